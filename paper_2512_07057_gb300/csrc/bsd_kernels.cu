// bsd_kernels.cu -- sm_103a kernels of the BP-guided beam search decoder.
//
// One warp owns one BP candidate (the seed path of a shot, or one child of a
// beam round) and keeps its whole state in shared memory: the edge messages
// E_{j->i}, over which the single-warp and jagged engines write the
// detector-to-error messages D_{i->j} and back (the generic engine keeps a
// compact 8-byte per-detector record, min1 and min2 with the sign parity in both
// sign bits, in D's place), sum_LLR, and the bit vectors s', mask, vals, e^ and the running syndrome parity.
//
// Kernels (all persistent: candidate groups claim shots with one atomic and leave
// when the counter runs out, or draw children from the beam's ring and leave when
// every shot has ended, so uneven iteration counts balance):
//   k_screen<DV>  (generic engines, every Lambda_j > 0, one result) a warp per
//                 shot forms e^(1) from the columns next to flipped detectors;
//                 finalises the shots that converge there, queues the rest
//   k_screen2<DV> the same for e^(2) of the shots k_screen passes on, from the
//                 columns that may flip (sparse syndromes)
//   k_seed<DV>    the seed BP of every shot in a chunk, or of the queued ones
//                 (Alg. 3, first BP run)
//   k_round<DV>   the beam of every shot: expand + masked BP of its children
//                 (Alg. 2) round by round; after the last child of a round
//                 select_entry takes the first success in visit order, the
//                 results, the top-w pruning and the next round's children
//                 (Alg. 3, App. B)
//   k_bp_llr<DV>  plain BP for a fixed number of iterations (LLR measurement)
//
// Arithmetic follows the readings stated in include/bsd.h: D = alpha * sign *
// min with the minimum over no other unmasked neighbour equal to L_MAX;
// E clamped to [-L_MAX, L_MAX]; the sums of Eqs. 2-3 start at Lambda_j and
// add the incoming messages in ascending order; every add and multiply is a
// single IEEE round-to-nearest operation (__fadd_rn / __fmul_rn, so no FMA
// contraction); scores and weights are summed exactly on a 2^-16 grid.
//
// Masked nodes: the messages of a masked error node are set to +L_MAX when it
// is masked.  A +L_MAX input (or a larger one, which the check pass caps) never
// lowers a minimum below that of the other inputs and never flips a sign, so the
// check pass needs no mask test.  The generic engine's error-node pass skips masked
// nodes; the others take Lambda_j = +inf for them, which makes their messages +inf.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cmath>

#include "bsd_device.cuh"
#include "bsd_internal.cuh"
#include "bsd_ring.cuh"

namespace bsd {

// bytes and 16-byte vectors of one E snapshot (Epad is a multiple of 8)
__host__ __device__ __forceinline__ size_t snap_bytes(const DevGraph& g) { return (size_t)g.Epad * (size_t)g.msg_bytes; }
__host__ __device__ __forceinline__ int snap_vec16(const DevGraph& g) { return (int)(snap_bytes(g) / 16); }

// Early abort of a beam child (num_results = 1): once a child of the same shot
// with a lower canonical index has succeeded in this round, this child's
// result can no longer be the first success in visit order and is never read.
// The shot's key holds (round stamp << 32) | ~c of the lowest successful index
// c so far (atomicMax); a run loads it at the start of an iteration and
// checks it at the end, so the load's latency hides behind the iteration.
struct AbortCheck {
    const unsigned long long* key;   // null: never abort
    unsigned long long stamp;        // this round's stamp << 32
    unsigned c;                      // this child's canonical index
    __device__ __forceinline__ bool hit(unsigned long long v) const
    {
        return (v & 0xffffffff00000000ull) == stamp && (0xffffffffu - (unsigned)v) < c;
    }
};

// copy n16 16-byte vectors (the E snapshot) with the threads of a candidate
// group; kL2: the source was written by other SMs during this kernel, so it is
// read past the L1 cache, which is not coherent between them
template <bool kL2 = false, class G>
__device__ __forceinline__ void group_copy16(const G& grp, void* dst, const void* src, int n16)
{
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    for (int q = grp.rank(); q < n16; q += grp.size()) d[q] = kL2 ? __ldcg(s + q) : s[q];
}


// ----------------------------------------------------------------------------
// candidate groups: the threads that process one BP candidate together.
// WarpGroup is one warp (a block holds several candidates); BlockGroup is a
// whole block (one candidate per block), for codes whose per-candidate state
// leaves room for only a few warps per SM.  Every row and column is computed
// by one thread and every reduction is exact (minima with index ties, integer
// sums, XOR), so both give the same results bit for bit.
// ----------------------------------------------------------------------------
struct ArgRec {                // per-warp partial of the argmin / score reduction
    float best, second;
    int bj, pad;
    unsigned long long s;
};

struct WarpGroup {
    static constexpr bool kBlock = false;
    __device__ static WarpGroup make(char*) { return WarpGroup{}; }
    __device__ __forceinline__ int rank() const { return threadIdx.x & 31; }
    __device__ __forceinline__ int size() const { return 32; }
    __device__ __forceinline__ int warp() const { return 0; }
    __device__ __forceinline__ int nwarps() const { return 1; }
    __device__ __forceinline__ int index() const { return threadIdx.x >> 5; }       // candidate slot of the block
    __device__ __forceinline__ int per_block() const { return blockDim.x >> 5; }
    __device__ __forceinline__ void sync() const { __syncwarp(); }
    __device__ __forceinline__ bool any(bool p) const
    {
        const bool r = __any_sync(FULLMASK, p);
        __syncwarp();
        return r;
    }
    // (a shuffle passes the value, the barrier what lane 0 has seen before it)
    __device__ __forceinline__ int bcast(int v) const
    {
        const int r = __shfl_sync(FULLMASK, v, 0);
        __syncwarp();
        return r;
    }
    __device__ __forceinline__ uint32_t xor_all(uint32_t v) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v ^= __shfl_xor_sync(FULLMASK, v, o);
        return v;
    }
};

struct BlockGroup {
    static constexpr bool kBlock = true;
    ArgRec* rec;               // shared scratch: one record per warp (16 at most)
    __device__ static BlockGroup make(char* scratch) { return BlockGroup{reinterpret_cast<ArgRec*>(scratch)}; }
    __device__ __forceinline__ int rank() const { return threadIdx.x; }
    __device__ __forceinline__ int size() const { return blockDim.x; }
    __device__ __forceinline__ int warp() const { return threadIdx.x >> 5; }
    __device__ __forceinline__ int nwarps() const { return blockDim.x >> 5; }
    __device__ __forceinline__ int index() const { return 0; }
    __device__ __forceinline__ int per_block() const { return 1; }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    __device__ __forceinline__ bool any(bool p) const { return __syncthreads_or(p ? 1 : 0) != 0; }
    __device__ __forceinline__ int bcast(int v) const
    {
        if (threadIdx.x == 0) rec[0].bj = v;
        __syncthreads();
        const int r = rec[0].bj;
        __syncthreads();
        return r;
    }
    __device__ __forceinline__ uint32_t xor_all(uint32_t v) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v ^= __shfl_xor_sync(FULLMASK, v, o);
        if ((threadIdx.x & 31) == 0) rec[threadIdx.x >> 5].pad = (int)v;
        __syncthreads();
        uint32_t r = 0;
        for (int q = 0; q < nwarps(); ++q) r ^= (uint32_t)rec[q].pad;
        __syncthreads();
        return r;
    }
};

// shared scratch a candidate group needs beyond the candidate's own state

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// per-warp shared-memory footprint of one BP candidate
// detector-side region: M records of 8 bytes (GenericEngine), one D per word
// (SmallEngine with 16-bit messages), nothing where D lies over E; g.det_bytes is
// set with the engine choice
__host__ __device__ inline size_t det_region_bytes(const DevGraph& g) { return (size_t)g.det_bytes; }

constexpr size_t kSelectBytes = 2 * kMaxBeam * (sizeof(double) + 2 * sizeof(int));
__host__ __device__ inline size_t warp_smem_bytes(const DevGraph& g)
{
    const size_t n = align16((size_t)g.e_bytes * (size_t)g.Epad) + det_region_bytes(g) +
                     align16(sizeof(float) * (size_t)g.Npad) + align16(sizeof(uint32_t) * (size_t)(2 * g.WM + 3 * g.WN + 1));
    return n > kSelectBytes ? n : kSelectBytes;   // the selection's scratch lies over the candidate's state
}

struct WarpState {
    void* E;           // [Epad] E_{j->i} in the storage format, CSR edge order
    float2* rs;        // [M]    (min1, min2), s'_i xor the parity of the negative messages in both sign bits
    float* D;          // [Epad] D_{i->j} per CSR edge (same storage as rs)
    float* sumllr;     // [Npad]
    uint32_t* sp;      // [WM] s' = s with the columns of nodes fixed to 1 folded in
    uint32_t* par;     // [WM] s' xor H e^ (zero iff converged)
    uint32_t* mask;    // [WN]
    uint32_t* vals;    // [WN]
    uint32_t* ehat;    // [WN]
    uint32_t* ab;      // [1] a lower-index sibling has succeeded (early abort)
};

__device__ inline WarpState carve(char* base, const DevGraph& g)
{
    WarpState s;
    char* p = base;
    s.E = p;                                 p += align16((size_t)g.e_bytes * (size_t)g.Epad);
    s.rs = reinterpret_cast<float2*>(p);
    s.D = reinterpret_cast<float*>(p);       p += det_region_bytes(g);
    s.sumllr = reinterpret_cast<float*>(p);  p += align16(sizeof(float) * (size_t)g.Npad);
    uint32_t* b = reinterpret_cast<uint32_t*>(p);
    s.sp = b;
    s.par = b + g.WM;
    s.mask = b + 2 * g.WM;
    s.vals = b + 2 * g.WM + g.WN;
    s.ehat = b + 2 * g.WM + 2 * g.WN;
    s.ab = b + 2 * g.WM + 3 * g.WN;
    return s;
}

// round(x * 2^16) to the nearest integer, ties to even: scaling a float by a
// power of two is exact, so single precision gives the value double would
// (GB300's double-precision pipe is narrow)
__device__ inline unsigned long long fixq(float x)
{
    return (unsigned long long)__float2ll_rn(__fmul_rn(x, (float)kFixScale));
}

// ----------------------------------------------------------------------------
// BP iterations on one candidate (Eqs. 1-4 with the masking of Alg. 2)
// ----------------------------------------------------------------------------
// Runs up to max_iters flooding iterations from the messages in st.E.  With
// stop = true it returns at the first t with H e^(t) = s' (Alg. 2).  On return
// st.ehat holds e^(t) of the last iteration (masked positions 0), st.sumllr
// holds the sum over the iterations run of Lambda_j(t).  With kPostOut,
// Lambda_j(max_iters) is written to post_out.
template <int DV, int P, bool W, bool kPostOut, class G>
__device__ int bp_iterate(const G& grp, const DevGraph& g, const DecCfg& cfg, const WarpState& st, int max_iters,
                          bool stop, int* success, float* post_out, bool from_prior, const AbortCheck& ab)
{
    using S = Store<P>;
    using T = typename S::T;
    T* const E = reinterpret_cast<T*>(st.E);
    const int lane = threadIdx.x & 31;
    const float alpha = cfg.alpha;
    const float L = cfg.L;
    int iters = 0;
    int ok = 0;
    for (int t = 1; t <= max_iters; ++t) {
        unsigned long long ab_key = 0ull;
        if (ab.key != nullptr && grp.rank() == 0) ab_key = *((volatile const unsigned long long*)ab.key);
        for (int q = grp.rank(); q < g.WM; q += grp.size()) st.par[q] = st.sp[q];
        // weighted min-sum: row min(t, wT) - 1 of the weights in place of alpha
        const float* wt = W ? cfg.weights + (size_t)((t < cfg.wT ? t : cfg.wT) - 1) * (size_t)g.Epad : nullptr;

        // a run from E(0) (seed, LLRs): the first check pass is the
        // precomputed E(0) record of each row with the syndrome bit folded into
        // the sign parity, and E(0) itself (clamp(Lambda), the same on every
        // edge of a column) is read from the graph, not from the candidate
        const bool prior = from_prior && t == 1;
        if (prior) {
            for (int i = grp.rank(); i < g.M; i += grp.size()) {
                const float4 r = __ldg(g.rs0 + i);
                const uint32_t sb = (((st.sp[i >> 5] >> (i & 31)) ^ __float_as_uint(r.w)) & 1u) << 31;
                st.rs[i] = make_float2(__uint_as_float(__float_as_uint(r.x) | sb),
                                       __uint_as_float(__float_as_uint(r.y) | sb));
            }
        }
        // ---- detector pass (Eq. 1): min1, min2 and the sign parity per row
        // (8-byte records: the error pass tells the edge holding the minimum
        // by its magnitude -- where the minimum is attained twice, min2 =
        // min1, so this equals the lowest-index argmin rule)
        for (int i = prior ? g.M : grp.rank(); i < g.M; i += grp.size()) {
            const int rb = __ldg(g.row_ptr + i), re = __ldg(g.row_ptr + i + 1);
            float m1 = L, m2 = L;
            uint32_t sg = ((st.sp[i >> 5] >> (i & 31)) & 1u) << 31;
            // branch-free: the runner-up is min(m2, max(m1, a)); a stored
            // message is never -0 (a clamped sum that starts at Lambda_j), so
            // its sign bit is exactly x < 0
            // (four messages per step; past the row's end a lane takes
            // +L_MAX, which changes neither minimum nor the parity)
            for (int e = rb; e < re; e += 4) {
                float x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = (e + u < re) ? S::ld(E, e + u) : L;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float a = fabsf(x[u]);
                    m2 = fminf(m2, fmaxf(m1, a));
                    m1 = fminf(m1, a);
                    sg ^= __float_as_uint(x[u]);
                }
            }
            sg &= 0x80000000u;
            st.rs[i] = make_float2(__uint_as_float(__float_as_uint(m1) | sg), __uint_as_float(__float_as_uint(m2) | sg));
        }
        grp.sync();

        // D_{i->j} of column j's edges in ascending order (padding +inf last),
        // with their CSR edge ids; returns the column's degree
        auto gather = [&](int j, float (&v)[DV], int (&ed)[DV]) -> int {
            const int kb = __ldg(g.col_ptr + j), deg = __ldg(g.col_ptr + j + 1) - kb;
            // E(0) is the same on every edge of a column: one load
            const float x0 = prior ? S::ld(reinterpret_cast<const T*>(g.lamEc), j) : 0.f;
#pragma unroll
            for (int k = 0; k < DV; ++k) {
                if (k < deg) {
                    const int e = __ldg(g.col_edge + kb + k);
                    const int r = __ldg(g.col_row + kb + k);
                    const float2 r2 = st.rs[r];
                    const float x = prior ? x0 : S::ld(E, e);
                    // the minimum over the row's other edges: min2 on an edge
                    // holding the minimum, min1 elsewhere; sign: the row's
                    // parity without the edge's own sign
                    const float m = (fabsf(x) == fabsf(r2.x)) ? fabsf(r2.y) : fabsf(r2.x);
                    const uint32_t sg = (__float_as_uint(r2.x) ^ __float_as_uint(x)) & 0x80000000u;
                    const float d = __fmul_rn(W ? __ldg(wt + e) : alpha, m);
                    v[k] = __uint_as_float(__float_as_uint(d) ^ sg);
                    ed[k] = e;
                } else {
                    v[k] = INFINITY;
                    ed[k] = -1;
                }
            }
            // ascending order of value (exchange network)
#pragma unroll
            for (int a = 0; a < DV; ++a) {
#pragma unroll
                for (int k = 0; k + 1 < DV - a; ++k) {
                    if (v[k] > v[k + 1]) {
                        const float tv = v[k]; v[k] = v[k + 1]; v[k + 1] = tv;
                        const int te = ed[k]; ed[k] = ed[k + 1]; ed[k + 1] = te;
                    }
                }
            }
            return deg;
        };
        auto flip_rows = [&](int j, int deg) {                 // s' xor H e^: the rows of column j
            for (int k = 0; k < deg; ++k) {
                const int r = __ldg(g.col_row + __ldg(g.col_ptr + j) + k);
                atomicXor(&st.par[r >> 5], 1u << (r & 31));
            }
        };

        // ---- error-node pass (Eqs. 2-4) and syndrome parity; each warp owns
        // whole 32-column words of e^ (one column per lane)
        auto column = [&](int jb) -> uint32_t {
            const int j = jb + lane;
            uint32_t ebit = 0;
            const bool act = (j < g.N) && !((st.mask[jb >> 5] >> lane) & 1u);
            if (act) {
                float v[DV];
                int ed[DV];
                const int deg = gather(j, v, ed);
                const float lj = __ldg(g.lam + j);
#pragma unroll
                for (int k = 0; k < DV; ++k) {                    // Eq. 2: leave d_i out
                    if (k < deg) {
                        float acc = lj;
#pragma unroll
                        for (int k2 = 0; k2 < DV; ++k2)
                            if (k2 != k && k2 < deg) acc = __fadd_rn(acc, v[k2]);
                        S::st(E, ed[k], fminf(fmaxf(acc, -L), L));
                    }
                }
                float post = lj;                                  // Eq. 3
#pragma unroll
                for (int k = 0; k < DV; ++k)
                    if (k < deg) post = __fadd_rn(post, v[k]);
                // a run from E(0) starts its sums here (0 + post, as a sum from zero)
                st.sumllr[j] = __fadd_rn(prior ? 0.f : st.sumllr[j], post);
                if (kPostOut && t == max_iters) post_out[j] = post;
                ebit = (post <= 0.f) ? 1u : 0u;                   // Eq. 4
                if (ebit) flip_rows(j, deg);
            }
            return ebit;
        };
        for (int jb = 32 * grp.warp(); jb < g.N; jb += 32 * grp.nwarps()) {
            const uint32_t bal = __ballot_sync(FULLMASK, column(jb));
            if (lane == 0) st.ehat[jb >> 5] = bal;
        }
        grp.sync();

        // ---- stopping rule: H e^(t) = s'
        uint32_t nz = 0;
        for (int q = grp.rank(); q < g.WM; q += grp.size()) nz |= st.par[q];
        ok = !grp.any(nz != 0u);
        iters = t;
        grp.sync();
        if (ok && stop) break;
        if (ab.key != nullptr && grp.any(grp.rank() == 0 && ab.hit(ab_key))) { ok = 0; break; }
    }
    *success = ok;
    return iters;
}

// reduction of per-thread (two smallest |sum_LLR|, node of the smallest, sum
// of q(|sum_LLR|)) over a candidate group: the smaller value wins, equal
// values go to the lower node index; every step is exact, so the result does
// not depend on the group's shape.  *tie is set when the relative margin
// between the smallest and the second smallest lies strictly inside
// (0, guard).
__device__ __forceinline__ void merge_argmin(float& best, float& second, int& bj, float ob, float os, int oj)
{
    second = fminf(fmaxf(best, ob), fminf(second, os));
    if (oj >= 0 && (bj < 0 || ob < best || (ob == best && oj < bj))) { best = ob; bj = oj; }
}

template <class G>
__device__ inline void reduce_argmin_score(const G& grp, float best, float second, int bj, unsigned long long s,
                                           double guard, int* next_pos, long long* S, int* tie)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(FULLMASK, best, o);
        const float os = __shfl_xor_sync(FULLMASK, second, o);
        const int oj = __shfl_xor_sync(FULLMASK, bj, o);
        merge_argmin(best, second, bj, ob, os, oj);
        s += __shfl_xor_sync(FULLMASK, s, o);
    }
    if constexpr (G::kBlock) {
        if ((threadIdx.x & 31) == 0) grp.rec[threadIdx.x >> 5] = ArgRec{best, second, bj, 0, s};
        __syncthreads();
        best = INFINITY; second = INFINITY; bj = -1; s = 0;
        for (int q = 0; q < grp.nwarps(); ++q) {
            const ArgRec r = grp.rec[q];
            merge_argmin(best, second, bj, r.best, r.second, r.bj);
            s += r.s;
        }
        __syncthreads();
    }
    *next_pos = bj;
    *S = (long long)s;
    int t = 0;
    if (guard > 0.0 && bj >= 0 && second != INFINITY) {
        const double den = fabs((double)second) > 1.0 ? fabs((double)second) : 1.0;
        const double gap = ((double)second - (double)best) / den;
        t = (gap > 0.0 && gap < guard) ? 1 : 0;
    }
    *tie = t;
}

// per-lane update of (smallest, second smallest, node of the smallest); nodes
// arrive in ascending order, so the lowest index keeps ties
__device__ __forceinline__ void two_smallest(float a, int j, float* best, float* second, int* bj)
{
    if (*bj < 0 || a < *best) {
        *second = *best;
        *best = a;
        *bj = j;
    } else if (a < *second) {
        *second = a;
    }
}

// least reliable unmasked node (lowest index on ties) and the score numerator
template <class G>
__device__ inline void argmin_and_score(const G& grp, const DevGraph& g, const WarpState& st, double guard,
                                        int* next_pos, long long* S, int* tie)
{
    float best = INFINITY, second = INFINITY;
    int bj = -1;
    unsigned long long s = 0;
    for (int j = grp.rank(); j < g.N; j += grp.size()) {
        if ((st.mask[j >> 5] >> (j & 31)) & 1u) continue;
        const float a = fabsf(st.sumllr[j]);
        two_smallest(a, j, &best, &second, &bj);
        s += fixq(a);
    }
    reduce_argmin_score(grp, best, second, bj, s, guard, next_pos, S, tie);
}

// ----------------------------------------------------------------------------
// BP engines: how one warp runs the iterations of one candidate
// ----------------------------------------------------------------------------
// GenericEngine: any code whose column degree is at most DV (used for degrees
// above 6, and for 16-bit messages that do not fit on chip as the floats of the
// jagged engine); graph tables are read from global memory (L1-resident) and
// sum_LLR lives in shared memory.
template <int DV, int P, bool W = false, class G = WarpGroup>
struct GenericEngine {
    using Grp = G;
    static constexpr int kMinBlocks = 1;
    static constexpr int kMaxThreads = G::kBlock ? 512 : 256;
    static constexpr int kPrec = P;
    static constexpr bool kPriorStart = true;   // runs from E(0) need no copy of E(0)
    static constexpr bool kPriorSetsSums = true;  // ... nor cleared sums: their first iteration sets them
    G grp;
    __device__ void load_graph(const DevGraph&, const WarpState&) {}
    __device__ void start_prior(const DevGraph&, const WarpState&) const {}
    // snapshots: the messages as they are kept
    __device__ void load_E(const DevGraph& g, const WarpState& st, const void* src) const
    {
        group_copy16<true>(grp, st.E, src, snap_vec16(g));
    }
    __device__ void save_E(const DevGraph& g, const WarpState& st, void* dst) const
    {
        group_copy16(grp, dst, st.E, snap_vec16(g));
    }
    // the sentinel +L_MAX on every message of the newly fixed node j
    __device__ void fix_node(const DevGraph& g, const WarpState& st, int j, float L) const
    {
        typename Store<P>::T* const E = reinterpret_cast<typename Store<P>::T*>(st.E);
        for (int q = __ldg(g.col_ptr + j) + grp.rank(); q < __ldg(g.col_ptr + j + 1); q += grp.size())
            Store<P>::st(E, __ldg(g.col_edge + q), L);
    }
    __device__ void clear_sums(const DevGraph& g, const WarpState& st)
    {
        for (int j = grp.rank(); j < g.N; j += grp.size()) st.sumllr[j] = 0.f;
    }
    template <bool kPostOut = false>
    __device__ int run(const DevGraph& g, const DecCfg& cfg, const WarpState& st, int max_iters, bool stop,
                       int* success, float* post_out, bool from_prior = false, const AbortCheck& ab = AbortCheck{})
    {
        return bp_iterate<DV, P, W, kPostOut>(grp, g, cfg, st, max_iters, stop, success, post_out, from_prior, ab);
    }
    __device__ void argmin_score(const DevGraph& g, const WarpState& st, double guard, int* np, long long* S,
                                 int* tie)
    {
        argmin_and_score(grp, g, st, guard, np, S, tie);
    }
    __device__ void write_sums(const DevGraph& g, const WarpState& st, float* dst)
    {
        for (int j = grp.rank(); j < g.N; j += grp.size()) dst[j] = st.sumllr[j];
    }
};

// SmallEngine: codes with every column of degree exactly 3, every row of
// degree exactly RD = 6, N <= 32*CPL, M <= 32*RPL -- the bivariate bicycle
// codes.  A candidate's messages sit at the words of the code's placement
// (bsd_layout.cu): the pair h of row i at h kPlane + 2 i, so the detector pass
// moves 32 consecutive pairs per access.  The columns are dealt to the lanes so
// that each row of a full group of 32 rows has two columns in its own lane: the
// messages on these edges (128 of 432 on [[144,12,12]]) stay in registers between
// the passes.  The other words are spread over the banks of their column group.
// With single-precision storage D is written over E (each word belongs to one
// row and to one (column, k), so either pass reads its words before it writes
// them); 16-bit storage keeps D in float beside E.  Each lane keeps its columns'
// shared-memory addresses, Lambda_j, sum_LLR and its first row's columns in
// registers.
//
// What bounds the iteration: 4 shared-memory transfers per edge that is not held
// in a register (44 wavefronts on [[144,12,12]], 54 if all 432 edges were in
// memory), and the ALU pipe, which runs min, max, compare, select and logic at 64
// lanes per clock (an add or multiply runs on the other pipe at 128).  So the
// detector pass takes each edge's minimum over the other five directly, with the
// sign product in the same instruction (min.xorsign.abs: the sign of the result is
// the xor of the operands'), 15 such operations per row of six instead of 13
// min/max, 6 compares, 6 selects and 12 logic operations; the cap at L_MAX carries
// the syndrome sign.  The
// stopping rule tests the parity of e^ on rows 0..31 from registers and goes on
// to the others only if these agree with s' (before: XOR of the set columns of
// H in every column pass and three warp reductions).  The beam of 10^6
// [[144,12,12]] shots at p = 0.05: 25.9 -> 17.4 ms, 15.1 with the ring and the
// register-held messages: issue, ALU and shared memory at about 60% each.
//
// Every value it produces is the one GenericEngine produces (same operations,
// same order; the placement only permutes where a row's edges and a column's
// edges are kept, and neither pass depends on that order).
__device__ __forceinline__ float xmin(float a, float b)
{
    float r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// two single-precision operations in one instruction, each rounded to nearest
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;}" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;}" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
// shared-memory accesses by 32-bit address, kept in program order (the code
// below loads a step ahead of its stores; the compiler cannot see that the
// words differ)
__device__ __forceinline__ float lds(uint32_t a)
{
    float r;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(r) : "r"(a) : "memory");
    return r;
}
__device__ __forceinline__ float2 lds2(uint32_t a)
{
    float2 r;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "r"(a) : "memory");
    return r;
}
__device__ __forceinline__ void sts(uint32_t a, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sts2(uint32_t a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

template <int CPL, int RPL, int RD, int P, bool W = false>
struct SmallEngine {
    using Grp = WarpGroup;
    // three 8-warp blocks per SM (at most 80 registers): k_round of 10^6
    // [[144,12,12]] shots at p = 0.05 took 17.4 ms against 18.0 with two
    // blocks (128 registers) and 18.1 with four (64 registers, 4 bytes spilled)
    static constexpr int kMinBlocks = 3;
    static constexpr int kMaxThreads = 256;
    static constexpr int kPrec = P;
    static constexpr bool kPriorStart = !W;  // unweighted runs from E(0) start from the table D0
    static constexpr bool kPriorSetsSums = false;
    static constexpr bool kInPlace = P == 0; // D over E
    static constexpr int LC = 2 * (RPL - 1); // column groups with a register-held message
    WarpGroup grp;
    using S = Store<P>;
    static_assert(RD == 6, "the placement holds rows of degree 6");
    static_assert(CPL == LC + 1, "every full row group has two column groups of its own, the last columns one");
    static constexpr int kPlane = small_plane_stride_rpl(RPL);   // words between a row's pairs
    uint32_t ca[CPL][3];   // shared-memory address of the D message on the k-th edge of the lane's column c
    uint32_t hq[CPL];      // the columns of row `lane` of H, by position
    float sum[CPL];
    uint32_t mb;           // bit c: the lane's column c is masked or there is none

    static __device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
    // the storage format's value of a message
    static __device__ __forceinline__ float rnd(float x)
    {
        if constexpr (P == 0) return x;
        typename S::T t;
        S::st(&t, 0, x);
        return S::ld(&t, 0);
    }
    static __device__ __forceinline__ int column(const DevGraph& g, int c)
    {
        return __ldg(&g.scol[(threadIdx.x & 31) + 32 * c].x);
    }
    __device__ void load_graph(const DevGraph& g, const WarpState& st)
    {
        const int lane = threadIdx.x & 31;
        const uint32_t base = saddr(kInPlace ? st.E : (void*)st.D);
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int4 q = __ldg(g.scol + lane + 32 * c);
            hq[c] = __ldg(g.shrow + (size_t)kSmallRowWords * lane + c);
            ca[c][0] = base + 4u * (uint32_t)q.y;
            ca[c][1] = base + 4u * (uint32_t)q.z;
            ca[c][2] = base + 4u * (uint32_t)q.w;
        }
    }
    __device__ void start_prior(const DevGraph& g, const WarpState& st) const
    {
        group_copy16(grp, st.E, g.slamE, snap_vec16(g));
    }
    // snapshots: the messages as they are kept
    __device__ void load_E(const DevGraph& g, const WarpState& st, const void* src) const
    {
        group_copy16<true>(grp, st.E, src, snap_vec16(g));
    }
    __device__ void save_E(const DevGraph& g, const WarpState& st, void* dst) const
    {
        group_copy16(grp, dst, st.E, snap_vec16(g));
    }
    __device__ void fix_node(const DevGraph& g, const WarpState& st, int j, float L) const
    {
        const int lane = threadIdx.x & 31;
        if (lane < 3)
            Store<P>::st(reinterpret_cast<typename Store<P>::T*>(st.E), __ldg(g.sword + 3 * j + lane), L);
    }
    __device__ void clear_sums(const DevGraph&, const WarpState&)
    {
#pragma unroll
        for (int c = 0; c < CPL; ++c) sum[c] = 0.f;
    }
    template <bool kPostOut = false>
    __device__ int run(const DevGraph& g, const DecCfg& cfg, const WarpState& st, int max_iters, bool stop,
                       int* success, float* post_out, bool from_prior = false, const AbortCheck& ab = AbortCheck{})
    {
        const int lane = threadIdx.x & 31;
        const float2 alpha2 = make_float2(cfg.alpha, cfg.alpha);
        typename S::T* const E = reinterpret_cast<typename S::T*>(st.E);
        const uint32_t dbase = saddr(kInPlace ? st.E : (void*)st.D);
        const uint32_t drow = dbase + 8u * lane;         // D of the lane's first row
        // Lambda_j of the lane's columns; +inf for a masked column or a position
        // without one: its messages and posterior are then +inf, which the
        // detector pass reads as L_MAX and positive (the sentinel of a masked
        // node) and Eq. 4 as e^_j = 0, with no test in the loop
        float l[CPL];
        // the messages of the edges between the lane's rows and its columns:
        // E after the error-node pass, D after the detector pass
        float own[LC];
        mb = 0u;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int j = column(g, c);
            const bool out = j < 0 || ((st.mask[j >> 5] >> (j & 31)) & 1u);
            if (out) mb |= 1u << c;
            l[c] = out ? INFINITY : __ldg(g.lam + j);
            if (c < LC) own[c] = S::ld(E, 2 * (lane + 32 * (c / 2)) + (c & 1));
        }
        // L_MAX with the sign (-1)^{s'_i} of the lane's rows (s' is fixed for the run)
        float sL[RPL];
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const uint32_t sb = (lane + 32 * r < g.M) ? ((st.sp[r] >> lane) & 1u) << 31 : 0u;
            sL[r] = __uint_as_float(__float_as_uint(cfg.L) | sb);
        }
        int iters = 0;
        int ok = 0;
        uint32_t bal[CPL];     // e^ by position in the last iteration (the same in every lane)
#pragma unroll
        for (int c = 0; c < CPL; ++c) bal[c] = 0u;
        for (int t = 1; t <= max_iters; ++t) {
            unsigned long long ab_key = 0ull;
            if (ab.key != nullptr && lane == 0) ab_key = *((volatile const unsigned long long*)ab.key);
            // weighted min-sum: row min(t, wT) - 1 of the weights in place of alpha
            const float* wt = W ? cfg.sweights + (size_t)((t < cfg.wT ? t : cfg.wT) - 1) * (size_t)g.Epad : nullptr;
            // ---- detector pass (Eq. 1)
            if (!W && from_prior && t == 1) {
                // a run from E(0) takes its first check messages from the table
                // D0, flipping the sign where s_i = 1
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    const int i = lane + 32 * r;
                    if (i < g.M) {
                        const uint32_t sb = __float_as_uint(sL[r]) & 0x80000000u;
#pragma unroll
                        for (int h = 0; h < 3; ++h) {
                            const float2 v = __ldg(reinterpret_cast<const float2*>(g.sD0 + h * kPlane + 2 * i));
                            const float2 d = make_float2(__uint_as_float(__float_as_uint(v.x) ^ sb),
                                                         __uint_as_float(__float_as_uint(v.y) ^ sb));
                            if (h == 0 && r < RPL - 1) {
                                own[2 * (r < RPL - 1 ? r : 0)] = d.x;
                                own[2 * (r < RPL - 1 ? r : 0) + 1] = d.y;
                            } else {
                                sts2(drow + 4u * (h * kPlane + 64 * r), d);
                            }
                        }
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < RPL; ++r) {
                    const int i = lane + 32 * r;
                    const bool held = r < RPL - 1;       // the row's pair 0 is in registers (a full row group)
                    const int o = held ? 2 * r : 0;
                    if (held || i < g.M) {
                        float2 x[3];
#pragma unroll
                        for (int h = 0; h < 3; ++h) {
                            if (held && h == 0) x[h] = make_float2(own[o], own[o + 1]);
                            else
                                x[h] = kInPlace ? lds2(drow + 4u * (h * kPlane + 64 * r)) : S::ld2(E, h * kPlane + 2 * i);
                        }
                        // D_{i->j} = alpha (-1)^{s_i} prod sign min over the other
                        // five messages (R3, R4): p[h] the signed minimum of pair
                        // h, q[h] that of the other two pairs capped at L_MAX with
                        // the syndrome sign (a stored message is never -0, so its
                        // sign bit is exactly x < 0; min(|x|, L_MAX) is exact)
                        float p[3], q[3];
#pragma unroll
                        for (int h = 0; h < 3; ++h) p[h] = xmin(x[h].x, x[h].y);
                        q[0] = xmin(xmin(p[1], p[2]), sL[r]);
                        q[1] = xmin(xmin(p[0], p[2]), sL[r]);
                        q[2] = xmin(xmin(p[0], p[1]), sL[r]);
#pragma unroll
                        for (int h = 0; h < 3; ++h) {
                            float2 w2 = alpha2;
                            if (W) w2 = __ldg(reinterpret_cast<const float2*>(wt + h * kPlane + 2 * i));
                            const float2 d = mul2(w2, make_float2(xmin(x[h].y, q[h]), xmin(x[h].x, q[h])));
                            if (held && h == 0) {
                                own[o] = d.x;
                                own[o + 1] = d.y;
                            } else {
                                sts2(drow + 4u * (h * kPlane + 64 * r), d);
                            }
                        }
                    }
                }
            }
            __syncwarp();
            // ---- error-node pass (Eqs. 2-4), the next column's messages loaded
            // before this one's are stored
            float v[2][3];
            auto load_column = [&](int c, float (&d)[3]) {
#pragma unroll
                for (int k = 0; k < 3; ++k) d[k] = (k == 0 && c < LC) ? own[c < LC ? c : 0] : lds(ca[c][k]);
            };
            load_column(0, v[0]);
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                if (c + 1 < CPL) load_column(c + 1, v[(c + 1) & 1]);
                const float v0 = v[c & 1][0], v1 = v[c & 1][1], v2 = v[c & 1][2];
                // Eq. 2: each message leaves its own detector out; the other two
                // are added in ascending order.  Messages are stored unclamped:
                // the detector pass reads min(|E|, L_MAX) and the sign, which is
                // what a clamp at store time (R4) would leave.  Eq. 3 in ascending
                // order: smallest, median (the least of the pair maxima), largest.
                const float lo12 = fminf(v1, v2), hi12 = fmaxf(v1, v2);
                const float lo02 = fminf(v0, v2), hi02 = fmaxf(v0, v2);
                const float lo01 = fminf(v0, v1), hi01 = fmaxf(v0, v1);
                const float2 ll = make_float2(l[c], l[c]);
                const float2 e01 = add2(add2(ll, make_float2(lo12, lo02)), make_float2(hi12, hi02));
                const float2 e2p = add2(add2(ll, make_float2(lo01, fminf(lo01, v2))),
                                        make_float2(hi01, fmin3(hi01, hi02, hi12)));
                const float post = __fadd_rn(e2p.y, fmaxf(hi01, v2));
                const bool inr = c < LC || lane + 32 * c < g.N;   // only the last group may pass N
                const float e[3] = {e01.x, e01.y, e2p.x};
                if (c < LC) own[c < LC ? c : 0] = rnd(e[0]);
                if (inr) {
#pragma unroll
                    for (int k = c < LC ? 1 : 0; k < 3; ++k) {
                        if (kInPlace) sts(ca[c][k], e[k]);
                        else S::st(E, (ca[c][k] - dbase) >> 2, e[k]);
                    }
                }
                sum[c] = __fadd_rn(sum[c], post);           // unused for masked columns
                if (kPostOut && t == max_iters && inr) st.sumllr[column(g, c)] = post;
                bal[c] = __ballot_sync(FULLMASK, post <= 0.f);                       // Eq. 4
            }
            __syncwarp();
            // ---- stopping rule H e^ = s': the parity of e^ on the lane's row
            // against s'_i, first on rows 0..31 (their columns stay in
            // registers: most iterations end here), then on the others
            uint32_t acc = 0u;
#pragma unroll
            for (int c = 0; c < CPL; ++c) acc ^= bal[c] & hq[c];
            ok = !__any_sync(FULLMASK, ((__popc(acc) & 1u) ^ (__float_as_uint(sL[0]) >> 31)) != 0u);
            if (RPL > 1 && ok) {
                uint32_t bad = 0u;
#pragma unroll
                for (int r = 1; r < RPL; ++r) {
                    const uint32_t* hr = g.shrow + (size_t)kSmallRowWords * (lane + 32 * r);
                    uint32_t a2 = 0u;
#pragma unroll
                    for (int c = 0; c < CPL; ++c) a2 ^= bal[c] & __ldg(hr + c);
                    bad |= (__popc(a2) & 1u) ^ (__float_as_uint(sL[r]) >> 31);
                }
                ok = !__any_sync(FULLMASK, bad != 0u);
            }
            iters = t;
            if (ok && stop) break;
            if (ab.key != nullptr && __any_sync(FULLMASK, lane == 0 && ab.hit(ab_key))) { ok = 0; break; }
        }
        if constexpr (kPostOut) {
            copy_row(g, st.sumllr, post_out);            // (messages and e^ are not read)
        } else {
            // the register-held messages join the others, and e^ of the last
            // iteration run goes back to natural order
#pragma unroll
            for (int c = 0; c < LC; ++c) S::st(E, 2 * (lane + 32 * (c / 2)) + (c & 1), own[c]);
            if (iters > 0) {
                if (lane < CPL) st.ehat[lane] = 0u;
                __syncwarp();
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    if ((bal[c] >> lane) & 1u) {
                        const int j = column(g, c);
                        atomicOr(&st.ehat[j >> 5], 1u << (j & 31));
                    }
                }
            }
        }
        *success = ok;
        return iters;
    }
    __device__ void argmin_score(const DevGraph& g, const WarpState&, double guard, int* np, long long* S,
                                 int* tie)
    {
        float best = INFINITY, second = INFINITY;
        int bj = -1;
        unsigned long long s = 0;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            if ((mb >> c) & 1u) continue;
            const float a = fabsf(sum[c]);
            merge_argmin(best, second, bj, a, INFINITY, column(g, c));
            s += fixq(a);
        }
        reduce_argmin_score(grp, best, second, bj, s, guard, np, S, tie);
    }
    // a row of N values in the columns' own order, staged in shared memory: stores by
    // the lanes' columns touch a sector each (plain BP of 8000 shots of [[144,12,12]],
    // T = 20: 87.6 -> 84.1 us, with the messages and e^ not put back either)
    __device__ void copy_row(const DevGraph& g, const float* src, float* dst) const
    {
        __syncwarp();
        for (int j = threadIdx.x & 31; j < g.N; j += 32) dst[j] = src[j];
        __syncwarp();
    }
    __device__ void write_sums(const DevGraph& g, const WarpState& st, float* dst)
    {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const int j = column(g, c);
            if (j >= 0) st.sumllr[j] = sum[c];
        }
        copy_row(g, st.sumllr, dst);
    }
};

// exchange networks of 2 to 6 inputs (the last three with the fewest
// comparators known): comparator c orders inputs x(c) < y(c), the c-th digits of
// two hexadecimal numbers
template <int N> struct SortNet;
template <> struct SortNet<1> { static constexpr int n = 0; static constexpr unsigned long long x = 0x0ull, y = 0x0ull; };
template <> struct SortNet<2> { static constexpr int n = 1; static constexpr unsigned long long x = 0x0ull, y = 0x1ull; };
template <> struct SortNet<3> { static constexpr int n = 3; static constexpr unsigned long long x = 0x100ull, y = 0x212ull; };
template <> struct SortNet<4> { static constexpr int n = 5; static constexpr unsigned long long x = 0x12010ull, y = 0x23132ull; };
template <> struct SortNet<5> { static constexpr int n = 9; static constexpr unsigned long long x = 0x231201010ull, y = 0x342413243ull; };
template <> struct SortNet<6> { static constexpr int n = 12; static constexpr unsigned long long x = 0x314202031210ull, y = 0x425315342435ull; };

// JaggedEngine: any code whose column degree is at most DV <= 6 (the detector
// error models, stacked X and Z checks).  The rows stand in order of falling
// degree and the k-th edges of all rows lie side by side (jagged diagonals,
// DevGraph::jplane), so the detector pass -- lane = row -- moves 32 consecutive
// words per access whatever the degrees; a row's edges are permuted among its
// words and a column's among its slots so that the error pass meets few bank
// conflicts (bsd_layout.cu).  D is written over E: a row's and a column's words
// are its own in either pass.  Messages are floats holding values of the
// storage format; snapshots are converted.
//
// The detector pass takes each edge's minimum over the others with its sign
// from running signed minima from both ends (three min.xorsign.abs per edge, the
// cap at L_MAX with the syndrome sign in the first; rows above degree 16 read
// their messages twice instead).  The error pass runs the exact network of the
// columns' degree where the 32 columns of a group have the same one (degree 3
// without a sort, as the single-warp engine), and one padded to the largest
// degree where they differ; a code most of whose groups would differ has its
// columns dealt to the groups by degree (DevGraph::colJ).  Masked columns and the clamp are handled as in the
// single-warp engine.
//
// Before (records of the two smallest magnitudes per row, one thread per CSR
// row, networks of DV inputs for every column) the detector pass of rows of
// equal degree met 4- to 8-way bank conflicts and an iteration took 2.9 warp
// instructions per edge.
template <int DV, int P, bool W = false, class G = WarpGroup>
struct JaggedEngine {
    using Grp = G;
    // blocks of up to 16 warps in 64 registers: two of them resident on an SM;
    // one warp per candidate: 80 registers, three 8-warp blocks
    static constexpr int kMinBlocks = G::kBlock ? 2 : 3;
    static constexpr int kMaxThreads = G::kBlock ? 512 : 256;
    static constexpr int kPrec = P;
    static constexpr bool kPriorStart = !W;       // unweighted runs from E(0) start from the table D0
    static constexpr bool kPriorSetsSums = true;  // a run from E(0) needs no cleared sums
    using S = Store<P>;
    static constexpr int kRegWords = G::kBlock ? 1 : 6;
    G grp;

    // the storage format's value of a message
    static __device__ __forceinline__ float rnd(float x)
    {
        if constexpr (P == 0) return x;
        typename S::T t;
        S::st(&t, 0, x);
        return S::ld(&t, 0);
    }
    static __device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
    __device__ void load_graph(const DevGraph&, const WarpState&) {}
    __device__ void start_prior(const DevGraph& g, const WarpState& st) const
    {
        float* const E = reinterpret_cast<float*>(st.E);
        for (int j = grp.rank(); j < g.N; j += grp.size()) {
            const float v = S::ld(reinterpret_cast<const typename S::T*>(g.lamEc), j);
#pragma unroll
            for (int k = 0; k < DV; ++k) {
                const int e = __ldg(g.colN + (size_t)k * g.Npad + j);
                if (e >= 0) E[e] = v;
            }
        }
    }
    __device__ void load_E(const DevGraph& g, const WarpState& st, const void* src) const
    {
        if constexpr (P == 0) {
            group_copy16<true>(grp, st.E, src, snap_vec16(g));
        } else {
            const uint4* s = reinterpret_cast<const uint4*>(src);
            float4* d = reinterpret_cast<float4*>(st.E);
            for (int q = grp.rank(); q < snap_vec16(g); q += grp.size()) {
                const uint4 v = __ldcg(s + q);
                const typename S::T* h = reinterpret_cast<const typename S::T*>(&v);
                d[2 * q] = make_float4(S::ld(h, 0), S::ld(h, 1), S::ld(h, 2), S::ld(h, 3));
                d[2 * q + 1] = make_float4(S::ld(h, 4), S::ld(h, 5), S::ld(h, 6), S::ld(h, 7));
            }
        }
    }
    __device__ void save_E(const DevGraph& g, const WarpState& st, void* dst) const
    {
        if constexpr (P == 0) {
            group_copy16(grp, dst, st.E, snap_vec16(g));
        } else {
            uint4* d = reinterpret_cast<uint4*>(dst);
            const float* s = reinterpret_cast<const float*>(st.E);
            for (int q = grp.rank(); q < snap_vec16(g); q += grp.size()) {
                uint4 v;
                typename S::T* h = reinterpret_cast<typename S::T*>(&v);
#pragma unroll
                for (int u = 0; u < 8; ++u) S::st(h, u, s[8 * q + u]);
                d[q] = v;
            }
        }
    }
    // the sentinel +L_MAX on every message of the newly fixed node j
    __device__ void fix_node(const DevGraph& g, const WarpState& st, int j, float L) const
    {
        for (int k = grp.rank(); k < DV; k += grp.size()) {
            const int e = __ldg(g.colN + (size_t)k * g.Npad + j);
            if (e >= 0) reinterpret_cast<float*>(st.E)[e] = L;
        }
    }
    __device__ void clear_sums(const DevGraph& g, const WarpState& st)
    {
        for (int j = grp.rank(); j < g.N; j += grp.size()) st.sumllr[j] = 0.f;
    }

    // D over E on the row of rank q, of degree RD (kSame) or deg <= RD
    template <int RD, bool kSame>
    static __device__ __forceinline__ void row_pass(const DevGraph& g, uint32_t eb, int q, int deg, float sL, float alpha,
                                                    const float* wt)
    {
        float x[RD], after[RD];
        uint32_t a[RD];
#pragma unroll
        for (int k = 0; k < RD; ++k) {
            a[k] = eb + 4u * (uint32_t)(g.jplane[k] + q);
            x[k] = kSame || k < deg ? lds(a[k]) : INFINITY;
        }
        after[RD - 1] = INFINITY;                  // the messages after k
#pragma unroll
        for (int k = RD - 1; k > 0; --k) after[k - 1] = k == RD - 1 ? x[k] : xmin(x[k], after[k]);
        float before = sL;                         // those before k, capped, with the syndrome sign
#pragma unroll
        for (int k = 0; k < RD; k += 2) {
            const int k1 = k + 1 < RD ? k + 1 : k;
            const float m0 = k == RD - 1 ? before : xmin(before, after[k]);
            before = xmin(before, x[k]);
            const float m1 = k1 == RD - 1 ? before : xmin(before, after[k1]);
            if (k1 + 1 < RD) before = xmin(before, x[k1]);
            float2 w2 = make_float2(alpha, alpha);
            if (W) {
                if (kSame || k < deg) w2.x = __ldg(wt + g.jplane[k] + q);
                if (kSame || k1 < deg) w2.y = __ldg(wt + g.jplane[k1] + q);
            }
            const float2 d = mul2(w2, make_float2(m0, m1));
            if (kSame || k < deg) sts(a[k], d.x);
            if (k1 > k && (kSame || k1 < deg)) sts(a[k1], d.y);
        }
    }

    // Eqs. 2-3 for a column of degree DD (kSame), or at most DD with holes in its
    // slots: the messages over the column's words, the posterior returned
    template <int DD, bool kSame>
    static __device__ __forceinline__ float column(uint32_t eb, const int (&word)[DV], float l)
    {
        if constexpr (DD == 0) {
            return l;
        } else {
            float v[DD];
            uint32_t a[DD];
#pragma unroll
            for (int k = 0; k < DD; ++k) a[k] = (kSame || word[k] >= 0) ? eb + 4u * (uint32_t)word[k] : 0xffffffffu;
#pragma unroll
            for (int k = 0; k < DD; ++k) v[k] = (kSame || a[k] != 0xffffffffu) ? lds(a[k]) : INFINITY;
            if constexpr (DD == 3 && kSame) {
                const float lo12 = fminf(v[1], v[2]), hi12 = fmaxf(v[1], v[2]);
                const float lo02 = fminf(v[0], v[2]), hi02 = fmaxf(v[0], v[2]);
                const float lo01 = fminf(v[0], v[1]), hi01 = fmaxf(v[0], v[1]);
                const float2 ll = make_float2(l, l);
                const float2 e01 = add2(add2(ll, make_float2(lo12, lo02)), make_float2(hi12, hi02));
                const float2 e2p = add2(add2(ll, make_float2(lo01, fminf(lo01, v[2]))),
                                        make_float2(hi01, fmin3(hi01, hi02, hi12)));
                sts(a[0], rnd(e01.x));
                sts(a[1], rnd(e01.y));
                sts(a[2], rnd(e2p.x));
                return __fadd_rn(e2p.y, fmaxf(hi01, v[2]));
            } else {
                // ascending order of value, the addresses along
#pragma unroll
                for (int c = 0; c < SortNet<DD>::n; ++c) {
                    const int x = (int)((SortNet<DD>::x >> (4 * c)) & 15u), y = (int)((SortNet<DD>::y >> (4 * c)) & 15u);
                    const bool sw = v[x] > v[y];
                    const float lo = fminf(v[x], v[y]), hi = fmaxf(v[x], v[y]);
                    const uint32_t al = sw ? a[y] : a[x], ah = sw ? a[x] : a[y];
                    v[x] = lo; v[y] = hi;
                    a[x] = al; a[y] = ah;
                }
                // (a hole adds +0, which changes no sum)
                if (!kSame) {
#pragma unroll
                    for (int k = 0; k < DD; ++k) v[k] = a[k] == 0xffffffffu ? 0.f : v[k];
                }
                float pre = l;
#pragma unroll
                for (int k = 0; k < DD; ++k) {                    // Eq. 2: leave d_i out
                    float acc = pre;
#pragma unroll
                    for (int k2 = k + 1; k2 < DD; ++k2) acc = __fadd_rn(acc, v[k2]);
                    if (kSame || a[k] != 0xffffffffu) sts(a[k], rnd(acc));
                    pre = __fadd_rn(pre, v[k]);
                }
                return pre;                                       // Eq. 3
            }
        }
    }

    template <bool kPostOut = false>
    __device__ int run(const DevGraph& g, const DecCfg& cfg, const WarpState& st, int max_iters, bool stop,
                       int* success, float* post_out, bool from_prior = false, const AbortCheck& ab = AbortCheck{})
    {
        const int lane = threadIdx.x & 31;
        const uint32_t eb = saddr(st.E);
        int iters = 0;
        int ok = 0;
        for (int t = 1; t <= max_iters; ++t) {
            unsigned long long ab_key = 0ull;
            if (ab.key != nullptr && grp.rank() == 0) ab_key = *((volatile const unsigned long long*)ab.key);
            // H e^(t): with a warp per candidate and few words of rows, the XOR of
            // the set columns of H in the lanes' registers, else of their rows
            // in shared memory
            const bool inreg = !G::kBlock && g.WM <= kRegWords;
            uint32_t hx[kRegWords];
            if (inreg) {
#pragma unroll
                for (int q = 0; q < kRegWords; ++q) hx[q] = 0u;
            } else {
                for (int q = grp.rank(); q < g.WM; q += grp.size()) st.par[q] = st.sp[q];
            }
            if (g.colJ != nullptr)
                for (int q = grp.rank(); q < g.WN; q += grp.size()) st.ehat[q] = 0u;
            // weighted min-sum: row min(t, wT) - 1 of the weights in place of alpha
            const float* wt = W ? cfg.weights + (size_t)((t < cfg.wT ? t : cfg.wT) - 1) * (size_t)g.Epad : nullptr;
            // ---- detector pass (Eq. 1); a run from E(0) takes its first check
            // messages from the table D0, flipping the sign where s_i = 1
            const bool prior = from_prior && t == 1;
            for (int q = grp.rank(); q < g.M; q += grp.size()) {
                const int2 rd = __ldg(g.rowQ + q);
                const uint32_t sb = ((st.sp[rd.x >> 5] >> (rd.x & 31)) & 1u) << 31;
                if (!W && prior) {
                    for (int k = 0; k < rd.y; ++k) {
                        const int e = __ldg(g.jplanes + k) + q;
                        sts(eb + 4u * (uint32_t)e, __uint_as_float(__float_as_uint(__ldg(g.jD0 + e)) ^ sb));
                    }
                    continue;
                }
                const float sL = __uint_as_float(__float_as_uint(cfg.L) | sb);
                // the warp's largest degree, + 32 when its rows have another too
                const int dmax = __ldg(g.rowG + (q >> 5));
                if (dmax == 8) {
                    row_pass<8, true>(g, eb, q, 8, sL, cfg.alpha, wt);
                } else if (dmax == 12) {
                    row_pass<12, true>(g, eb, q, 12, sL, cfg.alpha, wt);
                } else if ((dmax & 31) <= 8 && dmax < 64) {
                    row_pass<8, false>(g, eb, q, rd.y, sL, cfg.alpha, wt);
                } else if ((dmax & 31) <= 16 && dmax < 64) {
                    row_pass<16, false>(g, eb, q, rd.y, sL, cfg.alpha, wt);
                } else {
                    // the two smallest magnitudes and the sign parity, then D:
                    // the minimum over the others is m2 on an edge holding the
                    // minimum (a tie makes m2 = m1), m1 elsewhere
                    float m1 = cfg.L, m2 = cfg.L;
                    uint32_t sg = sb;
#pragma unroll 4
                    for (int k = 0; k < rd.y; ++k) {
                        const float x = lds(eb + 4u * (uint32_t)(__ldg(g.jplanes + k) + q)), m = fabsf(x);
                        m2 = fminf(m2, fmaxf(m1, m));
                        m1 = fminf(m1, m);
                        sg ^= __float_as_uint(x) & 0x80000000u;
                    }
#pragma unroll 4
                    for (int k = 0; k < rd.y; ++k) {
                        const int e = __ldg(g.jplanes + k) + q;
                        const float x = lds(eb + 4u * (uint32_t)e);
                        const float d = __fmul_rn(W ? __ldg(wt + e) : cfg.alpha, fabsf(x) == m1 ? m2 : m1);
                        sts(eb + 4u * (uint32_t)e,
                            __uint_as_float(__float_as_uint(d) ^ sg ^ (__float_as_uint(x) & 0x80000000u)));
                    }
                }
            }
            if (ab.key != nullptr && grp.rank() == 0) st.ab[0] = ab.hit(ab_key) ? 1u : 0u;
            grp.sync();
            // ---- error-node pass (Eqs. 2-4) and syndrome parity; each warp owns
            // whole 32-column words of e^ (one column per lane)
            // (the next group's table entries are loaded while this one runs)
            int nj = 0, nw[DV], ng = 0;
            float nl = 0.f;
            auto fetch = [&](int jb) {
                if (jb >= g.N) return;
                const int p = min(jb + lane, g.N - 1);
                ng = __ldg(g.colG + (jb >> 5));
                nj = g.colJ != nullptr ? __ldg(g.colJ + p) : p;
#pragma unroll
                for (int k = 0; k < DV; ++k) nw[k] = __ldg(g.colW + (size_t)k * g.Npad + p);
                nl = __ldg(g.lam + nj);
            };
            fetch(32 * grp.warp());
            for (int jb = 32 * grp.warp(); jb < g.N; jb += 32 * grp.nwarps()) {
                const int gd = ng, j = nj, p = jb + lane;
                int wd[DV];
#pragma unroll
                for (int k = 0; k < DV; ++k) wd[k] = nw[k];
                const float lj = nl;
                fetch(jb + 32 * grp.nwarps());
                bool ebit = false;
                if (p < g.N) {
                    const float l = ((st.mask[j >> 5] >> (j & 31)) & 1u) ? INFINITY : lj;
                    const float before = prior ? 0.f : st.sumllr[j];
                    float post;
                    switch (gd) {
                        case 0: post = column<0, true>(eb, wd, l); break;
                        case 1: post = column<1, true>(eb, wd, l); break;
                        case 2: post = column<2, true>(eb, wd, l); break;
                        case 3: post = column<3, true>(eb, wd, l); break;
                        case 9: case 10: case 11: post = column<3, false>(eb, wd, l); break;
                        default:
                            if constexpr (DV == 6) {
                                if (gd == 4) post = column<4, true>(eb, wd, l);
                                else if (gd == 5) post = column<5, true>(eb, wd, l);
                                else if (gd == 6) post = column<6, true>(eb, wd, l);
                                else post = column<6, false>(eb, wd, l);
                            } else {
                                post = l;
                            }
                    }
                    // a run from E(0) starts its sums here (0 + post, as a sum from zero)
                    st.sumllr[j] = __fadd_rn(before, post);
                    if (kPostOut && t == max_iters) post_out[j] = post;
                    ebit = post <= 0.f;                               // Eq. 4
                    if (ebit) {
                        if (g.colJ != nullptr) atomicOr(&st.ehat[j >> 5], 1u << (j & 31));
                        if (inreg) {
#pragma unroll
                            for (int q = 0; q < kRegWords; ++q)
                                if (q < g.WM) hx[q] ^= __ldg(g.hcol + (size_t)j * g.WM + q);
                        } else {
                            int rr[DV];
#pragma unroll
                            for (int k = 0; k < DV; ++k) rr[k] = __ldg(g.colF + (size_t)k * g.Npad + p);
#pragma unroll
                            for (int k = 0; k < DV; ++k)
                                if (rr[k] >= 0) atomicXor(&st.par[rr[k] >> 5], 1u << (rr[k] & 31));
                        }
                    }
                }
                if (g.colJ == nullptr) {
                    const uint32_t bal = __ballot_sync(FULLMASK, ebit);
                    if (lane == 0) st.ehat[jb >> 5] = bal;
                }
            }
            grp.sync();
            // ---- stopping rule: H e^(t) = s' (the vote's barrier also keeps the
            // next iteration's writes to par behind these reads); a child that
            // succeeds in the iteration at whose end it would stop has succeeded
            uint32_t nz = 0;
            if (inreg) {
#pragma unroll
                for (int q = 0; q < kRegWords; ++q)
                    if (q < g.WM) nz |= __reduce_xor_sync(FULLMASK, hx[q]) ^ st.sp[q];
            } else {
                for (int q = grp.rank(); q < g.WM; q += grp.size()) nz |= st.par[q];
            }
            const bool gone = ab.key != nullptr && st.ab[0] != 0u;
            ok = !grp.any(nz != 0u);
            iters = t;
            if (ok && stop) break;
            if (gone) { ok = 0; break; }
        }
        *success = ok;
        return iters;
    }
    __device__ void argmin_score(const DevGraph& g, const WarpState& st, double guard, int* np, long long* S,
                                 int* tie)
    {
        argmin_and_score(grp, g, st, guard, np, S, tie);
    }
    __device__ void write_sums(const DevGraph& g, const WarpState& st, float* dst)
    {
        for (int j = grp.rank(); j < g.N; j += grp.size()) dst[j] = st.sumllr[j];
    }
};

// write one shot's outputs: e^, A e^, status, iteration count
// (kSparse: A e^ from the set bits of e^, for the seed kernel, where e^ is
// long and sparse; kL2: e^ is in global memory and was written by other SMs
// during this kernel)
template <class G = WarpGroup, bool kSparse = false, bool kL2 = false>
__device__ void finalize_shot(const DevGraph& g, const Outputs& out, long long gb, const uint32_t* ehat,
                              uint32_t status, unsigned long long iters, const G& grp = G{})
{
    uint32_t* corr = out.corr + gb * g.WN;
    auto word = [&](int q) -> uint32_t { return kL2 ? __ldcg(ehat + q) : ehat[q]; };
    for (int q = grp.rank(); q < g.WN; q += grp.size()) corr[q] = word(q);
    if (out.obs != nullptr) {
        for (int wq = 0; wq < g.WK; ++wq) {
            uint32_t acc = 0;
            if constexpr (kSparse) {
                // over the set bits of e^ only (bits past N are never set)
                for (int q = grp.rank(); q < g.WN; q += grp.size()) {
                    uint32_t bits = word(q);
                    while (bits != 0u) {
                        const int b = __ffs(bits) - 1;
                        bits &= bits - 1u;
                        acc ^= __ldg(g.acol + (size_t)(32 * q + b) * g.WK + wq);
                    }
                }
            } else {
                for (int j = grp.rank(); j < g.N; j += grp.size())
                    if ((word(j >> 5) >> (j & 31)) & 1u) acc ^= __ldg(g.acol + (size_t)j * g.WK + wq);
            }
            acc = grp.xor_all(acc);
            if (grp.rank() == 0) out.obs[gb * g.WK + wq] = acc;
        }
    }
    if (grp.rank() == 0) {
        out.status[gb] = status;
        if (out.iters != nullptr) out.iters[gb] = iters > 0xffffffffull ? 0xffffffffu : (uint32_t)iters;
    }
}

// weight of a bit vector on the 2^-16 grid: sum of q(Lambda_j) over its support
__device__ inline long long vector_weight(const DevGraph& g, const uint32_t* bits)
{
    const int lane = threadIdx.x & 31;
    unsigned long long s = 0;
    for (int j = lane; j < g.N; j += 32)
        if ((__ldcg(bits + (j >> 5)) >> (j & 31)) & 1u) s += (unsigned long long)__ldg(g.lamq + j);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULLMASK, s, o);
    return (long long)s;
}

// slot of child c of window entry a in bank `bank`
__device__ inline size_t slot_index(const Work& w, int bank, int a, int c, int W2)
{
    return ((size_t)bank * (size_t)w.A + (size_t)a) * (size_t)W2 + (size_t)c;
}

// a parent in round r: the seed-store entry of the shot for r = 1, else child
// `slot` of the round before
struct SlotRef {
    const unsigned char* E;   // snapshot, Epad messages in the storage format
    const uint32_t* bits;
};

__device__ inline SlotRef parent_ref(const DevGraph& g, const DecCfg& cfg, const Work& w, int r, int seed, int a,
                                     int slot)
{
    SlotRef s;
    if (r == 1) {
        const size_t e = (size_t)seed;
        s.E = w.seedE + e * snap_bytes(g);
        s.bits = w.seedBits + e * (size_t)w.SB;
    } else {
        const size_t e = slot_index(w, (r - 1) & 1, a, slot, 2 * cfg.w);
        s.E = w.slotE + e * snap_bytes(g);
        s.bits = w.slotBits + e * (size_t)w.SB;
    }
    return s;
}

// records written by other SMs during the beam kernel, read past L1
__device__ inline SlotMeta load_meta(const SlotMeta* p)
{
    static_assert(sizeof(SlotMeta) == 24, "three 8-byte loads");
    const unsigned long long* q = reinterpret_cast<const unsigned long long*>(p);
    const unsigned long long x = __ldcg(q), y = __ldcg(q + 1), z = __ldcg(q + 2);
    SlotMeta m;
    m.S = (long long)x;
    m.iters = (int)(uint32_t)y;
    m.next_pos = (int)(uint32_t)(y >> 32);
    m.success = (int)(uint32_t)z;
    m.flags = (int)(uint32_t)(z >> 32);
    return m;
}
__device__ inline BeamEntry load_entry(const BeamEntry* p)
{
    const int4 v = __ldcg(reinterpret_cast<const int4*>(p));
    return BeamEntry{v.x, v.y, v.z, v.w};
}

// ----------------------------------------------------------------------------
// chunk set-up and beam set-up
// ----------------------------------------------------------------------------
__device__ inline void count_launch(const Work& w)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&w.stats[2], 1ull);
}

__global__ void k_begin_chunk(Work w, const uint32_t* synd, Outputs out, long long base, long long n)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        w.ctr->claim_seed = 0;
        w.ctr->n_active = 0;
        w.ctr->n_queue = 0;
        w.ctr->n_queue1 = 0;
        w.ctr->err = 0;
        w.ctr->bs_claim = 0;
        w.ctr->bs_run = 0;
        w.ctr->bs_active_next = 0;
        w.ctr->bs_done_blocks = 0;
        w.ctr->n_fail = 0;
        RunDesc d;
        d.synd = synd;
        d.out = out;
        d.chunk_base = base;
        d.chunk_n = n;
        d.win_base = 0;
        *w.desc = d;
    }
}

// graph only, after the seed kernel: run the beam only if some shot of the
// chunk needs it, and (windows) the loop over windows after it only if a shot
// found the seed store full
__global__ void k_beam_gate(Work w, cudaGraphConditionalHandle cond, cudaGraphConditionalHandle cwin, int windows)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        cudaGraphSetConditional(cond, w.ctr->n_active > 0 ? 1u : 0u);
        if (windows) cudaGraphSetConditional(cwin, w.ctr->n_fail > 0 ? 1u : 0u);
    }
}

// counters of a beam search over the n_active entries of the seed store: the
// first of them take the window entries, the others follow as entries end
__global__ void k_beam_begin(Work w, int beam_width)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        const int n = (int)((long long)w.ctr->n_active < w.S ? (long long)w.ctr->n_active : w.S);
        const int cnt = (long long)n < w.A ? n : (int)w.A;
        w.ctr->n_active = n;
        w.ctr->b_head = 0u;
        w.ctr->b_tail = 2u * (unsigned)cnt;
        w.ctr->b_left = n;
        w.ctr->b_next = cnt;
        // the ring for these entries: at most 2w items of each are on it at once
        uint32_t slots = 4;
        while ((unsigned long long)slots < 2ull * (unsigned long long)cnt * (unsigned)beam_width) slots *= 2;
        w.ctr->b_mask = slots - 1;
    }
}

// the first items of the ring, two children per window entry, and empty
// slots after them
__global__ void k_beam_ring(Work w)
{
    count_launch(w);
    const uint32_t n = w.ctr->b_tail, mask = w.ctr->b_mask;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q <= mask; q += gridDim.x * blockDim.x)
        w.ring[q] = q < n ? ring_item((int)(q >> 1), (int)(q & 1u)) : kRingEmpty;
}

// every shot of the beam ended with its outputs written, or the device-side
// error word says so (the beam kernel cannot leave one behind by design)
__global__ void k_beam_end(Work w)
{
    count_launch(w);
    if (threadIdx.x == 0 && w.ctr->b_left != 0) w.ctr->err = kErrBeam;
}

// batched seed BP: the shots it hands on are decoded from the seed on in
// windows of at most S shots (the seed store); graph only: enter the loop
// over windows if there is any
__global__ void k_win_gate(Work w, cudaGraphConditionalHandle cond)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        w.desc->win_base = 0;
        cudaGraphSetConditional(cond, *((volatile int*)&w.ctr->n_fail) > 0 ? 1u : 0u);
    }
}

// start of a window: the per-window counters start afresh, as at the start of
// a chunk (base < 0: keep the window base)
__global__ void k_win_begin(Work w, int base)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        w.ctr->claim_seed = 0;
        w.ctr->n_active = 0;
        if (base >= 0) w.desc->win_base = base;
    }
}

// end of a window: graph only, another window if the fail list goes on
__global__ void k_win_end(Work w, cudaGraphConditionalHandle cond)
{
    count_launch(w);
    if (threadIdx.x == 0) {
        const long long nb = (long long)w.desc->win_base + w.S;
        w.desc->win_base = (int)(nb < 0x7fffffffll ? nb : 0x7fffffffll);
        cudaGraphSetConditional(cond, nb < (long long)*((volatile int*)&w.ctr->n_fail) ? 1u : 0u);
    }
}

// ----------------------------------------------------------------------------
// first-iteration screen of the seed runs (generic engines)
// ----------------------------------------------------------------------------
// With every Lambda_j > 0, the scale alpha and one result, E(0) carries no
// negative sign, so at t = 1 a detector i with s_i = 0 sends
// D_{i->j}(1) = alpha min_{j' != j} Lambda_{j'} > 0 to every neighbour, and a
// column none of whose detectors is flipped has Lambda_j(1) > 0, e^_j(1) = 0.
// One warp per shot forms e^(1) from the columns next to flipped detectors
// (each once), by the operations and in the order of the seed BP's first
// iteration (its check messages are the create-time table D0 of E(0) with the
// syndrome sign, the values bp_iterate forms from the E(0) records; the sums
// of Eq. 3 in ascending order), and tests H e^(1) = s.  A shot
// that converges (or has s = 0) is finalised here: its seed BP would stop at
// t = 1 with this e^, and a converged seed with one result reads neither E(1)
// nor sum_LLR.  The others go to the seed BP through the queue.  The state of
// a warp is four bit vectors, so many shots are in flight per SM.
//
// Most columns next to a flipped detector are next to one only, and whether
// that flip alone makes e^_j(1) = 1 does not depend on the shot: it is a bit of
// the edge (DevGraph::scrC).  So Eqs. 2-4 are formed only for the columns met
// a second time and those whose bit is set (of about 285 columns per shot of
// the synthetic DEM some 10 are; 10^6 shots 5.4 -> 2.1 ms).
constexpr int kScreenWarps = 8;
constexpr int kMaxFlip = 128;

__host__ __device__ inline size_t screen_warp_words(const DevGraph& g)
{
    return 2 * (size_t)g.WN + 2 * (size_t)g.WM + 2 * (size_t)kMaxFlip + 64;
}

// (more: the shots that do not converge go to the second-iteration screen)
template <int DV>
__global__ void k_screen(DevGraph g, DecCfg cfg, Work w, int more)
{
    extern __shared__ __align__(16) uint32_t ssm[];
    const int lane = threadIdx.x & 31;
    uint32_t* seen = ssm + (size_t)(threadIdx.x >> 5) * screen_warp_words(g);
    uint32_t* eh = seen + g.WN;
    uint32_t* sp = eh + g.WN;
    uint32_t* par = sp + g.WM;
    int* fst = reinterpret_cast<int*>(par + g.WM);    // [kMaxFlip] flipped detectors, then their first edges
    int* foff = fst + kMaxFlip;                       // [kMaxFlip] their edges' offsets in the shot's list
    int* cand = foff + kMaxFlip;                      // [64] columns to form
    count_launch(w);
    const RunDesc* dp = w.desc;
    const long long n = dp->chunk_n;
    const long long nw = (long long)gridDim.x * kScreenWarps;
    unsigned long long upd = 0;                  // message updates formed (lane)
    for (long long b = (long long)blockIdx.x * kScreenWarps + (threadIdx.x >> 5); b < n; b += nw) {
        const long long gb = dp->chunk_base + b;
        const uint32_t* s = dp->synd + gb * g.WM;
        uint32_t nz = 0;
        for (int q = lane; q < g.WM; q += 32) {
            const uint32_t x = s[q];
            sp[q] = x;
            par[q] = x;
            nz |= x;
        }
        for (int q = lane; q < g.WN; q += 32) { seen[q] = 0u; eh[q] = 0u; }
        __syncwarp();
        bool conv = !__any_sync(FULLMASK, nz != 0u);
        if (!conv) {
            // the flipped detectors, in order (a shot with more than kMaxFlip
            // goes to the seed BP unscreened)
            int nflip = 0;
            for (int q0 = 0; q0 < g.WM; q0 += 32) {
                const int q = q0 + lane;
                const uint32_t word = q < g.WM ? sp[q] : 0u;
                const int c = __popc(word);
                int incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULLMASK, incl, o);
                    if (lane >= o) incl += y;
                }
                int k = nflip + incl - c;
                if (k + c <= kMaxFlip) {
                    for (uint32_t w2 = word; w2 != 0u; w2 &= w2 - 1u) fst[k++] = 32 * q + __ffs(w2) - 1;
                }
                nflip += __shfl_sync(FULLMASK, incl, 31);
            }
            if (nflip <= kMaxFlip) {
                __syncwarp();
                // each flipped detector's first edge and its edges' offset in
                // the shot's list of (detector, edge) pairs
                int tot = 0;
                for (int k0 = 0; k0 < nflip; k0 += 32) {
                    const int k = k0 + lane;
                    int rb = 0, d = 0;
                    if (k < nflip) {
                        const int i = fst[k];
                        rb = __ldg(g.row_ptr + i);
                        d = __ldg(g.row_ptr + i + 1) - rb;
                    }
                    int incl = d;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(FULLMASK, incl, o);
                        if (lane >= o) incl += y;
                    }
                    if (k < nflip) {
                        fst[k] = rb;
                        foff[k] = tot + incl - d;
                    }
                    tot += __shfl_sync(FULLMASK, incl, 31);
                }
                __syncwarp();
                // D_{i'->j}(1) on the column's edges: the check message of
                // E(0) on the edge (the same for every shot: E(0) > 0 on
                // every edge, so it is alpha times the row's minimum over the
                // other edges, positive) with the syndrome bit of its row as
                // the sign; two (message, row) pairs per 16-byte load, padding
                // (+inf, -1) past the column's degree.  (A column listed twice
                // is formed twice with the same result.)
                auto form = [&](int j) {
                    constexpr int KD = DV == 3 ? 4 : DV;
                    const float4* cr = g.colRD + (size_t)j * (KD / 2);
                    float v[KD];
                    int rr[KD];
                    int deg = 0;
#pragma unroll
                    for (int h = 0; h < KD / 2; ++h) {
                        const float4 q = __ldg(cr + h);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int r = __float_as_int(u ? q.w : q.y);
                            const float d = u ? q.z : q.x;
                            const int rs = r >= 0 ? r : 0;
                            const uint32_t si = (r >= 0) ? (sp[rs >> 5] >> (rs & 31)) & 1u : 0u;
                            v[2 * h + u] = __uint_as_float(__float_as_uint(d) ^ (si << 31));
                            rr[2 * h + u] = r;
                            deg += (r >= 0) ? 1 : 0;
                        }
                    }
#pragma unroll
                    for (int a = 0; a < KD; ++a) {
#pragma unroll
                        for (int k = 0; k + 1 < KD - a; ++k) {
                            if (v[k] > v[k + 1]) { const float tv = v[k]; v[k] = v[k + 1]; v[k + 1] = tv; }
                        }
                    }
                    float post = __ldg(g.lam + j);               // Eq. 3 in ascending order
#pragma unroll
                    for (int k = 0; k < KD; ++k)
                        if (k < deg) post = __fadd_rn(post, v[k]);
                    upd += (unsigned long long)deg;
                    const uint32_t bit = 1u << (j & 31);
                    if (post <= 0.f && !(atomicOr(&eh[j >> 5], bit) & bit)) {   // Eq. 4
#pragma unroll
                        for (int k = 0; k < KD; ++k)
                            if (rr[k] >= 0) atomicXor(&par[rr[k] >> 5], 1u << (rr[k] & 31));
                    }
                };
                // one (detector, edge) pair per lane: the column on the edge,
                // listed when another flipped detector had it or its bit is set
                int nc = 0;
                for (int t0 = 0; t0 < tot; t0 += 32) {
                    const int t = t0 + lane;
                    bool add = false;
                    int j = 0;
                    if (t < tot) {
                        int lo = 0, hi = nflip - 1;                // last detector with foff <= t
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (foff[mid] <= t) lo = mid; else hi = mid - 1;
                        }
                        const uint32_t c = __ldg(g.scrC + fst[lo] + (t - foff[lo]));
                        j = (int)(c & 0x7fffffffu);
                        const uint32_t bit = 1u << (j & 31);
                        add = (atomicOr(&seen[j >> 5], bit) & bit) || (c >> 31);
                    }
                    const uint32_t bal = __ballot_sync(FULLMASK, add);
                    if (add) cand[nc + __popc(bal & ((1u << lane) - 1u))] = j;
                    nc += __popc(bal);
                    __syncwarp();
                    if (nc >= 32) {
                        form(cand[lane]);
                        const int rest = lane < nc - 32 ? cand[32 + lane] : 0;
                        __syncwarp();
                        cand[lane] = rest;
                        nc -= 32;
                        __syncwarp();
                    }
                }
                if (lane < nc) form(cand[lane]);
                __syncwarp();
                nz = 0;
                for (int q = lane; q < g.WM; q += 32) nz |= par[q];
                conv = !__any_sync(FULLMASK, nz != 0u);
            }
        }
        if (conv) {
            finalize_shot<WarpGroup, true>(g, dp->out, gb, eh, ST_SEED, 1ull);
        } else if (lane == 0) {
            const int k = atomicAdd(more ? &w.ctr->n_queue1 : &w.ctr->n_queue, 1);
            (more ? w.queue1 : w.queue)[k] = (int)b;
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) upd += __shfl_xor_sync(FULLMASK, upd, o);
    if (lane == 0 && upd != 0ull) atomicAdd(&w.stats[3], upd);
}

// ----------------------------------------------------------------------------
// second-iteration screen (generic engines, sparse syndromes)
// ----------------------------------------------------------------------------
// E(1) differs from its value for s = 0 (the create-time E0(1) > 0) only on the
// columns next to flipped detectors.  So the row records of E(1) -- the two
// smallest magnitudes and the parity P_i of s_i and the negative messages --
// follow from the row's few smallest E0(1) on other columns (DevGraph::row4)
// and those columns' messages, and at t = 2 a column meets a negative check
// message, without which Lambda_j(2) > 0, only in a row with P_i odd or through
// a negative E(1) of its own.  One warp per shot forms Lambda_j(2) for these
// columns, by the operations and in the order of the seed BP's second
// iteration, and tests H e^(2) = s.  A shot that converges is finalised here
// with two iterations; the others (and any whose lists overflow) go to the seed
// BP.
//
// It pays where the flipped detectors' columns are few (configure_kernels): of
// the synthetic 936 x 8800 DEM's shots 14% pass the first screen and 97% of
// those end here, after about 300 columns each way instead of two passes over
// 35110 edges.
constexpr int kScreen2Cols = 1024;       // columns next to flipped detectors, and
constexpr int kScreen2Cand = 512;        // columns to form at t = 2 (some of them more than once), of one shot

__host__ __device__ inline size_t screen2_warp_words(const DevGraph& g)
{
    return (size_t)g.WN + 3 * (size_t)g.WM + 3 * (size_t)kMaxFlip + (kScreen2Cols + kScreen2Cand) / 2 +
           2 * (size_t)g.M;
}

// the set rows of a bit set (rows): each one's first edge (first) and its
// edges' offset (off) in the list of all their edges; returns their number,
// *tot = the edges (nothing is listed when there are more than kMaxFlip)
__device__ inline int list_rows(const DevGraph& g, const uint32_t* bits, int* rows, int* first, int* off, int* tot)
{
    const int lane = threadIdx.x & 31;
    int n = 0;
    for (int q0 = 0; q0 < g.WM; q0 += 32) {
        const int q = q0 + lane;
        const uint32_t word = q < g.WM ? bits[q] : 0u;
        const int c = __popc(word);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULLMASK, incl, o);
            if (lane >= o) incl += y;
        }
        int k = n + incl - c;
        if (k + c <= kMaxFlip) {
            for (uint32_t w2 = word; w2 != 0u; w2 &= w2 - 1u) rows[k++] = 32 * q + __ffs(w2) - 1;
        }
        n += __shfl_sync(FULLMASK, incl, 31);
    }
    *tot = 0;
    if (n > kMaxFlip) return n;
    __syncwarp();
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int k = k0 + lane;
        int rb = 0, d = 0;
        if (k < n) {
            const int i = rows[k];
            rb = __ldg(g.row_ptr + i);
            d = __ldg(g.row_ptr + i + 1) - rb;
        }
        int incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULLMASK, incl, o);
            if (lane >= o) incl += y;
        }
        if (k < n) {
            first[k] = rb;
            off[k] = *tot + incl - d;
        }
        *tot += __shfl_sync(FULLMASK, incl, 31);
    }
    __syncwarp();
    return n;
}

// the columns on the listed rows' edges, appended to list[cap]: those `seen` does
// not hold yet, or with m2 (the rows' second smallest magnitudes at m2[2 i + 1])
// those it holds and those whose Lambda_j one negative message of the row could
// bring to 0; returns the list's length, above cap when it overflows
template <bool kBound>
__device__ inline int list_columns(const DevGraph& g, const int* rows, const int* first, const int* off, int n, int tot,
                                   uint32_t* seen, uint16_t* list, int len, int cap, const uint32_t* m2, float alpha)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 2
    for (int t0 = 0; t0 < tot; t0 += 32) {
        const int t = t0 + lane;
        bool add = false;
        int j = 0;
        if (t < tot) {
            int lo = 0, hi = n - 1;                        // last row with off <= t
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (off[mid] <= t) lo = mid; else hi = mid - 1;
            }
            j = __ldg(g.row_col + first[lo] + (t - off[lo]));
            const uint32_t bit = 1u << (j & 31);
            const bool had = atomicOr(&seen[j >> 5], bit) & bit;
            if (kBound)
                add = had || !(__fsub_rn(__ldg(g.lam + j), __fmul_rn(alpha, __uint_as_float(m2[2 * rows[lo] + 1]))) > 0.f);
            else
                add = !had;
        }
        const uint32_t bal = __ballot_sync(FULLMASK, add);
        const int at = len + __popc(bal & ((1u << lane) - 1u));
        if (add && at < cap) list[at] = (uint16_t)j;
        len += __popc(bal);
    }
    __syncwarp();
    return len;
}

// E_{j->i}(1) of column j in the storage format's values: v[k] on row rr[k],
// k < the column's degree (returned); its table entry is loaded ahead
template <int KD>
struct ColumnIn {
    float4 q[KD / 2];
    float lam;
};
template <int KD>
__device__ __forceinline__ void load_column(const DevGraph& g, int j, ColumnIn<KD>& in)
{
#pragma unroll
    for (int h = 0; h < KD / 2; ++h) in.q[h] = __ldg(g.colRD + (size_t)j * (KD / 2) + h);
    in.lam = __ldg(g.lam + j);
}
template <int KD, int P>
__device__ __forceinline__ int column_E1(const ColumnIn<KD>& in, const uint32_t* sp, float L, float (&v)[KD],
                                         int (&rr)[KD])
{
    using S = Store<P>;
    float d[KD];
    int deg = 0;
#pragma unroll
    for (int h = 0; h < KD / 2; ++h) {
        const float4 q = in.q[h];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int r = __float_as_int(u ? q.w : q.y);
            const uint32_t si = (r >= 0) ? (sp[(r >= 0 ? r : 0) >> 5] >> (r & 31)) & 1u : 0u;
            d[2 * h + u] = __uint_as_float(__float_as_uint(u ? q.z : q.x) ^ (si << 31));
            rr[2 * h + u] = r;
            deg += (r >= 0) ? 1 : 0;
        }
    }
    // ascending order of value, the padding (+inf) last
#pragma unroll
    for (int a = 0; a < KD; ++a) {
#pragma unroll
        for (int k = 0; k + 1 < KD - a; ++k) {
            if (d[k] > d[k + 1]) {
                const float tv = d[k]; d[k] = d[k + 1]; d[k + 1] = tv;
                const int tr = rr[k]; rr[k] = rr[k + 1]; rr[k + 1] = tr;
            }
        }
    }
    const float lj = in.lam;
#pragma unroll
    for (int k = 0; k < KD; ++k) {                            // Eq. 2: leave d_i out
        float acc = lj;
#pragma unroll
        for (int k2 = 0; k2 < KD; ++k2)
            if (k2 != k && k2 < deg) acc = __fadd_rn(acc, d[k2]);
        typename S::T x;
        S::st(&x, 0, fminf(fmaxf(acc, -L), L));
        v[k] = S::ld(&x, 0);
    }
    return deg;
}

template <int DV, int P>
__global__ void __launch_bounds__(32 * kScreenWarps) k_screen2(DevGraph g, DecCfg cfg, Work w, int min_queue)
{
    extern __shared__ __align__(16) uint32_t ssm[];
    constexpr int KD = DV == 3 ? 4 : DV;
    const int lane = threadIdx.x & 31;
    const size_t stride = screen2_warp_words(g);
    uint32_t* rec = ssm + (size_t)(threadIdx.x >> 5) * stride;      // [M] (min1, min2)
    uint32_t* bits = rec + 2 * (size_t)g.M;                          // [WN] columns listed, then e^(2)
    uint32_t* sp = bits + g.WN;
    uint32_t* pr = sp + g.WM;                                        // P_i
    uint32_t* par = pr + g.WM;                                       // s xor H e^(2)
    int* rows = reinterpret_cast<int*>(par + g.WM);
    int* first = rows + kMaxFlip;
    int* off = first + kMaxFlip;
    uint16_t* cols = reinterpret_cast<uint16_t*>(off + kMaxFlip);
    uint16_t* cand = cols + kScreen2Cols;
    count_launch(w);
    const RunDesc* dp = w.desc;
    const int nq = *((volatile int*)&w.ctr->n_queue1);
    const int nw = gridDim.x * kScreenWarps;
    // few shots: a warp here takes longer over one than the seed kernel's
    // candidate group over two iterations, and the groups are free
    if (nq < min_queue) {
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nq; k += gridDim.x * blockDim.x) w.queue[k] = w.queue1[k];
        if (blockIdx.x == 0 && threadIdx.x == 0) w.ctr->n_queue = nq;
        return;
    }
    const float L = cfg.L;
    unsigned long long upd = 0;                                      // message updates formed (lane)
    unsigned long long ended = 0;
    for (int k0 = blockIdx.x * kScreenWarps + (threadIdx.x >> 5); k0 < nq; k0 += nw) {
        const int b = w.queue1[k0];
        const long long gb = dp->chunk_base + b;
        const uint32_t* s = dp->synd + gb * g.WM;
        for (int q = lane; q < g.WM; q += 32) sp[q] = pr[q] = par[q] = s[q];
        for (int q = lane; q < g.WN; q += 32) bits[q] = 0u;
        __syncwarp();
        bool conv = false;
        int tot;
        const int nflip = list_rows(g, sp, rows, first, off, &tot);
        const int nc = nflip <= kMaxFlip ? list_columns<false>(g, rows, first, off, nflip, tot, bits, cols, 0,
                                                               kScreen2Cols, nullptr, 0.f)
                                         : kScreen2Cols + 1;
        if (nc <= kScreen2Cols) {
            // the records of E0(1) over the other columns: none on a flipped
            // row, whose columns are all listed; else the first two of the row's
            // four smallest, and a row that has fewer (more than two of the four
            // are next to flipped detectors) is read whole
#pragma unroll 4
            for (int i = lane; i < g.M; i += 32) {
                const float4 a0 = __ldg(g.row4 + 2 * i), a1 = __ldg(g.row4 + 2 * i + 1);
                const float x[4] = {a0.x, a0.z, a1.x, a1.z};
                const int c[4] = {__float_as_int(a0.y), __float_as_int(a0.w), __float_as_int(a1.y),
                                  __float_as_int(a1.w)};
                float m1 = L, m2 = L;
                int n = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool other = c[u] < 0 || !((bits[c[u] >> 5] >> (c[u] & 31)) & 1u);
                    if (other) {
                        if (n == 0) m1 = x[u];
                        else if (n == 1) m2 = x[u];
                        ++n;
                    }
                }
                if ((sp[i >> 5] >> (i & 31)) & 1u) {
                    m1 = m2 = L;
                } else if (n < 2) {
                    m1 = m2 = L;
                    for (int e = __ldg(g.row_ptr + i); e < __ldg(g.row_ptr + i + 1); ++e) {
                        const int j = __ldg(g.row_col + e);
                        if ((bits[j >> 5] >> (j & 31)) & 1u) continue;
                        const float a = __ldg(g.E1 + e);
                        m2 = fminf(m2, fmaxf(m1, a));
                        m1 = fminf(m1, a);
                    }
                }
                rec[2 * i] = __float_as_uint(m1);
                rec[2 * i + 1] = __float_as_uint(m2);
            }
            __syncwarp();
            for (int q = lane; q < g.WN; q += 32) bits[q] = 0u;
            __syncwarp();
            // the messages of the columns next to flipped detectors; the larger
            // of a message and the minimum it meets goes on to the second one,
            // which in the end is the least of all but the minimum (and one that
            // is not below the second one now never changes either)
            int ncand = 0;
            ColumnIn<KD> in, next;
            int j = lane < nc ? cols[lane] : 0;
            load_column<KD>(g, j, in);
            for (int t0 = 0; t0 < nc; t0 += 32) {
                bool neg = false;
                const int jn = t0 + 32 + lane < nc ? cols[t0 + 32 + lane] : 0;
                load_column<KD>(g, jn, next);
                if (t0 + lane < nc) {
                    float v[KD];
                    int rr[KD];
                    const int deg = column_E1<KD, P>(in, sp, L, v, rr);
#pragma unroll
                    for (int k = 0; k < KD; ++k) {
                        if (k < deg) {
                            const uint32_t a = __float_as_uint(fabsf(v[k]));
                            if (a < *((volatile uint32_t*)&rec[2 * rr[k] + 1])) {
                                const uint32_t old = atomicMin(&rec[2 * rr[k]], a);
                                atomicMin(&rec[2 * rr[k] + 1], old > a ? old : a);
                            }
                            if (v[k] < 0.f) {
                                neg = true;
                                atomicXor(&pr[rr[k] >> 5], 1u << (rr[k] & 31));
                            }
                        }
                    }
                    upd += (unsigned long long)deg;
                }
                const uint32_t bal = __ballot_sync(FULLMASK, neg);
                const int at = ncand + __popc(bal & ((1u << lane) - 1u));
                if (neg) {
                    atomicOr(&bits[j >> 5], 1u << (j & 31));
                    if (at < kScreen2Cand) cand[at] = (uint16_t)j;
                }
                ncand += __popc(bal);
                in = next;
                j = jn;
            }
            __syncwarp();
            if (ncand <= kScreen2Cand) {
                const int nodd = list_rows(g, pr, rows, first, off, &tot);
                ncand = nodd <= kMaxFlip ? list_columns<true>(g, rows, first, off, nodd, tot, bits, cand, ncand,
                                                              kScreen2Cand, rec, cfg.alpha)
                                         : kScreen2Cand + 1;
            }
            if (ncand <= kScreen2Cand) {
                for (int q = lane; q < g.WN; q += 32) bits[q] = 0u;
                __syncwarp();
                for (int t = lane; t < ncand; t += 32) {
                    const int j = cand[t];
                    float v[KD];
                    int rr[KD];
                    ColumnIn<KD> in;
                    load_column<KD>(g, j, in);
                    const int deg = column_E1<KD, P>(in, sp, L, v, rr);
#pragma unroll
                    for (int k = 0; k < KD; ++k) {            // Eq. 1
                        if (k < deg) {
                            const float m1 = __uint_as_float(rec[2 * rr[k]]), m2 = __uint_as_float(rec[2 * rr[k] + 1]);
                            const float d = __fmul_rn(cfg.alpha, fabsf(v[k]) == m1 ? m2 : m1);
                            const uint32_t sg = ((pr[rr[k] >> 5] >> (rr[k] & 31)) << 31) ^
                                                (__float_as_uint(v[k]) & 0x80000000u);
                            v[k] = __uint_as_float(__float_as_uint(d) ^ sg);
                        } else {
                            v[k] = INFINITY;
                        }
                    }
#pragma unroll
                    for (int a = 0; a < KD; ++a) {
#pragma unroll
                        for (int k = 0; k + 1 < KD - a; ++k) {
                            if (v[k] > v[k + 1]) { const float tv = v[k]; v[k] = v[k + 1]; v[k + 1] = tv; }
                        }
                    }
                    float post = in.lam;                      // Eq. 3 in ascending order
#pragma unroll
                    for (int k = 0; k < KD; ++k)
                        if (k < deg) post = __fadd_rn(post, v[k]);
                    upd += (unsigned long long)deg;
                    const uint32_t bit = 1u << (j & 31);
                    if (post <= 0.f && !(atomicOr(&bits[j >> 5], bit) & bit)) {   // Eq. 4
#pragma unroll
                        for (int k = 0; k < KD; ++k)
                            if (k < deg) atomicXor(&par[rr[k] >> 5], 1u << (rr[k] & 31));
                    }
                }
                __syncwarp();
                uint32_t nz = 0;
                for (int q = lane; q < g.WM; q += 32) nz |= par[q];
                conv = !__any_sync(FULLMASK, nz != 0u);
            }
        }
        if (conv) {
            finalize_shot<WarpGroup, true>(g, dp->out, gb, bits, ST_SEED, 2ull);
            ended += 2ull;
        } else if (lane == 0) {
            w.queue[atomicAdd(&w.ctr->n_queue, 1)] = b;
        }
        __syncwarp();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) upd += __shfl_xor_sync(FULLMASK, upd, o);
    if (lane == 0 && upd != 0ull) {
        atomicAdd(&w.stats[3], upd);
        if (ended != 0ull) atomicAdd(&w.stats[0], ended);
    }
}

// ----------------------------------------------------------------------------
// seed BP
// ----------------------------------------------------------------------------
template <class Eng>
__global__ void __launch_bounds__(Eng::kMaxThreads, Eng::kMinBlocks) k_seed(DevGraph g, DecCfg cfg, Work w,
                                                                             int screened)
{
    extern __shared__ __align__(16) char smem[];
    Eng eng;
    eng.grp = Eng::Grp::make(smem + warp_smem_bytes(g));
    const auto& grp = eng.grp;
    const WarpState st = carve(smem + (size_t)grp.index() * warp_smem_bytes(g), g);
    const RunDesc* dp = w.desc;                  // read fields when needed (keeps registers free)
    count_launch(w);
    eng.load_graph(g, st);
    unsigned long long seed_iters = 0;           // BP iterations (group rank 0)
    // a warp claims its shots four at a time (one atomic per batch on the
    // chunk's counter, which a million one-iteration seeds would otherwise hit a
    // million times), but one at a time once the shots left are few for the
    // grid, and where each is many iterations: a block candidate's, and those a
    // screen passed on (four failing seeds in one warp held up the end of the
    // kernel: 10^5 shots of depolarizing noise on [[144,12,12]] 6.7 -> 4.4 ms)
    const int total_warps = (int)(gridDim.x * grp.per_block());
    // the shots: every shot of the chunk (screened = 0), those the screen
    // passed on (1), or the current window of the fail list (2: those the
    // batched seed BP passed on, or that found the seed store full)
    const int wb = screened == 2 ? *((volatile int*)&w.desc->win_base) : 0;
    const int* list = screened == 2 ? w.fail + wb : w.queue;
    int nq = screened ? *((volatile int*)&w.ctr->n_queue) : 0;
    if (screened == 2) {
        // the current window of the fail list: at most S shots (the seed store)
        const long long left = (long long)*((volatile int*)&w.ctr->n_fail) - wb;
        nq = (int)(left < w.S ? (left > 0 ? left : 0) : w.S);
    }
    int kcur = 0, kend = 0;                      // claimed slots [kcur, kend), the same in the whole group
    for (;;) {
        if (kcur >= kend) {
            const int batch = (Eng::Grp::kBlock || screened || dp->chunk_n - kend < 16ll * total_warps) ? 1 : 4;
            int base = 0;
            if (grp.rank() == 0) base = atomicAdd(&w.ctr->claim_seed, batch);
            kcur = grp.bcast(base);
            kend = kcur + batch;
        }
        const int k = kcur++;
        // after a screen, the shots it passed on; else every shot of the chunk
        const int b = !screened ? k : (k < nq ? list[k] : (int)dp->chunk_n);
        if (b >= dp->chunk_n) break;
        const long long gb = dp->chunk_base + b;
        const uint32_t* s = dp->synd + gb * g.WM;
        uint32_t nz = 0;
        for (int q = grp.rank(); q < g.WM; q += grp.size()) {
            const uint32_t x = s[q];
            st.sp[q] = x;
            nz |= x;
        }
        for (int q = grp.rank(); q < g.WN; q += grp.size()) { st.mask[q] = 0u; st.vals[q] = 0u; st.ehat[q] = 0u; }
        grp.sync();
        // s = 0 with every Lambda_j > 0: D > 0 at t = 1, so e^(1) = 0 and the
        // seed converges after one iteration (exact, no BP needed)
        if (!grp.any(nz != 0u) && cfg.num_results == 1 && g.all_lam_pos) {
            finalize_shot<typename Eng::Grp, true>(g, dp->out, gb, st.ehat, ST_SEED, 1ull, grp);
            grp.sync();
            continue;
        }
        if (!Eng::kPriorStart) eng.start_prior(g, st);
        if (!Eng::kPriorSetsSums) eng.clear_sums(g, st);
        grp.sync();
        int succ = 0;
        const int it = eng.run(g, cfg, st, cfg.initial_iters, true, &succ, nullptr, true);
        if (grp.rank() == 0) seed_iters += (unsigned long long)it;
        grp.sync();
        if ((succ && cfg.num_results == 1) || cfg.max_rounds == 0) {
            finalize_shot<typename Eng::Grp, true>(g, dp->out, gb, st.ehat, succ ? ST_SEED : ST_FAILED,
                                                   (unsigned long long)it, grp);
            grp.sync();
            continue;
        }
        int np, tie;
        long long S;
        eng.argmin_score(g, st, cfg.tie_guard, &np, &S, &tie);
        int a = 0;
        if (grp.rank() == 0) {
            a = atomicAdd(&w.ctr->n_active, 1);
            // a full store (a chunk may be larger): the shot is decoded again in
            // a window after this one's beam
            if (a >= w.S) w.fail[atomicAdd(&w.ctr->n_fail, 1)] = b;
        }
        a = grp.bcast(a);
        if (a >= w.S) continue;
        // the seed path (Alg. 3): snapshot, s' = s, no fixed node, e^, next_pos
        eng.save_E(g, st, w.seedE + (size_t)a * snap_bytes(g));
        uint32_t* bits = w.seedBits + (size_t)a * (size_t)w.SB;
        for (int q = grp.rank(); q < g.WM; q += grp.size()) bits[q] = st.sp[q];
        for (int q = grp.rank(); q < g.WN; q += grp.size()) {
            bits[g.WM + q] = 0u;
            bits[g.WM + g.WN + q] = 0u;
            bits[g.WM + 2 * g.WN + q] = st.ehat[q];
        }
        if (grp.rank() == 0) {
            SlotMeta m;
            m.S = 0; m.iters = it; m.next_pos = np; m.success = succ; m.flags = tie;
            w.seedMeta[a] = m;
            w.seed_shot[a] = b;
        }
        grp.sync();
    }
    if (grp.rank() == 0 && seed_iters != 0ull) atomicAdd(&w.stats[0], seed_iters);
}

// ----------------------------------------------------------------------------
// the beam: every round of every shot in one kernel
// ----------------------------------------------------------------------------
// A shot's rounds depend only on one another, so no round waits for another
// shot: the children to run are items of a ring that the candidate groups of
// one persistent kernel draw from; the group that finishes the last child of a
// shot's round selects (k_round's select_entry), and pushes the children of
// the next round or, when the shot has ended, gives its window entry to the
// next shot of the seed store.  (Before: a launch of all children and one of
// all selections per round and window of shots, each ending with most of the
// GPU idle: 10^6 [[144,12,12]] shots at p = 0.05 took 280 launches of 21.3 ms
// in all.)
//
// The ring (bsd_ring.cuh): a group draws a ticket and waits for the item that will
// be put at its slot; it draws the next one when its child, and the selection after
// it, are done.  The running groups alone finish the work: a group that has waited a
// second without an item leaves.
// orders this thread's memory operations, and those of the threads it has
// synchronised with, before and after an atomic that passes them on
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

struct GpuRing {
    static __device__ __forceinline__ uint32_t add(uint32_t* p, uint32_t v) { return atomicAdd(p, v); }
    static __device__ __forceinline__ uint32_t cas(uint32_t* p, uint32_t want, uint32_t v) { return atomicCAS(p, want, v); }
    static __device__ __forceinline__ uint32_t and_(uint32_t* p, uint32_t v) { return atomicAnd(p, v); }
    static __device__ __forceinline__ uint32_t load(const uint32_t* p) { return ld_relaxed(p); }
    static __device__ __forceinline__ void pause() { __nanosleep(200); }
    static __device__ __forceinline__ unsigned long long now() { return global_ns(); }
};

__device__ inline void push_pair(const Work& w, uint32_t item)
{
    ring_push_pair<GpuRing>(w.ring, &w.ctr->b_tail, w.ctr->b_mask, item);
}

__device__ inline uint32_t draw_item(const Work& w, uint32_t ticket)
{
    const uint32_t it = ring_draw<GpuRing>(w.ring, w.ctr->b_mask, reinterpret_cast<const uint32_t*>(&w.ctr->b_left), ticket);
    if (it != kRingEmpty) fence_gpu();         // the item before what it names
    return it;
}

struct SelScratch {
    double score[2 * kMaxBeam];
    int iters[2 * kMaxBeam];
    int flags[2 * kMaxBeam];     // bit0 exists, bit1 success, bit2 argmin near-tie
};
static_assert(sizeof(SelScratch) == kSelectBytes, "the scratch warp_smem_bytes makes room for");

// window entry a takes the shot of seed-store entry e (one warp): the seed
// path is its only path (Alg. 3)
__device__ inline void init_entry(const DevGraph& g, const DecCfg& cfg, const Work& w, int a, int e, int stamp)
{
    const int lane = threadIdx.x & 31;
    const SlotMeta sm = w.seedMeta[e];
    if (sm.success) {                  // num_results > 1: the seed result opens `results`
        const uint32_t* eb = w.seedBits + (size_t)e * (size_t)w.SB + g.WM + 2 * g.WN;
        uint32_t* rb = w.res_bits + (size_t)a * cfg.num_results * g.WN;
        for (int q = lane; q < g.WN; q += 32) rb[q] = eb[q];
        const long long W = vector_weight(g, eb);
        if (lane == 0) {
            w.res_w[(size_t)a * cfg.num_results] = W;
            w.res_origin[(size_t)a * cfg.num_results] = 0;
        }
    }
    if (lane == 0) {
        w.shot_of[a] = w.seed_shot[e];
        w.set_size[a] = 1;
        w.iters_acc[a] = (unsigned long long)sm.iters;
        w.res_n[a] = sm.success ? 1 : 0;
        w.near[a] = sm.flags & 1;      // the seed path branches on its argmin
        w.ent[a] = BeamEntry{e, 1, 2, stamp};
        w.kid[(size_t)a * 2 * cfg.w] = w.kid[(size_t)a * 2 * cfg.w + 1] = make_int2(-1, sm.next_pos);
    }
    __syncwarp();
}

// the entries of the first items (the ring is filled by k_beam_ring)
__global__ void k_beam_entries(DevGraph g, DecCfg cfg, Work w)
{
    count_launch(w);
    const int cnt = w.ctr->b_next;
    const int nw = (int)((gridDim.x * blockDim.x) >> 5);
    for (int a = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); a < cnt; a += nw) {
        init_entry(g, cfg, w, a, a, 1);
        if ((threadIdx.x & 31) == 0) w.first_ok[a] = 0ull;   // no stamp is 0
    }
}

__device__ void finalize_results(const DevGraph& g, const DecCfg& cfg, const Work& w, const Outputs& out,
                                 int a, long long gb, unsigned long long total, uint32_t extra)
{
    const int n = __ldcg(w.res_n + a);
    const long long* rw = w.res_w + (size_t)a * cfg.num_results;
    int bi = 0;
    long long wb = __ldcg(rw);
    for (int q = 1; q < n; ++q) {
        const long long wq = __ldcg(rw + q);
        if (wq < wb) { bi = q; wb = wq; }
    }
    const uint32_t st = (__ldcg(w.res_origin + (size_t)a * cfg.num_results + bi) == 0) ? ST_SEED : ST_BEAM;
    finalize_shot<WarpGroup, false, true>(g, out, gb, w.res_bits + ((size_t)a * cfg.num_results + bi) * g.WN,
                                          st | extra, total);
}

// one warp, after the last child of the round of window entry a: first success
// in visit order, `results`, top-w pruning (Alg. 3, App. B), then the next
// round's items, or the shot's outputs and the entry's next shot.  Everything
// read here was written by other SMs during this kernel (__ldcg).
__device__ __noinline__ void select_entry(const DevGraph& g, const DecCfg& cfg, const Work& w, int a, SelScratch* sc)
{
    const int lane = threadIdx.x & 31;
    const int W2 = 2 * cfg.w;
    const RunDesc d = *w.desc;
    const BeamEntry ent = load_entry(w.ent + a);
    const int r = ent.round;
    const int cb = r & 1;
    const long long gb = d.chunk_base + __ldcg(w.shot_of + a);
    const int npar = __ldcg(w.set_size + a);
    const int nch = 2 * npar;
    // gather the children of this round in canonical order c = 2 * rank + val
    for (int c = lane; c < nch; c += 32) {
        const int pnp = __ldcg(w.kid + (size_t)a * W2 + c).y;
        int fl = 0, it = 0;
        double scv = 0.0;
        if (pnp >= 0) {
            const SlotMeta m = load_meta(w.slotMeta + slot_index(w, cb, a, c, W2));
            fl = 1 | (m.success ? 2 : 0) | ((m.flags & 1) << 2);
            it = m.iters;
            scv = ((double)m.S / kFixScale) / (double)m.iters;
        }
        sc->flags[c] = fl;
        sc->iters[c] = it;
        sc->score[c] = scv;
    }
    __syncwarp();
    unsigned long long acc = __ldcg(w.iters_acc + a);
    bool done = false;
    // near-tie record: argmin margins of the children the sequential
    // algorithm visits, and the pruning margin of the round
    int near = __ldcg(w.near + a);
    auto near_upto = [&](int last) {
        int f = 0;
        for (int c = lane; c <= last && c < nch; c += 32) f |= (sc->flags[c] >> 2) & 1;
        return __any_sync(FULLMASK, f != 0) ? 1 : 0;
    };
    if (cfg.num_results == 1) {
        // Alg. 3: the first successful child in visit order ends the search
        int first = 0x7fffffff;
        for (int c = lane; c < nch; c += 32)
            if ((sc->flags[c] & 3) == 3 && c < first) first = c;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) first = min(first, __shfl_xor_sync(FULLMASK, first, o));
        if (first != 0x7fffffff) {
            unsigned long long sum = 0;
            for (int c = lane; c <= first; c += 32)
                if (sc->flags[c] & 1) sum += (unsigned long long)sc->iters[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULLMASK, sum, o);
            const uint32_t* eb = w.slotBits + slot_index(w, cb, a, first, W2) * (size_t)w.SB + g.WM + 2 * g.WN;
            near |= near_upto(first);
            finalize_shot<WarpGroup, false, true>(g, d.out, gb, eb, ST_BEAM | (near ? ST_NEAR : 0u), acc + sum);
            done = true;
        }
    } else {
        // results collection in visit order (dedupe by equality, App. B)
        unsigned long long sum = 0;
        int nres = __ldcg(w.res_n + a);
        for (int c = 0; c < nch && !done; ++c) {
            const int fl = sc->flags[c];
            if (!(fl & 1)) continue;
            sum += (unsigned long long)sc->iters[c];
            if (!(fl & 2)) continue;
            const uint32_t* eb = w.slotBits + slot_index(w, cb, a, c, W2) * (size_t)w.SB + g.WM + 2 * g.WN;
            bool dup = false;
            if (g.WN <= 32) {
                // a stored result per lane (one memory round trip per success
                // instead of one per stored result)
                bool same = false;
                for (int q = lane; q < nres; q += 32) {
                    const uint32_t* rb = w.res_bits + ((size_t)a * cfg.num_results + q) * g.WN;
                    uint32_t diff = 0u;
                    for (int x = 0; x < g.WN; ++x) diff |= __ldcg(rb + x) ^ __ldcg(eb + x);
                    same = same || diff == 0u;
                }
                dup = __any_sync(FULLMASK, same);
            } else {
                for (int q = 0; q < nres && !dup; ++q) {
                    const uint32_t* rb = w.res_bits + ((size_t)a * cfg.num_results + q) * g.WN;
                    bool eq = true;
                    for (int x = lane; x < g.WN; x += 32) eq = eq && (__ldcg(rb + x) == __ldcg(eb + x));
                    dup = __all_sync(FULLMASK, eq);
                }
            }
            if (!dup) {
                uint32_t* rb = w.res_bits + ((size_t)a * cfg.num_results + nres) * g.WN;
                for (int x = lane; x < g.WN; x += 32) rb[x] = __ldcg(eb + x);
                const long long W = vector_weight(g, eb);
                __syncwarp();
                if (lane == 0) {
                    w.res_w[(size_t)a * cfg.num_results + nres] = W;
                    w.res_origin[(size_t)a * cfg.num_results + nres] = 1;
                    w.res_n[a] = nres + 1;
                }
                __syncwarp();
                if (++nres >= cfg.num_results) {
                    near |= near_upto(c);
                    finalize_results(g, cfg, w, d.out, a, gb, acc + sum, near ? ST_NEAR : 0u);
                    done = true;
                }
            }
        }
    }
    if (!done) {
        unsigned long long sum = 0;
        int nex = 0;
        for (int c = lane; c < nch; c += 32) {
            if (sc->flags[c] & 1) { sum += (unsigned long long)sc->iters[c]; ++nex; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sum += __shfl_xor_sync(FULLMASK, sum, o);
            nex += __shfl_xor_sync(FULLMASK, nex, o);
        }
        acc += sum;
        near |= near_upto(nch - 1);
        // rank of each existing child under (score desc, canonical index asc)
        int myrank[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = lane + 32 * q;
            myrank[q] = -1;
            if (c < nch && (sc->flags[c] & 1)) {
                const double s0 = sc->score[c];
                int rk = 0;
                for (int c2 = 0; c2 < nch; ++c2) {
                    if (!(sc->flags[c2] & 1)) continue;
                    const double s2 = sc->score[c2];
                    rk += (s2 > s0 || (s2 == s0 && c2 < c)) ? 1 : 0;
                }
                myrank[q] = rk;
            }
        }
        // the kept paths of a round before the last, and how many of them
        // have a node left to branch on (their children make round r + 1)
        const bool last = (r >= cfg.max_rounds || nex == 0);
        int keep = 0, tot = 0;
        if (!last) {
            __syncwarp();
            keep = nex < cfg.w ? nex : cfg.w;
            if (cfg.tie_guard > 0.0 && nex > keep) {
                // pruning margin: last kept (rank keep-1) against first dropped (rank keep)
                double s_in = -INFINITY, s_out = -INFINITY;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (myrank[q] == keep - 1) s_in = sc->score[lane + 32 * q];
                    if (myrank[q] == keep) s_out = sc->score[lane + 32 * q];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s_in = fmax(s_in, __shfl_xor_sync(FULLMASK, s_in, o));
                    s_out = fmax(s_out, __shfl_xor_sync(FULLMASK, s_out, o));
                }
                const double den = fabs(s_in) > 1.0 ? fabs(s_in) : 1.0;
                const double gap = (s_in - s_out) / den;
                if (gap > 0.0 && gap < cfg.tie_guard) near = 1;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (myrank[q] >= 0 && myrank[q] < keep)
                    w.set_idx[(size_t)a * cfg.w + myrank[q]] = (uint8_t)(lane + 32 * q);
            __syncwarp();
            int cntp = 0;
            for (int k = lane; k < keep; k += 32) {
                const int c = w.set_idx[(size_t)a * cfg.w + k];
                cntp += (__ldcg(&w.slotMeta[slot_index(w, cb, a, c, W2)].next_pos) >= 0) ? 1 : 0;
            }
            tot = cntp;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(FULLMASK, tot, o);
        }
        if (last || tot == 0) {
            // the search ends here: the last round, no child, or no kept
            // path with a node left (the next round would have no child)
            if (cfg.num_results > 1 && __ldcg(w.res_n + a) > 0) {
                finalize_results(g, cfg, w, d.out, a, gb, acc, near ? ST_NEAR : 0u);
            } else {
                // no valid solution: the best path of the final set
                int best = 0x7fffffff;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (myrank[q] == 0) best = lane + 32 * q;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(FULLMASK, best, o));
                const uint32_t* eb;
                if (best != 0x7fffffff)
                    eb = w.slotBits + slot_index(w, cb, a, best, W2) * (size_t)w.SB + g.WM + 2 * g.WN;
                else
                    eb = parent_ref(g, cfg, w, r, ent.seed, a, __ldcg(w.kid + (size_t)a * W2).x).bits + g.WM + 2 * g.WN;
                finalize_shot<WarpGroup, false, true>(g, d.out, gb, eb, ST_FAILED | (near ? ST_NEAR : 0u), acc);
            }
            done = true;
        } else {
            // the kept slots become the next round's parents: two children per
            // kept path that has a next_pos
            if (lane == 0) {
                w.set_size[a] = keep;
                w.iters_acc[a] = acc;
                w.near[a] = near;
                w.ent[a] = BeamEntry{ent.seed, r + 1, 2 * tot, ent.stamp + 1};
            }
            __syncwarp();
            for (int k = lane; k < keep; k += 32) {
                const int c = __ldcg(w.set_idx + (size_t)a * cfg.w + k);
                const int np = __ldcg(&w.slotMeta[slot_index(w, cb, a, c, W2)].next_pos);
                w.kid[(size_t)a * W2 + 2 * k] = w.kid[(size_t)a * W2 + 2 * k + 1] = make_int2(c, np);
                if (np >= 0) {
                    fence_gpu();               // the entry and the child before its items
                    push_pair(w, ring_item(a, 2 * k));
                }
            }
        }
    }
    if (done) {
        // the entry's next shot, then this one is counted off
        __syncwarp();
        int e = 0;
        if (lane == 0) e = atomicAdd(&w.ctr->b_next, 1);
        e = __shfl_sync(FULLMASK, e, 0);
        if (e < w.ctr->n_active) {
            init_entry(g, cfg, w, a, e, ent.stamp + 1);
            if (lane == 0) {
                fence_gpu();
                push_pair(w, ring_item(a, 0));
            }
        }
        __syncwarp();
        if (lane == 0) {
            fence_gpu();
            atomicSub(&w.ctr->b_left, 1);
        }
    }
}

// expand a child and run masked BP (Alg. 2), item by item
template <class Eng>
__global__ void __launch_bounds__(Eng::kMaxThreads, Eng::kMinBlocks) k_round(DevGraph g, DecCfg cfg, Work w)
{
    extern __shared__ __align__(16) char smem[];
    count_launch(w);
    Eng eng;
    eng.grp = Eng::Grp::make(smem + warp_smem_bytes(g));
    const auto& grp = eng.grp;
    char* const own = smem + (size_t)grp.index() * warp_smem_bytes(g);
    const WarpState st = carve(own, g);
    // no more tickets waiting than slots
    if ((uint32_t)(blockIdx.x * grp.per_block() + grp.index()) > w.ctr->b_mask) return;
    const int W2 = 2 * cfg.w;
    unsigned long long ran = 0;                // BP iterations (group rank 0)
    for (;;) {
        uint32_t item = kRingEmpty;
        if (grp.rank() == 0) item = draw_item(w, atomicAdd(&w.ctr->b_head, 1u));
        item = (uint32_t)grp.bcast((int)item);
        if (item == kRingEmpty) break;
        const int a = ring_entry(item), c = ring_child(item);
        const BeamEntry ent = load_entry(w.ent + a);
        const int2 kid = __ldcg(w.kid + (size_t)a * W2 + c);
        const int r = ent.round;
        const int v = c & 1, pos = kid.y;
        const SlotRef par = parent_ref(g, cfg, w, r, ent.seed, a, kid.x);
        if (pos >= 0) {                        // (a path with no unmasked node has no children)
            const size_t cslot = slot_index(w, r & 1, a, c, W2);
            // s' of the child: flip the detectors of pos when it is fixed to 1
            for (int q = grp.rank(); q < g.WM; q += grp.size()) {
                uint32_t x = __ldcg(par.bits + q);
                if (v) x ^= __ldg(g.hcol + (size_t)pos * g.WM + q);
                st.sp[q] = x;
            }
            for (int q = grp.rank(); q < g.WN; q += grp.size()) {
                uint32_t m = __ldcg(par.bits + g.WM + q);
                uint32_t vv = __ldcg(par.bits + g.WM + g.WN + q);
                if (q == (pos >> 5)) {
                    m |= 1u << (pos & 31);
                    if (v) vv |= 1u << (pos & 31);
                }
                st.mask[q] = m;
                st.vals[q] = vv;
            }
            // (the engine's tables are read again for each child: nothing of them
            // is kept in registers across the selection's call)
            eng.load_graph(g, st);
            // warm start from the parent's snapshot
            eng.load_E(g, st, par.E);
            eng.clear_sums(g, st);
            grp.sync();
            eng.fix_node(g, st, pos, cfg.L);
            grp.sync();
            // with num_results = 1, only the first success in visit order matters:
            // a child stops once a lower-index sibling of this round has succeeded
            AbortCheck ab{};
            if (cfg.num_results == 1) {
                ab.key = w.first_ok + a;
                ab.stamp = (unsigned long long)(unsigned)ent.stamp << 32;
                ab.c = (unsigned)c;
            }
            int succ = 0;
            const int iters = eng.run(g, cfg, st, cfg.iters_per_round, true, &succ, nullptr, false, ab);
            int superseded = 0;
            if (grp.rank() == 0) {
                ran += (unsigned long long)iters;
                if (ab.key != nullptr) {
                    if (succ) atomicMax(w.first_ok + a, ab.stamp | (0xffffffffull - (unsigned)c));
                    else superseded = ab.hit(*((volatile const unsigned long long*)ab.key)) ? 1 : 0;
                }
            }
            // a superseded child's slot is never read: record only that it exists
            if (grp.bcast(superseded)) {
                if (grp.rank() == 0) {
                    SlotMeta m;
                    m.S = 0; m.iters = iters; m.next_pos = -1; m.success = 0; m.flags = 0;
                    w.slotMeta[cslot] = m;
                }
            } else {
                grp.sync();
                for (int q = grp.rank(); q < g.WN; q += grp.size())
                    st.ehat[q] = (st.ehat[q] & ~st.mask[q]) | st.vals[q];
                grp.sync();
                int np, tie;
                long long S;
                eng.argmin_score(g, st, cfg.tie_guard, &np, &S, &tie);
                eng.save_E(g, st, w.slotE + cslot * snap_bytes(g));
                uint32_t* cbits = w.slotBits + cslot * (size_t)w.SB;
                for (int q = grp.rank(); q < g.WM; q += grp.size()) cbits[q] = st.sp[q];
                for (int q = grp.rank(); q < g.WN; q += grp.size()) {
                    cbits[g.WM + q] = st.mask[q];
                    cbits[g.WM + g.WN + q] = st.vals[q];
                    cbits[g.WM + 2 * g.WN + q] = st.ehat[q];
                }
                if (grp.rank() == 0) {
                    SlotMeta m;
                    m.S = S; m.iters = iters; m.next_pos = np; m.success = succ; m.flags = tie;
                    w.slotMeta[cslot] = m;
                }
            }
        }
        // the slot before the count; the round's last child selects
        grp.sync();
        int last = 0;
        if (grp.rank() == 0) {
            fence_gpu();
            last = atomicSub(&w.ent[a].pending, 1) == 1 ? 1 : 0;
            if (last) fence_gpu();
        }
        last = grp.bcast(last);
        grp.sync();
        if (last) {
            if (grp.warp() == 0) select_entry(g, cfg, w, a, reinterpret_cast<SelScratch*>(own));
            grp.sync();
        }
    }
    if (grp.rank() == 0 && ran != 0ull) atomicAdd(&w.stats[1], ran);
}

// ----------------------------------------------------------------------------
// plain BP for a fixed number of iterations (LLR measurement)
// ----------------------------------------------------------------------------
template <class Eng>
__global__ void __launch_bounds__(Eng::kMaxThreads, Eng::kMinBlocks) k_bp_llr(DevGraph g, DecCfg cfg,
                                                                           const uint32_t* __restrict__ synd,
                                                                           long long B, int T, float* llr,
                                                                           float* sum_llr)
{
    extern __shared__ __align__(16) char smem[];
    Eng eng;
    eng.grp = Eng::Grp::make(smem + warp_smem_bytes(g));
    const auto& grp = eng.grp;
    const WarpState st = carve(smem + (size_t)grp.index() * warp_smem_bytes(g), g);
    eng.load_graph(g, st);
    const long long nw = (long long)gridDim.x * grp.per_block();
    for (long long b = (long long)blockIdx.x * grp.per_block() + grp.index(); b < B; b += nw) {
        for (int q = grp.rank(); q < g.WM; q += grp.size()) st.sp[q] = synd[b * g.WM + q];
        for (int q = grp.rank(); q < g.WN; q += grp.size()) { st.mask[q] = 0u; st.vals[q] = 0u; }
        if (!Eng::kPriorStart) eng.start_prior(g, st);
        if (!Eng::kPriorSetsSums) eng.clear_sums(g, st);
        grp.sync();
        int succ;
        eng.template run<true>(g, cfg, st, T, false, &succ, llr + b * g.N, true);
        grp.sync();
        if (sum_llr != nullptr) eng.write_sums(g, st, sum_llr + b * g.N);
        grp.sync();
    }
}

// ----------------------------------------------------------------------------
// host-side launch helpers
// ----------------------------------------------------------------------------
// engine id = 3 * kind + storage precision, or 15 + kind for weighted min-sum;
// kinds: 0, 1 jagged with column degree bound 3 / 6, 2 generic (16), 3: small (CPL 3,
// RPL 2, row degree 6), 4: small (CPL 5, RPL 3, row degree 6); precision 0
// float, 1 binary16, 2 bfloat16; then the blocks of warps and the wide engines below
#define BSD_KIND_ALIASES(P, SFX)                          \
    using Jagged3##SFX = JaggedEngine<3, P>;              \
    using Jagged6##SFX = JaggedEngine<6, P>;              \
    using Generic16##SFX = GenericEngine<16, P>;          \
    using Small326##SFX = SmallEngine<3, 2, 6, P>;        \
    using Small536##SFX = SmallEngine<5, 3, 6, P>;
BSD_KIND_ALIASES(0, _f32)
BSD_KIND_ALIASES(1, _f16)
BSD_KIND_ALIASES(2, _bf16)
// weighted min-sum (per-edge, per-iteration weights), single-precision messages: id 15 + kind
using Jagged3_w = JaggedEngine<3, 0, true>;
using Jagged6_w = JaggedEngine<6, 0, true>;
using Generic16_w = GenericEngine<16, 0, true>;
using Small326_w = SmallEngine<3, 2, 6, 0, true>;
using Small536_w = SmallEngine<5, 3, 6, 0, true>;
constexpr int kWeightedEngine = 15;
// a block of warps per candidate (jagged and generic engines): id 20 + 4 * kind + (0 float, 1 binary16,
// 2 bfloat16, 3 weighted float)
#define BSD_BLOCK_ALIASES(DV, ENGINE)                                    \
    using Block##DV##_f32 = ENGINE<DV, 0, false, BlockGroup>;            \
    using Block##DV##_f16 = ENGINE<DV, 1, false, BlockGroup>;            \
    using Block##DV##_bf16 = ENGINE<DV, 2, false, BlockGroup>;           \
    using Block##DV##_w = ENGINE<DV, 0, true, BlockGroup>;
BSD_BLOCK_ALIASES(3, JaggedEngine)
BSD_BLOCK_ALIASES(6, JaggedEngine)
BSD_BLOCK_ALIASES(16, GenericEngine)
constexpr int kBlockEngine = 20;
// the generic engine with 16-bit messages on chip, for codes of column degree up to 6
// whose messages do not fit there as floats: id 32 + 4 * kind + 2 (a block) +
// (0 binary16, 1 bfloat16)
#define BSD_WIDE_ALIASES(DV)                                             \
    using Wide##DV##_f16 = GenericEngine<DV, 1>;                         \
    using Wide##DV##_bf16 = GenericEngine<DV, 2>;                        \
    using WideBlock##DV##_f16 = GenericEngine<DV, 1, false, BlockGroup>; \
    using WideBlock##DV##_bf16 = GenericEngine<DV, 2, false, BlockGroup>;
BSD_WIDE_ALIASES(3)
BSD_WIDE_ALIASES(6)
constexpr int kWideEngine = 32;
#define BSD_ENGINES(X)                                                                          \
    X(0, Jagged3_f32) X(1, Jagged3_f16) X(2, Jagged3_bf16)                                      \
    X(3, Jagged6_f32) X(4, Jagged6_f16) X(5, Jagged6_bf16)                                      \
    X(6, Generic16_f32) X(7, Generic16_f16) X(8, Generic16_bf16)                                \
    X(9, Small326_f32) X(10, Small326_f16) X(11, Small326_bf16)                                 \
    X(12, Small536_f32) X(13, Small536_f16) X(14, Small536_bf16)                                \
    X(15, Jagged3_w) X(16, Jagged6_w) X(17, Generic16_w) X(18, Small326_w) X(19, Small536_w)    \
    X(20, Block3_f32) X(21, Block3_f16) X(22, Block3_bf16) X(23, Block3_w)                      \
    X(24, Block6_f32) X(25, Block6_f16) X(26, Block6_bf16) X(27, Block6_w)                      \
    X(28, Block16_f32) X(29, Block16_f16) X(30, Block16_bf16) X(31, Block16_w)                  \
    X(32, Wide3_f16) X(33, Wide3_bf16) X(34, WideBlock3_f16) X(35, WideBlock3_bf16)             \
    X(36, Wide6_f16) X(37, Wide6_bf16) X(38, WideBlock6_f16) X(39, WideBlock6_bf16)

template <class Eng>
static int set_attrs(size_t smem_bp)
{
    if (CUDA_FAILED(cudaFuncSetAttribute(k_seed<Eng>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bp)) ||
        CUDA_FAILED(cudaFuncSetAttribute(k_round<Eng>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bp)) ||
        CUDA_FAILED(cudaFuncSetAttribute(k_bp_llr<Eng>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bp)))
        return -2;
    return 0;
}

template <class Eng>
static int occupancy(int threads, size_t smem_bp, int* bps)
{
    int a = 0, b = 0;
    if (CUDA_FAILED(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_round<Eng>, threads, smem_bp))) return -2;
    if (CUDA_FAILED(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_seed<Eng>, threads, smem_bp))) return -2;
    *bps = a < b ? a : b;
    return 0;
}

// the second screen runs on at least this many shots: two for every candidate
// group of the seed kernel
static int screen2_min_queue(const LaunchShape& ls)
{
    return 2 * ls.grid_seed * (ls.group_warps >= 2 ? 1 : ls.warps_per_block);
}
static void* screen2_func(int dv, int prec)
{
    if (dv == 0)
        return prec == 0 ? (void*)k_screen2<3, 0> : prec == 1 ? (void*)k_screen2<3, 1> : (void*)k_screen2<3, 2>;
    if (dv == 1)
        return prec == 0 ? (void*)k_screen2<6, 0> : prec == 1 ? (void*)k_screen2<6, 1> : (void*)k_screen2<6, 2>;
    return prec == 0 ? (void*)k_screen2<16, 0> : prec == 1 ? (void*)k_screen2<16, 1> : (void*)k_screen2<16, 2>;
}

// can the small engine run this code? (column degree 3, row degree 6, with
// the placement of its messages built)
static bool small_fits(const DevGraph& g, int cpl, int rpl)
{
    if (g.scol == nullptr) return false;
    if (g.max_col_deg != 3 || g.max_row_deg != 6 || g.E != 3 * g.N || g.E != 6 * g.M) return false;
    if (g.E >= 65536 || g.M >= 65536) return false;
    return g.WN == cpl && (g.M + 31) / 32 == rpl;
}

int configure_kernels(DevGraph& g, const DecCfg& cfg, int device, int group_warps, int warps_per_block,
                      LaunchShape* ls)
{
    if (cfg.weights != nullptr && g.prec != 0) return -5;   // weights: single-precision messages only
    if (group_warps < 0 || group_warps > 16 || warps_per_block < 0 || warps_per_block > 8) return -5;
    int gkind;                                               // generic kind: column degree bound 3 / 6 / 16
    if (g.max_col_deg <= 3) gkind = 0;
    else if (g.max_col_deg <= 6) gkind = 1;
    else if (g.max_col_deg <= 16) gkind = 2;
    else return -5;
    if (gkind < 2 && g.colK != (gkind == 0 ? 3 : 6)) return -5;   // the column table matches the engine
    int skind = -1;                                          // small engine kind, if the code has its layout
    if (small_fits(g, 3, 2)) skind = 3;
    else if (small_fits(g, 5, 3)) skind = 4;
    int max_optin = 0, sms = 0;
    if (CUDA_FAILED(cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device)) ||
        CUDA_FAILED(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device)))
        return -2;
    g.sms = sms;
    g.max_smem = max_optin;
    // per-candidate state: the jagged engine keeps float messages, D over E;
    // the generic one the stored format and a record per detector
    g.e_bytes = gkind < 2 ? (int)sizeof(float) : g.msg_bytes;
    g.det_bytes = gkind < 2 ? 0 : (int)align16(sizeof(float2) * (size_t)g.M);
    // automatic choice: the small engine where it fits; otherwise a warp per
    // candidate while eight or more candidates fit on an SM, a block of 16
    // warps per candidate beyond (8 / 16 warps: 10^5 shots of the
    // phenomenological DEM at p = 3e-3 3.42 / 2.88 ms, 5 x 10^4 in half
    // precision 0.87 / 0.74, 3 x 10^5 of the synthetic DEM 11.2 / 10.7).  The rule
    // does not know the batch: of depolarizing noise on [[144,12,12]] at p = 0.03, 1 /
    // 8 / 16 warps, 10^5 shots take 7.6 / 9.8 / 14.3 ms, 3000 1.22 / 0.58 / 0.66, 300
    // 0.81 / 0.31 / 0.28 (bsd_autotune and group_warps choose otherwise)
    int gw = group_warps;
    if (gw == 0) gw = (skind >= 0 || warp_smem_bytes(g) * 8 <= (size_t)max_optin) ? 1 : 16;
    // 16-bit messages that do not fit as floats stay in 16 bits on chip (the
    // generic engine's state: 2 E + 8 M + 4 N bytes against 4 E + 4 N): from about
    // 45000 edges; 2 x 10^4 shots of a 1200 x 20000 code of 60000 edges 1.9 ms
    const bool wide = gkind < 2 && skind < 0 && g.prec != 0 &&
                      warp_smem_bytes(g) + (gw >= 2 ? 16 * sizeof(ArgRec) : 0) > (size_t)max_optin;
    if (wide) {
        g.e_bytes = g.msg_bytes;
        g.det_bytes = (int)align16(sizeof(float2) * (size_t)g.M);
    }
    const bool weighted = cfg.weights != nullptr;
    int eng, wpb;
    if (gw >= 2) {
        eng = wide ? kWideEngine + 4 * gkind + 2 + (g.prec - 1) : kBlockEngine + 4 * gkind + (weighted ? 3 : g.prec);
        wpb = gw;
    } else {
        const int kind = skind >= 0 ? skind : gkind;
        eng = weighted ? kWeightedEngine + kind : wide ? kWideEngine + 4 * gkind + (g.prec - 1) : 3 * kind + g.prec;
        // the small engine keeps D per edge in float (over E with single-precision
        // messages, else beside it)
        if (kind >= 3) {
            g.e_bytes = g.msg_bytes;
            g.det_bytes = g.prec == 0 ? 0 : (int)align16(sizeof(float) * (size_t)g.Epad);
        }
        const size_t per_warp = warp_smem_bytes(g);
        if (per_warp > (size_t)max_optin) return -5;
        wpb = warps_per_block > 0 ? warps_per_block : (int)((96 * 1024) / per_warp);
        if (wpb > 8) wpb = 8;
        if (wpb < 1) wpb = 1;
        if (per_warp * (size_t)wpb > (size_t)max_optin) return -5;
    }
    const size_t per_cand = warp_smem_bytes(g);
    ls->group_warps = gw >= 2 ? gw : 1;
    ls->warps_per_block = wpb;
    ls->smem_bp = gw >= 2 ? per_cand + 16 * sizeof(ArgRec) : per_cand * (size_t)wpb;
    if (ls->smem_bp > (size_t)max_optin) return -5;
    ls->dv = eng;
    const int threads = 32 * wpb;
    int rc = 0, bps_bp = 0;
    // The dynamic shared-memory limit is a property of the kernel, shared by
    // every decoder that launches it; it is raised to the device maximum so
    // that no decoder created later can lower it below what an earlier one
    // launches with (a CUDA graph keeps the value it was instantiated with,
    // a direct launch checks the current one).
    switch (eng) {
#define X(id, E)                                                                \
    case id:                                                                    \
        rc = set_attrs<E>((size_t)max_optin);                       \
        if (!rc) rc = occupancy<E>(threads, ls->smem_bp, &bps_bp);  \
        break;
        BSD_ENGINES(X)
#undef X
        default: return -5;
    }
    if (rc) return rc;
    if (bps_bp < 1) return -5;
    // the first-iteration screen: generic engines, the scale alpha, every
    // Lambda_j > 0, one result
    ls->screen = 0;
    ls->grid_screen = 0;
    ls->grid_screen2 = 0;
    ls->smem_screen = sizeof(uint32_t) * screen_warp_words(g) * kScreenWarps;
    if (eng < 9 || eng >= kBlockEngine) {                   // not a small engine
        if (!weighted && g.all_lam_pos && cfg.num_results == 1 && ls->smem_screen <= (size_t)max_optin) {
            void* kf = gkind == 0 ? (void*)k_screen<3> : gkind == 1 ? (void*)k_screen<6> : (void*)k_screen<16>;
            int bps_scr = 0;
            // a screen warp's state is a few KB of bit sets and lists: prefer the
            // shared-memory carveout that lets the register file, not the
            // carveout, bound the resident blocks
            if (CUDA_FAILED(cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin)) ||
                CUDA_FAILED(cudaFuncSetAttribute(kf, cudaFuncAttributePreferredSharedMemoryCarveout,
                                                 cudaSharedmemCarveoutMaxShared)) ||
                CUDA_FAILED(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps_scr, kf, 32 * kScreenWarps,
                                                                          ls->smem_screen)))
                return -2;
            if (bps_scr >= 1) {
                ls->screen = 1;
                ls->grid_screen = sms * bps_scr;
                ls->dv_screen = gkind;
            }
            // the second-iteration screen where its tables were built (sparse
            // syndromes) and the seed BP has a second iteration
            ls->smem_screen2 = sizeof(uint32_t) * (screen2_warp_words(g)) * kScreenWarps;
            if (ls->screen && g.row4 != nullptr && cfg.initial_iters >= 2 &&
                ls->smem_screen2 <= (size_t)max_optin) {
                kf = screen2_func(gkind, g.prec);
                if (CUDA_FAILED(cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, max_optin)) ||
                    CUDA_FAILED(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps_scr, kf, 32 * kScreenWarps,
                                                                              ls->smem_screen2)))
                    return -2;
                if (bps_scr >= 1) ls->grid_screen2 = sms * bps_scr;
            }
        }
    }
    ls->grid_seed = sms * bps_bp;
    ls->grid_round = sms * bps_bp;
    // the batched seed BP: generic engines with the scale alpha and one result
    // (the shots it finishes need no snapshot; the others are decoded again by
    // the per-candidate seed kernel)
    ls->batch = (eng < 9 || eng >= kBlockEngine) && !weighted && cfg.num_results == 1 ? 1 : 0;
    ls->grid_bs = batch_grid(device);
    return 0;
}

static void* screen_func(const LaunchShape& ls)
{
    return ls.dv_screen == 0 ? (void*)k_screen<3> : ls.dv_screen == 1 ? (void*)k_screen<6> : (void*)k_screen<16>;
}

template <class Eng>
static int launch_chunk_t(const DevGraph& g, const DecCfg& cfg, const Work& w, const LaunchShape& ls,
                          const uint32_t* synd, long long base, long long n, const Outputs& out, cudaStream_t s,
                          const LaunchHooks* hk, cudaGraphExec_t gx, int* host_n_active)
{
    const int threads = 32 * ls.warps_per_block;
    k_begin_chunk<<<1, 32, 0, s>>>(w, synd, out, base, n);
    if (CUDA_FAILED(cudaGetLastError())) return -2;
    if (gx != nullptr) return !CUDA_FAILED(cudaGraphLaunch(gx, s)) ? 0 : -2;
    if (ls.screen) {
        if (hk) hk->before(hk->ctx, 11);
        DevGraph gg = g;
        DecCfg cc = cfg;
        Work ww = w;
        int more = ls.grid_screen2 > 0, min_queue = screen2_min_queue(ls);
        void* cargs[] = {&gg, &cc, &ww, &more};
        void* margs[] = {&gg, &cc, &ww, &min_queue};
        if (CUDA_FAILED(cudaLaunchKernel(screen_func(ls), dim3((unsigned)ls.grid_screen), dim3(32 * kScreenWarps),
                                         cargs, ls.smem_screen, s)) ||
            (more && CUDA_FAILED(cudaLaunchKernel(screen2_func(ls.dv_screen, g.prec), dim3((unsigned)ls.grid_screen2),
                                                  dim3(32 * kScreenWarps), margs, ls.smem_screen2, s))))
            return -2;
        if (hk) hk->after(hk->ctx, 11);
    }
    // the seed kernel on its shots, then the beam if any needs it (without a
    // graph the number of active entries is read back)
    auto seed_and_beam = [&](int seed_src) -> int {
        if (hk) hk->before(hk->ctx, 0);
        k_seed<Eng><<<ls.grid_seed, threads, ls.smem_bp, s>>>(g, cfg, w, seed_src);
        if (hk) hk->after(hk->ctx, 0);
        if (CUDA_FAILED(cudaGetLastError())) return -2;
        if (cfg.max_rounds == 0) return 0;
        if (CUDA_FAILED(cudaMemcpyAsync(host_n_active, &w.ctr->n_active, sizeof(int), cudaMemcpyDeviceToHost, s)) ||
            CUDA_FAILED(cudaStreamSynchronize(s)))
            return -2;
        if (*host_n_active == 0) return 0;
        if (hk) hk->before(hk->ctx, 2);
        k_beam_begin<<<1, 32, 0, s>>>(w, cfg.w);
        k_beam_ring<<<ls.grid_seed, 256, 0, s>>>(w);
        k_beam_entries<<<ls.grid_seed, 256, 0, s>>>(g, cfg, w);
        if (hk) { hk->after(hk->ctx, 2); hk->before(hk->ctx, 1); }
        k_round<Eng><<<ls.grid_round, threads, ls.smem_bp, s>>>(g, cfg, w);
        if (hk) hk->after(hk->ctx, 1);
        k_beam_end<<<1, 32, 0, s>>>(w);
        return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
    };
    // the seed BP of the chunk: batched, or per candidate with the beam of the
    // shots that fit the seed store; then the shots handed on, in windows of at
    // most S (the store)
    const bool batched = ls.batch && w.bs_slots > 0;
    if (batched) {
        if (launch_batch_direct(g, cfg, w, ls, ls.screen, s, hk, host_n_active)) return -2;
    } else {
        const int rc = seed_and_beam(ls.screen);
        if (rc || w.S1 <= w.S || cfg.max_rounds == 0) return rc;
    }
    if (CUDA_FAILED(cudaMemcpyAsync(host_n_active, &w.ctr->n_fail, sizeof(int), cudaMemcpyDeviceToHost, s)) ||
        CUDA_FAILED(cudaStreamSynchronize(s)))
        return -2;
    const long long n_fail = *host_n_active;
    for (long long wb = 0; wb < n_fail; wb += w.S) {
        k_win_begin<<<1, 32, 0, s>>>(w, (int)wb);
        if (CUDA_FAILED(cudaGetLastError())) return -2;
        const int rc = seed_and_beam(2);
        if (rc) return rc;
    }
    return 0;
}

int launch_chunk(const DevGraph& g, const DecCfg& cfg, const Work& w, const LaunchShape& ls, const uint32_t* synd,
                 long long base, long long n, const Outputs& out, void* stream, const LaunchHooks* hooks,
                 void* graph_exec, int* host_n_active)
{
    cudaStream_t s = (cudaStream_t)stream;
    cudaGraphExec_t gx = (cudaGraphExec_t)graph_exec;
    switch (ls.dv) {
#define X(id, E) \
    case id: return launch_chunk_t<E>(g, cfg, w, ls, synd, base, n, out, s, hooks, gx, host_n_active);
        BSD_ENGINES(X)
#undef X
        default: return -5;
    }
}

// ---- the per-chunk graph: k_seed, then IF (a shot needs the beam) { the beam }
static int add_kernel(cudaGraph_t graph, cudaGraphNode_t* node, const cudaGraphNode_t* dep, void* func, int grid,
                      int block, size_t smem, void** args)
{
    cudaKernelNodeParams p{};
    p.func = func;
    p.gridDim = dim3((unsigned)grid);
    p.blockDim = dim3((unsigned)block);
    p.sharedMemBytes = (unsigned)smem;
    p.kernelParams = args;
    return !CUDA_FAILED(cudaGraphAddKernelNode(node, graph, dep, dep ? 1 : 0, &p)) ? 0 : -2;
}

// IF (a shot needs the beam) { its set-up, the beam, the check that no shot is
// left } after `dep` in `graph`
template <class Eng>
static int add_beam_nodes(cudaGraph_t graph, cudaGraphNode_t dep, cudaGraphNode_t* last, DevGraph& g, DecCfg& cfg,
                          Work& w, const LaunchShape& ls, cudaGraphConditionalHandle cwin = 0, int windows = 0)
{
    int rc = 0;
    cudaGraphConditionalHandle cbeam;
    cudaGraphNode_t gate, beam, begin, ring, entries, round, end;
    if (CUDA_FAILED(cudaGraphConditionalHandleCreate(&cbeam, graph, 0, cudaGraphCondAssignDefault))) rc = -2;
    if (!rc) {
        void* gargs[] = {&w, &cbeam, &cwin, &windows};
        rc = add_kernel(graph, &gate, &dep, (void*)k_beam_gate, 1, 32, 0, gargs);
    }
    cudaGraphNodeParams cp{};
    if (!rc) {
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = cbeam;
        cp.conditional.type = cudaGraphCondTypeIf;
        cp.conditional.size = 1;
        if (CUDA_FAILED(cudaGraphAddNode(&beam, graph, &gate, nullptr, 1, &cp))) rc = -2;
    }
    if (!rc) {
        // kernel parameters are copied when a node is added
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        void* wargs[] = {&w};
        void* rargs[] = {&g, &cfg, &w};
        void* bargs[] = {&w, &cfg.w};
        rc = add_kernel(body, &begin, nullptr, (void*)k_beam_begin, 1, 32, 0, bargs);
        if (!rc) rc = add_kernel(body, &ring, &begin, (void*)k_beam_ring, ls.grid_seed, 256, 0, wargs);
        if (!rc) rc = add_kernel(body, &entries, &ring, (void*)k_beam_entries, ls.grid_seed, 256, 0, rargs);
        if (!rc)
            rc = add_kernel(body, &round, &entries, (void*)k_round<Eng>, ls.grid_round, 32 * ls.warps_per_block,
                            ls.smem_bp, rargs);
        if (!rc) rc = add_kernel(body, &end, &round, (void*)k_beam_end, 1, 32, 0, wargs);
    }
    if (!rc) *last = beam;
    return rc;
}

template <class Eng>
static int build_graph_t(const DevGraph& g0, const DecCfg& cfg0, const Work& w0, const LaunchShape& ls,
                         cudaGraphExec_t* out)
{
    DevGraph g = g0;
    DecCfg cfg = cfg0;
    Work w = w0;
    const int threads = 32 * ls.warps_per_block;
    cudaGraph_t graph = nullptr;
    if (CUDA_FAILED(cudaGraphCreate(&graph, 0))) return -2;
    int rc = 0;
    cudaGraphNode_t seed, scr, last;
    const bool batched = ls.batch && w.bs_slots > 0;
    int screened = batched ? 2 : ls.screen;
    void* sargs[] = {&g, &cfg, &w, &screened};
    int more = ls.grid_screen2 > 0, min_queue = screen2_min_queue(ls);
    void* cargs[] = {&g, &cfg, &w, &more};
    void* margs[] = {&g, &cfg, &w, &min_queue};
    if (ls.screen)
        rc = add_kernel(graph, &scr, nullptr, screen_func(ls), ls.grid_screen, 32 * kScreenWarps, ls.smem_screen,
                        cargs);
    if (ls.screen && more && !rc) {
        cudaGraphNode_t scr1 = scr;
        rc = add_kernel(graph, &scr, &scr1, screen2_func(ls.dv_screen, g.prec), ls.grid_screen2, 32 * kScreenWarps,
                        ls.smem_screen2, margs);
    }
    // WHILE (shots handed on remain) { window start, the seed kernel on at most
    // S of them, the beam, window end } after `dep`
    auto add_windows = [&](cudaGraphNode_t dep, cudaGraphConditionalHandle cwin) {
        cudaGraphNode_t wwin;
        cudaGraphNodeParams cp{};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = cwin;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        if (CUDA_FAILED(cudaGraphAddNode(&wwin, graph, &dep, nullptr, 1, &cp))) { rc = -2; return; }
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        cudaGraphNode_t wbeg, wseed, wend;
        int keep = -1, from = 2;
        void* bargs[] = {&w, &keep};
        void* wargs[] = {&g, &cfg, &w, &from};
        rc = add_kernel(body, &wbeg, nullptr, (void*)k_win_begin, 1, 32, 0, bargs);
        if (!rc) rc = add_kernel(body, &wseed, &wbeg, (void*)k_seed<Eng>, ls.grid_seed, threads, ls.smem_bp, wargs);
        cudaGraphNode_t tail = wseed;
        if (!rc && cfg.max_rounds > 0) rc = add_beam_nodes<Eng>(body, wseed, &tail, g, cfg, w, ls);
        void* eargs[] = {&w, &cwin};
        if (!rc) rc = add_kernel(body, &wend, &tail, (void*)k_win_end, 1, 32, 0, eargs);
    };
    cudaGraphConditionalHandle cwin = 0;
    const int windows = !batched && w.S1 > w.S && cfg.max_rounds > 0;
    if (!rc && (batched || windows) &&
        CUDA_FAILED(cudaGraphConditionalHandleCreate(&cwin, graph, 0, cudaGraphCondAssignDefault)))
        rc = -2;
    if (!batched) {
        // seed, then the beam, then the shots that found the store full
        if (!rc)
            rc = add_kernel(graph, &seed, ls.screen ? &scr : nullptr, (void*)k_seed<Eng>, ls.grid_seed, threads,
                            ls.smem_bp, sargs);
        if (!rc && cfg.max_rounds > 0) rc = add_beam_nodes<Eng>(graph, seed, &last, g, cfg, w, ls, cwin, windows);
        if (!rc && windows) add_windows(last, cwin);
    } else {
        // the batched seed BP over the chunk, then the shots it handed on
        cudaGraphNode_t bs, wgate;
        if (!rc) rc = add_batch_nodes(graph, ls.screen ? scr : nullptr, &bs, g, cfg, w, ls, ls.screen);
        if (!rc) {
            void* gargs[] = {&w, &cwin};
            rc = add_kernel(graph, &wgate, &bs, (void*)k_win_gate, 1, 32, 0, gargs);
        }
        if (!rc) add_windows(wgate, cwin);
    }
    cudaGraphExec_t gx = nullptr;
    if (!rc && CUDA_FAILED(cudaGraphInstantiate(&gx, graph, 0))) rc = -2;
    cudaGraphDestroy(graph);
    if (rc) {
        cudaGetLastError();
        return rc;
    }
    *out = gx;
    return 0;
}

int build_graph(const DevGraph& g, const DecCfg& cfg, const Work& w, const LaunchShape& ls, void** graph_exec)
{
    cudaGraphExec_t gx = nullptr;
    int rc;
    switch (ls.dv) {
#define X(id, E) \
    case id: rc = build_graph_t<E>(g, cfg, w, ls, &gx); break;
        BSD_ENGINES(X)
#undef X
        default: rc = -5;
    }
    *graph_exec = rc ? nullptr : (void*)gx;
    return rc;
}

void destroy_graph(void* graph_exec)
{
    if (graph_exec) cudaGraphExecDestroy((cudaGraphExec_t)graph_exec);
}

// ---- workspace layout
static inline size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

size_t work_head_bytes()
{
    return a256(sizeof(Counters)) + a256(sizeof(RunDesc)) + a256(kStats * sizeof(unsigned long long));
}

size_t work_layout(const DevGraph& g, const DecCfg& cfg, long long S, long long A, char* base, Work* w,
                   int bs_slots, long long S1)
{
    if (S1 < S) S1 = S;
    const size_t W2 = 2 * (size_t)cfg.w;
    const size_t SB = (size_t)g.WM + 3 * (size_t)g.WN;
    const size_t NR = (size_t)cfg.num_results;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += a256(bytes > 0 ? bytes : 1);
        return p;
    };
    char* ctr = take(sizeof(Counters));
    char* desc = take(sizeof(RunDesc));
    char* stats = take(kStats * sizeof(unsigned long long));
    Work v{};
    v.S = S;
    v.S1 = S1;
    v.A = A;
    v.SB = (int)SB;
    v.ctr = reinterpret_cast<Counters*>(ctr);
    v.desc = reinterpret_cast<RunDesc*>(desc);
    v.stats = reinterpret_cast<unsigned long long*>(stats);
    v.seedE = (unsigned char*)take((size_t)S * snap_bytes(g));
    v.seedBits = (uint32_t*)take(sizeof(uint32_t) * (size_t)S * SB);
    v.seedMeta = (SlotMeta*)take(sizeof(SlotMeta) * (size_t)S);
    v.seed_shot = (int*)take(sizeof(int) * (size_t)S);
    v.queue = (int*)take(sizeof(int) * (size_t)S1);
    v.slotE = (unsigned char*)take(2 * (size_t)A * W2 * snap_bytes(g));
    v.slotBits = (uint32_t*)take(sizeof(uint32_t) * 2 * (size_t)A * W2 * SB);
    v.slotMeta = (SlotMeta*)take(sizeof(SlotMeta) * 2 * (size_t)A * W2);
    v.shot_of = (int*)take(sizeof(int) * (size_t)A);
    v.set_size = (int*)take(sizeof(int) * (size_t)A);
    v.ent = (BeamEntry*)take(sizeof(BeamEntry) * (size_t)A);
    v.set_idx = (uint8_t*)take((size_t)A * (size_t)cfg.w);
    v.iters_acc = (unsigned long long*)take(sizeof(unsigned long long) * (size_t)A);
    v.res_bits = (uint32_t*)take(sizeof(uint32_t) * (size_t)A * NR * (size_t)g.WN);
    v.res_w = (long long*)take(sizeof(long long) * (size_t)A * NR);
    v.res_origin = (int*)take(sizeof(int) * (size_t)A * NR);
    v.res_n = (int*)take(sizeof(int) * (size_t)A);
    v.first_ok = (unsigned long long*)take(sizeof(unsigned long long) * (size_t)A);
    v.near = (int*)take(sizeof(int) * (size_t)A);
    // a power of two of at least A * 2w slots (k_beam_begin)
    size_t slots = 4;
    while (slots < (size_t)A * W2) slots *= 2;
    v.ring = (uint32_t*)take(sizeof(uint32_t) * slots);
    v.kid = (int2*)take(sizeof(int2) * (size_t)A * W2);
    // the batched seed BP's slots and the shots it passes on
    v.bs_slots = bs_slots;
    if (bs_slots > 0) {
        const size_t Bs = (size_t)bs_slots;
        v.bsE = (unsigned char*)take(Bs * (size_t)g.Epad * (size_t)g.msg_bytes);
        v.bsR = (float2*)take(sizeof(float2) * Bs * (size_t)g.M);
        v.bs_shot = (int*)take(sizeof(int) * Bs);
        v.bs_t = (int*)take(sizeof(int) * Bs);
        v.bs_nl = (int*)take(sizeof(int) * Bs);
        v.bs_list = (int*)take(sizeof(int) * Bs * (size_t)kBsList);
    }
    if (bs_slots > 0 || S1 > S) v.fail = (int*)take(sizeof(int) * (size_t)S1);
    // the first screen's queue for the second lies where the chunk's later
    // steps write (the hand-on list of the batch, or the seed store's shots)
    v.queue1 = v.fail != nullptr || base == nullptr ? v.fail : v.seed_shot;
    if (w) *w = v;
    return off;
}

template <class Eng>
static void launch_llr_t(const DevGraph& g, const DecCfg& cfg, const LaunchShape& ls, const uint32_t* synd,
                         long long B, int T, float* llr, float* sum_llr, cudaStream_t s, int blocks)
{
    k_bp_llr<Eng><<<blocks, 32 * ls.warps_per_block, ls.smem_bp, s>>>(g, cfg, synd, B, T, llr, sum_llr);
}

// ----------------------------------------------------------------------------
// request loop for single syndromes (low-latency mode): one candidate group
// stays resident and answers requests posted in host-mapped memory, so a
// syndrome whose seed BP ends the search (Alg. 3: the first BP run converges,
// with one result) costs no launch and no host-side stream wait
// ----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_acquire_sys(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_sys(uint32_t* p, uint32_t v)
{
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The loop answers a request (ServeBox::req != the last answered number) by
// the seed BP of its syndrome -- the same engine, operations and order as
// k_seed, so the outputs are identical -- and writes e^, A e^, status and
// iterations, or status 0 when the beam search must decide (the host then
// takes the regular path).  Every wait is bounded: the loop leaves when the
// host sets ServeBox::stop or when no request comes for idle_ns.
template <class Eng>
__global__ void __launch_bounds__(Eng::kMaxThreads, Eng::kMinBlocks) k_serve(DevGraph g, DecCfg cfg, ServeBox* box,
                                                                           uint32_t last, unsigned long long idle_ns)
{
    extern __shared__ __align__(16) char smem[];
    Eng eng;
    eng.grp = Eng::Grp::make(smem + warp_smem_bytes(g));
    const auto& grp = eng.grp;
    const WarpState st = carve(smem, g);
    eng.load_graph(g, st);
    volatile uint32_t* const synd = reinterpret_cast<volatile uint32_t*>(box + 1);
    uint32_t* const obuf = reinterpret_cast<uint32_t*>(box + 1) + g.WM;
    const Outputs out{obuf, g.K > 0 ? obuf + g.WN : nullptr, &box->status, &box->iters};
    if (grp.rank() == 0) st_release_sys(&box->state, 1u);
    for (;;) {
        int what = 0;                             // 1 request, 2 stop, 3 idle
        if (grp.rank() == 0) {
            const unsigned long long t0 = global_ns();
            for (;;) {
                if (ld_acquire_sys(&box->stop) != 0u) { what = 2; break; }
                const uint32_t r = ld_acquire_sys(&box->req);
                if (r != last) { last = r; what = 1; break; }
                if (global_ns() - t0 > idle_ns) { what = 3; break; }
                __nanosleep(32);                  // each poll crosses to host memory
            }
        }
        what = grp.bcast(what);
        if (what != 1) {
            if (grp.rank() == 0) st_release_sys(&box->state, what == 2 ? 3u : 2u);
            return;
        }
        uint32_t nz = 0;
        for (int q = grp.rank(); q < g.WM; q += grp.size()) {
            const uint32_t x = synd[q];
            st.sp[q] = x;
            nz |= x;
        }
        for (int q = grp.rank(); q < g.WN; q += grp.size()) { st.mask[q] = 0u; st.vals[q] = 0u; st.ehat[q] = 0u; }
        grp.sync();
        if (!grp.any(nz != 0u) && cfg.num_results == 1 && g.all_lam_pos) {
            // s = 0 with every Lambda_j > 0: the seed converges at t = 1 with e^ = 0
            finalize_shot<typename Eng::Grp, true>(g, out, 0, st.ehat, ST_SEED, 1ull, grp);
        } else {
            if (!Eng::kPriorStart) eng.start_prior(g, st);
            if (!Eng::kPriorSetsSums) eng.clear_sums(g, st);
            grp.sync();
            int succ = 0;
            const int it = eng.run(g, cfg, st, cfg.initial_iters, true, &succ, nullptr, true);
            grp.sync();
            if ((succ && cfg.num_results == 1) || cfg.max_rounds == 0)
                finalize_shot<typename Eng::Grp, true>(g, out, 0, st.ehat, succ ? ST_SEED : ST_FAILED,
                                                       (unsigned long long)it, grp);
            else if (grp.rank() == 0)
                box->status = 0u;
        }
        __threadfence_system();
        grp.sync();
        if (grp.rank() == 0) st_release_sys(&box->done, last);
    }
}

template <class Eng>
static int launch_serve_t(const DevGraph& g, const DecCfg& cfg, const LaunchShape& ls, ServeBox* box,
                          uint32_t last, unsigned long long idle_ns, cudaStream_t s)
{
    const bool block = ls.group_warps >= 2;
    const size_t smem = block ? ls.smem_bp : warp_smem_bytes(g);
    // (the device maximum: see configure_kernels)
    if (CUDA_FAILED(cudaFuncSetAttribute(k_serve<Eng>, cudaFuncAttributeMaxDynamicSharedMemorySize, g.max_smem)))
        return -2;
    k_serve<Eng><<<1, 32 * (block ? ls.group_warps : 1), smem, s>>>(g, cfg, box, last, idle_ns);
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}

int launch_serve(const DevGraph& g, const DecCfg& cfg, const LaunchShape& ls, ServeBox* box, uint32_t last,
                 unsigned long long idle_ns, void* stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    switch (ls.dv) {
#define X(id, E) \
    case id: return launch_serve_t<E>(g, cfg, ls, box, last, idle_ns, s);
        BSD_ENGINES(X)
#undef X
        default: return -5;
    }
}

int launch_bp_llr(const DevGraph& g, const DecCfg& cfg, const LaunchShape& ls, const uint32_t* synd, long long B,
                  int T, float* llr, float* sum_llr, void* stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    if (g.scol == nullptr) {                                 // (the single-warp engine's codes run there)
        const int rc = launch_llr_tiles(g, cfg, ls, synd, B, T, llr, sum_llr, stream);
        if (rc <= 0) return rc;
    }
    const int per_block = ls.group_warps > 1 ? 1 : ls.warps_per_block;     // candidates
    long long blocks = (B + per_block - 1) / per_block;
    if (blocks > ls.grid_round) blocks = ls.grid_round;
    if (blocks < 1) blocks = 1;
    switch (ls.dv) {
#define X(id, E) \
    case id: launch_llr_t<E>(g, cfg, ls, synd, B, T, llr, sum_llr, s, (int)blocks); break;
        BSD_ENGINES(X)
#undef X
        default: return -5;
    }
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}

}  // namespace bsd

// ----------------------------------------------------------------------------
// single-precision re-runs of near-tie shots (16-bit messages)
// ----------------------------------------------------------------------------
namespace bsd {

__global__ void k_collect_flagged(const uint32_t* __restrict__ status, long long B, long long* list, int* count)
{
    for (long long b = (long long)blockIdx.x * blockDim.x + threadIdx.x; b < B; b += (long long)gridDim.x * blockDim.x)
        if (status[b] & ST_NEAR) list[atomicAdd(count, 1)] = b;
}

__global__ void k_gather_rows(const uint32_t* __restrict__ src, const long long* __restrict__ list, int n, int W,
                              uint32_t* __restrict__ dst)
{
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < (long long)n * W;
         k += (long long)gridDim.x * blockDim.x) {
        const long long i = k / W, q = k % W;
        dst[k] = src[list[i] * W + q];
    }
}

__global__ void k_scatter_results(const long long* __restrict__ list, int n, int WN, int WK, Outputs from, Outputs to)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long b = list[i];
        for (int q = 0; q < WN; ++q) to.corr[b * WN + q] = from.corr[i * WN + q];
        if (to.obs != nullptr)
            for (int q = 0; q < WK; ++q) to.obs[b * WK + q] = from.obs[i * WK + q];
        to.status[b] = from.status[i] | ST_NEAR | ST_RERUN;
        if (to.iters != nullptr) to.iters[b] = from.iters[i];
    }
}

int launch_collect_flagged(const uint32_t* status, long long B, long long* list, int* count, void* stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    if (CUDA_FAILED(cudaMemsetAsync(count, 0, sizeof(int), s))) return -2;
    long long blocks = (B + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_collect_flagged<<<(int)(blocks > 0 ? blocks : 1), 256, 0, s>>>(status, B, list, count);
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}

int launch_gather_rows(const uint32_t* src, const long long* list, int n, int W, uint32_t* dst, void* stream)
{
    long long blocks = ((long long)n * W + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_gather_rows<<<(int)(blocks > 0 ? blocks : 1), 256, 0, (cudaStream_t)stream>>>(src, list, n, W, dst);
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}

int launch_scatter_results(const long long* list, int n, int WN, int WK, const Outputs& from, const Outputs& to,
                           void* stream)
{
    long long blocks = ((long long)n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_scatter_results<<<(int)(blocks > 0 ? blocks : 1), 256, 0, (cudaStream_t)stream>>>(list, n, WN, WK, from, to);
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}

}  // namespace bsd
