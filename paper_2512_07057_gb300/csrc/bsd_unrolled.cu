// bsd_unrolled.cu -- unrolled weighted min-sum: forward, loss and adjoint.
//
// Training the weights w[t][e] of weighted min-sum (a weight per edge and
// iteration in place of the scale of Eq. 1) runs T flooding iterations of
// Eqs. 1-3 on a batch of B shots, with no stopping rule, and differentiates
//     loss = sum_{t=1..T} mean_{b,j} BCE(sigmoid(-Lambda_j(t)), e_j)
// with respect to the weights.
//
// Codes with rows and columns of at most 8 edges whose messages fit in shared
// memory for 8 shots run on chip, one block per tile of shots (described at
// kShots below).  The other codes run the passes described here.
//
// Layout: every per-edge array is [E][Bp] and every per-node array [N][Bp]
// (shots contiguous; Bp = B rounded up to the 512-shot tile of a block), so a
// warp's 32 threads x 4 shots move 512 contiguous bytes of one edge.  The
// passes stream coalesced float4 vectors; the graph tables are read-only and
// cache resident.  Syndromes and true errors are transposed once into bit
// planes [M][Bp/32] and [N][Bp/32].
//
//   check pass (block = row i x 512 shots):
//       D_e(t) = w[t-1][e] * (-1)^{s_i} * prod_{e' != e} sign(E_e') * min_{e' != e} |E_e'|
//   error pass (block = column j x 512 shots):
//       Lambda_j(t) = Lambda_j + sum_{e in N(j)} D_e(t),  E_e(t) = clamp(Lambda_j(t) - D_e(t))
// The forward keeps E at the checkpoints t = 0, k, 2k, ...  The backward
// recomputes each segment of k iterations from its checkpoint, keeping E(t)
// and Lambda(t) of the segment, then runs the adjoint passes from t = T down:
//   error pass adjoint: gLam_j = dloss/dLambda_j(t) + sum_e [|E_e(t)| < L] gE_e
//                       gD_e = gLam_j - [|E_e(t)| < L] gE_e
//   check pass adjoint: gw[t-1][e] += gD_e sigma_e m_e,  gm_e = gD_e w[t-1][e] sigma_e
//                       gE_{i1}(t-1) = sign(E_{i1}) sum_{e != i1} gm_e
//                       gE_{i2}(t-1) = sign(E_{i2}) gm_{i1}
// with i1, i2 the edges of the row holding the smallest and second smallest
// |E(t-1)| (lowest edge index among equal magnitudes), sigma_e = (-1)^{s_i}
// prod_{e' != e} sign(E_e'), and m_e = |E_{i1}| for e != i1, |E_{i2}| for
// e = i1, or the constant L_MAX when no such edge exists (a row of weight 1,
// or every |E| at L_MAX).  sign() has zero derivative, d|x|/dx = sign(x) with
// 0 at 0, and a message at +-L_MAX passes none.  Loss and weight gradients
// are reduced through per-warp partial sums added in a fixed order, so every
// result is deterministic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "bsd.h"
#include "bsd_internal.cuh"

namespace bsd {
namespace {

constexpr int kThreads = 128;            // threads per block
constexpr int kTile = 4 * kThreads;      // shots per block (4 per thread)
// a row or column of degree <= CAP (4 or 8) keeps its vectors in registers
// between passes; CAP = 0 loads them again
constexpr int kWarps = kThreads / 32;    // partial sums are kept per warp (no block barrier)

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

struct UArgs {
    const int* row_ptr;
    const int* col_ptr;
    const int* col_edge;
    const float* lam;
    int M, N, E;
    float L;
    long long B, Bp;
    int ntile;
    int T;
    const float* w;          // [T][E]
    const uint32_t* sT;      // [M][Bp/32]
    const uint32_t* yT;      // [N][Bp/32]
};

struct ULayout {
    uint32_t* sT;
    uint32_t* yT;
    float* ck;               // [C][E][Bp]: E at t = c k
    float* seg;              // [k][E][Bp]: E(t0 + 1 .. t0 + k) of the segment being differentiated
    float* lamT;             // [k][N][Bp]: Lambda(t0 + 1 .. t0 + k)
    float* D;                // [E][Bp]
    float* gE[2];            // [E][Bp]
    float* gD;               // [E][Bp]
    float* loss_part;        // [T][N][ntile * kWarps]: per-warp loss sums
    float* gw_part;          // [T][ntile * kWarps][E]: per-warp weight-gradient sums
    size_t bytes;
};

ULayout layout(const DevGraph& g, long long B, int T, int k, char* base)
{
    ULayout u{};
    const long long Bp = (B + kTile - 1) / kTile * kTile;
    const size_t W32 = (size_t)(Bp / 32), EB = (size_t)g.E * (size_t)Bp, NB = (size_t)g.N * (size_t)Bp;
    const int C = (T + k - 1) / k;
    const size_t ntile = (size_t)(Bp / kTile);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += a256(bytes);
        return p;
    };
    u.sT = (uint32_t*)take(sizeof(uint32_t) * (size_t)g.M * W32);
    u.yT = (uint32_t*)take(sizeof(uint32_t) * (size_t)g.N * W32);
    u.ck = (float*)take(sizeof(float) * EB * (size_t)C);
    u.seg = (float*)take(sizeof(float) * EB * (size_t)k);
    u.lamT = (float*)take(sizeof(float) * NB * (size_t)k);
    u.D = (float*)take(sizeof(float) * EB);
    u.gE[0] = (float*)take(sizeof(float) * EB);
    u.gE[1] = (float*)take(sizeof(float) * EB);
    u.gD = (float*)take(sizeof(float) * EB);
    u.loss_part = (float*)take(sizeof(float) * (size_t)T * (size_t)g.N * ntile * kWarps);
    u.gw_part = (float*)take(sizeof(float) * (size_t)T * ntile * kWarps * (size_t)g.E);
    u.bytes = off;
    return u;
}

__device__ __forceinline__ float4 ld4(const float* base, int row, long long Bp, long long b)
{
    return *reinterpret_cast<const float4*>(base + (size_t)row * (size_t)Bp + (size_t)b);
}
__device__ __forceinline__ void st4(float* base, int row, long long Bp, long long b, float4 v)
{
    *reinterpret_cast<float4*>(base + (size_t)row * (size_t)Bp + (size_t)b) = v;
}
__device__ __forceinline__ float comp(const float4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }
__device__ __forceinline__ void setc(float4& v, int c, float x)
{
    if (c == 0) v.x = x; else if (c == 1) v.y = x; else if (c == 2) v.z = x; else v.w = x;
}
// the 4 bits of shots b .. b+3 (b a multiple of 4) from a bit plane row
__device__ __forceinline__ uint32_t bits4(const uint32_t* plane, int row, long long Bp, long long b)
{
    return (plane[(size_t)row * (size_t)(Bp / 32) + (size_t)(b >> 5)] >> (b & 31)) & 0xFu;
}
__device__ __forceinline__ float softplus(float x) { return fmaxf(x, 0.f) + log1pf(expf(-fabsf(x))); }
__device__ __forceinline__ float sgn0(float x) { return x > 0.f ? 1.f : (x < 0.f ? -1.f : 0.f); }

// sum over the warp; every lane gets the total
__device__ __forceinline__ float warp_sum(float v)
{
_Pragma("unroll")
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// slot of this warp among the per-warp partial sums of a tile
__device__ __forceinline__ int warp_slot() { return (int)blockIdx.x * kWarps + (int)(threadIdx.x >> 5); }

// ---------------------------------------------------------------------------
// batch intake: bitpacked [B][W] words -> bit planes [nbits][Bp/32]
// ---------------------------------------------------------------------------
__global__ void k_u_planes(const uint32_t* __restrict__ src, long long B, int W, int nbits, long long Bp,
                           uint32_t* __restrict__ dst)
{
    // one warp per (32 shots, one source word): lane l loads shot 32 wd + l's
    // word, and the ballot over bit k is row 32 w + k of those 32 shots
    const long long W32 = Bp / 32;
    const long long nwarp = W32 * (long long)W;
    const int lane = threadIdx.x & 31;
    for (long long q = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < nwarp;
         q += ((long long)gridDim.x * blockDim.x) >> 5) {
        const long long wd = q / W;
        const int w = (int)(q % W);
        const long long b = 32 * wd + lane;
        const uint32_t v = (b < B) ? src[(size_t)b * W + w] : 0u;
        for (int k = 0; k < 32; ++k) {
            const uint32_t bal = __ballot_sync(0xffffffffu, (v >> k) & 1u);
            const int i = 32 * w + k;
            if (lane == k && i < nbits) dst[(size_t)i * (size_t)W32 + (size_t)wd] = bal;
        }
    }
}

// E(0) = clamp(Lambda_j) on every edge of column j, for every shot
__global__ void k_u_init(UArgs a, float* __restrict__ E0)
{
    const long long b = (long long)blockIdx.x * kTile + 4 * threadIdx.x;
    for (int j = blockIdx.y; j < a.N; j += gridDim.y) {
        const float v = fminf(fmaxf(__ldg(a.lam + j), -a.L), a.L);
        const float4 v4 = make_float4(v, v, v, v);
        for (int q = __ldg(a.col_ptr + j); q < __ldg(a.col_ptr + j + 1); ++q) st4(E0, __ldg(a.col_edge + q), a.Bp, b, v4);
    }
}

// Loops over the edges of a row or column: with CAP > 0 the loop is unrolled
// up to CAP with compile-time indices, so each edge's vector stays in a
// register between passes; with CAP = 0 the vector is loaded again.
#define U_FOR_EDGES(CAP, k, deg, ...)                        \
    if (CAP > 0) {                                          \
        _Pragma("unroll") for (int k = 0; k < CAP; ++k)     \
            if (k < (deg)) { __VA_ARGS__ }                  \
    } else {                                                \
        for (int k = 0; k < (deg); ++k) { __VA_ARGS__ }     \
    }

// ---------------------------------------------------------------------------
// check pass (Eq. 1 with weights): D(t) from E(t-1)
// ---------------------------------------------------------------------------
template <int CAP>
__global__ void __launch_bounds__(kThreads) k_u_check(UArgs a, const float* __restrict__ Ein, float* __restrict__ D,
                                                      int t)
{
    const long long b = (long long)blockIdx.x * kTile + 4 * threadIdx.x;
    const float* wt = a.w + (size_t)(t - 1) * (size_t)a.E;
    for (int i = blockIdx.y; i < a.M; i += gridDim.y) {
        const int rb = __ldg(a.row_ptr + i), deg = __ldg(a.row_ptr + i + 1) - rb;
        const uint32_t s4 = bits4(a.sT, i, a.Bp, b);
        float m1[4], m2[4];
        uint32_t neg[4];
_Pragma("unroll")
        for (int c = 0; c < 4; ++c) { m1[c] = a.L; m2[c] = a.L; neg[c] = (s4 >> c) & 1u; }
        float4 x[CAP > 0 ? CAP : 1];
        U_FOR_EDGES(CAP, k, deg, {
            const float4 v = ld4(Ein, rb + k, a.Bp, b);
            if (CAP > 0) x[CAP > 0 ? k : 0] = v;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) {
                const float y = comp(v, c), m = fabsf(y);
                m2[c] = fminf(m2[c], fmaxf(m1[c], m));
                m1[c] = fminf(m1[c], m);
                neg[c] ^= (y < 0.f) ? 1u : 0u;
            }
        })
        U_FOR_EDGES(CAP, k, deg, {
            const float4 v = CAP > 0 ? x[CAP > 0 ? k : 0] : ld4(Ein, rb + k, a.Bp, b);
            const float wv = __ldg(wt + rb + k);
            float4 d;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) {
                const float y = comp(v, c);
                const float m = (fabsf(y) == m1[c]) ? m2[c] : m1[c];
                const float dd = __fmul_rn(wv, m);
                setc(d, c, (neg[c] ^ ((y < 0.f) ? 1u : 0u)) ? -dd : dd);
            }
            st4(D, rb + k, a.Bp, b, d);
        })
    }
}

// ---------------------------------------------------------------------------
// error pass (Eqs. 2-3): Lambda(t), E(t), loss terms
// ---------------------------------------------------------------------------
template <int CAP>
__global__ void __launch_bounds__(kThreads) k_u_var(UArgs a, const float* __restrict__ D, float* __restrict__ Eout,
                                                    float* __restrict__ lamT, float* __restrict__ llr,
                                                    float* __restrict__ loss_part)
{
    const long long b = (long long)blockIdx.x * kTile + 4 * threadIdx.x;
    for (int j = blockIdx.y; j < a.N; j += gridDim.y) {
        const int kb = __ldg(a.col_ptr + j), deg = __ldg(a.col_ptr + j + 1) - kb;
        const float lj = __ldg(a.lam + j);
        float4 post = make_float4(lj, lj, lj, lj);
        float4 x[CAP > 0 ? CAP : 1];
        U_FOR_EDGES(CAP, k, deg, {
            const float4 v = ld4(D, __ldg(a.col_edge + kb + k), a.Bp, b);
            if (CAP > 0) x[CAP > 0 ? k : 0] = v;
            post.x = __fadd_rn(post.x, v.x);
            post.y = __fadd_rn(post.y, v.y);
            post.z = __fadd_rn(post.z, v.z);
            post.w = __fadd_rn(post.w, v.w);
        })
        U_FOR_EDGES(CAP, k, deg, {
            const int e = __ldg(a.col_edge + kb + k);
            const float4 v = CAP > 0 ? x[CAP > 0 ? k : 0] : ld4(D, e, a.Bp, b);
            float4 o;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) setc(o, c, fminf(fmaxf(__fsub_rn(comp(post, c), comp(v, c)), -a.L), a.L));
            st4(Eout, e, a.Bp, b, o);
        })
        if (lamT) st4(lamT, j, a.Bp, b, post);
        if (llr) {
_Pragma("unroll")
            for (int c = 0; c < 4; ++c)
                if (b + c < a.B) llr[(size_t)(b + c) * (size_t)a.N + j] = comp(post, c);
        }
        if (loss_part) {
            const uint32_t y4 = bits4(a.yT, j, a.Bp, b);
            float l = 0.f;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) {
                const float p = comp(post, c);
                if (b + c < a.B) l += ((y4 >> c) & 1u) ? softplus(p) : softplus(-p);
            }
            l = warp_sum(l);
            if ((threadIdx.x & 31) == 0) loss_part[(size_t)j * a.ntile * kWarps + warp_slot()] = l;
        }
    }
}

// loss term of iteration t (block t): its partial sums added in a fixed order, in double
__global__ void k_u_loss(const float* __restrict__ loss_part, int N, int nslot, double scale, float* __restrict__ out)
{
    __shared__ double red[256];
    const int t = blockIdx.x;
    const float* p = loss_part + (size_t)t * N * nslot;
    double s = 0.0;
    for (long long q = threadIdx.x; q < (long long)N * nslot; q += blockDim.x) s += (double)p[q];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[1 + t] = (float)(red[0] * scale);
}

// the loss: the T terms added in order
__global__ void k_u_loss_total(int T, float* __restrict__ out)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int t = 0; t < T; ++t) s += (double)out[1 + t];
        out[0] = (float)s;
    }
}

// ---------------------------------------------------------------------------
// adjoint of the error pass at iteration t: gD(t) from gE(t) and the loss
// ---------------------------------------------------------------------------
template <int CAP>
__global__ void __launch_bounds__(kThreads) k_u_bvar(UArgs a, const float* __restrict__ gEin,
                                                     const float* __restrict__ Et, const float* __restrict__ lamT,
                                                     const float* __restrict__ gout, double scale, int t,
                                                     float* __restrict__ gD)
{
    const long long b = (long long)blockIdx.x * kTile + 4 * threadIdx.x;
    // the objective's derivative with respect to the term of iteration t:
    // through the total ([0]) and through the term itself ([t])
    const float gs = (float)(((double)__ldg(gout) + (double)__ldg(gout + t)) * scale);
    for (int j = blockIdx.y; j < a.N; j += gridDim.y) {
        const int kb = __ldg(a.col_ptr + j), deg = __ldg(a.col_ptr + j + 1) - kb;
        const float4 post = ld4(lamT, j, a.Bp, b);
        const uint32_t y4 = bits4(a.yT, j, a.Bp, b);
        float4 gl;
_Pragma("unroll")
        for (int c = 0; c < 4; ++c) {
            // d BCE / d Lambda = sigmoid(Lambda) - 1 + e_j
            const float p = comp(post, c);
            const float sg = 1.f / (1.f + expf(-p));
            setc(gl, c, (b + c < a.B) ? gs * (sg - 1.f + (float)((y4 >> c) & 1u)) : 0.f);
        }
        // gE(t) where the clamp let the derivative through, 0 elsewhere
        auto gE_of = [&](int e) {
            float4 g = ld4(gEin, e, a.Bp, b);
            const float4 v = ld4(Et, e, a.Bp, b);
_Pragma("unroll")
            for (int c = 0; c < 4; ++c)
                if (!(fabsf(comp(v, c)) < a.L)) setc(g, c, 0.f);
            return g;
        };
        float4 ge[CAP > 0 ? CAP : 1];
        if (gEin) {
            U_FOR_EDGES(CAP, k, deg, {
                const float4 g = gE_of(__ldg(a.col_edge + kb + k));
                if (CAP > 0) ge[CAP > 0 ? k : 0] = g;
                gl.x += g.x; gl.y += g.y; gl.z += g.z; gl.w += g.w;
            })
        }
        U_FOR_EDGES(CAP, k, deg, {
            const int e = __ldg(a.col_edge + kb + k);
            float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gEin) g = CAP > 0 ? ge[CAP > 0 ? k : 0] : gE_of(e);
            st4(gD, e, a.Bp, b, make_float4(gl.x - g.x, gl.y - g.y, gl.z - g.z, gl.w - g.w));
        })
    }
}

// ---------------------------------------------------------------------------
// adjoint of the check pass at iteration t: weight gradients and gE(t-1)
// ---------------------------------------------------------------------------
template <int CAP>
__global__ void __launch_bounds__(kThreads) k_u_bcheck(UArgs a, const float* __restrict__ Eprev,
                                                       const float* __restrict__ gD, float* __restrict__ gEprev,
                                                       float* __restrict__ gw_part, int t)
{
    const long long b = (long long)blockIdx.x * kTile + 4 * threadIdx.x;
    const float* wt = a.w + (size_t)(t - 1) * (size_t)a.E;
    for (int i = blockIdx.y; i < a.M; i += gridDim.y) {
        const int rb = __ldg(a.row_ptr + i), deg = __ldg(a.row_ptr + i + 1) - rb;
        const uint32_t s4 = bits4(a.sT, i, a.Bp, b);
        float m1[4], m2[4], v1[4], v2[4];
        int i1[4], i2[4];
        uint32_t neg[4];
_Pragma("unroll")
        for (int c = 0; c < 4; ++c) {
            m1[c] = a.L; m2[c] = a.L; v1[c] = 0.f; v2[c] = 0.f; i1[c] = -1; i2[c] = -1;
            neg[c] = (s4 >> c) & 1u;
        }
        float4 x[CAP > 0 ? CAP : 1];
        // the two smallest magnitudes with their edges (lowest index among equals)
        U_FOR_EDGES(CAP, k, deg, {
            const float4 v = ld4(Eprev, rb + k, a.Bp, b);
            if (CAP > 0) x[CAP > 0 ? k : 0] = v;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) {
                const float y = comp(v, c), m = fabsf(y);
                if (m < m1[c]) {
                    m2[c] = m1[c]; i2[c] = i1[c]; v2[c] = v1[c];
                    m1[c] = m; i1[c] = k; v1[c] = y;
                } else if (m < m2[c]) {
                    m2[c] = m; i2[c] = k; v2[c] = y;
                }
                neg[c] ^= (y < 0.f) ? 1u : 0u;
            }
        })
        float acc1[4] = {0.f, 0.f, 0.f, 0.f}, g1[4] = {0.f, 0.f, 0.f, 0.f};
        U_FOR_EDGES(CAP, k, deg, {
            const float4 v = CAP > 0 ? x[CAP > 0 ? k : 0] : ld4(Eprev, rb + k, a.Bp, b);
            const float4 g = ld4(gD, rb + k, a.Bp, b);
            const float wv = __ldg(wt + rb + k);
            float gw = 0.f;
_Pragma("unroll")
            for (int c = 0; c < 4; ++c) {
                const float y = comp(v, c);
                const float sig = (neg[c] ^ ((y < 0.f) ? 1u : 0u)) ? -1.f : 1.f;
                const float m = (k == i1[c]) ? m2[c] : m1[c];
                const float gd = comp(g, c);
                gw += gd * sig * m;
                const float gm = gd * wv * sig;
                if (k == i1[c]) g1[c] = gm; else acc1[c] += gm;
            }
            gw = warp_sum(gw);
            if ((threadIdx.x & 31) == 0) gw_part[(size_t)warp_slot() * a.E + rb + k] = gw;
        })
        if (gEprev) {
            U_FOR_EDGES(CAP, k, deg, {
                float4 o;
_Pragma("unroll")
                for (int c = 0; c < 4; ++c) {
                    float r = 0.f;
                    if (k == i1[c]) r = sgn0(v1[c]) * acc1[c];
                    else if (k == i2[c] && i1[c] >= 0) r = sgn0(v2[c]) * g1[c];
                    setc(o, c, r);
                }
                st4(gEprev, rb + k, a.Bp, b, o);
            })
        }
    }
}

// weight gradients: the per-warp partial sums added in a fixed order
__global__ void k_u_gw(const float* __restrict__ gw_part, int T, int ntile, int E, float* __restrict__ grad)
{
    const long long total = (long long)T * E;
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const long long t = q / E, e = q % E;
        const float* p = gw_part + (size_t)t * ntile * E + e;
        float s = 0.f;
        for (int k = 0; k < ntile; ++k) s += p[(size_t)k * E];
        grad[q] = s;
    }
}

// ---------------------------------------------------------------------------
// the whole forward, and the whole backward, of a tile of shots on chip
// ---------------------------------------------------------------------------
// For codes with rows and columns of degree at most 8 whose messages of
// kShots shots fit in an SM's shared memory, one block runs every iteration of
// a tile of kShots shots there, so the messages never leave the SM: per
// iteration a row pass (E -> D, or gD -> gE) and a column pass (D -> E, or gE ->
// gD), each over the same words.  A thread handles one row or column for four
// shots (16-byte accesses); edge e's kShots values start at word
// kShots * tile_slot(e), which puts the accesses of consecutive rows of degree 8
// in different banks.  The forward keeps what the adjoint needs of every
// iteration, in place of the message checkpoints: per (row, shot) the two
// smallest magnitudes, their edges and the signs (10 bytes), per (node, shot)
// Lambda_j(t).  gE(t) is zero but on the two edges of a row that hold its
// minima, whose magnitudes lie below L_MAX, so the adjoint of the clamp needs no
// look at E(t).  Weight gradients are summed over a block's tiles in order in
// the block's own partial, then over the blocks: deterministic.
//
// Bound: 4 shared-memory transfers per edge and shot (6912 wavefronts per
// iteration of 8 shots on the phenomenological DEM, 3.3 us) and the issue slots
// of both passes, against HBM traffic of 20 bytes per edge, pass and shot
// before.
constexpr int kShots = kTileShots;
// the forward's row pass holds a row's messages and weights (128 registers; 640
// threads spill: 1.24 against 1.21 ms at B = 4096, T = 20 on the phenomenological
// DEM); the backward fits in 80 (512 threads 1.64 ms, 640 1.49, 768 1.47, 1024 1.57)
constexpr int kFwdThreads = 512;
constexpr int kBwdThreads = 768;
constexpr int kMaxDeg = 8;

struct TileArgs {
    const int* row_ptr;
    const int* row_col;
    const uint2* col_slot;   // [N][CAP / 4]: tile_slot of the column's edges, 16 bits each, 0xffff past its degree
    const float* lam;
    int M, N, E, T;
    float L;
    long long B;
    int ntile;               // tiles of kShots shots
    const float* w;          // [T][E]
    unsigned char* s8;       // [ntile][M] the syndrome bits of the tile's shots
    unsigned char* y8;       // [ntile][N] their errors
    float* m1;               // [ntile][T][M][kShots]
    float* m2;
    uint16_t* pk;            // own signs of the row's edges (bits 0..7), edges of m1 and m2 (4 bits each, 15: none)
    float* lamT;             // [ntile][T][N][kShots]
    float* loss_part;        // [T][ntile]
    float* gw_part;          // [blocks][T][E]
    int* hazard;             // [kHazardBlocks] a weight that may make a message NaN was found
    int blocks, threads;
};
constexpr int kHazardBlocks = 64;

// A weight that is not finite, or large enough that a sum of eight check messages
// overflows, may make Lambda_j(t) infinite or NaN, and then Lambda_j(t) - D NaN,
// which the clamp makes -L_MAX.  The forward leaves its messages unclamped, so it
// sets these in a pass of its own, and only when this scan finds such a weight
// (of a training step of 4096 shots, 2.78 ms, it takes 0.6%; the clamp on every
// message, or a test of each posterior, 2.2%).
__global__ void k_u_hazard(const float* __restrict__ w, size_t n, float limit, int* __restrict__ out)
{
    bool bad = false;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x)
        bad = bad || !(fabsf(__ldg(w + q)) <= limit);
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) out[blockIdx.x] = any;
}

__host__ __device__ inline size_t tile_smem(int M, int N, int E)
{
    const size_t e4 = ((size_t)E + 3) & ~size_t(3);
    return e4 * kShots * sizeof(float) + (((size_t)M + (size_t)N + 15) & ~size_t(15)) + 2 * 32 * sizeof(float) +
           sizeof(uint16_t) * ((size_t)M + 1);
}
__device__ __forceinline__ float4* tile_at(float* x, int e, int half)
{
    return reinterpret_cast<float4*>(x + kShots * tile_slot(e) + 4 * half);
}
// the places of a column's edges, as they are stored and one by one
template <int CAP>
struct ColumnSlots {
    uint2 v[CAP / 4];
    __device__ __forceinline__ void load(const TileArgs& a, int j)
    {
#pragma unroll
        for (int h = 0; h < CAP / 4; ++h) v[h] = __ldg(a.col_slot + (size_t)j * (CAP / 4) + h);
    }
    __device__ __forceinline__ uint32_t at(int k) const
    {
        const uint32_t w = (k & 2) ? v[k / 4].y : v[k / 4].x;
        return (k & 1) ? w >> 16 : w & 0xffffu;
    }
};
__device__ __forceinline__ float4* slot_at(float* x, uint32_t slot, int half)
{
    return reinterpret_cast<float4*>(x + kShots * slot + 4 * half);
}
// signed minimum of two messages: the magnitude's minimum with the product's sign
__device__ __forceinline__ float xmin(float a, float b)
{
    float r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// bits << 1 with the sign of v below
__device__ __forceinline__ uint32_t push_sign(uint32_t bits, float v)
{
    return __funnelshift_l(__float_as_uint(v), bits, 1);
}
// the row's weights or gradients as two 16-byte accesses where it has eight
// edges at an aligned place
__device__ __forceinline__ bool row_aligned(const float* p, int rb, int deg)
{
    return deg == kMaxDeg && ((reinterpret_cast<uintptr_t>(p + rb) & 15u) == 0);
}
__device__ __forceinline__ bool row_weights(const float* wt, int rb, int deg, float (&wv)[kMaxDeg])
{
    const bool wide = row_aligned(wt, rb, deg);
    if (wide) {
        const float4 w0 = __ldg(reinterpret_cast<const float4*>(wt + rb));
        const float4 w1 = __ldg(reinterpret_cast<const float4*>(wt + rb) + 1);
        wv[0] = w0.x; wv[1] = w0.y; wv[2] = w0.z; wv[3] = w0.w;
        wv[4] = w1.x; wv[5] = w1.y; wv[6] = w1.z; wv[7] = w1.w;
    } else {
#pragma unroll
        for (int k = 0; k < kMaxDeg; ++k) wv[k] = k < deg ? __ldg(wt + rb + k) : 0.f;
    }
    return wide;
}
// softplus(x) as above; below 2^-12 the two terms of log1p's series are within
// e^2 / 3 of it, and most nodes are there
__device__ __forceinline__ float softplus_tail(float x)
{
    const float e = expf(-fabsf(x));
    const float l = e < 0x1p-12f ? fmaf(-0.5f * e, e, e) : log1pf(e);
    return fmaxf(x, 0.f) + l;
}

template <int CAP>
__global__ void __launch_bounds__(kFwdThreads, 1) k_u_forward(TileArgs a, const uint32_t* __restrict__ synd,
                                                            const uint32_t* __restrict__ errs, int WM, int WN,
                                                            float* __restrict__ llr)
{
    extern __shared__ __align__(16) float sm[];
    float* const x = sm;
    unsigned char* const sb = reinterpret_cast<unsigned char*>(sm + (((size_t)a.E + 3) & ~size_t(3)) * kShots);
    unsigned char* const yb = sb + a.M;
    float* const red = reinterpret_cast<float*>(sb + (((size_t)a.M + (size_t)a.N + 15) & ~size_t(15)));   // [2][32]
    uint16_t* const rp = reinterpret_cast<uint16_t*>(red + 64);                                           // row_ptr
    for (int q = threadIdx.x; q <= a.M; q += blockDim.x) rp[q] = (uint16_t)__ldg(a.row_ptr + q);
    const int nw = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool hazard = __syncthreads_or((int)threadIdx.x < kHazardBlocks && a.hazard[threadIdx.x] != 0);
    for (int tile = blockIdx.x; tile < a.ntile; tile += gridDim.x) {
        const long long b0 = (long long)tile * kShots;
        // the tile's syndrome and error bits, one byte per row and node
        for (int q = threadIdx.x; q < a.M + a.N; q += blockDim.x) {
            const bool row = q < a.M;
            const int i = row ? q : q - a.M, W = row ? WM : WN;
            const uint32_t* src = row ? synd : errs;
            uint32_t v = 0;
#pragma unroll
            for (int c = 0; c < kShots; ++c)
                if (b0 + c < a.B) v |= ((__ldg(src + (size_t)(b0 + c) * W + (i >> 5)) >> (i & 31)) & 1u) << c;
            sb[q] = (unsigned char)v;
            if (row) a.s8[(size_t)tile * a.M + i] = (unsigned char)v;
            else a.y8[(size_t)tile * a.N + i] = (unsigned char)v;
        }
        for (int q = threadIdx.x; q < 2 * a.E; q += blockDim.x) {          // E(0)
            const float v = fminf(fmaxf(__ldg(a.lam + __ldg(a.row_col + (q >> 1))), -a.L), a.L);
            *tile_at(x, q >> 1, q & 1) = make_float4(v, v, v, v);
        }
        __syncthreads();
        for (int t = 1; t <= a.T; ++t) {
            const float* wt = a.w + (size_t)(t - 1) * (size_t)a.E;
            const size_t rec = ((size_t)tile * a.T + (size_t)(t - 1)) * (size_t)a.M * kShots;
            // (each task's table entries are loaded while the one before runs)
            float wn[kMaxDeg];
            if ((int)threadIdx.x < 2 * a.M)
                row_weights(wt, rp[threadIdx.x >> 1], rp[(threadIdx.x >> 1) + 1] - rp[threadIdx.x >> 1], wn);
            for (int q = threadIdx.x; q < 2 * a.M; q += blockDim.x) {
                const int i = q >> 1, half = q & 1;
                const int rb = rp[i], deg = rp[i + 1] - rb;
                const uint32_t s4 = (uint32_t)sb[i] >> (4 * half);
                float wv[kMaxDeg];
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k) wv[k] = wn[k];
                if (q + (int)blockDim.x < 2 * a.M) {
                    const int in = (q + (int)blockDim.x) >> 1;
                    row_weights(wt, rp[in], rp[in + 1] - rp[in], wn);
                }
                float4 v[kMaxDeg];
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k)
                    v[k] = k < deg ? *tile_at(x, rb + k, half) : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                float r1[4], r2[4];
                uint32_t packed[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // each edge's signed minimum over the others (capped at
                    // L_MAX, with the syndrome sign) from running minima from
                    // both ends; the two smallest magnitudes are the least of
                    // all and the largest of these
                    float out[kMaxDeg];
                    out[kMaxDeg - 1] = INFINITY;
#pragma unroll
                    for (int k = kMaxDeg - 1; k > 0; --k)
                        out[k - 1] = k == kMaxDeg - 1 ? comp(v[k], c) : xmin(comp(v[k], c), out[k]);
                    float pre = __uint_as_float(__float_as_uint(a.L) | (((s4 >> c) & 1u) << 31));
#pragma unroll
                    for (int k = 0; k < kMaxDeg; ++k) {
                        out[k] = k == kMaxDeg - 1 ? pre : xmin(pre, out[k]);
                        pre = xmin(pre, comp(v[k], c));
                    }
                    const float m1 = fabsf(pre);
                    float m2 = m1;
#pragma unroll
                    for (int k = 0; k < kMaxDeg; ++k) m2 = fmaxf(m2, fabsf(out[k]));   // (past the degree: m1)
                    // their edges (the lowest among equals, none at L_MAX) and
                    // the own signs, bit by bit: m - |x| has its sign bit set
                    // where |x| > m
                    uint32_t above1 = ~0u, above2 = ~0u, neg = 0u;
#pragma unroll
                    for (int k = kMaxDeg - 1; k >= 0; --k) {
                        const float y = comp(v[k], c);
                        above1 = push_sign(above1, m1 - fabsf(y));
                        above2 = push_sign(above2, m2 - fabsf(y));
                        neg = push_sign(neg, y);
                        setc(v[k], c, __fmul_rn(wv[k], out[k]));
                    }
                    const uint32_t at1 = m1 < a.L ? ~above1 : 0u;
                    const uint32_t first = at1 & (0u - at1);
                    const uint32_t at2 = m2 < a.L ? ~above2 & ~first : 0u;
                    const uint32_t i1 = at1 ? (uint32_t)__ffs((int)at1) - 1u : 15u;
                    const uint32_t i2 = at2 ? (uint32_t)__ffs((int)at2) - 1u : 15u;
                    r1[c] = m1;
                    r2[c] = m2;
                    packed[c] = (neg & 0xFFu) | (i1 << 8) | (i2 << 12);
                }
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k)
                    if (k < deg) *tile_at(x, rb + k, half) = v[k];
                const size_t at = rec + (size_t)i * kShots + 4 * half;
                *reinterpret_cast<float4*>(a.m1 + at) = make_float4(r1[0], r1[1], r1[2], r1[3]);
                *reinterpret_cast<float4*>(a.m2 + at) = make_float4(r2[0], r2[1], r2[2], r2[3]);
                *reinterpret_cast<uint2*>(a.pk + at) = make_uint2(packed[0] | (packed[1] << 16), packed[2] | (packed[3] << 16));
            }
            __syncthreads();
            float loss = 0.f;
            const size_t nod = ((size_t)tile * a.T + (size_t)(t - 1)) * (size_t)a.N * kShots;
            ColumnSlots<CAP> en;
            float ln = 0.f;
            if ((int)threadIdx.x < 2 * a.N) {
                en.load(a, threadIdx.x >> 1);
                ln = __ldg(a.lam + (threadIdx.x >> 1));
            }
            for (int q = threadIdx.x; q < 2 * a.N; q += blockDim.x) {
                const int j = q >> 1, half = q & 1;
                const ColumnSlots<CAP> e = en;
                const float lj = ln;
                if (q + (int)blockDim.x < 2 * a.N) {
                    en.load(a, (q + (int)blockDim.x) >> 1);
                    ln = __ldg(a.lam + ((q + (int)blockDim.x) >> 1));
                }
                float4 post = make_float4(lj, lj, lj, lj);
                float4 v[CAP];
#pragma unroll
                for (int k = 0; k < CAP; ++k) {
                    if (e.at(k) != 0xffffu) {
                        v[k] = *slot_at(x, e.at(k), half);
                        post.x = __fadd_rn(post.x, v[k].x);
                        post.y = __fadd_rn(post.y, v[k].y);
                        post.z = __fadd_rn(post.z, v[k].z);
                        post.w = __fadd_rn(post.w, v[k].w);
                    }
                }
                // (unclamped: the row pass caps the magnitudes at L_MAX; a NaN below)
#pragma unroll
                for (int k = 0; k < CAP; ++k) {
                    if (e.at(k) != 0xffffu)
                        *slot_at(x, e.at(k), half) =
                            make_float4(__fsub_rn(post.x, v[k].x), __fsub_rn(post.y, v[k].y),
                                        __fsub_rn(post.z, v[k].z), __fsub_rn(post.w, v[k].w));
                }
                *reinterpret_cast<float4*>(a.lamT + nod + (size_t)j * kShots + 4 * half) = post;
                const uint32_t y4 = (uint32_t)yb[j] >> (4 * half);
                const long long b = b0 + 4 * half;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float p = comp(post, c);
                    const float l = softplus_tail(((y4 >> c) & 1u) ? p : -p);
                    loss += b + c < a.B ? l : 0.f;
                    if (llr && b + c < a.B)
                        llr[((size_t)(t - 1) * (size_t)a.B + (size_t)(b + c)) * (size_t)a.N + j] = p;
                }
            }
            if (hazard) {                              // the NaN among this thread's own messages
                for (int q = threadIdx.x; q < 2 * a.N; q += blockDim.x) {
                    ColumnSlots<CAP> e;
                    e.load(a, q >> 1);
                    for (int k = 0; k < CAP; ++k) {
                        if (e.at(k) == 0xffffu) continue;
                        float4* const m = slot_at(x, e.at(k), q & 1);
                        *m = make_float4(fmaxf(m->x, -a.L), fmaxf(m->y, -a.L), fmaxf(m->z, -a.L), fmaxf(m->w, -a.L));
                    }
                }
            }
            loss = warp_sum(loss);
            if (lane == 0) red[32 * (t & 1) + wid] = loss;
            __syncthreads();
            if (threadIdx.x == 0) {
                double l = 0.0;
                for (int k = 0; k < nw; ++k) l += (double)red[32 * (t & 1) + k];
                a.loss_part[(size_t)(t - 1) * a.ntile + tile] = (float)l;
            }
        }
        __syncthreads();
    }
}

template <int CAP>
__global__ void __launch_bounds__(kBwdThreads, 1) k_u_backward(TileArgs a, const float* __restrict__ gout, double scale)
{
    extern __shared__ __align__(16) float sm[];
    float* const x = sm;
    unsigned char* const sb = reinterpret_cast<unsigned char*>(sm + (((size_t)a.E + 3) & ~size_t(3)) * kShots);
    unsigned char* const yb = sb + a.M;
    uint16_t* const rp = reinterpret_cast<uint16_t*>(
        reinterpret_cast<float*>(sb + (((size_t)a.M + (size_t)a.N + 15) & ~size_t(15))) + 64);                // row_ptr
    for (int q = threadIdx.x; q <= a.M; q += blockDim.x) rp[q] = (uint16_t)__ldg(a.row_ptr + q);
    float* const part = a.gw_part + (size_t)blockIdx.x * (size_t)a.T * (size_t)a.E;
    for (int tile = blockIdx.x; tile < a.ntile; tile += gridDim.x) {
        const bool fresh = tile == (int)blockIdx.x;
        const long long b0 = (long long)tile * kShots;
        for (int q = threadIdx.x; q < a.M; q += blockDim.x) sb[q] = a.s8[(size_t)tile * a.M + q];
        for (int q = threadIdx.x; q < a.N; q += blockDim.x) yb[q] = a.y8[(size_t)tile * a.N + q];
        __syncthreads();
        for (int t = a.T; t >= 1; --t) {
            // the objective's derivative with respect to the term of iteration t:
            // through the total ([0]) and through the term itself ([t])
            const float gs = (float)(((double)__ldg(gout) + (double)__ldg(gout + t)) * scale);
            const size_t nod = ((size_t)tile * a.T + (size_t)(t - 1)) * (size_t)a.N * kShots;
            // (each task's loads are issued while the one before runs; a task's
            // Lambda lies at nod + 4 q)
            ColumnSlots<CAP> en;
            float4 pn = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((int)threadIdx.x < 2 * a.N) {
                en.load(a, threadIdx.x >> 1);
                pn = __ldg(reinterpret_cast<const float4*>(a.lamT + nod) + threadIdx.x);
            }
            for (int q = threadIdx.x; q < 2 * a.N; q += blockDim.x) {
                const int j = q >> 1, half = q & 1;
                const ColumnSlots<CAP> e = en;
                const float4 post = pn;
                if (q + (int)blockDim.x < 2 * a.N) {
                    en.load(a, (q + (int)blockDim.x) >> 1);
                    pn = __ldg(reinterpret_cast<const float4*>(a.lamT + nod) + q + blockDim.x);
                }
                const uint32_t y4 = (uint32_t)yb[j] >> (4 * half);
                const long long b = b0 + 4 * half;
                float4 gl;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // d BCE / d Lambda = sigmoid(Lambda) - 1 + e_j
                    // (1 + e^-Lambda rounds to 1 above 16.64, where most nodes are)
                    const float p = comp(post, c);
                    const float sg = p > 16.7f ? 1.f : 1.f / (1.f + expf(-p));
                    setc(gl, c, (b + c < a.B) ? gs * (sg - 1.f + (float)((y4 >> c) & 1u)) : 0.f);
                }
                float4 g[CAP];
#pragma unroll
                for (int k = 0; k < CAP; ++k) {
                    g[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (t < a.T && e.at(k) != 0xffffu) {
                        g[k] = *slot_at(x, e.at(k), half);
                        gl.x += g[k].x; gl.y += g[k].y; gl.z += g[k].z; gl.w += g[k].w;
                    }
                }
#pragma unroll
                for (int k = 0; k < CAP; ++k)
                    if (e.at(k) != 0xffffu)
                        *slot_at(x, e.at(k), half) =
                            make_float4(gl.x - g[k].x, gl.y - g[k].y, gl.z - g[k].z, gl.w - g[k].w);
            }
            __syncthreads();
            const float* wt = a.w + (size_t)(t - 1) * (size_t)a.E;
            float* gwt = part + (size_t)(t - 1) * (size_t)a.E;
            const size_t rec = ((size_t)tile * a.T + (size_t)(t - 1)) * (size_t)a.M * kShots;
            // (a task's records lie at rec + 4 q)
            float4 m1n, m2n;
            uint2 pvn;
            auto load_record = [&](int q) {
                m1n = __ldg(reinterpret_cast<const float4*>(a.m1 + rec) + q);
                m2n = __ldg(reinterpret_cast<const float4*>(a.m2 + rec) + q);
                pvn = __ldg(reinterpret_cast<const uint2*>(a.pk + rec) + q);
            };
            load_record((int)threadIdx.x < 2 * a.M ? (int)threadIdx.x : 0);
            for (int q = threadIdx.x; q < ((2 * a.M + 31) & ~31); q += blockDim.x) {
                const bool in = q < 2 * a.M;
                const int i = in ? q >> 1 : 0, half = q & 1;
                const int rb = rp[i], deg = in ? rp[i + 1] - rb : 0;
                const float4 m1v = m1n, m2v = m2n;
                const uint2 pv = pvn;
                if (q + (int)blockDim.x < 2 * a.M) load_record(q + (int)blockDim.x);
                const uint32_t s4 = (uint32_t)sb[i] >> (4 * half);
                uint32_t neg[4], sig[4];
                int i1[4], i2[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t p = (c < 2 ? pv.x : pv.y) >> (16 * (c & 1));
                    neg[c] = p & 0xFFu;
                    i1[c] = (int)((p >> 8) & 15u);
                    i2[c] = (int)((p >> 12) & 15u);
                    // bit k: the sign of the product over the other edges
                    sig[c] = (((uint32_t)__popc(neg[c]) ^ (s4 >> c)) & 1u) ? ~neg[c] : neg[c];
                }
                float acc1[4] = {0.f, 0.f, 0.f, 0.f}, g1[4] = {0.f, 0.f, 0.f, 0.f}, gw[kMaxDeg], wv[kMaxDeg];
                const bool wide = row_weights(wt, rb, deg, wv);
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k) {
                    gw[k] = 0.f;
                    if (k < deg) {
                        const float4 g = *tile_at(x, rb + k, half);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float gd = __uint_as_float(__float_as_uint(comp(g, c)) ^ (((sig[c] >> k) & 1u) << 31));
                            gw[k] += gd * (k == i1[c] ? comp(m2v, c) : comp(m1v, c));
                            const float gm = gd * wv[k];
                            if (k == i1[c]) g1[c] = gm; else acc1[c] += gm;
                        }
                    }
                    // the tile's other four shots are in the next lane
                    gw[k] += __shfl_xor_sync(0xffffffffu, gw[k], 1);
                }
                if (wide && row_aligned(gwt, rb, deg)) {
                    float4* o = reinterpret_cast<float4*>(gwt + rb) + half;
                    float4 r = half ? make_float4(gw[4], gw[5], gw[6], gw[7]) : make_float4(gw[0], gw[1], gw[2], gw[3]);
                    if (!fresh) {
                        const float4 p = *o;
                        r.x += p.x; r.y += p.y; r.z += p.z; r.w += p.w;
                    }
                    *o = r;
                } else if (half == 0) {
#pragma unroll
                    for (int k = 0; k < kMaxDeg; ++k)
                        if (k < deg) gwt[rb + k] = fresh ? gw[k] : gwt[rb + k] + gw[k];
                }
                if (t > 1) {
#pragma unroll
                    for (int k = 0; k < kMaxDeg; ++k) {
                        if (k < deg) {
                            float4 o;
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                // d|E|/dE = sign(E), 0 at 0
                                const float m = k == i1[c] ? comp(m1v, c) : comp(m2v, c);
                                float r = k == i1[c] ? acc1[c] : g1[c];
                                r = __uint_as_float(__float_as_uint(r) ^ (((neg[c] >> k) & 1u) << 31));
                                setc(o, c, (k == i1[c] || (k == i2[c] && i1[c] != 15)) && m > 0.f ? r : 0.f);
                            }
                            *tile_at(x, rb + k, half) = o;
                        }
                    }
                }
            }
            __syncthreads();
        }
    }
}

// weight gradients of the tiled backward: the blocks' partial sums in order
__global__ void k_u_gw_blocks(const float* __restrict__ part, long long n, int blocks, float* __restrict__ grad)
{
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int k = 0; k < blocks; ++k) s += (double)part[(size_t)k * (size_t)n + (size_t)q];
        grad[q] = (float)s;
    }
}

// the limit belongs to the kernel, not to a decoder: always the device maximum, so
// that a thread with a smaller code does not lower it between another's call and
// its launch
template <class F>
bool allow_smem(const DevGraph& g, F* kernel)
{
    return !CUDA_FAILED(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, g.max_smem));
}

// The tiled path's arrays in the caller's workspace (base may be null: their size
// only).  It runs wherever the code allows it, whatever ckpt_every is: the interval
// changes no bit of the results.  It keeps 10 bytes per (row, shot) and 4 per (node,
// shot) of every iteration, on the phenomenological DEM 0.96 of what the passes need
// with their best interval at T = 20 and 1.27 at T = 30; so that no training that fit
// the device stops fitting, a workspace above kTileBytes is taken only where the
// passes' smallest is no smaller.
constexpr size_t kTileBytes = size_t(8) << 30;
bool tile_plan(const DevGraph& g, const DecCfg& cfg, long long B, int T, const float* w, char* base, TileArgs* out,
               size_t* bytes)
{
    if (g.max_row_deg > kMaxDeg || g.tile_slots == nullptr || g.E > 65528 || g.max_row_deg < 1) return false;
    const size_t smem = tile_smem(g.M, g.N, g.E);
    if (smem > (size_t)g.max_smem) return false;
    TileArgs a{};
    a.row_ptr = g.row_ptr; a.row_col = g.row_col; a.col_slot = g.tile_slots; a.lam = g.lam;
    a.M = g.M; a.N = g.N; a.E = g.E; a.T = T; a.L = cfg.L; a.B = B; a.w = w;
    a.ntile = (int)((B + kShots - 1) / kShots);
    // a thread per four shots of a row or of two columns, at most kFwdThreads or kBwdThreads;
    // as many blocks as fit at once, or fewer with the same number of tiles each
    const int want = std::max(2 * g.M, g.N);
    a.threads = std::max(64, (want + 31) / 32 * 32);
    const int fit = g.sms * std::max(1, std::min((int)((size_t)g.max_smem / smem), kFwdThreads / a.threads));
    const int rounds = (a.ntile + fit - 1) / fit;
    a.blocks = (a.ntile + rounds - 1) / rounds;
    const size_t nt = (size_t)a.ntile, TM = (size_t)T * (size_t)g.M * kShots, TN = (size_t)T * (size_t)g.N * kShots;
    size_t off = 0;
    auto take = [&](size_t n) {
        char* p = base ? base + off : nullptr;
        off += a256(n);
        return p;
    };
    a.s8 = (unsigned char*)take(nt * (size_t)g.M);
    a.y8 = (unsigned char*)take(nt * (size_t)g.N);
    a.m1 = (float*)take(sizeof(float) * nt * TM);
    a.m2 = (float*)take(sizeof(float) * nt * TM);
    a.pk = (uint16_t*)take(sizeof(uint16_t) * nt * TM);
    a.lamT = (float*)take(sizeof(float) * nt * TN);
    a.loss_part = (float*)take(sizeof(float) * nt * (size_t)T);
    a.gw_part = (float*)take(sizeof(float) * (size_t)a.blocks * (size_t)T * (size_t)g.E);
    a.hazard = (int*)take(sizeof(int) * kHazardBlocks);
    if (off > kTileBytes) {
        // (the passes' size falls, then rises with the interval, turning below sqrt(T) + 1)
        size_t least = SIZE_MAX;
        for (long long k = 1; k <= T && (k - 1) * (k - 1) <= T; ++k)
            least = std::min(least, layout(g, B, T, (int)k, nullptr).bytes);
        if (off > least) return false;
    }
    if (out) *out = a;
    *bytes = off;
    return true;
}

// bytes of the caller's workspace, on the path that runs
size_t work_bytes_of(const DevGraph& g, const DecCfg& cfg, long long B, int T, int k)
{
    size_t bytes = 0;
    return tile_plan(g, cfg, B, T, nullptr, nullptr, nullptr, &bytes) ? bytes : layout(g, B, T, k, nullptr).bytes;
}

// plain BP (Eqs. 1-3 with the scale alpha, the sums in ascending order) for T
// iterations on the same tiles: Lambda_j(T), and the sum of Lambda_j(t) held by the
// thread of (column, half tile) over the iterations.  For column degrees up to 3,
// whose ordered sums need no sort.  Bound by shared memory (each message read and
// written twice per iteration).  8192 shots of the phenomenological DEM, T = 20:
// 2.47 ms as candidates of 16 warps, 1.08 here; the sums in memory 1.36 (3.5 GB
// through L2), 640 threads and 9 sums 1.13, 768 and 7 1.21 (both spill).
constexpr int kLlrThreads = 512, kLlrHeld = 11;

__global__ void __launch_bounds__(kLlrThreads, 1) k_llr_tiles(TileArgs a, float alpha, const uint32_t* __restrict__ synd,
                                                              int WM, float* __restrict__ llr,
                                                              float* __restrict__ sum_llr)
{
    extern __shared__ __align__(16) float sm[];
    float* const x = sm;
    unsigned char* const sb = reinterpret_cast<unsigned char*>(sm + (((size_t)a.E + 3) & ~size_t(3)) * kShots);
    uint16_t* const rp = reinterpret_cast<uint16_t*>(
        reinterpret_cast<float*>(sb + (((size_t)a.M + (size_t)a.N + 15) & ~size_t(15))) + 64);                // row_ptr
    for (int q = threadIdx.x; q <= a.M; q += blockDim.x) rp[q] = (uint16_t)__ldg(a.row_ptr + q);
    for (int tile = blockIdx.x; tile < a.ntile; tile += gridDim.x) {
        const long long b0 = (long long)tile * kShots;
        for (int i = threadIdx.x; i < a.M; i += blockDim.x) {
            uint32_t v = 0;
#pragma unroll
            for (int c = 0; c < kShots; ++c)
                if (b0 + c < a.B) v |= ((__ldg(synd + (size_t)(b0 + c) * WM + (i >> 5)) >> (i & 31)) & 1u) << c;
            sb[i] = (unsigned char)v;
        }
        for (int q = threadIdx.x; q < 2 * a.E; q += blockDim.x) {          // E(0)
            const float v = fminf(fmaxf(__ldg(a.lam + __ldg(a.row_col + (q >> 1))), -a.L), a.L);
            *tile_at(x, q >> 1, q & 1) = make_float4(v, v, v, v);
        }
        __syncthreads();
        float4 sum[kLlrHeld];
#pragma unroll
        for (int r = 0; r < kLlrHeld; ++r) sum[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t = 1; t <= a.T; ++t) {
            for (int q = threadIdx.x; q < 2 * a.M; q += blockDim.x) {
                const int i = q >> 1, half = q & 1;
                const int rb = rp[i], deg = rp[i + 1] - rb;
                const uint32_t s4 = (uint32_t)sb[i] >> (4 * half);
                float4 v[kMaxDeg];
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k)
                    v[k] = k < deg ? *tile_at(x, rb + k, half) : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    // signed minima over the others from running ones from both
                    // ends, capped at L_MAX with the syndrome sign
                    float out[kMaxDeg];
                    out[kMaxDeg - 1] = INFINITY;
#pragma unroll
                    for (int k = kMaxDeg - 1; k > 0; --k)
                        out[k - 1] = k == kMaxDeg - 1 ? comp(v[k], c) : xmin(comp(v[k], c), out[k]);
                    float pre = __uint_as_float(__float_as_uint(a.L) | (((s4 >> c) & 1u) << 31));
#pragma unroll
                    for (int k = 0; k < kMaxDeg; ++k) {
                        const float m = k == kMaxDeg - 1 ? pre : xmin(pre, out[k]);
                        if (k + 1 < kMaxDeg) pre = xmin(pre, comp(v[k], c));
                        setc(v[k], c, __fmul_rn(alpha, m));
                    }
                }
#pragma unroll
                for (int k = 0; k < kMaxDeg; ++k)
                    if (k < deg) *tile_at(x, rb + k, half) = v[k];
            }
            __syncthreads();
            ColumnSlots<4> en;
            float ln = 0.f;
            if ((int)threadIdx.x < 2 * a.N) {
                en.load(a, threadIdx.x >> 1);
                ln = __ldg(a.lam + (threadIdx.x >> 1));
            }
#pragma unroll
            for (int r = 0; r < kLlrHeld; ++r) {
                const int q = threadIdx.x + r * blockDim.x;
                if (q >= 2 * a.N) break;
                const int j = q >> 1, half = q & 1;
                const ColumnSlots<4> e = en;
                const float lj = ln;
                if (q + (int)blockDim.x < 2 * a.N) {
                    en.load(a, (q + (int)blockDim.x) >> 1);
                    ln = __ldg(a.lam + ((q + (int)blockDim.x) >> 1));
                }
                const long long b = b0 + 4 * half;
                float4 v[3];
                int deg = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (e.at(k) != 0xffffu) {
                        v[k] = *slot_at(x, e.at(k), half);
                        deg = k + 1;
                    }
                float4 post = make_float4(lj, lj, lj, lj);
                if (deg == 3) {
                    float4 o[3];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float v0 = comp(v[0], c), v1 = comp(v[1], c), v2 = comp(v[2], c);
                        const float lo12 = fminf(v1, v2), hi12 = fmaxf(v1, v2);
                        const float lo02 = fminf(v0, v2), hi02 = fmaxf(v0, v2);
                        const float lo01 = fminf(v0, v1), hi01 = fmaxf(v0, v1);
                        setc(o[0], c, __fadd_rn(__fadd_rn(lj, lo12), hi12));
                        setc(o[1], c, __fadd_rn(__fadd_rn(lj, lo02), hi02));
                        setc(o[2], c, __fadd_rn(__fadd_rn(lj, lo01), hi01));
                        // smallest, median (the least of the pair maxima), largest
                        const float mid = fminf(hi01, fminf(hi02, hi12));
                        setc(post, c, __fadd_rn(__fadd_rn(__fadd_rn(lj, fminf(lo01, v2)), mid), fmaxf(hi01, v2)));
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) *slot_at(x, e.at(k), half) = o[k];
                } else if (deg == 2) {
                    float4 o[2];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float v0 = comp(v[0], c), v1 = comp(v[1], c);
                        setc(o[0], c, __fadd_rn(lj, v1));
                        setc(o[1], c, __fadd_rn(lj, v0));
                        setc(post, c, __fadd_rn(__fadd_rn(lj, fminf(v0, v1)), fmaxf(v0, v1)));
                    }
                    *slot_at(x, e.at(0), half) = o[0];
                    *slot_at(x, e.at(1), half) = o[1];
                } else if (deg == 1) {
                    *slot_at(x, e.at(0), half) = post;
                    post = make_float4(__fadd_rn(lj, v[0].x), __fadd_rn(lj, v[0].y), __fadd_rn(lj, v[0].z),
                                       __fadd_rn(lj, v[0].w));
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    setc(sum[r], c, __fadd_rn(comp(sum[r], c), comp(post, c)));
                    if (t != a.T || b + c >= a.B) continue;
                    const size_t at = (size_t)(b + c) * (size_t)a.N + j;
                    llr[at] = comp(post, c);
                    if (sum_llr) sum_llr[at] = comp(sum[r], c);
                }
            }
            __syncthreads();
        }
    }
}

// register cache for rows / columns of degree at most 4 or 8, none beyond
int cap_of(int max_deg) { return max_deg <= 4 ? 4 : (max_deg <= 8 ? 8 : 0); }

int grid_y(int items) { return items < 65535 ? (items > 0 ? items : 1) : 65535; }

int check_args(const bsd_decoder* dec, int64_t B, int32_t T, int32_t k, const DevGraph** g, const DecCfg** cfg,
               int* device)
{
    if (!dec || B < 1 || T < 1 || k < 1 || k > T || B > (1ll << 30)) return BSD_ERR_INVALID_ARG;
    if (decoder_graph(dec, g, cfg, device) != BSD_OK) return BSD_ERR_INVALID_ARG;
    if ((*g)->prec != 0) return BSD_ERR_UNSUPPORTED;
    return BSD_OK;
}

UArgs make_args(const DevGraph& g, const DecCfg& cfg, long long B, int T, const float* w, const ULayout& u)
{
    UArgs a{};
    a.row_ptr = g.row_ptr;
    a.col_ptr = g.col_ptr;
    a.col_edge = g.col_edge;
    a.lam = g.lam;
    a.M = g.M; a.N = g.N; a.E = g.E;
    a.L = cfg.L;
    a.B = B;
    a.Bp = (B + kTile - 1) / kTile * kTile;
    a.ntile = (int)(a.Bp / kTile);
    a.T = T;
    a.w = w;
    a.sT = u.sT;
    a.yT = u.yT;
    return a;
}

struct DeviceScope {
    int prev = -1;
    bool ok = false;
    explicit DeviceScope(int dev)
    {
        if (CUDA_FAILED(cudaGetDevice(&prev))) prev = -1;
        ok = !CUDA_FAILED(cudaSetDevice(dev));
    }
    ~DeviceScope()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// event hooks around a launch when the decoder's kernel timing is on
enum { kKindCheck = 3, kKindVar = 4, kKindBVar = 5, kKindBCheck = 6, kKindOther = 7 };
struct Timed {
    const LaunchHooks* hk;
    int kind;
    Timed(const LaunchHooks* h, int k) : hk(h), kind(k) { if (hk) hk->before(hk->ctx, kind); }
    ~Timed() { if (hk) hk->after(hk->ctx, kind); }
};

void launch_check(const UArgs& a, const DevGraph& g, const float* Ein, float* D, int t, cudaStream_t s,
                  const LaunchHooks* hk)
{
    const dim3 grid(a.ntile, grid_y(a.M));
    Timed tm(hk, kKindCheck);
    switch (cap_of(g.max_row_deg)) {
        case 4: k_u_check<4><<<grid, kThreads, 0, s>>>(a, Ein, D, t); break;
        case 8: k_u_check<8><<<grid, kThreads, 0, s>>>(a, Ein, D, t); break;
        default: k_u_check<0><<<grid, kThreads, 0, s>>>(a, Ein, D, t); break;
    }
}

void launch_var(const UArgs& a, const DevGraph& g, const float* D, float* Eout, float* lamT, float* llr,
                float* loss_part, cudaStream_t s, const LaunchHooks* hk)
{
    const dim3 grid(a.ntile, grid_y(a.N));
    Timed tm(hk, kKindVar);
    switch (cap_of(g.max_col_deg)) {
        case 4: k_u_var<4><<<grid, kThreads, 0, s>>>(a, D, Eout, lamT, llr, loss_part); break;
        case 8: k_u_var<8><<<grid, kThreads, 0, s>>>(a, D, Eout, lamT, llr, loss_part); break;
        default: k_u_var<0><<<grid, kThreads, 0, s>>>(a, D, Eout, lamT, llr, loss_part); break;
    }
}

}  // namespace

// plain BP on tiles of shots where it applies: single precision, no weights, rows
// of at most 8 and columns of at most 3 edges, the tile in shared memory; 1 where
// not.  A wave of tiles takes the time of one tile: against candidates of one warp
// each (864 columns, T = 20) 82 us for any batch up to 8 per SM where they take
// 290-350; a candidate of 16 warps (2592 columns) is done sooner while each SM has
// at most two, 66-98 us against 150, and later from three on, 187.
int launch_llr_tiles(const DevGraph& g, const DecCfg& cfg, const LaunchShape& ls, const uint32_t* synd, long long B, int T, float* llr,
                     float* sum_llr, void* stream)
{
    const size_t smem = tile_smem(g.M, g.N, g.E);
    if (g.prec != 0 || cfg.weights != nullptr || g.max_row_deg > kMaxDeg || g.max_row_deg < 1 || g.max_col_deg > 3 ||
        g.tile_slots == nullptr || smem > (size_t)g.max_smem || (ls.group_warps > 1 && B < 3ll * g.sms))
        return 1;
    TileArgs a{};
    a.row_ptr = g.row_ptr; a.row_col = g.row_col; a.col_slot = g.tile_slots; a.lam = g.lam;
    a.M = g.M; a.N = g.N; a.E = g.E; a.T = T; a.L = cfg.L; a.B = B;
    a.ntile = (int)((B + kShots - 1) / kShots);
    const int threads = std::min(kLlrThreads, std::max(64, (std::max(2 * g.M, g.N) + 31) / 32 * 32));
    const int fit = g.sms * std::max(1, std::min((int)((size_t)g.max_smem / smem), kLlrThreads / threads));
    if (2ll * g.N > (long long)kLlrHeld * threads) return 1;
    if (!allow_smem(g, k_llr_tiles)) return -2;
    k_llr_tiles<<<std::min(a.ntile, fit), threads, smem, (cudaStream_t)stream>>>(a, cfg.alpha, synd, g.WM, llr, sum_llr);
    return CUDA_FAILED(cudaGetLastError()) ? -2 : 0;
}
}  // namespace bsd

using namespace bsd;

extern "C" {

int bsd_unrolled_workspace(const bsd_decoder* dec, int64_t B, int32_t T, int32_t ckpt_every, int64_t* bytes)
{
    const DevGraph* g;
    const DecCfg* cfg;
    int device;
    if (!bytes) return BSD_ERR_INVALID_ARG;
    const int rc = check_args(dec, B, T, ckpt_every, &g, &cfg, &device);
    if (rc) return rc;
    *bytes = (int64_t)work_bytes_of(*g, *cfg, B, T, ckpt_every);
    return BSD_OK;
}

int bsd_unrolled_forward(const bsd_decoder* dec, const uint32_t* d_syndromes, const uint32_t* d_errors, int64_t B,
                         int32_t T, int32_t ckpt_every, const float* d_weights, float* d_loss, float* d_llr,
                         void* d_work, int64_t work_bytes, void* cuda_stream)
{
    const DevGraph* g;
    const DecCfg* cfg;
    int device;
    int rc = check_args(dec, B, T, ckpt_every, &g, &cfg, &device);
    if (rc) return rc;
    if (!d_syndromes || !d_errors || !d_weights || !d_loss || !d_work) return BSD_ERR_INVALID_ARG;
    if (work_bytes < (int64_t)work_bytes_of(*g, *cfg, B, T, ckpt_every) || ((uintptr_t)d_work & 255u))
        return BSD_ERR_INVALID_ARG;
    DeviceScope ds(device);
    if (!ds.ok) return BSD_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    LaunchHooks hks;
    const LaunchHooks* hk = decoder_hooks(dec, s, &hks) ? &hks : nullptr;
    TileArgs ta;
    size_t tile_bytes;
    if (tile_plan(*g, *cfg, B, T, d_weights, (char*)d_work, &ta, &tile_bytes)) {
        const size_t smem = tile_smem(g->M, g->N, g->E);
        auto kf = g->max_col_deg <= 4 ? k_u_forward<4> : k_u_forward<8>;
        if (!allow_smem(*g, kf)) return BSD_ERR_CUDA;
        {
            Timed tm(hk, kKindOther);
            k_u_hazard<<<kHazardBlocks, 256, 0, s>>>(d_weights, (size_t)T * (size_t)g->E, FLT_MAX / (16.f * cfg->L),
                                                     ta.hazard);
        }
        {
            Timed tm(hk, kKindCheck);
            kf<<<ta.blocks, std::min(ta.threads, kFwdThreads), smem, s>>>(ta, d_syndromes, d_errors, g->WM, g->WN, d_llr);
        }
        Timed tm(hk, kKindOther);
        k_u_loss<<<T, 256, 0, s>>>(ta.loss_part, 1, ta.ntile, 1.0 / ((double)B * (double)g->N), d_loss);
        k_u_loss_total<<<1, 32, 0, s>>>(T, d_loss);
        return CUDA_FAILED(cudaGetLastError()) ? BSD_ERR_CUDA : BSD_OK;
    }
    const ULayout u = layout(*g, B, T, ckpt_every, (char*)d_work);
    const UArgs a = make_args(*g, *cfg, B, T, d_weights, u);
    const int k = ckpt_every;
    const size_t EB = (size_t)g->E * (size_t)a.Bp;
    {
        Timed tm(hk, kKindOther);
        k_u_planes<<<1024, 256, 0, s>>>(d_syndromes, B, g->WM, g->M, a.Bp, u.sT);
        k_u_planes<<<1024, 256, 0, s>>>(d_errors, B, g->WN, g->N, a.Bp, u.yT);
        k_u_init<<<dim3(a.ntile, grid_y(g->N)), kThreads, 0, s>>>(a, u.ck);
    }
    // E(t) lives in its checkpoint slot at t = c k, else in a scratch buffer
    const float* src = u.ck;
    for (int t = 1; t <= T; ++t) {
        launch_check(a, *g, src, u.D, t, s, hk);
        float* dst = (t % k == 0 && t < T) ? u.ck + (size_t)(t / k) * EB : u.seg;
        launch_var(a, *g, u.D, dst, nullptr, d_llr ? d_llr + (size_t)(t - 1) * (size_t)B * g->N : nullptr,
                   u.loss_part + (size_t)(t - 1) * g->N * a.ntile * kWarps, s, hk);
        src = dst;
    }
    {
        Timed tm(hk, kKindOther);
        k_u_loss<<<T, 256, 0, s>>>(u.loss_part, g->N, a.ntile * kWarps, 1.0 / ((double)B * (double)g->N), d_loss);
        k_u_loss_total<<<1, 32, 0, s>>>(T, d_loss);
    }
    return CUDA_FAILED(cudaGetLastError()) ? BSD_ERR_CUDA : BSD_OK;
}

int bsd_unrolled_backward(const bsd_decoder* dec, int64_t B, int32_t T, int32_t ckpt_every, const float* d_weights,
                          const float* d_grad_loss, float* d_grad_weights, void* d_work, int64_t work_bytes,
                          void* cuda_stream)
{
    const DevGraph* g;
    const DecCfg* cfg;
    int device;
    int rc = check_args(dec, B, T, ckpt_every, &g, &cfg, &device);
    if (rc) return rc;
    if (!d_weights || !d_grad_loss || !d_grad_weights || !d_work) return BSD_ERR_INVALID_ARG;
    if (work_bytes < (int64_t)work_bytes_of(*g, *cfg, B, T, ckpt_every) || ((uintptr_t)d_work & 255u))
        return BSD_ERR_INVALID_ARG;
    DeviceScope ds(device);
    if (!ds.ok) return BSD_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const double scale = 1.0 / ((double)B * (double)g->N);
    LaunchHooks hks;
    const LaunchHooks* hk = decoder_hooks(dec, s, &hks) ? &hks : nullptr;
    TileArgs ta;
    size_t tile_bytes;
    if (tile_plan(*g, *cfg, B, T, d_weights, (char*)d_work, &ta, &tile_bytes)) {
        const size_t smem = tile_smem(g->M, g->N, g->E);
        auto kb = g->max_col_deg <= 4 ? k_u_backward<4> : k_u_backward<8>;
        if (!allow_smem(*g, kb)) return BSD_ERR_CUDA;
        {
            Timed tm(hk, kKindBVar);
            kb<<<ta.blocks, std::min(ta.threads, kBwdThreads), smem, s>>>(ta, d_grad_loss, scale);
        }
        Timed tm(hk, kKindOther);
        k_u_gw_blocks<<<1024, 128, 0, s>>>(ta.gw_part, (long long)T * g->E, ta.blocks, d_grad_weights);
        return CUDA_FAILED(cudaGetLastError()) ? BSD_ERR_CUDA : BSD_OK;
    }
    const ULayout u = layout(*g, B, T, ckpt_every, (char*)d_work);
    const UArgs a = make_args(*g, *cfg, B, T, d_weights, u);
    const int k = ckpt_every;
    const size_t EB = (size_t)g->E * (size_t)a.Bp, NB = (size_t)g->N * (size_t)a.Bp;
    const int cap_c = cap_of(g->max_col_deg);
    const dim3 gcol(a.ntile, grid_y(g->N)), grow(a.ntile, grid_y(g->M));
    int cur = 0;                               // gE(t) lives in u.gE[cur]
    const int C = (T + k - 1) / k;
    for (int c = C - 1; c >= 0; --c) {
        const int t0 = c * k, t1 = (t0 + k < T) ? t0 + k : T;
        // recompute E(t) and Lambda(t) of the segment from its checkpoint
        const float* src = u.ck + (size_t)c * EB;
        for (int t = t0 + 1; t <= t1; ++t) {
            launch_check(a, *g, src, u.D, t, s, hk);
            float* dst = u.seg + (size_t)(t - t0 - 1) * EB;
            launch_var(a, *g, u.D, dst, u.lamT + (size_t)(t - t0 - 1) * NB, nullptr, nullptr, s, hk);
            src = dst;
        }
        for (int t = t1; t > t0; --t) {
            const float* Et = u.seg + (size_t)(t - t0 - 1) * EB;
            const float* lamT = u.lamT + (size_t)(t - t0 - 1) * NB;
            const float* gEin = (t == T) ? nullptr : u.gE[cur];
            {
                Timed tm(hk, kKindBVar);
                if (cap_c == 4)
                    k_u_bvar<4><<<gcol, kThreads, 0, s>>>(a, gEin, Et, lamT, d_grad_loss, scale, t, u.gD);
                else if (cap_c == 8)
                    k_u_bvar<8><<<gcol, kThreads, 0, s>>>(a, gEin, Et, lamT, d_grad_loss, scale, t, u.gD);
                else k_u_bvar<0><<<gcol, kThreads, 0, s>>>(a, gEin, Et, lamT, d_grad_loss, scale, t, u.gD);
            }
            const float* Eprev = (t == t0 + 1) ? u.ck + (size_t)c * EB : u.seg + (size_t)(t - t0 - 2) * EB;
            float* gEout = (t > 1) ? u.gE[cur ^ 1] : nullptr;
            float* gwp = u.gw_part + (size_t)(t - 1) * a.ntile * kWarps * g->E;
            {
                Timed tm(hk, kKindBCheck);
                // the check adjoint reloads its vectors (64 registers, 8 blocks per SM):
                // faster than holding them (96 registers, 5 blocks)
                k_u_bcheck<0><<<grow, kThreads, 0, s>>>(a, Eprev, u.gD, gEout, gwp, t);
            }
            cur ^= 1;
        }
    }
    {
        Timed tm(hk, kKindOther);
        k_u_gw<<<1024, 256, 0, s>>>(u.gw_part, T, a.ntile * kWarps, g->E, d_grad_weights);
    }
    return CUDA_FAILED(cudaGetLastError()) ? BSD_ERR_CUDA : BSD_OK;
}

}  // extern "C"
