// bsd_layout.cu -- where the BP engines keep each edge's messages in shared
// memory (host code, run once when a decoder is created).
//
// Jagged engine (column degree bound 3 or 6; generic_layout): a row's
// edges occupy the row's places (given by the caller) in any order (the detector
// pass reduces them with order-independent operations),
// and a column's edges may take any k slots of the padded column table (the
// error pass sorts its inputs).  A local search over swaps within rows
// spreads each group of 32 columns over the banks (at most the group's
// largest column degree per bank), and a colouring of the group's
// (column, bank) multigraph then gives each k slot distinct banks; where the
// search leaves a bank above that, each edge takes the free slot whose bank
// is least loaded.  Columns may keep holes in their slots.
//
// Single-warp engine: small_local_layout (described there) deals the columns to the
// lanes; small_layout, an earlier placement of the same words with the columns in
// their own order, is exported for inspection and described here:
//
// The single-warp engine (codes with every row of degree 6 and every column of
// degree 3) runs two passes per BP iteration over a candidate's messages in
// shared memory (Eqs. 1-3):
//   detector pass  lane l takes rows i = l + 32 r and loads / stores each
//                  row's messages as three 8-byte pairs;
//   error pass     lane l takes columns j = l + 32 c and gathers / scatters
//                  the message of its k-th edge, k = 0, 1, 2, one 4-byte word
//                  each, from a per-(column, k) address table.
// A warp's shared-memory access costs one wavefront per distinct word in the
// busiest of the 32 banks.  Storing row i's pairs at 6 i, 6 i + 2, 6 i + 4
// makes the detector pass conflict-free but leaves the error pass about 2.3
// wavefronts per access on [[144,12,12]].
//
// Placement used here: pair h of row i at word h P + 2 i, three planes of
// stride P = 64 ceil(M / 32) + 12 (a compile-time constant of the engine,
// which holds ceil(M / 32) rows per lane, so these addresses fold into its
// load and store offsets); every detector-pass access is 32 consecutive
// pairs, conflict-free.  Two choices leave every value the engine computes
// unchanged, and the search below uses them to make the error pass
// conflict-free too:
//   * the order of a row's six edges over its six positions (the two smallest
//     magnitudes and the sign parity of a row do not depend on it, and each
//     edge's outgoing message depends only on its own input and those);
//   * which of a column's three edges is its k-th (the error pass sorts the
//     three incoming messages before it adds them).
// The error-pass access (c, k) is conflict-free when the 32 k-th edges of
// columns 32 c .. 32 c + 31 sit in 32 distinct banks.  If every bank holds at
// most three of the 96 edges of that column group, such a k exists for every
// column (a bipartite multigraph of columns and banks with degrees <= 3 has a
// proper 3-edge-colouring, Koenig's theorem), built here by alternating
// paths.  The row orders are found by a deterministic local search over
// swaps within a row that lowers the bank loads above three, restarted from
// a few seeds; if no run reaches zero the best one is kept (the engine is
// correct for any placement, only slower).  The skew 12 is one for which an
// exact integer program finds a zero-load placement on the [[72,12,6]],
// [[144,12,12]] and [[108,8,10]] bivariate bicycle codes.
#include "bsd_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

namespace bsd {

namespace {

constexpr int kPlanes = 3;      // pairs per row of degree 6
constexpr int kRowDeg = 6;
constexpr int kColDeg = 3;
constexpr int kTries = 16;      // local-search restarts
constexpr int kSweeps = 200;    // sweeps per restart
constexpr int kLocalMoves = 10000; // moves of the single-warp engine's placement

struct Rng {                    // xorshift64*: a fixed, reproducible sequence
    uint64_t s;
    uint32_t next()
    {
        s ^= s >> 12;
        s ^= s << 25;
        s ^= s >> 27;
        return (uint32_t)((s * 2685821657736338717ull) >> 32);
    }
    uint32_t below(uint32_t n) { return next() % n; }
    uint32_t pick(uint32_t n) { return (uint32_t)(((uint64_t)next() * n) >> 32); }
};

int mod32(int x) { return ((x % 32) + 32) % 32; }

// proper k-colouring (k = 0..2) of the edges of one column group whose banks
// each hold at most three of its edges, the edge (column u, bank v) list
// given; colour[i] receives the colour of edge i
void colour_group(const std::vector<int>& eu, const std::vector<int>& ev, std::vector<int>* colour)
{
    const int n = (int)eu.size();
    colour->assign(n, -1);
    int atU[32][kColDeg], atV[32][kColDeg];
    for (int a = 0; a < 32; ++a)
        for (int c = 0; c < kColDeg; ++c) atU[a][c] = atV[a][c] = -1;
    for (int i = 0; i < n; ++i) {
        const int u = eu[i], v = ev[i];
        int a = -1, b = -1;
        for (int c = 0; c < kColDeg && a < 0; ++c)
            if (atU[u][c] < 0) a = c;
        for (int c = 0; c < kColDeg && b < 0; ++c)
            if (atV[v][c] < 0) b = c;
        if (atV[v][a] >= 0) {
            // swap colours a and b along the path from v that alternates
            // a, b, a, ...; in a bipartite graph it never reaches u, and
            // afterwards a is free at v (and still free at u)
            std::vector<int> path;
            int x = v, side = 1, c = a;            // side 1: x is a bank
            while ((int)path.size() <= n) {
                const int e = side ? atV[x][c] : atU[x][c];
                if (e < 0) break;
                path.push_back(e);
                x = side ? eu[e] : ev[e];
                side ^= 1;
                c = (c == a) ? b : a;
            }
            for (int e : path) {                   // clear, then set with the other colour
                atU[eu[e]][(*colour)[e]] = -1;
                atV[ev[e]][(*colour)[e]] = -1;
            }
            for (int e : path) {
                const int ce = (*colour)[e] == a ? b : a;
                (*colour)[e] = ce;
                atU[eu[e]][ce] = e;
                atV[ev[e]][ce] = e;
            }
        }
        (*colour)[i] = a;
        atU[u][a] = i;
        atV[v][a] = i;
    }
}

}  // namespace

bool small_layout(int M, int N, const int* row_ptr, const int* col_idx, SmallLayout* out)
{
    if (M < 1 || N < 1) return false;
    for (int i = 0; i < M; ++i)
        if (row_ptr[i + 1] - row_ptr[i] != kRowDeg) return false;
    const int E = row_ptr[M];
    std::vector<int> cdeg(N, 0);
    for (int e = 0; e < E; ++e) cdeg[col_idx[e]]++;
    for (int j = 0; j < N; ++j)
        if (cdeg[j] != kColDeg) return false;
    const int NG = (N + 31) / 32;

    const int P = small_plane_stride(M);
    const int A[kPlanes] = {0, P, 2 * P};
    Rng rng{0x9e3779b97f4a7c15ull};
    int best_ex = -1;
    std::vector<int> best_perm;
    std::vector<int> perm((size_t)M * kRowDeg), cnt((size_t)NG * 32);
    for (int t = 0; t < kTries && best_ex != 0; ++t) {
        auto bank = [&](int i, int q) { return mod32(A[q >> 1] + 2 * i + (q & 1)); };
        auto grp = [&](int i, int q) { return col_idx[row_ptr[i] + perm[(size_t)i * kRowDeg + q]] >> 5; };
        for (int i = 0; i < M; ++i)
            for (int q = 0; q < kRowDeg; ++q) perm[(size_t)i * kRowDeg + q] = q;
        std::fill(cnt.begin(), cnt.end(), 0);
        for (int i = 0; i < M; ++i)
            for (int q = 0; q < kRowDeg; ++q) cnt[(size_t)grp(i, q) * 32 + bank(i, q)]++;
        auto over = [&](int g, int b) { return std::max(0, cnt[(size_t)g * 32 + b] - kColDeg); };
        int ex = 0;
        for (int x : cnt) ex += std::max(0, x - kColDeg);
        std::vector<int> order(M);
        for (int i = 0; i < M; ++i) order[i] = i;
        for (int sw = 0; sw < kSweeps && ex > 0; ++sw) {
            for (int i = M - 1; i > 0; --i) std::swap(order[i], order[rng.below((uint32_t)i + 1)]);
            for (int i : order) {
                for (int a = 0; a < kRowDeg; ++a) {
                    for (int b = a + 1; b < kRowDeg; ++b) {
                        const int ga = grp(i, a), gb = grp(i, b);
                        if (ga == gb) continue;
                        const int ba = bank(i, a), bb = bank(i, b);
                        const int before = over(ga, ba) + over(gb, bb) + over(ga, bb) + over(gb, ba);
                        cnt[(size_t)ga * 32 + ba]--; cnt[(size_t)gb * 32 + bb]--;
                        cnt[(size_t)ga * 32 + bb]++; cnt[(size_t)gb * 32 + ba]++;
                        const int after = over(ga, ba) + over(gb, bb) + over(ga, bb) + over(gb, ba);
                        // keep improvements, and one equal move in four to move on a plateau
                        if (after < before || (after == before && rng.below(4) == 0)) {
                            std::swap(perm[(size_t)i * kRowDeg + a], perm[(size_t)i * kRowDeg + b]);
                            ex += after - before;
                        } else {
                            cnt[(size_t)ga * 32 + ba]++; cnt[(size_t)gb * 32 + bb]++;
                            cnt[(size_t)ga * 32 + bb]--; cnt[(size_t)gb * 32 + ba]--;
                        }
                    }
                }
            }
        }
        if (best_ex < 0 || ex < best_ex) {
            best_ex = ex;
            best_perm = perm;
        }
    }

    // word address of every CSR edge
    out->addr.assign(E, 0);
    for (int i = 0; i < M; ++i)
        for (int q = 0; q < kRowDeg; ++q)
            out->addr[row_ptr[i] + best_perm[(size_t)i * kRowDeg + q]] = A[q >> 1] + 2 * i + (q & 1);
    for (int h = 0; h < kPlanes; ++h) out->A[h] = A[h];
    out->A[3] = 0;
    out->extent = A[kPlanes - 1] + 2 * M;
    out->excess = best_ex;

    // the k order of every column from a colouring per column group
    std::vector<int> erow(E);
    for (int i = 0; i < M; ++i)
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) erow[e] = i;
    std::vector<std::vector<int>> cedges(N);
    for (int e = 0; e < E; ++e) cedges[col_idx[e]].push_back(e);
    out->col.assign((size_t)N * kColDeg, 0u);
    for (int g = 0; g < NG; ++g) {
        std::vector<int> ids, eu, ev, colour;
        for (int j = 32 * g; j < std::min(N, 32 * g + 32); ++j)
            for (int e : cedges[j]) {
                ids.push_back(e);
                eu.push_back(j - 32 * g);
                ev.push_back(out->addr[e] & 31);
            }
        // a bank above three edges (a search that did not reach zero) admits
        // no proper colouring: the group keeps the column lists' order
        int vdeg[32] = {0};
        for (int v : ev) vdeg[v]++;
        bool proper = *std::max_element(vdeg, vdeg + 32) <= kColDeg;
        if (proper) colour_group(eu, ev, &colour);
        // every column must take k = 0, 1, 2 once (the engine reads all three)
        for (size_t x = 0; proper && x < ids.size(); x += kColDeg) {
            int seen = 0;
            for (int y = 0; y < kColDeg; ++y) seen |= colour[x + y] >= 0 ? 1 << colour[x + y] : 8;
            proper = seen == 7;
        }
        if (!proper) {
            colour.resize(ids.size());
            for (size_t x = 0; x < ids.size(); ++x) colour[x] = (int)(x % kColDeg);
        }
        for (size_t x = 0; x < ids.size(); ++x) {
            const int e = ids[x], j = col_idx[e];
            out->col[(size_t)j * kColDeg + colour[x]] = ((uint32_t)out->addr[e] << 16) | (uint32_t)erow[e];
        }
    }
    return true;
}

}  // namespace bsd

namespace bsd {

namespace {

constexpr int kMaxColour = 16;
constexpr int kPatience = 4;

// proper colouring with `ncol` colours of the edges of one column group whose
// banks each hold at most ncol of its edges and whose columns have at most
// ncol edges (Koenig's theorem; alternating paths, as colour_group)
void colour_group_n(const std::vector<int>& eu, const std::vector<int>& ev, int ncol, std::vector<int>* colour)
{
    const int n = (int)eu.size();
    colour->assign(n, -1);
    int atU[32][kMaxColour], atV[32][kMaxColour];
    for (int a = 0; a < 32; ++a)
        for (int c = 0; c < kMaxColour; ++c) atU[a][c] = atV[a][c] = -1;
    for (int i = 0; i < n; ++i) {
        const int u = eu[i], v = ev[i];
        int a = -1, b = -1;
        for (int c = 0; c < ncol && a < 0; ++c)
            if (atU[u][c] < 0) a = c;
        for (int c = 0; c < ncol && b < 0; ++c)
            if (atV[v][c] < 0) b = c;
        if (atV[v][a] >= 0) {
            std::vector<int> path;
            int x = v, side = 1, c = a;
            while ((int)path.size() <= n) {
                const int e = side ? atV[x][c] : atU[x][c];
                if (e < 0) break;
                path.push_back(e);
                x = side ? eu[e] : ev[e];
                side ^= 1;
                c = (c == a) ? b : a;
            }
            for (int e : path) {
                atU[eu[e]][(*colour)[e]] = -1;
                atV[ev[e]][(*colour)[e]] = -1;
            }
            for (int e : path) {
                const int ce = (*colour)[e] == a ? b : a;
                (*colour)[e] = ce;
                atU[eu[e]][ce] = e;
                atV[ev[e]][ce] = e;
            }
        }
        (*colour)[i] = a;
        atU[u][a] = i;
        atV[v][a] = i;
    }
}

}  // namespace

bool generic_layout(int M, int N, const int* row_ptr, const int* col_idx, int colK, GenericLayout* out,
                    const int* start, bool quick)
{
    if (M < 1 || N < 1 || colK < 1 || colK > kMaxColour) return false;
    const int E = row_ptr[M];
    if (E > kGenericLayoutMaxEdges) return false;
    std::vector<int> cdeg(N, 0);
    for (int e = 0; e < E; ++e) cdeg[col_idx[e]]++;
    for (int j = 0; j < N; ++j)
        if (cdeg[j] > colK) return false;
    const int NG = (N + 31) / 32;
    std::vector<int> cap(NG, 0);                  // the largest column degree of each group
    for (int j = 0; j < N; ++j) cap[j >> 5] = std::max(cap[j >> 5], cdeg[j]);
    // position of every CSR edge among its row's words: start from the given
    // order (the CSR order) and swap within rows while the bank loads above
    // each group's cap fall
    std::vector<int> pos(E);
    for (int e = 0; e < E; ++e) pos[e] = start ? start[e] : e;
    std::vector<int> cnt((size_t)NG * 32, 0);
    for (int e = 0; e < E; ++e) cnt[(size_t)(col_idx[e] >> 5) * 32 + (pos[e] & 31)]++;
    auto over = [&](int g, int b) { return std::max(0, cnt[(size_t)g * 32 + b] - cap[g]); };
    int ex = 0;
    for (int g = 0; g < NG; ++g)
        for (int b = 0; b < 32; ++b) ex += over(g, b);
    Rng rng{0x243f6a8885a308d3ull};
    std::vector<int> order(M);
    for (int i = 0; i < M; ++i) order[i] = i;
    // a bounded effort: at most ~5e7 swap trials, and kPatience sweeps
    // without a lower load end the search
    double per_sweep = 1.0;
    for (int i = 0; i < M; ++i) {
        const double d = row_ptr[i + 1] - row_ptr[i];
        per_sweep += d * (d - 1) / 2;
    }
    const int max_sweeps = (int)std::min<double>(kSweeps, 5e7 / per_sweep);
    // (quick: the given order starts close to what the search reaches, and it
    // ends at the first sweep that takes off less than a tenth)
    std::vector<int> next;
    int best = ex, stale = 0;
    for (int sw = 0; sw < max_sweeps && ex > 0 && stale < (quick ? 1 : kPatience); ++sw) {
        if (ex < (quick && sw > 0 ? 0.9 * best : best)) { best = ex; stale = 0; } else if (sw > 0) { ++stale; }
        if (quick && stale) break;
        for (int i = M - 1; i > 0; --i) std::swap(order[i], order[rng.below((uint32_t)i + 1)]);
        for (int i : order) {
            if (quick && ex == 0) break;
            // a swap gains only where one of its words is on an overloaded bank, so the
            // others are not tried (quick): next[x] = the first such word from x on
            const int rb = row_ptr[i], re = row_ptr[i + 1];
            next.assign(re - rb + 1, re - rb);
            auto mark = [&] {
                for (int x = re - rb - 1; x >= 0; --x)
                    next[x] = !quick || over(col_idx[rb + x] >> 5, pos[rb + x] & 31) > 0 ? x : next[x + 1];
            };
            mark();
            for (int a = rb; a < re && next[0] < re - rb; ++a) {
                for (int b = a + 1;; ++b) {
                    if (b < re && next[a - rb] != a - rb) b = rb + next[b - rb];
                    if (b >= re) break;
                    const int ga = col_idx[a] >> 5, gb = col_idx[b] >> 5;
                    if (ga == gb) continue;
                    const int ba = pos[a] & 31, bb = pos[b] & 31;
                    const int before = over(ga, ba) + over(gb, bb) + over(ga, bb) + over(gb, ba);
                    cnt[(size_t)ga * 32 + ba]--; cnt[(size_t)gb * 32 + bb]--;
                    cnt[(size_t)ga * 32 + bb]++; cnt[(size_t)gb * 32 + ba]++;
                    const int after = over(ga, ba) + over(gb, bb) + over(ga, bb) + over(gb, ba);
                    if (after < before || (after == before && rng.below(4) == 0)) {
                        std::swap(pos[a], pos[b]);
                        ex += after - before;
                        if (quick) mark();
                    } else {
                        cnt[(size_t)ga * 32 + ba]++; cnt[(size_t)gb * 32 + bb]++;
                        cnt[(size_t)ga * 32 + bb]--; cnt[(size_t)gb * 32 + ba]--;
                    }
                }
            }
        }
    }
    out->pos = pos;
    out->excess = ex;
    // the k slot of every column's edges: a proper colouring per group where
    // the loads allow one (holes where a column has fewer edges than colours),
    // else the column lists' order
    std::vector<std::vector<int>> cedges(N);
    for (int e = 0; e < E; ++e) cedges[col_idx[e]].push_back(e);
    out->kedge.assign((size_t)colK * N, -1);
    for (int g = 0; g < NG; ++g) {
        std::vector<int> ids, eu, ev, colour;
        for (int j = 32 * g; j < std::min(N, 32 * g + 32); ++j)
            for (int e : cedges[j]) {
                ids.push_back(e);
                eu.push_back(j - 32 * g);
                ev.push_back(pos[e] & 31);
            }
        int vdeg[32] = {0};
        for (int v : ev) vdeg[v]++;
        bool proper = cap[g] > 0 && *std::max_element(vdeg, vdeg + 32) <= cap[g];
        if (proper) colour_group_n(eu, ev, cap[g], &colour);
        // every column's edges take distinct slots below colK
        if (proper) {
            std::vector<int> seen((size_t)32 * kMaxColour, 0);
            for (size_t x = 0; x < ids.size() && proper; ++x) {
                const int c = colour[x];
                if (c < 0 || c >= colK || seen[(size_t)eu[x] * kMaxColour + c]++) proper = false;
            }
        }
        if (!proper) {
            // greedy: each edge takes the free slot of its column whose bank
            // is least loaded so far
            colour.assign(ids.size(), 0);
            std::vector<int> load((size_t)colK * 32, 0);
            for (size_t x = 0; x < ids.size();) {
                size_t y = x;
                while (y < ids.size() && eu[y] == eu[x]) ++y;
                uint32_t used = 0;
                for (size_t z = x; z < y; ++z) {
                    int bestk = -1;
                    for (int k = 0; k < colK; ++k) {
                        if ((used >> k) & 1u) continue;
                        if (bestk < 0 || load[(size_t)k * 32 + ev[z]] < load[(size_t)bestk * 32 + ev[z]]) bestk = k;
                    }
                    colour[z] = bestk;
                    used |= 1u << bestk;
                    load[(size_t)bestk * 32 + ev[z]]++;
                }
                x = y;
            }
        }
        for (size_t x = 0; x < ids.size(); ++x) out->kedge[(size_t)colour[x] * N + col_idx[ids[x]]] = ids[x];
    }
    return true;
}

}  // namespace bsd

namespace bsd {

// The single-warp engine's placement: rows in natural order, columns in the order
// of the lanes that process them.
//
// Each full row (of a group of 32 rows) owns two of its columns; they are dealt to
// its lane in the groups 2 r and 2 r + 1, and their messages on that row stay in a
// register.  The other columns form the last group.  The row's other four edges take
// its words 2..5 (all six in the last rows).  An access of the error pass is free of
// conflicts when each bank holds at most two words of a full group's columns (three
// of the last one's): exactly two, as 64 words meet 32 banks, so a placement by
// chance leaves some 20 words over.
//
// Annealing over the words within a row, the two sides of a row's own columns, and
// the columns that rows own (one of the last group taken in, or one of another row,
// which takes one of the last group instead); the cost is the sum of squared loads.
// Four moves of five start at a word of an overloaded bank.  kLocalMoves bound it,
// about 1 ms; some codes end earlier.  Extra wavefronts, beside the error pass's 11 (7
// for up to 96 columns), on average and at most: 2.7 and 4 over 20 numberings of the
// rows and columns of [[144,12,12]], 0.7 and 2 of [[72,12,6]], 2.6 and 5 over 20 random
// (3, 6)-regular codes of 40 to 78 rows; with twice the moves and time 2.0, 0.9 and
// 1.8.  With the owned columns drawn at random and only words and sides moved it was
// 6.3, 2.8 and 5.5, in six times the time.
bool small_local_layout(int M, int N, const int* row_ptr, const int* col_idx, SmallLocal* out)
{
    const int RPL = (M + 31) / 32, CPL = (N + 31) / 32, LC = 2 * (RPL - 1);
    if (RPL < 2 || CPL != LC + 1 || N != 2 * M || CPL > kSmallMaxCpl) return false;
    const int E = row_ptr[M];
    std::vector<int> cedge((size_t)kColDeg * N), deg(N, 0), erow(E);
    for (int i = 0; i < M; ++i) {
        if (row_ptr[i + 1] - row_ptr[i] != kRowDeg) return false;
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int j = col_idx[e];
            if (deg[j] == kColDeg) return false;
            erow[e] = i;
            cedge[(size_t)kColDeg * j + deg[j]++] = e;
        }
    }
    const int full = 32 * (RPL - 1), P = small_plane_stride(M);
    Rng rng{1};
    for (int k = 0; k < 8; ++k) rng.next();                    // (its first draws are small)
    // two columns of its own for every full row (augmenting paths; a row has six
    // columns and a column three rows, so the assignment exists)
    std::vector<int> own(N, -1), seen(N, -1), via(N, -1), queue, rp(M + 1), ci, id, start, pos(N);
    std::vector<int> has(2 * (size_t)full, -1);
    for (int n = 0; n < 2 * full; ++n) {
        // breadth-first over columns from row n / 2, through the rows that own them
        queue.clear();
        int end = -1;
        std::vector<int> from(full, -1);                       // the column a row would give up
        std::vector<char> met(full, 0);
        met[n / 2] = 1;
        std::vector<int> rows(1, n / 2);
        for (size_t q = 0; q < rows.size() && end < 0; ++q) {
            for (int e = row_ptr[rows[q]]; e < row_ptr[rows[q] + 1] && end < 0; ++e) {
                const int j = col_idx[e];
                if (seen[j] == n || own[j] == rows[q]) continue;
                seen[j] = n;
                via[j] = rows[q];
                if (own[j] < 0) end = j;
                else if (!met[own[j]]) { met[own[j]] = 1; from[own[j]] = j; rows.push_back(own[j]); }
            }
        }
        if (end < 0) return false;
        for (int j = end;;) {
            const int i = via[j], given = i == n / 2 ? -1 : from[i];
            own[j] = i;
            int* const h = &has[2 * (size_t)i];
            if (given < 0) { h[n % 2] = j; break; }
            h[h[0] == given ? 0 : 1] = j;
            j = given;
        }
    }
    std::vector<int> grp(N, LC);
    for (int n = 0; n < 2 * full; ++n) grp[has[n]] = 2 * (n / 2 / 32) + n % 2;
    // the words: word[6 i + q] the edge at word q of row i, at[e] its q, bk[e] its bank (-1: in a register)
    std::vector<int> word((size_t)kRowDeg * M, -1), at(E, -1), bk(E, -1);
    std::vector<std::vector<int>> words_of(32);                // word indices by bank
    auto bank = [&](int i, int q) { return ((q >> 1) * P + 2 * i + (q & 1)) & 31; };
    int cnt[kSmallMaxCpl * 32] = {0}, over[kSmallMaxCpl * 32], overpos[kSmallMaxCpl * 32], nover = 0;
    int d = 0;                                                 // cost of the current move
    auto cap = [&](int cell) { return cell < 32 * LC ? 2 : 3; };
    auto shift = [&](int g, int b, int by) {
        const int cell = 32 * g + b, c = cnt[cell];
        cnt[cell] = c + by;
        d += g < LC ? 2 * by * c + 1 : 4 * (std::max(0, c + by - 3) - std::max(0, c - 3));
        if (by > 0 && c == cap(cell)) { overpos[cell] = nover; over[nover++] = cell; }
        if (by < 0 && c == cap(cell) + 1) {
            over[overpos[cell]] = over[--nover];
            overpos[over[nover]] = overpos[cell];
        }
    };
    for (int i = 0; i < M; ++i) {
        int q = i < full ? 2 : 0;
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            if (own[col_idx[e]] == i) continue;
            word[(size_t)kRowDeg * i + q] = e;
            at[e] = q;
            bk[e] = bank(i, q);
            words_of[bk[e]].push_back(kRowDeg * i + q);
            shift(grp[col_idx[e]], bk[e], 1);
            ++q;
        }
    }
    auto count = [&](int j, int by) {                          // column j's words in the loads
        for (int k = 0; k < kColDeg; ++k) {
            const int e = cedge[(size_t)kColDeg * j + k];
            if (bk[e] >= 0) shift(grp[j], bk[e], by);
        }
    };
    auto edge_in = [&](int j, int i) {
        const int* e = &cedge[(size_t)kColDeg * j];
        return erow[e[0]] == i ? e[0] : erow[e[1]] == i ? e[1] : e[2];
    };
    uint32_t odds[32] = {0};                                   // of taking a move that costs d
    auto pass = [&] { return d <= 0 || (d < 32 && rng.next() < odds[d]); };
    // edge e takes the word x of its row's edge f, which goes into a register
    auto put = [&](int e, int f) {
        at[e] = at[f];
        bk[e] = bk[f];
        bk[f] = -1;
        word[(size_t)kRowDeg * erow[e] + at[e]] = e;
    };
    for (int n = 0; n < kLocalMoves && nover > 0; ++n) {
        if (n % 512 == 0) {
            const double T = 0.7 * std::pow(0.35, (double)n / kLocalMoves);
            for (int k = 0; k < 32; ++k) odds[k] = (uint32_t)(4294967295.0 * std::exp(-k / T));
        }
        // a word of an overloaded bank, or one in five times any word
        int e = -1;
        if (rng.pick(5) != 0) {
            const int cell = over[rng.pick((uint32_t)nover)];
            const std::vector<int>& w = words_of[cell & 31];
            uint32_t q = rng.pick((uint32_t)w.size());
            while (grp[col_idx[word[w[q]]]] != cell >> 5) q = q + 1 < w.size() ? q + 1 : 0;
            e = word[w[q]];
        } else {
            do e = (int)rng.pick((uint32_t)E); while (bk[e] < 0);
        }
        const int i = erow[e], j = col_idx[e], lo = i < full ? 2 : 0;
        const uint32_t kind = rng.pick(10);
        d = 0;
        if (kind < 6 || (i >= full && own[j] < 0)) {
            int y = lo + (int)rng.pick((uint32_t)(kRowDeg - lo - 1));
            if (y >= at[e]) ++y;
            const int f = word[(size_t)kRowDeg * i + y], ge = grp[j], gf = grp[col_idx[f]], be = bk[e], bf = bk[f];
            if (ge == gf) continue;
            // (what shifting one word from bank to bank costs, without doing it)
            auto moved = [&](int g, int from, int to) {
                const int a = cnt[32 * g + from], b = cnt[32 * g + to];
                return g < LC ? 2 * (b - a + 1) : 4 * ((b >= 3) - (a > 3));
            };
            d = moved(ge, be, bf) + moved(gf, bf, be);
            if (pass()) {
                shift(ge, be, -1); shift(ge, bf, 1); shift(gf, bf, -1); shift(gf, be, 1);
                std::swap(word[(size_t)kRowDeg * i + at[e]], word[(size_t)kRowDeg * i + y]);
                std::swap(at[e], at[f]);
                std::swap(bk[e], bk[f]);
            }
        } else if (own[j] >= 0 && (kind == 6 || i >= full)) {
            int* const h = &has[2 * (size_t)own[j]];           // the two sides
            auto swap_sides = [&] {
                count(h[0], -1); count(h[1], -1);
                std::swap(grp[h[0]], grp[h[1]]);
                count(h[0], 1); count(h[1], 1);
            };
            swap_sides();
            if (pass()) std::swap(h[0], h[1]); else swap_sides();
        } else {
            // row i owns j in place of its column g; the row i2 that owned j takes
            // a column l of the last group, or g
            const int side = (int)rng.pick(2), g = has[2 * (size_t)i + side], i2 = own[j], eg = edge_in(g, i);
            int l = -1, el = -1, ej = -1, side2 = 0;
            if (i2 >= 0) {
                int cand[kRowDeg], nc = 0;
                for (int q = 2; q < kRowDeg; ++q) {
                    const int f = word[(size_t)kRowDeg * i2 + q];
                    if (own[col_idx[f]] < 0 || col_idx[f] == g) cand[nc++] = f;
                }
                if (nc == 0) continue;
                el = cand[rng.pick((uint32_t)nc)];
                l = col_idx[el];
                ej = edge_in(j, i2);
                side2 = has[2 * (size_t)i2] == j ? 0 : 1;
            }
            const int gg = grp[g], gj = grp[j];
            auto count_all = [&](int by) {
                count(g, by); count(j, by);
                if (l >= 0 && l != g) count(l, by);
            };
            count_all(-1);
            put(eg, e);
            own[g] = -1; grp[g] = LC;
            own[j] = i; grp[j] = gg; has[2 * (size_t)i + side] = j;
            if (l >= 0) { put(ej, el); own[l] = i2; grp[l] = gj; has[2 * (size_t)i2 + side2] = l; }
            count_all(1);
            if (pass()) continue;
            count_all(-1);
            if (l >= 0) { put(el, ej); own[l] = -1; grp[l] = LC; has[2 * (size_t)i2 + side2] = j; }
            put(e, eg);
            own[j] = i2; grp[j] = gj;
            own[g] = i; grp[g] = gg; has[2 * (size_t)i + side] = g;
            count_all(1);
        }
    }
    SmallLocal s;
    s.col.assign((size_t)32 * CPL, -1);
    int next = 32 * LC;
    for (int j = 0; j < N; ++j) {
        const int i = own[j];
        pos[j] = i < 0 ? next++ : 32 * grp[j] + i % 32;
        s.col[pos[j]] = j;
    }
    s.word.assign(E, 0);
    rp[0] = 0;
    for (int i = 0; i < M; ++i) {
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int j = col_idx[e];
            if (own[j] == i) {
                s.word[e] = 2 * i + (grp[j] & 1);
                continue;
            }
            ci.push_back(pos[j]);
            id.push_back(e);
            start.push_back((at[e] >> 1) * P + 2 * i + (at[e] & 1));
        }
        rp[i + 1] = (int)ci.size();
    }
    GenericLayout gl;
    if (!generic_layout(M, N, rp.data(), ci.data(), kColDeg, &gl, start.data(), true)) return false;
    for (size_t x = 0; x < id.size(); ++x) s.word[id[x]] = gl.pos[x];
    // the columns' slots: the register-held word first; the two others of a full
    // group's columns so that each bank's words fall to the two accesses in equal
    // parts or one more to the one (colours in turn along trails through columns
    // and banks, from banks of an odd load first)
    s.slot.assign((size_t)32 * CPL * kColDeg, 0);
    for (int g = 0; g < LC; ++g) {
        int two[32][2], left[32] = {0}, who[32][2 * kRowDeg];
        bool used[32] = {false};
        for (int u = 0; u < 32; ++u) {
            const int j = s.col[32 * g + u];
            int k = 0;
            for (int c = 0; c < kColDeg; ++c) {
                const int e = cedge[(size_t)kColDeg * j + c];
                if (own[j] == erow[e]) s.slot[(size_t)kColDeg * (32 * g + u)] = s.word[e];
                else two[u][k++] = s.word[e];
            }
            for (k = 0; k < 2; ++k) {
                const int b = two[u][k] & 31;
                who[b][left[b]++] = u;
            }
        }
        int load[32];
        std::copy(left, left + 32, load);
        for (int n = 0; n < 96; ++n) {                         // odd loads above two, the other odd ones, the rest
            const int b0 = n & 31;
            if (n < 64 ? !(load[b0] & 1) || (n < 32 && load[b0] < 3) : false) continue;
            for (;;) {
                int b = b0, steps = 0;
                for (;; ++steps) {
                    while (left[b] > 0 && used[who[b][left[b] - 1]]) --left[b];
                    if (left[b] == 0) break;
                    const int u = who[b][--left[b]];
                    used[u] = true;
                    const int first = (two[u][0] & 31) == b ? 0 : 1;
                    int* const w = &s.slot[(size_t)kColDeg * (32 * g + u)];
                    w[1] = two[u][first];
                    w[2] = two[u][1 - first];
                    b = two[u][1 - first] & 31;
                }
                if (steps == 0 || n < 64) break;
            }
        }
    }
    for (int q = 32 * LC; q < N; ++q) {
        int k = 0;
        for (int c = 0; c < kColDeg; ++c) {
            const int x = gl.kedge[(size_t)c * N + q];
            if (x >= 0 && k < kColDeg) s.slot[(size_t)kColDeg * q + k++] = s.word[id[x]];
        }
        if (k != kColDeg) return false;
    }
    s.extent = 2 * P + 2 * M;
    s.extra = 0;                                               // wavefronts that conflicts add to the error pass
    for (int g = 0; g < CPL; ++g)
        for (int k = g < LC ? 1 : 0; k < kColDeg; ++k) {
            int load[32] = {0}, most = 0;
            for (int q = 32 * g; q < std::min(N, 32 * g + 32); ++q)
                most = std::max(most, ++load[s.slot[(size_t)kColDeg * q + k] & 31]);
            s.extra += most - 1;
        }
    *out = s;
    return true;
}

void jagged_layout(int M, int N, const int* row_ptr, const int* col_idx, int colK, JaggedLayout* out)
{
    const int E = row_ptr[M], WN = (N + 31) / 32;
    JaggedLayout l;
    auto rdeg = [&](int i) { return row_ptr[i + 1] - row_ptr[i]; };
    for (int i = 0; i < M; ++i) l.row.push_back(i);
    std::stable_sort(l.row.begin(), l.row.end(), [&](int x, int y) { return rdeg(x) > rdeg(y); });
    std::vector<int> start((size_t)std::max(E, 1), 0);
    l.plane.assign(std::max(1, rdeg(l.row[0])), 0);
    for (int k = 0, at = 0; k < rdeg(l.row[0]); ++k) {
        l.plane[k] = at;
        for (int q = 0; q < M && rdeg(l.row[q]) > k; ++q) start[(size_t)row_ptr[l.row[q]] + k] = at++;
    }
    // the columns' positions: natural, or by degree where more than a quarter
    // of the groups would hold several (columns of degree 2 to 6 at random,
    // 35110 edges: the seed BP of 4300 shots 4.2 -> 3.5 ms together with the tables loaded ahead)
    std::vector<int> cdeg(N, 0);
    for (int e = 0; e < E; ++e) cdeg[col_idx[e]]++;
    for (int j = 0; j < N; ++j) l.order.push_back(j);
    int several = 0;
    for (int q = 0; q < WN; ++q) {
        bool same = true;
        for (int j = 32 * q; j < std::min(N, 32 * q + 32); ++j) same = same && cdeg[j] == cdeg[32 * q];
        several += same ? 0 : 1;
    }
    l.dealt = 4 * several > WN;
    if (l.dealt) std::stable_sort(l.order.begin(), l.order.end(), [&](int x, int y) { return cdeg[x] < cdeg[y]; });
    // the search over the rows' words, with the edges' columns by position
    std::vector<int> at(N), ci((size_t)std::max(E, 1));
    for (int p = 0; p < N; ++p) at[l.order[p]] = p;
    for (int e = 0; e < E; ++e) ci[e] = at[col_idx[e]];
    GenericLayout gl;
    if (generic_layout(M, N, row_ptr, ci.data(), colK, &gl, start.data(), true)) {
        l.word = gl.pos;
        l.slot = gl.kedge;
    } else {                                   // too many edges to search: as they come
        l.word = start;
        l.slot.assign((size_t)colK * N, -1);
        std::vector<int> fill(N, 0);
        for (int e = 0; e < E; ++e) l.slot[(size_t)fill[ci[e]]++ * N + ci[e]] = e;
    }
    for (int q = 0; q < WN; ++q) {
        int hi = 0;
        for (int p = 32 * q; p < std::min(N, 32 * q + 32); ++p) hi = std::max(hi, cdeg[l.order[p]]);
        for (int p = 32 * q; p < std::min(N, 32 * q + 32); ++p) {
            int free = 0;
            for (int k = hi; k < colK; ++k) {
                int& from = l.slot[(size_t)k * N + p];
                if (from < 0) continue;
                while (l.slot[(size_t)free * N + p] >= 0) ++free;
                l.slot[(size_t)free * N + p] = from;
                from = -1;
            }
        }
    }
    *out = l;
}

// H as the exports take it: rows of ascending columns in range
static bool csr_valid(int M, int N, const int32_t* row_ptr, const int32_t* col_idx)
{
    if (row_ptr[0] != 0) return false;
    for (int i = 0; i < M; ++i) {
        if (row_ptr[i + 1] < row_ptr[i]) return false;
        for (int e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            if (col_idx[e] < 0 || col_idx[e] >= N) return false;
            if (e > row_ptr[i] && col_idx[e] <= col_idx[e - 1]) return false;
        }
    }
    return true;
}

}  // namespace bsd

extern "C" int bsd_small_layout(int32_t M, int32_t N, const int32_t* H_row_ptr, const int32_t* H_col_idx,
                                int32_t* plane, int32_t* edge_word, int32_t* col_word, int32_t* extent,
                                int32_t* excess)
{
    if (M < 1 || N < 1 || !H_row_ptr || !H_col_idx || !plane || !edge_word || !col_word || !extent || !excess)
        return BSD_ERR_INVALID_ARG;
    if (!bsd::csr_valid(M, N, H_row_ptr, H_col_idx)) return BSD_ERR_INVALID_ARG;
    bsd::SmallLayout sl;
    if (!bsd::small_layout(M, N, H_row_ptr, H_col_idx, &sl)) return BSD_ERR_UNSUPPORTED;
    for (int h = 0; h < 3; ++h) plane[h] = sl.A[h];
    for (size_t e = 0; e < sl.addr.size(); ++e) edge_word[e] = sl.addr[e];
    for (size_t q = 0; q < sl.col.size(); ++q) col_word[q] = (int32_t)(sl.col[q] >> 16);
    *extent = sl.extent;
    *excess = sl.excess;
    return BSD_OK;
}

extern "C" int bsd_lane_layout(int32_t M, int32_t N, const int32_t* H_row_ptr, const int32_t* H_col_idx,
                               int32_t* edge_word, int32_t* lane_col, int32_t* lane_word, int32_t* extent,
                               int32_t* extra)
{
    if (M < 1 || N < 1 || !H_row_ptr || !H_col_idx || !edge_word || !lane_col || !lane_word || !extent || !extra)
        return BSD_ERR_INVALID_ARG;
    if (!bsd::csr_valid(M, N, H_row_ptr, H_col_idx)) return BSD_ERR_INVALID_ARG;
    bsd::SmallLocal sl;
    if (N > 32 * bsd::kSmallMaxCpl || M > 32 * bsd::kSmallMaxRpl ||
        !bsd::small_local_layout(M, N, H_row_ptr, H_col_idx, &sl))
        return BSD_ERR_UNSUPPORTED;
    std::copy(sl.word.begin(), sl.word.end(), edge_word);
    std::copy(sl.col.begin(), sl.col.end(), lane_col);
    std::copy(sl.slot.begin(), sl.slot.end(), lane_word);
    *extent = sl.extent;
    *extra = sl.extra;
    return BSD_OK;
}

extern "C" int bsd_generic_layout(int32_t M, int32_t N, const int32_t* H_row_ptr, const int32_t* H_col_idx,
                                  int32_t* edge_word, int32_t* slot_edge, int32_t* colK, int32_t* excess)
{
    if (M < 1 || N < 1 || !H_row_ptr || !H_col_idx || !edge_word || !slot_edge || !colK || !excess)
        return BSD_ERR_INVALID_ARG;
    if (!bsd::csr_valid(M, N, H_row_ptr, H_col_idx)) return BSD_ERR_INVALID_ARG;
    const int E = H_row_ptr[M];
    std::vector<int> cdeg(N, 0);
    for (int e = 0; e < E; ++e) cdeg[H_col_idx[e]]++;
    const int max_col = N > 0 ? *std::max_element(cdeg.begin(), cdeg.end()) : 0;
    if (max_col > 6) return BSD_ERR_UNSUPPORTED;
    const int K = max_col <= 3 ? 3 : 6;
    bsd::GenericLayout gl;
    if (!bsd::generic_layout(M, N, H_row_ptr, H_col_idx, K, &gl)) return BSD_ERR_UNSUPPORTED;
    for (int e = 0; e < E; ++e) edge_word[e] = gl.pos[e];
    for (size_t q = 0; q < gl.kedge.size(); ++q) slot_edge[q] = gl.kedge[q];
    *colK = K;
    *excess = gl.excess;
    return BSD_OK;
}

extern "C" int bsd_jagged_layout(int32_t M, int32_t N, const int32_t* H_row_ptr, const int32_t* H_col_idx,
                                 int32_t* rank_row, int32_t* edge_word, int32_t* column, int32_t* slot_edge,
                                 int32_t* colK)
{
    if (M < 1 || N < 1 || !H_row_ptr || !H_col_idx || !rank_row || !edge_word || !column || !slot_edge || !colK)
        return BSD_ERR_INVALID_ARG;
    if (!bsd::csr_valid(M, N, H_row_ptr, H_col_idx)) return BSD_ERR_INVALID_ARG;
    std::vector<int> cdeg(N, 0);
    for (int e = 0; e < H_row_ptr[M]; ++e) cdeg[H_col_idx[e]]++;
    const int max_col = *std::max_element(cdeg.begin(), cdeg.end());
    if (max_col > 6) return BSD_ERR_UNSUPPORTED;
    *colK = max_col <= 3 ? 3 : 6;
    bsd::JaggedLayout l;
    bsd::jagged_layout(M, N, H_row_ptr, H_col_idx, *colK, &l);
    std::copy(l.row.begin(), l.row.end(), rank_row);
    std::copy(l.word.begin(), l.word.begin() + H_row_ptr[M], edge_word);
    std::copy(l.order.begin(), l.order.end(), column);
    std::copy(l.slot.begin(), l.slot.end(), slot_edge);
    return BSD_OK;
}
