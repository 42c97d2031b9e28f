// Per-vertex and per-edge counts of roots of out-degree at most 128.
//
// Alg. 2 credits every member of every root-to-leaf path: a leaf with h hold
// and p pivot links has the clique polynomial x^h (1+x)^p (coefficient of x^k:
// its k-cliques), a hold vertex of it lies in all of them and a pivot vertex
// in x^(h+1) (1+x)^(p-1).  Walked leaf by leaf that is a path listing and a
// row of multi-word atomics per member and leaf, on rows of the same few hub
// vertices for millions of leaves.  Here
//   * most leaves lie one or two links below an inner node (h, p) and are
//     credited with it: what the closed children of a node give a vertex is
//     x^h (1+x)^p (A0 + A1 x + A2 x^2 + A3 x^3) with small integers A that
//     follow from bit counts, so a node costs one pass over its members
//     whatever the number of its leaves (for a pivot vertex of the path the
//     same A over x^(h+1) (1+x)^(p-1));
//   * a warp adds these polynomials to a table of its root's members in
//     shared memory, one lane per member and so without atomics, for sizes up
//     to LocalWork's window; sums stay below C(128, 11) < 2^64.  The table
//     goes to the caller's table once per root.  In an edge table it is the
//     rows of the root's own edges; member pairs are credited per node.
//   * sizes above the window (cliques of more than 8 to 12 vertices) and edge
//     rows go to the caller's table with carry-propagating atomics.
// Dense roots are not walked where they are gathered: the warp stores the
// rows, and a second launch walks each in parts that deal out the hold
// children along the root's pivot chain, so one such root does not occupy one
// warp after all others have finished.
// What bounds it: load latency in the gathers (the one-word one issues on 61 %
// of the slots), dependent instructions and instruction fetch in the parts of
// dense roots, at 11 to 32 warps per SM (the table takes 2 to 8 KB of shared
// memory per warp).  Start -> now, whole
// calls: per-vertex, 500k vertices, 8.25M edges, k <= 40: 23.6 -> 3.9 ms;
// 90k vertices, k <= 5: 4.3 -> 0.85 ms; per-edge, 2M edges, k <= 12: 5.3 ->
// 2.4 ms; 56k edges, k <= 22: 0.56 -> 0.23 ms.
#pragma once

#include "walk.cuh"

namespace pvt {

// A root is walked in parts from LOCAL_HEAVY_EDGES member edges on, in one
// part for LOCAL_PART_EDGES edges, more when they are dense: the tree grows
// with the edges of a sparse member graph and far faster in a dense one, and
// each part walks the root's pivot chain again.
// A near-clique's tree is small: at most LOCAL_FEW_MISSING edges short of one,
// a root is not split.  Measured on per-vertex tables of 500k vertices (3.96 ms)
// and per-edge tables of 56k edges (0.22 ms) and of dense groups (2.38 ms): parts
// of 96 edges 4.35, 0.20 and 2.54 ms, of 384 edges 3.76, 0.23 and 2.52; a density
// factor of 4 in place of 16 3.91, 0.25 and 2.65, of 64 4.39, 0.20 and 2.64.  The
// first edge count (24 to 96), the most parts (16 to 256) and the edges short of
// a clique (0 to 32) made no difference beyond that of two runs.
constexpr unsigned LOCAL_HEAVY_EDGES = 48, LOCAL_PART_EDGES = 192, LOCAL_MAX_PARTS = 64, LOCAL_FEW_MISSING = 8;
__device__ __forceinline__ unsigned local_parts(unsigned edges, int d)
{
    const float density = 2.0f * (float)edges / ((float)d * (float)(d - 1));
    return min((unsigned)((float)edges * (1.0f + 16.0f * density * density) / LOCAL_PART_EDGES) + 1u, LOCAL_MAX_PARTS);
}
constexpr int LOCAL_BINOM = 24;              // block table of C(a, b), a < LOCAL_BINOM, in 32 bits

template <int NW>
struct LocalWork {
    static constexpr int D = 32 * NW;
    static constexpr int RS = (NW & 1) ? NW : NW + 1;
    static constexpr int FILTER_LOG = 12;
    static constexpr bool GSTACK = NW > 2;
    static constexpr int FW = 3 * NW;    // stack frame: label, hold members, pivot members of the path
    static constexpr int WINDOW = NW == 1 ? 12 : (NW == 2 ? 10 : 8);  // largest size in the table
    int64_t rs[D];
    uint32_t ids[D];
    uint32_t off[D + 1];
    uint32_t adj[D * RS];
    union {
        struct {
            uint32_t filter[(1 << FILTER_LOG) / 32];
            uint2 hits[64];
        };
        uint32_t stk_s[GSTACK ? 1 : (D + 1) * FW];
    };
    uint8_t mem[D];    // members of a clique leaf
    // walk of a label of at most 32 members below a wider root (NW > 1): its
    // members (relabel_rows), rows and stack
    alignas(8) uint16_t cm[NW > 1 ? 32 : 4];
    uint32_t crow[NW > 1 ? 32 : 1];
    uint32_t cstk[NW > 1 ? 33 * 3 : 1];
    uint32_t *gstk;
    uint32_t *etab;    // edge ids of member pairs, D x D
    __device__ __forceinline__ uint32_t *stk() { return GSTACK ? gstk : stk_s; }
};

// Dense roots between the two launches.
struct LocalHeavy {
    uint32_t *rows;     // [cap][D][NW] adjacency rows
    uint32_t *etab;     // [cap][D][D] edge ids (per-edge counts)
    uint32_t *root;     // [cap] vertex
    uint2 *items;       // [cap * LOCAL_MAX_PARTS] (slot, part | parts << 16)
    unsigned *count;    // [0] slots, [1] items taken for writing, [2] queue head of the second launch
    unsigned cap;
};

// a[0..W) += n * b[0..W), carries propagated (n < 2^32).
__device__ __forceinline__ void atomic_add_scaled(unsigned long long *a, const unsigned long long *__restrict__ b,
                                                  unsigned n, int W, unsigned *err)
{
    unsigned long long c = 0;
    for (int j = 0; j < W; ++j) {
        const unsigned long long bj = b[j];
        if (bj == 0 && c == 0) continue;
        const unsigned long long lo = bj * n, add = lo + c;
        const unsigned long long up = __umul64hi(bj, n) + (add < lo ? 1ull : 0ull);
        const unsigned long long old = add ? atomicAdd(a + j, add) : 0ull;
        c = up + (old + add < old ? 1ull : 0ull);
    }
    if (c) atomicOr(err, DERR_OVERFLOW);
}

// Coefficients A0..A3 of one member's share of a node's closed leaves.
struct Share {
    unsigned a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    __device__ __forceinline__ bool any() const { return (a0 | a1 | a2 | a3) != 0; }
};

// Walk of one root (or part q of Q of it) and its credits.  tab[k * D + m]:
// count of size k <= kt of member m, zero on entry and on return.
template <int NW, int MODE>
struct LocalWalk {
    using Work = LocalWork<NW>;
    static constexpr int D = Work::D, RS = Work::RS, FW = Work::FW;
    Work &Wk;
    unsigned long long *tab;
    const uint32_t *bin;     // block table of small binomials
    const CountArgs &A;
    const int lane, kt;
    const uint32_t r;
    const int64_t rbeg;
    const int d;
    unsigned long long acc = 0;  // lane k: the root's own count of size k <= kt (per-vertex)
    int ktop = 0;                // largest size in the table

    __device__ __forceinline__ unsigned long long *cell(int m) const
    {
        const size_t row = MODE == MODE_VERTEX ? (size_t)Wk.ids[m] : (size_t)A.oeid[rbeg + m];
        return A.out + row * (A.kmax + 1) * A.W;
    }
    __device__ __forceinline__ unsigned long long binom64(int a, int b) const
    {
        if (b < 0 || b > a) return 0ull;
        return a < LOCAL_BINOM ? bin[a * (a + 1) / 2 + b] : __ldg(binom_at(A.B, a, b, A.Bw));
    }
    // count of size k += v.  No count of a size up to ksafe passes 2^64: its
    // low word cannot wrap, and the addition need not come back.
    __device__ __forceinline__ void add_count(unsigned long long *row, int k, unsigned long long v) const
    {
        if (k <= A.ksafe) atomicAdd(row + (size_t)k * A.W, v);
        else atomic_add_u64_carry(row + (size_t)k * A.W, v, A.W, A.err);
    }
    // coefficient of x^e in (1+x)^a (a0 + a1 x + a2 x^2 + a3 x^3), modulo 2^64
    __device__ __forceinline__ unsigned long long coeff(int a, int e, const Share &s) const
    {
        unsigned long long v = 0;
        if (s.a0) v += s.a0 * binom64(a, e);
        if (s.a1) v += s.a1 * binom64(a, e - 1);
        if (s.a2) v += s.a2 * binom64(a, e - 2);
        if (s.a3) v += s.a3 * binom64(a, e - 3);
        return v;
    }
    // row += x^h (1+x)^a (share), sizes from k0 to kmax, multi-word
    __device__ __noinline__ void add_high(unsigned long long *row, int h, int a, const Share &s, int k0) const
    {
        const unsigned n[4] = {s.a0, s.a1, s.a2, s.a3};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (!n[i]) continue;
            for (int k = max(k0, h + i); k <= min(A.kmax, h + i + a); ++k)
                atomic_add_scaled(row + (size_t)k * A.W, binom_at(A.B, a, k - h - i, A.Bw), n[i], A.W, A.err);
        }
    }

    // Credit every member: H the hold and Pm the pivot members of the path,
    // with share `path` over x^h (1+x)^p (the root is one more hold vertex);
    // own[j]: the share of this lane's member of word j outside the path.
    // top: degree of the path's share polynomial (no other share's is larger).
    __device__ __forceinline__ void credit(int h, int p, const uint32_t *H, const uint32_t *Pm, const Share &path,
                                           const Share *own, int top)
    {
        const int kmost = min(A.kmax, h + p + top);
        const int kin = min(kt, kmost);
        ktop = max(ktop, kin);
        const bool small = p < LOCAL_BINOM;
#pragma unroll
        for (int j = 0; j < NW; ++j) {
            const bool inH = (H[j] >> lane) & 1u, inP = (Pm[j] >> lane) & 1u;
            const Share s = inH || inP ? path : own[j];
            const bool has = s.any();
            if (!__any_sync(FULL, has)) continue;
            const int hl = inP ? h + 1 : h, pl = inP ? p - 1 : p;
            if (small) {
                // C(p, e) < 2^21 for p < LOCAL_BINOM and shares below 2^9: 32 bits hold each sum
                const uint32_t *row = bin + (inP ? pl * (pl + 1) / 2 : p * (p + 1) / 2);
                uint32_t c1 = 0, c2 = 0, c3 = 0;
                for (int e = 0; h + e <= kin; ++e) {
                    const uint32_t c0 = e <= pl ? row[e] : 0u;
                    const uint32_t v = s.a0 * c0 + s.a1 * c1 + s.a2 * c2 + s.a3 * c3;
                    if (has && v && hl + e <= kin) tab[(hl + e) * D + j * 32 + lane] += v;
                    c3 = c2;
                    c2 = c1;
                    c1 = c0;
                }
            } else if (has) {
                for (int k = hl; k <= min(kin, hl + pl + 3); ++k)
                    tab[k * D + j * 32 + lane] += coeff(pl, k - hl, s);
            }
            if (kmost > kt && has) add_high(cell(j * 32 + lane), hl, pl, s, kt + 1);
        }
        if (MODE == MODE_VERTEX) {
            if (lane >= h && lane <= kin) acc += coeff(p, lane - h, path);
            if (kmost > kt) high_root(h, p, path);
        }
        __syncwarp();
    }

    // row of edge e += x^h (1+x)^a (share)
    __device__ __noinline__ void add_edge(uint32_t e, int h, int a, const Share &s) const
    {
        unsigned long long *row = A.out + (size_t)e * (A.kmax + 1) * A.W;
        if (a > 50) {
            add_high(row, h, a, s, 0);
            return;
        }
        // C(a, b) < 2^47 and shares below 2^9: 64 bits hold each sum
        const int k1 = min(A.kmax, h + a + (s.a3 ? 3 : (s.a2 ? 2 : (s.a1 ? 1 : 0))));
        const bool small = a < LOCAL_BINOM;
        const uint32_t *brow = bin + a * (a + 1) / 2;
        unsigned long long c1 = 0, c2 = 0, c3 = 0;
        for (int k = h; k <= k1; ++k) {
            const unsigned long long c0 = k - h > a ? 0ull : (small ? brow[k - h] : binom64(a, k - h));
            const unsigned long long v = s.a0 * c0 + s.a1 * c1 + s.a2 * c2 + s.a3 * c3;
            if (v) add_count(row, k, v);
            c3 = c2;
            c2 = c1;
            c1 = c0;
        }
    }
    __device__ __forceinline__ void add_edge(uint32_t e, int h, int a) const
    {
        Share one;
        one.a0 = 1;
        add_edge(e, h, a, one);
    }
    // Credit every pair of a clique leaf's members, hold H and pivot Pm, dealt
    // to the lanes pair by pair.
    __device__ __forceinline__ void credit_clique_pairs(int h, int p, const uint32_t *H, const uint32_t *Pm)
    {
        int nh = 0, np = 0, L = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) nh += __popc(H[w]);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const uint32_t low = (1u << lane) - 1u;
            if ((H[w] >> lane) & 1u) Wk.mem[L + __popc(H[w] & low)] = (uint8_t)(w * 32 + lane);
            if ((Pm[w] >> lane) & 1u) Wk.mem[nh + np + __popc(Pm[w] & low)] = (uint8_t)(w * 32 + lane);
            L += __popc(H[w]);
            np += __popc(Pm[w]);
        }
        L = nh + np;
        __syncwarp();
        // pair t: a < b < L, numbered column by column (b(b-1)/2 + a)
        for (int t = lane; t < L * (L - 1) / 2; t += 32) {
            int b = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)t)) * 0.5f);
            while (b * (b - 1) / 2 > t) --b;
            while ((b + 1) * b / 2 <= t) ++b;
            const int a = t - b * (b - 1) / 2;
            const int n = (a >= nh) + (b >= nh);
            add_edge(Wk.etab[(size_t)Wk.mem[a] * D + Wk.mem[b]], h + n, p - n);
        }
    }

    // Credit the member pairs that contain a path member (arguments as
    // credit): a pair's polynomial loses one (1+x) and gains one x for each of
    // its pivot members.
    __device__ __forceinline__ void credit_pairs(int h, int p, const uint32_t *H, const uint32_t *Pm,
                                                 const Share &path, const Share *own)
    {
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            for (uint32_t us = H[w] | Pm[w]; us; us &= us - 1) {
                const int b = __ffs(us) - 1, u = w * 32 + b;
                const int up = (Pm[w] >> b) & 1u;
                const uint32_t *eu = Wk.etab + (size_t)u * D;
#pragma unroll
                for (int j = 0; j < NW; ++j) {
                    const int m = j * 32 + lane;
                    const bool inH = (H[j] >> lane) & 1u, inP = (Pm[j] >> lane) & 1u;
                    const Share s = inH || inP ? path : own[j];
                    if ((inH || inP) && m <= u) continue;
                    if (!s.any()) continue;
                    const int np = up + (inP ? 1 : 0);
                    add_edge(eu[m], h + np, p - np, s);
                }
            }
        }
    }

    // The subtree of a label S of s <= 32 members below a wider root, entered
    // with (h, p) and the path members H, P (the prefix): relabelled to
    // one-word rows, one member per lane.  A node costs a few one-word
    // operations instead of NW times as many, and the prefix's share of it is
    // summed, one size per lane, and credited once at the end.
    __device__ void run_small(const uint32_t (&S)[NW], const uint32_t (&H)[NW], const uint32_t (&P)[NW], int s, int h,
                              int p, WalkCounters &wc)
    {
        uint32_t cw = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w)
            if (lane == w) cw = S[w];
        int sz = 0;
        const uint32_t r1 = relabel_rows<NW, RS>(Wk.adj, Wk.cm, lane, cw, sz);
        const int mk = lane < s ? (int)(Wk.cm[lane] ^ 31) : 0;  // this lane's member
        Wk.crow[lane] = r1;
        __syncwarp();
        auto adjacent = [&](int a, int b) { return (Wk.crow[a] >> b) & 1u; };
        auto member = [&](int a) { return (int)(Wk.cm[a] ^ 31); };
        const uint32_t low = (1u << lane) - 1u;
        uint32_t S1 = s >= 32 ? FULL : (1u << s) - 1u, H1 = 0, P1 = 0;
        int hh = h, pp = p, top = 0;
        unsigned long long pre = 0;  // lane k: what a hold member of the prefix gains at size k <= kt
        int kpre = 0;
        for (;;) {
            const int s1 = __popc(S1);
            const bool in = (S1 >> lane) & 1u;
            const uint32_t c = in ? (uint32_t)__popc(r1 & S1) : 0u;
            const uint32_t best = __reduce_max_sync(FULL, in ? ((c + 1u) << 5 | (31u - (uint32_t)lane)) : 0u);
            const uint32_t dsum = __reduce_add_sync(FULL, c);
            wc.nodes++;
            wc.words += (unsigned)s1;
            bool closed = true;
            Share path, own;
            uint32_t PX = P1, N = 0;
            int pc = pp, piv = 0;
            if (dsum == (uint32_t)s1 * (uint32_t)(s1 - 1)) {
                wc.leaves++;
                path.a0 = 1;
                pc = pp + s1;
                PX = P1 | S1;
            } else {
                piv = 31 - (int)(best & 31u);
                const uint32_t a0 = __shfl_sync(FULL, r1, piv);
                N = a0 & S1;
                const uint32_t R = hh + 1 > A.kmax ? 0u : S1 & ~a0 & ~(1u << piv);
                const bool inR = (R >> lane) & 1u;
                const uint32_t child = inR ? r1 & S1 & ~(R & low) : 0u;
                const int cs = __popc(child);
                const int a = child ? __ffs(child) - 1 : 0, b = child ? 31 - __clz(child) : 0;
                const bool pair = inR && cs == 2 && adjacent(a, b);
                const unsigned b1 = __ballot_sync(FULL, inR && cs == 1), b2 = __ballot_sync(FULL, pair);
                const unsigned bn = __ballot_sync(FULL, inR && cs == 2 && !pair);
                const unsigned bp = __ballot_sync(FULL, inR && cs > 2);
                const unsigned n1 = __popc(b1), n2 = __popc(b2), nn = __popc(bn);
                const unsigned n0 = __popc(R & ~(b1 | b2 | bn | bp));
                if (inR && cs <= 2) {
                    own.a1 = 1;
                    own.a2 = cs;
                    own.a3 = pair;
                    if (MODE == MODE_EDGE && cs) {
                        const uint32_t *em = Wk.etab + (size_t)mk * D;
                        const int ma = member(a), mb = member(b);
                        add_edge(em[ma], hh + 2, pair ? pp + 1 : pp);
                        if (cs == 2) add_edge(em[mb], hh + 2, pair ? pp + 1 : pp);
                        if (pair) add_edge(Wk.etab[(size_t)ma * D + mb], hh + 3, pp);
                    }
                }
                if (top + __popc(bp) > 33) {
                    if (lane == 0) atomicOr(A.err, DERR_STACK);
                    return;
                }
                __syncwarp();
                if ((bp >> lane) & 1u) {
                    uint32_t *f = Wk.cstk + (top + __popc(bp & low)) * 3;
                    f[0] = child;
                    f[1] = H1 | 1u << lane;
                    f[2] = P1;
                }
                top += __popc(bp);
                const unsigned held = hh + 2 <= A.kmax ? nn : 0u;
                wc.nodes += n0 + n1 + n2 + 2 * nn + held;
                wc.leaves += n0 + n1 + n2 + nn + held;
                wc.words += n1 + 2 * (n2 + nn);
                path.a1 = n0 + n1 + n2 + nn;
                path.a2 = n1 + 2 * (n2 + nn);
                path.a3 = n2;
                if (in) {
                    const uint32_t lim = r1 & (inR ? low : FULL);
                    const unsigned t1 = __popc(lim & (b1 | bn)), t2 = __popc(lim & b2);
                    own.a2 += t1 + t2;
                    own.a3 += t2;
                }
                const int ps = __popc(N);
                if (ps <= 2) {
                    const int na = N ? __ffs(N) - 1 : 0, nb = N ? 31 - __clz(N) : 0;
                    const bool adjp = ps == 2 && adjacent(na, nb);
                    const bool split = ps == 2 && !adjp;
                    const bool hold = split && hh + 1 <= A.kmax;
                    wc.nodes += 1 + split + hold;
                    wc.leaves += 1 + hold;
                    wc.words += (unsigned)ps;
                    path.a0 += 1;
                    path.a1 += 1 + (unsigned)ps;
                    path.a2 += ps == 0 ? 0u : (ps == 1 ? 1u : (adjp ? 3u : 2u));
                    path.a3 += adjp;
                    if (lane == piv) {
                        own.a1 += 1;
                        own.a2 += (unsigned)ps;
                        own.a3 += adjp;
                    } else if ((ps >= 1 && lane == na) || (ps == 2 && lane == nb)) {
                        own.a1 += 1;
                        own.a2 += adjp ? 2u : 1u;
                        own.a3 += adjp;
                    }
                    if (MODE == MODE_EDGE && ps) {
                        int x = -1, y = 0;
                        if (lane == 0) { x = piv; y = na; }
                        if (lane == 1 && ps == 2) { x = piv; y = nb; }
                        if (lane == 2 && adjp) { x = na; y = nb; }
                        if (x >= 0) add_edge(Wk.etab[(size_t)member(x) * D + member(y)], hh + 2, adjp ? pp + 1 : pp);
                    }
                } else {
                    closed = false;
                }
            }
            if (path.any()) {
                const int kmost = min(A.kmax, hh + pc + (path.a3 ? 3 : (path.a2 ? 2 : (path.a1 ? 1 : 0))));
                const int kin = min(kt, kmost);
                kpre = max(kpre, kin);
                // this lane's member
                const bool inH = (H1 >> lane) & 1u, inP = (PX >> lane) & 1u;
                const Share sh = inH || inP ? path : own;
                const bool has = sh.any();
                const int hl = inP ? hh + 1 : hh, pl = inP ? pc - 1 : pc;
                if (pc < LOCAL_BINOM) {
                    const uint32_t *row = bin + pl * (pl + 1) / 2;
                    uint32_t c1 = 0, c2 = 0, c3 = 0;
                    for (int e = 0; hh + e <= kin; ++e) {
                        const uint32_t c0 = e <= pl ? row[e] : 0u;
                        const uint32_t v = sh.a0 * c0 + sh.a1 * c1 + sh.a2 * c2 + sh.a3 * c3;
                        if (has && v && hl + e <= kin) tab[(hl + e) * D + mk] += v;
                        c3 = c2;
                        c2 = c1;
                        c1 = c0;
                    }
                } else if (has) {
                    for (int k = hl; k <= min(kin, hl + pl + 3); ++k) tab[k * D + mk] += coeff(pl, k - hl, sh);
                }
                if (lane >= hh && lane <= kin) pre += coeff(pc, lane - hh, path);
                if (kmost > kt) {  // sizes above the table: everyone at once
                    if (has) add_high(cell(mk), hl, pl, sh, kt + 1);
                    high_prefix(hh, pc, H, P, path);
                }
                if (MODE == MODE_EDGE) {
                    // pairs of this lane's member with a path member of the label
                    for (uint32_t us = H1 | PX; us; us &= us - 1) {
                        const int u = __ffs(us) - 1;
                        if (has && !((inH || inP) && lane <= u)) {
                            const int np = (int)((PX >> u) & 1u) + (inP ? 1 : 0);
                            add_edge(Wk.etab[(size_t)member(u) * D + mk], hh + np, pc - np, sh);
                        }
                    }
                    // pairs with and inside the prefix
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        for (uint32_t us = H[w] | P[w]; us; us &= us - 1) {
                            const int b = __ffs(us) - 1, u = w * 32 + b;
                            const int up = (P[w] >> b) & 1u;
                            const uint32_t *eu = Wk.etab + (size_t)u * D;
                            if (has) add_edge(eu[mk], hh + up + (inP ? 1 : 0), pc - up - (inP ? 1 : 0), sh);
#pragma unroll
                            for (int j = 0; j < NW; ++j) {
                                const int m = j * 32 + lane, mp = (P[j] >> lane) & 1u;
                                if (m > u && (((H[j] | P[j]) >> lane) & 1u)) add_edge(eu[m], hh + up + mp, pc - up - mp, path);
                            }
                        }
                    }
                }
            }
            __syncwarp();
            if (!closed) {
                S1 = N;
                P1 |= 1u << piv;
                pp += 1;
                continue;
            }
            if (top == 0) break;
            --top;
            S1 = Wk.cstk[top * 3];
            H1 = Wk.cstk[top * 3 + 1];
            P1 = Wk.cstk[top * 3 + 2];
            hh = h + __popc(H1);
            pp = p + __popc(P1);
        }
        // ---- the prefix: hold members gain pre, pivot members x / (1+x) of it
        // (every leaf here has them as pivots, so the division is exact)
        unsigned long long div = 0;
        for (int k = 1; k <= kpre; ++k) {
            const unsigned long long x = __shfl_sync(FULL, pre, k - 1), y = __shfl_sync(FULL, div, k - 1);
            if (lane == k) div = x - y;
        }
#pragma unroll
        for (int w = 0; w < NW; ++w)
            for (uint32_t us = H[w] | P[w]; us; us &= us - 1) {
                const int b = __ffs(us) - 1;
                if (lane <= kpre) tab[lane * D + w * 32 + b] += (P[w] >> b) & 1u ? div : pre;
            }
        acc += pre;
        ktop = max(ktop, kpre);
        __syncwarp();
    }
    // A node's share of the sizes above the table for the prefix members and
    // the root (as credit's).
    __device__ __noinline__ void high_prefix(int h, int p, const uint32_t *H, const uint32_t *Pm, const Share &path) const
    {
#pragma unroll
        for (int j = 0; j < NW; ++j) {
            const bool inP = (Pm[j] >> lane) & 1u;
            if (((H[j] | Pm[j]) >> lane) & 1u) add_high(cell(j * 32 + lane), inP ? h + 1 : h, inP ? p - 1 : p, path, kt + 1);
        }
        high_root(h, p, path);
    }
    // ... for the root, one size per lane (per-vertex)
    __device__ __forceinline__ void high_root(int h, int p, const Share &path) const
    {
        if (MODE != MODE_VERTEX) return;
        unsigned long long *row = A.out + (size_t)r * (A.kmax + 1) * A.W;
        const unsigned n[4] = {path.a0, path.a1, path.a2, path.a3};
        for (int k = kt + 1 + lane; k <= min(A.kmax, h + p + 3); k += 32)
            for (int i = 0; i < 4; ++i)
                if (n[i] && k - h - i >= 0 && k - h - i <= p)
                    atomic_add_scaled(row + (size_t)k * A.W, binom_at(A.B, p, k - h - i, A.Bw), n[i], A.W, A.err);
    }

    __device__ void run(unsigned q, unsigned Q, WalkCounters &wc)
    {
        uint32_t row[NW][NW];  // this lane's rows
#pragma unroll
        for (int j = 0; j < NW; ++j)
#pragma unroll
            for (int w = 0; w < NW; ++w) row[j][w] = j * 32 + lane < d ? Wk.adj[(j * 32 + lane) * RS + w] : 0u;
        auto adjacent = [&](int a, int b) { return (Wk.adj[a * RS + (b >> 5)] >> (b & 31)) & 1u; };
        const uint32_t low = (1u << lane) - 1u;
        uint32_t S[NW], H[NW], P[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int bits = d - 32 * w;
            S[w] = bits >= 32 ? FULL : (bits <= 0 ? 0u : ((1u << bits) - 1u));
            H[w] = P[w] = 0;
        }
        int h = 1, p = 0, top = 0;
        bool chain = true;      // on the root's pivot chain, which every part walks
        unsigned dealt = 0;     // hold children met along it
        uint32_t *stk = Wk.stk();
        auto pop = [&]() {
            --top;
            const uint32_t *f = stk + (size_t)top * FW;
            h = 1;
            p = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                S[w] = f[w];
                H[w] = f[NW + w];
                P[w] = f[2 * NW + w];
                h += __popc(H[w]);
                p += __popc(P[w]);
            }
        };
        for (;;) {
            const bool mine = !chain || q == 0;  // the chain's own leaves are part 0's
            int s = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) s += __popc(S[w]);
            if (NW > 1 && s <= 32 && (!chain || Q == 1)) {
                run_small(S, H, P, s, h, p, wc);
                chain = false;
                if (top == 0) break;
                pop();
                continue;
            }
            uint32_t best = 0, dsum = 0;
#pragma unroll
            for (int j = 0; j < NW; ++j) {
                if ((S[j] >> lane) & 1u) {
                    uint32_t c = 0;
#pragma unroll
                    for (int w = 0; w < NW; ++w) c += __popc(row[j][w] & S[w]);
                    best = max(best, ((c + 1u) << 10) | (1023u - (uint32_t)(j * 32 + lane)));
                    dsum += c;
                }
            }
            best = __reduce_max_sync(FULL, best);
            dsum = __reduce_add_sync(FULL, dsum);
            if (mine) {
                wc.nodes++;
                wc.words += (unsigned long long)s * (unsigned)((s + 31) >> 5);
            }
            bool closed = true;
            // what the node credits: share `path` over x^h (1+x)^pc with the pivot
            // members PX of the path, own for the members outside it
            Share path, own[NW];
            uint32_t PX[NW];
            int pc = p, piv = 0;
            uint32_t N[NW];  // the pivot's neighbours in S
            if (dsum == (uint32_t)s * (uint32_t)(s - 1)) {
                // S is a clique: one leaf with all of S as pivot vertices
                if (mine) {
                    wc.leaves++;
                    path.a0 = 1;
                }
                pc = p + s;
#pragma unroll
                for (int w = 0; w < NW; ++w) PX[w] = P[w] | S[w];
            } else {
                piv = 1023 - (int)(best & 1023u);
                uint32_t R[NW];  // non-neighbours of the pivot
                int nR = 0, ps = 0, na = 0, nb = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const uint32_t a = Wk.adj[piv * RS + w];
                    PX[w] = P[w];
                    N[w] = a & S[w];
                    R[w] = S[w] & ~a;
                    if (w == (piv >> 5)) R[w] &= ~(1u << (piv & 31));
                    if (h + 1 > A.kmax) R[w] = 0;  // no further hold link
                    nR += __popc(R[w]);
                    if (N[w]) {
                        if (ps == 0) na = w * 32 + __ffs(N[w]) - 1;
                        nb = w * 32 + 31 - __clz(N[w]);
                    }
                    ps += __popc(N[w]);
                }
                // ---- hold children: member m = j*32+lane of R holds the label
                // N(S, m) without the earlier members of R
                uint32_t M1[NW], M2[NW];  // holders of a single member or a non-adjacent pair; of an adjacent pair
                unsigned n0 = 0, n1 = 0, n2 = 0, nn = 0;
                int fresh = 0;            // children pushed
                if (top + nR > D + 1) {
                    if (lane == 0) atomicOr(A.err, DERR_STACK);
                    return;
                }
                __syncwarp();
                uint32_t M[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) M[w] = S[w];
#pragma unroll
                for (int j = 0; j < NW; ++j) {
                    M1[j] = M2[j] = 0;
                    if (R[j] == 0) continue;
                    const bool inR = (R[j] >> lane) & 1u;
                    uint32_t c[NW];
                    int cs = 0;
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        c[w] = inR ? row[j][w] & M[w] & (w == j ? ~(R[j] & low) : FULL) : 0u;
                        cs += __popc(c[w]);
                    }
                    bool pair = false;
                    int a = 0, b = 0;
                    if (inR && (cs == 1 || cs == 2)) {
#pragma unroll
                        for (int w = NW - 1; w >= 0; --w)
                            if (c[w]) {
                                a = w * 32 + __ffs(c[w]) - 1;
                                b = max(b, w * 32 + 31 - __clz(c[w]));
                            }
                        pair = cs == 2 && adjacent(a, b);
                    }
                    const unsigned b0 = __ballot_sync(FULL, inR && cs == 0), b1 = __ballot_sync(FULL, inR && cs == 1);
                    const unsigned b2 = __ballot_sync(FULL, inR && cs == 2 && pair);
                    const unsigned bn = __ballot_sync(FULL, inR && cs == 2 && !pair);
                    n0 += __popc(b0);
                    n1 += __popc(b1);
                    n2 += __popc(b2);
                    nn += __popc(bn);
                    M1[j] = b1 | bn;
                    M2[j] = b2;
                    if (inR && cs <= 2) {
                        own[j].a1 = 1;
                        own[j].a2 = cs;         // x, x(1+x), x(1+x)^2 or x(1+x) + x^2
                        own[j].a3 = pair;
                        if (MODE == MODE_EDGE && mine && cs) {
                            // pairs of the held member and its label
                            const int m = j * 32 + lane;
                            const uint32_t *em = Wk.etab + (size_t)m * D;
                            const uint32_t ea = em[a], eb = cs == 2 ? em[b] : 0u;
                            const uint32_t eab = pair ? Wk.etab[(size_t)a * D + b] : 0u;
                            add_edge(ea, h + 2, pair ? p + 1 : p);
                            if (cs == 2) add_edge(eb, h + 2, pair ? p + 1 : p);
                            if (pair) add_edge(eab, h + 3, p);
                        }
                    }
                    // the others to the stack (this part's share of them)
                    const unsigned bp = __ballot_sync(FULL, inR && cs > 2);
                    bool push = inR && cs > 2;
                    if (chain) {
                        push = push && (dealt + __popc(bp & low)) % Q == q;
                        dealt += __popc(bp);
                    }
                    const unsigned bq = __ballot_sync(FULL, push);
                    if (push) {
                        uint32_t *f = stk + (size_t)(top + fresh + __popc(bq & low)) * FW;
#pragma unroll
                        for (int w = 0; w < NW; ++w) {
                            f[w] = c[w];
                            f[NW + w] = H[w] | (w == j ? 1u << lane : 0u);
                            f[2 * NW + w] = P[w];
                        }
                    }
                    fresh += __popc(bq);
#pragma unroll
                    for (int w = 0; w < NW; ++w)
                        if (w == j) M[w] &= ~R[j];
                }
                top += fresh;
                if (mine) {
                    const unsigned held = h + 2 <= A.kmax ? nn : 0u;
                    wc.nodes += n0 + n1 + n2 + 2 * nn + held;
                    wc.leaves += n0 + n1 + n2 + nn + held;
                    wc.words += n1 + 2 * (n2 + nn);
                    path.a1 = n0 + n1 + n2 + nn;
                    path.a2 = n1 + 2 * (n2 + nn);
                    path.a3 = n2;
                    // members of the closed labels: x^2 for a single member or
                    // either of a non-adjacent pair, x^2 (1+x) in an adjacent pair
#pragma unroll
                    for (int j = 0; j < NW; ++j) {
                        if (!((S[j] >> lane) & 1u)) continue;
                        const bool inR = (R[j] >> lane) & 1u;
                        unsigned t1 = 0, t2 = 0;
#pragma unroll
                        for (int w = 0; w < NW; ++w) {
                            const uint32_t lim = row[j][w] & (inR ? (w < j ? FULL : (w == j ? low : 0u)) : FULL);
                            t1 += __popc(lim & M1[w]);
                            t2 += __popc(lim & M2[w]);
                        }
                        own[j].a2 += t1 + t2;
                        own[j].a3 += t2;
                    }
                }
                // ---- the pivot child N: closed here if it has at most two members
                const bool adjp = ps == 2 && adjacent(na, nb);
                if (ps <= 2) {
                    if (mine) {
                        const bool split = ps == 2 && !adjp;
                        const bool held = split && h + 1 <= A.kmax;
                        wc.nodes += 1 + split + held;
                        wc.leaves += 1 + held;
                        wc.words += (unsigned)ps;
                        // path: (1+x)^(1+ps), or (1+x)^2 + x(1+x)
                        path.a0 += 1;
                        path.a1 += 1 + (unsigned)ps;
                        path.a2 += ps == 0 ? 0u : (ps == 1 ? 1u : (adjp ? 3u : 2u));
                        path.a3 += adjp;
#pragma unroll
                        for (int j = 0; j < NW; ++j) {
                            const int m = j * 32 + lane;
                            if (m == piv) {  // x(1+x)^ps, or x(1+x) + x^2
                                own[j].a1 += 1;
                                own[j].a2 += (unsigned)ps;
                                own[j].a3 += adjp;
                            } else if ((ps >= 1 && m == na) || (ps == 2 && m == nb)) {  // x(1+x), or x(1+x)^2 in a pair
                                own[j].a1 += 1;
                                own[j].a2 += adjp ? 2u : 1u;
                                own[j].a3 += adjp;
                            }
                        }
                        if (MODE == MODE_EDGE && ps) {
                            const int a2 = adjp ? p + 1 : p;
                            int x = -1, y = 0;
                            if (lane == 0) { x = piv; y = na; }
                            if (lane == 1 && ps == 2) { x = piv; y = nb; }
                            if (lane == 2 && adjp) { x = na; y = nb; }
                            if (x >= 0) add_edge(Wk.etab[(size_t)x * D + y], h + 2, a2);
                        }
                    }
                } else {
                    closed = false;
                }
            }
            if (path.any()) {
                credit(h, pc, H, PX, path, own, path.a3 ? 3 : (path.a2 ? 2 : (path.a1 ? 1 : 0)));
                if (MODE == MODE_EDGE) {
                    if (pc > p) credit_clique_pairs(h, pc, H, PX);
                    else credit_pairs(h, pc, H, PX, path, own);
                }
            }
            __syncwarp();
            if (!closed) {
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    S[w] = N[w];
                    if (w == (piv >> 5)) P[w] |= 1u << (piv & 31);
                }
                p += 1;
                continue;
            }
            chain = false;
            if (top == 0) break;
            pop();
        }
        __syncwarp();
        // ---- the root's table to the caller's
#pragma unroll
        for (int j = 0; j < NW; ++j) {
            const int m = j * 32 + lane;
            if (m >= d) continue;
            unsigned long long *out = cell(m);
            for (int k = 1; k <= ktop; ++k) {
                const unsigned long long v = tab[k * D + m];
                if (!v) continue;
                add_count(out, k, v);
                tab[k * D + m] = 0;
            }
        }
        if (MODE == MODE_VERTEX && acc) add_count(A.out + (size_t)r * (A.kmax + 1) * A.W, lane, acc);
        __syncwarp();
    }
};

// Per-warp shared memory: the work area, then the table.
template <int NW>
__host__ __device__ constexpr size_t local_warp_bytes(int kt)
{
    return sizeof(LocalWork<NW>) + (size_t)(kt + 1) * 32 * NW * sizeof(unsigned long long);
}
template <int NW>
constexpr int local_wpb()
{
    return NW <= 2 ? 8 : 4;
}
// resident blocks the kernels' registers are held to
template <int NW>
constexpr int local_blocks()
{
    return NW == 1 ? 4 : (NW == 2 ? 3 : 5);
}

template <int NW>
__device__ __forceinline__ unsigned long long *local_set_up(unsigned char *smem, uint32_t *bin, const CountArgs &A,
                                                            int kt, int amax, int lane, int wid)
{
    for (int i = threadIdx.x; i < LOCAL_BINOM * (LOCAL_BINOM + 1) / 2; i += blockDim.x) {
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= i) ++a;
        bin[i] = a <= amax ? (uint32_t)*binom_at(A.B, a, i - a * (a + 1) / 2, A.Bw) : 0u;
    }
    unsigned long long *tab = reinterpret_cast<unsigned long long *>(smem + (size_t)wid * local_warp_bytes<NW>(kt) +
                                                                     sizeof(LocalWork<NW>));
    for (int i = lane; i < (kt + 1) * 32 * NW; i += 32) tab[i] = 0;
    __syncthreads();
    return tab;
}

// First launch: every root of the class, by persistent warps; dense roots go
// to hv (split) instead of being walked.
template <int NW, int MODE>
__global__ void __launch_bounds__(32 * local_wpb<NW>(), local_blocks<NW>()) k_local(CountArgs A, LocalHeavy hv, int kt, int amax, int split)
{
    constexpr int WPB = local_wpb<NW>(), D = 32 * NW;
    using Work = LocalWork<NW>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t bin[LOCAL_BINOM * (LOCAL_BINOM + 1) / 2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *tab = local_set_up<NW>(smem, bin, A, kt, amax, lane, wid);
    Work &Wk = *reinterpret_cast<Work *>(smem + (size_t)wid * local_warp_bytes<NW>(kt));
    const unsigned warp = blockIdx.x * WPB + wid;
    if (Work::GSTACK) Wk.gstk = A.gstack + (size_t)warp * (D + 1) * Work::FW;
    Wk.etab = MODE == MODE_EDGE ? A.eidtab + (size_t)warp * D * D : nullptr;
    WalkCounters wc;
    for (;;) {
        unsigned qi = 0;
        if (lane == 0) qi = atomicAdd(A.qhead, A.chunk);
        qi = __shfl_sync(FULL, qi, 0);
        if (qi >= A.nroots) break;
        const unsigned qend = min(qi + A.chunk, A.nroots);
        for (; qi < qend; ++qi) {
            const uint32_t r = A.roots[qi];
            const int64_t rbeg = A.orow[r];
            const int d = (int)(A.orow[r + 1] - rbeg);
            if (d > D) {
                if (lane == 0) atomicOr(A.err, DERR_RANGE);
                continue;
            }
            gather_rows<NW, MODE>(Wk, A, lane, rbeg, d);
            if (split) {
                unsigned bits = 0;
                for (int t = lane; t < d * Work::RS; t += 32) bits += __popc(Wk.adj[t]);
                const unsigned edges = __reduce_add_sync(FULL, bits) / 2;
                if (edges >= LOCAL_HEAVY_EDGES && (unsigned)(d * (d - 1) / 2) - edges > LOCAL_FEW_MISSING) {
                    const unsigned parts = local_parts(edges, d);
                    unsigned slot = 0, at = 0;
                    if (lane == 0) {
                        slot = atomicAdd(hv.count, 1u);
                        if (slot < hv.cap) at = atomicAdd(hv.count + 1, parts);
                    }
                    slot = __shfl_sync(FULL, slot, 0);
                    at = __shfl_sync(FULL, at, 0);
                    if (slot < hv.cap) {  // else walked here
                        uint32_t *rows = hv.rows + (size_t)slot * D * NW;
                        for (int t = lane; t < d * NW; t += 32) rows[t] = Wk.adj[(t / NW) * Work::RS + t % NW];
                        if (MODE == MODE_EDGE) {
                            uint32_t *et = hv.etab + (size_t)slot * D * D;
                            for (int t = lane; t < d * D; t += 32) et[t] = Wk.etab[t];
                        }
                        if (lane == 0) hv.root[slot] = r;
                        for (unsigned q = lane; q < parts; q += 32) hv.items[at + q] = make_uint2(slot, q | parts << 16);
                        __syncwarp();
                        continue;
                    }
                }
            }
            LocalWalk<NW, MODE> w{Wk, tab, bin, A, lane, kt, r, rbeg, d};
            w.run(0, 1, wc);
        }
        if (vload(A.err) & (DERR_STACK | DERR_RANGE)) break;
    }
    wc.flush(A.stats, A.cls, lane);
}

// Second launch: the parts of the dense roots.
template <int NW, int MODE>
__global__ void __launch_bounds__(32 * local_wpb<NW>(), local_blocks<NW>()) k_local_parts(CountArgs A, LocalHeavy hv, int kt, int amax)
{
    constexpr int WPB = local_wpb<NW>(), D = 32 * NW;
    using Work = LocalWork<NW>;
    const unsigned nitems = *(volatile unsigned *)(hv.count + 1);
    if (nitems == 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t bin[LOCAL_BINOM * (LOCAL_BINOM + 1) / 2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long *tab = local_set_up<NW>(smem, bin, A, kt, amax, lane, wid);
    Work &Wk = *reinterpret_cast<Work *>(smem + (size_t)wid * local_warp_bytes<NW>(kt));
    if (Work::GSTACK) Wk.gstk = A.gstack + (size_t)(blockIdx.x * WPB + wid) * (D + 1) * Work::FW;
    WalkCounters wc;
    for (;;) {
        unsigned i = 0;
        if (lane == 0) i = atomicAdd(hv.count + 2, 1u);
        i = __shfl_sync(FULL, i, 0);
        if (i >= nitems) break;
        const uint2 it = hv.items[i];
        const uint32_t r = hv.root[it.x];
        const int64_t rbeg = A.orow[r];
        const int d = (int)(A.orow[r + 1] - rbeg);
        const uint32_t *rows = hv.rows + (size_t)it.x * D * NW;
        for (int t = lane; t < d; t += 32) Wk.ids[t] = A.ocol[rbeg + t];
        for (int t = lane; t < d * NW; t += 32) Wk.adj[(t / NW) * Work::RS + t % NW] = rows[t];
        Wk.etab = MODE == MODE_EDGE ? hv.etab + (size_t)it.x * D * D : nullptr;
        __syncwarp();
        LocalWalk<NW, MODE> w{Wk, tab, bin, A, lane, kt, r, rbeg, d};
        w.run(it.y & 0xFFFFu, it.y >> 16, wc);
        if (vload(A.err) & (DERR_STACK | DERR_RANGE)) break;
    }
    wc.flush(A.stats, A.cls, lane);
}

// Roots of many graphs (k_count_batch for out-degrees of at most 128).
template <int NW, int MODE>
__global__ void __launch_bounds__(32 * local_wpb<NW>(), local_blocks<NW>())
    k_local_batch(const BatchGraph *gs, const uint64_t *entries, unsigned nentries, unsigned *qhead,
                  const unsigned long long *B, int Bw, int amax, unsigned *err, unsigned long long *stats,
                  uint32_t *gstack, uint32_t *eidtab)
{
    constexpr int WPB = local_wpb<NW>(), D = 32 * NW, KT = LocalWork<NW>::WINDOW;
    using Work = LocalWork<NW>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t bin[LOCAL_BINOM * (LOCAL_BINOM + 1) / 2];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    CountArgs A{};
    A.B = B;
    A.Bw = Bw;
    A.err = err;
    A.stats = stats;
    unsigned long long *tab = local_set_up<NW>(smem, bin, A, KT, amax, lane, wid);
    Work &Wk = *reinterpret_cast<Work *>(smem + (size_t)wid * local_warp_bytes<NW>(KT));
    const unsigned warp = blockIdx.x * WPB + wid;
    if (Work::GSTACK) Wk.gstk = gstack + (size_t)warp * (D + 1) * Work::FW;
    Wk.etab = MODE == MODE_EDGE ? eidtab + (size_t)warp * D * D : nullptr;
    WalkCounters wc;
    for (;;) {
        unsigned qi = 0;
        if (lane == 0) qi = atomicAdd(qhead, 1u);
        qi = __shfl_sync(FULL, qi, 0);
        if (qi >= nentries) break;
        const uint64_t e = entries[qi];
        const BatchGraph &G = gs[e >> 32];
        const uint32_t r = (uint32_t)e;
        A.orow = G.orow;
        A.ocol = G.ocol;
        A.oeid = G.oeid;
        A.out = G.out;
        A.W = G.W;
        A.kmax = G.kmax;
        A.ksafe = G.ksafe;
        const int64_t rbeg = A.orow[r];
        const int d = (int)(A.orow[r + 1] - rbeg);
        if (d > D) {
            if (lane == 0) atomicOr(err, DERR_RANGE);
            break;
        }
        if (d == 0) {  // one path (h = 1, p = 0): c_1(r)
            if (MODE == MODE_VERTEX && lane == 0 && A.kmax >= 1)
                atomic_add_u64_carry(A.out + ((size_t)r * (A.kmax + 1) + 1) * A.W, 1ull, A.W, err);
            wc.nodes++;
            wc.leaves++;
            continue;
        }
        gather_rows<NW, MODE>(Wk, A, lane, rbeg, d);
        LocalWalk<NW, MODE> w{Wk, tab, bin, A, lane, min(KT, A.kmax), r, rbeg, d};
        w.run(0, 1, wc);
        if (vload(err) & (DERR_STACK | DERR_RANGE)) break;
    }
    wc.flush(stats, -1, lane);
}

// Resident blocks of a kernel per SM with its dynamic shared memory allowed.
template <typename K>
static pvt_status local_occupancy(K kern, int threads, size_t smem, int *per_sm)
{
    PVT_CK(resident_blocks((const void *)kern, threads, smem, per_sm));
    if (*per_sm < 1) {
        set_error("local count kernel cannot be resident (shared memory)");
        return PVT_ECUDA;
    }
    return PVT_OK;
}

template <int NW, int MODE>
pvt_status launch_local(pvt_dag *g, const CountArgs &base, int cls, cudaStream_t s)
{
    const unsigned cnt = (unsigned)g->wcnt[cls];
    if (cnt == 0) return PVT_OK;
    constexpr int WPB = local_wpb<NW>();
    constexpr size_t D = 32 * NW;
    CountArgs A = base;
    A.roots = g->wroots + g->wstart[cls];
    A.nroots = cnt;
    A.qhead = g->d_q + cls;
    A.cls = cls;
    const int kt = std::min(A.kmax, LocalWork<NW>::WINDOW), amax = g->alpha + 2;
    const size_t smem = local_warp_bytes<NW>(kt) * WPB;
    int per_sm = 0;
    pvt_status st;
    if ((st = local_occupancy(k_local<NW, MODE>, 32 * WPB, smem, &per_sm)) != PVT_OK) return st;
    const unsigned full = (unsigned)(g->num_sms * per_sm);
    A.chunk = NW == 1 ? claim_size(g, cnt, full * WPB) : 1u;
    const unsigned per_block = WPB * A.chunk;
    const unsigned grid = std::max(1u, std::min(full, (cnt + per_block - 1) / per_block));
    if (LocalWork<NW>::GSTACK) {
        if ((st = grow(g, g->gstack[cls], (size_t)full * WPB * (D + 1) * LocalWork<NW>::FW, s)) != PVT_OK) return st;
        A.gstack = g->gstack[cls].p;
    }
    if (MODE == MODE_EDGE) {
        if ((st = grow(g, g->etab[cls], (size_t)grid * WPB * D * D, s)) != PVT_OK) return st;
        A.eidtab = g->etab[cls].p;
    }
    if (g->sizing) return PVT_OK;
    // dense roots: at most 2^16, and 1 GB of edge-id tables; those that find no
    // room are walked by the warp that took them
    bool split = g->policy.persistent != 0;
    LocalHeavy hv{};
    if (split) {
        unsigned cap = std::min(cnt, 1u << 16);
        if (MODE == MODE_EDGE) cap = std::min(cap, (unsigned)(((size_t)1 << 28) / (D * D)));
        const size_t words = 2 * LOCAL_MAX_PARTS + D * NW + 1 + (MODE == MODE_EDGE ? D * D : 0);
        st = grow_least(g, g->lheavy[cls], cap, std::min(cap, 64u), words, s);
        if (st != PVT_OK && st != PVT_ENOMEM) return st;
        split = st == PVT_OK;
        hv.cap = cap;
    }
    if (split) {
        const size_t cap = hv.cap;
        uint32_t *w = g->lheavy[cls].p;
        hv.items = reinterpret_cast<uint2 *>(w);
        hv.rows = w + cap * 2 * LOCAL_MAX_PARTS;
        hv.root = hv.rows + cap * D * NW;
        hv.etab = hv.root + cap;
        hv.count = g->qctl + QCTL_WORDS * cls;
        PVT_CK(cudaMemsetAsync(hv.count, 0, 3 * sizeof(unsigned), s));
    }
    phase_begin(g, 1 + cls, s);
    k_local<NW, MODE><<<grid, 32 * WPB, smem, s>>>(A, hv, kt, amax, split ? 1 : 0);
    PVT_CK(cudaGetLastError());
    g->stats.launches++;
    if (split) {
        if ((st = local_occupancy(k_local_parts<NW, MODE>, 32 * WPB, smem, &per_sm)) != PVT_OK) return st;
        k_local_parts<NW, MODE><<<std::min(full, (unsigned)(g->num_sms * per_sm)), 32 * WPB, smem, s>>>(A, hv, kt, amax);
        PVT_CK(cudaGetLastError());
        g->stats.launches++;
    }
    phase_end(g, 1 + cls, s);
    return PVT_OK;
}

// scratch_room: bytes its stacks and edge tables may take.  Any number of warps
// walks the entries, so it makes do with less, down to a block's.
template <int NW, int MODE>
pvt_status launch_local_batch(const BatchGraph *gs, const uint64_t *entries, unsigned cnt, unsigned *qhead,
                              const unsigned long long *B, int Bw, unsigned *err, unsigned long long *stats, int num_sms,
                              size_t scratch_room, cudaStream_t s)
{
    constexpr int WPB = local_wpb<NW>();
    constexpr size_t D = 32 * NW;
    constexpr size_t smem = local_warp_bytes<NW>(LocalWork<NW>::WINDOW) * WPB;
    int per_sm = 0;
    pvt_status st = local_occupancy(k_local_batch<NW, MODE>, 32 * WPB, smem, &per_sm);
    if (st != PVT_OK) return st;
    unsigned grid = std::max(1u, std::min<unsigned>((unsigned)(num_sms * per_sm), (cnt + WPB - 1) / WPB));
    constexpr size_t stack = LocalWork<NW>::GSTACK ? (size_t)WPB * (D + 1) * LocalWork<NW>::FW : 0;  // words of a block
    constexpr size_t etab = MODE == MODE_EDGE ? (size_t)WPB * D * D : 0;
    constexpr size_t block_bytes = (stack + etab) * sizeof(uint32_t);
    Scratch mem(s);
    if constexpr (block_bytes > 0) {
        grid = (unsigned)std::max<size_t>(1, std::min<size_t>(grid, scratch_room / block_bytes));
        cudaError_t e;
        while ((e = mem.take(grid * block_bytes)) == cudaErrorMemoryAllocation && grid > 1) {
            (void)cudaGetLastError();
            grid = std::max(1u, grid / 4);
        }
        PVT_CK(e);
    }
    uint32_t *scratch = mem.as<uint32_t>();
    k_local_batch<NW, MODE><<<grid, 32 * WPB, smem, s>>>(gs, entries, cnt, qhead, B, Bw, BATCH_MAX_ALPHA + 2, err, stats,
                                                       scratch, scratch ? scratch + stack * grid : nullptr);
    PVT_CK(cudaGetLastError());
    return PVT_OK;
}

}  // namespace pvt
