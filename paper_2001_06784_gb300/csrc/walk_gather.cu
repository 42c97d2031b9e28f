// Gather of the <= 32 out-degree class of a two-phase global count.
//
// A root of out-degree d <= 32 needs its members' out-lists read once and
// each entry looked up among the members; the tree below it is small.  A
// kernel that does both is bound by issue slots (the lookups and the per-node
// control of a warp walk), and one warp that meets a dense root walks its
// whole tree while the others finish.  So this kernel only gathers: it closes
// the roots whose tree has a closed form (no edge among the members, or a
// clique) and emits every other root as a frame of the lane walk (lanes.cuh),
// where 32 subtrees share a warp and a heavy one is split by donation.
//
// The gather works on registers.  Lane i holds member i (id, out-list start
// and length) and a 1024-bit filter of the member ids, one word per lane; the
// concatenated out-lists are read 32 entries at a time, four rounds in
// flight.  An entry's list is found from the bit mask of list starts inside
// the round, an entry that passes the filter (about d in 1024 of the others)
// is compared with all members at once, and a match sets one bit in two
// lanes' rows.  What bounds it: issue slots, about 30 warp instructions per 32
// out-list entries (521M entries for the 941k such roots of the 1M-vertex,
// 10.8M-edge graph).  There the class took 3.13 ms as a warp walk and takes
// 0.93 ms here plus about 0.3 ms of the lane walk; on a 61k-vertex graph with
// planted communities, where one warp's dense root was the time, 1.10 ms
// became 0.17 + 0.22 ms.
#include <type_traits>

#include "lanes.cuh"

namespace pvt {

constexpr int G1_WPB = 8;              // warps per block
constexpr unsigned G1_RESERVE = 16;    // frame slots a warp reserves at once
constexpr int G1_ROUNDS = 4;           // rounds of 32 entries with loads in flight

// NARROW: the graph has fewer than 2^32 edges, so positions in the out-lists
// fit 32 bits.
template <bool NARROW>
__global__ void __launch_bounds__(32 * G1_WPB) k_gather1(CountArgs A)
{
    using Pos = std::conditional_t<NARROW, uint32_t, int64_t>;
    __shared__ unsigned sh32[HIST_H * HIST_P];
    __shared__ uint32_t s_tmp[G1_WPB][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
    uint32_t *tmp = s_tmp[wid];
    for (int i = threadIdx.x; i < HIST_H * HIST_P; i += blockDim.x) sh32[i] = 0;
    __syncthreads();
    unsigned long long nodes = 0, leaves = 0, words = 0;  // uniform
    unsigned slot = 0, slot_end = 0;                      // reserved frame slots (uniform)
    const bool hold = A.kmax >= 2;                        // hold children of a root (h = 2) are walked
    for (;;) {
        // ---- claim up to A.chunk (<= 32) roots; lane i holds the i-th
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(A.qhead, A.chunk);
        base = __shfl_sync(FULL, base, 0);
        if (base >= A.nroots) break;
        const unsigned nc = min(A.chunk, A.nroots - base);
        int64_t cb = 0;
        int cd = 0;
        if ((unsigned)lane < nc) {
            const uint32_t r = A.roots[base + lane];
            cb = A.orow[r];
            cd = (int)(A.orow[r + 1] - cb);
        }
        for (unsigned ci = 0; ci < nc; ++ci) {
            const int64_t rbeg = __shfl_sync(FULL, cb, ci);
            const int d = __shfl_sync(FULL, cd, ci);
            if (d > 32) {
                if (lane == 0) atomicOr(A.err, DERR_RANGE);
                continue;
            }
            // ---- members: id, out-list start and length
            uint32_t id = 0xFFFFFFFFu, od = 0;
            int64_t rs = 0;
            if (lane < d) {
                id = A.ocol[rbeg + lane];
                if (d > 1) {  // a single member has no edge to find
                    rs = A.orow[id];
                    od = (uint32_t)(A.orow[id + 1] - rs);
                }
            }
            uint32_t inc = od;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, inc, o);
                if (lane >= o) inc += t;
            }
            const uint32_t T = __shfl_sync(FULL, inc, 31);
            const uint32_t off = inc - od;
            // filter of the member ids: bit hash(id) of 1024, word w in lane w
            const uint32_t hash = id * FIB_HASH;
            tmp[lane] = 0;
            __syncwarp();
            if (lane < d) atomicOr(&tmp[hash >> 27], 1u << ((hash >> 22) & 31u));
            __syncwarp();
            const uint32_t filter = tmp[lane];
            __syncwarp();
            // k-th member with a nonempty list in lane k: its index, and the
            // distance from a position in the concatenation to its entry
            const unsigned some = __ballot_sync(FULL, od != 0);
            uint32_t mk = (uint32_t)lane;
            if (some & (some + 1u)) {  // an empty list before another
                if (od) tmp[__popc(some & lt)] = (uint32_t)lane;
                __syncwarp();
                mk = tmp[lane] & 31u;
            }
            const Pos delta = __shfl_sync(FULL, (Pos)(rs - (int64_t)off), (int)mk);
            __syncwarp();
            uint32_t row = 0;   // this member's row
            int started = -1;   // lists started before the current round, less one
            for (uint32_t t0 = 0; t0 < T; t0 += 32 * G1_ROUNDS) {
                uint32_t x[G1_ROUNDS];
                int own[G1_ROUNDS];
#pragma unroll
                for (int q = 0; q < G1_ROUNDS; ++q) {
                    const uint32_t w0 = t0 + 32u * q;
                    const bool here = od && off - w0 < 32u;
                    const uint32_t starts = __reduce_or_sync(FULL, here ? 1u << (off - w0) : 0u);
                    own[q] = started + __popc(starts & le);
                    started += __popc(starts);
                    const uint32_t t = w0 + lane;
                    const Pos at = __shfl_sync(FULL, delta, own[q]) + (Pos)t;  // (modulo 2^32 in 32 bits)
                    x[q] = t < T ? A.ocol[at] : 0xFFFFFFFFu;
                }
#pragma unroll
                for (int q = 0; q < G1_ROUNDS; ++q) {
                    const uint32_t hx = x[q] * FIB_HASH;
                    const uint32_t word = __shfl_sync(FULL, filter, (int)(hx >> 27));
                    const uint32_t t = t0 + 32u * q + lane;
                    unsigned cand = __ballot_sync(FULL, t < T && ((word >> ((hx >> 22) & 31u)) & 1u));
                    while (cand) {
                        const int l = __ffs(cand) - 1;
                        cand &= cand - 1;
                        const unsigned hit = __ballot_sync(FULL, id == __shfl_sync(FULL, x[q], l));
                        if (!hit) continue;
                        const int a = __ffs(hit) - 1;
                        const int u = (int)__shfl_sync(FULL, mk, __shfl_sync(FULL, own[q], l));
                        if (lane == u) row |= 1u << a;
                        if (lane == a) row |= 1u << u;
                    }
                }
            }
            // ---- closed forms: no edge (the pivot leaf (1, 1) and a hold leaf
            // (2, 0) per other member), a clique (one leaf (1, d))
            const unsigned dsum = __reduce_add_sync(FULL, (unsigned)__popc(row));
            if (dsum == (unsigned)(d * (d - 1))) {
                ++nodes;
                ++leaves;
                words += (unsigned)d;
                if (lane == 0) tally_n<true>(sh32, A, 1, d, 1u);
            } else if (dsum == 0) {
                const unsigned held = hold ? (unsigned)(d - 1) : 0u;
                nodes += 2 + held;
                leaves += 1 + held;
                words += (unsigned)d;
                if (lane == 0) {
                    tally_n<true>(sh32, A, 1, 1, 1u);
                    if (held) tally_n<true>(sh32, A, 2, 0, held);
                }
            } else {
                if (slot == slot_end) {
                    if (lane == 0) slot = atomicAdd(A.emit1_count, G1_RESERVE);
                    slot = __shfl_sync(FULL, slot, 0);
                    slot_end = slot + G1_RESERVE;
                    if (slot_end > A.emit1_cap) {  // cannot happen (gather1_slots)
                        if (lane == 0) atomicOr(A.err, DERR_RANGE);
                        slot = slot_end = 0;
                        continue;
                    }
                }
                uint32_t *fr = A.emit1 + (size_t)slot * FRAME_WORDS;
                ++slot;
                fr[4 + lane] = row;
                if (lane == 0)
                    *reinterpret_cast<uint4 *>(fr) =
                        make_uint4(FRAME_COMPACT, 1u << 16, d >= 32 ? FULL : (1u << d) - 1u, (uint32_t)A.cls);
            }
        }
    }
    // slots reserved and not used
    if (slot + (unsigned)lane < slot_end) A.emit1[(size_t)(slot + lane) * FRAME_WORDS] = FRAME_NONE;
    if (lane == 0 && nodes) {
        atomicAdd(&A.stats[0], nodes);
        atomicAdd(&A.stats[1], leaves);
        atomicAdd(&A.stats[2], words);
        atomicAdd(&A.stats[3 + A.cls], words);
    }
    hist_flush(sh32, A);
}

using Gather1 = void (*)(CountArgs);
static Gather1 gather1_kernel(const pvt_dag *g) { return g->m < (1ll << 32) ? k_gather1<true> : k_gather1<false>; }

static cudaError_t gather1_grid(const pvt_dag *g, unsigned *blocks)
{
    int per_sm = 0;
    const cudaError_t e = resident_blocks((const void *)gather1_kernel(g), 32 * G1_WPB, 0, &per_sm);
    *blocks = (unsigned)(g->num_sms * std::max(per_sm, 1));
    return e;
}

unsigned gather1_slots(const pvt_dag *g, unsigned cnt)
{
    unsigned blocks = 0;
    gather1_grid(g, &blocks);
    return cnt + blocks * G1_WPB * G1_RESERVE;
}

pvt_status launch_gather1(pvt_dag *g, const CountArgs &base, const uint32_t *roots, unsigned cnt, unsigned slots,
                          cudaStream_t s)
{
    CountArgs A = base;
    A.cls = 1;
    A.roots = roots;
    A.nroots = cnt;
    A.qhead = g->d_q + 1;
    A.emit1_cap = slots;
    unsigned blocks = 0;
    PVT_CK(gather1_grid(g, &blocks));
    A.chunk = claim_size(g, cnt, blocks * G1_WPB);
    const unsigned per_block = G1_WPB * A.chunk;
    blocks = std::max(1u, std::min(blocks, (cnt + per_block - 1) / per_block));
    gather1_kernel(g)<<<blocks, 32 * G1_WPB, 0, s>>>(A);
    PVT_CK(cudaGetLastError());
    g->stats.launches++;
    return PVT_OK;
}

}  // namespace pvt
