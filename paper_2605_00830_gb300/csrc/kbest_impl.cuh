// kbest_impl.cuh -- sm_103a K-Best kernels (templates; instantiated per edge-label plane
// count in kbest_b0.cu, kbest_b2.cu and kbest_b8.cu; the S0 packing kernel and the dispatch
// live in kbest_kernels.cu).
//
//   kbest_kernel          S1-S5 for every pair of a size class: persistent one-CTA teams pull
//                         pairs from a device work queue; per level they find the target
//                         vertices still open to some node, build per-node neighbour bitsets,
//                         score every open (node, column) with AND/XOR + popcount into one
//                         byte and one histogram count, select the best K exactly (threshold
//                         bucket, a stable compaction of the bytes, a counting placement),
//                         write the kept children in key order and stage the next cost row;
//                         finally they complete the leaves and take the argmin.
//   kbest_cluster_kernel  the same with a team of 2-16 CTAs in a thread-block cluster, for
//                         classes with fewer pairs than SMs and large pairs or beams.
//
// Method: Algorithm 1 of Dabah & Herten (branching Sec. 4.1.1, evaluation Sec. 4.1.2 and
// Algorithm 2, selection Sec. 4.2, leaf insertions Sec. 4.4). The paper's GPU design
// (one block per node, a lambda walk per successor, atomic top-L lists) is replaced here:
// the implied edge cost of substituting v_i by u is computed from bitsets,
//     P     = images of the already-substituted g1 neighbours of v_i,
//     Img   = images of every substituted g1 vertex,
//     A2[u] = neighbours of u in g2,
//   inserted edges   = popc(A2[u] & Img & ~P)
//   deleted edges    = popc(P & ~A2[u]) + (# g1 neighbours of v_i that were deleted)
//   relabelled edges = popc(A2[u] & P & OR_b(PL_b ^ L2_b[u]))
// and when insertion and deletion cost the same, the first two fold into one
// popc((A2[u] & Img) ^ P) since P is a subset of Img.
#pragma once
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "fastged_internal.h"

namespace fastged {

__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ int warp_sum(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// bits k of word w with k < i
__device__ __forceinline__ uint64_t low_mask(int i, int w)
{
    const int lo = w * 64;
    if (i >= lo + 64) return ~0ull;
    if (i <= lo) return 0ull;
    return (1ull << (i - lo)) - 1ull;
}

// ------------------------------------------------------------------------------------
// K-Best teams
// ------------------------------------------------------------------------------------
// Team scalars: in shared memory for a one-CTA team, in the cluster's global scratch for a
// cluster team (MW = warps the team may have).
template <int MW>
struct TeamSharedT {
    int pair;
    int wcode[MW];                  // best successor of each warp (variant B)
    unsigned long long wbest[MW];   // best completion key of each warp
};
using TeamShared = TeamSharedT<kMaxWarps>;
using TeamSharedCl = TeamSharedT<kMaxClusterWarps>;

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cluster_size()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// Barrier over every thread of the cluster; writes before it (shared or global) are visible
// to every thread of the cluster after it (release / acquire at cluster scope).
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
                 ::: "memory");
}

// The threads solving one pair: one CTA, or every CTA of a cluster (CL).
template <bool CL>
struct Team {
    int tid, T, warp, NW;
    __device__ __forceinline__ Team()
    {
        if (CL) {
            tid = (int)cluster_rank() * (int)blockDim.x + (int)threadIdx.x;
            T = (int)cluster_size() * (int)blockDim.x;
        } else {
            tid = (int)threadIdx.x;
            T = (int)blockDim.x;
        }
        warp = tid >> 5;
        NW = T >> 5;
    }
    __device__ __forceinline__ void sync() const
    {
        if (CL) cluster_barrier();
        else __syncthreads();
    }
};

template <typename Word>
struct Regions {
    int32_t *hist, *alpha2, *crow, *sbase, *sel, *selped, *klist, *kped, *noff, *nbr, *chist;
    int32_t *ped0, *ped1;
    uint32_t *allm;
    uint16_t *act;
    uint8_t *score, *rec, *et0, *et1;
    Word *a2t, *l2t, *img0, *img1, *P, *PL, *imgl;
    uint8_t *map0, *map1;
};

// A kept child is stored in the selection list as (parent slot << 11) | j, j = 0..n2.
constexpr int kSelShift = 11;

__device__ __forceinline__ int popcw(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int popcw(uint64_t x) { return __popcll(x); }

#ifdef FASTGED_PHASE_TIMERS
// profiling builds only: cycles thread 0 of every team spends in each phase
#define PHASE_MARK(k)                                        \
    do {                                                     \
        if (threadIdx.x == 0) {                              \
            const long long t_ = clock64();                  \
            ph[k] += t_ - ph_last;                           \
            ph_last = t_;                                    \
        }                                                    \
    } while (0)
#else
#define PHASE_MARK(k) do { } while (0)
#endif

// Lanes of the warp whose 5-bit value equals `v`, among the lanes in `valid`, given the
// ballots b[k] of bit k of every lane's value.
__device__ __forceinline__ unsigned same_value_lanes(unsigned valid, const unsigned b[5], int v)
{
    unsigned m = valid;
#pragma unroll
    for (int k = 0; k < 5; ++k) m &= ((v >> k) & 1) ? b[k] : ~b[k];
    return m;
}

// One active column of a level for the single-word teams: adjacency word and label planes of
// the target vertex, its cost-row entry, padded to 16 bytes so that one vector load or two
// bring it. All lanes of a warp read the same record (a broadcast).
template <typename Word, int NPL>
struct __align__(16) ColRec {
    Word a2;
    Word l[NPL > 0 ? NPL : 1];
    int32_t crow;
};

static_assert(sizeof(ColRec<uint32_t, 0>) == col_rec_bytes(true, 0), "record size");
static_assert(sizeof(ColRec<uint32_t, 2>) == col_rec_bytes(true, 2), "record size");
static_assert(sizeof(ColRec<uint32_t, kMaxB>) == col_rec_bytes(true, kMaxB), "record size");
static_assert(sizeof(ColRec<uint64_t, 0>) == col_rec_bytes(false, 0), "record size");
static_assert(sizeof(ColRec<uint64_t, 2>) == col_rec_bytes(false, 2), "record size");
static_assert(sizeof(ColRec<uint64_t, kMaxB>) == col_rec_bytes(false, kMaxB), "record size");

// Score bytes: one per (parent node, active column) of the nodes a CTA owns, row after row.
// 0..126 is the successor's PED offset from the pass's anchor (0 also stands for one below an
// anchor that is a guess), 127 stands for an offset past
// the window and for a column that is no successor of the node (its vertex is used).
constexpr int kScoreMax = 127;
constexpr int kAnchorSlack = 48;   // of the 127 offsets, kept for a level that starts lower
constexpr int kBuckets = kHistRow;   // histogram counters: offsets 0..126, [127] the successors

// Everything a warp needs to score its nodes at one level.
template <typename Word>
struct LevelView {
    const Word *imgw;       // Img rows: the CTA's staged copy (cluster) or the beam's
    const int32_t *crow;    // S1 cost row
    int ioff, cs0;          // first node of imgw's rows, of the CTA's node tables
    int s_lo, s_hi;         // nodes of this warp
    int nact;               // active columns of the level
    int stride;             // bytes per row of score bytes (>= nact)
    int64_t nimg;           // elements behind imgw
    // eight and more words: the level's rows of neighbour counts (null: none are kept), the
    // beam's maps and their stride, v_i's prior neighbours in the list
    const uint8_t *et;
    const uint16_t *map;
    int64_t mt;
    int n0, deg;
};

// PED of successor (node s, column j). Column j == n2 is the deletion v_i -> eps: its A2
// column is empty, so the implied-edge terms count every substituted neighbour in P as a
// deleted edge (with the dcnt deleted neighbours in sbase, all deg edges to v_0..v_{i-1}),
// and the cost row holds c_vdel there.
template <int W, typename Word>
__device__ __forceinline__ int succ_ped(const KParams &p, const Regions<Word> &R,
                                        const LevelView<Word> &V, int B, int s, int j)
{
    const int64_t im = (int64_t)(s - V.ioff) * W, Ps = (int64_t)(s - V.cs0) * W;
    const bool fold_ie = p.cost.eins == p.cost.edel;
    const int N2S = p.lay.n2s;
    int x = 0, y = 0, z = 0;
    for (int w = 0; w < W; ++w) {
        const Word aw = FG_AT(R.a2t, w * N2S + j, FG_N(Word, p.lay.rsize[RG_A2T]));
        const Word ai = aw & FG_AT(V.imgw, im + w, V.nimg);
        const Word pw = FG_AT(R.P, Ps + w, FG_N(Word, p.lay.rsize[RG_P]));
        if (fold_ie) {
            x += popcw((Word)(ai ^ pw));
        } else {
            x += popcw((Word)(ai & ~pw));
            y += popcw((Word)(pw & ~aw));
        }
        Word ld = (Word)0;
        for (int b = 0; b < B; ++b)
            ld |= FG_AT(R.PL, ((int64_t)b * p.lay.kloc + (s - V.cs0)) * W + w, FG_N(Word, p.lay.rsize[RG_PL])) ^
                  FG_AT(R.l2t, (b * W + w) * N2S + j, FG_N(Word, p.lay.rsize[RG_L2T]));
        z += popcw((Word)(aw & pw & ld));
    }
    return FG_AT(R.sbase, s - V.cs0, FG_N(int32_t, p.lay.rsize[RG_SBASE])) +
           FG_AT(V.crow, j, N2S) + p.cost.eins * x + p.cost.edel * y + p.cost.esub * z;
}

// Score byte of PED offset d in a pass of the exact selection: with sh > 0 in units of 2^sh,
// offsets below 0 left out; sh == 0 gives 0 below 0 and 1 + d from there on.
__device__ __forceinline__ int exact_byte(int d, int sh)
{
    if (sh > 0) return d < 0 ? kScoreMax : min(d >> sh, kScoreMax);
    return d < 0 ? 0 : min(d, kScoreMax - 1) + 1;
}

// S3 over nodes [g0, g0 + ng) of this warp, lanes <-> active columns.
//
// Bound: the integer pipes. A column costs W popcounts of 64 bits (two 32-bit POPC each, 16
// lanes per clock and SM), so a chunk of 32 columns takes at least 4 W clocks of an SM. Only
// columns some node still has free are scored (1.02-1.3 times the free ones on dense pairs, 2.1
// times on a beam of 20,000). A score leaves one byte instead of the 8-byte
// entry that was written once and read back twice, and its histogram count is taken here: a
// shared increment costs 6 clocks of an SM per warp for any mix of buckets, what counting in
// packed registers costs too, but on the memory pipe. 1,024 dense pairs of 50-200 vertices,
// K = 256: 41.9 -> 19.6 ms; one G(200, 0.4) pair, K = 5,000: 40.1 -> 29.3 ms. (Large sparse
// pairs without edge labels are scored by score_table.)
//
// Every column's target
// tables stay in registers while the warp walks its nodes, whose vectors are read as
// broadcasts. With few active columns a warp scores several nodes per step. Each score leaves
// one byte and one count in the warp's histogram row (a shared-memory increment, which the
// hardware aggregates over lanes with the same bucket).
// EXACT = 0: offset from `anchor`, offsets below it counting as 0. EXACT = 1 (selection
// past the histogram window): see exact_byte.
template <int W, typename Word, int BK, bool FOLD, bool EXACT>
__device__ __forceinline__ void score_nodes(const KParams &p, const Regions<Word> &R,
                                            const LevelView<Word> &V, int B, int n2, int nw,
                                            int g0, int ng, int anchor, int sh, int32_t *hrow)
{
    constexpr int WB = 8 * (int)sizeof(Word);
    constexpr int NPL = BK == 8 ? kMaxB : BK;
    constexpr bool kRegLab = W * NPL <= 4;   // label planes of a column held in registers
    const int lane = threadIdx.x & 31;
    const int N2S = p.lay.n2s, KM = p.lay.kloc, nact = V.nact;
    const int c_eins = p.cost.eins, c_edel = p.cost.edel, c_esub = p.cost.esub;
    // columns per node in a step: 32, or a power of two that covers the active ones
    const int cs = nact > 16 ? 5 : nact > 8 ? 4 : nact > 4 ? 3 : nact > 2 ? 2 : nact > 1 ? 1 : 0;
    const int step = 32 >> cs, sub = lane >> cs;
    for (int a0 = 0; a0 < nact; a0 += 1 << cs) {
        const int a = a0 + (lane & ((1 << cs) - 1));
        const bool col = a < nact;
        const int j = col ? (int)FG_AT(R.act, a, FG_N(uint16_t, p.lay.rsize[RG_ACT])) : n2;
        const int jw = min(j >> 5, W * WB / 32 - 1);
        const uint32_t jm = j < n2 ? 1u << (j & 31) : 0u;   // 0: the deletion is never used up
        Word aw[W], lw[kRegLab && NPL > 0 ? W * NPL : 1];
#pragma unroll
        for (int w = 0; w < W; ++w)
            aw[w] = FG_AT(R.a2t, w * N2S + j, FG_N(Word, p.lay.rsize[RG_A2T]));
        if (kRegLab && NPL > 0) {
#pragma unroll
            for (int x = 0; x < W * NPL; ++x)
                lw[x] = x < B * W ? FG_AT(R.l2t, x * N2S + j, FG_N(Word, p.lay.rsize[RG_L2T])) : (Word)0;
        }
        const int cj = FG_AT(V.crow, j, N2S) - anchor;
        // (sixteen words with label planes leave no registers for two nodes at once: 20 pairs of
        // 500-1,000 vertices, K = 256, labels 0-200, 200 -> 138 ms; unlabelled ones lose 1-4 %)
#pragma unroll (W > 8 && NPL > 0 ? 1 : 2)
        for (int t0 = 0; t0 < ng; t0 += step) {
            const bool ok = col && t0 + sub < ng;
            const int s = g0 + (t0 + sub < ng ? t0 + sub : 0);
            const int64_t im = (int64_t)(s - V.ioff) * W, Ps = (int64_t)(s - V.cs0) * W;
            int x = 0, y = 0, z = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (W > 4 && w >= nw) break;
                const Word ai = aw[w] & FG_AT(V.imgw, im + w, V.nimg);
                const Word pw = FG_AT(R.P, Ps + w, FG_N(Word, p.lay.rsize[RG_P]));
                if (FOLD) {
                    x += popcw((Word)(ai ^ pw));
                } else {
                    x += popcw((Word)(ai & ~pw));
                    y += popcw((Word)(pw & ~aw[w]));
                }
                // (large pairs: most words hold no image of v_i's few prior neighbours; such 20 pairs,
                // labels 0-200, 1,360 -> 200 ms, labels 0-2, 199 -> 92)
                if (NPL > 0 && B > 0 && (W < 8 || pw != (Word)0)) {
                    Word ld = (Word)0;
#pragma unroll
                    for (int b = 0; b < NPL; ++b)
                        if (b < B)
                            ld |= FG_AT(R.PL, ((int64_t)b * KM + (s - V.cs0)) * W + w, FG_N(Word, p.lay.rsize[RG_PL])) ^
                                  (kRegLab ? lw[kRegLab ? b * W + w : 0]
                                           : FG_AT(R.l2t, (b * W + w) * N2S + j, FG_N(Word, p.lay.rsize[RG_L2T])));
                    z += popcw((Word)(aw[w] & pw & ld));
                }
            }
            int d = FG_AT(R.sbase, s - V.cs0, FG_N(int32_t, p.lay.rsize[RG_SBASE])) + cj + c_eins * x;
            if (!FOLD) d += c_edel * y;
            if (NPL > 0) d += c_esub * z;
            const uint32_t uw = FG_AT((const uint32_t *)V.imgw, im * (int)(sizeof(Word) / 4) + jw,
                                      V.nimg * (int)(sizeof(Word) / 4));
            int v;
            if (EXACT) v = exact_byte(d, sh);
            else v = max(0, min(d, kScoreMax));
            if (uw & jm) v = kScoreMax;
            if (ok) {
                FG_AT(R.score, (int64_t)(s - V.cs0) * V.stride + a, FG_N(uint8_t, p.lay.rsize[RG_SCORE])) = (uint8_t)v;
                if (v < kScoreMax) atomicAdd(&FG_AT(hrow, v, kBuckets), 1);
            }
        }
    }
}

// S3 for single-word teams, lanes <-> parent nodes. With 10-40 target vertices a chunk of 32
// columns is half empty (1.9-2.3 lane slots per successor measured on the workload's levels)
// and every node's vectors are loaded per chunk; this way round it is 1.6, the column records
// are broadcasts, and four scores make one store (4,096 served molecule pairs, a third of them
// with K = 512 here: 3.51 -> 2.98 ms). A node's vectors stay in its lane's
// registers and the warp walks the level's active columns four at a time (one store of four
// score bytes). A group of at most 16 nodes is spread over the lanes, 2^qs lanes per node
// taking every 2^qs-th quad. nd: the lane's node in the group (valid when `act`), base: its
// base PED less the anchor. Rows are an odd number of quads long, so the lanes' stores fall
// into different banks.
template <typename Word, int BK, bool FOLD>
__device__ __forceinline__ void score_quads(const KParams &p, const Regions<Word> &R,
                                            const LevelView<Word> &V, int B, int row, bool act,
                                            int r, int qs, Word im, Word P, const Word *PL,
                                            int base, int32_t *hrow)
{
    constexpr int NPL = BK == 8 ? kMaxB : BK;
    using Rec = ColRec<Word, NPL>;
    const Rec *rec = (const Rec *)R.rec;
    const Word *jm = (const Word *)((const uint8_t *)R.rec + p.lay.jm_off);
    const int c_eins = p.cost.eins, c_edel = p.cost.edel, c_esub = p.cost.esub;
    const int nq = V.stride >> 2, nk = (V.nact + 3) >> 2;   // quads of a row, with columns
    if (!act) base = 1 << 28;   // past every bucket
    for (int k = r; k < nq; k += 1 << qs) {
        uint32_t v4 = k < nk ? 0u : 0x7f7f7f7fu;
        if (k < nk) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const Rec c = FG_AT(rec, 4 * k + u, FG_N(Rec, p.lay.jm_off));
            const Word used = im & FG_AT(jm, 4 * k + u, FG_N(Word, p.lay.rsize[RG_REC] - p.lay.jm_off));
            const Word ai = c.a2 & im;
            int d = base + c.crow;
            if (FOLD) d += c_eins * popcw((Word)(ai ^ P));
            else d += c_eins * popcw((Word)(ai & ~P)) + c_edel * popcw((Word)(P & ~c.a2));
            if (NPL > 0) {
                Word ld = (Word)0;
#pragma unroll
                for (int b = 0; b < NPL; ++b)
                    if (b < B) ld |= PL[b] ^ c.l[b];
                d += c_esub * popcw((Word)(c.a2 & P & ld));
            }
            const int v = used ? kScoreMax : max(0, min(d, kScoreMax));
            atomicAdd(&FG_AT(hrow, v, kBuckets), 1);   // [127] is not read as a count
            v4 |= (uint32_t)v << (8 * u);
        }
        }
        if (act) FG_AT((uint32_t *)R.score, (int64_t)row * nq + k, FG_N(uint32_t, p.lay.rsize[RG_SCORE])) = v4;
    }
}

// four bits of x (from bit 0) -> four bytes of 0 or 1
__device__ __forceinline__ uint32_t nibble_bytes(uint32_t x)
{
    return ((x & 15u) * 0x00204081u) & 0x01010101u;
}

// Node vectors of a group in the lanes (lane t: node g0 + t) for score_table.
struct TableNode {
    int code;        // the node in the last level's selection: parent slot << kSelShift | j
    int base;        // base PED less the anchor
    int nimg;        // images in P
    uint32_t ph[2];  // the first four prior neighbours' images, 16 bits each (0xffff: deleted)
};

// S3 over nodes [g0, g0 + ng) for targets of eight and more words and sparse, unlabelled pairs.
// The implied edges of (s, j) need only two counts: E = g2 neighbours of j in Img(s), and T =
// those in P(s). E differs from the parent's E by one row of A2, so each kept node keeps a row
// of counts (a byte per column, double buffered): reading the parent's row, adding the bits
// of A2[j_s] and writing it back replaces 2 W popcounts per column by about one addition, and
// T is the sum of the bits of a few rows of A2 (deg of them).
//   inserted = E - T, deleted = |P| - T, PED = base + C + eins (E - T) + edel (|P| - T)
// Lanes <-> eight columns each (256 columns per step); the counts of four columns share a
// 32-bit word, and no byte of E + |P| can pass 255 (the caller checks the degrees). Every column
// is scored, used ones too (a row of counts has to stay complete for the children): about twice
// a node's successors on 64 pairs of 500-1,000 vertices, K = 1,024, whose time went 327 -> 199 ms
// with this path and the row prefetch below. Bound: latency of the rows and maps in L2 and DRAM
// at 16 warps per SM.
template <int W, typename MapT, typename Word, bool FOLD>
__device__ __forceinline__ void score_table(const KParams &p, const Regions<Word> &R,
                                            const LevelView<Word> &V, int n2, int g0, int ng,
                                            const TableNode &nd, const MapT *map, int64_t mt,
                                            int n0, int deg, const uint8_t *ec, uint8_t *en,
                                            bool root, int32_t *hrow)
{
    const int lane = threadIdx.x & 31;
    const int N2S = p.lay.n2s;
    const int c_eins = p.cost.eins, c_edel = p.cost.edel;
    const uint8_t *a2b = (const uint8_t *)R.a2t, *imb = (const uint8_t *)V.imgw;
    const int64_t NA = p.lay.rsize[RG_A2T], NE = p.lay.rsize[RG_ET0];
    constexpr int WBY = (int)sizeof(Word);
    // the parents' rows come from L2 or DRAM (all teams' rows: 150 MB on 64 large pairs), so a
    // whole row of the next node is under way while a node is scored
    constexpr int KS = (64 * W + 8 + 255) / 256;   // steps of a row at most
    uint2 nxt[KS];
    auto fetch = [&](int t) {
        const int par = __shfl_sync(0xffffffffu, nd.code, t) >> kSelShift;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int c0 = 256 * k + 8 * lane;
            nxt[k] = make_uint2(0u, 0u);
            if (!root && c0 < V.stride) nxt[k] = FG_AT((const uint2 *)ec, ((int64_t)par * N2S + c0) >> 3, NE >> 3);
        }
    };
    fetch(0);
    for (int t = 0; t < ng; ++t) {
        const int s = g0 + t;
        uint2 cur[KS];
#pragma unroll
        for (int k = 0; k < KS; ++k) cur[k] = nxt[k];
        if (t + 1 < ng) fetch(t + 1);
        const int code = __shfl_sync(0xffffffffu, nd.code, t);
        const int np = __shfl_sync(0xffffffffu, nd.nimg, t);
        const int base = __shfl_sync(0xffffffffu, nd.base, t) + (FOLD ? 0 : c_edel * np);
        const uint32_t p0 = __shfl_sync(0xffffffffu, nd.ph[0], t), p1 = __shfl_sync(0xffffffffu, nd.ph[1], t);
        const int jc = code & ((1 << kSelShift) - 1);
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int c0 = 256 * k + 8 * lane;
            if (c0 >= V.stride) break;
            const int wrow = (c0 / (8 * WBY)) * N2S, by = (c0 >> 3) % WBY;   // word row, byte in it
            // bits c0 .. c0 + 7 of row u of A2 (columns and rows of A2 are alike; row n2 is empty)
            // (columns past the last word: none)
            const bool in = c0 < 8 * WBY * W;
            auto bits = [&](int u) -> uint32_t {
                return in ? (uint32_t)FG_AT(a2b, (int64_t)(wrow + u) * WBY + by, NA) : 0u;
            };
            uint32_t e[2] = {0u, 0u};
            if (!root) {
                const uint32_t a = bits(jc);
                e[0] = cur[k].x + nibble_bytes(a);
                e[1] = cur[k].y + nibble_bytes(a >> 4);
            }
            FG_AT((uint2 *)en, ((int64_t)s * N2S + c0) >> 3, NE >> 3) = make_uint2(e[0], e[1]);
            uint32_t tt[2] = {0u, 0u};
            auto image = [&](uint32_t u) {
                if (u == 0xffffu) return;
                const uint32_t a = bits((int)u);
                tt[0] += nibble_bytes(a);
                tt[1] += nibble_bytes(a >> 4);
            };
            if (deg > 0) image(p0 & 0xffffu);
            if (deg > 1) image(p0 >> 16);
            if (deg > 2) image(p1 & 0xffffu);
            if (deg > 3) image(p1 >> 16);
            for (int q = 4; q < deg; ++q) {
                const int v = FG_AT(R.nbr, n0 + q, FG_N(int32_t, p.lay.rsize[RG_NBR])) & 0xffff;
                image((uint32_t)FG_AT(map, (int64_t)s * mt + v, FG_N(MapT, p.lay.rsize[RG_MAP0])));
            }
            // used columns and the ones past the deletion
            uint32_t um = c0 < n2 ? (uint32_t)FG_AT(imb, (int64_t)(s - V.ioff) * W * WBY + (c0 >> 3), V.nimg * WBY) : 0u;
            if (c0 + 8 > n2 + 1) um |= c0 > n2 ? 0xffu : 0xffu << (n2 + 1 - c0);
            uint32_t v4[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int4 cr = FG_AT((const int4 *)V.crow, (c0 >> 2) + h, N2S >> 2);
                const int cw[4] = {cr.x, cr.y, cr.z, cr.w};
                // FOLD: (E - T) + (|P| - T); else E - T, T apart
                const uint32_t f = FOLD ? e[h] + (uint32_t)np * 0x01010101u - 2u * tt[h] : e[h] - tt[h];
                v4[h] = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    int d = base + cw[u] + c_eins * (int)((f >> (8 * u)) & 0xffu);
                    if (!FOLD) d -= c_edel * (int)((tt[h] >> (8 * u)) & 0xffu);
                    int v = max(0, min(d, kScoreMax));
                    if ((um >> (4 * h + u)) & 1u) v = kScoreMax;
                    if (v < kScoreMax) atomicAdd(&FG_AT(hrow, v, kBuckets), 1);
                    v4[h] |= (uint32_t)v << (8 * u);
                }
            }
            FG_AT((uint2 *)R.score, ((int64_t)(s - V.cs0) * V.stride + c0) >> 3, FG_N(uint2, p.lay.rsize[RG_SCORE])) = make_uint2(v4[0], v4[1]);
        }
    }
}

// The scores of the exact selection from the level's own rows of counts, which score_table left:
// E is read as it stands, T summed from the rows of A2 of the images as there. (With passes over
// 2 W popcounts per column, 20 pairs of 500-1,000 vertices at K = 256 and costs of 700-3,001,
// where nearly every level comes here, took 378 ms; 86 ms so.)
template <int W, typename Word, bool FOLD>
__device__ __forceinline__ void score_counts(const KParams &p, const Regions<Word> &R,
                                             const LevelView<Word> &V, int n2, int anchor, int sh,
                                             int32_t *hrow)
{
    constexpr int WBY = (int)sizeof(Word);
    const int lane = threadIdx.x & 31;
    const int N2S = p.lay.n2s;
    const int c_eins = p.cost.eins, c_edel = p.cost.edel;
    const uint8_t *a2b = (const uint8_t *)R.a2t, *imb = (const uint8_t *)V.imgw;
    const int64_t NA = p.lay.rsize[RG_A2T], NE = p.lay.rsize[RG_ET0];
    for (int s = V.s_lo; s < V.s_hi; ++s) {
        for (int c0 = 8 * lane; c0 - 8 * lane < V.stride; c0 += 256) {   // the whole warp
            const bool on = c0 < V.stride;
            const int wrow = (c0 / (8 * WBY)) * N2S, by = (c0 >> 3) % WBY;
            const bool in = c0 < 8 * WBY * W;   // (columns past the last word: no bits)
            uint2 e = make_uint2(0u, 0u);
            if (on) e = FG_AT((const uint2 *)V.et, ((int64_t)s * N2S + c0) >> 3, NE >> 3);
            uint32_t tt[2] = {0u, 0u};
            int np = 0;   // images of v_i's prior neighbours
            for (int q0 = 0; q0 < V.deg; q0 += 32) {
                int u = 0xffff;
                if (q0 + lane < V.deg) {
                    const int v = FG_AT(R.nbr, V.n0 + q0 + lane, FG_N(int32_t, p.lay.rsize[RG_NBR])) & 0xffff;
                    u = FG_AT(V.map, (int64_t)s * V.mt + v, FG_N(uint16_t, p.lay.rsize[RG_MAP0]));
                }
                unsigned m = __ballot_sync(0xffffffffu, u != 0xffff);
                np += __popc(m);
                for (; m; m &= m - 1u) {
                    const int img = __shfl_sync(0xffffffffu, u, __ffs((int)m) - 1);
                    const uint32_t a = in ? (uint32_t)FG_AT(a2b, (int64_t)(wrow + img) * WBY + by, NA) : 0u;
                    tt[0] += nibble_bytes(a);
                    tt[1] += nibble_bytes(a >> 4);
                }
            }
            if (!on) continue;
            const int base = FG_AT(R.sbase, s - V.cs0, FG_N(int32_t, p.lay.rsize[RG_SBASE])) - anchor +
                             (FOLD ? 0 : c_edel * np);
            uint32_t um = c0 < n2 ? (uint32_t)FG_AT(imb, (int64_t)(s - V.ioff) * W * WBY + (c0 >> 3), V.nimg * WBY) : 0u;
            if (c0 + 8 > n2 + 1) um |= c0 > n2 ? 0xffu : 0xffu << (n2 + 1 - c0);
            uint32_t v4[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int4 cr = FG_AT((const int4 *)V.crow, (c0 >> 2) + h, N2S >> 2);
                const int cw[4] = {cr.x, cr.y, cr.z, cr.w};
                const uint32_t eh = h ? e.y : e.x;
                const uint32_t f = FOLD ? eh + (uint32_t)np * 0x01010101u - 2u * tt[h] : eh - tt[h];
                v4[h] = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    int d = base + cw[u] + c_eins * (int)((f >> (8 * u)) & 0xffu);
                    if (!FOLD) d -= c_edel * (int)((tt[h] >> (8 * u)) & 0xffu);
                    const int v = (um >> (4 * h + u)) & 1u ? kScoreMax : exact_byte(d, sh);
                    if (v < kScoreMax) atomicAdd(&FG_AT(hrow, v, kBuckets), 1);
                    v4[h] |= (uint32_t)v << (8 * u);
                }
            }
            FG_AT((uint2 *)R.score, ((int64_t)(s - V.cs0) * V.stride + c0) >> 3, FG_N(uint2, p.lay.rsize[RG_SCORE])) = make_uint2(v4[0], v4[1]);
        }
    }
}

// Scores this warp's nodes again for the exact selection (the node vectors are in place). A warp
// without nodes must not enter the scoring, which reads a column's tables before its first node:
// the CTA may have none at all, and then no list of columns. (The test stands here and not in
// solve_pair's column count, where two more conditions cost two-word clusters 15 %: 16 wide
// beams 13.1 -> 15.0 ms.)
template <int W, typename Word, int BK>
__device__ __noinline__ void score_exact(const KParams &p, const Regions<Word> &R,
                                         const LevelView<Word> &V, int B, int n2, int nw,
                                         int anchor, int sh, int32_t *hrow)
{
    const int lane = threadIdx.x & 31;
    for (int b = lane; b < kBuckets; b += 32) FG_AT(hrow, b, kBuckets) = 0;
    __syncwarp();
    if (V.s_lo >= V.s_hi) return;
    if (W >= 8 && V.et) {
        if (p.cost.eins == p.cost.edel) score_counts<W, Word, true>(p, R, V, n2, anchor, sh, hrow);
        else score_counts<W, Word, false>(p, R, V, n2, anchor, sh, hrow);
    } else if (p.cost.eins == p.cost.edel)
        score_nodes<W, Word, BK, true, true>(p, R, V, B, n2, nw, V.s_lo, V.s_hi - V.s_lo, anchor, sh, hrow);
    else
        score_nodes<W, Word, BK, false, true>(p, R, V, B, n2, nw, V.s_lo, V.s_hi - V.s_lo, anchor, sh, hrow);
    __syncwarp();
}

// Turns the warps' histogram rows into exclusive prefixes over the team's warps (in
// enumeration order) and leaves the bucket totals in the row after the CTA's last warp.
// A cluster's CTAs exchange their totals through its global scratch.
template <bool CL, typename Word>
__device__ __forceinline__ void prefix_buckets(const KParams &p, const Regions<Word> &R,
                                               const Team<CL> &tm)
{
    const int nwl = (int)blockDim.x >> 5;
    const int64_t NH = FG_N(int32_t, p.lay.rsize[RG_HIST]);
    __syncthreads();
    if (CL) {
        const int cr = (int)cluster_rank();
        for (int b = threadIdx.x; b < kBuckets; b += blockDim.x) {
            int t = 0;
            for (int w = 0; w < nwl; ++w) t += FG_AT(R.hist, w * kBuckets + b, NH);
            FG_AT(R.chist, cr * kBuckets + b, FG_N(int32_t, p.lay.rsize[RG_CHIST])) = t;
        }
        tm.sync();
    }
    for (int b = threadIdx.x; b < kBuckets; b += blockDim.x) {
        int run = 0, all = 0;
        if (CL) {
            const int cr = (int)cluster_rank(), ncta = (int)cluster_size();
            for (int c0 = 0; c0 < ncta; c0 += 4) {   // four loads in flight
                int v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = c0 + u < ncta ? FG_AT(R.chist, (c0 + u) * kBuckets + b, FG_N(int32_t, p.lay.rsize[RG_CHIST])) : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    all += v[u];
                    run += c0 + u < cr ? v[u] : 0;
                }
            }
        }
        for (int w = 0; w < nwl; ++w) {
            const int t = FG_AT(R.hist, w * kBuckets + b, NH);
            FG_AT(R.hist, w * kBuckets + b, NH) = run;
            run += t;
        }
        FG_AT(R.hist, nwl * kBuckets + b, NH) = CL ? all : run;
    }
    __syncthreads();
}

// The bucket where the cumulative count reaches `want` (kScoreMax when it lies past the
// window), the successors below it, and the lowest bucket that holds any. Lane l holds
// buckets 4l..4l+3.
__device__ __forceinline__ void find_threshold(const KParams &p, const int32_t *htot, int want,
                                               int &thr, int &below, int &first)
{
    const int lane = threadIdx.x & 31;
    int c[4], sum = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        c[u] = 4 * lane + u < kScoreMax ? FG_AT(htot, 4 * lane + u, kBuckets) : 0;
        sum += c[u];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    int run = incl - sum, mt = kScoreMax, mb = 0, mf = kScoreMax;
#pragma unroll
    for (int u = 3; u >= 0; --u)
        if (c[u]) mf = 4 * lane + u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (mt == kScoreMax && run < want && run + c[u] >= want) {
            mt = 4 * lane + u;
            mb = run;
        }
        run += c[u];
    }
    thr = (int)__reduce_min_sync(0xffffffffu, (unsigned)mt);
    first = (int)__reduce_min_sync(0xffffffffu, (unsigned)mf);
    below = __shfl_sync(0xffffffffu, mb, (thr >> 2) & 31);   // of the lane that holds thr
}

// Bit index of the k-th set bit (from 0) of a 16-bit mask that has more than k.
__device__ __forceinline__ int nth_bit16(uint32_t m, int k)
{
    int at = 0;
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {
        const int c = __popc((m >> at) & ((1u << h) - 1u));
        if (k >= c) {
            k -= c;
            at += h;
        }
    }
    return at;
}

// Stable compaction of the kept ones among score bytes [lo, hi), in the order of the bytes: every
// byte below `thr`, and the first q bytes equal to it counted over the whole team, of which eq
// lie before lo. A step takes 16 bytes per lane and leaves a 16-bit mask of the kept ones in
// each; then the lanes take the kept ones of all masks by rank, 32 at a time (the best
// parents' children crowd into a few lanes: their own loops over up to 16 hits made the
// one-warp kernel 4 % slower), or each its own when no lane has more than three (sparse
// masks: ranking them costs large pairs 15 %). put(position, index, byte) receives each kept one; positions run from
// `pos` and the walk ends once `last` is reached. Returns the number kept.
template <typename Put>
__device__ __forceinline__ int compact_bytes(const KParams &p, const uint8_t *score, int64_t n,
                                             int64_t lo, int64_t hi, int thr, int q, int pos,
                                             int eq, int last, Put put)
{
    const int lane = threadIdx.x & 31;
    const int pos0 = pos;
    const uint32_t t4 = (uint32_t)thr * 0x01010101u;
    for (int64_t b0 = lo & ~(int64_t)15; b0 < hi && pos < last; b0 += 512) {
        const int64_t o = b0 + 16 * lane;
        uint32_t le = 0, eqm = 0;
        if (o < hi) {
            const uint4 x = FG_AT((const uint4 *)score, o >> 4, n >> 4);
            const uint32_t v[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // bytes are at most 127: bit 7 of a byte says byte <= thr, byte == thr; the
                // product gathers bits 7, 15, 23 and 31 into a nibble
                const uint32_t a = ((t4 | 0x80808080u) - v[u]) & 0x80808080u;
                const uint32_t e = (0x80808080u - (v[u] ^ t4)) & 0x80808080u;
                le |= (((a >> 7) * 0x10204080u) >> 28) << (4 * u);
                eqm |= (((e >> 7) * 0x10204080u) >> 28) << (4 * u);
            }
            if (o < lo || o + 16 > hi) {   // bytes of the warps before and after this one
                uint32_t in = 0xffffu;
                if (o < lo) in &= 0xffffu << (int)(lo - o);
                if (o + 16 > hi) in &= 0xffffu >> (int)(o + 16 - hi);
                le &= in;
                eqm &= in;
            }
        }
        if (!__any_sync(0xffffffffu, le != 0)) continue;
        const int neq = __popc(eqm), nlt = __popc(le) - neq;
        int incl = nlt | (neq << 16);   // at most 512 each
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += y;
        }
        const int aeq = __shfl_sync(0xffffffffu, incl, 31) >> 16;
        const int e1 = eq + (incl >> 16), e0 = e1 - neq;   // ties up to this lane, before it
        // kept up to this lane: the smaller ones, and the ties within the quota
        const int kin = (incl & 0xffff) + (min(e1, q) - min(eq, q));
        uint32_t m = le;
        if (e1 > q) {   // the lane where the ties run out, and those after it
            m ^= eqm;
            for (int k = e0; k < q; ++k) {   // back in: the first q - e0 of them
                m |= eqm & (0u - eqm);
                eqm &= eqm - 1u;
            }
        }
        const int cnt = __shfl_sync(0xffffffffu, kin, 31);
        if (__reduce_max_sync(0xffffffffu, (unsigned)__popc(m)) <= 3u) {
            for (int r = kin - __popc(m); m; ++r) {   // few: each lane its own
                const int64_t idx = o + __ffs((int)m) - 1;
                m &= m - 1u;
                put(pos + r, (int)idx, (int)FG_AT(score, idx, n));
            }
        } else
        for (int r0 = 0; r0 < cnt; r0 += 32) {
            const int r = r0 + lane;
            // the first lane that holds more than r kept ones up to itself
            int src = 0;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
                if (__shfl_sync(0xffffffffu, kin, src + s - 1) <= r) src += s;
            const uint32_t ms = __shfl_sync(0xffffffffu, m, src & 31);
            const int ks = __shfl_sync(0xffffffffu, kin, src & 31);
            if (r < cnt) {
                const int64_t idx = b0 + 16 * src + nth_bit16(ms, r - (ks - __popc(ms)));
                put(pos + r, (int)idx, (int)FG_AT(score, idx, n));
            }
        }
        pos += cnt;
        eq += aeq;
    }
    return pos - pos0;
}

// The same for this warp's nodes of a team: klist receives the byte's index in the CTA's score
// bytes (its node and column follow when all lanes have one to decode, in kept_code) and kped
// the byte.
template <typename Word>
__device__ __forceinline__ int compact_kept(const KParams &p, const Regions<Word> &R,
                                            const LevelView<Word> &V, int thr, int q, int pos,
                                            int eq)
{
    return compact_bytes(p, R.score, p.lay.rsize[RG_SCORE],
                         (int64_t)(V.s_lo - V.cs0) * V.stride, (int64_t)(V.s_hi - V.cs0) * V.stride,
                         thr, q, pos, eq, INT_MAX, [&](int at, int idx, int v) {
                             FG_AT(R.klist, at, FG_N(int32_t, p.lay.rsize[RG_KLIST])) = idx;
                             FG_AT(R.kped, at, FG_N(int32_t, p.lay.rsize[RG_KPED])) = v;
                         });
}

// (parent slot << kSelShift) | j of score byte idx.
template <typename Word>
__device__ __forceinline__ int kept_code(const KParams &p, const Regions<Word> &R,
                                         const LevelView<Word> &V, int idx)
{
    const uint32_t row = (uint32_t)idx / (uint32_t)V.stride;
    const int j = (int)FG_AT(R.act, (uint32_t)idx - row * (uint32_t)V.stride, FG_N(uint16_t, p.lay.rsize[RG_ACT]));
    return ((V.cs0 + (int)row) << kSelShift) | j;
}

// Region pointers of a team from a region -> base address function.
template <typename Word, typename F>
__device__ __forceinline__ Regions<Word> make_regions(F base)
{
    Regions<Word> R;
    R.hist = (int32_t *)base(RG_HIST);
    R.alpha2 = (int32_t *)base(RG_ALPHA2);
    R.crow = (int32_t *)base(RG_CROW);
    R.a2t = (Word *)base(RG_A2T);
    R.l2t = (Word *)base(RG_L2T);
    R.sbase = (int32_t *)base(RG_SBASE);
    R.ped0 = (int32_t *)base(RG_PED0);
    R.ped1 = (int32_t *)base(RG_PED1);
    R.sel = (int32_t *)base(RG_SEL);
    R.selped = (int32_t *)base(RG_SELPED);
    R.klist = (int32_t *)base(RG_KLIST);
    R.kped = (int32_t *)base(RG_KPED);
    R.noff = (int32_t *)base(RG_NOFF);
    R.nbr = (int32_t *)base(RG_NBR);
    R.img0 = (Word *)base(RG_IMG0);
    R.img1 = (Word *)base(RG_IMG1);
    R.P = (Word *)base(RG_P);
    R.PL = (Word *)base(RG_PL);
    R.score = base(RG_SCORE);
    R.et0 = base(RG_ET0);
    R.et1 = base(RG_ET1);
    R.chist = (int32_t *)base(RG_CHIST);
    R.map0 = base(RG_MAP0);
    R.map1 = base(RG_MAP1);
    R.imgl = (Word *)base(RG_IMGL);
    return R;
}

// The regions that every layout keeps in shared memory: histogram rows, active columns and
// their records, and the used-by-all mask. Taken from the shared window directly, their accesses (the
// histogram's increments above all) need no generic addressing.
template <typename Word>
__device__ __forceinline__ void smem_regions(const KParams &p, Regions<Word> &R, uint8_t *smem)
{
    R.hist = (int32_t *)(smem + p.lay.off[RG_HIST]);
    R.act = (uint16_t *)(smem + p.lay.off[RG_ACT]);
    R.allm = (uint32_t *)(smem + p.lay.off[RG_ALL]);
    R.rec = smem + p.lay.off[RG_REC];
}

// A team's regions from the layout alone: what the kernels below build, with every base chosen
// by the layout's masks.
template <typename Word, bool CL>
__device__ __forceinline__ Regions<Word> team_regions(const KParams &p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const unsigned team = CL ? blockIdx.x / cluster_size() : blockIdx.x;
    uint8_t *gs = p.gscratch + (int64_t)team * p.lay.slice_bytes;
    uint8_t *gc = CL ? gs + p.lay.cta_off + (int64_t)cluster_rank() * p.lay.cta_bytes : gs;
    Regions<Word> R = make_regions<Word>([&](int r) -> uint8_t * {
        if ((p.lay.smem_mask >> r) & 1u) return smem + p.lay.off[r];
        return (CL && ((p.lay.cta_mask >> r) & 1u) ? gc : gs) + p.lay.off[r];
    });
    smem_regions(p, R, smem);
    return R;
}

// What the exact selection's functions know of level i (L nodes, nact columns in rows of `stride`
// bytes). They build the team's regions and the warp's view of the level anew: handed over by
// reference, both would live in the caller's local memory.
struct ExactLevel {
    int i, L, nact, stride, B, n2, nw;
    bool table;   // rows of neighbour counts are kept
};

template <int W, typename Word, bool CL>
__device__ __forceinline__ LevelView<Word> exact_view(const KParams &p, const Regions<Word> &R,
                                                      const Team<CL> &tm, const ExactLevel &x)
{
    LevelView<Word> V;
    const bool odd = x.i & 1;   // the beam buffers alternate
    V.cs0 = CL ? (int)((int64_t)(tm.warp - (int)(threadIdx.x >> 5)) * x.L / tm.NW) : 0;
    V.ioff = V.cs0;
    V.imgw = CL ? R.imgl : odd ? R.img1 : R.img0;
    V.nimg = FG_N(Word, p.lay.rsize[CL ? RG_IMGL : RG_IMG0]);
    V.crow = R.crow + (odd ? p.lay.n2s : 0);
    V.s_lo = (int)((int64_t)tm.warp * x.L / tm.NW);
    V.s_hi = (int)((int64_t)(tm.warp + 1) * x.L / tm.NW);
    V.nact = x.nact;
    V.stride = x.stride;
    if (W >= 8) {
        V.et = x.table ? (odd ? R.et0 : R.et1) : nullptr;
        V.map = (const uint16_t *)(odd ? R.map1 : R.map0);
        V.mt = p.lay.mrow / (int64_t)sizeof(uint16_t);
        V.n0 = FG_AT(R.noff, x.i, FG_N(int32_t, p.lay.rsize[RG_NOFF]));
        V.deg = FG_AT(R.noff, x.i + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) - V.n0;
    }
    return V;
}

// Exact selection, first part, for a K-th PED past the histogram window or below a guessed
// anchor: the level is scored again over coarser, then finer PED windows until the K-th PED is
// known. Returns the score byte of the K-th PED, the successors below it, and what added to a byte
// gives its PED (byte 0: below the last window). The bytes and the histogram rows are those of
// the last pass.
template <int W, typename Word, int BK, bool CL>
__device__ __noinline__ int4 rescore_exact(const KParams &p, const ExactLevel x, int newL, int anchor)
{
    const Team<CL> tm;
    const Regions<Word> R = team_regions<Word, CL>(p);
    const LevelView<Word> V = exact_view<W, Word, CL>(p, R, tm, x);
    const int nwl = (int)blockDim.x >> 5, lw = (int)threadIdx.x >> 5;
    int32_t *hrow = R.hist + lw * kBuckets;
    const int32_t *htot = R.hist + nwl * kBuckets;
    // windows of 127 buckets, each 64 times as wide as the one before, until one holds the K-th
    // PED (PEDs are below 2^31, so a bucket width of 2^30 does); then 64 buckets of 1/64 the
    // width inside the bucket found
    int sh = 0, pre = 0, thr = 0, below = 0, first;
    bool down = false;
    for (int pass = 0; pass < 12; ++pass) {   // up to 30, then to 0
        sh += down ? -6 : 6;
        tm.sync();
        score_exact<W, Word, BK>(p, R, V, x.B, x.n2, x.nw, anchor, sh, hrow);
        prefix_buckets<CL>(p, R, tm);
        // (the last pass counts the successors below its window as well)
        find_threshold(p, htot, sh > 0 ? newL - pre : newL, thr, below, first);
        if (sh == 0) break;
        if (thr < kScoreMax) {
            down = true;
            pre += below;
            anchor += thr << sh;
        }
    }
    return make_int4(thr, below, anchor - 1, 0);
}

// Exact selection, second part: entries [kbeg, kbeg + kcnt) of the kept lists hold this warp's
// compacted children (index and score byte); their codes and PEDs follow, and the team orders
// all newL by (PED, enumeration order). low: byte 0 stands for any PED below.
template <int W, typename Word, int BK, bool CL>
__device__ __noinline__ void order_exact(const KParams &p, const ExactLevel x, int newL, int anchor,
                                         bool low, int kbeg, int kcnt)
{
    const Team<CL> tm;
    const Regions<Word> R = team_regions<Word, CL>(p);
    const LevelView<Word> V = exact_view<W, Word, CL>(p, R, tm, x);
    const int tid = tm.tid, T = tm.T, lane = threadIdx.x & 31;
#define NKP FG_N(int32_t, p.lay.rsize[RG_KPED])
#define NKL FG_N(int32_t, p.lay.rsize[RG_KLIST])
#define NSE FG_N(int32_t, p.lay.rsize[RG_SEL])
#define NSP FG_N(int32_t, p.lay.rsize[RG_SELPED])
    for (int a = kbeg + lane; a < kbeg + kcnt; a += 32) {
        const int code = kept_code<Word>(p, R, V, FG_AT(R.klist, a, NKL)), v = FG_AT(R.kped, a, NKP);
        FG_AT(R.klist, a, NKL) = code;
        FG_AT(R.kped, a, NKP) = low && v == 0 ? succ_ped<W, Word>(p, R, V, x.B, code >> kSelShift, code & ((1 << kSelShift) - 1))
                                              : anchor + v;
    }
    tm.sync();
    // order by (PED, enumeration order); klist is in enumeration order and its codes are
    // increasing, so (kped, klist) is that key
    if (newL <= 2048) {
        for (int a = tid; a < newL; a += T) {
            const int pa = FG_AT(R.kped, a, NKP);
            int rank = 0;
            for (int b = 0; b < newL; ++b) {
                const int pb = FG_AT(R.kped, b, NKP);
                rank += (pb < pa) || (pb == pa && b < a);
            }
            FG_AT(R.sel, rank, NSE) = FG_AT(R.klist, a, NKL);
            FG_AT(R.selped, rank, NSP) = pa;
        }
        return;
    }
    // large beams: bitonic sort of (kped, klist) in place. Every comparator puts the smaller
    // key at the lower index (each merge starts with a reversed-partner stage), so entries
    // past newL act as +infinity padding up to the next power of two and are never touched.
    int N = 1;
    while (N < newL) N <<= 1;
    auto cmpswap = [&](int i, int j) {
        if (j >= newL) return;
        const int pi = FG_AT(R.kped, i, NKP), pj = FG_AT(R.kped, j, NKP);
        const int li = FG_AT(R.klist, i, NKL), lj = FG_AT(R.klist, j, NKL);
        if (pj < pi || (pj == pi && lj < li)) {
            FG_AT(R.kped, i, NKP) = pj;
            FG_AT(R.kped, j, NKP) = pi;
            FG_AT(R.klist, i, NKL) = lj;
            FG_AT(R.klist, j, NKL) = li;
        }
    };
    for (int size = 2; size <= N; size <<= 1) {
        const int half = size >> 1;
        for (int t = tid; t < N / 2; t += T) {
            const int blk = t / half, off = t - blk * half;
            cmpswap(blk * size + off, blk * size + size - 1 - off);
        }
        tm.sync();
        for (int stride = half >> 1; stride > 0; stride >>= 1) {
            for (int t = tid; t < N / 2; t += T) {
                const int blk = t / stride, off = t - blk * stride;
                const int i = blk * 2 * stride + off;
                cmpswap(i, i + stride);
            }
            tm.sync();
        }
    }
    for (int a = tid; a < newL; a += T) {
        FG_AT(R.sel, a, NSE) = FG_AT(R.klist, a, NKL);
        FG_AT(R.selped, a, NSP) = FG_AT(R.kped, a, NKP);
    }
#undef NKP
#undef NKL
#undef NSE
#undef NSP
}

// BK: edge-label planes known at compile time: 0 (unlabelled), 2 (exactly two planes), or
// 8 (any count up to 8, read from the layout)
// CL: the team is a whole cluster (S then lives in global scratch); regions the team
// writes are global, the read-only target-graph tables are per CTA in shared memory.
template <int W, typename MapT, typename Word, int BK, bool CL, typename TS>
__device__ __forceinline__ void solve_pair(const KParams &p, const Regions<Word> R, TS &S,
                                           const int pair)
{
    constexpr int WB = 8 * (int)sizeof(Word);
    const Team<CL> tm;
    const int tid = tm.tid, lane = threadIdx.x & 31, warp = tm.warp;
    const int T = tm.T, NW = tm.NW;
    // CTA-local threads (staging of the per-CTA read-only tables)
    const int ltid = threadIdx.x, LT = blockDim.x;
    const int g1 = FG_AT(p.pairs, 2 * pair, 2 * p.n_pairs);
    const int g2 = FG_AT(p.pairs, 2 * pair + 1, 2 * p.n_pairs);
    const GraphMeta m1 = FG_AT(p.gmeta, g1, p.n_graphs), m2 = FG_AT(p.gmeta, g2, p.n_graphs);
    const int n1 = m1.n, n2 = m2.n, W1 = m1.W, W2 = m2.W;
    const int K = p.kpp ? FG_AT(p.kpp, pair, p.n_pairs) : p.K;
    const int Bc = BK == 0 ? 0 : (BK == 2 ? 2 : p.lay.B);   // planes of the class
    const int N2S = p.lay.n2s;
    const int KM = p.lay.kloc;   // node slots of the P / PL / sbase tables this CTA indexes
    constexpr int W32 = W * (int)sizeof(Word) / 4;   // 32-bit words of a bitset
    const int nwl = (int)blockDim.x >> 5;            // warps of this CTA
    const int nw = min(W, max(1, (n2 + WB - 1) / WB));   // words this pair's bitsets use
    int32_t *hrow = R.hist + (threadIdx.x >> 5) * kBuckets;   // this warp's histogram row
    const int32_t *htot = R.hist + nwl * kBuckets;            // team totals (prefix_buckets)
    const int64_t mrow = p.lay.mrow;
    const MapT DEL = (MapT)~(MapT)0;
    const CostModel c = p.cost;
    const int hwin = p.hwin;     // PEDs a kept list may span without the exact selection
    const bool fold_ie = (c.eins == c.edel);
    // lane-constant masks: lane b answers for histogram bucket b
    unsigned lanebit[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) lanebit[k] = ((lane >> k) & 1) ? 0xffffffffu : 0u;
#ifdef FASTGED_PHASE_TIMERS
    long long ph[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    long long ph_last = clock64();
#endif

    // stage g2: transposed adjacency and label planes, vertex labels; g1 degrees (these
    // tables are per CTA)
    bool lab = false;   // some edge of the pair has a label
    {
        const uint64_t *adj2 = p.adj + m2.adj_off;
        for (int idx = ltid; idx < W * n2; idx += LT) {
            const int w = idx / n2, u = idx - w * n2;
            const int w64 = (w * WB) >> 6, sh = (w * WB) & 63;
            FG_AT(R.a2t, w * N2S + u, FG_N(Word, p.lay.rsize[RG_A2T])) =
                (w64 < W2) ? (Word)(FG_AT(adj2, (int64_t)u * W2 + w64, p.adj_words - m2.adj_off) >> sh)
                           : (Word)0;
        }
        for (int b = 0; b < Bc; ++b) {
            const uint64_t *pl2 = p.planes + m2.plane_off + (int64_t)b * n2 * W2;
            for (int idx = ltid; idx < W * n2; idx += LT) {
                const int w = idx / n2, u = idx - w * n2;
                const int w64 = (w * WB) >> 6, sh = (w * WB) & 63;
                const Word l = (w64 < W2) ? (Word)(FG_AT(pl2, (int64_t)u * W2 + w64,
                                                         p.plane_words - m2.plane_off - (int64_t)b * n2 * W2) >> sh)
                                          : (Word)0;
                FG_AT(R.l2t, (b * W + w) * N2S + u, FG_N(Word, p.lay.rsize[RG_L2T])) = l;
                lab |= l != (Word)0;
            }
        }
        for (int u = ltid; u < n2; u += LT)
            FG_AT(R.alpha2, u, FG_N(int32_t, p.lay.rsize[RG_ALPHA2])) = FG_AT(p.vlab, m2.lab_off + u, p.n_vlab);
        // column n2 of the target tables is the deletion v_i -> eps: no g2 neighbours, so the
        // substitution formula scores it with the deletion's edge costs (see succ_ped)
        for (int w = ltid; w < W; w += LT) FG_AT(R.a2t, w * N2S + n2, FG_N(Word, p.lay.rsize[RG_A2T])) = (Word)0;
        for (int x = ltid; x < Bc * W; x += LT) FG_AT(R.l2t, x * N2S + n2, FG_N(Word, p.lay.rsize[RG_L2T])) = (Word)0;
        // S1 cost row of level 0 (the row of level i + 1 is written during level i)
        if (n1 > 0) {
            const int a10 = FG_AT(p.vlab, m1.lab_off, p.n_vlab);
            for (int u = ltid; u <= n2; u += LT)
                FG_AT(R.crow, u, FG_N(int32_t, p.lay.rsize[RG_CROW])) =
                    u < n2 ? ((FG_AT(p.vlab, m2.lab_off + u, p.n_vlab) != a10) ? c.vsub : 0) : c.vdel;
        }
        // number of neighbours v_k of v_i with k < i
        for (int v = ltid; v < n1; v += LT) {
            const int64_t row = m1.adj_off + (int64_t)v * W1;
            int d = 0;
            for (int w = 0; w < W1; ++w)
                d += __popcll(FG_AT(p.adj, row + w, p.adj_words) & low_mask(v, w));
            FG_AT(R.noff, v + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) = d;
        }
        if (ltid == 0) FG_AT(R.noff, 0, FG_N(int32_t, p.lay.rsize[RG_NOFF])) = 0;
        for (int x = ltid; x < W32; x += LT) FG_AT(R.allm, x, FG_N(uint32_t, p.lay.rsize[RG_ALL])) = ~0u;
        // root node: empty lambda, R_V2 = V2, PED 0
        for (int w = tid; w < W; w += T) FG_AT(R.img0, w, FG_N(Word, p.lay.rsize[RG_IMG0])) = (Word)0;
        if (tid == 0) FG_AT(R.ped0, 0, FG_N(int32_t, p.lay.rsize[RG_PED0])) = 0;
    }
    __syncthreads();
    // prior-neighbour lists of g1: nbr[noff[i] .. noff[i+1]) = k | (edge label << 16)
    if (ltid < 32) {
        int carry = 0;
        for (int v0 = 0; v0 < n1; v0 += 32) {
            const int v = v0 + lane;
            const int d = v < n1 ? FG_AT(R.noff, v + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) : 0;
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (v < n1) FG_AT(R.noff, v + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) = carry + incl;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();
    for (int v = ltid; v < n1; v += LT) {
        const int64_t row = m1.adj_off + (int64_t)v * W1;
        const int64_t pl = m1.plane_off + (int64_t)v * W1;
        const int64_t pstep = (int64_t)n1 * W1;
        int o = FG_AT(R.noff, v, FG_N(int32_t, p.lay.rsize[RG_NOFF]));
        for (int w = 0; w < W1; ++w) {
            uint64_t bits = FG_AT(p.adj, row + w, p.adj_words) & low_mask(v, w);
            while (bits) {
                const int t = __ffsll((long long)bits) - 1;
                bits &= bits - 1ull;
                int el = 0;
                for (int b = 0; b < Bc; ++b)
                    el |= (int)((FG_AT(p.planes, pl + b * pstep + w, p.plane_words) >> t) & 1ull) << b;
                lab |= el != 0;
                FG_AT(R.nbr, o++, FG_N(int32_t, p.lay.rsize[RG_NBR])) = (w * 64 + t) | (el << 16);
            }
        }
    }
    // a pair without edge labels in a labelled batch pays nothing for the planes
    const int B = BK == 0 ? 0 : (__syncthreads_or(lab ? 1 : 0) ? Bc : 0);
    // Neighbour counts kept per node (score_table): for eight and more words, without edge
    // labels, when v_i has eight prior neighbours at most on average (each costs about one
    // addition per column, the counts replace 2 W popcounts) and no count can pass 127.
    bool table = false;
    if (W >= 8) {
        bool over = m1.m > 8 * n1;
        for (int u = ltid; u < n2; u += LT) {
            int d = 0;
            for (int w = 0; w < nw; ++w) d += popcw(FG_AT(R.a2t, w * N2S + u, FG_N(Word, p.lay.rsize[RG_A2T])));
            over |= d > 127;
        }
        for (int v = ltid; v < n1; v += LT)
            over |= FG_AT(R.noff, v + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) -
                        FG_AT(R.noff, v, FG_N(int32_t, p.lay.rsize[RG_NOFF])) > 127;
        table = !__syncthreads_or(over ? 1 : 0) && B == 0;
    }
    uint8_t *ecur = R.et0, *enext = R.et1;   // the parents' counts, and this level's
    long long nevals = 0;
    int L = 1, rise = 0;
    // current / next beam buffers, swapped after every level
    uint8_t *mapc = R.map0, *mapn = R.map1;
    Word *imgc = R.img0, *imgn = R.img1;
    int32_t *pedc = R.ped0, *pedn = R.ped1;
    int32_t *crc = R.crow, *crn = R.crow + N2S;   // S1 cost rows of this level and the next
    // elements of the beam buffers (both buffers of a pair have the same size), the cost-row
    // halves, the P / PL / sbase tables, the maps in MapT and 16-byte units
#define NIMG FG_N(Word, p.lay.rsize[RG_IMG0])
#define NPED FG_N(int32_t, p.lay.rsize[RG_PED0])
#define NSW ((int64_t)(sizeof(S.wbest) / sizeof(S.wbest[0])))   // warps the team scalars hold
#define NP FG_N(Word, p.lay.rsize[RG_P])
#define NMAPT FG_N(MapT, p.lay.rsize[RG_MAP0])
#define NMAP16 FG_N(uint4, p.lay.rsize[RG_MAP0])
#define NIMGW (CL ? FG_N(Word, p.lay.rsize[RG_IMGL]) : NIMG)
    tm.sync();
    PHASE_MARK(0);

    for (int i = 0; i < n1; ++i) {
        const int n0 = FG_AT(R.noff, i, FG_N(int32_t, p.lay.rsize[RG_NOFF])), deg = FG_AT(R.noff, i + 1, FG_N(int32_t, p.lay.rsize[RG_NOFF])) - n0;
        // 64-bit products: K can be 2^20 and a team 256 warps
        const int s_lo = (int)((int64_t)warp * L / NW), s_hi = (int)((int64_t)(warp + 1) * L / NW);
        // node tables the warp prepares and evaluates are indexed from cs0: 0 for a one-CTA
        // team; for a cluster, the first node of this CTA (its P, PL, sbase and score bytes
        // are CTA-local and its nodes' Img rows are staged into shared memory)
        int cs0 = 0, ioff = 0, cs1 = L;
        const Word *imgw = imgc;
        if (CL) {
            const int r0 = (int)cluster_rank() * nwl;
            cs0 = (int)((int64_t)r0 * L / NW);
            cs1 = (int)((int64_t)(r0 + nwl) * L / NW);
            imgw = R.imgl;
            ioff = cs0;
        }
        // target vertices that every node of this CTA uses: the beam's nodes share most of
        // their ancestors, so the columns left are little more than a node's own successors.
        // A thread reads one 32-bit word index of every row it visits (W32 divides the warp).
        {
            uint32_t am = ~0u;
            const int64_t n32 = (int64_t)(cs1 - cs0) * W32, b32 = (int64_t)cs0 * W32;
            for (int64_t x = ltid; x < n32; x += LT) {
                const uint32_t v = FG_AT((const uint32_t *)imgc, b32 + x, NIMG * (int)(sizeof(Word) / 4));
                if (CL) FG_AT((uint32_t *)R.imgl, x, NIMGW * (int)(sizeof(Word) / 4)) = v;
                am &= v;
            }
#pragma unroll
            for (int o = 16; o >= W32; o >>= 1) am &= __shfl_xor_sync(0xffffffffu, am, o);
            if (table) am = 0u;   // rows of counts keep every column
            if (lane < W32) atomicAnd(&FG_AT(R.allm, lane, FG_N(uint32_t, p.lay.rsize[RG_ALL])), am);
        }
        __syncthreads();
        // active columns, increasing: the vertices not used by all, and the deletion n2. A
        // cluster CTA without nodes (levels of fewer nodes than CTAs) has no such list: its
        // mask is still all ones, its count means nothing, and score_exact does not read them
        int nact = n2 + 1, stride;
        {
            using Rec = ColRec<Word, (BK == 8 ? kMaxB : BK)>;
            constexpr int NPL = BK == 8 ? kMaxB : BK;
            Word *jm = (Word *)((uint8_t *)R.rec + p.lay.jm_off);   // one-hot vertex bits
#define NJM FG_N(Word, p.lay.rsize[RG_REC] - p.lay.jm_off)
            for (int w = 0; w < W32; ++w) nact -= __popc(FG_AT(R.allm, w, FG_N(uint32_t, p.lay.rsize[RG_ALL])));
            for (int j = ltid; j <= n2; j += LT) {
                int pos = j;
                bool fr = true;
                if (cs1 > cs0) {
                    for (int w = 0; w < W32; ++w) {
                        const uint32_t m = FG_AT(R.allm, w, FG_N(uint32_t, p.lay.rsize[RG_ALL]));
                        if (w < (j >> 5)) pos -= __popc(m);
                        if (w == (j >> 5)) {
                            pos -= __popc(m & ((1u << (j & 31)) - 1u));
                            fr = !((m >> (j & 31)) & 1u);
                        }
                    }
                    if (fr) {
                        FG_AT(R.act, pos, FG_N(uint16_t, p.lay.rsize[RG_ACT])) = (uint16_t)j;
                        if (W == 1) {
                            Rec c;
                            c.a2 = FG_AT(R.a2t, j, FG_N(Word, p.lay.rsize[RG_A2T]));
#pragma unroll
                            for (int b = 0; b < NPL; ++b)
                                c.l[b] = b < B ? FG_AT(R.l2t, b * N2S + j, FG_N(Word, p.lay.rsize[RG_L2T])) : (Word)0;
                            c.crow = FG_AT(crc, j, N2S);
                            FG_AT((Rec *)R.rec, pos, FG_N(Rec, p.lay.jm_off)) = c;
                            FG_AT(jm, pos, NJM) = j < n2 ? (Word)1 << (j % WB) : (Word)0;
                        }
                    }
                }
            }
            stride = W >= 8 && table ? (nact + 7) / 8 * 8 : nact;
            // single-word rows: whole quads of columns, an odd number of them; the columns
            // past the active ones score past every bucket
            if (W == 1) {
                stride = ((nact + 3) / 4 | 1) * 4;
                for (int a = nact + ltid; cs1 > cs0 && a < stride; a += LT) {
                    Rec c = {};
                    c.crow = 1 << 29;
                    FG_AT((Rec *)R.rec, a, FG_N(Rec, p.lay.jm_off)) = c;
                    FG_AT(jm, a, NJM) = (Word)0;
                }
            }
        }
#undef NJM
        LevelView<Word> V;
        V.imgw = imgw;
        V.crow = crc;
        V.ioff = ioff;
        V.cs0 = cs0;
        V.s_lo = s_lo;
        V.s_hi = s_hi;
        V.nact = nact;
        V.stride = stride;
        V.nimg = NIMGW;
        // anchor of the level's PED offsets. No child's PED is below the best parent's, but in
        // dense graphs all lie far above it, at a distance that changes little from one level
        // to the next: the window starts kAnchorSlack below where the last level's began. If
        // that is too high, bucket 0 is not empty and the exact selection takes over.
        const int A0 = FG_AT(pedc, 0, NPED);
        const int A = A0 + max(0, rise - kAnchorSlack);
        const bool last_b = p.variant == 1 && i == n1 - 1;
        for (int b = lane; b < kBuckets; b += 32) FG_AT(hrow, b, kBuckets) = 0;
        __syncthreads();
        PHASE_MARK(7);
        // ---- S1 + S2 per-node vectors, S3 scores and their histogram -------------------
        int kw = 0;          // successors of this lane's nodes so far
        for (int g0 = s_lo; g0 < s_hi; g0 += 32) {
            const int ng = min(32, s_hi - g0);
            const int s = g0 + lane;
            constexpr int NPL = BK == 8 ? kMaxB : (BK == 2 ? 2 : 1);
            Word pr = (Word)0, plr[NPL], imr = (Word)0;   // single-word node vectors
            int nbase = 0;
            TableNode tn = {0, 0, 0, {0xffffffffu, 0xffffffffu}};
#pragma unroll
            for (int b = 0; b < NPL; ++b) plr[b] = (Word)0;
            if (lane < ng) {
                // S2: P = images of the substituted g1 neighbours of v_i (their edge labels in
                // bit-planes PL at the image positions); dcnt = deleted neighbours
                const int64_t Ps = (int64_t)(s - cs0) * W;   // this node's row of R.P
                const int64_t ms = (int64_t)s * (mrow / (int64_t)sizeof(MapT));   // its map row
                int dcnt = 0;
                if (W > 1) {
#pragma unroll
                    for (int w = 0; w < W; ++w) FG_AT(R.P, Ps + w, NP) = (Word)0;
                    for (int b = 0; b < B; ++b)
                        for (int w = 0; w < W; ++w) FG_AT(R.PL, ((int64_t)b * KM + (s - cs0)) * W + w, FG_N(Word, p.lay.rsize[RG_PL])) = (Word)0;
                }
                // several neighbours per step: list and map loads first, then the bits
                constexpr int NU = W > 1 ? 8 : 4;
                for (int t0 = 0; t0 < deg; t0 += NU) {
                    int e[NU];
                    MapT phi[NU];
#pragma unroll
                    for (int u = 0; u < NU; ++u) e[u] = t0 + u < deg ? FG_AT(R.nbr, n0 + t0 + u, FG_N(int32_t, p.lay.rsize[RG_NBR])) : -1;
#pragma unroll
                    for (int u = 0; u < NU; ++u)
                        phi[u] = e[u] >= 0 ? FG_AT((const MapT *)mapc, ms + (e[u] & 0xffff), NMAPT) : DEL;
#pragma unroll
                    for (int u = 0; u < NU; ++u) {
                        const bool sub = phi[u] != DEL;
                        dcnt += (e[u] >= 0 && !sub) ? 1 : 0;
                        if (W >= 8 && t0 == 0 && u < 4)
                            tn.ph[u >> 1] = (tn.ph[u >> 1] & (u & 1 ? 0xffffu : 0xffff0000u)) |
                                            (uint32_t)(uint16_t)phi[u] << (16 * (u & 1));
                        if (W == 1) {
                            const Word pb = sub ? (Word)1 << ((int)phi[u] % WB) : (Word)0;
                            pr |= pb;
#pragma unroll
                            for (int b = 0; b < NPL; ++b)
                                if (b < B && ((e[u] >> (16 + b)) & 1)) plr[b] |= pb;
                        } else if (sub) {
                            const int pw = (int)phi[u] / WB;
                            const Word pb = (Word)1 << ((int)phi[u] % WB);
                            FG_AT(R.P, Ps + pw, NP) |= pb;
                            for (int b = 0; b < B; ++b)
                                if ((e[u] >> (16 + b)) & 1) FG_AT(R.PL, ((int64_t)b * KM + (s - cs0)) * W + pw, FG_N(Word, p.lay.rsize[RG_PL])) |= pb;
                        }
                    }
                }
                if (W == 1) {
                    FG_AT(R.P, Ps, NP) = pr;
#pragma unroll
                    for (int b = 0; b < NPL; ++b)
                        if (b < B) FG_AT(R.PL, (int64_t)b * KM + (s - cs0), FG_N(Word, p.lay.rsize[RG_PL])) = plr[b];
                }
                nbase = FG_AT(pedc, s, NPED) + c.edel * dcnt;
                FG_AT(R.sbase, s - cs0, FG_N(int32_t, p.lay.rsize[RG_SBASE])) = nbase;
                const int64_t im = (int64_t)(s - ioff) * W;   // this node's Img row in imgw
                int used = 0;
#pragma unroll
                for (int w = 0; w < W; ++w) used += popcw(FG_AT(imgw, im + w, NIMGW));
                kw += n2 - used + 1;   // free g2 vertices (R_V2) and the deletion
                if (W == 1) imr = FG_AT(imgw, im, NIMGW);
                if (W >= 8 && table) {
                    tn.code = i > 0 ? FG_AT(R.sel, s, FG_N(int32_t, p.lay.rsize[RG_SEL])) : 0;
                    tn.base = nbase - A;
                    tn.nimg = deg - dcnt;
                }
            }
            __syncwarp();   // the group's node vectors (P, PL, base) are in place
            PHASE_MARK(5);
            if (W == 1 && !last_b) {
                const int qs = ng > 16 ? 0 : ng > 8 ? 1 : ng > 4 ? 2 : ng > 2 ? 3 : ng > 1 ? 4 : 5;
                const int nd = lane >> qs;   // this lane's node of the group
                if (qs) {
                    pr = __shfl_sync(0xffffffffu, pr, nd);
                    imr = __shfl_sync(0xffffffffu, imr, nd);
                    nbase = __shfl_sync(0xffffffffu, nbase, nd);
#pragma unroll
                    for (int b = 0; b < NPL; ++b) plr[b] = __shfl_sync(0xffffffffu, plr[b], nd);
                }
                const int r = lane & ((1 << qs) - 1);
                if (fold_ie) score_quads<Word, BK, true>(p, R, V, B, g0 + nd - cs0, nd < ng, r, qs, imr, pr, plr, nbase - A, hrow);
                else score_quads<Word, BK, false>(p, R, V, B, g0 + nd - cs0, nd < ng, r, qs, imr, pr, plr, nbase - A, hrow);
                PHASE_MARK(1);
            } else if (W >= 8 && table && !last_b) {
                const MapT *mp = (const MapT *)mapc;
                const int64_t mt = mrow / (int64_t)sizeof(MapT);
                if (fold_ie) score_table<W, MapT, Word, true>(p, R, V, n2, g0, ng, tn, mp, mt, n0, deg, ecur, enext, i == 0, hrow);
                else score_table<W, MapT, Word, false>(p, R, V, n2, g0, ng, tn, mp, mt, n0, deg, ecur, enext, i == 0, hrow);
                PHASE_MARK(1);
            } else if (!last_b) {
                if (fold_ie) score_nodes<W, Word, BK, true, false>(p, R, V, B, n2, nw, g0, ng, A, 0, hrow);
                else score_nodes<W, Word, BK, false, false>(p, R, V, B, n2, nw, g0, ng, A, 0, hrow);
                PHASE_MARK(1);
            }
        }
        kw = warp_sum(kw);   // (the scoring's last increments are done: [127] is overwritten)
        __syncwarp();
        if (lane == 0) FG_AT(hrow, kScoreMax, kBuckets) = kw;
        if (ltid < W32) FG_AT(R.allm, ltid, FG_N(uint32_t, p.lay.rsize[RG_ALL])) = ~0u;   // for the next level
        prefix_buckets<CL>(p, R, tm);
        const int total = FG_AT(htot, kScoreMax, kBuckets);   // successors of the level
        PHASE_MARK(2);

        if (last_b) {
            // variant B: every successor of the last level is completed (insertions of the
            // free g2 vertices and their edges) and the least (total, PED, enumeration order)
            // wins. Lanes <-> active columns; per node: nimg = |Img|, e2 = g2 edges inside Img.
            unsigned long long key = ~0ull;   // total << 32 | PED
            int code = INT_MAX;               // parent slot << kSelShift | j
            for (int s = s_lo; s < s_hi; ++s) {
                const int64_t im = (int64_t)(s - ioff) * W;   // the node's Img row
                int nimg = 0, acc = 0;
                for (int u = lane; u < n2; u += 32) {
                    if ((FG_AT(imgw, im + u / WB, NIMGW) >> (u % WB)) & (Word)1) {
                        ++nimg;
#pragma unroll
                        for (int w = 0; w < W; ++w)
                            acc += popcw((Word)(FG_AT(R.a2t, w * N2S + u, FG_N(Word, p.lay.rsize[RG_A2T])) &
                                                FG_AT(imgw, im + w, NIMGW)));
                    }
                }
                nimg = warp_sum(nimg);
                acc = warp_sum(acc) / 2;
                for (int a = lane; a < nact; a += 32) {
                    const int j = (int)FG_AT(R.act, a, FG_N(uint16_t, p.lay.rsize[RG_ACT]));
                    if (j < n2 && ((FG_AT(imgw, im + j / WB, NIMGW) >> (j % WB)) & (Word)1)) continue;
                    int e2 = acc;
#pragma unroll
                    for (int w = 0; w < W; ++w)   // none for the deletion's empty column
                        e2 += popcw((Word)(FG_AT(R.a2t, w * N2S + j, FG_N(Word, p.lay.rsize[RG_A2T])) &
                                           FG_AT(imgw, im + w, NIMGW)));
                    const int d = succ_ped<W, Word>(p, R, V, B, s, j);
                    const long long tt = (long long)d + (long long)c.vins * (n2 - nimg - (j < n2 ? 1 : 0)) +
                                         (long long)c.eins * (m2.m - e2);
                    const unsigned long long kk = ((unsigned long long)tt << 32) | (unsigned)d;
                    const int cc = (s << kSelShift) | j;
                    if (kk < key || (kk == key && cc < code)) {
                        key = kk;
                        code = cc;
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
                const int c2 = __shfl_xor_sync(0xffffffffu, code, o);
                if (k2 < key || (k2 == key && c2 < code)) {
                    key = k2;
                    code = c2;
                }
            }
            if (lane == 0) {
                FG_AT(S.wbest, warp, NSW) = key;
                FG_AT(S.wcode, warp, NSW) = code;
            }
            tm.sync();
            key = FG_AT(S.wbest, 0, NSW);
            code = FG_AT(S.wcode, 0, NSW);
            for (int w = 1; w < NW; ++w) {
                const unsigned long long k2 = FG_AT(S.wbest, w, NSW);
                const int c2 = FG_AT(S.wcode, w, NSW);
                if (k2 < key || (k2 == key && c2 < code)) {
                    key = k2;
                    code = c2;
                }
            }
            const int ws = code >> kSelShift, wj = code & ((1 << kSelShift) - 1);
            if (tid == 0) {
                FG_AT(p.out_cost, pair, p.n_pairs) = (int32_t)(key >> 32);
                if (p.out_nevals) FG_AT(p.out_nevals, pair, p.n_pairs) = nevals + 2LL * total;
            }
            const int64_t mb = (int64_t)ws * (mrow / (int64_t)sizeof(MapT));   // the winner's map row
            const int64_t om = FG_AT(p.map_off, pair, p.n_pairs);
            for (int k = tid; k < n1; k += T) {
                const MapT v = (k == i) ? ((wj < n2) ? (MapT)wj : DEL) : FG_AT((const MapT *)mapc, mb + k, NMAPT);
                FG_AT(p.out_map, om + k, p.map_total) = (v == DEL) ? -1 : (int32_t)v;
            }
            tm.sync();
            return;
        }

        // ---- S4 selection ---------------------------------------------------------
        const int newL = min(K, total);
        if (tid == 0) nevals += total;
        int thr, below, first;
        find_threshold(p, htot, newL, thr, below, first);
        const bool fits = A == A0 || first > 0;   // nothing below the anchor
        rise = A - A0 + (first < kScoreMax ? first : kScoreMax);
        // kept = every successor below the threshold bucket and the first q in it. Each warp
        // compacts its kept successors in enumeration order, then places them at their rank in
        // (PED, parent slot, j) order: position = #(smaller PED) + #(equal PED earlier); lane b
        // answers for bucket first + b. Kept sets past the window or over too many buckets go
        // through the exact selection instead.
        const bool known = fits && thr < kScoreMax;
        if (known && thr - first < hwin - 1) {
            const int q = newL - below;
            const bool in = first + lane <= thr;
            int incl = in ? FG_AT(htot, first + lane, kBuckets) : 0;
            const int tot = incl;
            const int mine = in ? FG_AT(hrow, first + lane, kBuckets) : 0;   // of earlier warps
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int bexcl = incl - tot;
            const int eq_before = __shfl_sync(0xffffffffu, mine, thr - first);
            const int lt_before = warp_sum(first + lane < thr ? mine : 0);
            const int kbeg = lt_before + min(q, eq_before);
            const int kcnt = compact_kept<Word>(p, R, V, thr, q, kbeg, eq_before);
            __syncwarp();
            PHASE_MARK(8);
            // kept of bucket first + lane before the warp's next 32
            int run = first + lane < thr ? mine : min(q, eq_before);
            for (int xb = 0; xb < kcnt; xb += 32) {
                const int x = kbeg + xb + lane;
                const bool v = xb + lane < kcnt;
                const int d = v ? FG_AT(R.kped, x, FG_N(int32_t, p.lay.rsize[RG_KPED])) - first : 0;
                const unsigned V32 = __ballot_sync(0xffffffffu, v);
                unsigned bb[5];
#pragma unroll
                for (int b = 0; b < 5; ++b) bb[b] = __ballot_sync(0xffffffffu, (d >> b) & 1);
                const int pos = __shfl_sync(0xffffffffu, bexcl, d) +
                                __shfl_sync(0xffffffffu, run, d) +
                                __popc(same_value_lanes(V32, bb, d) & lanemask_lt());
                if (v) {
                    FG_AT(R.sel, pos, FG_N(int32_t, p.lay.rsize[RG_SEL])) = kept_code<Word>(p, R, V, FG_AT(R.klist, x, FG_N(int32_t, p.lay.rsize[RG_KLIST])));
                    FG_AT(R.selped, pos, FG_N(int32_t, p.lay.rsize[RG_SELPED])) = A + first + d;
                }
                unsigned m = V32;
#pragma unroll
                for (int b = 0; b < 5; ++b) m &= ~(bb[b] ^ lanebit[b]);
                run += __popc(m);
            }
            PHASE_MARK(9);
        } else {
            const ExactLevel x = {i, L, nact, stride, B, n2, nw, W >= 8 && table};
            int anchor = A;
            if (!known) {
                const int4 found = rescore_exact<W, Word, BK, CL>(p, x, newL, fits ? A : A0);
                thr = found.x;
                below = found.y;
                anchor = found.z;
            }
            const int q = newL - below;
            int lt = 0;   // successors of earlier warps in the buckets below thr
            for (int b = lane; b < thr; b += 32) lt += FG_AT(hrow, b, kBuckets);
            lt = warp_sum(lt);
            const int eq = FG_AT(hrow, thr, kBuckets);
            const int kbeg = lt + min(q, eq);
            const int kcnt = compact_kept<Word>(p, R, V, thr, q, kbeg, eq);
            __syncwarp();
            order_exact<W, Word, BK, CL>(p, x, newL, anchor, !known, kbeg, kcnt);
            PHASE_MARK(10);
        }
        tm.sync();
        PHASE_MARK(6);

        // ---- kept children, in key order (slot = rank) -----------------------------
        {
            const int nvec = (int)((i * (int)sizeof(MapT) + 15) >> 4);
            const int64_t m16 = mrow >> 4, mt = mrow / (int64_t)sizeof(MapT);   // a map row in
                                                                                // 16 B / MapT units
            if (mrow <= 128) {
                for (int r = tid; r < newL; r += T) {
                    const int v = FG_AT(R.sel, r, FG_N(int32_t, p.lay.rsize[RG_SEL]));
                    const int s = v >> kSelShift, j = v & ((1 << kSelShift) - 1);
                    for (int t = 0; t < nvec; ++t)
                        FG_AT((uint4 *)mapn, r * m16 + t, NMAP16) = FG_AT((const uint4 *)mapc, s * m16 + t, NMAP16);
                    FG_AT((MapT *)mapn, r * mt + i, NMAPT) = (j < n2) ? (MapT)j : DEL;
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        Word x = FG_AT(imgc, (int64_t)s * W + w, NIMG);
                        if (j < n2 && j / WB == w) x |= (Word)1 << (j % WB);
                        FG_AT(imgn, (int64_t)r * W + w, NIMG) = x;
                    }
                    FG_AT(pedn, r, NPED) = FG_AT(R.selped, r, FG_N(int32_t, p.lay.rsize[RG_SELPED]));
                }
            } else if (!CL) {
                // long maps, one-CTA team: every thread takes (child, 16-byte vector) items
                // (the last vector of a child also carries its new entry i) and one more item
                // per child writes Img, the PED and entry i when it starts a new vector
                const int nb = i * (int)sizeof(MapT);
                const int per = nvec + 1;
                const int items = newL * per;
                for (int t = tid; t < items; t += T) {
                    const int r = t / per, v = t - r * per;
                    const int sv = FG_AT(R.sel, r, FG_N(int32_t, p.lay.rsize[RG_SEL]));
                    const int s = sv >> kSelShift, j = sv & ((1 << kSelShift) - 1);
                    const MapT val = (j < n2) ? (MapT)j : DEL;
                    if (v < nvec) {
                        uint4 x = FG_AT((const uint4 *)mapc, s * m16 + v, NMAP16);
                        if (v == nvec - 1 && nb < 16 * nvec)
                            ((MapT *)&x)[(nb - 16 * v) / (int)sizeof(MapT)] = val;
                        FG_AT((uint4 *)mapn, r * m16 + v, NMAP16) = x;
                    } else {
                        if (nb == 16 * nvec) FG_AT((MapT *)mapn, r * mt + i, NMAPT) = val;
                        for (int w = 0; w < W; ++w) {
                            Word x = FG_AT(imgc, (int64_t)s * W + w, NIMG);
                            if (j < n2 && j / WB == w) x |= (Word)1 << (j % WB);
                            FG_AT(imgn, (int64_t)r * W + w, NIMG) = x;
                        }
                        FG_AT(pedn, r, NPED) = FG_AT(R.selped, r, FG_N(int32_t, p.lay.rsize[RG_SELPED]));
                    }
                }
            } else {
                // cluster teams: a warp copies its children two at a time. Its next 32 codes and
                // PEDs come in one load each, and up to four map vectors per lane are under way
                // (rows of up to 2 KB from L2: with one vector under way the copies took a
                // fifth of the time on large pairs)
                for (int rb = warp; rb < newL; rb += 32 * NW) {
                    const int mine = rb + lane * NW;
                    const int mc = mine < newL ? FG_AT(R.sel, mine, FG_N(int32_t, p.lay.rsize[RG_SEL])) : 0;
                    const int md = mine < newL ? FG_AT(R.selped, mine, FG_N(int32_t, p.lay.rsize[RG_SELPED])) : 0;
                    const int cnt = min(32, (newL - rb + NW - 1) / NW);
                    for (int t = 0; t < cnt; t += 2) {
                        const int ca = __shfl_sync(0xffffffffu, mc, t), cb = __shfl_sync(0xffffffffu, mc, (t + 1) & 31);
                        const int da = __shfl_sync(0xffffffffu, md, t), db = __shfl_sync(0xffffffffu, md, (t + 1) & 31);
                        const bool two = t + 1 < cnt;
                        const int64_t ra = rb + (int64_t)t * NW, rc = two ? ra + NW : ra;
                        const int64_t sa = ca >> kSelShift, sb = (two ? cb : ca) >> kSelShift;
                        for (int v = lane; v < nvec; v += 64) {
                            const bool w2 = v + 32 < nvec;
                            uint4 x[4];
                            x[0] = FG_AT((const uint4 *)mapc, sa * m16 + v, NMAP16);
                            x[1] = FG_AT((const uint4 *)mapc, sb * m16 + v, NMAP16);
                            if (w2) {
                                x[2] = FG_AT((const uint4 *)mapc, sa * m16 + v + 32, NMAP16);
                                x[3] = FG_AT((const uint4 *)mapc, sb * m16 + v + 32, NMAP16);
                            }
                            FG_AT((uint4 *)mapn, ra * m16 + v, NMAP16) = x[0];
                            if (two) FG_AT((uint4 *)mapn, rc * m16 + v, NMAP16) = x[1];
                            if (w2) {
                                FG_AT((uint4 *)mapn, ra * m16 + v + 32, NMAP16) = x[2];
                                if (two) FG_AT((uint4 *)mapn, rc * m16 + v + 32, NMAP16) = x[3];
                            }
                        }
                        __syncwarp();
                        // half a warp per child: Img words (16 at most), entry i, PED
                        const bool hi = lane >= 16;
                        if (!hi || two) {
                            const int j = (hi ? cb : ca) & ((1 << kSelShift) - 1), w = lane & 15;
                            const int64_t r = hi ? rc : ra, s = hi ? sb : sa;
                            if (w < W) {
                                Word x = FG_AT(imgc, s * W + w, NIMG);
                                if (j < n2 && j / WB == w) x |= (Word)1 << (j % WB);
                                FG_AT(imgn, r * W + w, NIMG) = x;
                            }
                            if (w == 0) {
                                FG_AT((MapT *)mapn, r * mt + i, NMAPT) = (j < n2) ? (MapT)j : DEL;
                                FG_AT(pedn, r, NPED) = hi ? db : da;
                            }
                        }
                    }
                }
            }
        }
        // S1 cost row of the next level (each CTA keeps its own copy)
        if (i + 1 < n1) {
            const int a1n = FG_AT(p.vlab, m1.lab_off + i + 1, p.n_vlab);
            for (int u = ltid; u <= n2; u += LT)
                FG_AT(crn, u, N2S) = u < n2 ? ((FG_AT(R.alpha2, u, FG_N(int32_t, p.lay.rsize[RG_ALPHA2])) != a1n) ? c.vsub : 0) : c.vdel;
        }
        tm.sync();
        PHASE_MARK(3);
        { int32_t *t = crc; crc = crn; crn = t; }
        { uint8_t *t = mapc; mapc = mapn; mapn = t; }
        { uint8_t *t = ecur; ecur = enext; enext = t; }
        { Word *t = imgc; imgc = imgn; imgn = t; }
        { int32_t *t = pedc; pedc = pedn; pedn = t; }
        L = newL;
    }

    // ---- S5 leaf completion (insert the free g2 vertices and their edges) + argmin ------
    {
        unsigned long long best = ~0ull;
        for (int s = warp; s < L; s += NW) {
            const int64_t im = (int64_t)s * W;   // the leaf's Img row
            int acc = 0;
            for (int u = lane; u < n2; u += 32) {
                if ((FG_AT(imgc, im + u / WB, NIMG) >> (u % WB)) & (Word)1) {
#pragma unroll
                    for (int w = 0; w < W; ++w)
                        acc += popcw((Word)(FG_AT(R.a2t, w * N2S + u, FG_N(Word, p.lay.rsize[RG_A2T])) &
                                            FG_AT(imgc, im + w, NIMG)));
                }
            }
            int nimg = 0;
            for (int w = lane; w < W; w += 32) nimg += popcw(FG_AT(imgc, im + w, NIMG));
            acc = warp_sum(acc);
            nimg = warp_sum(nimg);
            // g2 edges with both ends used were counted twice in acc
            const long long total = (long long)FG_AT(pedc, s, NPED) + (long long)c.vins * (n2 - nimg) +
                                    (long long)c.eins * (m2.m - acc / 2);
            const unsigned long long key = ((unsigned long long)total << 32) | (unsigned)s;
            best = key < best ? key : best;
        }
        if (lane == 0) FG_AT(S.wbest, warp, NSW) = best;
        tm.sync();
        if (tid == 0) {
            unsigned long long b = FG_AT(S.wbest, 0, NSW);
            for (int w = 1; w < NW; ++w) b = FG_AT(S.wbest, w, NSW) < b ? FG_AT(S.wbest, w, NSW) : b;
            FG_AT(S.wbest, 0, NSW) = b;
            FG_AT(p.out_cost, pair, p.n_pairs) = (int32_t)(b >> 32);
            if (p.out_nevals) FG_AT(p.out_nevals, pair, p.n_pairs) = nevals + L;
        }
        tm.sync();
        const int bs = (int)(FG_AT(S.wbest, 0, NSW) & 0xffffffffull);
        const int64_t mb = (int64_t)bs * (mrow / (int64_t)sizeof(MapT));   // the winner's map row
        const int64_t om = FG_AT(p.map_off, pair, p.n_pairs);
        for (int k = tid; k < n1; k += T) {
            const MapT v = FG_AT((const MapT *)mapc, mb + k, NMAPT);
            FG_AT(p.out_map, om + k, p.map_total) = (v == DEL) ? -1 : (int32_t)v;
        }
        tm.sync();
        PHASE_MARK(4);
    }
#ifdef FASTGED_PHASE_TIMERS
    if (tid == 0 && p.phase_cycles)
        for (int k = 0; k < 16; ++k) atomicAdd(&p.phase_cycles[k], (unsigned long long)ph[k]);
#endif
#undef NIMG
#undef NPED
#undef NSW
#undef NP
#undef NMAPT
#undef NMAP16
#undef NIMGW
}

// SM: every region but the neighbour lists and the vertex maps lives in shared memory (addresses then stay in the
// shared window)
template <int W, typename MapT, typename Word, bool SM, int BK>
__global__ void __launch_bounds__(512, (W <= 4) ? 2 : 1) kbest_kernel(const KParams p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ TeamShared S;
    uint8_t *gs = p.gscratch + (int64_t)blockIdx.x * p.lay.slice_bytes;
    auto base = [&](int r) -> uint8_t * {
        if (SM && r != RG_NBR && r != RG_MAP0 && r != RG_MAP1) return smem + p.lay.off[r];
        return ((p.lay.smem_mask >> r) & 1u ? smem : gs) + p.lay.off[r];
    };
    Regions<Word> R = make_regions<Word>(base);
    smem_regions(p, R, smem);
    for (;;) {
        if (threadIdx.x == 0) S.pair = atomicAdd(p.queue_head, 1);
        __syncthreads();
        const int qi = S.pair;
        __syncthreads();
        if (qi >= p.n_order) break;
        solve_pair<W, MapT, Word, BK, false, TeamShared>(p, R, S, FG_AT(p.order, qi, p.n_order));
    }
}

// One pair per thread-block cluster: every CTA of the cluster belongs to the team. Each
// CTA keeps its own copy of the read-only target-graph tables; what the team writes lives in
// the cluster's slice of global scratch, together with the team scalars. Two-word teams are
// held to 64 registers so that two CTAs share an SM (more clusters resident at once); wider
// ones keep 128 (their 16-word evaluation would spill).
template <int W, typename MapT, typename Word, int BK>
__global__ void __launch_bounds__(512, (W <= 2) ? 2 : 1) kbest_cluster_kernel(const KParams p)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const unsigned crank = cluster_rank(), csize = cluster_size();
    uint8_t *gs = p.gscratch + (int64_t)(blockIdx.x / csize) * p.lay.slice_bytes;
    uint8_t *gc = gs + p.lay.cta_off + (int64_t)crank * p.lay.cta_bytes;   // this CTA's block
    auto base = [&](int r) -> uint8_t * {
        if ((p.lay.smem_mask >> r) & 1u) return smem + p.lay.off[r];
        return ((p.lay.cta_mask >> r) & 1u ? gc : gs) + p.lay.off[r];
    };
    Regions<Word> R = make_regions<Word>(base);
    smem_regions(p, R, smem);
    TeamSharedCl &S = *(TeamSharedCl *)(gs + p.lay.team_off);
    for (;;) {
        if (crank == 0 && threadIdx.x == 0) S.pair = atomicAdd(p.queue_head, 1);
        cluster_barrier();
        const int qi = *(volatile int *)&S.pair;
        cluster_barrier();
        if (qi >= p.n_order) break;
        solve_pair<W, MapT, Word, BK, true, TeamSharedCl>(p, R, S, FG_AT(p.order, qi, p.n_order));
    }
}

// ------------------------------------------------------------------------------------
// launch wrappers (host side)
// ------------------------------------------------------------------------------------
// Opts the kernel into the device's full dynamic shared memory (needed above 48 KB) before
// it is launched or queried for occupancy.
template <int W, typename MapT, typename Word, bool SM, int BK>
static cudaError_t ensure_smem_attr()
{
    static bool done = false;
    if (done) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kbest_kernel<W, MapT, Word, SM, BK>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kbest_kernel<W, MapT, Word, SM, BK>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) done = true;
    return e;
}

template <int W, typename MapT, typename Word, bool SM, int BK>
static cudaError_t launch_one(const KParams &p, int grid, int block, size_t smem,
                              cudaStream_t st)
{
    cudaError_t e = ensure_smem_attr<W, MapT, Word, SM, BK>();
    if (e != cudaSuccess) return e;
    kbest_kernel<W, MapT, Word, SM, BK><<<grid, block, smem, st>>>(p);
    return cudaGetLastError();
}

template <int W, typename MapT, typename Word, bool SM, int BK>
static cudaError_t occupancy_one(int block, size_t smem, int *out)
{
    cudaError_t e = ensure_smem_attr<W, MapT, Word, SM, BK>();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kbest_kernel<W, MapT, Word, SM, BK>,
                                                         block, smem);
}

// size class -> template instance. 16-bit maps only occur with W >= 4 (n2 >= 255), and the
// all-shared-memory variant is built for bitsets of up to 4 words.
#define FASTGED_DISPATCH(W_, wide, w32, sm, CALL)                                        \
    do {                                                                                 \
        if (sm) {                                                                        \
            if (w32) return CALL(1, uint8_t, uint32_t, true);                            \
            if (W_ == 1 && !wide) return CALL(1, uint8_t, uint64_t, true);               \
            if (W_ == 2 && !wide) return CALL(2, uint8_t, uint64_t, true);               \
            if (W_ == 4 && !wide) return CALL(4, uint8_t, uint64_t, true);               \
        }                                                                                \
        if (w32) return CALL(1, uint8_t, uint32_t, false);                               \
        switch (W_) {                                                                    \
        case 1: if (!wide) return CALL(1, uint8_t, uint64_t, false); break;              \
        case 2: if (!wide) return CALL(2, uint8_t, uint64_t, false); break;              \
        case 4: if (wide) return CALL(4, uint16_t, uint64_t, false);                     \
                else return CALL(4, uint8_t, uint64_t, false);                           \
        case 8: return CALL(8, uint16_t, uint64_t, false);                               \
        case 16: return CALL(16, uint16_t, uint64_t, false);                             \
        default: break;                                                                  \
        }                                                                                \
        return cudaErrorInvalidValue;                                                    \
    } while (0)

template <int W, typename MapT, typename Word, int BK>
static cudaError_t ensure_cluster_attr()
{
    static bool done = false;
    if (done) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kbest_cluster_kernel<W, MapT, Word, BK>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kbest_cluster_kernel<W, MapT, Word, BK>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kbest_cluster_kernel<W, MapT, Word, BK>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) done = true;
    return e;
}

template <int W, typename MapT, typename Word, int BK>
static cudaError_t cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, int grid,
                                  int block, size_t smem, int cluster, cudaStream_t st)
{
    cudaError_t e = ensure_cluster_attr<W, MapT, Word, BK>();
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3((unsigned)block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cluster;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return e;
}

template <int W, typename MapT, typename Word, int BK>
static cudaError_t launch_cluster_one(const KParams &p, int grid, int block, size_t smem,
                                      int cluster, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cudaError_t e = cluster_config<W, MapT, Word, BK>(cfg, attr, grid, block, smem, cluster, st);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, kbest_cluster_kernel<W, MapT, Word, BK>, p);
}

template <int W, typename MapT, typename Word, int BK>
static cudaError_t cluster_occupancy_one(int block, size_t smem, int cluster, int *out)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr;
    cudaError_t e = cluster_config<W, MapT, Word, BK>(cfg, attr, cluster, block, smem, cluster,
                                                      nullptr);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveClusters(out, kbest_cluster_kernel<W, MapT, Word, BK>, &cfg);
}

// cluster teams are built for the 8-bit-map classes of 2 and 4 words and the 16-bit-map
// classes of 4, 8 and 16 words
#define FASTGED_CLUSTER_DISPATCH(W_, wide, CALL)                                         \
    do {                                                                                 \
        switch (W_) {                                                                    \
        case 2: return CALL(2, uint8_t, uint64_t);                                       \
        case 4: if (wide) return CALL(4, uint16_t, uint64_t);                            \
                else return CALL(4, uint8_t, uint64_t);                                  \
        case 8: return CALL(8, uint16_t, uint64_t);                                      \
        case 16: return CALL(16, uint16_t, uint64_t);                                    \
        default: return cudaErrorInvalidValue;                                           \
        }                                                                                \
    } while (0)

template <int BK>
cudaError_t launch_kbest_cluster_bk(int W, bool wide, const KParams &p, int grid, int block,
                                    size_t smem, int cluster, cudaStream_t st)
{
#define CALL_CL(w, M, Wd) launch_cluster_one<w, M, Wd, BK>(p, grid, block, smem, cluster, st)
    FASTGED_CLUSTER_DISPATCH(W, wide, CALL_CL);
#undef CALL_CL
}

template <int BK>
cudaError_t kbest_cluster_occupancy_bk(int W, bool wide, int block, size_t smem, int cluster,
                                       int *out)
{
#define CALL_CO(w, M, Wd) cluster_occupancy_one<w, M, Wd, BK>(block, smem, cluster, out)
    FASTGED_CLUSTER_DISPATCH(W, wide, CALL_CO);
#undef CALL_CO
}

template <int BK>
cudaError_t launch_kbest_bk(int W, bool wide_map, bool w32, bool sm, const KParams &p, int grid,
                            int block, size_t smem, cudaStream_t st)
{
#define CALL_LAUNCH(w, M, Wd, S_) launch_one<w, M, Wd, S_, BK>(p, grid, block, smem, st)
    FASTGED_DISPATCH(W, wide_map, w32, sm, CALL_LAUNCH);
#undef CALL_LAUNCH
}

template <int BK>
cudaError_t kbest_occupancy_bk(int W, bool wide_map, bool w32, bool sm, int block, size_t smem,
                               int *out)
{
#define CALL_OCC(w, M, Wd, S_) occupancy_one<w, M, Wd, S_, BK>(block, smem, out)
    FASTGED_DISPATCH(W, wide_map, w32, sm, CALL_OCC);
#undef CALL_OCC
}

}  // namespace fastged
