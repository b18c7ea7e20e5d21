// kbest_warp.cuh -- sm_103a K-Best kernel with one warp per pair, for pairs whose target graph
// fits one bitset word with a bit to spare (n2 <= 63; the bit after the last vertex stands for
// the deletion), whose source has at most 64 vertices and whose beam is small (the
// molecule-like batches). Instantiated per edge-label plane count in kbest_b0.cu,
// kbest_b2.cu and kbest_b8.cu next to the team kernels of kbest_impl.cuh.
//
// Method: Algorithm 1 of Dabah & Herten (branching Sec. 4.1.1, evaluation Sec. 4.1.2 and
// Algorithm 2, selection Sec. 4.2, leaf insertions Sec. 4.4), with the bitset form of the
// implied edge costs stated at the top of kbest_impl.cuh. Results are identical to the team
// kernels' (same key order, same tie-breaking); only the mapping onto the hardware differs:
//
//   * a warp owns a pair, so a level needs no block barrier and no cross-warp table;
//   * a level scores only the active columns: the target vertices some kept node still has
//     free, and the deletion. Their records (adjacency word, label planes, cost entry) are
//     gathered once per level;
//   * evaluation runs lane <-> parent node: each lane keeps its node's vectors (Img, P, label
//     planes of P, base PED) in registers and all lanes walk the same columns, so a record is
//     one broadcast load. A group of at most 16 nodes (the tail of the beam, or an early
//     level) gives each node 2-32 lanes, which share its columns in quads;
//   * each score leaves one byte (PED offset from the best parent's PED, a lower bound of every
//     child: costs are non-negative and slot 0 holds the least PED of the kept list; 127 when
//     it is larger or the node has used the column's vertex), four to a store, and one count
//     in the warp's histogram by a shared-memory increment;
//   * the kept ones are compacted in enumeration order (node by node, j increasing, the
//     deletion last) from the bytes, 16 per lane and load, and then placed at their rank by a
//     counting sort over the buckets;
//   * when the kept PEDs reach past the window, the level is scored again over coarser, then
//     finer windows until the K-th PED is known, and the kept children are ranked by (PED,
//     enumeration order).
//
// Bound: the integer ALU pipe (half the issue rate) in the scoring loop, and the latency of one
// pair's levels when a batch holds fewer pairs than warps fit the GPU. The loop before this one
// walked each lane's own free bits (find-first-set, a record load with 32 addresses, a 16-bit
// entry and a packed-register count per successor), and its 15-bucket window sent cost setting
// 2 to a bisection on many levels. Measured, before -> after: 20,000 pairs, setting 1, resident:
// 2.82 -> 2.76 ms; 5,003 pairs, setting 2, from host memory: 2.08 -> 1.32 ms; 61 x 256 distance
// matrix, K = 20: 1.28 -> 1.19 ms. (One pair from host memory: 302 -> 296 us; a batch that small
// takes a CTA per pair, 209 us. team_beats_warps in fastged_runtime.cu says where the line lies.)
// Registers are capped at 96 by the launch bounds; the instances with 0 and 2 label planes spill
// 20-40 bytes for it.
#pragma once
#include "kbest_impl.cuh"

namespace fastged {

// kept successors a warp places at once: the largest K of a one-warp class, in 32s
constexpr int kWarpChunks = 4;
// cost entry of the columns that pad the active ones to whole quads: past every bucket, and
// no PED offset (below 2^16) added to it leaves the range
constexpr int kWarpPadCost = 1 << 24;

// Target record of g2 vertex u at index u, or of the deletion column at index n2 (no
// neighbours, no labels): adjacency word and NPL edge-label planes. (WarpRec, one per active
// column of a level, also holds the cost entry.)
template <typename Word, int NPL>
struct __align__(16) TgtRec {
    Word a2;
    Word l[NPL];
};
template <typename Word>
struct __align__(16) TgtRec<Word, 0> {
    Word a2;
};

static_assert(sizeof(TgtRec<uint32_t, 0>) == warp_rec_bytes(true, 0), "record size");
static_assert(sizeof(TgtRec<uint32_t, 2>) == warp_rec_bytes(true, 2), "record size");
static_assert(sizeof(TgtRec<uint32_t, kMaxB>) == warp_rec_bytes(true, kMaxB), "record size");
static_assert(sizeof(TgtRec<uint64_t, 0>) == warp_rec_bytes(false, 0), "record size");
static_assert(sizeof(TgtRec<uint64_t, 2>) == warp_rec_bytes(false, 2), "record size");
static_assert(sizeof(TgtRec<uint64_t, kMaxB>) == warp_rec_bytes(false, kMaxB), "record size");

template <typename Word, int NPL>
__device__ __forceinline__ Word rec_plane(const TgtRec<Word, NPL> &r, int b) { return r.l[b]; }
template <typename Word>
__device__ __forceinline__ Word rec_plane(const TgtRec<Word, 0> &, int) { return (Word)0; }
template <typename Word, int NPL>
__device__ __forceinline__ void rec_set_plane(TgtRec<Word, NPL> &r, int b, Word v) { r.l[b] = v; }
template <typename Word>
__device__ __forceinline__ void rec_set_plane(TgtRec<Word, 0> &, int, Word) {}

#ifdef FASTGED_PHASE_TIMERS
// profiling builds only: cycles lane 0 of every warp spends in each phase
#define WPHASE(k)                                            \
    do {                                                     \
        if ((threadIdx.x & 31) == 0) {                       \
            const long long t_ = clock64();                  \
            ph[k] += t_ - ph_last;                           \
            ph_last = t_;                                    \
        }                                                    \
    } while (0)
#else
#define WPHASE(k) do { } while (0)
#endif

// Record of an active column of a level: adjacency word, the g2 neighbours whose edge's label
// differs from the level's (v_i's edges to its prior neighbours, when all have one label), the
// vertex's one-hot bit (0: the deletion, or a column that pads the row) and the cost entry.
template <typename Word>
struct __align__(16) WarpRec {
    Word a2, mis, bit;
    int32_t crow;
};
static_assert(sizeof(WarpRec<uint32_t>) == warp_col_bytes(true), "record size");
static_assert(sizeof(WarpRec<uint64_t>) == warp_col_bytes(false), "record size");

// Dynamic shared memory of the one-warp kernel (every warp of a CTA has its block in it).
extern __shared__ __align__(16) uint8_t g_warp_smem[];

// Working set of one warp (see WarpRegion): the warp's block is addressed by 32-bit offsets
// into shared memory; only the vertex maps (shared or global) need full pointers. The beam
// buffers alternate: cur selects which of each pair holds the current level.
template <typename Word, int NPL>
struct WarpRegs {
    uint32_t wb;     // start of the warp's block in dynamic shared memory
    int cur;         // 0: buffers *0 are current, *1 next; 1: the reverse
    uint8_t *mb;     // base of the vertex-map buffers
    template <typename T>
    __device__ __forceinline__ T *at(int32_t off) const { return (T *)(g_warp_smem + wb + (uint32_t)off); }
    __device__ __forceinline__ TgtRec<Word, NPL> *tgt(const WarpLayout &wl) const { return at<TgtRec<Word, NPL>>(wl.off[WR_TGT]); }
    __device__ __forceinline__ int32_t *lab2(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_LAB2]); }
    __device__ __forceinline__ int32_t *noff(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_NOFF]); }
    __device__ __forceinline__ int32_t *nbr(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_NBR]); }
    __device__ __forceinline__ Word *imgc(const WarpLayout &wl) const { return at<Word>(cur ? wl.off[WR_IMG1] : wl.off[WR_IMG0]); }
    __device__ __forceinline__ Word *imgn(const WarpLayout &wl) const { return at<Word>(cur ? wl.off[WR_IMG0] : wl.off[WR_IMG1]); }
    __device__ __forceinline__ int32_t *pedc(const WarpLayout &wl) const { return at<int32_t>(cur ? wl.off[WR_PED1] : wl.off[WR_PED0]); }
    __device__ __forceinline__ int32_t *pedn(const WarpLayout &wl) const { return at<int32_t>(cur ? wl.off[WR_PED0] : wl.off[WR_PED1]); }
    __device__ __forceinline__ uint16_t *e2c(const WarpLayout &wl) const { return at<uint16_t>(cur ? wl.off[WR_E21] : wl.off[WR_E20]); }
    __device__ __forceinline__ uint16_t *e2n(const WarpLayout &wl) const { return at<uint16_t>(cur ? wl.off[WR_E20] : wl.off[WR_E21]); }
    __device__ __forceinline__ uint8_t *score(const WarpLayout &wl) const { return at<uint8_t>(wl.off[WR_SCORE]); }
    __device__ __forceinline__ int32_t *hist(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_SCORE] + wl.hist_off); }
    __device__ __forceinline__ WarpRec<Word> *rec(const WarpLayout &wl) const { return at<WarpRec<Word>>(wl.off[WR_SCORE] + wl.rec_off); }
    __device__ __forceinline__ Word *planes(const WarpLayout &wl) const { return at<Word>(wl.off[WR_SCORE] + wl.pl_off); }
    __device__ __forceinline__ uint32_t *klist(const WarpLayout &wl) const { return at<uint32_t>(wl.off[WR_KLIST]); }
    __device__ __forceinline__ int32_t *sel(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_SEL]); }
    __device__ __forceinline__ int32_t *selped(const WarpLayout &wl) const { return at<int32_t>(wl.off[WR_SELPED]); }
    __device__ __forceinline__ uint8_t *mapc(const WarpLayout &wl) const { return mb + (cur ? wl.off[WR_MAP1] : wl.off[WR_MAP0]); }
    __device__ __forceinline__ uint8_t *mapn(const WarpLayout &wl) const { return mb + (cur ? wl.off[WR_MAP0] : wl.off[WR_MAP1]); }
};

// elements of the arrays inside WR_SCORE (bounds-checked builds check indexes against them)
#define NSC ((int64_t)wl.hist_off)
#define NRC FG_N(WarpRec<Word>, wl.pl_off - wl.rec_off)
#define NPA FG_N(Word, wl.size[WR_SCORE] - wl.pl_off)

// What scoring a level needs beside the warp's regions.
struct WarpLevel {
    int L, n0, deg, n2, mrow;   // nodes, v_i's prior neighbours, target vertices, map row bytes
    int nq, nk;                 // quads of columns per row of score bytes (odd), with a column
    int m2;                     // g2 edges (variant B)
    bool one_label;             // v_i's edges to its prior neighbours have one label
};

// Scores every successor of level i. MODE 0: bytes and counts of the offsets from A; returns the
// successors of the level. MODE 1 (selection past the window): with sh > 0 the offsets from A
// in units of 2^sh, PEDs below A left out; sh == 0 gives 0 below A and 1 + the offset from A on.
// MODE 2 (variant B's last level): no bytes; the lane's least (total, PED, code) of the
// completed successors goes to key and code.
// FOLD: insertion and deletion of an edge cost the same, so the two implied-edge terms are
// one popcount.
template <typename Word, int BK, bool FOLD, int MODE>
__device__ __forceinline__ int eval_level(const KParams &p,
                                          const WarpRegs<Word, (BK == 8 ? kMaxB : BK)> &R,
                                          const WarpLevel &lv, int A, int sh,
                                          unsigned long long &key, int &code,
                                          long long *prof = nullptr)
{
    constexpr int WB = 8 * (int)sizeof(Word);
    constexpr int NPL = BK == 8 ? kMaxB : BK;
    using CRec = WarpRec<Word>;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const WarpLayout &wl = p.wl;
    const int L = lv.L, n0 = lv.n0, deg = lv.deg, n2 = lv.n2, mrow = lv.mrow, nq = lv.nq;
    const int B = BK == 0 ? 0 : (BK == 2 ? 2 : p.lay.B);
    const int c_eins = p.cost.eins, c_edel = p.cost.edel, c_esub = p.cost.esub;
    const uint8_t *mapc = R.mapc(wl);
    const CRec *rec = R.rec(wl);
    const Word *planes = R.planes(wl);
    int32_t *hist = R.hist(wl);
    uint32_t *score = (uint32_t *)R.score(wl);
    int tot = 0;
    // v_i's first prior neighbour (the same for every node): most levels of tree-like source
    // graphs have at most one, and those take the short S2 path below
    const int e0 = deg > 0 ? FG_AT(R.nbr(wl), n0, FG_N(int32_t, wl.size[WR_NBR])) : -1;
#ifdef FASTGED_PHASE_TIMERS
    long long tprof = clock64();
#endif
    for (int g0 = 0; g0 < L; g0 += 32) {
        // a group of ng nodes: one lane per node when ng > 16, else 2^qs lanes per node, lane
        // part r taking every 2^qs-th quad of columns
        const int ng = min(32, L - g0);
        const int qs = ng > 16 ? 0 : ng > 8 ? 1 : ng > 4 ? 2 : ng > 2 ? 3 : ng > 1 ? 4 : 5;
        const int r = lane & ((1 << qs) - 1);
        const int s = g0 + (lane >> qs);
        const bool act = (lane >> qs) < ng;
        // S2: P = images of the substituted g1 neighbours of v_i, their edge labels as planes
        // at the image positions, dcnt = deleted neighbours (the neighbour list is the same
        // for every lane: v_i's prior neighbours)
        Word P = (Word)0;
        Word PL[NPL > 0 ? NPL : 1];
#pragma unroll
        for (int b = 0; b < (NPL > 0 ? NPL : 1); ++b) PL[b] = (Word)0;
        int dcnt = 0;
        const int64_t ms = (int64_t)(act ? s : 0) * mrow;   // the node's map row
        if (deg <= 1) {   // warp-uniform
            if (deg == 1) {
                const uint8_t ph = act ? FG_AT(mapc, ms + (e0 & 0xffff), wl.size[WR_MAP0]) : (uint8_t)0xff;
                const bool sub = ph != 0xff;
                dcnt = sub ? 0 : 1;
                P = sub ? (Word)1 << ph : (Word)0;
#pragma unroll
                for (int b = 0; b < NPL; ++b)
                    if (b < B && ((e0 >> (16 + b)) & 1)) PL[b] = P;
            }
        } else
        for (int t0 = 0; t0 < deg; t0 += 4) {
            int e[4];
            uint8_t phi[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                e[u] = t0 + u < deg ? FG_AT(R.nbr(wl), n0 + t0 + u, FG_N(int32_t, wl.size[WR_NBR])) : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                phi[u] = (e[u] >= 0 && act) ? FG_AT(mapc, ms + (e[u] & 0xffff), wl.size[WR_MAP0])
                                            : (uint8_t)0xff;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool sub = phi[u] != 0xff;
                dcnt += (e[u] >= 0 && !sub) ? 1 : 0;
                const Word pb = sub ? (Word)1 << phi[u] : (Word)0;
                P |= pb;
#pragma unroll
                for (int b = 0; b < NPL; ++b)
                    if (b < B && ((e[u] >> (16 + b)) & 1)) PL[b] |= pb;
            }
        }
        const Word im = act ? FG_AT(R.imgc(wl), s, FG_N(Word, wl.size[WR_IMG0])) : (Word)0;
        // (lanes without a node score past every bucket)
        const int base = act ? FG_AT(R.pedc(wl), s, FG_N(int32_t, wl.size[WR_PED0])) - A + c_edel * dcnt : kWarpPadCost;
        const int nimg = popcw(im);
        if (act && r == 0) tot += n2 - nimg + 1;   // free target vertices and the deletion
        const int e2 = MODE == 2 && act ? (int)FG_AT(R.e2c(wl), s, FG_N(uint16_t, wl.size[WR_E20])) : 0;
#ifdef FASTGED_PHASE_TIMERS
        // profiling builds: cycles of the group set-up (prof[12])
        if (prof && lane == 0) {
            const long long tn = clock64();
            prof[12] += tn - tprof;
            tprof = tn;
        }
#endif
        for (int k = r; k < nq; k += 1 << qs) {
            uint32_t v4 = k < lv.nk ? 0u : 0x7f7f7f7fu;
            if (k < lv.nk) {
                // sums of products go to the FMA pipe: the integer ALU, at half the issue rate,
                // is what bounds this loop
                int dd[4];
                Word us[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const CRec c = FG_AT(rec, 4 * k + u, NRC);
                    const Word ai = c.a2 & im;
                    us[u] = im & c.bit;
                    int d = base + c.crow;
                    if (FOLD) d += c_eins * popcw((Word)(ai ^ P));
                    else d += c_eins * popcw((Word)(ai & ~P)) + c_edel * popcw((Word)(P & ~c.a2));
                    if (NPL > 0) {
                        if (lv.one_label) {   // warp-uniform
                            d += c_esub * popcw((Word)(c.mis & P));
                        } else {
                            Word ld = (Word)0;
#pragma unroll
                            for (int b = 0; b < NPL; ++b)
                                if (b < B) ld |= PL[b] ^ FG_AT(planes, b * 4 * nq + 4 * k + u, NPA);
                            d += c_esub * popcw((Word)(c.a2 & P & ld));
                        }
                    }
                    if (MODE == 2 && act && !us[u] && c.crow < kWarpPadCost) {
                        const int j = c.bit ? popcw((Word)(c.bit - 1)) : n2;
                        const long long tt = (long long)d + A + (long long)p.cost.vins * (n2 - nimg - (j < n2 ? 1 : 0)) +
                                             (long long)c_eins * (lv.m2 - e2 - popcw(ai));
                        const unsigned long long kk = ((unsigned long long)tt << 32) | (unsigned)(d + A);
                        const int cc = (s << 8) | j;
                        if (kk < key || (kk == key && cc < code)) {
                            key = kk;
                            code = cc;
                        }
                    }
                    dd[u] = d;
                }
                if (MODE != 2) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int d = dd[u];
                        int v;
                        if (MODE == 0) v = min(d, kScoreMax);
                        else if (sh > 0) v = d < 0 ? kScoreMax : min(d >> sh, kScoreMax);
                        else v = d < 0 ? 0 : min(d + 1, kScoreMax);
                        if (us[u]) v = kScoreMax;
                        dd[u] = v;
                        atomicAdd(&FG_AT(hist, v, kBuckets), 1);   // [127] is not read
                    }
                    v4 = (uint32_t)dd[0] + (uint32_t)dd[1] * 256u + (uint32_t)dd[2] * 65536u + (uint32_t)dd[3] * 16777216u;
                }
            }
            if (MODE != 2 && act) FG_AT(score, s * nq + k, NSC / 4) = v4;
        }
#ifdef FASTGED_PHASE_TIMERS
        // profiling builds: cycles of the scoring loop (prof[13])
        if (prof && lane == 0) {
            const long long tn = clock64();
            prof[13] += tn - tprof;
            tprof = tn;
        }
#endif
    }
    __syncwarp();
    return warp_sum(tot);
}

// Parent slot << 8 | target vertex (n2: the deletion) of score byte idx. inv = ceil(2^21 /
// row bytes): idx < 128 rows and rows below 72 bytes make the product exact.
template <typename Word, int NPL>
__device__ __forceinline__ int warp_code(const KParams &p, const WarpRegs<Word, NPL> &R, int idx,
                                         int row, uint32_t inv, int n2)
{
    const WarpLayout &wl = p.wl;
    const int s = (int)(((uint32_t)idx * inv) >> 21);
    const Word bit = FG_AT(R.rec(wl), idx - s * row, NRC).bit;
    return (s << 8) | (bit ? popcw((Word)(bit - 1)) : n2);
}

// Exact selection: the kept PEDs reach past the histogram window (which starts at A), or over
// too many of its buckets. thr >= 0: offset of the K-th PED, with `below` successors below it;
// the score bytes then hold the kept PEDs already. Otherwise the level is scored again, two or
// four times, and the bytes of the last pass select (no further pass marks the kept ones: 5,000
// molecule pairs with costs of 700-3,001, where nearly every level comes here, 9.0 -> 8.4 ms).
template <typename Word, int BK, bool FOLD>
__device__ __noinline__ void select_exact_warp(const KParams &p,
                                               const WarpRegs<Word, (BK == 8 ? kMaxB : BK)> R,
                                               const WarpLevel lv, int A, int newL, int thr,
                                               int below, uint32_t inv)
{
    constexpr int NPL = BK == 8 ? kMaxB : BK;
    const WarpLayout &wl = p.wl;
    const int lane = threadIdx.x & 31, row = 4 * lv.nq;
    const int B = BK == 0 ? 0 : (BK == 2 ? 2 : p.lay.B);
    int32_t *hist = R.hist(wl);
    unsigned long long key = 0;
    int code = 0;
    const bool known = thr >= 0;
    int anchor = A;
    if (!known) {
        // windows 64 times as wide as the one before until one holds the K-th PED (PEDs are
        // below 2^16 here), then 64 buckets of 1/64 the width inside the bucket found
        int sh = 0, pre = 0, first;
        bool down = false;
        for (int pass = 0; pass < 12; ++pass) {
            sh += down ? -6 : 6;
            for (int b = lane; b < kBuckets; b += 32) FG_AT(hist, b, kBuckets) = 0;
            __syncwarp();
            eval_level<Word, BK, FOLD, 1>(p, R, lv, anchor, sh, key, code);
            // (the last pass counts the successors below its window as well)
            find_threshold(p, hist, sh > 0 ? newL - pre : newL, thr, below, first);
            __syncwarp();
            if (sh == 0) break;
            if (thr < kScoreMax) {
                down = true;
                pre += below;
                anchor += thr << sh;
            }
        }
    }
    uint32_t *klist = R.klist(wl);
    compact_bytes(p, R.score(wl), NSC, 0, lv.L * row, thr, newL - below, 0, 0, newL,
                  [&](int at, int idx, int v) {
                      FG_AT(klist, at, FG_N(uint32_t, wl.size[WR_KLIST])) = ((uint32_t)v << 16) | (uint32_t)idx;
                  });
    __syncwarp();
    // code and PED of every kept child, in enumeration order: the PED from its byte, or from the
    // definition for those below the last window
    for (int x = lane; x < newL; x += 32) {
        const uint32_t kv = FG_AT(klist, x, FG_N(uint32_t, wl.size[WR_KLIST]));
        const int idx = (int)(kv & 0xffffu), v = (int)(kv >> 16);
        const int cc = warp_code<Word, NPL>(p, R, idx, row, inv, lv.n2);
        int ped = known ? A + v : anchor + v - 1;
        if (!known && v == 0) {
            const int s = cc >> 8, j = cc & 0xff;
            const TgtRec<Word, NPL> t = FG_AT(R.tgt(wl), j, (int64_t)wl.size[WR_TGT] / (int64_t)sizeof(TgtRec<Word, NPL>));
            Word P = (Word)0, z = (Word)0;
            int dcnt = 0;
            for (int q = 0; q < lv.deg; ++q) {
                const int e = FG_AT(R.nbr(wl), lv.n0 + q, FG_N(int32_t, wl.size[WR_NBR]));
                const uint8_t ph = FG_AT(R.mapc(wl), (int64_t)s * lv.mrow + (e & 0xffff), wl.size[WR_MAP0]);
                if (ph == 0xff) { ++dcnt; continue; }
                const Word pb = (Word)1 << ph;
                P |= pb;
                for (int b = 0; b < B; ++b)
                    z |= (((e >> (16 + b)) & 1 ? pb : (Word)0) ^ rec_plane(t, b)) & pb;
            }
            const Word im = FG_AT(R.imgc(wl), s, FG_N(Word, wl.size[WR_IMG0])), ai = t.a2 & im;
            ped = FG_AT(R.pedc(wl), s, FG_N(int32_t, wl.size[WR_PED0])) + p.cost.edel * dcnt +
                  FG_AT(R.rec(wl), idx - s * row, NRC).crow + p.cost.eins * popcw((Word)(ai & ~P)) +
                  p.cost.edel * popcw((Word)(P & ~t.a2)) + p.cost.esub * popcw((Word)(t.a2 & z));
        }
        FG_AT(klist, x, FG_N(uint32_t, wl.size[WR_KLIST])) = (uint32_t)cc;
        FG_AT(R.selped(wl), x, FG_N(int32_t, wl.size[WR_SELPED])) = ped;
    }
    __syncwarp();
    // rank by (PED, enumeration order); at most kWarpChunks children per lane, and PEDs below 2^16
    // beside seven bits of the order
    int rk[kWarpChunks], pd[kWarpChunks];
#pragma unroll
    for (int ch = 0; ch < kWarpChunks; ++ch) {
        const int x = 32 * ch + lane;
        rk[ch] = 0;
        pd[ch] = x < newL ? FG_AT(R.selped(wl), x, FG_N(int32_t, wl.size[WR_SELPED])) : 0;
    }
    for (int y = 0; y < newL; ++y) {
        const int ky = FG_AT(R.selped(wl), y, FG_N(int32_t, wl.size[WR_SELPED])) << 7 | y;
#pragma unroll
        for (int ch = 0; ch < kWarpChunks; ++ch) rk[ch] += ky < (pd[ch] << 7 | (32 * ch + lane));
    }
    __syncwarp();
#pragma unroll
    for (int ch = 0; ch < kWarpChunks; ++ch) {
        const int x = 32 * ch + lane;
        if (x < newL) {
            FG_AT(R.sel(wl), rk[ch], FG_N(int32_t, wl.size[WR_SEL])) = (int)FG_AT(klist, x, FG_N(uint32_t, wl.size[WR_KLIST]));
            FG_AT(R.selped(wl), rk[ch], FG_N(int32_t, wl.size[WR_SELPED])) = pd[ch];
        }
    }
    __syncwarp();
}

template <typename Word, int BK, bool FOLD>
__device__ __forceinline__ void solve_pair_warp(const KParams &p, uint32_t wb, uint8_t *gw,
                                                const int pair)
{
    constexpr int NPL = BK == 8 ? kMaxB : BK;
    constexpr int WB = 8 * (int)sizeof(Word);
    using Rec = TgtRec<Word, NPL>;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const WarpLayout &wl = p.wl;
    WarpRegs<Word, NPL> R;
    R.wb = wb;
    R.cur = 0;
    R.mb = wl.gmap ? gw : g_warp_smem + wb;

// elements of warp region r viewed as type T (bounds-checked builds check indexes against it)
#define WN(T, r) FG_N(T, wl.size[r])
    const int g1 = FG_AT(p.pairs, 2 * pair, 2 * p.n_pairs);
    const int g2 = FG_AT(p.pairs, 2 * pair + 1, 2 * p.n_pairs);
    const GraphMeta m1 = FG_AT(p.gmeta, g1, p.n_graphs), m2 = FG_AT(p.gmeta, g2, p.n_graphs);
    const int n1 = m1.n, n2 = m2.n, W1 = m1.W;
    const int K = p.kpp ? FG_AT(p.kpp, pair, p.n_pairs) : p.K;
    const int B = BK == 0 ? 0 : (BK == 2 ? 2 : p.lay.B);
    const int mrow = wl.mrow;
    const CostModel c = p.cost;
    const int hwin = p.hwin;   // PEDs a kept list may span without the exact selection
    constexpr uint8_t DEL = 0xff;
    // m &= ballot(bit b of an offset) ^ lb[b] keeps the lanes whose bit b equals bit b of
    // this lane's index
    unsigned lb[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) lb[k] = ((lane >> k) & 1) ? 0u : 0xffffffffu;
#ifdef FASTGED_PHASE_TIMERS
    long long ph[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    long long ph_last = clock64();
#endif

    // ---- stage the target graph (record u target vertex u, record n2 the deletion) and the
    // source graph's prior-neighbour lists
    {
        const uint64_t *adj2 = p.adj + m2.adj_off;
        const uint64_t *pl2 = p.planes + m2.plane_off;
        const int W2 = m2.W;
        for (int u = lane; u <= n2; u += 32) {
            const bool vtx = u < n2;
            Rec r;
            r.a2 = vtx ? (Word)FG_AT(adj2, (int64_t)u * W2, p.adj_words - m2.adj_off) : (Word)0;
#pragma unroll
            for (int b = 0; b < NPL; ++b)
                rec_set_plane(r, b, (vtx && b < B)
                                        ? (Word)FG_AT(pl2, ((int64_t)b * n2 + u) * W2,
                                                      p.plane_words - m2.plane_off)
                                        : (Word)0);
            FG_AT(R.tgt(wl), u, WN(Rec, WR_TGT)) = r;
            if (vtx)
                FG_AT(R.lab2(wl), u, WN(int32_t, WR_LAB2)) =
                    FG_AT(p.vlab, m2.lab_off + u, p.n_vlab);
        }
        // prior neighbours v_k (k < v) of every g1 vertex v, with their edge labels
        for (int v = lane; v < n1; v += 32) {
            const int64_t row = m1.adj_off + (int64_t)v * W1;
            int d = 0;
            for (int w = 0; w < W1; ++w)
                d += __popcll(FG_AT(p.adj, row + w, p.adj_words) & low_mask(v, w));
            FG_AT(R.noff(wl), v + 1, WN(int32_t, WR_NOFF)) = d;
        }
        __syncwarp();
        int carry = 0;
        for (int v0 = 0; v0 < n1; v0 += 32) {
            const int v = v0 + lane;
            const int d = v < n1 ? FG_AT(R.noff(wl), v + 1, WN(int32_t, WR_NOFF)) : 0;
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += y;
            }
            __syncwarp();
            if (v < n1) FG_AT(R.noff(wl), v + 1, WN(int32_t, WR_NOFF)) = carry + incl;
            carry += __shfl_sync(FULL, incl, 31);
        }
        if (lane == 0) FG_AT(R.noff(wl), 0, WN(int32_t, WR_NOFF)) = 0;
        __syncwarp();
        const int64_t pstep = (int64_t)n1 * W1;
        for (int v = lane; v < n1; v += 32) {
            const int64_t row = m1.adj_off + (int64_t)v * W1;
            const int64_t pl = m1.plane_off + (int64_t)v * W1;
            int o = FG_AT(R.noff(wl), v, WN(int32_t, WR_NOFF));
            for (int w = 0; w < W1; ++w) {
                uint64_t bits = FG_AT(p.adj, row + w, p.adj_words) & low_mask(v, w);
                while (bits) {
                    const int t = __ffsll((long long)bits) - 1;
                    bits &= bits - 1ull;
                    int lab = 0;
                    for (int b = 0; b < B; ++b)
                        lab |= (int)((FG_AT(p.planes, pl + b * pstep + w, p.plane_words) >> t) & 1ull) << b;
                    FG_AT(R.nbr(wl), o, WN(int32_t, WR_NBR)) = (w * 64 + t) | (lab << 16);
                    ++o;
                }
            }
        }
        // root: empty map, Img empty, PED 0
        if (lane == 0) {
            FG_AT(R.imgc(wl), 0, WN(Word, WR_IMG0)) = (Word)0;
            FG_AT(R.pedc(wl), 0, WN(int32_t, WR_PED0)) = 0;
            FG_AT(R.e2c(wl), 0, WN(uint16_t, WR_E20)) = 0;
        }
        __syncwarp();
    }

    long long nevals = 0;
    int L = 1;
    Word all = (Word)0;   // target vertices that every node uses
    const Word nmask = n2 >= WB ? ~(Word)0 : (((Word)1 << n2) - (Word)1);
    using CRec = WarpRec<Word>;
    WPHASE(0);
    for (int i = 0; i < n1; ++i) {
        // the level's active columns, increasing: vertices not used by every node, and the
        // deletion as bit n2 (n2 < WB); their records with S1, the vertex-cost row C[i][.], and
        // one-hot vertex bits; past them, up to an odd number of quads (the lanes' rows then
        // fall into different banks), columns that score past every bucket
        const Word actm = (Word)((~all & nmask) | ((Word)1 << n2));
        const int nact = popcw(actm), nq = (nact + 3) / 4 | 1;
        WarpLevel lv;
        lv.L = L;
        lv.n0 = FG_AT(R.noff(wl), i, WN(int32_t, WR_NOFF));
        lv.deg = FG_AT(R.noff(wl), i + 1, WN(int32_t, WR_NOFF)) - lv.n0;
        lv.n2 = n2;
        lv.mrow = mrow;
        lv.nq = nq;
        lv.nk = (nact + 3) / 4;
        lv.m2 = m2.m;
        // the label of v_i's edges to its prior neighbours, when they have one
        int lab = 0;
        lv.one_label = true;
        if (NPL > 0 && lv.deg > 0) {
            lab = FG_AT(R.nbr(wl), lv.n0, WN(int32_t, WR_NBR)) >> 16;
            for (int t = 1; t < lv.deg; ++t)
                lv.one_label &= (FG_AT(R.nbr(wl), lv.n0 + t, WN(int32_t, WR_NBR)) >> 16) == lab;
        }
        {
            const int a1 = FG_AT(p.vlab, m1.lab_off + i, p.n_vlab);
            for (int u = lane; u <= n2; u += 32) {
                if (!((actm >> u) & (Word)1)) continue;
                const int pos = popcw((Word)(actm & (((Word)1 << u) - (Word)1)));
                const Rec t = FG_AT(R.tgt(wl), u, WN(Rec, WR_TGT));
                CRec cr;
                cr.a2 = t.a2;
                Word ld = (Word)0;
#pragma unroll
                for (int b = 0; b < NPL; ++b) {
                    ld |= rec_plane(t, b) ^ ((lab >> b) & 1 ? ~(Word)0 : (Word)0);
                    if (!lv.one_label && b < B) FG_AT(R.planes(wl), b * 4 * nq + pos, NPA) = rec_plane(t, b);
                }
                cr.mis = t.a2 & ld;
                cr.bit = u < n2 ? (Word)1 << u : (Word)0;
                cr.crow = u < n2 ? ((FG_AT(R.lab2(wl), u, WN(int32_t, WR_LAB2)) != a1) ? c.vsub : 0) : c.vdel;
                FG_AT(R.rec(wl), pos, NRC) = cr;
            }
            if (lane < 4 * nq - nact) {   // fewer than eight
                CRec cr = {};
                cr.crow = kWarpPadCost;
                FG_AT(R.rec(wl), nact + lane, NRC) = cr;
                if (!lv.one_label)
                    for (int b = 0; b < B; ++b) FG_AT(R.planes(wl), b * 4 * nq + nact + lane, NPA) = (Word)0;
            }
            for (int b = lane; b < kBuckets; b += 32) FG_AT(R.hist(wl), b, kBuckets) = 0;
        }
        __syncwarp();
        WPHASE(7);
        const int A = FG_AT(R.pedc(wl), 0, WN(int32_t, WR_PED0));   // least PED of the kept list: a lower bound of every child
        unsigned long long key = ~0ull;
        int code = INT_MAX;
        if (p.variant == 1 && i == n1 - 1) {
            // variant B: every successor of the last level is completed, and the least (total,
            // PED, enumeration order) wins
            const int tot = eval_level<Word, BK, FOLD, 2>(p, R, lv, A, 0, key, code);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(FULL, key, o);
                const int c2 = __shfl_xor_sync(FULL, code, o);
                if (k2 < key || (k2 == key && c2 < code)) {
                    key = k2;
                    code = c2;
                }
            }
            if (lane == 0) {
                FG_AT(p.out_cost, pair, p.n_pairs) = (int32_t)(key >> 32);
                if (p.out_nevals) FG_AT(p.out_nevals, pair, p.n_pairs) = nevals + 2LL * tot;
            }
            const int64_t mo = FG_AT(p.map_off, pair, p.n_pairs);
            const int ws = code >> 8, wj = code & 0xff;
            for (int k = lane; k < n1; k += 32) {
                const uint8_t v = k == i ? (wj < n2 ? (uint8_t)wj : DEL)
                                         : FG_AT(R.mapc(wl), (int64_t)ws * mrow + k, wl.size[WR_MAP0]);
                FG_AT(p.out_map, mo + k, p.map_total) = v == DEL ? -1 : (int32_t)v;
            }
            __syncwarp();
            return;
        }
#ifdef FASTGED_PHASE_TIMERS
        const int tot = eval_level<Word, BK, FOLD, 0>(p, R, lv, A, 0, key, code, ph);
        ph[10] += tot;   // successors
        ph[11] += 1;     // levels
#else
        const int tot = eval_level<Word, BK, FOLD, 0>(p, R, lv, A, 0, key, code);
#endif
        nevals += tot;
        WPHASE(1);
        const int newL = min(K, tot);
        const int row = 4 * nq;
        const uint32_t inv = ((1u << 21) + (uint32_t)row - 1u) / (uint32_t)row;
        // S4: bucket b = PED - A; kept PEDs past the window or over too many buckets go to the
        // exact selection
        int thr, below, first;
        find_threshold(p, R.hist(wl), newL, thr, below, first);
        if (thr < kScoreMax && thr - first < hwin - 1) {
            // kept: every successor below bucket thr and the first q of bucket thr, compacted
            // in enumeration order (score byte << 16 | its index; at most 128 * 72 bytes)
            const int q = newL - below;
            uint32_t *klist = R.klist(wl);
            compact_bytes(p, R.score(wl), NSC, 0, L * row, thr, q, 0, 0, newL,
                          [&](int at, int idx, int v) {
                              FG_AT(klist, at, WN(uint32_t, WR_KLIST)) = ((uint32_t)(v - first) << 16) | (uint32_t)idx;
                          });
            __syncwarp();
            WPHASE(3);
            // place every kept successor at its rank: (smaller offsets) + (equal offsets
            // earlier in enumeration order). All chunks of the kept list are handled at once;
            // lane b carries the kept successors of bucket first + b in the chunks before each
            // one.
            int incl = first + lane < thr ? FG_AT(R.hist(wl), first + lane, kBuckets) : 0;
            const int cb = incl;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            const int bexcl = incl - cb;
            uint32_t kv[kWarpChunks];
            int dk[kWarpChunks], pos[kWarpChunks];
            bool vk[kWarpChunks];
            int run = 0;
#pragma unroll
            for (int ch = 0; ch < kWarpChunks; ++ch) {
                const int x = 32 * ch + lane;
                vk[ch] = x < newL;
                kv[ch] = vk[ch] ? FG_AT(R.klist(wl), x, WN(uint32_t, WR_KLIST)) : 0u;
                dk[ch] = (int)(kv[ch] >> 16);
            }
#pragma unroll
            for (int ch = 0; ch < kWarpChunks; ++ch) {
                if (32 * ch >= newL) break;
                const unsigned V = __ballot_sync(FULL, vk[ch]);
                // same: lanes whose offset equals this lane's; m: lanes whose offset is this
                // lane's index
                unsigned same = V, m = V;
#pragma unroll
                for (int b = 0; b < 5; ++b) {
                    if ((thr - first) >> b == 0) break;   // no offset has this bit
                    const unsigned bb = __ballot_sync(FULL, (dk[ch] >> b) & 1);
                    same &= ((dk[ch] >> b) & 1) ? bb : ~bb;
                    m &= bb ^ lb[b];
                }
                pos[ch] = __shfl_sync(FULL, bexcl, dk[ch]) + __shfl_sync(FULL, run, dk[ch]) +
                          __popc(same & lanemask_lt());
                run += __popc(m);
            }
#pragma unroll
            for (int ch = 0; ch < kWarpChunks; ++ch) {
                if (vk[ch]) {
                    FG_AT(R.sel(wl), pos[ch], WN(int32_t, WR_SEL)) =
                        warp_code<Word, NPL>(p, R, (int)(kv[ch] & 0xffffu), row, inv, n2);
                    FG_AT(R.selped(wl), pos[ch], WN(int32_t, WR_SELPED)) = A + first + dk[ch];
                }
            }
            WPHASE(4);
        } else {
            select_exact_warp<Word, BK, FOLD>(p, R, lv, A, newL, thr < kScoreMax ? thr : -1, below, inv);
            WPHASE(5);
        }
        __syncwarp();
        // kept children in key order (slot = rank): parent map + entry i, Img, PED, and the
        // g2 edges inside Img (for the leaf completion)
        {
            const int nvec = (i + 15) >> 4;
            const uint8_t *__restrict__ mapc = R.mapc(wl);
            uint8_t *__restrict__ mapn = R.mapn(wl);
            Word am = ~(Word)0;
            for (int r = lane; r < newL; r += 32) {
                const int v = FG_AT(R.sel(wl), r, WN(int32_t, WR_SEL));
                const int s = v >> 8, j = v & 0xff;   // parent, vertex (n2: deletion)
                const int64_t src = (int64_t)s * (mrow >> 4), dst = (int64_t)r * (mrow >> 4);
                for (int t = 0; t < nvec; ++t)
                    FG_AT((uint4 *)mapn, dst + t, FG_N(uint4, wl.size[WR_MAP0])) =
                        FG_AT((const uint4 *)mapc, src + t, FG_N(uint4, wl.size[WR_MAP0]));
                FG_AT(mapn, (int64_t)r * mrow + i, wl.size[WR_MAP0]) = j < n2 ? (uint8_t)j : DEL;
                const Word im = FG_AT(R.imgc(wl), s, WN(Word, WR_IMG0));
                int e2 = FG_AT(R.e2c(wl), s, WN(uint16_t, WR_E20));
                Word imn = im;
                if (j < n2) {
                    e2 += popcw((Word)(FG_AT(R.tgt(wl), j, WN(Rec, WR_TGT)).a2 & im));
                    imn |= (Word)1 << j;
                }
                FG_AT(R.imgn(wl), r, WN(Word, WR_IMG0)) = imn;
                am &= imn;
                FG_AT(R.e2n(wl), r, WN(uint16_t, WR_E20)) = (uint16_t)e2;
                FG_AT(R.pedn(wl), r, WN(int32_t, WR_PED0)) = FG_AT(R.selped(wl), r, WN(int32_t, WR_SELPED));
            }
            all = (Word)__reduce_and_sync(FULL, (unsigned)am);
            if (WB == 64)
                all |= (Word)((uint64_t)__reduce_and_sync(FULL, (unsigned)((uint64_t)am >> 32)) << 32);
        }
        __syncwarp();
        R.cur ^= 1;
        L = newL;
        WPHASE(6);
    }

    // ---- S5: complete every kept leaf (insert the free g2 vertices and their edges), least
    // (total, slot)
    unsigned long long best = ~0ull;
    for (int s = lane; s < L; s += 32) {
        const int nimg = popcw(FG_AT(R.imgc(wl), s, WN(Word, WR_IMG0)));
        const long long total = (long long)FG_AT(R.pedc(wl), s, WN(int32_t, WR_PED0)) +
                                (long long)c.vins * (n2 - nimg) +
                                (long long)c.eins * (m2.m - (int)FG_AT(R.e2c(wl), s, WN(uint16_t, WR_E20)));
        const unsigned long long key = ((unsigned long long)total << 32) | (unsigned)s;
        best = key < best ? key : best;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(FULL, best, o);
        best = y < best ? y : best;
    }
    if (lane == 0) {
        FG_AT(p.out_cost, pair, p.n_pairs) = (int32_t)(best >> 32);
        if (p.out_nevals) FG_AT(p.out_nevals, pair, p.n_pairs) = nevals + L;
    }
    const int bs = (int)(best & 0xffffffffull);
    const int64_t mo = FG_AT(p.map_off, pair, p.n_pairs);
    for (int k = lane; k < n1; k += 32) {
        const uint8_t v = FG_AT(R.mapc(wl), (int64_t)bs * mrow + k, wl.size[WR_MAP0]);
        FG_AT(p.out_map, mo + k, p.map_total) = v == DEL ? -1 : (int32_t)v;
    }
    __syncwarp();
    WPHASE(8);
#ifdef FASTGED_PHASE_TIMERS
    if (lane == 0 && p.phase_cycles)
        for (int k = 0; k < 16; ++k) atomicAdd(&p.phase_cycles[k], (unsigned long long)ph[k]);
#endif
#undef WN
#undef NSC
#undef NRC
#undef NPA
}

// Persistent one-warp teams: each warp pops pairs from the class's queue until it is empty. Five
// CTAs per SM (96 registers) hide the latency of the maps; eight label planes need 128 and have
// shared memory for four anyway (5,000 molecule pairs, labels 0-6: 1.48 -> 1.37 ms).
template <typename Word, int BK>
__global__ void __launch_bounds__(128, BK == 8 ? 4 : 5) kbest_warp_kernel(const KParams p)
{
    const int wic = (int)(threadIdx.x >> 5);
    const int gwarp = (int)blockIdx.x * (int)(blockDim.x >> 5) + wic;
    const uint32_t wb = (uint32_t)wic * (uint32_t)p.wl.warp_bytes;
    uint8_t *gw = p.wl.gmap ? p.gscratch + (int64_t)gwarp * p.wl.gmap_bytes : nullptr;
    const bool fold = p.cost.eins == p.cost.edel;
    for (;;) {
        int qi = 0;
        if ((threadIdx.x & 31) == 0) qi = atomicAdd(p.queue_head, 1);
        qi = __shfl_sync(0xffffffffu, qi, 0);
        if (qi >= p.n_order) break;
        const int pair = FG_AT(p.order, qi, p.n_order);
        if (fold) solve_pair_warp<Word, BK, true>(p, wb, gw, pair);
        else solve_pair_warp<Word, BK, false>(p, wb, gw, pair);
    }
}

template <typename Word, int BK>
static cudaError_t ensure_warp_attr()
{
    static bool done = false;
    if (done) return cudaSuccess;
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kbest_warp_kernel<Word, BK>);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kbest_warp_kernel<Word, BK>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) done = true;
    return e;
}

template <int BK>
cudaError_t launch_kbest_warp_bk(bool w32, const KParams &p, int grid, int block, size_t smem,
                                 cudaStream_t st)
{
    if (w32) {
        cudaError_t e = ensure_warp_attr<uint32_t, BK>();
        if (e != cudaSuccess) return e;
        kbest_warp_kernel<uint32_t, BK><<<grid, block, smem, st>>>(p);
    } else {
        cudaError_t e = ensure_warp_attr<uint64_t, BK>();
        if (e != cudaSuccess) return e;
        kbest_warp_kernel<uint64_t, BK><<<grid, block, smem, st>>>(p);
    }
    return cudaGetLastError();
}

template <int BK>
cudaError_t kbest_warp_occupancy_bk(bool w32, int block, size_t smem, int *out)
{
    if (w32) {
        cudaError_t e = ensure_warp_attr<uint32_t, BK>();
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kbest_warp_kernel<uint32_t, BK>,
                                                             block, smem);
    }
    cudaError_t e = ensure_warp_attr<uint64_t, BK>();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kbest_warp_kernel<uint64_t, BK>,
                                                         block, smem);
}

}  // namespace fastged
