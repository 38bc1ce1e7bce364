// walk_dev.cuh -- device code of the tree walk shared by the walk kernel
// (walk.cu) and its warp-specialised form (walk_ws.cu): parameters, shared
// buffers, the evaluation of far cells, leaf particles, big-list corrections
// and analytic halos for a lane's rays (Sec. 3.2), and the traversal with its
// buffer appends, written against a context whose flush either evaluates a
// full buffer or hands it to another warp.
#pragma once

#include "local.cuh"
#include "profiles.cuh"
#include "walk_shared.cuh"

namespace lens {

// A group's walk can be cut: the warp that walks it hands the boxes still on
// its stack (and, deferred, big lists) to `parts` work items of the next
// launch, each of which walks every parts-th box of them for the same rays.
// A warp's walk is a serial chain of dependent steps, so a launch of few
// groups leaves most of the chip idle (295 groups of a 97^2-ray map: 2.9 ms
// for 295 warps of 3,648), and a group over a density cusp runs alone at the
// end of a launch of many (walk_rounds says when groups are cut).  Every item
// writes its rays' totals to a place of its own; k_cut_sum adds those of a
// group in order.
//
// The bits do not depend on which warp ran what.  Where a cut finds its pool
// full, the warp itself walks the parts one after another, cuts them again
// where a part of the pool would be, and adds all totals in the same order.
// The number of parts is fixed then; only where the pool has room for every
// group does it follow from how many are cut.
constexpr int kCutNodes = 384;   // boxes handed over per cut
constexpr int kCutRanges = 96;   // deferred big lists per cut
constexpr int kLongList = 8;     // chunks of a big list that is deferred wherever a group may be cut
constexpr uint32_t kNoItem = 0xffffffffu, kNoCut = 0xffffffffu;

struct alignas(16) CutSlot {
    uint32_t g;        // group
    uint32_t n_nodes, n_ranges;
    int32_t parent;    // the totals go to this part of the pool before, or -1: the outputs
    int2 ranges[kCutRanges];  // big lists {first entry, entries}
    int nodes[kCutNodes];
};

static_assert(sizeof(CutSlot) == kCutSlotBytes, "scratch layout");

// The cuts of one launch.
template <typename T> struct CutPool {
    uint32_t* cnt = nullptr;  // cuts made (above max_cuts: by their own warp)
    CutSlot* slots = nullptr;
    uint32_t max_cuts = 0;
    uint32_t parts = 0;     // parts per cut
    uint32_t items = 0;     // if not 0: fewer parts, so that there are at most these in all
    T* head = nullptr;      // max_cuts x 5 x 32R totals: of the walk up to the cut
    T* part = nullptr;      // of part j of cut i: (i x parts + j) x 5 x 32R
    LENS_DEV uint32_t cuts() const { return min(*cnt, max_cuts); }
    LENS_DEV uint32_t parts_of(uint32_t n_cuts) const
    {
        return items == 0 || n_cuts == 0 ? parts : max(1u, min(parts, items / n_cuts));
    }
};

template <typename T> struct CutParams {
    CutPool<T> in;          // the items of this launch (null: whole groups)
    CutPool<T> out;         // where this launch's cuts go (null: no cuts)
    uint32_t limit = 0;     // evaluated entries before a group is cut
    uint32_t limit_stretched = 0;  // the same for a stretched group (0: as the others)
    uint32_t few_parts = 0;    // parts of cuts into fewer than this are cut again at 4 x limit
    int min_nodes = 0;      // boxes on the stack to be worth a cut
    int defer = 0;          // every big list met before the cut goes to the parts
    unsigned char* local = nullptr;  // per warp: deferred lists, and a cut's slot and sums if its pool is full
    size_t local_bytes = 0;          // of one warp: cut_local_bytes, twice where its parts may be cut too
    // the cuts of parts that the warp walks itself (as in the next launch)
    uint32_t again_limit = kNoCut, again_parts = 0;
    int again_min_nodes = 0;
};

template <int R, typename T> constexpr size_t cut_local_bytes() { return kCutSlotBytes + 2 * 5 * 32 * R * sizeof(T); }

// A supergroup: kSuperGroups consecutive groups whose common part of the walk
// is done once (k_super).  Boxes that every group accepts, and leaves that
// every group opens, and that lie far from the supergroup seen from its size,
// are in its expansion h (local.cuh) about (cx, cy) in the frame anchored at
// (hx, hy), scale 1/id; the boxes that are left are where each group's own
// walk starts.  sdelta[g] corrects the expansion's alpha and gamma for group
// g: at the centre of the group's box, the sum of the same sources one by one,
// in the order and with the compensated partial sums of a group's own walk,
// minus the expansion's value.  Over a patch much smaller than the distances
// every ray of a group shares the rounding of that sum, and the results keep
// it (a component that happens to be 1e-3 of the sum of |terms| otherwise
// moves by 2e-5).
struct SuperRec {
    // 1: use it; 0: each group starts at the root; 2: and takes no expansions
    // of its own; 3 (of all records): as 2, in the plain kernel
    int ok;
    int n;         // boxes left
    float hx, hy, cx, cy, id, pad;
    float h[kLocH];
    int nodes[kCutNodes];
};
static_assert(sizeof(SuperRec) == kSuperBytes, "scratch layout");

// A species' constants in the evaluation.
template <typename T> struct EvalConsts {
    T Uq, invNq, Uq2, Nq, eU;
};

template <typename T> struct WalkParams : EvalConsts<T> {
    const vec4_t<T>* nodeA;
    const v2_t<T>* nodeB;
    const int4* link;
    const float* node_rcm;
    const vec4_t<T>* leaf0;   // near records (listed particles marked)
    const vec4_t<T>* leaf1;   // NFW second record
    const vec4_t<T>* big0;       // {x, y, s^2, r0^2}
    const vec4_t<T>* big1;       // {m, c | A, B, 0}
    const vec4_t<T>* big_chunk;  // support bounding box per 32 entries
    const vec4_t<T>* node_bigbox;
    int64_t n_part;
    const v2_t<T>* gH;
    const vec4_t<T>* gbox;
    const uint2* grange;
    int64_t n_rays;
    const v2_t<T>* ray_l;
    const uint32_t* ray_idx;
    int64_t n_groups;
    const HaloDev* halos;
    int n_halos;
    T* out[5];
    int accumulate;
    uint32_t* counter;
    int* stack;
    uint32_t* err;
    unsigned long long* stats;  // optional walk counters
    long long wait_cycles;      // bound of every wait between cooperating warps (SM clock cycles)
    // direct sum split over particle slices (n_slices > 1): work item
    // g * n_slices + k sums slice k of the particles for group g's rays into
    // split[(k * 5 + q) * split_n + ray]; k_split_sum adds the slices
    int n_slices;
    int64_t split_n;
    T* split;
    // group order and work record (walk_shared.cuh): item g walks group
    // order[g] (identity if null); the walk adds each group's work to gcost[g]
    const uint32_t* order;
    uint32_t* gcost;
    // interaction lists kept for the adjoint (LENS_KEEP_LISTS): group g's
    // tagged box indices at list_ids + g * list_K, their count in list_n[g]
    uint32_t* list_ids;
    uint32_t* list_n;
    int list_K;
    CutParams<T> cut;  // parts of groups whose walk is shared by several warps
    const uint8_t* gflag;     // per group: 1 if stretched (walk_shared.cuh)
    // only the groups sub[0 .. *sub_n) (null: all); skip: all but the stretched ones
    const uint32_t* sub;
    const uint32_t* sub_n;
    int skip;
    const SuperRec* super;   // supergroups' records (null: every group starts at the root)
    const float4* sdelta;    // per group: see SuperRec
};

// Record one traversal step's boxes that matter to the adjoint (one entry
// per box, lane order) into the context's list, if it keeps one.  The parts of
// a cut group share the group's count in memory (rec_shared); an overflow
// leaves it above the room.
template <class Ctx>
LENS_DEV void record_step(Ctx& C, int v, bool acc, bool leaf, bool big)
{
    if (!C.rec) return;
    const int lane = threadIdx.x & 31;
    const uint32_t tag = (acc ? kListFar : 0u) | (leaf ? kListLeaf : 0u) | (big ? kListBig : 0u);
    const unsigned m = __ballot_sync(0xffffffffu, tag != 0u);
    if (m == 0u) return;
    if (C.rec_shared) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(C.rec_shared, (uint32_t)__popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        C.rec_n = (int)min(at, (uint32_t)C.rec_cap);
    }
    const int pos = C.rec_n + __popc(m & ((1u << lane) - 1u));
    if (tag != 0u && pos < C.rec_cap) C.rec[pos] = (uint32_t)v | tag;
    C.rec_n += __popc(m);
}

// The shared-memory tiles of the near field: TILE 0 holds kNearCap leaf
// particles and kBigCap big-list entries per warp, TILE 1 twice as many
// (fewer flushes and folds, more shared memory per warp); the autotuner
// times both.
template <int KIND, typename T, int TILE = 0> struct WalkBuf {
    static constexpr int kNear = TILE ? 2 * kNearCap : kNearCap;
    static constexpr int kBig = TILE ? 2 * kBigCap : kBigCap;
    // FP32 Gaussian big entries are stored one array per field, so that two
    // consecutive entries load as one float2 operand of the packed form
    static constexpr bool kPackedBig = KIND == LENS_GAUSS && sizeof(T) == 4;
    static constexpr int kB = kPackedBig ? kBig : 1;
    T fdx[kFarCap], fdy[kFarCap], fM[kFarCap], fqr[kFarCap], fqi[kFarCap];
    vec4_t<T> n0[kNear];
    vec4_t<T> n1[KIND == LENS_NFW ? kNear : 1];
    vec4_t<T> b0[KIND == LENS_POINT || kPackedBig ? 1 : kBig];
    vec4_t<T> b1[KIND == LENS_POINT || kPackedBig ? 1 : kBig];
    // -x, -y (from the group anchor), -c log2 e, m/N_q, -(m/N_q) e^-q^2/2,
    // m c/N_q, the flag or 1/r0^2 (b0.w of the generic layout) and 1/c.
    // Entries whose support contains every ray of the group fill slots
    // [0, n_in) from the bottom; the others fill [kBig - n_out, kBig)
    // from the top (the buffer count packs n_in | n_out << 16).
    float bnx[kB], bny[kB], bcl[kB], bm[kB], bme[kB], bk[kB], bw[kB], bic[kB];
};

// The work item a warp walks (a whole group, or a part of a cut one) and its
// cut.  Warp-uniform and touched once per item or cut, so it lives in shared
// memory: in registers it pushed the walk's hot loops into spills (headline
// walk 22.6 -> 24.6 ms).
struct WalkCut {
    // the item
    uint32_t g;          // group
    uint32_t item;       // the part's place in the in pool (kNoItem: a whole group)
    int sp;              // boxes on the stack
    const CutSlot* cs;   // the cut it is a part of, or null
    int j, parts;        // part j of parts
    int rn;              // deferred big lists to scan (every parts-th chunk from j), at rs
    const int2* rs;
    // its cut
    uint32_t limit;      // evaluated entries before the cut (kNoCut: none)
    int min_nodes;
    int n_ranges;        // big lists deferred so far (in the warp's own slot)
    uint32_t chunks;     // their chunks
    int fired;           // was cut
    int local;           // the parts are walked here (the pool was full)
    uint32_t cut;        // its place in the out pool
    int seg;             // local: the part being walked
    int sub, seg2;       // that part was cut too: its subpart being walked
    CutSlot* own;        // the warp's place for what is cut or put aside now
};

// The list ranges of one traversal step (one per lane) and the Neumaier-
// compensated totals of each lane's rays ([component][ray][lane]; touched once
// per buffer flush, so they live here rather than in registers).
struct WalkRanges {
    int rs_off[33];
    int rs_first[32];
    int rs_end[32];
};

// NR: rays per lane the totals have room for (2, or 4 for 128-ray groups).
template <typename T, int NR = 2> struct WalkTot {
    T tot_s[5][NR][32], tot_c[5][NR][32];
};

// The local expansion of the group (FP32 trees) and the entries of a flush
// that are evaluated ray by ray.
struct WalkLocal {
    LocalSum sum;
    float rho2;                // sources with (d/|w0|)^2 up to this are expanded
    float d;                   // the expansion's scale (local_scale)
    uint8_t idx[2 * kBigCap];  // (buffers hold at most 256 entries)
};
struct NoLocal {};
template <typename T> struct LocalBuf;
template <> struct LocalBuf<float> { using type = WalkLocal; };
template <> struct LocalBuf<double> { using type = NoLocal; };

// What a flush needs beside its buffer: the species' constants, the group's
// anchor and box, and every lane's rays.
template <typename T, int NR> struct WalkRays {
    EvalConsts<T> K;
    v2_t<T> H;
    vec4_t<T> box;
    T lx[NR][32], ly[NR][32];
};

// Shared memory of one warp of the walk kernel.
template <int KIND, typename T, int TILE = 0, int NR = 2> struct WalkShared {
    WalkBuf<KIND, T, TILE> buf;
    WalkRanges rng;
    WalkTot<T, NR> tot;
    WalkCut cut;
    WalkRays<T, NR> ray;
    typename LocalBuf<T>::type loc;
};

// Shared memory of one warp of the plain walk kernel.
template <int KIND, typename T, int TILE = 0, int NR = 2> struct PlainShared {
    WalkBuf<KIND, T, TILE> buf;
    WalkRanges rng;
    WalkTot<T, NR> tot;
    WalkCut cut;
};

// Room in the totals for R rays per lane.
template <int R> constexpr int tot_rays() { return R > 2 ? R : 2; }

template <int KIND, typename T, int R, bool AO, int TILE = 0> struct WalkEval {
    static_assert(R <= kMaxRaysPerLane, "rays per lane");
    static constexpr int kQ = AO ? 2 : 5;  // components accumulated
    static constexpr int kNR = tot_rays<R>();
    using Buf = WalkBuf<KIND, T, TILE>;
    const EvalConsts<T>& K;  // the species' constants
    Buf* B;                // the buffers being evaluated
    WalkTot<T, kNR>* Tt;   // compensated totals of the lane's rays
    T lx[R], ly[R];
    Acc5<T> part[R];
    v2_t<T> H;
    vec4_t<T> box;

    LENS_DEV WalkEval(const EvalConsts<T>& k, Buf* b, WalkTot<T, kNR>* t) : K(k), B(b), Tt(t) {}

    LENS_DEV void tot_zero()
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < kQ; ++q) Tt->tot_s[q][r][lane] = Tt->tot_c[q][r][lane] = T(0);
    }

    LENS_DEV T tot_get(int r, int q) const
    {
        const int lane = threadIdx.x & 31;
        return Tt->tot_s[q][r][lane] + Tt->tot_c[q][r][lane];
    }

    // Add the partial sums of the last flush to the compensated totals.
    LENS_DEV void fold()
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T v[5] = {part[r].a1, part[r].a2, part[r].k, part[r].g1, part[r].g2};
#pragma unroll
            for (int q = 0; q < kQ; ++q) {
                T ts = Tt->tot_s[q][r][lane], tc = Tt->tot_c[q][r][lane];
                Comp5<T>::add1(ts, tc, v[q]);
                Tt->tot_s[q][r][lane] = ts;
                Tt->tot_c[q][r][lane] = tc;
            }
            part[r].zero();
        }
    }

    // (idx: only those nf entries)
    LENS_DEV void eval_far(int nf, const uint8_t* idx = nullptr)
    {
        for (int i = 0; i < nf; ++i) {
            const int c = idx ? idx[i] : i;
            T dx = B->fdx[c], dy = B->fdy[c], M = B->fM[c], qr = B->fqr[c], qi = B->fqi[c];
#pragma unroll
            for (int r = 0; r < R; ++r) cell_terms<T, AO>(part[r], lx[r] - dx, ly[r] - dy, M, qr, qi);
        }
        fold();
    }

    // Leaf particles: full profile unless marked as a listed (softened) point.
    LENS_DEV void eval_near(int nn, const uint8_t* idx = nullptr)
    {
        for (int e = 0; e < nn; ++e) {
            const int i = idx ? idx[e] : e;
            vec4_t<T> q = B->n0[i];
            vec4_t<T> q1;
            if constexpr (KIND == LENS_NFW) q1 = B->n1[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                T wx = lx[r] - q.x, wy = ly[r] - q.y;
                T r2 = fma(wx, wx, wy * wy);
                T kb, kap = T(0), Dp;
                if (KIND == LENS_POINT) {
                    point_terms(q.z, r2, kb, Dp);
                } else if (KIND == LENS_GAUSS) {
                    if (q.w > T(0)) gauss_terms(q.z, q.w, r2, K.Uq, K.invNq, kb, kap, Dp);
                    else point_terms(q.z, fmax(r2, -q.w), kb, Dp);
                } else {
                    if (q.w > T(0)) nfw_terms(q.z, q.w, q1.x, q1.y, r2, kb, kap, Dp);
                    else point_terms(q.z, fmax(r2, -q.w), kb, Dp);
                }
                part[r].template radial<AO>(wx, wy, kb, kap, Dp);
            }
        }
        fold();
    }

    // One packed-layout entry for every ray, in scalar arithmetic (entries
    // with a ray inside the softening radius, and unpaired entries).
    LENS_DEV void big_entry_scalar(int i, Acc5x2 (&pa)[R])
    {
        const float nx = B->bnx[i], ny = B->bny[i], w = B->bw[i];
        const float4 q = make_float4(0.0f, 0.0f, 0.0f, w);
        const float4 q1 = make_float4(B->bm[i], -B->bcl[i], B->bk[i], B->bic[i]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            Acc5<float> a;
            a.zero();
            if (w < 0.0f) gauss_correction_fast<AO>(a, lx[r] + nx, ly[r] + ny, q1, K.Uq2, K.eU);
            else gauss_correction<AO>(a, lx[r] + nx, ly[r] + ny, q, q1, K.Uq2, K.Nq);
            pa[r].na1.x -= a.a1;
            pa[r].na2.x -= a.a2;
            if (!AO) {
                pa[r].k.x += a.k;
                pa[r].g1p.x += a.g1;
                pa[r].hg2.x = fmaf(0.5f, a.g2, pa[r].hg2.x);
            }
        }
    }

    // Two entries of the other region of which some ray may come inside a
    // softening radius: the packed general form.
    LENS_DEV void big_pair_soft(int i, Acc5x2 (&pa)[R], const float2 (&LX)[R], const float2 (&LY)[R])
    {
        const float2 nx = *reinterpret_cast<const float2*>(&B->bnx[i]);
        const float2 ny = *reinterpret_cast<const float2*>(&B->bny[i]);
        const float2 cl = *reinterpret_cast<const float2*>(&B->bcl[i]);
        const float2 mN = *reinterpret_cast<const float2*>(&B->bm[i]);
        const float2 kz = *reinterpret_cast<const float2*>(&B->bk[i]);
        const float2 w = *reinterpret_cast<const float2*>(&B->bw[i]);
        const float2 ic = *reinterpret_cast<const float2*>(&B->bic[i]);
        const float2 t_c = make_float2(-cl.x, -cl.y);
        const float2 nmass = make_float2(-(mN.x * K.Nq), -(mN.y * K.Nq));
        const float2 ws = make_float2(w.x < 0.0f ? INFINITY : w.x, w.y < 0.0f ? INFINITY : w.y);
#pragma unroll
        for (int r = 0; r < R; ++r)
            gauss_correction_soft_x2<AO>(pa[r], LX[r], LY[r], nx, ny, t_c, kz, mN, nmass, ws, ic, K.Uq2, K.eU);
    }

    template <bool EDGE>
    LENS_DEV void big_pair_packed(int i, Acc5x2 (&pa)[R], const float2 (&LX)[R], const float2 (&LY)[R])
    {
        const float2 nx = *reinterpret_cast<const float2*>(&B->bnx[i]);
        const float2 ny = *reinterpret_cast<const float2*>(&B->bny[i]);
        const float2 cl = *reinterpret_cast<const float2*>(&B->bcl[i]);
        const float2 mN = *reinterpret_cast<const float2*>(&B->bm[i]);
        const float2 nmE = *reinterpret_cast<const float2*>(&B->bme[i]);
        const float2 kz = *reinterpret_cast<const float2*>(&B->bk[i]);
#pragma unroll
        for (int r = 0; r < R; ++r)
            gauss_correction_x2<AO, EDGE>(pa[r], LX[r], LY[r], nx, ny, cl, mN, nmE, kz, -K.Uq2);
    }

    // FP32 Gaussian big buffer in packed arithmetic: the whole-group-inside
    // region four entries at a time without tests, then the other region
    // pair by pair (packed closed form with the support edge; where a ray may
    // be inside a softening radius, the packed general form for alpha only,
    // else entry by entry).
    LENS_DEV void eval_big_packed(int nbuf)
    {
        const int n_in = nbuf & 0xffff, n_out = nbuf >> 16;
        Acc5x2 pa[R];
        float2 LX[R], LY[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            pa[r].zero();
            LX[r] = make_float2(lx[r], lx[r]);
            LY[r] = make_float2(ly[r], ly[r]);
        }
        int i = 0;
        for (; i + 3 < n_in; i += 4) {
            big_pair_packed<false>(i, pa, LX, LY);
            big_pair_packed<false>(i + 2, pa, LX, LY);
        }
        if (i + 1 < n_in) {
            big_pair_packed<false>(i, pa, LX, LY);
            i += 2;
        }
        if (i < n_in) big_entry_scalar(i, pa);
        i = Buf::kBig - n_out;
        if ((i & 1) && i < Buf::kBig) big_entry_scalar(i++, pa);
        for (; i + 1 < Buf::kBig; i += 2) {
            const float2 w = *reinterpret_cast<const float2*>(&B->bw[i]);
            if (w.x < 0.0f && w.y < 0.0f) {
                big_pair_packed<true>(i, pa, LX, LY);
            } else if constexpr (AO) {
                // (alpha only: the registers allow the packed general form;
                // with kappa and gamma it would push the walk's hot loop
                // into spills)
                big_pair_soft(i, pa, LX, LY);
            } else {
                big_entry_scalar(i, pa);
                big_entry_scalar(i + 1, pa);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            part[r].a1 -= pa[r].na1.x + pa[r].na1.y;
            part[r].a2 -= pa[r].na2.x + pa[r].na2.y;
            if (!AO) {
                part[r].k += pa[r].k.x + pa[r].k.y;
                part[r].g1 += (pa[r].g1p.x + pa[r].g1p.y) - 2.0f * (pa[r].g1y.x + pa[r].g1y.y);
                part[r].g2 += 2.0f * (pa[r].hg2.x + pa[r].hg2.y);
            }
        }
        fold();
    }

    // Big-list corrections: (full profile - softened point); zero outside the
    // support, where both are the same point mass.
    // b0 = {x - H.x, y - H.y, s^2, 1/r0^2}; b1 = {m/N_q, c log2 e, m c / N_q,
    // 1/c} (GAUSS) or {m, A, B, 0} (NFW).  1/max(r^2, r0^2) = min(1/r^2, 1/r0^2).
    // The generic layout takes two entries per iteration for instruction-level
    // parallelism.
    LENS_DEV void eval_big(int nb)
    {
        if constexpr (Buf::kPackedBig) {
            eval_big_packed(nb);
            return;
        }
        int i = 0;
        if constexpr (KIND == LENS_GAUSS) {
            // b0.w < 0 marks an entry whose softening radius no ray of the
            // group reaches (the common case); b0.w = -2 also that its
            // support contains every ray of the group
            for (; i + 1 < nb; i += 2) {
                vec4_t<T> q = B->b0[i], q1 = B->b1[i], p = B->b0[i + 1], p1 = B->b1[i + 1];
                if (q.w < T(-1.5) && p.w < T(-1.5)) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        gauss_correction_inside<AO>(part[r], lx[r] - q.x, ly[r] - q.y, q1, K.eU);
                        gauss_correction_inside<AO>(part[r], lx[r] - p.x, ly[r] - p.y, p1, K.eU);
                    }
                } else if (q.w < T(0) && p.w < T(0)) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        gauss_correction_fast<AO>(part[r], lx[r] - q.x, ly[r] - q.y, q1, K.Uq2, K.eU);
                        gauss_correction_fast<AO>(part[r], lx[r] - p.x, ly[r] - p.y, p1, K.Uq2, K.eU);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        if (q.w < T(0)) gauss_correction_fast<AO>(part[r], lx[r] - q.x, ly[r] - q.y, q1, K.Uq2, K.eU);
                        else gauss_correction<AO>(part[r], lx[r] - q.x, ly[r] - q.y, q, q1, K.Uq2, K.Nq);
                        if (p.w < T(0)) gauss_correction_fast<AO>(part[r], lx[r] - p.x, ly[r] - p.y, p1, K.Uq2, K.eU);
                        else gauss_correction<AO>(part[r], lx[r] - p.x, ly[r] - p.y, p, p1, K.Uq2, K.Nq);
                    }
                }
            }
        }
        for (; i < nb; ++i) {
            vec4_t<T> q = B->b0[i], q1 = B->b1[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                T wx = lx[r] - q.x, wy = ly[r] - q.y;
                if constexpr (KIND == LENS_GAUSS) {
                    if (q.w < T(0)) gauss_correction_fast<AO>(part[r], wx, wy, q1, K.Uq2, K.eU);
                    else gauss_correction<AO>(part[r], wx, wy, q, q1, K.Uq2, K.Nq);
                } else {
                    T r2 = fma(wx, wx, wy * wy);
                    T inv = r2 > T(0) ? rcp(r2) : T(0);
                    T inv_s = fmin(inv, q.w);
                    T kbp = q1.x * inv_s;
                    T kb, kap, Dp;
                    nfw_terms(q1.x, q.z, q1.y, q1.z, r2, kb, kap, Dp);
                    part[r].template radial<AO>(wx, wy, kb - kbp, kap, Dp - kbp * inv_s);
                }
            }
        }
        fold();
    }

    // Analytic components for every ray (Sec. 3.2 analytic models, App. B).
    LENS_DEV void halos(const HaloDev* halos, int n_halos)
    {
        for (int h = 0; h < n_halos; ++h) {
            const HaloDev& hd = halos[h];
            T hx = (T)((double)H.x - hd.x), hy = (T)((double)H.y - hd.y);
            int kind = hd.kind;
            T m = (T)hd.m;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                T wx = lx[r] + hx, wy = ly[r] + hy;
                T r2 = fma(wx, wx, wy * wy);
                T kb = T(0), kap = T(0), Dp = T(0);
                if (kind == LENS_POINT) {
                    point_terms(m, r2, kb, Dp);
                } else if (kind == LENS_GAUSS) {
                    gauss_terms(m, (T)hd.c0, r2, (T)hd.c1, (T)hd.c2, kb, kap, Dp);
                } else if (kind == LENS_NFW) {
                    nfw_terms(m, (T)hd.c2, (T)hd.c0, (T)hd.c1, r2, kb, kap, Dp);
                } else if (kind == LENS_SIS) {
                    if (r2 > T(0)) {
                        T rr = sqrt(r2), re = (T)hd.p0;
                        kb = re / rr;
                        kap = T(0.5) * kb;
                        Dp = kap / r2;
                    }
                } else {  // uniform disk
                    T R2 = (T)hd.c2;
                    if (r2 < R2) {
                        kb = m / R2;
                        kap = kb;
                        Dp = T(0);
                    } else {
                        point_terms(m, r2, kb, Dp);
                    }
                }
                part[r].template radial<AO>(wx, wy, kb, kap, Dp);
            }
        }
        fold();
    }
};

// The walk kernel's context: evaluation plus the buffer counts, where a full
// buffer is evaluated on the spot.
// The flushes of the walk kernel: everything a full buffer's evaluation needs
// is in shared memory, so each is one function (its code inlined at every
// flush site overflowed the instruction cache: 6.3 of 10 stall cycles) and the
// traversal keeps none of its registers.  LOC (FP32 tree walks): the entries
// far from the group, seen from its size, go to the group's local expansion
// (local.cuh), one lane per entry; the others are evaluated for every ray.
template <int KIND, typename T, int R, bool AO, int TILE, bool LOC> struct WalkFlush {
    using WS = WalkShared<KIND, T, TILE, tot_rays<R>()>;
    using Eval = WalkEval<KIND, T, R, AO, TILE>;
    using Buf = WalkBuf<KIND, T, TILE>;

    // The warp's shared memory (named here, not passed: a pointer argument
    // would be a generic one, and every access a generic load).
    static LENS_DEV WS& mine()
    {
        extern __shared__ __align__(16) unsigned char smem_raw[];
        return reinterpret_cast<WS*>(smem_raw)[threadIdx.x >> 5];
    }
    static LENS_DEV Eval eval(WS& S)
    {
        const int lane = threadIdx.x & 31;
        Eval E(S.ray.K, &S.buf, &S.tot);
        E.H = S.ray.H;
        E.box = S.ray.box;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            E.lx[r] = S.ray.lx[r][lane];
            E.ly[r] = S.ray.ly[r][lane];
            E.part[r].zero();
        }
        return E;
    }
    // Add entry i (this lane's, if it has one) to the list of those evaluated
    // ray by ray; n entries are in it.
    static LENS_DEV int keep_direct(WS& S, bool direct, int i, int n)
    {
        const unsigned m = __ballot_sync(0xffffffffu, direct);
        if (direct) S.loc.idx[n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = (uint8_t)i;
        return n + __popc(m);
    }

    // Add the lanes' shares of h to the running coefficients (one copy of the
    // code: the exchanges of 24 values are some 150 instructions).
    static __device__ __noinline__ void add_h24(float4 a, float4 b, float4 c, float4 e, float4 f, float4 g)
    {
        WS& S = mine();
        float u[16] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w, e.x, e.y, e.z, e.w};
        float v[8] = {f.x, f.y, f.z, f.w, g.x, g.y, g.z, g.w};
        local_add(S.loc.sum, 0, lane_totals<16>(u));
        local_add(S.loc.sum, 1, lane_totals<8>(v));
    }
    static LENS_DEV void add_h(const LocalH& H)
    {
        const float* v = H.v;
        add_h24(make_float4(v[0], v[1], v[2], v[3]), make_float4(v[4], v[5], v[6], v[7]),
                make_float4(v[8], v[9], v[10], v[11]), make_float4(v[12], v[13], v[14], v[15]),
                make_float4(v[16], v[17], v[18], v[19]), make_float4(v[20], v[21], v[22], v[23]));
    }

    static __device__ __noinline__ void far(int nf)
    {
        WS& S = mine();
        __syncwarp();
        if constexpr (LOC) {
            const int lane = threadIdx.x & 31;
            const float4 box = S.ray.box;
            const float d = S.loc.d;
            LocalH H;
            H.zero();
            int nd = 0;
#pragma unroll 1
            for (int b = 0; b < nf; b += 32) {
                const int i = b + lane;
                bool direct = i < nf;
                if (direct) {
                    const float wx = box.x - S.buf.fdx[i], wy = box.y - S.buf.fdy[i];
                    const float inv = rcp(fmaf(wx, wx, wy * wy));
                    if (d * d * inv <= S.loc.rho2) {
                        direct = false;
                        H.cell(wx, wy, inv, d, S.buf.fM[i], S.buf.fqr[i], S.buf.fqi[i]);
                    }
                }
                nd = keep_direct(S, direct, i, nd);
            }
            if (nd < nf) add_h(H);
            __syncwarp();
            if (nd > 0) eval(S).eval_far(nd, S.loc.idx);
        } else {
            eval(S).eval_far(nf);
        }
    }

    static __device__ __noinline__ void near(int nn)
    {
        WS& S = mine();
        __syncwarp();
        if constexpr (LOC) {
            const int lane = threadIdx.x & 31;
            const float4 box = S.ray.box;
            const float d = S.loc.d;
            LocalH H;
            H.zero();
            int nd = 0;
#pragma unroll 1
            for (int b = 0; b < nn; b += 32) {
                const int i = b + lane;
                bool direct = i < nn;
                if (direct) {
                    const float4 q = S.buf.n0[i];
                    const float wx = box.x - q.x, wy = box.y - q.y;
                    const float r2 = fmaf(wx, wx, wy * wy), inv = rcp(r2);
                    // a point mass for every ray of the group: beyond the
                    // softening radius, or outside the support
                    bool point = true;
                    if constexpr (KIND != LENS_POINT) {
                        const float lo2 = kLocNear2 * r2;
                        point = q.w <= 0.0f ? lo2 >= -q.w : lo2 > q.w;
                    }
                    if (point && d * d * inv <= S.loc.rho2) {
                        direct = false;
                        H.point(wx, wy, inv, d, q.z);
                    }
                }
                nd = keep_direct(S, direct, i, nd);
            }
            if (nd < nn) add_h(H);
            __syncwarp();
            if (nd > 0) eval(S).eval_near(nd, S.loc.idx);
        } else {
            eval(S).eval_near(nn);
        }
    }

    // After the last flush: the group's expansion for every ray, that of its
    // supergroup (sr, if any) with its correction, and the analytic halos.
    static __device__ __noinline__ void finish(const HaloDev* halos, int n_halos, const SuperRec* sr, float4 delta)
    {
        WS& S = mine();
        __syncwarp();
        if constexpr (LOC) {
            if (sr) {
                LocalFields& F = *reinterpret_cast<LocalFields*>(S.buf.n0);  // (flushed: free)
                const int lane = threadIdx.x & 31;
                if (lane < kLocH) F.h[lane] = sr->h[lane];
                __syncwarp();
                Eval E = eval(S);
                const float ox = (E.H.x - sr->hx) - sr->cx, oy = (E.H.y - sr->hy) - sr->cy;
                const float id = sr->id;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    local_eval<AO>(F, (E.lx[r] + ox) * id, (E.ly[r] + oy) * id, id, E.part[r]);
                E.fold();
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    E.part[r].a1 = delta.x;
                    E.part[r].a2 = delta.y;
                    E.part[r].g1 = delta.z;
                    E.part[r].g2 = delta.w;
                }
                E.fold();
                __syncwarp();
            }
            LocalFields& F = *reinterpret_cast<LocalFields*>(S.buf.n0);  // (flushed: free)
            local_finish(S.loc.sum, F);
            Eval E = eval(S);
            const float id = 1.0f / S.loc.d;
            // (id = 0: a ray at infinity makes the box infinite.  Nothing is
            // expanded then, and 0 * (x - inf) would be NaN for every ray)
            if (id > 0.0f) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    local_eval<AO>(F, (E.lx[r] - E.box.x) * id, (E.ly[r] - E.box.y) * id, id, E.part[r]);
                E.fold();
            }
            __syncwarp();
        }
        if (n_halos > 0) eval(S).halos(halos, n_halos);
    }
};

// The walk kernel's context: the buffers' counts, where a full buffer is
// evaluated on the spot.
template <int KIND, typename T, int R, bool AO, int TILE = 0, bool LOC = false> struct WalkCtx {
    using value_type = T;
    using Buf = WalkBuf<KIND, T, TILE>;
    using Flush = WalkFlush<KIND, T, R, AO, TILE, LOC>;
    static constexpr int kKind = KIND, kR = R;
    static constexpr bool kCuts = true, kDefer = true;  // may be cut; puts long lists aside
    static constexpr int kNear = Buf::kNear, kBig = Buf::kBig;
    const WalkParams<T>& P;
    typename Flush::WS& S;
    Buf* B;
    WalkRanges* Rg;
    WalkCut* Cut;
    v2_t<T> H;
    vec4_t<T> box;
    // boxes visited, cells accepted, leaf particles, big entries scanned, kept
    uint32_t c_vis = 0, c_acc = 0, c_near = 0, c_bigs = 0, c_bigk = 0;
    int nf = 0, nn = 0, nb = 0;  // entries in the far, near and big buffers
    uint32_t* rec = nullptr;     // the group's kept interaction list, or null
    uint32_t* rec_shared = nullptr;  // a part's: the group's count in memory
    int rec_n = 0, rec_cap = 0;

    LENS_DEV WalkCtx(const WalkParams<T>& p, typename Flush::WS& s)
        : P(p), S(s), B(&s.buf), Rg(&s.rng), Cut(&s.cut) {}

    // Load group g's anchor, box and rays (lanes without a ray take the centre).
    LENS_DEV void load_group(uint32_t g)
    {
        const int lane = threadIdx.x & 31;
        H = P.gH[g];
        box = P.gbox[g];
        const uint2 rg = P.grange[g];
        if (lane == 0) {
            S.ray.K.Uq = P.Uq;
            S.ray.K.invNq = P.invNq;
            S.ray.K.Uq2 = P.Uq2;
            S.ray.K.Nq = P.Nq;
            S.ray.K.eU = P.eU;
            S.ray.H = H;
            S.ray.box = box;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r * 32 + lane;
            v2_t<T> l;
            l.x = box.x;
            l.y = box.y;
            if (k < (int)rg.y) l = P.ray_l[rg.x + k];
            S.ray.lx[r][lane] = l.x;
            S.ray.ly[r][lane] = l.y;
        }
        nf = nn = nb = 0;
        c_vis = c_acc = c_near = c_bigs = c_bigk = 0;
    }
    // Zero the totals and the expansion.
    LENS_DEV void start()
    {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < (AO ? 2 : 5); ++q) S.tot.tot_s[q][r][lane] = S.tot.tot_c[q][r][lane] = T(0);
        if constexpr (LOC) {
            local_zero(S.loc.sum);
            if (lane == 0) {
                S.loc.rho2 = P.super && P.super[Cut->g / kSuperGroups].ok >= 2 ? -1.0f : kLocRho2;
                S.loc.d = local_scale(box.z, box.w, P.node_rcm[0]);
            }
        }
        __syncwarp();
    }
    LENS_DEV T total(int r, int q) const
    {
        const int lane = threadIdx.x & 31;
        return S.tot.tot_s[q][r][lane] + S.tot.tot_c[q][r][lane];
    }
    LENS_DEV void flush_far()
    {
        if (nf > 0) Flush::far(nf);
        nf = 0;
    }
    LENS_DEV void flush_near()
    {
        if (nn > 0) Flush::near(nn);
        nn = 0;
    }
    LENS_DEV void flush_big()
    {
        if constexpr (KIND != LENS_POINT) {
            Flush::eval(S).eval_big(nb);
            nb = 0;
        }
    }
};

// The context of the plain walk kernel (whole groups, no expansions): the rays
// stay in registers and full buffers are evaluated inline.  With CUTS a heavy
// group's walk may end in a cut, but no list is put aside for it.
template <int KIND, typename T, int R, bool AO, int TILE, bool CUTS> struct PlainCtx : WalkEval<KIND, T, R, AO, TILE> {
    using value_type = T;
    using Buf = WalkBuf<KIND, T, TILE>;
    static constexpr int kKind = KIND, kR = R;
    static constexpr bool kCuts = CUTS, kDefer = false;
    static constexpr int kNear = Buf::kNear, kBig = Buf::kBig;
    const WalkParams<T>& P;
    WalkRanges* Rg;
    WalkCut* Cut;
    // boxes visited, cells accepted, leaf particles, big entries scanned, kept
    uint32_t c_vis = 0, c_acc = 0, c_near = 0, c_bigs = 0, c_bigk = 0;
    int nf = 0, nn = 0, nb = 0;
    uint32_t* rec = nullptr;
    uint32_t* rec_shared = nullptr;
    int rec_n = 0, rec_cap = 0;

    LENS_DEV PlainCtx(const WalkParams<T>& p, Buf* b, WalkTot<T, tot_rays<R>()>* t, WalkRanges* r, WalkCut* c)
        : WalkEval<KIND, T, R, AO, TILE>(p, b, t), P(p), Rg(r), Cut(c) {}
    LENS_DEV void flush_far()
    {
        this->eval_far(nf);
        nf = 0;
    }
    LENS_DEV void flush_near()
    {
        this->eval_near(nn);
        nn = 0;
    }
    LENS_DEV void flush_big()
    {
        this->eval_big(nb);
        nb = 0;
    }
};

// Append, in order, the leaf particles of up to 32 index ranges (one per
// lane) to the near buffer, flushing it whenever fewer than 32 slots remain.
template <class Ctx, typename T = typename Ctx::value_type>
LENS_DEV void append_ranges(Ctx& C, int cnt, int first, const vec4_t<T>* src0, const vec4_t<T>* src1)
{
    constexpr int KIND = Ctx::kKind;
    const unsigned full = 0xffffffffu;
    int lane = threadIdx.x & 31;
    int tot;
    int off = warp_exclusive_scan(cnt, &tot);
    if (tot == 0) return;
    C.c_near += (uint32_t)tot;
    C.Rg->rs_off[lane] = off;
    C.Rg->rs_first[lane] = first;
    if (lane == 31) C.Rg->rs_off[32] = tot;
    __syncwarp();
    for (int base = 0; base < tot; base += 32) {
        if (C.nn + 32 > Ctx::kNear) {
            C.flush_near();
            __syncwarp();
        }
        int i = base + lane;
        bool have = i < tot;
        vec4_t<T> q0, q1;
        bool keep = false;
        if (have) {
            int lo = 0, hi = 32;  // last lane o with rs_off[o] <= i
            while (hi - lo > 1) {
                int mid = (lo + hi) >> 1;
                if (C.Rg->rs_off[mid] <= i) lo = mid;
                else hi = mid;
            }
            int p = C.Rg->rs_first[lo] + (i - C.Rg->rs_off[lo]);
            q0 = src0[p];
            if constexpr (KIND == LENS_NFW) q1 = src1[p];
            q0.x -= C.H.x;
            q0.y -= C.H.y;
            keep = true;
        }
        unsigned ball = __ballot_sync(full, keep);
        if (keep) {
            int slot = C.nn + __popc(ball & ((1u << lane) - 1u));
            C.B->n0[slot] = q0;
            if constexpr (KIND == LENS_NFW) C.B->n1[slot] = q1;
        }
        C.nn += __popc(ball);
        __syncwarp();
    }
}

// Slots in use in the big buffer (the packed layout counts both regions).
template <int KIND, typename T> LENS_DEV int big_used(int nbuf)
{
    if constexpr (WalkBuf<KIND, T>::kPackedBig) return (nbuf & 0xffff) + (nbuf >> 16);
    else return nbuf;
}

// Big lists of the visited boxes (one list per lane: entries [z, z + w) of
// the big arrays, cnt 32-entry chunks; 0: none, or its support box misses the
// group).  The chunks are tested by their support boxes and the
// entries of the chunks that pass are tested one by one; entries whose
// support reaches the group's box are appended to the big buffer.
// With a stride, only every cstep-th chunk from c0 is taken (a part's share).
template <class Ctx, typename T = typename Ctx::value_type>
LENS_DEV void append_big(Ctx& C, int cnt, int z, int w, int c0 = 0, int cstep = 1)
{
    constexpr int KIND = Ctx::kKind;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const WalkParams<T>& P = C.P;
    int tot;
    int off = warp_exclusive_scan(cnt, &tot);
    if (tot == 0) return;
    int n_seen = 0, n_kept = 0;
    C.Rg->rs_off[lane] = off;
    C.Rg->rs_first[lane] = z;
    C.Rg->rs_end[lane] = z + w;
    if (lane == 31) C.Rg->rs_off[32] = tot;
    __syncwarp();
    for (int base = c0; base < tot; base += 32 * cstep) {
        int i = base + lane * cstep;
        int cid = -1, own = 0;
        bool pass = false;
        if (i < tot) {
            int lo = 0, hi = 32;
            while (hi - lo > 1) {
                int mid = (lo + hi) >> 1;
                if (C.Rg->rs_off[mid] <= i) lo = mid;
                else hi = mid;
            }
            own = lo;
            cid = (C.Rg->rs_first[lo] >> 5) + (i - C.Rg->rs_off[lo]);
            pass = box_reaches_group<T>(P.big_chunk[cid], C.H, C.box);
        }
        unsigned ball = __ballot_sync(full, pass);
        while (ball) {
            int src = __ffs(ball) - 1;
            ball &= ball - 1;
            int c = __shfl_sync(full, cid, src);
            int o = __shfl_sync(full, own, src);
            if (big_used<KIND, T>(C.nb) + 32 > Ctx::kBig) {
                C.flush_big();
                __syncwarp();
            }
            int e = 32 * c + lane;
            bool keep = false;
            vec4_t<T> q0, q1;
            bool inr = e >= C.Rg->rs_first[o] && e < C.Rg->rs_end[o];
            n_seen += __popc(__ballot_sync(full, inr));
            if (inr) {
                q0 = P.big0[e];
                q0.x -= C.H.x;
                q0.y -= C.H.y;
                T ex = fmax(fabs(q0.x - C.box.x) - C.box.z, T(0));
                T ey = fmax(fabs(q0.y - C.box.y) - C.box.w, T(0));
                T near2 = fma(ex, ex, ey * ey);
                keep = near2 < q0.z;
                if constexpr (KIND == LENS_GAUSS) {
                    // every ray of the group beyond the softening radius?  and
                    // all inside the support?
                    if (keep && near2 > T(0) && near2 * q0.w >= T(1.000001)) {
                        T fx = fabs(q0.x - C.box.x) + C.box.z, fy = fabs(q0.y - C.box.y) + C.box.w;
                        T far2 = fma(fx, fx, fy * fy) * T(1.000001);
                        q0.w = far2 < q0.z ? T(-2) : T(-1);
                    }
                }
            }
            unsigned kb = __ballot_sync(full, keep);
            if constexpr (Ctx::Buf::kPackedBig) {
                const bool in = keep && q0.w < T(-1.5);
                const unsigned bi = __ballot_sync(full, in), lt = (1u << lane) - 1u;
                if (keep) {
                    q1 = P.big1[e];
                    int slot = in ? (C.nb & 0xffff) + __popc(bi & lt)
                                  : Ctx::kBig - 1 - ((C.nb >> 16) + __popc(kb & ~bi & lt));
                    C.B->bnx[slot] = -q0.x;
                    C.B->bny[slot] = -q0.y;
                    C.B->bcl[slot] = -q1.y;
                    C.B->bm[slot] = q1.x;
                    C.B->bme[slot] = -q1.x * P.eU;
                    C.B->bk[slot] = q1.z;
                    C.B->bw[slot] = q0.w;
                    C.B->bic[slot] = q1.w;
                }
                C.nb += __popc(bi) + (__popc(kb & ~bi) << 16);
            } else {
                if (keep) {
                    q1 = P.big1[e];
                    int slot = C.nb + __popc(kb & ((1u << lane) - 1u));
                    C.B->b0[slot] = q0;
                    C.B->b1[slot] = q1;
                }
                C.nb += __popc(kb);
            }
            n_kept += __popc(kb);
            __syncwarp();
        }
    }
    C.c_bigs += (uint32_t)n_seen;
    C.c_bigk += (uint32_t)n_kept;
}


// The warp's own cut slot (the lists deferred so far, and the boxes of a cut
// whose pool is full) and the sums beside it; level 1: of a part's cut.
template <int R, typename T> LENS_DEV unsigned char* cut_own(const CutParams<T>& cp, int level = 0)
{
    const int64_t w = (int64_t)blockIdx.x * kWalkWarps + (threadIdx.x >> 5);
    return cp.local + w * (int64_t)cp.local_bytes + level * (int64_t)cut_local_bytes<R, T>();
}

// Cut the walk: the boxes at the bottom of the stack (the shallowest) and the
// deferred lists go to a slot of the pool, or stay in the warp's own if the
// pool is full.  Returns how many boxes stay (at the bottom of the stack).
// DEFER: the walk puts lists aside (one that does not has no slot of its own,
// and is only cut where every group has a place: cuts_fit).
template <int R, bool DEFER = true, typename T> LENS_DEV int cut_now(const CutParams<T>& cp, WalkCut& K, int* stack, int sp)
{
    const uint32_t lane = threadIdx.x & 31;
    const CutPool<T>& pool = cp.out;
    const bool part = DEFER && K.local;  // a part that the warp walks itself
    uint32_t ci = 0;
    if (lane == 0 && !part) ci = atomicAdd(pool.cnt, 1u);
    ci = __shfl_sync(0xffffffffu, ci, 0);
    const bool pooled = !DEFER || (!part && ci < pool.max_cuts);
    CutSlot* own = DEFER ? K.own : nullptr;
    CutSlot* s = pooled ? pool.slots + ci : own;
    const int nd = sp < kCutNodes ? sp : kCutNodes;
    if (DEFER && pooled)
        for (int i = (int)lane; i < K.n_ranges; i += 32) s->ranges[i] = own->ranges[i];
    for (int i = (int)lane; i < nd; i += 32) s->nodes[i] = stack[i];
    if (lane == 0) {
        s->g = K.g;
        s->n_nodes = (uint32_t)nd;
        s->n_ranges = DEFER ? (uint32_t)K.n_ranges : 0u;
        s->parent = K.item == kNoItem ? -1 : (int32_t)K.item;
        if (part) {
            K.sub = 1;
            K.seg2 = 0;
        } else {
            K.fired = 1;
            K.local = !pooled;
            K.cut = ci;
        }
    }
    __syncwarp();
    for (int i = nd; i < sp; i += 32) {
        const int m = i + (int)lane < sp ? stack[i + lane] : 0;
        __syncwarp();
        if (i + (int)lane < sp) stack[i + lane - nd] = m;
        __syncwarp();
    }
    return sp - nd;
}

// Walk the tree for the context's group (Sec. 3.2) from the sp boxes on the
// stack: up to 32 candidate boxes per step, one per lane, tested against the
// group's bounding box; accepted boxes go to the far buffer, opened leaves to
// the near buffer, opened internal boxes push their children, and every
// visited box's big list is scanned.  Full buffers are flushed through the
// context (evaluated on the spot, or handed to an evaluating warp); the caller
// flushes what remains.  Where the walk may be cut (C.Cut->limit), long big
// lists are put aside, and once the walk has evaluated `limit` entries (or
// has only long lists left) it is cut.  The deferred lists of the item itself
// (C.Cut->rn) are scanned 32 to a step, in steps without boxes.
// A context that puts no lists aside stops there instead, the boxes left on the
// stack (C.Cut->sp).
// Returns false if the warp's stack overflowed (the error word is set).
template <class Ctx, typename T = typename Ctx::value_type>
LENS_DEV bool traverse(Ctx& C, int* stack, int sp)
{
    constexpr int KIND = Ctx::kKind;
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const WalkParams<T>& P = C.P;
    uint32_t limit = Ctx::kDefer ? C.Cut->limit : kNoCut;
    int rn = Ctx::kDefer ? C.Cut->rn : 0;
    for (;;) {
        bool lists = false;  // a step of deferred lists
        if constexpr (Ctx::kDefer && KIND != LENS_POINT) {
            lists = rn > 0;
            if (sp == 0 && !lists && limit != kNoCut && C.Cut->n_ranges > 0) {
                // only deferred lists are left: worth a cut (a list's chunk
                // keeps about half of its entries), or scanned here
                const bool cut = 16 * C.Cut->chunks >= limit + 512;
                limit = kNoCut;
                if (cut) {
                    cut_now<Ctx::kR>(P.cut, *C.Cut, stack, 0);
                } else {
                    rn = C.Cut->n_ranges;
                    if (lane == 0) {
                        C.Cut->rs = C.Cut->own->ranges;
                        C.Cut->j = 0;
                        C.Cut->parts = 1;
                    }
                    __syncwarp();
                    lists = true;
                }
            }
        }
        if (sp == 0 && !lists) break;
        int k = lists ? 0 : sp < 32 ? sp : 32;
        sp -= k;
        int v = lane < k ? stack[sp + lane] : -1;
        __syncwarp();
        bool valid = v >= 0, acc = false, leaf = false, open = false;
        vec4_t<T> A;
        int4 Lk = make_int4(0, 0, 0, 0);
        T dxv = T(0), dyv = T(0);
        if (valid) {
            A = P.nodeA[v];
            Lk = P.link[v];
            dxv = A.x - C.H.x;
            dyv = A.y - C.H.y;
            T ex = fmax(fabs(dxv - C.box.x) - C.box.z, T(0));
            T ey = fmax(fabs(dyv - C.box.y) - C.box.w, T(0));
            acc = fma(ex, ex, ey * ey) > A.w;
            leaf = !acc && (Lk.y & kLeafBit);
            open = !acc && !leaf;
        }
        unsigned ball = __ballot_sync(full, acc);
        if (acc) {
            int pos = C.nf + __popc(ball & ((1u << lane) - 1u));
            v2_t<T> Q = P.nodeB[v];
            C.B->fdx[pos] = dxv;
            C.B->fdy[pos] = dyv;
            C.B->fM[pos] = A.z;
            C.B->fqr[pos] = Q.x;
            C.B->fqi[pos] = Q.y;
        }
        C.nf += __popc(ball);
        C.c_vis += (uint32_t)k;
        C.c_acc += (uint32_t)__popc(ball);
        int nc = open ? Lk.y : 0;
        int totc;
        int offc = warp_exclusive_scan(nc, &totc);
        if (sp + totc > kStackCap) {
            if (lane == 0) atomicOr(P.err, DERR_STACK_OVERFLOW);
            return false;
        }
        for (int c = 0; c < nc; ++c) stack[sp + offc + c] = Lk.x + c;
        sp += totc;
        append_ranges(C, leaf ? (Lk.y & kCountMask) : 0, Lk.x, P.leaf0, P.leaf1);
        bool big = false;
        if constexpr (KIND != LENS_POINT) {
            int cnt = 0, c0 = 0, cstep = 1;
            if (lists) {
                const int i = rn - 1 - lane;
                if (i >= 0) {
                    const int2 r = C.Cut->rs[i];
                    Lk.z = r.x;
                    Lk.w = r.y;
                }
                c0 = C.Cut->j;
                cstep = C.Cut->parts;
                rn = rn > 32 ? rn - 32 : 0;
            } else if (valid && Lk.w > 0) {
                big = box_reaches_group<T>(P.node_bigbox[v], C.H, C.box);
                if (!big) Lk.w = 0;
            }
            if (Lk.w > 0 && (lists || big)) cnt = ((Lk.z + Lk.w - 1) >> 5) - (Lk.z >> 5) + 1;
            if constexpr (Ctx::kDefer) {
                if (!lists && limit != kNoCut) {
                    // (a part that the warp walks itself: as in the next launch)
                    const bool put = cnt > (P.cut.defer && !C.Cut->local ? 0 : kLongList);
                    const unsigned bm = __ballot_sync(full, put);
                    if (bm) {
                        const int n0 = C.Cut->n_ranges, pos = n0 + __popc(bm & ((1u << lane) - 1u));
                        uint32_t ch = 0;
                        if (put && pos < kCutRanges) {
                            C.Cut->own->ranges[pos] = make_int2(Lk.z, Lk.w);
                            ch = (uint32_t)cnt;
                            cnt = 0;
                        }
                        ch = __reduce_add_sync(full, ch);
                        if (lane == 0) {
                            C.Cut->n_ranges = min(n0 + __popc(bm), kCutRanges);
                            C.Cut->chunks += ch;
                        }
                        __syncwarp();
                    }
                }
            }
            append_big(C, cnt, Lk.z, Lk.w, c0, cstep);
        }
        record_step(C, v, acc, leaf, big);
        __syncwarp();
        if (C.nf >= 32) {
            C.flush_far();
            __syncwarp();
        }
        if constexpr (Ctx::kCuts) {
            const uint32_t work = C.c_near + C.c_bigk + (C.c_acc >> 1) + (C.c_bigs >> 4);
            if constexpr (Ctx::kDefer) {
                if (work >= limit && sp >= C.Cut->min_nodes) {
                    sp = cut_now<Ctx::kR>(P.cut, *C.Cut, stack, sp);
                    limit = kNoCut;
                }
            } else if (work >= C.Cut->limit && sp >= C.Cut->min_nodes && sp <= kCutNodes) {
                // (the kernel cuts once the buffers are flushed: the code of
                // the cut in here cost it registers)
                if (lane == 0) C.Cut->sp = sp;
                __syncwarp();
                break;
            }
        }
    }
    return true;
}

// Put the boxes of the item's part on the stack, and its share of the lists.
LENS_DEV void load_part(WalkCut& K, int* stack)
{
    const int lane = threadIdx.x & 31, nn = (int)K.cs->n_nodes, j = K.j, parts = K.parts;
    const int sp = nn > j ? (nn - j + parts - 1) / parts : 0;
    for (int i = lane; i < sp; i += 32) stack[i] = K.cs->nodes[j + i * parts];
    __syncwarp();
    if (lane == 0) {
        K.sp = sp;
        K.rn = (int)K.cs->n_ranges;
        K.rs = K.cs->ranges;
    }
    __syncwarp();
}

// The work after which group g is cut (kNoCut: never).
template <typename T> LENS_DEV uint32_t cut_limit(const WalkParams<T>& P, uint32_t g)
{
    const CutParams<T>& cp = P.cut;
    if (!cp.out.cnt) return kNoCut;
    return cp.limit_stretched && P.gflag[g] ? cp.limit_stretched : cp.limit;
}

// A whole group for a kernel without parts: the root on the stack.
template <typename T> LENS_DEV void whole_group(const WalkParams<T>& P, WalkCut& K, uint32_t g, int* stack)
{
    if ((threadIdx.x & 31) == 0) {
        K.g = g;
        K.item = kNoItem;
        K.limit = cut_limit(P, g);
        K.min_nodes = P.cut.min_nodes;
        K.fired = K.local = 0;
        K.sp = 0;
        stack[0] = 0;
    }
    __syncwarp();
}

// Take the next item (false: none left); its boxes go on the stack.
template <int R, typename T> LENS_DEV bool next_item(const WalkParams<T>& P, int* stack, WalkCut& K)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const CutPool<T>& in = P.cut.in;
    const uint32_t cuts = in.cnt ? in.cuts() : 0u, parts = in.parts_of(cuts);
    const int64_t n = in.cnt ? (int64_t)cuts * parts
                      : P.sub ? (int64_t)*P.sub_n
                      : P.super && P.super[0].ok == 3 ? 0 : P.n_groups;
    uint32_t item = 0;
    if (lane == 0) item = atomicAdd(P.counter, 1u);
    item = __shfl_sync(full, item, 0);
    if ((int64_t)item >= n) return false;
    if (lane == 0) {
        K.min_nodes = P.cut.min_nodes;
        K.n_ranges = 0;
        K.chunks = 0;
        K.fired = K.local = 0;
        K.seg = K.sub = 0;
        K.own = (CutSlot*)cut_own<R>(P.cut);
        K.rn = 0;
        if (in.cnt) {
            const CutSlot* cs = in.slots + item / parts;
            K.cs = cs;
            K.j = (int)(item % parts);
            K.parts = (int)parts;
            K.g = cs->g;
            K.limit = !P.cut.out.cnt ? kNoCut : P.cut.limit << (parts < P.cut.few_parts ? 2 : 0);
            K.item = item;
        } else {
            K.cs = nullptr;
            K.g = P.sub ? P.sub[item] : P.order ? P.order[item] : item;
            K.limit = cut_limit(P, K.g);
            K.item = kNoItem;
            K.sp = 1;
            stack[0] = 0;
        }
    }
    __syncwarp();
    if (in.cnt) {
        load_part(K, stack);
    } else if (P.super) {
        // the boxes that the supergroup's walk left
        const SuperRec& sr = P.super[K.g / kSuperGroups];
        if (sr.ok == 1) {
            const int n = sr.n;
            for (int i = lane; i < n; i += 32) stack[i] = sr.nodes[i];
            __syncwarp();
            if (lane == 0) K.sp = n;
            __syncwarp();
        }
    }
    return true;
}

// A cut whose pool was full: after each segment (the item's own, then each
// part; after a part that was cut too, each of its subparts) its totals are
// added to the sums beside the warp's slot, as k_cut_sum adds them; then the
// next part's boxes go on the stack.  False: no part left.
template <int R, int NQ, typename T, class Tot>
LENS_DEV bool local_next_part(const CutParams<T>& cp, WalkCut& K, int* stack, Tot&& tot)
{
    const int lane = threadIdx.x & 31;
    auto at = [&](int level, int r, int q) {
        return (T*)(cut_own<R>(cp, level) + kCutSlotBytes) + ((q * R + r) * 2) * 32 + lane;
    };
    auto next = [&](int level, int j, uint32_t parts) {
        if (lane == 0) {
            K.cs = (CutSlot*)cut_own<R>(cp, level);
            K.j = j;
            K.parts = (int)parts;
            K.own = (CutSlot*)cut_own<R>(cp, 1);
            K.n_ranges = 0;
            K.chunks = 0;
            K.limit = level ? kNoCut : cp.again_limit;
            K.min_nodes = cp.again_min_nodes;
            if (level) {
                K.seg2 = j + 1;
            } else {
                K.seg = j + 1;
                K.sub = 0;
            }
        }
        __syncwarp();
        load_part(K, stack);
    };
    const int seg = K.seg, sub = K.sub, seg2 = K.seg2;
    for (int level = sub; level >= 0; --level) {
        const bool first = (level ? seg2 : seg) == 0;
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                T* a = at(level, r, q);
                T v = tot(r, q);
                if (sub && level == 0) {
                    const T* b = at(1, r, q);
                    v = b[0] + b[32];
                }
                T x = first ? v : a[0], c = first ? T(0) : a[32];
                if (!first) Comp5<T>::add1(x, c, v);
                a[0] = x;
                a[32] = c;
            }
        __syncwarp();
        const int j = level ? seg2 : seg;
        const uint32_t parts = level ? cp.again_parts : cp.out.parts;
        if (j < (int)parts) {
            next(level, j, parts);
            return true;
        }
    }
    return false;
}
template <int R, typename T> LENS_DEV T local_total(const CutParams<T>& cp, int r, int q)
{
    const T* a = (const T*)(cut_own<R>(cp) + kCutSlotBytes) + ((q * R + r) * 2) * 32 + (threadIdx.x & 31);
    return a[0] + a[32];
}

// Where an item's totals go: the outputs (null), its own place in its pool,
// or, when it was cut, the cut's.
template <int R, typename T> LENS_DEV T* item_totals(const CutParams<T>& cp, const WalkCut& K)
{
    if (K.fired && !K.local) return cp.out.head + (int64_t)K.cut * (5 * 32 * R);
    if (K.item != kNoItem) return cp.in.part + (int64_t)K.item * (5 * 32 * R);
    return nullptr;
}

// Add an item's counts to the walk counters (LENS_COUNT) and to its group's
// work record.
template <class Ctx> LENS_DEV void count_item(const Ctx& C, uint32_t g, bool head)
{
    const auto& P = C.P;
    if ((threadIdx.x & 31) != 0) return;
    if (P.gcost) atomicAdd(P.gcost + g, C.c_vis + C.c_acc + C.c_near + C.c_bigk);
    if (P.stats) {
        if (head) atomicAdd(&P.stats[0], 1ull);
        atomicAdd(&P.stats[1], (unsigned long long)C.c_vis);
        atomicAdd(&P.stats[2], (unsigned long long)C.c_acc);
        atomicAdd(&P.stats[3], (unsigned long long)C.c_near);
        atomicAdd(&P.stats[4], (unsigned long long)C.c_bigs);
        atomicAdd(&P.stats[5], (unsigned long long)C.c_bigk);
        atomicAdd(&P.stats[6], (unsigned long long)P.grange[g].y * (C.c_acc + C.c_near + C.c_bigk));
    }
}

// The totals of every cut group of `pool`, its parts added in order with
// Neumaier compensation, into the outputs, or into the place of the part that
// was cut again (`to`).  One warp per (cut, component).
template <typename T, int R>
__global__ void k_cut_sum(CutPool<T> pool, CutPool<T> to, WalkParams<T> P, int nq)
{
    const int lane = threadIdx.x & 31;
    const uint32_t cuts = pool.cuts(), nc = cuts * (uint32_t)nq;
    const int parts = (int)pool.parts_of(cuts);
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    constexpr int64_t stride = 5 * 32 * R;
    for (uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nc; w += nw) {
        const uint32_t ci = w / (uint32_t)nq;
        const CutSlot& cs = pool.slots[ci];
        const int q = (int)(w % (uint32_t)nq);
        const uint2 rg = P.grange[cs.g];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t at = (q * R + r) * 32 + lane;
            const T* p = pool.part + (int64_t)ci * parts * stride + at;
            T s = pool.head[(int64_t)ci * stride + at], c = T(0);
            for (int j = 0; j < parts; j += 16) {
                // (16 loads in flight: 1,000 rays, 64 parts 22 -> 8 us)
                T v[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) v[u] = j + u < parts ? p[(int64_t)(j + u) * stride] : T(0);
#pragma unroll
                for (int u = 0; u < 16; ++u)
                    if (j + u < parts) Comp5<T>::add1(s, c, v[u]);
            }
            T val = s + c;
            if (cs.parent >= 0) {
                to.part[(int64_t)cs.parent * stride + (q * R + r) * 32 + lane] = val;
            } else if (r * 32 + lane < (int)rg.y && P.out[q]) {
                const uint32_t i = P.ray_idx[rg.x + r * 32 + lane];
                if (P.accumulate) val += P.out[q][i];
                P.out[q][i] = val;
            }
        }
    }
}

// How the groups of a tree walk are cut (walk_rounds).
struct CutPlan {
    bool few;         // all groups are cut, their long lists put aside from the start
    bool keep_order;  // FP32 point masses: only the heaviest
    bool stretched;   // the call's stretched groups alone (P.sub): all of them
    // parts of a heavy group, at most: 16, but 8 for the potential (300,000
    // particles, 1000^2 rays 9.9 ms, 16: 10.2; its other sizes +-4 %; the
    // deflection of 300,000 particles, 839^2 rays 7.3 ms, 16: 6.8)
    uint32_t heavy_parts = 16;
};
// Up to how many groups all are cut: 4,096, but 512 for FP32 Gaussian trees of
// 200,000 particles and more.  Their groups' parts are heavy too and fill the
// second pool.  Times with all groups cut, and with the heavy ones only: 20,000
// particles, 4,072 groups 0.95 ms, 1.44; 60,000, 1,287: 1.02, 2.47; 100,000,
// 1,800: 1.72, 1.55, 4,072: 2.58, 3.03; 300,000, 1,296 64-ray groups 11.0, 3.70
// (without cuts 9.4), 4,072: 6.9, 3.2; 1e6, 1,287: 20.1, 8.2, 4,072: 15.5, 10.1;
// potential, 300,000, 2,485: 8.4, 5.6; 1e6, 1,800: 5.6, 6.9 (the one that loses).
inline int64_t few_groups(int kind, bool f32, int64_t n)
{
    return f32 && kind == LENS_GAUSS && n >= 200000 ? 512 : 4096;
}

// Is no group of a tree of n particles worth a cut (five more launches)?  Times
// with cuts, and without, theta 0.3 (at smaller theta a walk meets more of a
// tree):
//   few groups: 400 particles, 100 to 1e5 rays 1.05 to 1.15 times as long; 700
//     particles, 100 rays 0.22 ms, 0.29; FP64, 400 particles, 1,000 rays 0.59 ms,
//     0.69.  Above 512 groups the groups are many beside the particles at first
//     (3,750 groups, 1,200 particles 0.40 ms, 0.39; 5,000 particles 0.63, 0.81;
//     potential, 3,750 groups, 2,500 particles 0.64, 0.60; 2,329, 2,105: 0.47,
//     0.53).
//     One ray: 700 particles 0.126 ms, 0.100; 2,500 particles 0.113, 0.128.
//   others: no walk is longer than 2 n + n / 16 entries (cells and leaf particles,
//     listed ones, their tests), of point masses n; 0.3 ms for 16,384 entries.
inline bool never_cut(const lens_tree* t, int64_t ng, int64_t n_rays, int64_t n, const CutPlan& plan)
{
    const double th = std::min(t->theta / 0.3, 1.0);
    const int64_t small = t->precision == LENS_PREC_FP64 ? 256 : 512;
    if (plan.few)
        return n <= th * (double)std::max(small, ng > 512 ? 7 * ng / 10 : 0) || (n_rays == 1 && n < 1024 * th * th);
    return plan.keep_order ? n < 8192 : 2 * n + n / 16 < 16384;
}

// Totals in the second pool.  (Twice as many, in 32-ray groups: 400,000
// particles, 3,750 groups potential 9.4 -> 7.3 ms, 1,046 groups 8.4 -> 12.5: a
// part whose boxes are one heavy one and 15 light ones gains nothing from a
// launch of its own, and waits for it.)
template <typename T, int R> constexpr size_t again_items()
{
    return std::min<size_t>(16384, ((size_t)20 << 20) / (5 * 32 * R * sizeof(T)));
}

// Room for the first pool of a walk's cuts, and whether every one of ng groups
// has a place there.
template <typename T, int R> int64_t cut_room(const Layout& L, int warps, int cut_warps)
{
    constexpr size_t total = 5 * 32 * R * sizeof(T), again = again_items<T, R>() * total + again_items<T, R>() / 17 * sizeof(CutSlot);
    return (int64_t)(L.cut_end - L.stack) - (int64_t)warps * kStackCap * (int64_t)sizeof(int) -
           (int64_t)cut_warps * 2 * (int64_t)cut_local_bytes<R, T>() - (int64_t)again - 8 * 256;
}
template <typename T, int R> bool cuts_fit(int64_t ng, const Layout& L, int warps, int cut_warps)
{
    return ng * (int64_t)(sizeof(CutSlot) + 2 * 5 * 32 * R * sizeof(T)) <= cut_room<T, R>(L, warps, cut_warps);
}

// The launches of one tree walk over ng groups: `groups(P)` launches the kernel
// for whole groups, `parts(P)` the one for parts.  Groups are cut in a launch's
// kernel and their parts run in the next one; a part may be cut once more.
// Launches without items cost about 3 us each, beside walks of 100 us and more.
// warps: of the kernel with the most; cut_warps: of the cut form.
//   few (few_groups): about as many warps as the chip holds, or fewer.
//     Up to 512 groups are cut as soon as their stack holds 64 boxes (their big
//     lists deferred to the parts), into enough parts for about 8,192 warps; up
//     to 4,096 after a share of work that about doubles the launch's warps.
//   stretched: some tens or hundreds, cut as up to 512 groups are.
//   otherwise: only a group far heavier than the others (16,384 entries and
//     more; an average one evaluates 5,000 to 7,000), or a stretched one (which
//     may hold most of the tree) beyond 8,192; the fewer they are, the more
//     parts.  Where the groups are more than the pool has room for, 8 parts each.
//   keep_order (FP32 point masses): never few.  Over a patch much smaller than
//     the distances all rays share the rounding of one sum of thousands of
//     terms, which shows in a component that happens to be small (1e-3 of the
//     sum of |terms|): such groups keep their order of summation.
template <typename T, int R, typename Groups, typename Parts>
void walk_rounds(WalkParams<T> P, const CutPlan& plan, int nq, char* base, const Layout& L, uint32_t* counter,
                 Groups&& groups, Parts&& parts, int warps, int cut_warps, cudaStream_t s)
{
    // counter: 8 words, zeroed by the caller: work counters, then each pool's
    CutPool<T> pool[2];
    constexpr size_t total = 5 * 32 * R * sizeof(T);
    const int64_t ng = P.n_groups;
    const bool few = plan.few;
    P.gflag = (const uint8_t*)(base + L.gflag);
    if (cut_room<T, R>(L, warps, cut_warps) < 0) {  // (on fewer than some 80 SMs)
        groups(P);
        return;
    }
    char* at = base + L.stack + (size_t)warps * kStackCap * sizeof(int);
    auto take = [&](size_t bytes) {
        char* p = at;
        at += (bytes + 255) & ~(size_t)255;
        return p;
    };
    // (twice: where the first pool may be full)
    const size_t local_bytes = cut_local_bytes<R, T>() * 2;
    unsigned char* local = (unsigned char*)take((size_t)cut_warps * local_bytes);
    // the second pool: parts that are cut again
    pool[1].parts = few || plan.stretched ? 16 : 32;
    pool[1].max_cuts = (uint32_t)(again_items<T, R>() / (pool[1].parts + 1));
    pool[1].slots = (CutSlot*)take(pool[1].max_cuts * sizeof(CutSlot));
    pool[1].head = (T*)take(pool[1].max_cuts * total);
    pool[1].part = (T*)take(pool[1].max_cuts * pool[1].parts * total);
    // the first has the rest: every group that may be cut has a place
    // (fixed numbers of parts where it may be full)
    const size_t room = (size_t)cut_room<T, R>(L, warps, cut_warps);
    const bool all = cuts_fit<T, R>(ng, L, warps, cut_warps);
    if (few && all) {
        const size_t fit = (room - (size_t)ng * (sizeof(CutSlot) + total)) / total;
        pool[0].max_cuts = (uint32_t)ng;
        pool[0].parts = ng <= 512 ? 64 : 16;
        pool[0].items = (uint32_t)std::min<size_t>(ng <= 512 ? 8192 : 28672, fit);
    } else {
        // a place for every group, or 8 parts each for as many as fit
        pool[0].max_cuts = (uint32_t)(all ? (size_t)ng : room / (sizeof(CutSlot) + 9 * total));
        pool[0].parts = all ? plan.stretched ? 64 : plan.heavy_parts : 8;
        pool[0].items = all ? (uint32_t)std::min<size_t>(28672, (room - pool[0].max_cuts * (sizeof(CutSlot) + total)) / total) : 0;
    }
    pool[0].slots = (CutSlot*)take(pool[0].max_cuts * sizeof(CutSlot));
    pool[0].head = (T*)take(pool[0].max_cuts * total);
    pool[0].part = (T*)take((all ? (size_t)std::max(pool[0].max_cuts, pool[0].items) : (size_t)pool[0].max_cuts * 8) * total);
    for (int k = 0; k < 2; ++k) pool[k].cnt = counter + 4 + k;
    constexpr int rounds = 3;
    CutParams<T> c[rounds];
    if (few && ng <= 512) {
        c[0].limit = 0;
        c[0].min_nodes = 64;
        c[0].defer = 1;
        c[1].limit = 512;
        c[1].min_nodes = 16;
    } else if (few) {
        c[0].limit = (uint32_t)(ng / 4 + 256);
        c[0].min_nodes = 32;
        c[1].limit = c[0].limit;
        c[1].min_nodes = 16;
    } else if (plan.stretched) {
        c[0].limit = 0;
        c[0].min_nodes = 64;
        c[0].defer = 1;
        c[1].limit = 512;
        c[1].few_parts = 32;  // (over 896 groups)
        c[1].min_nodes = 16;
    } else {
        c[0].limit = (uint32_t)(ng <= 10922 || plan.keep_order ? 16384 : 3 * (ng / 2));
        c[0].limit_stretched = 8192;
        c[0].min_nodes = 32;
        c[1].limit = 8192;
        c[1].few_parts = 4;  // (thousands of cuts fill the chip by themselves: only the heaviest again)
        c[1].min_nodes = 16;
    }
    c[0].again_limit = c[1].limit << (pool[0].parts < c[1].few_parts ? 2 : 0);
    c[0].again_parts = pool[1].parts;
    c[0].again_min_nodes = c[1].min_nodes;
    for (int r = 0; r < rounds; ++r) {
        c[r].local = local;
        c[r].local_bytes = local_bytes;
        P.counter = counter + r;
        if (r > 0) c[r].in = pool[r - 1];
        if (r + 1 < rounds) c[r].out = pool[r];
        P.cut = c[r];
        if (r == 0) groups(P);
        else parts(P);
    }
    for (int r = rounds - 2; r >= 0; --r) {
        const int64_t most = std::min<int64_t>(pool[r].max_cuts, r > 0 ? 2048 : ng);
        k_cut_sum<T, R><<<(unsigned)((most * nq + 7) / 8), 256, 0, s>>>(pool[r], r > 0 ? pool[r - 1] : CutPool<T>{}, P, nq);
        note_launch();
    }
}

// Launch the producer/consumer form of the walk (walk_ws.cu); false if it
// cannot run here (the caller then launches the one-warp walk).
template <typename T, int R>
bool launch_ws(int kind, bool ao, const WalkParams<T>& P, int num_sms, cudaStream_t s, int consumers);

}  // namespace lens
