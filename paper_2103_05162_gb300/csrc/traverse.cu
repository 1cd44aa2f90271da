// The two traversal phases of the parallel disjoint-set DBSCAN (Sec. 3.2,
// Algorithm 3) over the BVH of Sec. 4.1/4.2, plus union-find initialisation,
// final compression (Sec. 4.3) and canonical relabelling.
//
// Work is organised per BVH leaf and per warp: a leaf is either a tile of up
// to 32 sorted points outside dense cells (one point per lane) or a whole
// dense cell (Sec. 4.2). A warp takes the next leaf from a global counter
// (persistent kernels) and goes through the leaves within eps of it, 32 at a
// time, one per lane: from the leaf's list, or from a walk of the tree that
// expands up to 32 nodes a step. Those that pass the lane's test give their
// points in one stream, one per lane; the points near the query box are
// staged, and a full stage is tested against the tile's points.
//
// Exact shortcuts cut the pair tests in dense regions:
//  * containment: when the farthest corners of a leaf's box and the query box
//    are within eps, every pair between them is (no per-point tests);
//  * solid leaves: a leaf whose points are all core and already one set
//    (every dense cell, and every tile that becomes so) behaves like a dense
//    cell of Sec. 4.2: one adjacent pair decides;
//  * sets: a pair whose points shared a set at any time needs no test (sets
//    never split). Consecutive leaves are united first (link_next), so that
//    dense regions start the main phase as a few sets.
//
// Preprocessing (minPts > 2 only): each point outside dense cells counts its
// neighbours (itself included) and stops at minPts; points of dense cells are
// core by construction.
// Intra: each tile unites its own pairs, records whether it is solid, and is
// united with the next leaf.
// Main: each leaf visits only the leaves with index > its own (the pair mask
// of Sec. 4.1, Figure "pair traversal"), so every pair is seen once, and
// applies the rule of Algorithm 3 as it finds each pair, with no neighbour
// list: core-core pairs are united, a core point claims a non-core neighbour
// with one compare-and-swap (Sec. 3.2).
#include <algorithm>
#include <climits>
#include <map>
#include <mutex>
#include <tuple>

#include "build.cuh"

namespace gbd {

namespace {

constexpr int TREE_DEPTH = 97;    // the largest possible tree depth (64-bit keys and an index tie-break)
constexpr int STACK = 384;        // a walk's stack: wide steps, which add up to 32 entries, up to STACK_WIDE,
constexpr int STACK_WIDE = 224;   // then one node a step, whose depth-first growth stays below the tree depth
static_assert(STACK_WIDE + 32 + TREE_DEPTH < STACK, "a walk's stack");

// Node access and the box tests of both children at once (packed pairs: the
// left child in the low half, the right child in the high half). The general
// template covers 4 to 8 dimensions; 2 and 3 are specialised.
template <int D> struct NB {
    using T = Traits<D>;
    struct PP { f32x2 c[D]; };
    __device__ static __forceinline__ PP pack(const typename T::Point& p)
    {
        PP r;
#pragma unroll
        for (int k = 0; k < D; ++k) r.c[k] = pk2(p.c[k], p.c[k]);
        return r;
    }
    __device__ static __forceinline__ typename T::Node load(const typename T::Node* n, int i)
    {
        typename T::Node r;
#pragma unroll
        for (int k = 0; k < D; ++k) r.ax[k] = __ldg(&n[i].ax[k]);
        r.m = __ldg(&n[i].m);
        return r;
    }
    __device__ static __forceinline__ void bd2(const typename T::Node& n, const typename T::Box& q, float& dl,
                                               float& dr)
    {
        GBD_COUNT(CNT_BOX, 2);
        f32x2 s = sqr2(gap2_rn2(pk2(q.lo.c[0], q.lo.c[0]), pk2(q.hi.c[0], q.hi.c[0]), pk2(n.ax[0].x, n.ax[0].y),
                                pk2(n.ax[0].z, n.ax[0].w)));
#pragma unroll
        for (int k = 1; k < D; ++k)
            s = add2(s, sqr2(gap2_rn2(pk2(q.lo.c[k], q.lo.c[k]), pk2(q.hi.c[k], q.hi.c[k]),
                                      pk2(n.ax[k].x, n.ax[k].y), pk2(n.ax[k].z, n.ax[k].w))));
        unpk2(s, dl, dr);
    }
    __device__ static __forceinline__ float pbox(const typename T::Point& p, const typename T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_dist2(p, b);
    }
    __device__ static __forceinline__ float bbox(const typename T::Box& q, const typename T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_box_dist2(q, b);
    }
    __device__ static __forceinline__ typename T::Point shfl(const typename T::Point& p, int src)
    {
        typename T::Point r = p;
#pragma unroll
        for (int k = 0; k < D; ++k) r.c[k] = __shfl_sync(FULL, p.c[k], src);
        return r;
    }
};
template <> struct NB<3> {
    using T = Traits<3>;
    struct PP { f32x2 x, y, z; };  // a point's coordinates, each twice
    __device__ static __forceinline__ PP pack(const T::Point& p) { return PP{pk2(p.x, p.x), pk2(p.y, p.y), pk2(p.z, p.z)}; }
    __device__ static __forceinline__ T::Node load(const T::Node* n, int i)
    {
        T::Node r;
        // 64-byte records at 64-byte boundaries: two 256-bit loads
        float4 mf;
        ldg256(&n[i].a, r.a, r.b);
        ldg256(&n[i].c, r.c, mf);
        r.m = make_int4(__float_as_int(mf.x), __float_as_int(mf.y), __float_as_int(mf.z), __float_as_int(mf.w));
        return r;
    }
    // squared box-to-box distances of both children from q (box_box_dist2's order)
    __device__ static __forceinline__ void bd2(const T::Node& n, const T::Box& q, float& dl, float& dr)
    {
        GBD_COUNT(CNT_BOX, 2);
        f32x2 s = sqr2(gap2_rn2(pk2(q.lo.x, q.lo.x), pk2(q.hi.x, q.hi.x), pk2(n.a.x, n.a.y), pk2(n.a.z, n.a.w)));
        s = add2(s, sqr2(gap2_rn2(pk2(q.lo.y, q.lo.y), pk2(q.hi.y, q.hi.y), pk2(n.b.x, n.b.y), pk2(n.b.z, n.b.w))));
        s = add2(s, sqr2(gap2_rn2(pk2(q.lo.z, q.lo.z), pk2(q.hi.z, q.hi.z), pk2(n.c.x, n.c.y), pk2(n.c.z, n.c.w))));
        unpk2(s, dl, dr);
    }
    __device__ static __forceinline__ float pbox(const T::Point& p, const T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_dist2(p, b.lo.x, b.lo.y, b.lo.z, b.hi.x, b.hi.y, b.hi.z);
    }
    __device__ static __forceinline__ float bbox(const T::Box& q, const T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_box_dist2(q, b.lo.x, b.lo.y, b.lo.z, b.hi.x, b.hi.y, b.hi.z);
    }
    __device__ static __forceinline__ T::Point shfl(const T::Point& p, int src)
    {
        return make_float4(__shfl_sync(FULL, p.x, src), __shfl_sync(FULL, p.y, src), __shfl_sync(FULL, p.z, src), 0.f);
    }
};
template <> struct NB<2> {
    using T = Traits<2>;
    struct PP { f32x2 x, y; };
    __device__ static __forceinline__ PP pack(const T::Point& p) { return PP{pk2(p.x, p.x), pk2(p.y, p.y)}; }
    __device__ static __forceinline__ T::Node load(const T::Node* n, int i)
    {
        T::Node r;
        r.a = __ldg(&n[i].a); r.b = __ldg(&n[i].b); r.m = __ldg(&n[i].m);
        return r;
    }
    __device__ static __forceinline__ void bd2(const T::Node& n, const T::Box& q, float& dl, float& dr)
    {
        GBD_COUNT(CNT_BOX, 2);
        f32x2 s = sqr2(gap2_rn2(pk2(q.lo.x, q.lo.x), pk2(q.hi.x, q.hi.x), pk2(n.a.x, n.a.y), pk2(n.a.z, n.a.w)));
        s = add2(s, sqr2(gap2_rn2(pk2(q.lo.y, q.lo.y), pk2(q.hi.y, q.hi.y), pk2(n.b.x, n.b.y), pk2(n.b.z, n.b.w))));
        unpk2(s, dl, dr);
    }
    __device__ static __forceinline__ float pbox(const T::Point& p, const T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_dist2(p, b.lo.x, b.lo.y, b.hi.x, b.hi.y);
    }
    __device__ static __forceinline__ float bbox(const T::Box& q, const T::Box& b)
    {
        GBD_COUNT(CNT_BOX, 1);
        return T::box_box_dist2(q, b.lo.x, b.lo.y, b.hi.x, b.hi.y);
    }
    __device__ static __forceinline__ T::Point shfl(const T::Point& p, int src)
    {
        return make_float2(__shfl_sync(FULL, p.x, src), __shfl_sync(FULL, p.y, src));
    }
};

// Up to 32 staged points by coordinate (structure of arrays): two
// neighbouring points load as one packed pair per axis.
template <int D> struct __align__(16) SoA {
    float c[D][32];
    __device__ __forceinline__ void put(int l, const typename Traits<D>::Point& p)
    {
#pragma unroll
        for (int k = 0; k < D; ++k) c[k][l] = p.c[k];
    }
    __device__ __forceinline__ typename Traits<D>::Point get(int l) const
    {
        typename Traits<D>::Point p{};
#pragma unroll
        for (int k = 0; k < D; ++k) p.c[k] = c[k][l];
        return p;
    }
    __device__ __forceinline__ void d2pair(const typename NB<D>::PP& p, int u, float& d0, float& d1) const
    {
        GBD_COUNT(CNT_DIST, 2);
        f32x2 s = sqr2(sub2(p.c[0], *reinterpret_cast<const f32x2*>(&c[0][u])));
#pragma unroll
        for (int k = 1; k < D; ++k) s = add2(s, sqr2(sub2(p.c[k], *reinterpret_cast<const f32x2*>(&c[k][u]))));
        unpk2(s, d0, d1);
    }
    __device__ __forceinline__ float d2(const typename Traits<D>::Point& p, int u) const
    {
        GBD_COUNT(CNT_DIST, 1);
        float s = sqr_rn(__fsub_rn(p.c[0], c[0][u]));
#pragma unroll
        for (int k = 1; k < D; ++k) s = __fadd_rn(s, sqr_rn(__fsub_rn(p.c[k], c[k][u])));
        return s;
    }
};
template <> struct __align__(16) SoA<3> {
    float x[32], y[32], z[32];
    __device__ __forceinline__ void put(int l, const float4& p) { x[l] = p.x; y[l] = p.y; z[l] = p.z; }
    __device__ __forceinline__ float4 get(int l) const { return make_float4(x[l], y[l], z[l], 0.f); }
    // dist2(p, point u) and dist2(p, point u + 1) for even u (p packed)
    __device__ __forceinline__ void d2pair(const NB<3>::PP& p, int u, float& d0, float& d1) const
    {
        GBD_COUNT(CNT_DIST, 2);
        const f32x2 bx = *reinterpret_cast<const f32x2*>(&x[u]);
        const f32x2 by = *reinterpret_cast<const f32x2*>(&y[u]);
        const f32x2 bz = *reinterpret_cast<const f32x2*>(&z[u]);
        f32x2 s = sqr2(sub2(p.x, bx));
        s = add2(s, sqr2(sub2(p.y, by)));
        s = add2(s, sqr2(sub2(p.z, bz)));
        unpk2(s, d0, d1);
    }
    __device__ __forceinline__ float d2(const float4& p, int u) const { return dist2(p, make_float4(x[u], y[u], z[u], 0.f)); }
};
template <> struct __align__(16) SoA<2> {
    float x[32], y[32];
    __device__ __forceinline__ void put(int l, const float2& p) { x[l] = p.x; y[l] = p.y; }
    __device__ __forceinline__ float2 get(int l) const { return make_float2(x[l], y[l]); }
    __device__ __forceinline__ void d2pair(const NB<2>::PP& p, int u, float& d0, float& d1) const
    {
        GBD_COUNT(CNT_DIST, 2);
        const f32x2 bx = *reinterpret_cast<const f32x2*>(&x[u]);
        const f32x2 by = *reinterpret_cast<const f32x2*>(&y[u]);
        f32x2 s = sqr2(sub2(p.x, bx));
        s = add2(s, sqr2(sub2(p.y, by)));
        unpk2(s, d0, d1);
    }
    __device__ __forceinline__ float d2(const float2& p, int u) const { return dist2(p, make_float2(x[u], y[u])); }
};

// a node or leaf box: one 256-bit load where it is a 32-byte record (2D, 3D)
template <int D>
__device__ __forceinline__ typename Traits<D>::Box load_box(const typename Traits<D>::Box* __restrict__ boxes,
                                                            int64_t i)
{
    typename Traits<D>::Box b;
    if constexpr (sizeof(typename Traits<D>::Box) == 32) ldg256(&boxes[i], b.lo, b.hi);
    else b = boxes[i];
    return b;
}

// The points of up to 32 leaves (one per lane with `on`: [us, ue)) in one
// stream, in lane order and ascending within a leaf: each lane gets one point
// a step, whatever the sizes of the leaves, and the next step's points are
// loaded while the current ones are looked at. Visiting the leaves one by one
// cost a chain of dependent loads for each, with a third of the lanes idle.
// (PointStream needs a leaf with `on` in some lane.)
struct StreamMem {
    int first[32];  // per leaf of the stream: its first point less its first position
};

template <int D>
struct PointStream {
    using P = typename Traits<D>::Point;
    const P* __restrict__ sp;
    StreamMem& st;
    int off;       // first position of this lane's leaf in the stream (no leaf: beyond any)
    int total;
    int before;    // leaves that start before the current 32 positions, less one
    int b;         // the step's first position
    int lane;
    // this lane's point of the step (in: it has one), and the next step's
    bool in;
    int j, jn;
    P p, pn;

    __device__ __forceinline__ PointStream(const P* sp_, StreamMem& st_, bool on, int us, int ue, int lane_)
        : sp(sp_), st(st_), lane(lane_)
    {
        const int size = on ? ue - us : 0;
        off = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, off, o);
            if (lane >= o) off += y;
        }
        total = __shfl_sync(FULL, off, 31);
        off -= size;
        const unsigned om = __ballot_sync(FULL, on);
        __syncwarp();
        if (on) {
            const int r = __popc(om & ((1u << lane) - 1u));
            st.first[r] = us - off;
        } else {
            off = INT_MAX;
        }
        __syncwarp();
        before = -1;
        b = -32;
        load(0);
    }
    __device__ __forceinline__ void load(int at)
    {
        const unsigned t = (unsigned)(off - at);
        const unsigned sm = __reduce_or_sync(FULL, t < 32u ? 1u << t : 0u);
        const int r = before + __popc(sm & (0xffffffffu >> (31 - lane)));
        before += __popc(sm);
        jn = st.first[r] + min(at + lane, total - 1);  // (past the end: the last point)
        pn = sp[jn];
    }
    __device__ __forceinline__ bool next()
    {
        b += 32;
        in = b + lane < total;
        j = jn;
        p = pn;
        if (b + 32 < total) load(b + 32);
        return b < total;
    }
};

// per leaf: at most SIBCAP sibling subtrees are recorded (more: the start
// node is used instead), and at most LEAFCAP leaves within eps
constexpr int SIBCAP = TRAVERSAL_SIBCAP;
constexpr int LEAFCAP = TRAVERSAL_LEAFCAP;

// The bounding box of the points of the lanes with `on` (empty if none): a
// query box for all of them at once. For p inside it every per-axis gap to a
// box is at least the box-to-box gap (monotone rounding, same order of the
// sum), so a box farther than eps from it is farther from each point.
template <int D>
__device__ __forceinline__ typename Traits<D>::Box warp_box(const typename Traits<D>::Point& p, bool on)
{
    using T = Traits<D>;
    typename T::Box b = on ? T::point_box(p) : T::empty_box();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) T::merge(b, T::shfl_xor(b, o));
    return b;
}

// the lanes of a tile of k <= 32 points
__device__ __forceinline__ unsigned tile_lanes(int k) { return k >= 32 ? FULL : ((1u << k) - 1u); }

// Per-warp shared memory of both phases.
template <int D>
struct WarpMem {
    SoA<D> soa;      // staged points
    int idx[32];     // and their indices (main phase: top bit: not core)
    StreamMem st;
    int stack[STACK];
    int cand[64];
};

template <int D>
struct DevArgs {
    const typename Traits<D>::Point* sp;
    const typename Traits<D>::Node* nodes;
    const typename Traits<D>::Box* leafbox;
    const int2* leafr;
    uint8_t* lsolid;
    int32_t* klist;  // m_cap entries per leaf kind
    int64_t m_cap;
    int32_t* labels;
    uint8_t* core;
    uint8_t* nbr;
    int32_t* nlist;
    int lcap;
    bool whole_intra;  // k_intra also makes the lists' claims and groups the leaves by kind
    uint32_t* ctrl;
    float e2;
    int min_pts;
    int mode;
    // batches of independent instances: per-leaf instance and per-instance
    // eps^2, minPts and subtree root (all null for a single instance)
    const int32_t* linst;
    const float* e2s;
    const int32_t* mps;
    const int32_t* iroot;
    // per leaf without a list: the node its traversals start at, and the
    // sibling subtrees on the way down that come within eps (tile_start)
    int32_t* tstart;
    int2* tsib;
    int8_t* tnsib;
    // multi-minPts runs: neighbour counts capped at min_pts (null otherwise)
    int32_t* ncount;
    // per leaf: the leaves within eps of its box (k_leaf_lists)
    int32_t* llist;
    int16_t* lcount;
};

// eps^2, minPts and the traversal start of the tile's instance
struct TileParams {
    float e2;
    int min_pts;
    int start;
};
template <int D>
__device__ __forceinline__ TileParams tile_params(const DevArgs<D>& a, int L)
{
    if (!a.linst) return TileParams{a.e2, a.min_pts, 0};
    const int b = a.linst[L];
    return TileParams{a.e2s[b], a.mps[b], a.iroot[b]};
}

// The lowest ancestor A of a leaf such that no point outside A's subtree is
// within eps of the leaf's box, and the sibling subtrees on the way down from
// A that come within eps of it: traversals for the leaf's points (each within
// the leaf box) then start at A, or at those siblings, instead of the root and
// skip the levels above, where only one path could lead to a neighbour. Found
// from the top: one node record per level holds both children's boxes and
// says on which side the leaf lies, so a level is one dependent load, and the
// upper levels are the same for all lanes. Climbing from the leaf took three
// per level (parent, its children, the sibling's box) and 409 us for the lists
// of 16.8M halos, where this takes 363: most of it is the walk below the
// siblings.
//
// Returns the number of siblings (-1: more than SIBCAP); the first SIBCAP go
// to near(k, sibling, last leaf under it) from the top down.
template <int D, typename Near>
__device__ __forceinline__ int tile_start(const DevArgs<D>& a, int L, int leaf0, const TileParams& tp,
                                          const typename Traits<D>::Box& q, int& start, Near near)
{
    int cur = tp.start, ns = 0;
    start = leaf0 + L;
    // a longer way down than the tree is deep means a corrupt tree: start at
    // the root
#pragma unroll 1
    for (int steps = 0; cur < leaf0; ++steps) {
        if (steps > TREE_DEPTH) {
            start = tp.start;
            return -1;
        }
        const auto nd = NB<D>::load(a.nodes, cur);
        float dl, dr;
        NB<D>::bd2(nd, q, dl, dr);
        const bool right = L > nd.m.z;
        if ((right ? dl : dr) <= tp.e2) {
            if (ns == 0) start = cur;
            if (ns < SIBCAP) near(ns, right ? nd.m.x : nd.m.y, right ? nd.m.z : nd.m.w);
            ++ns;
        }
        cur = right ? nd.m.y : nd.m.x;
    }
    return ns <= SIBCAP ? ns : -1;
}

// The roots of leaf L's walk onto an empty stack (the top is taken first):
// its sibling leaves from the farthest ancestor down, then the sibling
// subtrees from the nearest up, or the start node where there are more than
// SIBCAP of them. Subtrees whose leaves all precede mask_lo are left out.
template <int D>
__device__ __forceinline__ int walk_roots(const DevArgs<D>& a, int L, int leaf0, int mask_lo, int* stack, int lane)
{
    const int ns = a.tnsib[L];
    int item = -1;
    if (ns >= 0) {
        if (lane < ns) {
            const int2 t = a.tsib[(int64_t)L * SIBCAP + ns - 1 - lane];
            if (t.y >= mask_lo) item = t.x;
        }
    } else if (lane == 0) {
        item = a.tstart[L];
    }
    const unsigned lm = __ballot_sync(FULL, item >= leaf0), im = __ballot_sync(FULL, item >= 0 && item < leaf0);
    const int sp = __popc(lm) + __popc(im);
    const int pos = item >= leaf0 ? __popc(lm >> lane) - 1 : __popc(lm) + __popc(im & ((1u << lane) - 1u));
    if (item >= 0) stack[sp - 1 - pos] = item;
    __syncwarp();
    return sp;
}

// A node's children within eps of the box q, in the order they are taken:
// leaves before subtrees, left before right (RIGHT: the right one of two
// subtrees first; -1: none)
template <int D, bool RIGHT = false>
__device__ __forceinline__ int2 near_children(const DevArgs<D>& a, int node, const typename Traits<D>::Box& q, float e2,
                                              int leaf0, int mask_lo)
{
    const auto nd = NB<D>::load(a.nodes, node);
    float dl, dr;
    NB<D>::bd2(nd, q, dl, dr);
    int l = dl <= e2 && nd.m.z >= mask_lo ? nd.m.x : -1;
    int r = dr <= e2 && nd.m.w >= mask_lo ? nd.m.y : -1;
    if (l < 0 || (l < leaf0 && (r >= leaf0 || (RIGHT && r >= 0)))) { const int t = l; l = r; r = t; }
    return make_int2(l, r);
}

// Where a leaf has no list (more than LEAFCAP leaves within eps): the next
// leaves of its walk through the tree, up to 32 of them into wm.cand (mask_lo:
// only leaves from there on). Up to 32 nodes from the top of the stack are
// expanded a step, each in place, so that the leaves come out in the order of
// a walk that takes one node at a time -- whose chain of dependent loads, one
// per node, was a third of the main phase on dense data. Returns how many
// (fewer than 32: the walk is over).
template <int D, bool RIGHT = false>
__device__ __forceinline__ int walk_next(const DevArgs<D>& a, WarpMem<D>& wm, int& sp, int& nc, int64_t& steps,
                                         int64_t m, const typename Traits<D>::Box& q, float e2, int mask_lo, int lane)
{
    const int leaf0 = (int)(m - 1);
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
    while (sp > 0 && nc < 32) {
        // each step enters a node or emits a leaf, each at most once; more
        // steps can only come from a corrupt tree: flag it and stop
        if (++steps > 2 * m) {
            if (lane == 0) atomicOr(&a.ctrl[CTRL_ERR], ERR_STACK);
            sp = 0;
            break;
        }
        const int np = sp > STACK_WIDE ? 1 : min(sp, 32);
        const int item = lane < np ? wm.stack[sp - 1 - lane] : -1;
        __syncwarp();
        // the leaves before the first subtree are next in order
        const unsigned sub = __ballot_sync(FULL, item >= 0 && item < leaf0);
        const int lead = sub ? __ffs(sub) - 1 : np;
        const bool emit = lane < lead && item - leaf0 >= mask_lo;
        const unsigned em = __ballot_sync(FULL, emit);
        if (emit) wm.cand[nc + __popc(em & lt)] = item - leaf0;
        nc += __popc(em);
        // the others stay, subtrees replaced by their children
        int2 c = make_int2(-1, -1);
        if (lane >= lead && lane < np) {
            GBD_COUNT(CNT_NODE, item < leaf0);
            c = item >= leaf0 ? make_int2(item, -1) : near_children<D, RIGHT>(a, item, q, e2, leaf0, mask_lo);
        }
        const unsigned c1 = __ballot_sync(FULL, c.x >= 0), c2 = __ballot_sync(FULL, c.y >= 0);
        sp += __popc(c1) + __popc(c2) - np;
        if (sp > STACK) {
            if (lane == 0) atomicOr(&a.ctrl[CTRL_ERR], ERR_STACK);
            sp = 0;
            break;
        }
        const int pos = sp - 1 - __popc(c1 & lt) - __popc(c2 & lt);
        if (c.x >= 0) wm.stack[pos] = c.x;
        if (c.y >= 0) wm.stack[pos - 1] = c.y;
        __syncwarp();
    }
    return min(nc, 32);
}

// the leaves handed out by walk_next are done with: the rest moves up
template <int D>
__device__ __forceinline__ int walk_take(WarpMem<D>& wm, int& nc, int lane)
{
    const int U = lane < nc ? wm.cand[lane] : -1;
    const int V = lane + 32 < nc ? wm.cand[lane + 32] : -1;
    __syncwarp();
    if (V >= 0) wm.cand[lane] = V;
    nc = max(nc - 32, 0);
    __syncwarp();
    return U;
}

// The leaves whose boxes come within eps of each leaf's box (itself
// excluded), found once per leaf by one thread walking the subtrees recorded
// by tile_start with the leaf box as the query (box-to-box test, exact by
// the same monotone-rounding argument). Every neighbour of a point of the
// leaf lies in one of them, so the traversals of both phases can go through
// the list instead of the tree. More than LEAFCAP leaves: count -1, and the
// phases walk the tree for that leaf (walk_next).
// (each thread's walk stack lives in shared memory as column threadIdx.x of
// [depth][LL_THREADS]: lanes at different depths still fall in distinct
// banks, where a local-memory stack costs a transaction per distinct depth;
// a walk deeper than LL_STACK gives up its list as well)
constexpr int LL_THREADS = 256;
constexpr int LL_STACK = 48;
// Up to so many leaves per warp of the launch (of 8 in each of up to 1,216
// blocks, half of which are resident at once), a warp makes a list: a thread's
// walk is a chain of one load per node, a warp's of one per level or so (16,384
// blob points: 42 us by threads, 19 by warps). With more leaves, threads keep
// more walks in flight. Whole runs by threads and by warps, in us: below the
// line blobs 349 and 294 (262,144), 500 and 441 (1M), halos 358 and 331
// (262,144), roads, whose walks are short, 202 and 214 (262,144); above it
// halos 446 and 433 (524,287), 606 and 666 (1M), 4265 and 6200 (16.8M), roads
// 278 and 308 (524,287).
constexpr int LL_ROUNDS = 2;

// Leaf L's list by a whole warp: the same list in the same order (the nearest
// sibling leaves first, then the sibling subtrees from the farthest down, a
// node's leaves before its subtrees, its right subtree first).
template <int D>
__device__ __forceinline__ void warp_list(const DevArgs<D>& a, int L, int64_t m, WarpMem<D>& wm, int lane)
{
    const int leaf0 = (int)(m - 1);
    const TileParams tp = tile_params(a, L);
    const typename Traits<D>::Box q = load_box<D>(a.leafbox, L);
    int32_t* out = a.llist + (int64_t)L * LEAFCAP;
    int2 mine = make_int2(-1, 0);  // lane k: sibling k from the top and the last leaf under it
    int start, cnt = LEAFCAP + 1;
    const int ns = tile_start<D>(a, L, leaf0, tp, q, start, [&](int k, int sib, int last) {
        if (lane == k) mine = make_int2(sib, last);
    });
    if (ns >= 0) {
        const unsigned lm = __ballot_sync(FULL, mine.x >= leaf0);
        const unsigned im = __ballot_sync(FULL, mine.x >= 0 && mine.x < leaf0);
        if (mine.x >= leaf0) out[__popc(lm >> lane) - 1] = mine.x - leaf0;
        else if (mine.x >= 0) wm.stack[__popc(im >> lane) - 1] = mine.x;
        __syncwarp();
        cnt = __popc(lm);
        int sp = __popc(im), nc = 0;
        int64_t steps = 0;
        while (cnt <= LEAFCAP) {
            const int k = walk_next<D, true>(a, wm, sp, nc, steps, m, q, tp.e2, 0, lane);
            if (k == 0) break;
            const int U = walk_take<D>(wm, nc, lane);
            if (U >= 0 && cnt + lane < LEAFCAP) out[cnt + lane] = U;
            cnt += k;
        }
        __syncwarp();
    }
    if (lane == 0) a.lcount[L] = cnt <= LEAFCAP ? (int16_t)cnt : (int16_t)-1;
    if (cnt > LEAFCAP) {  // walks of this leaf begin at its siblings or its start
        if (lane < ns) a.tsib[(int64_t)L * SIBCAP + lane] = mine;
        if (lane == 0) {
            a.tnsib[L] = (int8_t)ns;
            a.tstart[L] = start;
        }
    }
}

template <int D>
__global__ void __launch_bounds__(LL_THREADS) k_leaf_lists(const __grid_constant__ DevArgs<D> a)
{
    stage_begin();
    using T = Traits<D>;
    const int64_t m = a.ctrl[CTRL_M];
    const int leaf0 = (int)(m - 1);
    __shared__ __align__(16) int s_stk[LL_STACK][LL_THREADS];
    int* const stk = &s_stk[0][threadIdx.x];  // stk[k * LL_THREADS]: entry k
    static_assert(sizeof(WarpMem<D>) * (LL_THREADS / 32) <= sizeof(s_stk), "the warps' walks fit");
    const int64_t warps = (int64_t)gridDim.x * (LL_THREADS / 32);
    if (m <= LL_ROUNDS * warps) {
        WarpMem<D>& wm = reinterpret_cast<WarpMem<D>*>(&s_stk[0][0])[threadIdx.x >> 5];
        for (int64_t L = blockIdx.x * (int64_t)(LL_THREADS / 32) + (threadIdx.x >> 5); L < m; L += warps)
            warp_list(a, (int)L, m, wm, threadIdx.x & 31);
        return;
    }
    for (int64_t L = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; L < m; L += (int64_t)gridDim.x * blockDim.x) {
        const TileParams tp = tile_params(a, (int)L);
        typename T::Box q;
        q = load_box<D>(a.leafbox, L);
        int32_t* out = a.llist + L * LEAFCAP;
        int cnt = 0, sp = 0, start;
        // the siblings wait at the end of the stack, the nearest first, and
        // are moved to its start (never past the next one to be read)
        static_assert(SIBCAP <= LL_STACK, "siblings fit the stack");
        const int ns = tile_start<D>(a, (int)L, leaf0, tp, q, start,
                                     [&](int k, int sib, int) { stk[LL_THREADS * (LL_STACK - 1 - k)] = sib; });
        if (ns < 0) cnt = LEAFCAP + 1;
        for (int j = LL_STACK - ns; j < LL_STACK; ++j) {
            const int r = stk[LL_THREADS * j];
            if (r >= leaf0) {  // a leaf sibling: within eps of the box by construction
                if (cnt < LEAFCAP) out[cnt] = r - leaf0;
                ++cnt;
            } else {
                stk[LL_THREADS * sp++] = r;
            }
        }
        int64_t steps = 0;
        while (sp > 0 && cnt <= LEAFCAP) {
            if (++steps > m) {
                atomicOr(&a.ctrl[CTRL_ERR], ERR_STACK);
                cnt = LEAFCAP + 1;
                break;
            }
            const int node = stk[LL_THREADS * --sp];
            const auto nd = NB<D>::load(a.nodes, node);
            float dl, dr;
            NB<D>::bd2(nd, q, dl, dr);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if ((c ? dr : dl) > tp.e2) continue;
                const int child = c ? nd.m.y : nd.m.x;
                if (child >= leaf0) {
                    if (child - leaf0 != (int)L) {
                        if (cnt < LEAFCAP) out[cnt] = child - leaf0;
                        ++cnt;
                    }
                } else if (sp < LL_STACK) {
                    stk[LL_THREADS * sp++] = child;
                } else {
                    cnt = LEAFCAP + 1;
                }
            }
        }
        a.lcount[L] = cnt <= LEAFCAP ? (int16_t)cnt : (int16_t)-1;
        if (cnt > LEAFCAP) {  // walks of this leaf begin at its siblings or its start
            a.tnsib[L] = (int8_t)tile_start<D>(a, (int)L, leaf0, tp, q, start, [&](int k, int sib, int last) {
                a.tsib[L * SIBCAP + k] = make_int2(sib, last);
            });
            a.tstart[L] = start;
        }
    }
}

__device__ __forceinline__ int next_leaf(uint32_t* ctr)
{
    int L = 0;
    if ((threadIdx.x & 31) == 0) L = (int)atomicAdd(ctr, 1u);
    return __shfl_sync(FULL, L, 0);
}

// Register caps of the preprocessing kernel: 48 in 3D (16.8M halos 1356 us when
// taken, 56: 1397), 56 in 2D (4.2M road points 314, 48: 328), 80 in 5D (400K points
// 239, 96: 252). Whole runs with this and the main phase's caps 8 to 24 lower or
// 8 to 32 higher, 2D to 8D, both algorithms: lower -1 to 8% slower; higher 2 to
// 8% slower from 400,000 points in 4D to 8D and 0.5 to 2% on 4.2M points, up to
// 1.5% faster in 2D and 3D and at 20,000 points.
template <int D>
constexpr int traversal_regs()
{
    return D == 2 ? 56 : (D == 3 ? 48 : (D <= 5 ? 80 : 112));
}

// (the main phase holds more state per lane and waits on union-find chains)
template <int D>
constexpr int main_regs()
{
    return D <= 3 ? 64 : (D <= 5 ? 96 : 128);
}

// Preprocessing: each point outside dense cells counts its neighbours (itself
// included) and stops at minPts (Sec. 3.2, 4.1, 4.2). A warp takes a tile,
// one point per lane: its own points first, then the points of the leaves
// within eps, 32 leaves at a time. Their points pass by in one stream, one per
// lane; those within eps of the box of the queries still counting are staged,
// and every 32 of them (or the last) are tested against the queries, looping
// over the smaller side. The order of the list and of the points in a leaf is
// kept, so a query's neighbours are found in the order of the lists.
// Issue-bound (79% of the slots on 4.2M halos): visiting leaf by leaf, with a
// test of each query against each leaf's box, took 1580 us on 16.8M halos and
// 338 us on 400K 5D points, this takes 1337 and 235 us.
constexpr int FEW_QUERIES = 8;

template <int D>
struct PreWarp {
    using T = Traits<D>;
    using P = typename T::Point;
    const DevArgs<D>& a;
    WarpMem<D>& wm;
    int lane;
    float e2;
    int min_pts;
    int qs;       // the tile's first point
    P p;
    bool act;     // this lane's query still counts
    int cnt;
    // lane l's query (point qs + l) records its out-of-tile neighbours while
    // its count is below minPts, so a query that ends non-core has all of
    // them (nl <= minPts - 1 = lcap; lcap 0: no lists)
    int nl;
    typename T::Box qbox;  // box of the queries that count when the walk starts

    // n staged points against the queries still counting
    __device__ __forceinline__ void flush(int n)
    {
        __syncwarp();
        unsigned am = __ballot_sync(FULL, act);
        const unsigned am0 = am;
        const bool list = a.lcap > 0;
        int32_t* row = a.nlist + (int64_t)(qs + lane) * a.lcap;
        if (2 * __popc(am) < n) {
            // lane per staged point, looping over the queries: a step of it
            // costs as much as a step of the other loop, which takes two
            // staged points (16.8M halos, when taken: 1397 us, 1461 without the factor)
            const bool in = lane < n;
            const P rp = wm.soa.get(lane);
            const int ri = wm.idx[lane];
#pragma unroll 1
            while (am) {
                const int q = __ffs(am) - 1;
                am &= am - 1;
                const P pq = NB<D>::shfl(p, q);
                const unsigned h = __ballot_sync(FULL, in && dist2(pq, rp) <= e2);
                if (!h) continue;  // the common case in sparse regions: nothing to record
                if (list) {
                    // each hit point writes itself into q's list
                    const int at = __shfl_sync(FULL, nl, q) + __popc(h & ((1u << lane) - 1u));
                    if (((h >> lane) & 1u) && at < a.lcap) a.nlist[(int64_t)(qs + q) * a.lcap + at] = ri;
                }
                if (lane == q) {
                    cnt += __popc(h);
                    nl += __popc(h);
                    act = cnt < min_pts;
                }
            }
        } else {
            // lane per query, looping over the staged points two at a time
            // (packed; of an odd count the last distance is of a slot not in
            // use); a count that reaches minPts stops
            const typename NB<D>::PP pp = NB<D>::pack(p);
#pragma unroll 1
            for (int u = 0; u < n && act; u += 2) {
                float d0, d1;
                wm.soa.d2pair(pp, u, d0, d1);
                const bool h0 = d0 <= e2, h1 = d1 <= e2 && u + 1 < n;
                if (h0 || h1) {
                    if (list) {
                        int at = nl;
                        if (h0 && at < a.lcap) row[at] = wm.idx[u];
                        at += h0;
                        if (h1 && at < a.lcap) row[at] = wm.idx[u + 1];
                    }
                    cnt += h0 + h1;
                    nl += h0 + h1;
                    act = cnt < min_pts;
                }
            }
        }
        __syncwarp();
        // fewer queries, a smaller box
        am = __ballot_sync(FULL, act);
        if (am && am != am0) qbox = warp_box<D>(p, act);
    }

    // up to 32 candidate leaves, one per lane (U < 0: none); whether any
    // query still counts
    __device__ __forceinline__ bool batch(int U, int64_t m)
    {
        int us = 0, ue = 0;
        bool cand = false, whole = false;
        typename T::Box bx = qbox;
        if (U >= 0) {
            const int2 r = __ldg(&a.leafr[U]);
            us = r.x;
            ue = r.y & 0x7fffffff;
            bx = load_box<D>(a.leafbox, U);
            cand = NB<D>::bbox(qbox, bx) <= e2;
            whole = cand && ue - us >= min_pts && T::box_far2(qbox, bx) <= e2;
        }
        if (!__any_sync(FULL, cand)) return true;
        if (__any_sync(FULL, whole)) {
            // a leaf of at least minPts points lies within eps of all queries
            if (act) cnt = min_pts;
            act = false;
            return false;
        }
        // a dense cell larger than a tile: the queries that it lies within
        // eps of as a whole are done, and it is not streamed unless another
        // query is within eps of its box
        unsigned bm = __ballot_sync(FULL, cand && ue - us > TILE);
        if (bm) {
            const bool was = act;
#pragma unroll 1
            while (bm) {
                const int src = __ffs(bm) - 1;
                bm &= bm - 1;
                const typename T::Box big = load_box<D>(a.leafbox, __shfl_sync(FULL, U, src));
                const int size = __shfl_sync(FULL, ue - us, src);
                if (act && size >= min_pts && T::far_dist2(p, big) <= e2) {
                    cnt = min_pts;
                    act = false;
                }
                const bool near = __any_sync(FULL, act && NB<D>::pbox(p, big) <= e2);
                if (lane == src) cand = near;
            }
            if (!__any_sync(FULL, act)) return false;
            if (__any_sync(FULL, act != was)) qbox = warp_box<D>(p, act);
            if (!__any_sync(FULL, cand)) return true;  // no leaf is left to stream
        }
        // few queries: their box says little, so each of them is tested against
        // the lanes' leaves
        unsigned am = __ballot_sync(FULL, act);
        if (__popc(am) <= FEW_QUERIES) {
            bool near = false;
#pragma unroll 1
            while (am) {
                const P pq = NB<D>::shfl(p, __ffs(am) - 1);
                am &= am - 1;
                near = near || NB<D>::pbox(pq, bx) <= e2;
            }
            cand = cand && near;
            if (!__any_sync(FULL, cand)) return true;
        }
        GBD_COUNT(CNT_LEAF, cand);
        PointStream<D> ps(a.sp, wm.st, cand, us, ue, lane);
        int n = 0;
#pragma unroll 1
        for (;;) {
            const bool more = ps.next();
            const bool keep = more && ps.in && NB<D>::pbox(ps.p, qbox) <= e2;
            const unsigned km = __ballot_sync(FULL, keep);
            if (more ? n + __popc(km) > 32 : n > 0) {
                flush(n);
                if (!__any_sync(FULL, act)) return false;
                n = 0;
            }
            if (!more) return true;
            if (keep) {
                const int at = n + __popc(km & ((1u << lane) - 1u));
                wm.soa.put(at, ps.p);
                wm.idx[at] = ps.j;
            }
            n += __popc(km);
        }
    }

    __device__ __forceinline__ void walk(int L, int64_t m)
    {
        const int lc = a.lcount[L];
        int sp = 0, nc = 0, j0 = 0;
        int64_t steps = 0;
        if (lc < 0) sp = walk_roots<D>(a, L, (int)(m - 1), 0, wm.stack, lane);
#pragma unroll 1
        for (;;) {
            int U = -1;
            if (lc >= 0) {
                if (j0 >= lc) return;
                if (j0 + lane < lc) U = a.llist[(int64_t)L * LEAFCAP + j0 + lane];
                j0 += 32;
            } else {
                if (walk_next<D>(a, wm, sp, nc, steps, m, qbox, e2, 0, lane) == 0) return;
                U = walk_take<D>(wm, nc, lane);
                if (U == L) U = -1;
            }
            if (!batch(U, m)) return;
        }
    }
};

template <int D>
__global__ void __maxnreg__(traversal_regs<D>()) k_pre(const __grid_constant__ DevArgs<D> a)
{
    stage_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    WarpMem<D>* wm = reinterpret_cast<WarpMem<D>*>(smem) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int64_t m = a.ctrl[CTRL_M];
    for (;;) {
        const int L = next_leaf(&a.ctrl[CTRL_WORK_PRE]);
        if (L >= m) break;
        const int2 r = a.leafr[L];
        if (r.y < 0) continue;  // dense cell: all core already
        const TileParams tp = tile_params(a, L);
        // Algorithm 3: no preprocessing for minPts <= 2 (counts for several
        // minPts are always taken)
        if (tp.min_pts <= 2 && !a.ncount) continue;
        const int s = r.x, e = r.y, k = e - s;
        const int q = s + lane;
        // points of dense cells inside the tile are core already
        const bool counts = q < e && !a.core[q];
        if (!__any_sync(FULL, counts)) continue;
        PreWarp<D> w{a, *wm};
        w.lane = lane;
        w.e2 = tp.e2;
        w.min_pts = tp.min_pts;
        w.qs = s;
        w.p = a.sp[q < e ? q : s];
        // the tile's own points first: in dense regions most queries reach
        // minPts here and need no traversal at all (two points at a time)
        wm->soa.put(lane, w.p);
        __syncwarp();
        int cnt = 0;
        if (counts) {
            const typename NB<D>::PP pp = NB<D>::pack(w.p);
            int u = 0;
#pragma unroll 2
            for (; u + 1 < k && cnt < tp.min_pts; u += 2) {
                float d0, d1;
                wm->soa.d2pair(pp, u, d0, d1);
                cnt += (d0 <= tp.e2) + (d1 <= tp.e2);
            }
            if (u < k && cnt < tp.min_pts && wm->soa.d2(w.p, u) <= tp.e2) ++cnt;
        }
        __syncwarp();
        w.act = counts && cnt < tp.min_pts;
        w.cnt = cnt;
        w.nl = 0;
        const unsigned am = __ballot_sync(FULL, w.act);
        if (am) {
            // every point of the tile still counting: their box is the
            // leaf's own (exact min/max of the same points), no reduction
            w.qbox = am == tile_lanes(k) ? load_box<D>(a.leafbox, L) : warp_box<D>(w.p, w.act);
            w.walk(L, m);
        }
        if (counts) {
            const bool c = w.cnt >= tp.min_pts;
            a.core[q] = c ? 1 : 0;
            // lists: how many out-of-tile neighbours the list of a non-core
            // point holds; else whether another point is within eps (the
            // count includes q)
            a.nbr[q] = a.lcap > 0 ? (c ? 0 : (uint8_t)w.nl) : (w.cnt >= 2 ? 1 : 0);
            if (a.ncount) a.ncount[q] = w.cnt;
        }
    }
}

// A border claim from preprocessing's list (DBSCAN mode): a non-core point q
// holds all its neighbours outside its tile; it joins the cluster of the first
// core one (Algorithm 3's claim of a border point, Sec. 3.2, made here from the
// border's side). Neighbours inside the tile are k_intra's, afterwards.
__device__ __forceinline__ void list_claim(const int32_t* nlist, int lcap, const uint8_t* nbr,
                                           const uint8_t* core, int32_t* labels, int64_t q)
{
    const int k = nbr[q];
    const int32_t* row = nlist + q * lcap;
    for (int j = 0; j < k; ++j) {
        const int y = row[j];
        if (core[y]) {
            uf_claim(labels, (int)q, y);
            break;
        }
    }
}

// In small runs k_intra also makes the lists' claims and groups the leaves by
// kind, which saves two launches of 5 us each. From SPLIT_INTRA points on both
// are kernels of their own: a thread per point has more of the lists' scattered
// reads in flight, and k_intra's warps take their leaves one by one, far apart,
// instead of consecutive ones of alike cost. Whole runs in one and in three
// kernels, in us: blobs 354 and 367 (524,287), 663 and 708 (2.1M), 962 and 1084
// (4.2M); halos 870 and 887 (2.1M), 1435 and 1425 (4.2M), 1848 and 1818 (6M), 4335
// and 4266 (16.8M); roads 278 and 277 (524,287), 701 and 706 (2.1M), 1370 and
// 1380 (4.2M), 2625 and 2672 (8.4M): the line is where the halos turn.
constexpr int64_t SPLIT_INTRA = 1 << 22;
__global__ void k_list_claims(const int32_t* __restrict__ nlist, int lcap, const uint8_t* __restrict__ nbr,
                              const uint8_t* core, int32_t* labels, int64_t n)
{
    stage_begin(nlist, nbr, core);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        if (!core[q]) list_claim(nlist, lcap, nbr, core, labels, q);
}

// Each tile resolves its own pairs (q, q') with q' > q. Every lane builds the
// bit mask of the tile points within eps of its point; the components of the
// core points follow by growing each from its first point with one warp
// reduction per step; each core point then joins its component's first point
// globally (at most one union per point), and a non-core point with a core
// neighbour in the tile claims it. Finally the tile records whether it is
// solid: all points core and in one set. Dense cells larger than a tile are
// solid by construction.
constexpr int INTRA_THREADS = 256;

// a leaf's flag: no core point and none to claim (the main phase skips it),
// solid (all points core and in one set), or neither
constexpr uint8_t LEAF_IDLE = 0, LEAF_SOLID = 1, LEAF_MIXED = 2;

// Leaf L (nA staged points in soa, of which those in `am` are core; staged
// point j is point sA + j * step) united with the next leaf in sorted order
// where a pair of their points (up to 32 of a dense cell) is within eps. In
// dense regions nearly every leaf is adjacent to the next one, so the main
// phase starts from sets that span stretches of the curve and drops most of
// its candidate leaves by their sets.
template <int D>
__device__ __forceinline__ void link_next(const DevArgs<D>& a, const SoA<D>& soa, int64_t L, int64_t m,
                                          const TileParams& tp, int nA, unsigned am, int sA, int step, int lane)
{
    using P = typename Traits<D>::Point;
    if (L + 1 >= m || (a.linst && a.linst[L + 1] != a.linst[L])) return;
    const int2 r = a.leafr[L + 1];
    const int n = (r.y & 0x7fffffff) - r.x;
    const int idx = r.x + (n <= 32 ? min(lane, n - 1) : (int)((int64_t)n * lane / 32));
    const P p = a.sp[idx];
    const typename Traits<D>::Box box = load_box<D>(a.leafbox, L);
    const bool c = lane < n && (tp.min_pts <= 2 || r.y < 0 || a.core[idx]) && NB<D>::pbox(p, box) <= tp.e2;
    if (!__any_sync(FULL, c)) return;
    unsigned hit = 0;
    if (c) {
        const typename NB<D>::PP pp = NB<D>::pack(p);
        for (int j = 0; j < nA; j += 2) {  // (an odd count: the last distance is of a slot that `am` drops)
            float d0, d1;
            soa.d2pair(pp, j, d0, d1);
            hit |= (d0 <= tp.e2 ? 1u : 0u) << j;
            hit |= (d1 <= tp.e2 ? 2u : 0u) << j;
        }
        hit &= am;
    }
    const unsigned hm = __ballot_sync(FULL, hit != 0);
    if (!hm) return;
    const int q = hit ? sA + (__ffs(hit) - 1) * step : sA;
    if (hit && tp.min_pts == 2) {
        a.core[idx] = 1;
        a.core[q] = 1;
    }
    // one lane first: the others mostly find their pair united then
    const bool lead = lane == __ffs(hm) - 1;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        if (hit && lead == (h == 0) && __ldcg(a.labels + idx) != __ldcg(a.labels + q)) uf_union(a.labels, idx, q);
        __syncwarp();
    }
}

// The lanes' leaves go to the lists of their kinds (0 a tile that is not solid,
// 1 a solid tile, 2 a dense cell larger than a tile, -1 nothing to do), in lane
// order, with one atomic per kind.
__device__ __forceinline__ void append_kinds(uint32_t* ctrl, int32_t* klist, int64_t m_cap, int kind, int64_t L, int lane)
{
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const unsigned b = __ballot_sync(FULL, kind == t);
        if (!b) continue;
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&ctrl[CTRL_KIND_COUNT + t], (uint32_t)__popc(b));
        at = __shfl_sync(FULL, at, 0);
        if (kind == t) klist[t * m_cap + at + __popc(b & ((1u << lane) - 1u))] = (int32_t)L;
    }
}

template <int D>
__global__ void __launch_bounds__(INTRA_THREADS) k_intra(DevArgs<D> a)
{
    stage_begin();
    using P = typename Traits<D>::Point;
    __shared__ SoA<D> soa_s[INTRA_THREADS / 32];
    SoA<D>& soa = soa_s[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t m = a.ctrl[CTRL_M];
    const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // up to 16 consecutive leaves per warp and round: their kinds go to the
    // main phase's lists with one atomic per kind
    const int64_t per = a.whole_intra ? max((int64_t)1, min((int64_t)16, (m + nw - 1) / nw)) : 1;
    for (int64_t L0 = wid * per; L0 < m; L0 += nw * per) {
        int kinds = -1;  // lane j: the kind of leaf L0 + j
        for (int j = 0; j < per && L0 + j < m; ++j) {
            const int64_t L = L0 + j;
            const int2 r = a.leafr[L];
            if (r.y < 0) {
                if (lane == j) kinds = 2;
                if (lane == 0) a.lsolid[L] = LEAF_SOLID;
                const int n = (r.y & 0x7fffffff) - r.x;
                soa.put(lane, a.sp[r.x + (int)((int64_t)n * lane / 32)]);
                __syncwarp();
                link_next<D>(a, soa, L, m, tile_params(a, (int)L), 32, FULL, r.x, 0, lane);
                __syncwarp();
                continue;
            }
            const int s = r.x, k = r.y - r.x;
            const TileParams tp = tile_params(a, (int)L);
            const bool valid = lane < k;
            bool c = valid && a.core[s + lane];
            if (a.whole_intra && a.lcap > 0 && tp.min_pts > 2 && valid && !c)
                list_claim(a.nlist, a.lcap, a.nbr, a.core, a.labels, s + lane);
            if (tp.min_pts > 2 && !__any_sync(FULL, c)) {
                // core flags known and none in the tile: no pair inside it
                // unites or claims anything; the main phase needs the tile only
                // where it claims border points
                const bool idle = a.lcap > 0 || a.mode != DBSCAN_MODE_DBSCAN;
                if (lane == 0) a.lsolid[L] = idle ? LEAF_IDLE : LEAF_MIXED;
                if (lane == j) kinds = idle ? -1 : 0;
                continue;
            }
            const P p = a.sp[valid ? s + lane : s];
            // the tile's adjacency, two points at a time (packed)
            soa.put(lane, p);
            __syncwarp();
            unsigned adj = 0;
            if (valid) {
                const typename NB<D>::PP pp = NB<D>::pack(p);
                int j = 0;
                for (; j + 1 < k; j += 2) {
                    float d0, d1;
                    soa.d2pair(pp, j, d0, d1);
                    adj |= (d0 <= tp.e2 ? 1u : 0u) << j;
                    adj |= (d1 <= tp.e2 ? 2u : 0u) << j;
                }
                if (j < k && soa.d2(p, j) <= tp.e2) adj |= 1u << j;
                adj &= ~(1u << lane);
            }
            __syncwarp();
            if (tp.min_pts == 2) {
                // no preprocessing: a neighbour inside the tile makes a point core
                // (neighbours in other tiles are found by the main phase)
                c = valid && (c || adj != 0);
                if (c) a.core[s + lane] = 1;
            }
            const unsigned cm = __ballot_sync(FULL, c);
            if (tp.min_pts > 2 && a.mode == DBSCAN_MODE_DBSCAN && valid && !c && (adj & cm))
                uf_claim(a.labels, s + lane, s + __ffs(adj & cm) - 1);
            // the components, each grown from its first point by one reduction
            // over the lanes already in it per step
            const unsigned near = c ? adj & cm : 0u;
            unsigned reach = 1u << lane;
            unsigned left = __ballot_sync(FULL, near != 0);
            const bool pairs = left != 0;
            while (left) {
                unsigned grown = left & (0u - left), set;
                do {
                    set = grown;
                    grown |= __reduce_or_sync(FULL, ((set >> lane) & 1u) ? near : 0u);
                } while (grown != set);
                if ((set >> lane) & 1u) reach = set;
                left &= ~set;
            }
            if (c) {
                const int lr = __ffs(reach) - 1;
                if (lr != lane) uf_union(a.labels, s + lane, s + lr);
            }
            __syncwarp();
            const int root = c ? uf_find(a.labels, s + lane) : -1;
            const int root0 = __shfl_sync(FULL, root, 0);
            const bool solid = __all_sync(FULL, !valid || (c && root == root0));
            if (lane == 0) a.lsolid[L] = solid ? LEAF_SOLID : LEAF_MIXED;
            if (lane == j) kinds = solid ? 1 : 0;
            if (pairs) link_next<D>(a, soa, L, m, tp, k, tp.min_pts <= 2 ? tile_lanes(k) : cm, s, 1, lane);
            __syncwarp();
        }
        if (a.whole_intra) append_kinds(a.ctrl, a.klist, a.m_cap, kinds, L0 + lane, lane);
    }
}

__global__ void k_kinds(const int2* __restrict__ leafr, const uint8_t* __restrict__ lsolid, uint32_t* ctrl,
                        int32_t* __restrict__ klist, int64_t m_cap)
{
    stage_begin(leafr, lsolid);
    const int lane = threadIdx.x & 31;
    const int64_t m = ctrl[CTRL_M];
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; base < m;
         base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t L = base + lane;
        int kind = -1;
        if (L < m) {
            const uint8_t f = lsolid[L];
            kind = leafr[L].y < 0 ? 2 : (f == LEAF_IDLE ? -1 : (f == LEAF_SOLID ? 1 : 0));
        }
        append_kinds(ctrl, klist, m_cap, kind, L, lane);
    }
}

// ---------------------------------------------------------------------------
// The main phase.
//
// A warp takes one leaf L (a tile of up to 32 points, one per lane, or a
// dense cell larger than a tile) and unites it with the leaves after it (the
// pair mask of Sec. 4.1). What bounds it is the latency of dependent loads
// (leaf record, points, union-find chains), not arithmetic, so the candidate
// leaves are taken 32 at a time, one per lane: each lane loads its leaf's
// record, box and flag and follows the chain of its first point, and only
// the leaves that can still change something are visited one after another
// by the whole warp. Three things decide that nothing can change: the boxes
// are farther apart than eps; the leaf holds no core point (and no border
// point can be claimed); or it is solid and already in the set that all of
// L's points are in. A visited tile is cut to its points near L's box whose
// set differs from L's before any distance is taken: sets never split, so a
// pair that shared a root at any time needs no test. Testing the pairs first
// and looking at the sets of those within eps, one leaf after another, took
// 1241 us on 16.8M halos, 1524 us on 8M halos at minPts 2 and 1243 us on 400K
// 5D points; this takes 495, 939 and 480 us (kernel times).
// ---------------------------------------------------------------------------

// What a point can still do, by its code: the root of its set (core points;
// for minPts <= 2 all points), CODE_FREE for a non-core point that no core
// point has claimed, CODE_DONE for all others.
constexpr int CODE_FREE = -1, CODE_DONE = -2;

// can a pair within eps change something: a core point with a point of
// another set, or with an unclaimed non-core one
__device__ __forceinline__ bool pairable(int x, int y) { return x != y && min(x, y) >= CODE_FREE; }

// The union-find steps of the main phase are calls, not inlined: with its
// visitors and their union-find loops inlined at every use the kernel was
// 279 KB of code, and a fifth to a third of its warps' stalls were waits for
// instructions.
__device__ __noinline__ int uf_find_call(int* L, int x) { return uf_find(L, x); }

// unites the sets of x and y; returns the root of the union
__device__ __noinline__ int uf_join(int* L, int x, int y)
{
#pragma unroll 1
    for (;;) {
        uf_find2(L, x, y);
        if (x == y) return x;
        if (x > y) { const int t = x; x = y; y = t; }
        if (atomicCAS(L + y, y, x) == y) return x;
    }
}

template <int D>
struct MainWarp {
    using T = Traits<D>;
    using P = typename T::Point;
    using B = typename T::Box;
    const DevArgs<D>& a;
    WarpMem<D>& wm;
    int64_t m;
    int lane;
    float e2;
    int min_pts;
    bool claims;  // core-to-non-core claims: DBSCAN mode without preprocessing lists
    bool cell;    // a dense cell larger than a tile (else a tile)
    int L;
    int s, e;     // its points
    P p;          // tile: this lane's point and its code
    int rq;
    bool uni;     // all of L's points that take part are in set R
    int R;
    B qbox;       // box of the points that take part

    __device__ __forceinline__ int find(int x) const { return uf_find_call(a.labels, x); }
    // the set of x where L is in one set: a parent that is R settles it, so
    // that the many points of a large set do not all read its root's word
    __device__ __forceinline__ int find_near(int x) const
    {
        return uni && __ldcg(a.labels + x) == R ? R : find(x);
    }
    // the root of x, the same in all lanes (they decide together on it)
    __device__ __forceinline__ int warp_root(int x) const { return __shfl_sync(FULL, find(x), 0); }

    // the code of point i (core flag c)
    __device__ __forceinline__ int code_of(int i, bool c) const
    {
        if (min_pts <= 2 || c) return find_near(i);
        return claims && __ldcg(a.labels + i) == i ? CODE_FREE : CODE_DONE;
    }
    // are all points that take part in one set (tiles)
    __device__ __forceinline__ void uniform()
    {
        const unsigned part = __ballot_sync(FULL, rq >= CODE_FREE);
        R = part ? __shfl_sync(FULL, rq, __ffs(part) - 1) : CODE_DONE;
        uni = __all_sync(FULL, rq == CODE_DONE || rq == R) && R >= 0;
    }
    // codes after unions and claims
    __device__ __forceinline__ void refresh()
    {
        if (rq >= 0) rq = find(rq);
        else if (rq == CODE_FREE && __ldcg(a.labels + s + lane) != s + lane) rq = CODE_DONE;
        uniform();
    }
    // the sets x and y united (codes are mostly roots still: then one
    // compare-and-swap does it); returns a node of the union near its root
    __device__ __forceinline__ int join(int x, int y) const
    {
        const int hi = max(x, y), lo = min(x, y);
        return atomicCAS(a.labels + hi, hi, lo) == hi ? lo : uf_join(a.labels, hi, lo);
    }
    // the rule of Algorithm 3 for a pair (i, j) within eps with codes ci, cj
    // (pairable); the union's node, or INT_MAX after a claim
    __device__ __forceinline__ int act(int i, int ci, int j, int cj) const
    {
        if (min(ci, cj) >= 0) return join(ci, cj);
        // a non-core point joins the core point's set, unless another claimed it first
        const int y = ci >= 0 ? j : i;
        atomicCAS(a.labels + y, y, max(ci, cj));
        return INT_MAX;
    }

    // L's set (uni) united with the sets ru of the lanes with `on`: all of
    // them are hooked under the smallest root at once, so no lane waits for
    // another's union. R becomes the set's root.
    __device__ __forceinline__ void unite_lanes(bool on, int ru)
    {
        const int lo = min(R, __reduce_min_sync(FULL, on ? ru : R));
        int r = lo;
        const unsigned peers = __match_any_sync(FULL, on ? ru : -1);
        if (on && ru != lo && lane == __ffs(peers) - 1) r = join(ru, lo);
        if (lane == 0 && R != lo) r = min(r, join(R, lo));
        R = __reduce_min_sync(FULL, r);
        if (rq >= 0) {
            rq = R;
            // (several points in one set are core already, a tile's only point is by this pair)
            if (min_pts == 2) a.core[s + lane] = 1;
        }
    }

    // One round of a tile against n staged points (within eps of the query
    // box, allowed to take part): their sets, the pairs that can still change
    // something, their distances, the unions. The smaller side is looped over
    // (the pivot), the other sits in the lanes; after a union the codes on
    // both sides are brought up to date by value, without reading them again.
    __device__ __forceinline__ void flush(int n)
    {
        __syncwarp();
        // lane u: staged point u
        int cu = CODE_DONE, ui = 0;
        P up = p;
        if (lane < n) {
            const int enc = wm.idx[lane];
            ui = enc & 0x7fffffff;
            cu = code_of(ui, enc >= 0);
            up = wm.soa.get(lane);
        }
        __syncwarp();
        if (uni && cu == R) cu = CODE_DONE;
        const unsigned km = __ballot_sync(FULL, cu >= CODE_FREE);
        if (!km) return;
        const unsigned mq = __ballot_sync(FULL, rq >= CODE_FREE);
        const bool byq = __popc(mq) <= __popc(km);  // the queries are the pivots
        const P x = byq ? up : p, y = byq ? p : up;
        const int ix = byq ? ui : s + lane, iy = byq ? s + lane : ui;
        int cx = byq ? cu : rq, cy = byq ? rq : cu;
        unsigned mask = byq ? mq : km;
#pragma unroll 1
        while (mask) {
            const int v = __ffs(mask) - 1;
            mask &= mask - 1;
            const P py = NB<D>::shfl(y, v);
            const int pc = __shfl_sync(FULL, cy, v);
            const bool hit = pairable(pc, cx) && dist2(py, x) <= e2;
            if (!__any_sync(FULL, hit)) continue;
            const int pi = __shfl_sync(FULL, iy, v);
            // one union per set that was hit
            bool lead = hit && min(pc, cx) < 0;
            for (unsigned mm = __ballot_sync(FULL, hit && !lead); mm;) {
                const int src = __ffs(mm) - 1;
                lead = lead || lane == src;
                mm &= ~__ballot_sync(FULL, cx == __shfl_sync(FULL, cx, src));
            }
            if (hit && min_pts == 2) { a.core[pi] = 1; a.core[ix] = 1; }
            int r = INT_MAX;
            if (lead) r = act(pi, pc, ix, cx);
            __syncwarp();
            if (pc == CODE_FREE) {  // claimed
                if (lane == v) cy = CODE_DONE;
                continue;
            }
            r = __reduce_min_sync(FULL, r);
            const int old = cx;
            if (hit && cx == CODE_FREE) cx = CODE_DONE;
            unsigned mm = __ballot_sync(FULL, hit && old >= 0);
            if (!mm) continue;
            if (cy == pc) cy = r;
            while (mm) {
                const int c = __shfl_sync(FULL, old, __ffs(mm) - 1);
                if (cx == c) cx = r;
                mm &= ~__ballot_sync(FULL, old == c);
            }
            // all that is left in one set
            if (!__any_sync(FULL, (cx >= CODE_FREE && cx != r) || (((mask >> lane) & 1u) && cy != r))) break;
        }
        rq = byq ? cy : cx;
        uniform();
    }

    // A tile that is not in one set against a dense cell larger than a tile:
    // each query of another set looks for one adjacent point.
    __device__ __forceinline__ void tile_big(int us, int ue, const B& box)
    {
        const int ru = warp_root(us);
        if (rq >= 0 && rq != ru) rq = find(rq);
        const bool need = pairable(rq, ru) && NB<D>::pbox(p, box) <= e2;
        if (!__any_sync(FULL, need)) return;
        unsigned hm = __ballot_sync(FULL, need && T::far_dist2(p, box) <= e2);
        unsigned open = __ballot_sync(FULL, need) & ~hm;
#pragma unroll 1
        for (int c = us; c < ue && open; c += 32) {
            // the cell's points within eps of the queries' box (exact pruning)
            const P rp = a.sp[min(c + lane, ue - 1)];
            const bool keep = c + lane < ue && NB<D>::pbox(rp, qbox) <= e2;
            if (!__any_sync(FULL, keep)) continue;
            unsigned mm = open;
#pragma unroll 1
            while (mm) {
                const int qq = __ffs(mm) - 1;
                mm &= mm - 1;
                const P pq = NB<D>::shfl(p, qq);
                if (__any_sync(FULL, keep && dist2(pq, rp) <= e2)) hm |= 1u << qq;
            }
            open &= ~hm;
        }
        if (!hm) return;
        if ((hm >> lane) & 1u) {
            if (min_pts == 2) { a.core[s + lane] = 1; a.core[us] = 1; }
            act(s + lane, rq, us, ru);
        }
        __syncwarp();
        refresh();
    }

    // L in one set (a tile or a dense cell) against a solid leaf: is there an
    // adjacent pair? Of L only the points within eps of the leaf's box can
    // have a partner, of the leaf only those within eps of L's box (exact
    // pruning). Up to 32 of L's are staged at a time; the leaf's points pass
    // by them, one per lane, four loads in flight.
    // [ls, le): the part of L looked at.
    __device__ __forceinline__ bool adjacent(int ls, int le, int us, int ue, const B& box)
    {
        const unsigned lt = (1u << lane) - 1u;
        int cq = ls;
#pragma unroll 1
        while (cq < le) {
            int n = 0;
            if (cell) {
#pragma unroll 1
                for (; cq < le; cq += 32) {
                    const P pq = a.sp[min(cq + lane, le - 1)];
                    const bool near = cq + lane < le && NB<D>::pbox(pq, box) <= e2;
                    const unsigned nm = __ballot_sync(FULL, near);
                    if (n + __popc(nm) > 32) break;
                    if (near) wm.soa.put(n + __popc(nm & lt), pq);
                    n += __popc(nm);
                }
            } else {
                const bool near = rq >= 0 && NB<D>::pbox(p, box) <= e2;
                const unsigned nm = __ballot_sync(FULL, near);
                if (near) wm.soa.put(__popc(nm & lt), p);
                n = __popc(nm);
                cq = le;
            }
            if (!n) continue;
            __syncwarp();
            // (the next points are loaded while the current ones are tested)
            P r = a.sp[min(us + lane, ue - 1)];
#pragma unroll 1
            for (int c = us; c < ue; c += 32) {
                const P rn = a.sp[min(c + 32 + lane, ue - 1)];
                bool hit = false;
                if (NB<D>::pbox(r, qbox) <= e2) {
                    const typename NB<D>::PP pr = NB<D>::pack(r);
#pragma unroll 1
                    for (int u = 0; u < n && !hit; u += 2) {
                        float d0, d1;
                        wm.soa.d2pair(pr, u, d0, d1);
                        hit = d0 <= e2 || (d1 <= e2 && u + 1 < n);
                    }
                }
                if (__any_sync(FULL, hit)) return true;
                r = rn;
            }
            __syncwarp();
        }
        return false;
    }

    // ---- dense cell against a tile that is not solid: lane per tile point
    __device__ __forceinline__ void cell_mixed(int us, int ue, const B& box)
    {
        const int k = ue - us;
        const bool in = lane < k;
        const int ri = us + (in ? lane : 0);
        const P rp = a.sp[ri];
        const bool rc = a.core[ri];
        int cu = CODE_DONE;
        if (in && NB<D>::pbox(rp, qbox) <= e2) cu = code_of(ri, rc);
        bool need = pairable(R, cu);
        if (!__any_sync(FULL, need)) return;
        bool found = need && T::far_dist2(rp, qbox) <= e2;
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll 1
        for (int cq = s; cq < e; cq += 32) {
            if (!__any_sync(FULL, need && !found)) break;
            const P ap = a.sp[min(cq + lane, e - 1)];
            const bool keep = cq + lane < e && NB<D>::pbox(ap, box) <= e2;
            const unsigned km = __ballot_sync(FULL, keep);
            if (!km) continue;
            if (keep) wm.soa.put(__popc(km & lt), ap);
            __syncwarp();
            const int kk = __popc(km);
            if (need)
#pragma unroll 1
                for (int u = 0; u < kk && !found; ++u) found = wm.soa.d2(rp, u) <= e2;
            __syncwarp();
        }
        if (need && found) {
            if (min_pts == 2) a.core[ri] = 1;
            act(s, R, ri, cu);
        }
        __syncwarp();
        R = warp_root(R);
    }

    // what the head of a batch needs to know of a lane's candidate leaf
    struct Head {
        int U, us, ue, fl;  // leaf (-1: none), its points, its flag
        B box;
    };
    __device__ __forceinline__ Head head(int U) const
    {
        Head h;
        h.U = U;
        h.us = h.ue = 0;
        h.fl = LEAF_IDLE;
        h.box = qbox;
        if (U >= 0) {
            h.fl = *(volatile const uint8_t*)&a.lsolid[U];
            const int2 r = __ldg(&a.leafr[U]);
            h.box = load_box<D>(a.leafbox, U);
            h.us = r.x;
            h.ue = r.y & 0x7fffffff;
        }
        return h;
    }

    // up to 32 candidate leaves, one per lane
    __device__ __forceinline__ void batch(const Head& h)
    {
        const int us = h.us, ue = h.ue;
        const bool solid = h.fl == LEAF_SOLID;
        const float near = NB<D>::bbox(qbox, h.box);
        bool cand = h.U >= 0 && h.fl != LEAF_IDLE && near <= e2;
        int ru = 0;
        if (uni) {
            if (cand && solid) cand = (ru = find_near(us)) != R;
            bool far = false;
            if (__any_sync(FULL, cand && solid)) {
                R = warp_root(R);
                if (rq >= 0) rq = R;
                if (cand && solid) cand = ru != R;
                far = cand && solid && T::box_far2(qbox, h.box) <= e2;
            }
            if (__any_sync(FULL, far)) {
                // leaves that lie within eps of all of L
                unite_lanes(far, ru);
                if (cand && solid) cand = !far && (ru = find_near(ru)) != R;
            }
        }
        if (!cell) {
            // tiles: their points in one stream, in any order. Of several
            // solid ones the nearest goes first: the others are often in L's
            // set once it is
            const bool small = cand && ue - us <= 32;
            const unsigned sm = __ballot_sync(FULL, small && solid);
            bool first = small;
            if (uni && __popc(sm) > 2) {
                const unsigned d = small && solid ? __float_as_uint(near) : 0xffffffffu;
                const unsigned best = __ballot_sync(FULL, d == __reduce_min_sync(FULL, d));
                first = lane == __ffs(best) - 1;
            }
            bool todo = small;
#pragma unroll 1
            while (__any_sync(FULL, todo)) {
                const bool firsts = __any_sync(FULL, todo && first);
                const bool on = todo && (first || !firsts);
                PointStream<D> ps(a.sp, wm.st, on, us, ue, lane);
                int n = 0;
#pragma unroll 1
                for (;;) {
                    const bool more = ps.next();
                    bool keep = more && ps.in && NB<D>::pbox(ps.p, qbox) <= e2;
                    const bool c = min_pts > 2 && keep && a.core[ps.j];
                    keep = keep && (c || min_pts <= 2 || claims);
                    const unsigned km = __ballot_sync(FULL, keep);
                    if (more ? n + __popc(km) > 32 : n > 0) {
                        flush(n);
                        n = 0;
                    }
                    if (!more) break;
                    if (keep) {
                        const int at = n + __popc(km & ((1u << lane) - 1u));
                        wm.soa.put(at, ps.p);
                        wm.idx[at] = c || min_pts <= 2 ? ps.j : (int)(ps.j | 0x80000000u);
                    }
                    n += __popc(km);
                }
                todo = todo && !on;
                if (todo && solid && uni) todo = (ru = find_near(ru)) != R;
            }
            cand = cand && !small;
            if (uni && cand) cand = find_near(us) != R;
        }
        // one leaf at a time, the nearer ones first (they are likely adjacent,
        // and then often join L with the farther ones)
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            unsigned cm = __ballot_sync(FULL, cand && (near <= 0.25f * e2) == (pass == 0));
#pragma unroll 1
            while (cm) {
                const int src = __ffs(cm) - 1;
                cm &= cm - 1;
                const int Us = __shfl_sync(FULL, h.U, src);
                const int vs = __shfl_sync(FULL, us, src), ve = __shfl_sync(FULL, ue, src);
                const bool sol = __shfl_sync(FULL, (int)solid, src);
                const B box = load_box<D>(a.leafbox, Us);
                GBD_COUNT(CNT_LEAF, lane == 0);
                if (!sol) {
                    cell_mixed(vs, ve, box);
                } else if (!uni) {
                    tile_big(vs, ve, box);
                } else {
                    // (the points of a dense cell are in input order, so its
                    // first ones are a sample of it: they settle most pairs)
                    bool adj = false;
#pragma unroll 1
                    for (int part = 0; part < 2 && !adj; ++part) {
                        const int le = part ? e : min(s + 64, e), v1 = part ? ve : min(vs + 64, ve);
                        if (part && le == min(s + 64, e) && v1 == min(vs + 64, ve)) break;
                        adj = adjacent(s, le, vs, v1, box);
                    }
                    if (adj) {
                        const int rv = warp_root(vs);
                        unite_lanes(lane == src, rv);
                        // the others may be in L's set now
                        if (cand && solid) cand = find_near(us) != R;
                        cm &= __ballot_sync(FULL, cand);
                    }
                }
                __syncwarp();
            }
        }
    }

    // the leaves after L within eps of the query box, from L's list or by
    // walking the tree
    __device__ __forceinline__ void walk(int lc, const Head& h0)
    {
        int j0 = 0, sp = 0, nc = 0;
        int64_t steps = 0;
        Head h = h0;
        bool have = lc >= 0;  // the first batch of a list comes loaded
        if (lc < 0) sp = walk_roots<D>(a, L, (int)(m - 1), L + 1, wm.stack, lane);
#pragma unroll 1
        for (;;) {
            int U = -1;
            if (lc >= 0) {
                if (j0 >= lc) return;
                if (!have && j0 + lane < lc) U = a.llist[(int64_t)L * LEAFCAP + j0 + lane];
                j0 += 32;
            } else {
                if (walk_next<D>(a, wm, sp, nc, steps, m, qbox, e2, L + 1, lane) == 0) return;
                U = walk_take<D>(wm, nc, lane);
            }
            if (!have) h = head(U > L ? U : -1);
            have = false;
            if (__any_sync(FULL, h.U >= 0)) batch(h);
        }
    }
};

template <int D>
__global__ void __maxnreg__(main_regs<D>()) k_main(const __grid_constant__ DevArgs<D> a)
{
    stage_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    WarpMem<D>* wm = reinterpret_cast<WarpMem<D>*>(smem) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int64_t m = a.ctrl[CTRL_M];
    const int64_t c0 = a.ctrl[CTRL_KIND_COUNT], c1 = a.ctrl[CTRL_KIND_COUNT + 1], c2 = a.ctrl[CTRL_KIND_COUNT + 2];
    // One warp per leaf, also when there are more warps than leaves: warps
    // sharing a leaf contend for the same sets (with up to eight per leaf the
    // phase took 97 us on 16K dense points, with one 59). The dense cells
    // larger than a tile come first -- few, each much work.
    const int64_t total = c0 + c1 + c2;
    // The chain of dependent loads at the start of a leaf is what a warp
    // would wait for most: the next leaf's index is taken while the current
    // one is worked on, and the first batch's lists and leaves are loaded
    // together with the leaf's own points.
    int L;
    auto resolve = [&](int64_t idx) {
        // (a list per kind, taken as 2, 1, 0)
        if (idx >= total) L = -1;
        else if (idx < c2) L = a.klist[2 * a.m_cap + idx];
        else L = a.klist[idx < c2 + c1 ? a.m_cap + (idx - c2) : idx - c2 - c1];
    };
    int pend = 0;
    if (lane == 0) pend = (int)atomicAdd(&a.ctrl[CTRL_KIND_WORK], 1u);
    resolve(__shfl_sync(FULL, pend, 0));
    while (L >= 0) {
        if (lane == 0) pend = (int)atomicAdd(&a.ctrl[CTRL_KIND_WORK], 1u);
        const TileParams tp = tile_params(a, L);
        const bool listed = a.lcap > 0 && tp.min_pts > 2;
        const int2 r = a.leafr[L];
        const int lc = a.lcount[L];
        MainWarp<D> w{a, *wm};
        w.m = m;
        w.lane = lane;
        w.e2 = tp.e2;
        w.min_pts = tp.min_pts;
        w.claims = a.mode == DBSCAN_MODE_DBSCAN && !listed && tp.min_pts > 2;
        w.L = L;
        w.s = r.x;
        w.e = r.y & 0x7fffffff;
        w.cell = r.y < 0;
        int U = -1;
        if (lane < lc) U = a.llist[(int64_t)L * LEAFCAP + lane];
        if (U <= L) U = -1;
        // a tile's points that take part: after preprocessing a non-core
        // point with no other point within eps takes part in no pair, and in
        // DBSCAN* no non-core point does (with lists, non-core points took
        // their pairs with core points from their lists)
        const int q = w.s + lane;
        const bool in = !w.cell && q < w.e;
        const bool c = in && a.core[q];
        w.p = a.sp[in ? q : w.s];
        w.qbox = load_box<D>(a.leafbox, L);
        const typename MainWarp<D>::Head h = w.head(U);
        w.rq = CODE_DONE;
        w.uni = false;
        if (in && (tp.min_pts <= 2 || c || (w.claims && a.nbr[q]))) w.rq = w.code_of(q, c);
        bool work = true;
        if (w.cell) {
            w.uni = true;
            w.R = w.warp_root(w.s);
        } else {
            w.uniform();
            const unsigned vm = __ballot_sync(FULL, w.rq >= CODE_FREE);
            work = vm != 0;
            if (vm == tile_lanes(w.e - w.s)) {
                // every point core and in one set by now: solid from here on
                // (others may read the old flag, which only costs them tests)
                if (w.uni && w.e - w.s > 1 && lane == 0) *(volatile uint8_t*)&a.lsolid[L] = LEAF_SOLID;
            } else {
                w.qbox = warp_box<D>(w.p, w.rq >= CODE_FREE);
            }
        }
        resolve(__shfl_sync(FULL, pend, 0));
        if (work) w.walk(lc, h);
    }
}

// the work counters of the phases that follow
__device__ __forceinline__ void clear_work(uint32_t* ctrl)
{
    if (blockIdx.x == 0 && threadIdx.x < CTRL_WORK_END - CTRL_WORK_PRE) ctrl[CTRL_WORK_PRE + threadIdx.x] = 0u;
}
constexpr int32_t CANON_NONE = 0x7f7f7f7f;  // above every index

// k_init for one minPts of a multi-minPts run, with core flags from the
// neighbour counts (capped at the largest minPts, which decides every smaller
// one); points of dense cells are core for every minPts of the run.
__global__ void k_init_from_counts(const uint8_t* __restrict__ pdense, const int32_t* __restrict__ dstart,
                                   const int32_t* __restrict__ ncount, int64_t n, int min_pts,
                                   int32_t* __restrict__ labels, uint8_t* __restrict__ core,
                                   int32_t* __restrict__ canon, uint32_t* __restrict__ ctrl)
{
    stage_begin(pdense, dstart, ncount);
    clear_work(ctrl);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (pdense && pdense[i]) {
            labels[i] = dstart[i];
            core[i] = 1;
        } else {
            labels[i] = (int32_t)i;
            core[i] = (min_pts <= 1 || ncount[i] >= min_pts) ? 1 : 0;
        }
        canon[i] = CANON_NONE;
    }
}

// Core flags given by the caller in input order (core_in[perm[i]]), for
// clustering a part of a larger point set whose flags were decided with the
// rest of it; points of dense cells are core in any case (every one of them
// has at least minPts neighbours inside its cell).
__global__ void k_core_from_input(const uint32_t* __restrict__ perm, const uint8_t* __restrict__ core_in,
                                  const uint8_t* __restrict__ pdense, int64_t n, uint8_t* __restrict__ core,
                                  const uint32_t* __restrict__ ctrl)
{
    stage_begin(perm, core_in, pdense, ctrl);
    if (!stage_on(ctrl, -1)) return;  // aborted run: perm may hold stale words
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        core[i] = ((pdense && pdense[i]) || core_in[perm[i]]) ? 1 : 0;
}

// labels[i] = i, or the first point of its dense cell (pre-united, Sec. 4.2);
// core = 1 in dense cells (and everywhere when minPts == 1); no list entries,
// no smallest index, the phases' work counters at 0
__global__ void k_init(const uint8_t* __restrict__ pdense, const int32_t* __restrict__ dstart, int64_t n,
                       int min_pts, int32_t* __restrict__ labels, uint8_t* __restrict__ core,
                       uint8_t* __restrict__ nbr, int32_t* __restrict__ canon, uint32_t* __restrict__ ctrl)
{
    stage_begin(pdense, dstart);
    clear_work(ctrl);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (pdense && pdense[i]) {
            labels[i] = dstart[i];
            core[i] = 1;
        } else {
            labels[i] = (int32_t)i;
            core[i] = min_pts == 1 ? 1 : 0;
        }
        nbr[i] = 0;
        canon[i] = CANON_NONE;
    }
}

// full compression (Sec. 4.3) and the smallest input index per root
__global__ void k_finalize(int32_t* labels, const uint8_t* __restrict__ core, const uint32_t* __restrict__ perm,
                           int64_t n, int32_t* __restrict__ canon, const uint32_t* __restrict__ ctrl)
{
    stage_begin(core, perm, ctrl);
    if (!stage_on(ctrl, -1)) return;
    // warp-uniform trip count: warp_atomic_min needs all 32 lanes
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const int64_t i = base + (threadIdx.x & 31);
        const bool in = i < n;
        const int r = in ? uf_find(labels, (int)i) : 0;
        // (permutation and core flags are read once: evict-first)
        warp_atomic_min(canon, r, in ? (int32_t)__ldcs(perm + i) : 0, in && __ldcs(core + i));
    }
}

// output in input order: canonical label of the cluster, or -1
__global__ void k_relabel(const int32_t* labels, const uint8_t* __restrict__ core, const uint32_t* __restrict__ perm,
                          int64_t n, int mode, const int32_t* __restrict__ canon, int32_t* __restrict__ out,
                          uint8_t* __restrict__ core_out, const uint32_t* __restrict__ ctrl)
{
    stage_begin(labels, core, perm, canon, ctrl);
    // aborted run (non-finite input, a sort that gave up): perm may hold
    // stale words, so nothing is written; the error is reported at the next
    // host sync point
    if (!stage_on(ctrl, -1)) return;
    // the sequential reads (core flags, permutation, own label) stream
    // through L2 with evict-first priority, so that the lines of the
    // scattered output stay cached until they are complete
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool c = __ldcs(core + i) != 0;
        int r = (int)i;
        for (int p = __ldcs(labels + i); p != r; p = __ldcg(labels + r)) r = p;
        const bool member = c || (mode == DBSCAN_MODE_DBSCAN && r != (int)i);
        const uint32_t o = __ldcs(perm + i);
        out[o] = member ? canon[r] : -1;
        if (core_out) core_out[o] = c ? 1 : 0;
    }
}

#ifdef GBD_COUNTERS
__global__ void k_count_phase(int phase) { g_count_phase = phase; }
#endif

// the traversal counters' phase for the kernels that follow (counters build)
void count_phase(int phase, cudaStream_t s)
{
#ifdef GBD_COUNTERS
    k_count_phase<<<1, 1, 0, s>>>(phase);
#else
    (void)phase;
    (void)s;
#endif
}

// Blocks of a persistent launch (as many as fit on all SMs at once), kept per
// kernel, device and block size. Blocks from some 600 threads on take more
// shared memory than a launch gets by default; that limit belongs to the kernel
// on its device, so it is set once, to what the largest block takes: set to each
// size at its first use, a smaller block's would lower it under a larger one's.
cudaError_t persistent_blocks(const void* kernel, int block, size_t warp_smem, unsigned* out)
{
    static std::mutex mu;
    static std::map<std::tuple<const void*, int, int>, unsigned> known;
    int dev = 0, sms = 0, per = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    unsigned& g = known[std::make_tuple(kernel, dev, block)];
    if (!g) {
        if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(warp_smem * (MAX_BLOCK / 32)))) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, block, warp_smem * (block / 32))) !=
                cudaSuccess)
            return e;
        g = (unsigned)((per > 0 ? per : 1) * sms);
    }
    *out = g;
    return cudaSuccess;
}

template <int D>
DevArgs<D> dev_args(const ClusterArgs& a)
{
    DevArgs<D> d;
    d.sp = static_cast<const typename Traits<D>::Point*>(a.sp);
    d.nodes = static_cast<const typename Traits<D>::Node*>(a.nodes);
    d.leafbox = static_cast<const typename Traits<D>::Box*>(a.leafbox);
    d.leafr = a.leafr;
    d.lsolid = a.lsolid;
    d.klist = a.klist;
    d.m_cap = a.m_cap;
    d.nbr = a.nbr;
    d.nlist = a.nlist;
    d.lcap = a.lcap;
    d.whole_intra = a.n < SPLIT_INTRA;
    d.labels = a.labels;
    d.core = a.core;
    d.ctrl = a.ctrl;
    d.e2 = a.e2;
    d.min_pts = a.min_pts;
    d.mode = a.mode;
    d.linst = a.linst;
    d.e2s = a.e2s;
    d.mps = a.mps;
    d.iroot = a.iroot;
    d.tstart = a.tstart;
    d.tsib = a.tsib;
    d.tnsib = a.tnsib;
    d.llist = a.llist;
    d.lcount = a.lcount;
    d.ncount = a.ncount;
    return d;
}

// (launch errors: cudaGetLastError)
template <int D>
cudaError_t run_persistent(void (*kernel)(DevArgs<D>), const ClusterArgs& a, cudaStream_t s)
{
    unsigned g = 0;
    const cudaError_t e = persistent_blocks((const void*)kernel, a.block, sizeof(WarpMem<D>), &g);
    if (e != cudaSuccess) return e;
    launch(kernel, g, a.block, sizeof(WarpMem<D>) * (size_t)(a.block / 32), s, dev_args<D>(a));
    return cudaSuccess;
}

template <int D>
cudaError_t run_main(const ClusterArgs& a, cudaStream_t s)
{
    const bool split = a.n >= SPLIT_INTRA;
    if (split && a.lcap > 0) {
        launch(k_list_claims, 152 * 16, 256, 0, s, a.nlist, a.lcap, a.nbr, a.core, a.labels, a.n);
        note_launches(1);
    }
    int64_t gw = (a.m_cap * 32 + INTRA_THREADS - 1) / INTRA_THREADS;
    if (gw > 152 * 16) gw = 152 * 16;
    launch(k_intra<D>, (unsigned)gw, INTRA_THREADS, 0, s, dev_args<D>(a));
    if (split) {
        int64_t gk = (a.m_cap + 255) / 256;
        if (gk > 152 * 8) gk = 152 * 8;
        launch(k_kinds, (unsigned)gk, 256, 0, s, a.leafr, a.lsolid, a.ctrl, a.klist, a.m_cap);
        note_launches(1);
    }
    return run_persistent<D>(k_main<D>, a, s);
}

}  // namespace

cudaError_t launch_cluster_init(const ClusterArgs& a, cudaStream_t s)
{
    int64_t gn = (a.n + 255) / 256;
    if (gn > 152 * 16) gn = 152 * 16;
    launch(k_init, (unsigned)gn, 256, 0, s, a.pdense, a.dstart, a.n, a.min_pts, a.labels, a.core, a.nbr, a.canon, a.ctrl);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cluster_from_counts(const ClusterArgs& a, int min_pts, cudaStream_t s)
{
    int64_t gn = (a.n + 255) / 256;
    if (gn > 152 * 16) gn = 152 * 16;
    launch(k_init_from_counts, (unsigned)gn, 256, 0, s, a.pdense, a.dstart, a.ncount, a.n, min_pts, a.labels, a.core,
                                                    a.canon, a.ctrl);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cluster_starts(const ClusterArgs& a, cudaStream_t s)
{
    count_phase(0, s);
    // (a thread per leaf, or up to the resident blocks a warp)
    int64_t gm = std::max<int64_t>((a.m_cap + LL_THREADS - 1) / LL_THREADS,
                                   std::min<int64_t>((a.m_cap + LL_THREADS / 32 - 1) / (LL_THREADS / 32), 152 * 4));
    if (gm > 152 * 8) gm = 152 * 8;
#define LL_LAUNCH(D) launch(k_leaf_lists<D>, (unsigned)gm, LL_THREADS, 0, s, dev_args<D>(a))
    GBD_DIM_SWITCH(a.dim, LL_LAUNCH)
#undef LL_LAUNCH
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cluster_pre(const ClusterArgs& a, cudaStream_t s)
{
    // Algorithm 3: no preprocessing for minPts <= 2 (counts for several minPts
    // are always taken)
    if (a.min_pts <= 2 && !a.ncount) return cudaSuccess;
    count_phase(1, s);
    cudaError_t e = cudaSuccess;
#define PRE_RUN(D) e = run_persistent<D>(k_pre<D>, a, s)
    GBD_DIM_SWITCH(a.dim, PRE_RUN)
#undef PRE_RUN
    if (e != cudaSuccess) return e;
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cluster_main(const ClusterArgs& a, cudaStream_t s)
{
    count_phase(2, s);
    cudaError_t e = cudaSuccess;
#define MAIN_RUN(D) e = run_main<D>(a, s)
    GBD_DIM_SWITCH(a.dim, MAIN_RUN)
#undef MAIN_RUN
    if (e != cudaSuccess) return e;
    note_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_cluster_core_from_input(const ClusterArgs& a, const uint8_t* core_in, cudaStream_t s)
{
    int64_t gn = (a.n + 255) / 256;
    if (gn > 152 * 16) gn = 152 * 16;
    launch(k_core_from_input, (unsigned)gn, 256, 0, s, a.perm, core_in, a.pdense, a.n, a.core, a.ctrl);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_cluster_final(const ClusterArgs& a, int32_t* labels_out, uint8_t* core_out, cudaStream_t s)
{
    int64_t gn = (a.n + 255) / 256;
    if (gn > 152 * 16) gn = 152 * 16;
    launch(k_finalize, (unsigned)gn, 256, 0, s, a.labels, a.core, a.perm, a.n, a.canon, a.ctrl);
    launch(k_relabel, (unsigned)gn, 256, 0, s, a.labels, a.core, a.perm, a.n, a.mode, a.canon, labels_out, core_out,
                                           a.ctrl);
    note_launches(2);
    return cudaGetLastError();
}

bool counters_built()
{
#ifdef GBD_COUNTERS
    return true;
#else
    return false;
#endif
}

// the traversal counters since the last read ([phase][kind]), then zeroed
cudaError_t counters_take(uint64_t* out)
{
#ifdef GBD_COUNTERS
    unsigned long long h[CNT_PHASES * CNT_KINDS] = {};
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(h, g_counts, sizeof(h));
    for (int i = 0; i < CNT_PHASES * CNT_KINDS; ++i) out[i] = h[i];
    const unsigned long long z[CNT_PHASES * CNT_KINDS] = {};
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_counts, z, sizeof(z));
    return e;
#else
    for (int i = 0; i < CNT_PHASES * CNT_KINDS; ++i) out[i] = 0;
    return cudaErrorNotSupported;
#endif
}

}  // namespace gbd
