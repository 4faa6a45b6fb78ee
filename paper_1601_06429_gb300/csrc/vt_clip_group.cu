// vt_clip_group.cu -- the bulk clipping kernels of the FP32 filter: G = 4 or 8 lanes per cell, 8 or 4 cells per warp.
//
// The warp kernel (vt_clip_impl.cuh) gives a cell 32 lanes, of which a cut's 6-7 new vertices, a facet's fan or a
// node's few children keep a handful busy: it issues 31,000 warp instructions per cell.  Here the work of a cell is
// split over two kernels that alternate, one pair per radius pass, over chunks of cells:
//   k_group_search  a warp takes 32 consecutive cells (a tree bucket) and searches for those that want a pass, eight at
//                   a time with one walk of the tree: a leaf's points are loaded once for all of them.  It needs little
//                   shared memory and few registers, so 32 warps an SM hide the walk's dependent loads.  The candidates
//                   of a cell, in order of distance, go to a list in global memory.
//   k_group_clip    G lanes take a cell: side tests with one candidate plane per lane, new vertices and facet sums one
//                   per lane; the 32/G cells of a warp take these steps together, so an instruction serves 8 (or 4)
//                   cells.  A group whose cell is finished, or wants another pass (its state goes to global memory),
//                   takes the next one.
// Both are bound by instruction issue and by the latency of dependent instructions (FP32 and integer; DRAM idles).  Two
// kernels, each with half the code: fused in one they stalled on instruction fetch and ran ten warps an SM (70.9 ms at
// 1,048,576 clustered points where the pair takes 31).  Clipping at 2,097,152 points, warp kernel -> these: uniform
// 114.5 -> 40.2 ms, clustered 128 -> 61.4 ms (9,500 warp instructions a uniform cell instead of 31,000).
//
// The arithmetic is the warp kernel's: the same first radius and start box, candidates cut in the same order (by
// |d|^2), the same vertex formula, predicates and FP64 re-decisions, and new vertices take the same slots in the
// same order, so a facet's fan starts at the same vertex and every sum has the same terms in the same order.  A
// cell's result does not depend on the group size or on the other cells of its warp.  A cell these kernels cannot
// finish (capacity, an ill-conditioned vertex, a test undecided in FP64, a start wall left, a search wider than their
// passes, a duplicate) goes to a list that the warp kernel takes from the start.
#include <climits>
#include <cstddef>

#include "vt_clip_impl.cuh"
#include "vt_grid.cuh"
#include "vt_polytope.cuh"

namespace vt {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int GNT = GROUP_NT;  // vertex slots of a cell (two mask words)
constexpr int GNP = GROUP_NP;    // planes: the six start walls and the cuts (compacted when full)
constexpr int GNC = GROUP_CAND;  // candidates of one radius pass (byte indices)
constexpr int GBND = 48;   // boundary edges of a cut
constexpr int SCELLS = 8;  // cells searched for together
constexpr int SSTK = 96;   // inner nodes waiting in a search
constexpr int SLEAF = 64;  // leaves waiting in it (a pop adds up to 32)
constexpr int SWARPS = 4;  // warps per block of the search kernel
constexpr int GBINS = 64;  // radial bins of the candidate ordering (one byte counter each)
// from this radius pass on points too are tested against the vertices' balls (nodes from the second pass on): from the
// second pass on it costs more than the tests it saves (59 against 53 ms at 1,048,576 clustered points)
constexpr uint32_t SWIDE = 3;
constexpr int GLIST = 3;
constexpr uint32_t GM_INIT = 1u << 17;  // header: the cell starts (again) from its start box
constexpr int IDB5 = 6;    // bits of a plane id
constexpr uint32_t IDM5 = (1u << IDB5) - 1u;
constexpr uint32_t IDS = (1u << (3 * IDB5)) - 1u;

// a cell being clipped, in shared memory (2.4 KB: 11 warps of eight cells an SM).  64 vertices and 40 planes hold all but
// 0.03 % of clustered cells; 56 and 32 (13 warps) left 0.6 %, which took the warp kernel as long as all the others.
struct __align__(16) GCell {
    // vertex relative to the site; w holds the bound of its error, rounded up to 5 bits of mantissa, and in the low 18
    // bits its three plane ids (as a number w is at least the bound, and at most 7 % above it)
    float4 V[GNT];
    float4 Pl[GNP];      // plane n.y <= h; |n| is 1 for a start wall and sqrt(2 h) for a bisector
    uint32_t Ad[GNT];    // neighbour slot across edge k (a->b, b->c, c->a), one byte each
    uint32_t Ps[GNP];    // the plane's particle (sorted index)
    uint8_t Sq[GNP];     // the plane's number among the start walls and all cuts so far (its id before any compaction)
    union {
        struct {
            uint32_t bnd[GBND];              // boundary edges of a cut (x, y, kept slot, its edge, new slot)
            uint8_t lnk_s[GNP], lnk_e[GNP];  // new vertex whose boundary edge starts / ends at a plane
            uint8_t lnk_n[GNP];              // the plane at which the boundary edge that starts at a plane ends
        };
        uint32_t first[GNP];                 // emission: a plane's first slot
    };
    uint32_t pad[4];
};
static_assert(sizeof(GCell) % 32 == 16, "an odd number of 16-byte units: reads of one slot of every cell do not conflict");
static_assert(offsetof(GCell, bnd) <= GROUP_STATE && GROUP_STATE % 16 == 0, "the state kept between passes: V, Pl, Ad, Ps, Sq");

// one cell's search, and a warp's shared memory in the search kernel (6.8 KB: 32 warps an SM)
struct __align__(16) SCell {
    float4 q, a, b0, b1;      // position and squared reach; inner, support tolerance, range of |d|^2; box low and slack;
    uint32_t slo, shi, self;  // box high and key steps
    uint32_t vlo, vhi, wide;  // vertex slots (0: none yet); points tested against the vertices too
    const float4* V;          // its vertices
};
struct __align__(16) SWarp {
    SCell par[SCELLS];
    uint32_t cj[SCELLS][GNC];   // candidates
    uint16_t ck[SCELLS][GNC];   // their |d|^2 in 65536 steps over the pass's range
    uint32_t stack[SSTK], leaf[SLEAF];
    uint32_t lm[32];            // cells each leaf of a batch matters to
    uint16_t pair[32 * SCELLS]; // (leaf, cell) pairs of a batch
    uint32_t hist[GBINS / 4];   // ordering: counts, then starts of the bins (bytes)
    uint8_t tmp[GNC], plc[GNC]; // candidates by bin, and their places in the bins
};

// why a cell is handed over (n_tfail of the status words counts them)
constexpr int GF_CAP = 1, GF_ILL = 2, GF_UNDECIDED = 3, GF_DUP = 4, GF_WALL = 5, GF_RADIUS = 6, GF_STACK = 7;

template <int G> __device__ __forceinline__ float gmax(float v) {
#pragma unroll
    for (int o = G / 2; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}
template <int G> __device__ __forceinline__ float gmin(float v) {
#pragma unroll
    for (int o = G / 2; o; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}
template <int G> __device__ __forceinline__ unsigned gor(unsigned v) {
#pragma unroll
    for (int o = G / 2; o; o >>= 1) v |= __shfl_xor_sync(FULL, v, o);
    return v;
}
template <bool SETS>
__device__ __forceinline__ const Geometry& geo_of(const ClipArgs& A, uint32_t set) {
    if constexpr (SETS) return A.sgeo[set];
    else return A.geo;
}

// displacement of particle j from the site (minimum image in a periodic box); batched sets are never periodic
template <typename P, bool SETS>
__device__ __forceinline__ void gdisp(const P& pj, const P& pi, const Geometry& g, float& dx, float& dy, float& dz) {
    if constexpr (SETS) {
        DispPlain<P, float>::get(pj, pi, dx, dy, dz);
    } else {
        int code;
        DispF<P, float>::get(pj, pi, g, dx, dy, dz, code);
    }
}

__device__ __forceinline__ void ids_of(float w, uint32_t& a, uint32_t& b, uint32_t& c) {
    const uint32_t t = __float_as_uint(w);
    a = t & IDM5; b = (t >> IDB5) & IDM5; c = (t >> (2 * IDB5)) & IDM5;
}
__device__ __forceinline__ uint32_t pack_ids(uint32_t a, uint32_t b, uint32_t c) {
    return a | (b << IDB5) | (c << (2 * IDB5));
}
// error bound (finite) and plane ids as one word
__device__ __forceinline__ float pack_w(float ev, uint32_t ids) {
    return __uint_as_float(((__float_as_uint(ev) + IDS) & ~IDS) | ids);
}
__device__ __forceinline__ bool in_set(unsigned lo, unsigned hi, uint32_t n) {
    return (((n & 32u) ? hi : lo) >> (n & 31u)) & 1u;
}

// vertex of planes a, b, c: position, error bound in w, and rr >= its squared distance
__device__ __forceinline__ float4 vertex_at(const GCell& C, uint32_t a, uint32_t b, uint32_t c, float& rr) {
    const float4 A = C.Pl[a], B = C.Pl[b], D = C.Pl[c];
    const float an = a < 6 ? 1.f : sqrtf(2.f * A.w), bn = b < 6 ? 1.f : sqrtf(2.f * B.w), cn = c < 6 ? 1.f : sqrtf(2.f * D.w);
    float4 v;
    make_vertex<float>(A.x, A.y, A.z, A.w, an, B.x, B.y, B.z, B.w, bn, D.x, D.y, D.z, D.w, cn, v.x, v.y, v.z, v.w, rr);
    return v;
}

// plane p as a predicate source: a start wall (artificial or of the box), or a bisector with its image shift
template <typename P>
__device__ PRef plane_ref(const GCell& C, uint32_t p, unsigned art, uint32_t self, const P* spos, const Geometry& g) {
    PRef r;
    if (p < 6) {
        r.code = (int)(((art >> p) & 1u) ? CODE_ART + p : CODE_WALL + p);
        r.src = ((art >> p) & 1u) ? __float_as_uint(C.Pl[p].w) : self;
        return r;
    }
    r.src = C.Ps[p];
    float dx, dy, dz;
    DispF<P, float>::get(spos[r.src], spos[self], g, dx, dy, dz, r.code);
    return r;
}

// FP64 re-decision of vertex slot s against the bisector with particle j: +1, -1, or 0 (undecided)
template <typename P>
__device__ __noinline__ int resolve64(const GCell& C, int s, uint32_t j, unsigned art, uint32_t self, const P* spos,
                                      const Geometry& g) {
    uint32_t a, b, c;
    ids_of(C.V[s].w, a, b, c);
    PRef rj;
    rj.src = j;
    float dx, dy, dz;
    DispF<P, float>::get(spos[j], spos[self], g, dx, dy, dz, rj.code);
    return side64<P>(spos, g, self, plane_ref<P>(C, a, art, self, spos, g), plane_ref<P>(C, b, art, self, spos, g),
                     plane_ref<P>(C, c, art, self, spos, g), rj);
}

// Offsets of the six start walls (x upper, x lower, y ...) for artificial walls at B, and which are artificial (or a
// bisector with an own image) rather than a wall of a bounded box
template <typename P>
__device__ __forceinline__ unsigned start_box(const Geometry& g, bool periodic, const P& pi, float B, float* w) {
    const double lmin = fmin(g.L[0], fmin(g.L[1], g.L[2]));
    unsigned art = 0u;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        const int axis = k >> 1;
        const double xi = axis == 0 ? (double)pi.x : axis == 1 ? (double)pi.y : (double)pi.z;
        // periodic: half the box (an FP32 number: the box sides are)
        const double real = periodic ? 0.5 * g.L[axis] : (k & 1) == 0 ? g.hi[axis] - xi : xi - g.lo[axis];
        const bool inside = (double)B < (periodic ? 0.49 * lmin : real);
        w[k] = inside ? B : (float)real;
        if (periodic || inside) art |= 1u << k;
    }
    return art;
}

// the kk-th smallest |d|^2 from particle self to the other 31 of its bucket (the whole warp; INFINITY past the last)
template <typename P, bool SETS>
__device__ __noinline__ float bucket_kth(const P* spos, const ClipArgs& A, uint32_t self, uint32_t slo, uint32_t shi, uint32_t set,
                                         int kk) {
    const unsigned lane = lane_id();
    const Geometry& g = geo_of<SETS>(A, set);
    const uint32_t j = (self & ~31u) + lane;
    float d2f = INFINITY;
    if (j >= slo && j < shi && j != self) {
        float dx, dy, dz;
        gdisp<P, SETS>(spos[j], spos[self], g, dx, dy, dz);
        d2f = f_fma<float>(dz, dz, f_fma<float>(dy, dy, dx * dx));
    }
#pragma unroll 1
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll 1
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            const float o = __shfl_xor_sync(FULL, d2f, jj);
            const bool up = ((lane & k) == 0), lower = (lane & jj) == 0;
            const float mn = fminf(d2f, o), mx = fmaxf(d2f, o);
            d2f = (lower == up) ? mn : mx;
        }
    return __shfl_sync(FULL, d2f, kk);
}

// whether particle a comes before particle b for equal keys: nearer to the site; at the same distance in the order in
// which the warp kernel's search meets them (the higher bucket first, then the lower index)
template <typename P, bool SETS>
__device__ __noinline__ bool nearer(uint32_t a, uint32_t b, uint32_t self, const P* spos, const Geometry& g) {
    float dx, dy, dz, ex, ey, ez;
    const P pi = spos[self];
    gdisp<P, SETS>(spos[a], pi, g, dx, dy, dz);
    gdisp<P, SETS>(spos[b], pi, g, ex, ey, ez);
    const float d = f_fma<float>(dz, dz, f_fma<float>(dy, dy, dx * dx)), e = f_fma<float>(ez, ez, f_fma<float>(ey, ey, ex * ex));
    return d < e || (d == e && (a >> 5 != b >> 5 ? a >> 5 > b >> 5 : a < b));
}

// first |d|^2 where no bucket mate gives one: from the mean spacing of the set
__device__ __noinline__ float spacing2(const Geometry& g, uint32_t n) {
    const double sp = cbrt(g.L[0] * g.L[1] * g.L[2] / (double)n);
    return (float)(4.0 * sp * sp);
}

// A node (its box relative to the site) that may hold a point to cut with: within the squared reach, not within the ball
// already searched, and not outside the support of the cell's box.
__device__ __forceinline__ bool node_may_cut(float x0, float y0, float z0, float x1, float y1, float z1, float reach2,
                                             const float4& a, const float4& b0, const float4& b1) {
    const float dx = fmaxf(fmaxf(x0, -x1), 0.f), dy = fmaxf(fmaxf(y0, -y1), 0.f), dz = fmaxf(fmaxf(z0, -z1), 0.f);
    const float fx = fmaxf(-x0, x1), fy = fmaxf(-y0, y1), fz = fmaxf(-z0, z1);
    return dx * dx + dy * dy + dz * dz <= reach2 && fx * fx + fy * fy + fz * fz >= a.x &&
           supp_gmax(x0 - b0.w, x1 + b0.w, b0.x, b1.x) + supp_gmax(y0 - b0.w, y1 + b0.w, b0.y, b1.y) +
                   supp_gmax(z0 - b0.w, z1 + b0.w, b0.z, b1.z) >= -a.y;
}

// A bisector with p cuts a vertex v off when p lies in the ball around v through the site: whether a box (or a point)
// reaches into the ball of any vertex of the cell.  2 p.v - |p|^2 = |v|^2 - |p - v|^2 is at most tol where it does not.
__device__ __forceinline__ bool ball_hit(const SCell& K, float x0, float y0, float z0, float x1, float y1, float z1,
                                             float tol) {
    const unsigned vlo = K.vlo, vhi = K.vhi;
    const int hw = vhi ? 64 - __clz(vhi) : 32 - __clz(vlo);
    float best = -INFINITY;
#pragma unroll 2
    for (int s = 0; s < hw; s++) {
        const float4 v = K.V[s];
        const float dx = fmaxf(fmaxf(x0 - v.x, v.x - x1), 0.f), dy = fmaxf(fmaxf(y0 - v.y, v.y - y1), 0.f),
                    dz = fmaxf(fmaxf(z0 - v.z, v.z - z1), 0.f);
        // the exact vertex is within v.w: its ball is at most 2 v.w wider
        const float e = (v.x * v.x + v.y * v.y + v.z * v.z) - (dx * dx + dy * dy + dz * dz) +
                        4.f * v.w * (fabsf(v.x) + fabsf(v.y) + fabsf(v.z) + v.w);
        if (in_set(vlo, vhi, (uint32_t)s)) best = fmaxf(best, e);
    }
    return best >= -tol;
}

// Candidates rlo2 <= |d|^2 < rhi2 of the cells [c0, c0 + nc) that want a pass.  FIRST: the cells of this kernel's mode
// start: first radius, start box.
template <typename P, bool SETS, bool FIRST>
__global__ void __launch_bounds__(SWARPS * 32, 8) k_group_search(const __grid_constant__ ClipArgs A,
                                                                 const __grid_constant__ GroupBuf B, uint32_t c0, uint32_t nc,
                                                                 uint32_t* ctr, uint32_t unit, int mode,
                                                                 const uint32_t* act_list, const uint32_t* n_act) {
    __shared__ SWarp smem[SWARPS];
    SWarp& S = smem[threadIdx.x >> 5];
    const unsigned lane = lane_id(), lt = lanemask_lt();
    if (*((volatile unsigned*)&A.st->invalid_input)) return;
    const P* const spos = (const P*)A.spos;
    const bool periodic = SETS ? false : A.geo.periodic != 0;
    unsigned c_coll = 0, c_found = 0;
    const uint32_t count = act_list ? *n_act : nc;
    for (;;) {
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(ctr, unit);
        b = __shfl_sync(FULL, b, 0);
        if (b >= count) break;
        // the lanes hold the cells of a bucket and the warp searches for `unit` of them, or the next `unit` listed cells
        uint32_t i = (b & ~31u) + lane;
        bool in = i < nc, active = in && i >= b && i < b + unit;
        if (act_list) {
            in = active = lane < unit && b + lane < count;
            i = in ? act_list[b + lane] : 0u;
        }
        const uint32_t self = c0 + i;
        uint32_t set = 0, slo = 0, shi = (uint32_t)A.N;
        int k_target = A.k_target;
        const bool mine = active;
        if (!FIRST && mine) active = B.stat[i] != 0;
        if (FIRST && A.n_own < A.N && mine) active = A.perm[self] < A.n_own;  // buffer particles get no cell
        if (SETS && active) {
            set = A.sset[self];
            slo = (uint32_t)A.soff[set];
            shi = (uint32_t)A.soff[set + 1];
            int m = A.tpc_mode;
            if (A.set_cfg) {
                k_target = A.set_cfg[set] & 0xffff;
                m = (A.set_cfg[set] >> 16) & 3;
            }
            if (FIRST && m != mode) active = false;  // another kernel's cell
        }
        if (FIRST && mine) B.stat[i] = active ? 1 : 0;
        unsigned am = __ballot_sync(FULL, active);
        if (!am) continue;
        const Geometry& g = geo_of<SETS>(A, set);
        const P pi = spos[in ? self : c0];
        GHdr h = {};
        if (FIRST) {
            // first radius: 1.6 x the distance of the ~(k_target / 4)th nearest of the other 31 particles of the bucket
            const int kk = min(max(k_target / 4, 4), 30);
            float s[8], mx = 0.f;
#pragma unroll
            for (int q = 0; q < 8; q++) s[q] = INFINITY;
#pragma unroll 1
            for (int l = 0; l < 32; l++) {
                P pj;
                pj.x = __shfl_sync(FULL, pi.x, l); pj.y = __shfl_sync(FULL, pi.y, l); pj.z = __shfl_sync(FULL, pi.z, l);
                const uint32_t j = c0 + (b & ~31u) + (uint32_t)l;
                float v = INFINITY;
                if (j >= slo && j < shi && l != (int)lane) {
                    float dx, dy, dz;
                    gdisp<P, SETS>(pj, pi, g, dx, dy, dz);
                    v = f_fma<float>(dz, dz, f_fma<float>(dy, dy, dx * dx));
                    mx = fmaxf(mx, v);
                }
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const float lo = fminf(s[q], v);
                    v = fmaxf(s[q], v);
                    s[q] = lo;
                }
            }
            float dk = kk == 4 ? s[4] : kk == 5 ? s[5] : kk == 6 ? s[6] : s[7];
#pragma unroll 1
            for (unsigned todo = __ballot_sync(FULL, active && kk > 7); todo; todo &= todo - 1u) {
                const int l = __ffs(todo) - 1;  // more than the eight nearest: the bucket's distances sorted, one cell at a time
                const float d = bucket_kth<P, SETS>(spos, A, __shfl_sync(FULL, self, l), __shfl_sync(FULL, slo, l),
                                                    __shfl_sync(FULL, shi, l), __shfl_sync(FULL, set, l), __shfl_sync(FULL, kk, l));
                if ((int)lane == l) dk = d;
            }
            if (active && !(dk < INFINITY)) dk = mx > 0.f ? mx : spacing2(g, shi - slo);
            h.first2 = dk * 2.6f;
            // start box: artificial walls at 3 r, or where they are nearer the box walls (bounded sets) or the bisectors
            // with the site's own periodic images (a cell that keeps a facet on one is the warp kernel's to refuse)
            h.B = (float)(3.0 * sqrt((double)h.first2));
            const double lmin = fmin(g.L[0], fmin(g.L[1], g.L[2]));
            h.cap2 = periodic ? (float)(0.249 * lmin * lmin)
                              : (float)(4.0 * (g.L[0] * g.L[0] + g.L[1] * g.L[1] + g.L[2] * g.L[2]));
            h.meta = GM_INIT;
        } else if (active) {
            h = B.hdr[i];
        }
        if (active && (h.meta & GM_INIT)) {
            // a cell that starts (or starts again without artificial walls): its box is the start box
            float w[6];
            start_box<P>(g, periodic, pi, h.B, w);
            const float wd = 1.f + 4e-6f;  // the box holds the exact corners
            h.bx0 = -w[1] * wd; h.by0 = -w[3] * wd; h.bz0 = -w[5] * wd;
            h.bx1 = w[0] * wd; h.by1 = w[2] * wd; h.bz1 = w[4] * wd;
            h.vlo = h.vhi = 0u;
            h.rlo2 = 0.f;
            h.rhi2 = fminf(h.first2, h.cap2);
        }
        bool fail = false;
#pragma unroll 1
        while (am) {
            // up to eight of the cells: c-th of them is the c-th lowest bit of sub
            unsigned sub = am;
#pragma unroll 1
            for (int k = __popc(am); k > SCELLS; k--) sub &= ~(0x80000000u >> __clz(sub));
            am &= ~sub;
            const int ncell = __popc(sub);
            const bool act = (sub >> lane) & 1u;
            const int own = __popc(sub & lt);
            float ux0 = INFINITY, uy0 = INFINITY, uz0 = INFINITY, ux1 = -INFINITY, uy1 = -INFINITY, uz1 = -INFINITY;
            uint32_t ulo = 0u, uhi = (uint32_t)A.N;
            bool cross = false;
            __syncwarp();
            if (act) {
                const float qx = (float)pi.x, qy = (float)pi.y, qz = (float)pi.z;
                const float rad = sqrtf(h.rhi2) * 1.0001f + 1e-30f;
                const float bext = fmaxf(fmaxf(fmaxf(-h.bx0, h.bx1), fmaxf(-h.by0, h.by1)), fmaxf(-h.bz0, h.bz1));
                const float stol = 1e-5f * (4.f * bext * rad + rad * rad) + 1e-30f;  // rounding of the support test
                const float big = fmaxf(fmaxf(fmaxf(fabsf(g.hif[0]), fabsf(g.lof[0])), fmaxf(fabsf(g.hif[1]), fabsf(g.lof[1]))),
                                        fmaxf(fabsf(g.hif[2]), fabsf(g.lof[2])));
                const float slack = 8.0f * 1.2e-7f * big;  // rounding of a shifted coordinate and of a difference of two
                const float reach = rad + 2.f * slack;
                // squared distances in the node and point tests carry the slack; the hits are then tested exactly
                const float inner = sqrtf(h.rlo2) * 0.9999f - 2.f * slack;  // nodes within it hold only examined points
                ux0 = qx - reach; uy0 = qy - reach; uz0 = qz - reach;
                ux1 = qx + reach; uy1 = qy + reach; uz1 = qz + reach;
                cross = periodic && !(ux0 > g.lof[0] && ux1 < g.hif[0] && uy0 > g.lof[1] && uy1 < g.hif[1] &&
                                      uz0 > g.lof[2] && uz1 < g.hif[2]);
                SCell& K = S.par[own];
                K.q = make_float4(qx, qy, qz, reach * reach);
                K.a = make_float4(inner > 0.f ? inner * inner : 0.f, stol, h.rlo2, h.rhi2);
                K.b0 = make_float4(h.bx0, h.by0, h.bz0, slack);
                K.b1 = make_float4(h.bx1, h.by1, h.bz1, 65535.f / (h.rhi2 - h.rlo2));
                K.slo = slo; K.shi = shi; K.self = self;
                K.vlo = h.vlo; K.vhi = h.vhi;
                K.wide = (h.meta >> 24) >= SWIDE;
                K.V = reinterpret_cast<const float4*>(B.state + (size_t)i * GROUP_STATE);
                c_coll++;
            }
            // the box around the search balls
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                ux0 = fminf(ux0, __shfl_xor_sync(FULL, ux0, o)); ux1 = fmaxf(ux1, __shfl_xor_sync(FULL, ux1, o));
                uy0 = fminf(uy0, __shfl_xor_sync(FULL, uy0, o)); uy1 = fmaxf(uy1, __shfl_xor_sync(FULL, uy1, o));
                uz0 = fminf(uz0, __shfl_xor_sync(FULL, uz0, o)); uz1 = fmaxf(uz1, __shfl_xor_sync(FULL, uz1, o));
            }
            if (SETS) {
                ulo = __reduce_min_sync(FULL, act ? slo : 0xffffffffu);
                uhi = __reduce_max_sync(FULL, act ? shi : 0u);
            }
            // ... and the ball around them: half of the box's leaves lie in its corners
            const float ucx = 0.5f * (ux0 + ux1), ucy = 0.5f * (uy0 + uy1), ucz = 0.5f * (uz0 + uz1);
            float ur2 = 0.f;
            if (act) {
                const float4 q = S.par[own].q;
                const float ax = q.x - ucx, ay = q.y - ucy, az = q.z - ucz;
                ur2 = (sqrtf(ax * ax + ay * ay + az * az) + sqrtf(q.w)) * (1.f + 1e-5f) + 2.f * S.par[own].b0.w;
                ur2 *= ur2;
            }
            ur2 = warp_max<float>(ur2);
            cross = __any_sync(FULL, cross);
            unsigned lost = 0u;  // cells whose search failed
            int n = 0;           // lane c: candidates of cell c
            __syncwarp();
            // the images of the box the union reaches into (image 0: the box itself); a ball is narrower than the box
#pragma unroll 1
            for (int img = 0; img < (cross ? 27 : 1); img++) {
                const int ia = img % 3, ib = (img / 3) % 3, ic = img / 9;  // 0: none, 1: +L, 2: -L added to the points
                float hx = 0.f, hy = 0.f, hz = 0.f;
                if (img) {
                    hx = ia == 0 ? 0.f : ia == 1 ? A.geo.Lf[0] : -A.geo.Lf[0];
                    hy = ib == 0 ? 0.f : ib == 1 ? A.geo.Lf[1] : -A.geo.Lf[1];
                    hz = ic == 0 ? 0.f : ic == 1 ? A.geo.Lf[2] : -A.geo.Lf[2];
                    if (A.geo.lof[0] + hx > ux1 || A.geo.hif[0] + hx < ux0 || A.geo.lof[1] + hy > uy1 || A.geo.hif[1] + hy < uy0 ||
                        A.geo.lof[2] + hz > uz1 || A.geo.hif[2] + hz < uz0)
                        continue;
                }
                if (lane == 0) S.stack[0] = (uint32_t)(A.tree.levels + 1) << 28;  // the root: a node above the top level
                int sp = 1, nl = 0;
                __syncwarp();
#pragma unroll 1
                while (sp + nl > 0) {
                    if (sp > 0 && nl < 32) {
                        const uint32_t ent = S.stack[--sp];
                        const int cl = (int)(ent >> 28) - 1;
                        const uint32_t c = (ent & ((1u << 28) - 1u)) * 32u + lane;
                        bool hit = c < (uint32_t)A.tree.count[cl];
                        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
                        if (hit) {
                            const int64_t o = A.tree.off[cl] + c;
                            lo = A.tree.lo[o]; hi = A.tree.hi[o];
                            hit = lo.x + hx <= ux1 && hi.x + hx >= ux0 && lo.y + hy <= uy1 && hi.y + hy >= uy0 &&
                                  lo.z + hz <= uz1 && hi.z + hz >= uz0;
                            const float ax = fmaxf(fmaxf(lo.x + hx - ucx, ucx - hi.x - hx), 0.f),
                                        ay = fmaxf(fmaxf(lo.y + hy - ucy, ucy - hi.y - hy), 0.f),
                                        az = fmaxf(fmaxf(lo.z + hz - ucz, ucz - hi.z - hz), 0.f);
                            hit = hit && ax * ax + ay * ay + az * az <= ur2;
                            if (SETS) {
                                const uint64_t f = (uint64_t)c << (5 * cl);
                                hit = hit && f < uhi && f + (1ull << (5 * cl)) > ulo;
                            }
                        }
                        if (!FIRST && cl > 1 && __any_sync(FULL, hit)) {
                            // an inner node of a later pass: some cell's annulus, support and vertices' balls must reach it
                            bool any = false;
#pragma unroll 1
                            for (int c2 = 0; c2 < ncell; c2++) {
                                const SCell& K = S.par[c2];
                                const float4 q = K.q, a = K.a, b0 = K.b0, b1 = K.b1;
                                const float x0 = lo.x + hx - q.x, y0 = lo.y + hy - q.y, z0 = lo.z + hz - q.z, x1 = hi.x + hx - q.x,
                                            y1 = hi.y + hy - q.y, z1 = hi.z + hz - q.z;
                                bool may = hit && !any && node_may_cut(x0, y0, z0, x1, y1, z1, q.w, a, b0, b1);
                                if (may && K.wide && (K.vlo | K.vhi))
                                    may = ball_hit(K, x0 - b0.w, y0 - b0.w, z0 - b0.w, x1 + b0.w, y1 + b0.w, z1 + b0.w, a.y);
                                any = any || may;
                            }
                            hit = hit && any;
                        }
                        const unsigned hm = __ballot_sync(FULL, hit);
                        const int nh = __popc(hm);
                        if (cl > 1 && sp + nh > SSTK) {
                            lost = (1u << ncell) - 1u;
                            break;
                        }
                        uint32_t* const to = cl == 1 ? &S.leaf[nl] : &S.stack[sp];
                        if (hit) to[__popc(hm & lt)] = ((uint32_t)cl << 28) | c;
                        if (cl == 1) nl += nh; else sp += nh;
                        __syncwarp();
                        continue;
                    }
                    // up to 32 leaves, one per lane: the cells each may matter to (its box within the cell's ball, not
                    // within the ball already searched, and not outside the support of the cell's box)
                    const int nb = min(nl, 32);
                    nl -= nb;
                    uint32_t lf = 0u;
                    float x0 = INFINITY, y0 = 0.f, z0 = 0.f, x1 = INFINITY, y1 = 0.f, z1 = 0.f;
                    if ((int)lane < nb) {
                        lf = S.leaf[nl + lane] & ((1u << 28) - 1u);
                        const int64_t o = A.tree.off[1] + lf;
                        const float4 lo = A.tree.lo[o], hi = A.tree.hi[o];
                        x0 = lo.x + hx; y0 = lo.y + hy; z0 = lo.z + hz;
                        x1 = hi.x + hx; y1 = hi.y + hy; z1 = hi.z + hz;
                    }
                    S.lm[lane] = 0u;
                    int npair = 0;
#pragma unroll 1
                    for (int c = 0; c < ncell; c++) {
                        const SCell& K = S.par[c];
                        const float4 q = K.q;
                        const float dx = fmaxf(fmaxf(x0 - q.x, q.x - x1), 0.f), dy = fmaxf(fmaxf(y0 - q.y, q.y - y1), 0.f),
                                    dz = fmaxf(fmaxf(z0 - q.z, q.z - z1), 0.f);
                        bool hit = dx * dx + dy * dy + dz * dz <= q.w;
                        if (SETS) hit = hit && lf * 32u < K.shi && lf * 32u + 32u > K.slo;
                        const unsigned hm = __ballot_sync(FULL, hit);
                        if (hit) S.pair[npair + __popc(hm & lt)] = (uint16_t)(lane | (c << 5));
                        npair += __popc(hm);
                    }
                    __syncwarp();
#pragma unroll 1
                    for (int k0 = 0; k0 < npair; k0 += 32) {
                        const int k = k0 + (int)lane;
                        const unsigned code = k < npair ? S.pair[k] : 0u;
                        const int l = (int)(code & 31u);
                        const SCell& K = S.par[code >> 5];
                        const float4 q = K.q, a = K.a, b0 = K.b0, b1 = K.b1;
                        const float ax = __shfl_sync(FULL, x0, l) - q.x, ay = __shfl_sync(FULL, y0, l) - q.y,
                                    az = __shfl_sync(FULL, z0, l) - q.z, ex = __shfl_sync(FULL, x1, l) - q.x,
                                    ey = __shfl_sync(FULL, y1, l) - q.y, ez = __shfl_sync(FULL, z1, l) - q.z;
                        bool hit = k < npair && node_may_cut(ax, ay, az, ex, ey, ez, q.w, a, b0, b1);
                        if (!FIRST && hit && (K.vlo | K.vhi))
                            hit = ball_hit(K, ax - b0.w, ay - b0.w, az - b0.w, ex + b0.w, ey + b0.w, ez + b0.w, a.y);
                        if (hit) atomicOr(&S.lm[l], 1u << (code >> 5));
                    }
                    __syncwarp();
                    const unsigned need = S.lm[lane] & ~lost;
#pragma unroll 1
                    for (unsigned lm = __ballot_sync(FULL, need != 0u); lm; lm &= lm - 1u) {
                        const int l = __ffs(lm) - 1;
                        const uint32_t j = __shfl_sync(FULL, lf, l) * 32u + lane;
                        unsigned todo = __shfl_sync(FULL, need, l) & ~lost;
                        const bool in = j < uhi;
                        const float4 pj = A.spos4[in ? j : 0u];
                        const float px = pj.x + hx, py = pj.y + hy, pz = pj.z + hz;
#pragma unroll 1
                        for (; todo; todo &= todo - 1u) {
                            const int c = __ffs(todo) - 1;
                            SCell& K = S.par[c];
                            const float4 q = K.q, a = K.a;
                            const float tx = px - q.x, ty = py - q.y, tz = pz - q.z;
                            const float t2 = tx * tx + ty * ty + tz * tz;
                            bool hit = in && t2 >= a.x && t2 <= q.w;
                            if (!__any_sync(FULL, hit)) continue;
                            float d2 = 0.f;
                            if (hit) {
                                const float4 b0 = K.b0, b1 = K.b1;
                                const uint32_t ks = K.self;
                                P pc;
                                if constexpr (sizeof(P) == 16) { pc.x = q.x; pc.y = q.y; pc.z = q.z; }
                                else pc = spos[ks];
                                float dx, dy, dz;
                                gdisp<P, SETS>(spos[j], pc, g, dx, dy, dz);
                                d2 = f_fma<float>(dz, dz, f_fma<float>(dy, dy, dx * dx));
                                hit = d2 >= a.z && d2 < a.w && j != ks &&
                                      supp_g(dx, b0.x, b1.x) + supp_g(dy, b0.y, b1.y) + supp_g(dz, b0.z, b1.z) >= -a.y;
                                if (SETS) hit = hit && j >= K.slo && j < K.shi;
                                if (!FIRST && hit && K.wide && (K.vlo | K.vhi)) hit = ball_hit(K, dx, dy, dz, dx, dy, dz, a.y);
                            }
                            unsigned hm = __ballot_sync(FULL, hit);
                            if (!hm) continue;
                            int nc = __shfl_sync(FULL, n, c);
#pragma unroll 1
                            for (int tries = 0; nc + __popc(hm) > GNC; tries++) {
                                // other lanes' entries of the leaves since the last barrier (a vote does not order them)
                                __syncwarp();
                                // a full list: the part nearer than the mean of it stays, and the pass ends there
                                int sum = 0;
                                for (int i = (int)lane; i < nc; i += 32) sum += S.ck[c][i];
                                sum = __reduce_add_sync(FULL, sum);
                                const float lo2 = K.a.z, hi2 = K.a.w;
                                const float rn = lo2 + (float)sum / (K.b1.w * (float)max(nc, 1));
                                if (!(rn > lo2) || !(rn < hi2) || tries == 24) {
                                    lost |= 1u << c;
                                    hm = 0u;
                                    nc = 0;
                                    hit = false;
                                    break;
                                }
                                const float nks = 65535.f / (rn - lo2);
                                int kept = 0;
                                for (int i0 = 0; i0 < nc; i0 += 32) {
                                    const int i = i0 + (int)lane;
                                    uint32_t jj = 0;
                                    float e2 = INFINITY;
                                    if (i < nc) {
                                        jj = S.cj[c][i];
                                        float dx, dy, dz;
                                        gdisp<P, SETS>(spos[jj], spos[K.self], g, dx, dy, dz);
                                        e2 = f_fma<float>(dz, dz, f_fma<float>(dy, dy, dx * dx));
                                    }
                                    const unsigned km = __ballot_sync(FULL, e2 < rn);
                                    if (e2 < rn) {
                                        const int o = kept + __popc(km & lt);
                                        S.ck[c][o] = (uint16_t)min(65535, max(0, (int)((e2 - lo2) * nks)));
                                        S.cj[c][o] = jj;
                                    }
                                    kept += __popc(km);
                                    __syncwarp();
                                }
                                nc = kept;
                                if (lane == 0) {
                                    const float re = sqrtf(rn) * 1.0001f + 1e-30f + 2.f * K.b0.w;
                                    K.q.w = re * re;
                                    K.a.w = rn;
                                    K.b1.w = nks;
                                }
                                __syncwarp();
                                hit = hit && d2 < rn;
                                hm = __ballot_sync(FULL, hit);
                            }
                            if (hit) {
                                const int o = nc + __popc(hm & lt);
                                S.ck[c][o] = (uint16_t)min(65535, max(0, (int)((d2 - K.a.z) * K.b1.w)));
                                S.cj[c][o] = j;
                            }
                            if ((int)lane == c) n = nc + __popc(hm);
                        }
                    }
                    __syncwarp();
                }
                __syncwarp();
            }
            if ((int)lane < ncell) c_found += n;
            __syncwarp();

            // ------------------------------------------------------------ order the candidates by |d|^2
            // cell by cell: radial bins (byte counters), candidates gathered by bin, then ranked within their bin (equal
            // keys by the distances themselves)
#pragma unroll 1
            for (int c = 0; c < ncell; c++) {
                const int m = __shfl_sync(FULL, n, c);
                const uint32_t ks = S.par[c].self;
                uint32_t* const out = B.list + (size_t)(ks - c0) * GNC;
                if (m == 0) continue;
                if (lane < GBINS / 4) S.hist[lane] = 0u;
                __syncwarp();
#pragma unroll 1
                for (int i = (int)lane; i < m; i += 32) {
                    const int b = S.ck[c][i] >> 10;
                    const unsigned old = atomicAdd(&S.hist[b >> 2], 1u << (8 * (b & 3)));
                    S.plc[i] = (uint8_t)(old >> (8 * (b & 3)));  // place within the bin
                }
                __syncwarp();
                {
                    const unsigned p = (lane < GBINS / 4 ? S.hist[lane] : 0u) * 0x01010101u;  // inclusive sums of the bytes
                    unsigned x = p >> 24;
#pragma unroll
                    for (int o = 1; o < GBINS / 4; o <<= 1) {
                        const unsigned y = __shfl_up_sync(FULL, x, o);
                        if ((int)lane >= o) x += y;
                    }
                    if (lane < GBINS / 4) S.hist[lane] = (p << 8) + (x - (p >> 24)) * 0x01010101u;
                }
                __syncwarp();
                const uint8_t* const start = reinterpret_cast<const uint8_t*>(S.hist);
#pragma unroll 1
                for (int i = (int)lane; i < m; i += 32) S.tmp[start[S.ck[c][i] >> 10] + S.plc[i]] = (uint8_t)i;
                __syncwarp();
#pragma unroll 1
                for (int q = (int)lane; q < m; q += 32) {
                    const int i = S.tmp[q];
                    const int key = S.ck[c][i], b = key >> 10;
                    const int b0 = start[b], b1 = b + 1 < GBINS ? (int)start[b + 1] : m;
                    int rank = b0;
#pragma unroll 1
                    for (int t = b0; t < b1; t++) {
                        const int k = S.tmp[t], kk = S.ck[c][k];
                        if (kk < key || (kk == key && k != i && nearer<P, SETS>(S.cj[c][k], S.cj[c][i], ks, spos, g))) rank++;
                    }
                    out[rank] = S.cj[c][i];
                }
                __syncwarp();
            }
            const int no = __shfl_sync(FULL, n, own & 31);
            if (act) {
                h.n = (h.n & 0xffff0000u) | (uint32_t)no;
                h.rhi2 = S.par[own].a.w;
                fail = (lost >> own) & 1u;
            }
            __syncwarp();
        }
        const bool was = active && !fail;
        if (was) {
            if (h.meta & GM_INIT) B.hdr[i] = h;
            else {
                B.hdr[i].rhi2 = h.rhi2;
                B.hdr[i].n = h.n;
            }
        }
        const unsigned fm = __ballot_sync(FULL, fail);
        if (fm) {
            unsigned slot = 0;
            if (lane == 0) {
                slot = atomicAdd(&A.st->n_warp_cells, (unsigned)__popc(fm));
                atomicAdd(&A.st->n_tfail[GF_STACK], (unsigned long long)__popc(fm));
            }
            slot = __shfl_sync(FULL, slot, 0);
            if (fail) {
                A.warp_list[slot + __popc(fm & lt)] = self;
                B.stat[i] = 0;
            }
        }
    }
    c_coll = __reduce_add_sync(FULL, c_coll);
    c_found = __reduce_add_sync(FULL, c_found);
    if (lane == 0) {
        atomicAdd(&A.st->n_collect, (unsigned long long)c_coll);
        atomicAdd(&A.st->n_collected, (unsigned long long)c_found);
    }
}

// The vertices of `in` reached from `seed` over edges within it, and the removed side of a cut by pl made whole, with the
// kept side (vt_polytope.cuh): what is apart from the vertex farthest out is kept, what is then apart from the vertex farthest in
// is removed.  One lane's work, for the few cuts whose signs contradict each other.
__device__ unsigned long long reach_of_slots(const GCell& C, int seed, unsigned long long in) {
    unsigned long long got = 1ull << seed, front = got;
    while (front) {
        unsigned long long to = 0ull;
        for (; front; front &= front - 1ull) {
            const uint32_t ad = C.Ad[__ffsll((long long)front) - 1];
            to |= (1ull << (ad & 63u)) | (1ull << ((ad >> 8) & 63u)) | (1ull << ((ad >> 16) & 63u));
        }
        front = to & in & ~got;
        got |= front;
    }
    return got;
}
__device__ __noinline__ unsigned long long whole_sides(const GCell& C, float4 pl, unsigned long long all, unsigned long long rem) {
    float so = -INFINITY, si = INFINITY;
    int far_out = 0, far_in = 0;
    for (unsigned long long m = all; m; m &= m - 1ull) {
        const int s = __ffsll((long long)m) - 1;
        const float4 v = C.V[s];
        const float d = beyond(pl, v.x, v.y, v.z);
        if ((rem >> s) & 1ull) {
            if (d > so) { so = d; far_out = s; }
        } else if (d < si) {
            si = d;
            far_in = s;
        }
    }
    rem = reach_of_slots(C, far_out, rem);
    return all & ~reach_of_slots(C, far_in, all & ~rem);
}

// Cut the cells of the groups with `cut` set by the plane that lane `src` of the group holds (pl, from its lane's particle
// `from`), which removes exactly the vertex slots rem: the plane gets an id, every edge between a removed and a kept vertex
// becomes a new vertex (w: the new slots).  fail is set where the cell outgrows its capacity or a vertex is
// ill-conditioned.  SIGNS: rem comes from plain signs, which may contradict each other; where the boundary is not one loop
// that meets a plane once, both sides are made whole first and rem returns what was removed; and new vertices are taken on
// their edges.  The whole warp calls.
constexpr int EARLY = 3;  // new vertices a lane holds before it writes them (SIGNS)
__device__ __forceinline__ float4 on_edge(const GCell& C, float4 pl, uint32_t p, uint32_t rec) {
    const float4 a = C.V[rec >> 26], b = C.V[(rec >> 12) & 63u];
    const float e = edge_part(beyond(pl, a.x, a.y, a.z), beyond(pl, b.x, b.y, b.z));
    return make_float4(fmaf(e, b.x - a.x, a.x), fmaf(e, b.y - a.y, a.y), fmaf(e, b.z - a.z, a.z),
                       pack_w(0.f, pack_ids(rec & 63u, (rec >> 6) & 63u, p)));
}
template <int G, bool SIGNS>
__device__ __forceinline__ void group_cut(GCell& C, bool& cut, int src, unsigned& rem0, unsigned& rem1, float4 pl, uint32_t from,
                                          unsigned& vlo, unsigned& vhi, int& np, int& nseq, int& fail, unsigned& w0,
                                          unsigned& w1) {
    const unsigned lane = lane_id();
    const int r = (int)(lane & (G - 1)), gsh = (int)(lane & ~(unsigned)(G - 1));
    if (__any_sync(FULL, cut && np == GNP)) {
        // planes no vertex uses any more are dropped (the start walls keep their ids, the others their order)
        const bool cp = cut && np == GNP;
        unsigned use0 = 0u, use1 = 0u;
#pragma unroll 1
        for (int s = r; s < GNT; s += G)
            if (cp && in_set(vlo, vhi, (uint32_t)s)) {
                uint32_t a, b, c;
                ids_of(C.V[s].w, a, b, c);
                const unsigned long long mk = (1ull << a) | (1ull << b) | (1ull << c);
                use0 |= (unsigned)mk; use1 |= (unsigned)(mk >> 32);
            }
        const unsigned long long use = ((unsigned long long)gor<G>(use1) << 32) | gor<G>(use0) | 0x3full;
#pragma unroll 1
        for (int p = r; p < GNP; p += G) {
            const bool mv = cp && ((use >> p) & 1ull);
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            uint32_t qs = 0u;
            uint8_t qq = 0;
            if (mv) { q = C.Pl[p]; qs = C.Ps[p]; qq = C.Sq[p]; }
            __syncwarp();
            const int d = __popcll(use & ((1ull << p) - 1ull));
            if (mv) { C.Pl[d] = q; C.Ps[d] = qs; C.Sq[d] = qq; }
            __syncwarp();
        }
#pragma unroll 1
        for (int s = r; s < GNT; s += G)
            if (cp && in_set(vlo, vhi, (uint32_t)s)) {
                uint32_t a, b, c;
                const uint32_t w = __float_as_uint(C.V[s].w);
                ids_of(C.V[s].w, a, b, c);
                C.V[s].w = __uint_as_float((w & ~IDS) | pack_ids(__popcll(use & ((1ull << a) - 1ull)), __popcll(use & ((1ull << b) - 1ull)),
                                                                  __popcll(use & ((1ull << c) - 1ull))));
            }
        if (cp) {
            np = __popcll(use);
            if (np == GNP || nseq > 127) { fail = GF_CAP; cut = false; }
        }
        __syncwarp();
    }
    const int p = np;
    if (cut) {
        if (lane == (unsigned)src) {
            C.Pl[p] = pl;
            C.Ps[p] = from;
            C.Sq[p] = (uint8_t)nseq;
        }
        np++;
        nseq++;
    }
    int nB = 0;
#pragma unroll 1
    for (int tries = 0;; tries++) {
        // boundary edges: edge k of a removed vertex whose neighbour across it is kept; numbered by chunk of
        // 32 slots, edge, slot
        nB = 0;
#pragma unroll 1
        for (int e = 0; e < 2; e++) {
            const unsigned re = cut ? (e ? rem1 : rem0) : 0u;
            if (!__any_sync(FULL, re != 0u)) continue;
            unsigned first = re;
#pragma unroll
            for (int q = 0; q < G - 1; q++)
                if (q < r) first &= first - 1u;
            unsigned b0 = 0u, b1 = 0u, b2 = 0u;
            unsigned mm = first;
#pragma unroll 1
            while (__any_sync(FULL, mm != 0u)) {
                if (mm) {
                    const unsigned bit = mm & (0u - mm);
                    const uint32_t ad = C.Ad[e * 32 + __ffs(mm) - 1];
                    if (!in_set(rem0, rem1, ad & 255u)) b0 |= bit;
                    if (!in_set(rem0, rem1, (ad >> 8) & 255u)) b1 |= bit;
                    if (!in_set(rem0, rem1, (ad >> 16) & 255u)) b2 |= bit;
                }
#pragma unroll
                for (int q = 0; q < G; q++) mm &= mm - 1u;
            }
            b0 = gor<G>(b0); b1 = gor<G>(b1); b2 = gor<G>(b2);
            const int n0 = __popc(b0), n1 = __popc(b1), n2 = __popc(b2);
            mm = first;
#pragma unroll 1
            while (__any_sync(FULL, mm != 0u)) {
                if (mm) {
                    const unsigned bit = mm & (0u - mm);
                    const uint32_t t = (uint32_t)(e * 32 + __ffs(mm) - 1);
                    const uint32_t ad = C.Ad[t], tr = __float_as_uint(C.V[t].w);
#pragma unroll
                    for (int q = 0; q < 3; q++) {
                        const unsigned bq = q == 0 ? b0 : q == 1 ? b1 : b2;
                        if (!(bq & bit)) continue;
                        const int o = nB + (q > 0 ? n0 : 0) + (q > 1 ? n1 : 0) + __popc(bq & (bit - 1u));
                        const uint32_t nb = (ad >> (8 * q)) & 63u;
                        const uint32_t na = C.Ad[nb];
                        const uint32_t kn = (na & 255u) == t ? 0u : ((na >> 8) & 255u) == t ? 1u : 2u;
                        const uint32_t x = (tr >> (IDB5 * q)) & IDM5, y = (tr >> (q == 2 ? 0 : IDB5 * (q + 1))) & IDM5;
                        if (o < GBND) C.bnd[o] = x | (y << 6) | (nb << 12) | (kn << 18) | (SIGNS ? t << 26 : 0u);
                    }
                }
#pragma unroll
                for (int q = 0; q < G; q++) mm &= mm - 1u;
            }
            nB += n0 + n1 + n2;
        }
        unsigned long long fr = ~((((unsigned long long)vhi << 32) | vlo) & ~(((unsigned long long)rem1 << 32) | rem0)) &
                                (GNT == 64 ? ~0ull : (1ull << (GNT & 63)) - 1ull);
        if (SIGNS && nB > EARLY * G) fr &= ~(((unsigned long long)rem1 << 32) | rem0);
        const bool over = cut && (nB > min(GBND, __popcll(fr)) || nB < 3);
        if (over && (!SIGNS || tries)) { fail = GF_CAP; cut = false; }
        if (!cut) nB = 0;
        __syncwarp();
        // the i-th boundary edge takes the i-th lowest free slot
        w0 = w1 = 0u;
#pragma unroll
        for (int q = 0; q < G - 1; q++)
            if (q < r) fr &= fr - 1ull;
        const int nl = over ? 0 : nB, nlmax = __reduce_max_sync(FULL, nl);
#pragma unroll 1
        for (int i = r; i < nlmax; i += G) {
            if (i < nl) {
                const uint32_t t = (uint32_t)__ffsll((long long)fr) - 1u;
                const uint32_t rec = C.bnd[i];
                C.lnk_s[rec & 63u] = (uint8_t)t;
                C.lnk_e[(rec >> 6) & 63u] = (uint8_t)t;
                if (SIGNS) C.lnk_n[rec & 63u] = (uint8_t)((rec >> 6) & 63u);
                C.bnd[i] = rec | (t << 20);
                if (t < 32) w0 |= 1u << t; else w1 |= 1u << (t - 32);
            }
#pragma unroll
            for (int q = 0; q < G; q++) fr &= fr - 1ull;
        }
        if (!SIGNS) break;
        __syncwarp();
        // one loop: from the first edge's plane on, back at it after nB steps and not before (an entry may be an older
        // cut's, or never written: the steps are bounded)
        bool bad = over;
        if (nl > 0) {
            const uint32_t x0 = C.bnd[0] & 63u;
            uint32_t x = x0;
            int k = 0;
            do {
                x = C.lnk_n[x];
                k++;
            } while (x != x0 && x < (uint32_t)GNP && k < nl);
            bad = x != x0 || k != nl;
        }
        if (!__any_sync(FULL, bad)) break;
        if (tries) {  // (both sides whole: not reached)
            if (bad) { fail = GF_CAP; cut = false; nB = 0; }
            break;
        }
        unsigned long long rem = ((unsigned long long)rem1 << 32) | rem0;
        const float4 f = C.Pl[cut ? p : 0];
        if (bad && r == 0) rem = whole_sides(C, f, ((unsigned long long)vhi << 32) | vlo, rem);
        rem0 = __shfl_sync(FULL, (unsigned)rem, gsh);
        rem1 = __shfl_sync(FULL, (unsigned)(rem >> 32), gsh);
        __syncwarp();
    }
    const int nBmax = __reduce_max_sync(FULL, nB);
    __syncwarp();
    if (SIGNS) {
        // a new vertex may take the slot of a removed one that another lane reads: the first ones are read by all lanes before
        // any is written, and a longer boundary keeps off the removed slots
        float4 v[EARLY];
#pragma unroll
        for (int q = 0; q < EARLY; q++)
            if (r + q * G < nB) v[q] = on_edge(C, C.Pl[p], (uint32_t)p, C.bnd[r + q * G]);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < EARLY; q++)
            if (r + q * G < nB) C.V[(C.bnd[r + q * G] >> 20) & 63u] = v[q];
    }
    bool ill = false;
#pragma unroll 1
    for (int i = r; i < nBmax; i += G) {
        if (i < nB) {
            const uint32_t rec = C.bnd[i];
            const uint32_t x = rec & 63u, y = (rec >> 6) & 63u, nb = (rec >> 12) & 63u, kn = (rec >> 18) & 3u,
                           t = SIGNS ? (rec >> 20) & 63u : rec >> 20;
            C.Ad[t] = nb | ((uint32_t)C.lnk_s[y] << 8) | ((uint32_t)C.lnk_e[x] << 16);
            reinterpret_cast<uint8_t*>(&C.Ad[nb])[kn] = (uint8_t)t;
            if (SIGNS) {
                if (i >= EARLY * G) C.V[t] = on_edge(C, C.Pl[p], (uint32_t)p, rec);
                continue;
            }
            float rr;
            const float4 v = vertex_at(C, x, y, (uint32_t)p, rr);
            C.V[t] = make_float4(v.x, v.y, v.z, pack_w(v.w, pack_ids(x, y, (uint32_t)p)));
            if (!(v.w < INFINITY)) ill = true;
        }
    }
    w0 = gor<G>(w0); w1 = gor<G>(w1);
    if (cut) {
        vlo = (vlo & ~rem0) | w0;
        vhi = (vhi & ~rem1) | w1;
    }
    if ((__ballot_sync(FULL, ill) >> gsh) & ((1u << G) - 1u)) fail = GF_ILL;
}

// Clip the cells [c0, c0 + nc) that want a pass by their candidate lists.  last: cells that want another pass are handed
// over.
template <typename P, int G, bool SETS>
__global__ void __launch_bounds__(32, G == 4 ? 11 : 20) k_group_clip(const __grid_constant__ ClipArgs A,
                                                                     const __grid_constant__ GroupBuf B, uint32_t c0, uint32_t nc,
                                                                     uint32_t* ctr, int last, const uint32_t* act_list,
                                                                     const uint32_t* n_act, uint32_t* next_list,
                                                                     uint32_t* n_next) {
    constexpr int W = 32 / G;   // cells per warp
    constexpr int IT = 32 / G;  // planes per lane
    extern __shared__ __align__(16) unsigned char gsmem[];
    const unsigned lane = lane_id();
    const int r = (int)(lane & (G - 1));
    const int gsh = (int)(lane & ~(unsigned)(G - 1));  // first lane of the group
    constexpr unsigned GM = (1u << G) - 1u;
    const unsigned rlt = (1u << r) - 1u;
    GCell& C = reinterpret_cast<GCell*>(gsmem)[gsh / G];
    if (*((volatile unsigned*)&A.st->invalid_input)) return;
    const P* const spos = (const P*)A.spos;
    const float u = Prec<float>::u();
    const unsigned lead = W == 8 ? 0x11111111u : 0x01010101u;  // the groups' first lanes
    auto gballot = [&](bool p) -> unsigned { return (__ballot_sync(FULL, p) >> gsh) & GM; };

    // the group's cell
    bool has = false;
    uint32_t ci = 0, self = 0, set = 0;
    P pi = {};
    GHdr H = {};
    const uint32_t* list = B.list;
    unsigned vlo = 0u, vhi = 0u;  // vertex slots in use
    int np = 6, nseq = 6, fail = 0;
    unsigned art = 0u, used64 = 0u;
    float R2 = 0.f, bx0 = 0.f, by0 = 0.f, bz0 = 0.f, bx1 = 0.f, by1 = 0.f, bz1 = 0.f;
    // the warp's part of the queue: the cells wcell of the lanes in wmask
    const uint32_t count = act_list ? *n_act : nc;
    uint32_t wbase = 0, wcell = 0;
    unsigned wmask = 0u;
    bool dry = false;
    unsigned c_cut = 0, c_tested = 0, c_pass = 0, c_fp64 = 0, c_faces = 0, c_maxf = 0;

    // R2 (a bound of every exact vertex's |v|^2) and the outward-rounded box of the exact vertices
    auto bounds = [&](bool on) {
        float v2 = 0.f, em = 0.f, x0 = 0.f, y0 = 0.f, z0 = 0.f, x1 = 0.f, y1 = 0.f, z1 = 0.f;
        const int hw = vhi ? 64 - __clz(vhi) : 32 - __clz(vlo);
#pragma unroll 1
        for (int s = r; s < hw; s += G)
            if (on && in_set(vlo, vhi, (uint32_t)s)) {
                const float4 v = C.V[s];
                v2 = fmaxf(v2, __fmaf_rn(v.z, v.z, __fmaf_rn(v.y, v.y, v.x * v.x)));
                em = fmaxf(em, v.w);
                x0 = fminf(x0, __fsub_rd(v.x, v.w)); x1 = fmaxf(x1, __fadd_ru(v.x, v.w));
                y0 = fminf(y0, __fsub_rd(v.y, v.w)); y1 = fmaxf(y1, __fadd_ru(v.y, v.w));
                z0 = fminf(z0, __fsub_rd(v.z, v.w)); z1 = fmaxf(z1, __fadd_ru(v.z, v.w));
            }
        v2 = gmax<G>(v2); em = gmax<G>(em);
        x0 = gmin<G>(x0); y0 = gmin<G>(y0); z0 = gmin<G>(z0);
        x1 = gmax<G>(x1); y1 = gmax<G>(y1); z1 = gmax<G>(z1);
        if (on) {
            const float rr = sqrtf(v2) * (1.f + 8.f * u) + em;
            R2 = rr * rr * (1.f + 8.f * u);
            bx0 = x0; by0 = y0; bz0 = z0; bx1 = x1; by1 = y1; bz1 = z1;
        }
    };


    for (;;) {
        // ---------------------------------------------------------------- new cells for the idle groups
        bool fresh = false;
        {
            unsigned need = __ballot_sync(FULL, !has) & lead;
#pragma unroll 1
            while (need && !dry) {
                if (wmask == 0u) {
                    uint32_t b = 0;
                    if (lane == 0) b = atomicAdd(ctr, 32u);
                    wbase = __shfl_sync(FULL, b, 0);
                    if (wbase >= count) { dry = true; break; }
                    const bool in = wbase + lane < count;
                    wcell = !in ? 0u : act_list ? act_list[wbase + lane] : wbase + lane;
                    wmask = __ballot_sync(FULL, in && B.stat[wcell] != 0);
                    continue;
                }
                const int give = min(__popc(need), __popc(wmask));
                const int rank = __popc(need & ((1u << gsh) - 1u));
                unsigned m = wmask;
#pragma unroll 1
                for (int k = 0; k < rank; k++) m &= m - 1u;
                const uint32_t cell = __shfl_sync(FULL, wcell, m ? __ffs(m) - 1 : 0);
                if (((need >> gsh) & 1u) && rank < give) {
                    ci = cell;
                    has = fresh = true;
                }
#pragma unroll 1
                for (int k = 0; k < give; k++) { need &= need - 1u; wmask &= wmask - 1u; }
            }
        }
        if (!__any_sync(FULL, has)) break;
        if (fresh) {
            self = c0 + ci;
            if (SETS) set = A.sset[self];
            pi = spos[self];
            H = B.hdr[ci];
            list = B.list + (size_t)ci * GNC;
            fail = 0;
            used64 = 0u;
        }
        const Geometry& g = geo_of<SETS>(A, set);
        const bool periodic = SETS ? false : g.periodic != 0;
        if (fresh) {
            if (H.meta & GM_INIT) {
                float w[6];
                art = start_box<P>(g, periodic, pi, H.B, w);
                np = nseq = 6;
                used64 = (H.meta >> 16) & 1u;
                for (int k = r; k < 6; k += G) {
                    const float sg = (k & 1) ? -1.f : 1.f;
                    const float wk = k == 0 ? w[0] : k == 1 ? w[1] : k == 2 ? w[2] : k == 3 ? w[3] : k == 4 ? w[4] : w[5];
                    C.Pl[k] = make_float4(k < 2 ? sg : 0.f, (k >> 1) == 1 ? sg : 0.f, k > 3 ? sg : 0.f, wk);
                    C.Ps[k] = self;
                    C.Sq[k] = (uint8_t)k;
                }
                // corners: planes x upper 0 / lower 1, y 2/3, z 4/5, counter-clockwise seen from outside, and their
                // adjacency (across x->y the corner that holds y->x).  A wall's offset has relative error u at most, so
                // 16u |v| bounds a corner's error and the rounding of its tests.
#pragma unroll 1
                for (int k = r; k < 8; k += G) {
                    const bool even = (__popc((unsigned)k) & 1) == 0;
                    const uint32_t X = (k & 1) ? 1 : 0, Y = (k & 2) ? 3 : 2, Z = (k & 4) ? 5 : 4;
                    const float x = (k & 1) ? -w[1] : w[0], y = (k & 2) ? -w[3] : w[2], z = (k & 4) ? -w[5] : w[4];
                    const float ev = 16.f * u * sqrtf(f_fma<float>(z, z, f_fma<float>(y, y, x * x)));
                    C.V[k] = make_float4(x, y, z, pack_w(ev, pack_ids(X, even ? Y : Z, even ? Z : Y)));
                    // neighbours: flip z, x, y in the order of the edges
                    const uint32_t fx = (uint32_t)k ^ 1u, fy = (uint32_t)k ^ 2u, fz = (uint32_t)k ^ 4u;
                    C.Ad[k] = even ? (fz | (fx << 8) | (fy << 16)) : (fy | (fx << 8) | (fz << 16));
                }
                vlo = 0xffu; vhi = 0u;
            } else {
                // the state as the last pass left it
                vlo = H.vlo; vhi = H.vhi;
                np = (int)(H.meta & 255u);
                nseq = (int)(H.n >> 16);
                art = (H.meta >> 8) & 63u;
                used64 = (H.meta >> 16) & 1u;
                const int hw = vhi ? 64 - __clz(vhi) : 32 - __clz(vlo);
                const GCell* const K = reinterpret_cast<const GCell*>(B.state + (size_t)ci * GROUP_STATE);
                for (int s = r; s < hw; s += G) { C.V[s] = K->V[s]; C.Ad[s] = K->Ad[s]; }
                for (int p = r; p < np; p += G) { C.Pl[p] = K->Pl[p]; C.Ps[p] = K->Ps[p]; C.Sq[p] = K->Sq[p]; }
            }
        }
        __syncwarp();

        // ---------------------------------------------------------------- cut by the candidates, in order of distance
        // Batches of G, one per lane: every lane tests its plane against all vertices; then the first cutting plane is
        // applied and the later ones are tested against the new vertices only, until none cuts (a plane that misses a
        // polytope misses every subset of it).
        bool cert = false;
        const int nlist = has ? (int)(H.n & 0xffffu) : 0;
        int lim = nlist;
        int dirty = has ? 1 : 0;
#pragma unroll 1
        for (int base = 0;; base += G) {
            bool open = has && !fail && base < lim;
            if (__any_sync(FULL, dirty >= 3 || (dirty > 0 && (base == 0 || !open)))) {
                bounds(dirty > 0);
                dirty = 0;
            }
            if (!__any_sync(FULL, open)) break;
            const int k = base + r;
            float cdx = 0.f, cdy = 0.f, cdz = 0.f, chh = 0.f, cnr = 0.f;
            uint32_t cjj = 0;
            if (open && k < lim) {
                cjj = list[k];
                gdisp<P, SETS>(spos[cjj], pi, g, cdx, cdy, cdz);
                const float d2 = f_fma<float>(cdz, cdz, f_fma<float>(cdy, cdy, cdx * cdx));
                chh = 0.5f * d2;
                cnr = sqrtf(d2);
                c_tested++;
            }
            const float chb = 16.f * u * chh;
            // the list is ordered: from the first |d| >= 2R on nothing can cut, and nothing farther either
            const unsigned fm = gballot(open && k < lim && 2.f * chh * (1.f - 8.f * u) > 4.f * R2);
            if (fm) {
                lim = base + __ffs(fm) - 1;
                cert = true;
            }
            bool on = open && k < lim;
            if (gballot(on && chh == 0.f)) { fail = GF_DUP; on = false; }
            unsigned olo = 0u, ohi = 0u, ulo = 0u, uhi = 0u;
            {
                const int hw = open ? (vhi ? 64 - __clz(vhi) : 32 - __clz(vlo)) : 0;
                const int hmax = __reduce_max_sync(FULL, hw);
#pragma unroll 1
                for (int s0 = 0; s0 < hmax; s0 += 4) {
                    unsigned o4 = 0u, u4 = 0u;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const float4 v = C.V[s0 + q];
                        const float sv = f_fma<float>(cdx, v.x, f_fma<float>(cdy, v.y, f_fma<float>(cdz, v.z, -chh)));
                        const float bd = f_fma<float>(cnr, v.w, chb);
                        if (sv > bd) o4 |= 1u << q;
                        if (!(sv < -bd)) u4 |= 1u << q;
                    }
                    if (s0 < 32) { olo |= o4 << s0; ulo |= u4 << s0; }
                    else { ohi |= o4 << (s0 - 32); uhi |= u4 << (s0 - 32); }
                }
            }
            olo = on ? olo & vlo : 0u; ohi = on ? ohi & vhi : 0u;
            ulo = on ? ulo & vlo & ~olo : 0u; uhi = on ? uhi & vhi & ~ohi : 0u;
#pragma unroll 1
            for (;;) {
                if (__any_sync(FULL, (ulo | uhi) != 0u)) {
                    // tests the error bound left undecided: FP64 from the inputs
                    bool und = false;
                    while (ulo | uhi) {
                        const int s = ulo ? __ffs(ulo) - 1 : 31 + __ffs(uhi);
                        if (ulo) ulo &= ulo - 1; else uhi &= uhi - 1;
                        const int sd = resolve64<P>(C, s, cjj, art, self, spos, g);
                        c_fp64++;
                        used64 = 1u;
                        if (sd == 0) und = true;
                        if (sd > 0) { if (s < 32) olo |= 1u << s; else ohi |= 1u << (s - 32); }
                    }
                    __syncwarp();
                    if (gballot(und)) fail = GF_UNDECIDED;
                }
                const unsigned cm = gballot((olo | ohi) != 0u);
                bool cut = open && !fail && cm != 0u;
                if (!__any_sync(FULL, cut)) break;
                const int src = gsh + (cut ? __ffs(cm) - 1 : 0);
                unsigned rem0 = __shfl_sync(FULL, olo, src), rem1 = __shfl_sync(FULL, ohi, src);
                unsigned w0, w1;
                c_cut += cut && r == 0;
                dirty += cut;
                group_cut<G, false>(C, cut, src, rem0, rem1, make_float4(cdx, cdy, cdz, chh), cjj, vlo, vhi, np, nseq, fail, w0, w1);
                __syncwarp();
                // the later planes against the new vertices
                olo &= ~rem0; ohi &= ~rem1;
                if ((int)lane <= src) olo = ohi = 0u;
                const bool later = on && cut && (int)lane > src;
                unsigned m0 = cut ? w0 : 0u, m1 = cut ? w1 : 0u;
#pragma unroll 1
                while (__any_sync(FULL, (m0 | m1) != 0u)) {
                    const int s = m0 ? __ffs(m0) - 1 : m1 ? 31 + __ffs(m1) : 0;
                    if (m0) m0 &= m0 - 1u; else m1 &= m1 - 1u;
                    const float4 v = C.V[s];
                    const float sv = f_fma<float>(cdx, v.x, f_fma<float>(cdy, v.y, f_fma<float>(cdz, v.z, -chh)));
                    const float bd = f_fma<float>(cnr, v.w, chb);
                    const unsigned b0 = s < 32 ? 1u << s : 0u, b1 = s < 32 ? 0u : 1u << (s - 32);
                    if (later) {
                        if (sv > bd) { olo |= b0; ohi |= b1; }
                        else if (!(sv < -bd)) { ulo |= b0; uhi |= b1; }
                    }
                }
                if (cut) {
                    // only the new slots hold undecided tests now; a group that did not cut is done with the batch
                    ulo &= w0; uhi &= w1;
                }
                if (!cut) olo = ohi = ulo = uhi = 0u;
            }
        }

        // ---------------------------------------------------------------- certified, or the next radius
        bool done = false, again = false;
        int pass = 0;
        if (has && !fail) {
            c_pass += r == 0;
            pass = (int)(H.meta >> 24) + 1;
            if (cert || H.rhi2 * (1.f - 8.f * u) >= 4.f * R2) done = true;
            else if (!(R2 < INFINITY)) fail = GF_ILL;
            else if (H.rhi2 >= H.cap2 || pass >= A.max_passes || last) fail = GF_RADIUS;
            else {
                // the annulus up to 2R, at most twice the radius (policy 1: also no further than the radius that the
                // density seen so far says holds three times a pass's capacity: the support test leaves fewer)
                const float nxt = 4.f * R2 * (1.f + 32.f * u);
                float lim2 = 4.f * H.rhi2;
                if (A.radius_policy == 1 && nlist > 0) {
                    const float rh = sqrtf(H.rhi2), rl = sqrtf(H.rlo2);
                    const float shell = rh * rh * rh - rl * rl * rl;
                    if (shell > 0.f) {
                        const float rr = cbrtf(rh * rh * rh + 3.f * GNC * shell / (float)nlist);
                        lim2 = fminf(lim2, fmaxf(rr * rr, 1.21f * H.rhi2));
                    }
                }
                H.rlo2 = H.rhi2;
                H.rhi2 = fminf(fminf(nxt, lim2), H.cap2);
                H.meta = ((uint32_t)pass << 24) | (art << 8) | (uint32_t)np;
                H.vlo = vlo; H.vhi = vhi;
                H.n = (uint32_t)nseq << 16;
                again = true;
            }
            if (done && periodic) {
                const double lmin = fmin(g.L[0], fmin(g.L[1], g.L[2]));
                if (!(16.f * R2 < (float)(lmin * lmin))) { done = false; fail = GF_RADIUS; }
            }
        }
        const unsigned w64 = gor<G>(used64);
        bool queue = again;  // the cell's next pass
        if (again) {
            GCell* const K = reinterpret_cast<GCell*>(B.state + (size_t)ci * GROUP_STATE);
            const int hw = vhi ? 64 - __clz(vhi) : 32 - __clz(vlo);
#pragma unroll 1
            for (int s = r; s < hw; s += G) { K->V[s] = C.V[s]; K->Ad[s] = C.Ad[s]; }
#pragma unroll 1
            for (int p = r; p < np; p += G) { K->Pl[p] = C.Pl[p]; K->Ps[p] = C.Ps[p]; K->Sq[p] = C.Sq[p]; }
            if (r == 0) {
                H.bx0 = bx0; H.by0 = by0; H.bz0 = bz0; H.bx1 = bx1; H.by1 = by1; H.bz1 = bz1;
                H.meta |= w64 << 16;
                B.hdr[ci] = H;
            }
            has = false;
        }

        // ---------------------------------------------------------------- emission
        if (__any_sync(FULL, done)) {
            __syncwarp();
            if (done) {
#pragma unroll 1
                for (int p = r; p < GNP; p += G) C.first[p] = 0xffffffffu;
            }
            __syncwarp();
            // the planes' first slots, and the bound of the cell's radius: the largest of the vertices' (the stored
            // error bounds are rounded up: the vertices within that of the largest are computed again)
            float rmax = 0.f, wmax = 0.f, rr2 = 0.f;
            unsigned pr0 = 0u, pr1 = 0u;
            auto reach_of = [&](const float4& v) -> float {
                const float vn = sqrtf(f_fma<float>(v.z, v.z, f_fma<float>(v.y, v.y, v.x * v.x)));
                return vn * (1.f + 4.f * u) + (v.w - 8.f * u * vn);
            };
#pragma unroll 1
            for (int s = r; s < GNT; s += G)
                if (done && in_set(vlo, vhi, (uint32_t)s)) {
                    uint32_t a, b, c;
                    const float4 v = C.V[s];
                    ids_of(v.w, a, b, c);
                    atomicMin(&C.first[a], (uint32_t)s);
                    atomicMin(&C.first[b], (uint32_t)s);
                    atomicMin(&C.first[c], (uint32_t)s);
                    const unsigned long long mk = (1ull << a) | (1ull << b) | (1ull << c);
                    pr0 |= (unsigned)mk; pr1 |= (unsigned)(mk >> 32);
                    rmax = fmaxf(rmax, reach_of(v));
                    wmax = fmaxf(wmax, v.w);
                }
            rmax = gmax<G>(rmax);
            wmax = gmax<G>(wmax);
            const unsigned long long present = ((unsigned long long)gor<G>(pr1) << 32) | gor<G>(pr0);
#pragma unroll 1
            for (int s = r; s < GNT; s += G)
                if (done && in_set(vlo, vhi, (uint32_t)s)) {
                    const float4 v = C.V[s];
                    if (reach_of(v) * (1.f + 1e-6f) + 0.08f * wmax >= rmax) {
                        uint32_t a, b, c;
                        ids_of(v.w, a, b, c);
                        float rr;
                        vertex_at(C, a, b, c, rr);
                        rr2 = fmaxf(rr2, rr);
                    }
                }
            rr2 = gmax<G>(rr2);
            __syncwarp();
            if (done && (present & art)) {
                // the start box was too small: the cell starts again without artificial walls (with the bisectors of its own
                // images in a periodic box; a facet on one of those is the warp kernel's to refuse)
                done = false;
                if (last || !(H.B < INFINITY) || pass >= A.max_passes) fail = GF_WALL;
                else {
                    queue = true;
                    if (r == 0) {
                        H.B = INFINITY;
                        H.meta = ((uint32_t)pass << 24) | GM_INIT | (w64 << 16);
                        B.hdr[ci] = H;
                    }
                    has = false;
                }
            }
            const int nf = done ? __popcll(present >> 6) : 0;
            // facet records of the warp's finished cells, reserved at once
            uint32_t start = 0;
            bool pool = true;
            {
                int inc = r == 0 ? nf : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(FULL, inc, o);
                    if ((int)lane >= o) inc += y;
                }
                const int all = __shfl_sync(FULL, inc, 31);
                unsigned long long b = 0ull;
                if (lane == 0 && all > 0) b = atomicAdd(&A.st->face_next, (unsigned long long)all);
                b = __shfl_sync(FULL, b, 0);
                const unsigned long long s0 = b + (unsigned long long)(__shfl_sync(FULL, inc, gsh) - nf);
                pool = s0 + (unsigned long long)nf <= A.face_cap;
                start = (uint32_t)s0;
            }
            if (done && !pool) {
                if (r == 0) {
                    A.cstat[self] = CS_ERROR;
                    B.stat[ci] = 0;
                    if (atomicCAS(&A.st->error, 0, RC_POOL) == 0) {
                        A.st->error_cell = (int)self;
                        A.st->error_detail = RC_POOL;
                    }
                }
                done = false;
                has = false;
            }
            // one plane per lane and turn: the facet's fan from its first vertex.  A plane's sums take the place of its
            // equation (only this lane reads it); planes without a facet get zeros.
            if (done) {
#pragma unroll 1
                for (int p = r; p < GNP; p += G)
                    if (!((present >> p) & 1ull)) {
                        C.Pl[p] = make_float4(0.f, 0.f, 0.f, 0.f);
                        C.Ps[p] = 0u;
                    }
            }
            unsigned long long pm = done ? present : 0ull;
#pragma unroll 1
            while (__any_sync(FULL, pm != 0ull)) {
                unsigned long long mm = pm;
#pragma unroll
                for (int q = 0; q < G; q++) {
                    if (q < r) mm &= mm - 1ull;
                    pm &= pm - 1ull;
                }
                if (mm) {
                    const int p = __ffsll((long long)mm) - 1;
                    const uint32_t t0 = C.first[p];
                    const float4 v0 = C.V[t0];
                    const float4 pp = C.Pl[p];
                    const float inrm = 1.f / (p < 6 ? 1.f : sqrtf(2.f * pp.w));
                    const float nhx = pp.x * inrm, nhy = pp.y * inrm, nhz = pp.z * inrm;
                    KSum<float> kA;
                    kA.zero();
                    float csx = 0.f, csy = 0.f, csz = 0.f, sm2 = 0.f;
                    // successor around the plane: the neighbour across the edge (corner before p) -> p
                    auto succ = [&](uint32_t t) -> uint32_t {
                        uint32_t a, b, c;
                        ids_of(C.V[t].w, a, b, c);
                        const int k = a == (uint32_t)p ? 2 : b == (uint32_t)p ? 0 : 1;
                        return (C.Ad[t] >> (8 * k)) & 63u;
                    };
                    uint32_t cur = succ(t0);
#pragma unroll 1
                    for (int guard = 0; guard < GNT && cur != t0; guard++) {
                        const uint32_t nxt = succ(cur);
                        if (nxt == t0) break;
                        const float4 v1 = C.V[cur], v2 = C.V[nxt];
                        const float e1x = v1.x - v0.x, e1y = v1.y - v0.y, e1z = v1.z - v0.z;
                        const float e2x = v2.x - v0.x, e2y = v2.y - v0.y, e2z = v2.z - v0.z;
                        const float crx = f_fma<float>(e1y, e2z, -e1z * e2y), cry = f_fma<float>(e1z, e2x, -e1x * e2z),
                                    crz = f_fma<float>(e1x, e2y, -e1y * e2x);
                        const float at = 0.5f * f_fma<float>(crx, nhx, f_fma<float>(cry, nhy, crz * nhz));
                        kA.add(at);
                        const float third = (float)(1.0 / 3.0);
                        csx = f_fma<float>(at * third, v0.x + v1.x + v2.x, csx);
                        csy = f_fma<float>(at * third, v0.y + v1.y + v2.y, csy);
                        csz = f_fma<float>(at * third, v0.z + v1.z + v2.z, csz);
                        float s2 = f_fma<float>(v0.x, v0.x + v1.x + v2.x, f_fma<float>(v0.y, v0.y + v1.y + v2.y, v0.z * (v0.z + v1.z + v2.z)));
                        s2 = f_fma<float>(v1.x, v1.x + v2.x, f_fma<float>(v1.y, v1.y + v2.y, f_fma<float>(v1.z, v1.z + v2.z, s2)));
                        s2 = f_fma<float>(v2.x, v2.x, f_fma<float>(v2.y, v2.y, f_fma<float>(v2.z, v2.z, s2)));
                        sm2 = f_fma<float>(at, s2, sm2);
                        cur = nxt;
                    }
                    const float A_ = kA.value();
                    const float dist = pp.w * inrm;
                    const float qv = dist * A_ * (float)(1.0 / 3.0);
                    const float qx = dist * csx * 0.25f;
                    const float qy = dist * csy * 0.25f;
                    const float qz = dist * csz * 0.25f;
                    const float q2 = dist * sm2;
                    if (p >= 6) {
                        Face f;
                        f.dx = pp.x; f.dy = pp.y; f.dz = pp.z;
                        f.area = A_;
                        if (A_ != 0.f) { f.cx = csx / A_; f.cy = csy / A_; f.cz = csz / A_; }
                        else { f.cx = f.cy = f.cz = 0.f; }
                        f.nbr = C.Ps[p];
                        A.faces[start + (uint32_t)__popcll((present >> 6) & ((1ull << (p - 6)) - 1ull))] = f;
                    }
                    C.Pl[p] = make_float4(qv, qx, qy, qz);
                    C.Ps[p] = __float_as_uint(q2);
                }
            }
            __syncwarp();
            // the sums over planes as a butterfly over 32 lanes would take them, each plane on the lane of its number (plane p on lane p)
            KSum<float> kv[IT];
            float zx[IT], zy[IT], zz[IT], z2[IT];
            const bool moved = done && np < nseq;  // planes were dropped: ids and numbers differ
#pragma unroll
            for (int e = 0; e < IT; e++) {
                const float4 v = C.Pl[e * G + r];
                kv[e].s = v.x; kv[e].c = 0.f;
                zx[e] = v.y; zy[e] = v.z; zz[e] = v.w;
                z2[e] = __fmul_rn(__uint_as_float(C.Ps[e * G + r]), (float)(1.0 / 30.0));
                if (e * G + 32 < GNP) {
                    const float4 x = C.Pl[32 + e * G + r];
                    kv[e].add(x.x);
                    zx[e] += x.y; zy[e] += x.z; zz[e] += x.w;
                    z2[e] = __fmaf_rn(__uint_as_float(C.Ps[32 + e * G + r]), (float)(1.0 / 30.0), z2[e]);
                }
            }
            if (__any_sync(FULL, moved)) {
#pragma unroll
                for (int e = 0; e < IT; e++) {
                    if (moved) {
                        kv[e].zero();
                        zx[e] = zy[e] = zz[e] = z2[e] = 0.f;
                    }
#pragma unroll 1
                    for (int p = 0; p < GNP; p++)
                        if (moved && p < np && (C.Sq[p] & 31) == e * G + r) {
                            const float4 x = C.Pl[p];
                            kv[e].add(x.x);
                            zx[e] += x.y; zy[e] += x.z; zz[e] += x.w;
                            z2[e] = __fmaf_rn(__uint_as_float(C.Ps[p]), (float)(1.0 / 30.0), z2[e]);
                        }
                }
            }
            auto join = [&](KSum<float>& a, float so, float co) {
                float t, e;
                tsum_f(a.s, so, t, e);
                a.s = t;
                a.c = __fadd_rn(__fadd_rn(a.c, co), e);
            };
#pragma unroll
            for (int o = IT / 2; o; o >>= 1)
#pragma unroll
                for (int e = 0; e < o; e++) {
                    join(kv[e], kv[e + o].s, kv[e + o].c);
                    zx[e] += zx[e + o]; zy[e] += zy[e + o]; zz[e] += zz[e + o]; z2[e] += z2[e + o];
                }
#pragma unroll
            for (int o = G / 2; o; o >>= 1) {
                const float so = __shfl_xor_sync(FULL, kv[0].s, o), co = __shfl_xor_sync(FULL, kv[0].c, o);
                join(kv[0], so, co);
                zx[0] += __shfl_xor_sync(FULL, zx[0], o);
                zy[0] += __shfl_xor_sync(FULL, zy[0], o);
                zz[0] += __shfl_xor_sync(FULL, zz[0], o);
                z2[0] += __shfl_xor_sync(FULL, z2[0], o);
            }
            if (done) {
                float vol = kv[0].value(), m2 = z2[0];
                const float sg = vol < 0.f ? -1.f : 1.f;
                vol *= sg; m2 *= sg;
                if (sg < 0.f) {
#pragma unroll 1
                    for (int k = r; k < nf; k += G) A.faces[start + k].area = -A.faces[start + k].area;
                }
                if (r == 0) {
                    CellOut co;
                    co.vol = (double)vol;
                    co.zx = vol > 0.f ? sg * zx[0] / vol : 0.f;
                    co.zy = vol > 0.f ? sg * zy[0] / vol : 0.f;
                    co.zz = vol > 0.f ? sg * zz[0] / vol : 0.f;
                    co.mom2 = m2;
                    A.cell[self] = co;
                    if (A.rad) A.rad[self] = (float)sqrt((double)rr2) * (1.f + 1e-6f);
                    A.face_start[self] = start;
                    A.face_count[self] = (uint16_t)nf;
                    A.cstat[self] = (uint8_t)(CS_DONE | (w64 ? CS_FP64 : 0));
                    B.stat[ci] = 0;
                    c_faces += nf;
                    c_maxf = max(c_maxf, (unsigned)nf);
                }
                has = false;
            }
            __syncwarp();
        }
        if (next_list) {
            const unsigned qm = __ballot_sync(FULL, queue) & lead;
            if (qm) {
                unsigned slot = 0;
                if (lane == 0) slot = atomicAdd(n_next, (unsigned)__popc(qm));
                slot = __shfl_sync(FULL, slot, 0);
                if (queue && r == 0) next_list[slot + __popc(qm & ((1u << lane) - 1u))] = ci;
            }
        }
        // ---------------------------------------------------------------- cells for the warp kernel
        const bool hand = has && fail != 0;
        const unsigned hm = __ballot_sync(FULL, hand) & lead;
        if (hm) {
            unsigned slot = 0;
            if (lane == 0) slot = atomicAdd(&A.st->n_warp_cells, (unsigned)__popc(hm));
            slot = __shfl_sync(FULL, slot, 0);
            if (hand && r == 0) {
                A.warp_list[slot + __popc(hm & ((1u << lane) - 1u))] = self;
                atomicAdd(&A.st->n_tfail[fail & 7], 1ull);
                B.stat[ci] = 0;
            }
        }
        if (hand) has = false;
    }
    // counters
    unsigned v[5] = {c_cut, c_tested, c_pass, c_fp64, c_faces};
#pragma unroll
    for (int k = 0; k < 5; k++) v[k] = __reduce_add_sync(FULL, v[k]);
    c_maxf = __reduce_max_sync(FULL, c_maxf);
    if (lane == 0) {
        atomicAdd(&A.st->n_cut, (unsigned long long)v[0]);
        atomicAdd(&A.st->n_tested, (unsigned long long)v[1]);
        atomicAdd(&A.st->n_passes, (unsigned long long)v[2]);
        atomicAdd(&A.st->n_fp64, (unsigned long long)v[3]);
        atomicAdd(&A.st->n_faces, (unsigned long long)v[4]);
        atomicMax(&A.st->max_faces, c_maxf);
    }
}

// blocks per SM of a kernel, with its shared-memory attribute set: once per device (no such call is made while a
// stream is being captured, after the first launch)
template <typename K>
int blocks_per_sm(K kernel, int threads, size_t smem, int* per_sm_dev) {
    int dev = 0;
    cudaGetDevice(&dev);
    int per_sm = (dev >= 0 && dev < 64) ? per_sm_dev[dev] : 0;
    if (per_sm == 0) {
        if (smem) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
        if (per_sm < 1) per_sm = 1;
        if (dev >= 0 && dev < 64) per_sm_dev[dev] = per_sm;
    }
    return per_sm;
}

template <typename P, bool SETS, bool FIRST>
void launch_search(const ClipArgs& a, const GroupBuf& b, uint32_t c0, uint32_t nc, uint32_t* ctr, int mode,
                   const uint32_t* act, const uint32_t* n_act, int sm_count, cudaStream_t s) {
    static int per_sm_dev[64] = {0};
    const int per_sm = blocks_per_sm(k_group_search<P, SETS, FIRST>, SWARPS * 32, 0, per_sm_dev);
    const unsigned all = (unsigned)(sm_count * per_sm);
    // cells a warp takes at a time: 32 share what is loaded for a bucket; 8 where 32 would leave the chip short of warps
    // listed cells one by one: they are the widest, and the slowest search is the launch's time
    const uint32_t unit = act ? 1u : FIRST && nc >= 64u * SWARPS * all ? 32u : 8u;
    const unsigned most = (nc + unit * SWARPS - 1) / (unit * SWARPS);
    k_group_search<P, SETS, FIRST><<<most < all ? most : all, SWARPS * 32, 0, s>>>(a, b, c0, nc, ctr, unit, mode, act, n_act);
}
template <typename P, int G, bool SETS>
void launch_gclip(const ClipArgs& a, const GroupBuf& b, uint32_t c0, uint32_t nc, uint32_t* ctr, int last,
                  const uint32_t* act, const uint32_t* n_act, uint32_t* next, uint32_t* n_next, int sm_count, cudaStream_t s) {
    static int per_sm_dev[64] = {0};
    constexpr int W = 32 / G;
    const size_t smem = W * sizeof(GCell);
    const int per_sm = blocks_per_sm(k_group_clip<P, G, SETS>, 32, smem, per_sm_dev);
    const unsigned most = (nc + W - 1) / W, all = (unsigned)(sm_count * per_sm);
    k_group_clip<P, G, SETS><<<most < all ? most : all, 32, smem, s>>>(a, b, c0, nc, ctr, last, act, n_act, next, n_next);
}

template <typename P, int G, bool SETS>
int launch_group(const ClipArgs& a, const GroupBuf& b, int sm_count, cudaStream_t s) {
    constexpr int MODE = G == 4 ? 2 : 3;
    const uint32_t N = (uint32_t)a.N;
    uint32_t* ctr = b.ctr + (G == 4 ? 0 : group_counters(a.N) / 2);
    // A pass over few cells costs its latency, 0.2 to 0.7 ms with the widest of them: a small set hands over early.  Clip
    // times of 65,537 / 200,000 / 1,000,000 clustered particles with 3 passes 5.2 / 9.35 / 35.0 ms, with 4 5.4 / 9.0 /
    // 32.1, with 6 5.8 / 10.2 / 32.1, with 8 6.4 / 10.75 / 32.9.
    const int passes = a.N < (int64_t)(1 << 17) ? 3 : a.N < (int64_t)(1 << 20) ? 4 : GROUP_PASSES;
    int n = 0;
    for (uint32_t c0 = 0; c0 < N; c0 += b.chunk) {
        const uint32_t nc = N - c0 < b.chunk ? N - c0 : b.chunk;
        // counters of a pass: search queue, clip queue, cells listed for the next pass.  The first passes take the
        // chunk's cells in order (neighbours search together); from pass GLIST on the few left are listed
        for (int p = 0; p < passes; p++, ctr += 4) {
            const int last = p == passes - 1;
            const uint32_t *act = p < GLIST ? nullptr : b.act + (size_t)(p & 1) * b.chunk, *n_act = p < GLIST ? nullptr : ctr - 2;
            uint32_t* next = p >= GLIST - 1 && !last ? b.act + (size_t)((p + 1) & 1) * b.chunk : nullptr;
            if (p == 0) launch_search<P, SETS, true>(a, b, c0, nc, ctr, MODE, act, n_act, sm_count, s);
            else launch_search<P, SETS, false>(a, b, c0, nc, ctr, MODE, act, n_act, sm_count, s);
            launch_gclip<P, G, SETS>(a, b, c0, nc, ctr + 1, last, act, n_act, next, ctr + 2, sm_count, s);
            n += 2;
        }
    }
    return n;
}
// ------------------------------------------------------------------ volume-averaged grid: (cell, voxel) pairs
// The part of a voxel inside a cell is the voxel cut by the cell's facet planes, and most pairs need no cutting: the
// voxel lies outside one plane (no part), or inside all of them (all of it); a cell whose ball lies in one voxel gives it
// its whole volume.  A warp takes 32 cells at a time, its lanes one pair each of all the voxels that the cells' balls
// meet.  The pairs that some plane crosses wait in queues (of about the same number of crossing planes) until there are
// enough, and are cut by the crossing planes alone, G lanes a pair as in k_group_clip, starting from the voxel's box (cut
// down to the ball's).  Sides are plain FP32 signs: a wrong sign within rounding of a plane moves a rounding-sized sliver,
// and signs that contradict each other are put right in the cut (group_cut).  What outgrows the polytope goes to a list.
// Cells whose balls meet more than GV_BIG voxels are listed, with the running count of their units of GV_BIG pairs, and
// the warps of a second launch take those units from a counter (2,097,152 clustered particles on 256^3 voxels: 166 ms;
// 8.1 s when every warp went through all listed cells, 6.9 s with one thread a cell).
// Bound by instruction issue, as k_group_clip.  131,072 clustered particles on 32^3 voxels: 4.8 ms (4.75 ms without the check
// of a cut's boundary, whose signs near a lattice left parts of voxels wrong by up to a tenth); 297 ms with one thread
// walking all voxels of a cell and clipping a copy of it by each voxel's walls; 13 ms with one thread a pair (5 of 32 lanes
// active, and the lanes' polytopes in local memory).
constexpr int GV_BIG = 512;
constexpr int GV_CLASSES = 4;
constexpr int BIG_BITS = 36;

struct GridWarp {
    int pref[33];
    int a0[3][32], n[3][32];  // first voxel and number of voxels per axis (unwrapped)
    int4 q[GV_CLASSES][64];   // pairs to cut, by class
};

template <typename P, bool BIG>
__global__ void __launch_bounds__(32, 9) k_group_voxels(const __grid_constant__ GridArgs A) {
    constexpr int G = 4, W = 32 / G;
    extern __shared__ __align__(16) unsigned char gsmem[];
    GCell* const cells = reinterpret_cast<GCell*>(gsmem);
    GridWarp& S = *reinterpret_cast<GridWarp*>(cells + W);
    const unsigned lane = lane_id(), lt = lanemask_lt();
    const int r = (int)(lane & (G - 1)), gsh = (int)(lane & ~(unsigned)(G - 1));
    constexpr unsigned GM = (1u << G) - 1u;
    GCell& C = cells[gsh / G];
    const P* const spos = (const P*)A.spos;
    const double vox = A.h[0] * A.h[1] * A.h[2];
    const unsigned long long listed = BIG ? *((volatile unsigned long long*)&A.ctr->n_big) : 0ull;
    const unsigned long long n_units = listed & ((1ull << BIG_BITS) - 1ull);
    auto gballot = [&](bool p) -> unsigned { return (__ballot_sync(FULL, p) >> gsh) & GM; };
    auto gsum = [&](float v) -> float {
#pragma unroll
        for (int o = G / 2; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    };
    int nq[GV_CLASSES];
#pragma unroll
    for (int c = 0; c < GV_CLASSES; c++) nq[c] = 0;

    unsigned b = 0;
    int64_t total = 0, t1 = 0;
    bool more = true;
    for (;;) {
        // ---------------------------------------------------------------- 32 pairs to look at
        if (t1 >= total && more) {
            total = 0;
            if (BIG) {
                // one unit of a listed cell: the last cell whose first unit is not beyond it
                unsigned long long u = 0;
                if (lane == 0) u = atomicAdd(&A.ctr->big_queue, 1ull);
                u = __shfl_sync(FULL, u, 0);
                if (u >= n_units) more = false;
                else {
                    uint32_t e = 0, e1 = (uint32_t)(listed >> BIG_BITS);
                    while (e1 - e > 1) {
                        const uint32_t mid = (e + e1) >> 1;
                        if (A.big_unit[mid] <= u) e = mid;
                        else e1 = mid;
                    }
                    const uint32_t k = A.big[e];
                    const P pi = spos[k];
                    const double xi[3] = {(double)pi.x, (double)pi.y, (double)pi.z};
                    int a0[3], n[3];
                    total = ball_voxels(A, xi, A.rad[k] * (1.f + 4e-6f), a0, n);
                    if (lane < 3) {
                        S.a0[lane][0] = lane == 0 ? a0[0] : lane == 1 ? a0[1] : a0[2];
                        S.n[lane][0] = lane == 0 ? n[0] : lane == 1 ? n[1] : n[2];
                    }
                    b = k;
                    t1 = (int64_t)(u - A.big_unit[e]) * GV_BIG;
                    total = min(total, t1 + GV_BIG);
                }
            } else {
                if (lane == 0) b = atomicAdd(&A.ctr->queue, 32u);
                b = __shfl_sync(FULL, b, 0);
                if ((int64_t)b >= A.N) more = false;
                else {
                    const int64_t k = (int64_t)b + lane;
                    int m = 0;
                    if (k < A.N && A.rad[k] > 0.f) {
                        const P pi = spos[k];
                        const double xi[3] = {(double)pi.x, (double)pi.y, (double)pi.z};
                        int a0[3], n[3];
                        const int64_t mm = ball_voxels(A, xi, A.rad[k] * (1.f + 4e-6f), a0, n);
                        if (mm == 1) {
                            int64_t v[3];
                            for (int c = 0; c < 3; c++) {
                                const int q = a0[c] % A.G;
                                v[c] = q < 0 ? q + A.G : q;
                            }
                            atomicAdd(&A.acc[(v[2] * A.G + v[1]) * A.G + v[0]], A.dens[k] * A.cell[k].vol);
                        } else if (mm > GV_BIG) {
                            const unsigned long long o =
                                atomicAdd(&A.ctr->n_big, (1ull << BIG_BITS) + (unsigned long long)((mm + GV_BIG - 1) / GV_BIG));
                            A.big[o >> BIG_BITS] = (uint32_t)k;
                            A.big_unit[o >> BIG_BITS] = o & ((1ull << BIG_BITS) - 1ull);
                        } else {
                            m = (int)mm;
                            for (int c = 0; c < 3; c++) { S.a0[c][lane] = a0[c]; S.n[c][lane] = n[c]; }
                        }
                    }
                    int x = m;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(FULL, x, o);
                        if ((int)lane >= o) x += y;
                    }
                    S.pref[lane + 1] = x;
                    if (lane == 0) S.pref[0] = 0;
                    total = __shfl_sync(FULL, x, 31);
                    t1 = 0;
                }
            }
            __syncwarp();
        }
        if (t1 < total) {
            const int64_t t = t1 + lane;
            int cross = -1;
            int4 ent = make_int4(0, 0, 0, 0);
            if (t < total) {
                int c = 0, i = (int)t;
                if (!BIG) {
                    // the cell of pair t: the last with pref <= t
#pragma unroll
                    for (int o = 16; o; o >>= 1)
                        if (S.pref[c + o] <= (int)t) c += o;
                    i -= S.pref[c];
                }
                const int n0 = S.n[0][c], n1 = S.n[1][c];
                const int ia[3] = {S.a0[0][c] + i % n0, S.a0[1][c] + (i / n0) % n1, S.a0[2][c] + i / (n0 * n1)};
                const uint32_t k = b + (uint32_t)c;
                const P pi = spos[k];
                const double xi[3] = {(double)pi.x, (double)pi.y, (double)pi.z};
                float lo[3], hi[3];
                const int64_t vi = voxel_box(A, xi, A.rad[k] * (1.f + 4e-6f), ia, lo, hi);
                cross = side_of_box(A, A.face_start[k], A.face_count[k], lo, hi);
                if (cross == 0) atomicAdd(&A.acc[vi], A.dens[k] * vox);
                ent = make_int4((int)k, ia[0], ia[1], ia[2]);
            }
            const int cls = cross <= 0 ? -1 : cross <= 2 ? 0 : cross <= 5 ? 1 : cross <= 10 ? 2 : 3;
#pragma unroll
            for (int c = 0; c < GV_CLASSES; c++) {
                const unsigned cm = __ballot_sync(FULL, cls == c);
                if (cls == c) S.q[c][nq[c] + __popc(cm & lt)] = ent;
                nq[c] += __popc(cm);
            }
            t1 += 32;
            __syncwarp();
        }
        // ---------------------------------------------------------------- eight pairs of a class, while one is full
        bool idle = true;
#pragma unroll 1
        for (;;) {
            int cl = -1, m = 0;
#pragma unroll
            for (int c = 0; c < GV_CLASSES; c++)
                if (nq[c] >= 32 || (!more && t1 >= total && nq[c] > 0)) { cl = c; m = nq[c]; }
            if (cl < 0) break;
            idle = false;
            const int take = m < W ? m : W;
            const bool has = gsh / G < take;
            const int4 ent = S.q[cl][has ? m - take + gsh / G : 0];
#pragma unroll
            for (int c = 0; c < GV_CLASSES; c++)
                if (c == cl) nq[c] -= take;
            const uint32_t k = (uint32_t)ent.x, st = A.face_start[k];
            const int cnt = has ? (int)A.face_count[k] : 0;
            float lo[3], hi[3];
            int64_t vi;
            {
                const P pi = spos[k];
                const double xi[3] = {(double)pi.x, (double)pi.y, (double)pi.z};
                const int ia[3] = {ent.y, ent.z, ent.w};
                vi = voxel_box(A, xi, A.rad[k] * (1.f + 4e-6f), ia, lo, hi);
            }
            // start: the box (walls and corners as in k_group_clip)
            __syncwarp();
#pragma unroll 1
            for (int w = r; w < 6; w += G) {
                const float sg = (w & 1) ? -1.f : 1.f;
                const float h = w == 0 ? hi[0] : w == 1 ? -lo[0] : w == 2 ? hi[1] : w == 3 ? -lo[1] : w == 4 ? hi[2] : -lo[2];
                C.Pl[w] = make_float4(w < 2 ? sg : 0.f, (w >> 1) == 1 ? sg : 0.f, w > 3 ? sg : 0.f, h);
                C.Ps[w] = 0u;
                C.Sq[w] = (uint8_t)w;
            }
#pragma unroll 1
            for (int q = r; q < 8; q += G) {
                const bool even = (__popc((unsigned)q) & 1) == 0;
                const uint32_t X = (q & 1) ? 1 : 0, Y = (q & 2) ? 3 : 2, Z = (q & 4) ? 5 : 4;
                C.V[q] = make_float4((q & 1) ? lo[0] : hi[0], (q & 2) ? lo[1] : hi[1], (q & 4) ? lo[2] : hi[2],
                                     pack_w(0.f, pack_ids(X, even ? Y : Z, even ? Z : Y)));
                const uint32_t fx = (uint32_t)q ^ 1u, fy = (uint32_t)q ^ 2u, fz = (uint32_t)q ^ 4u;
                C.Ad[q] = even ? (fz | (fx << 8) | (fy << 16)) : (fy | (fx << 8) | (fz << 16));
            }
            unsigned vlo = has ? 0xffu : 0u, vhi = 0u;
            int np = 6, nseq = 6, fail = 0;
            bool empty = !has;
            __syncwarp();
            // the planes in batches of G, one per lane, as in k_group_clip
#pragma unroll 1
            for (int base = 0;; base += G) {
                const bool open = !fail && !empty && base < cnt;
                if (!__any_sync(FULL, open)) break;
                float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
                bool on = open && base + r < cnt;
                if (on) {
                    f = *reinterpret_cast<const float4*>(&A.faces[st + base + r]);
                    f.w = 0.5f * __fmaf_rn(f.z, f.z, __fmaf_rn(f.y, f.y, f.x * f.x));
                    on = fmaxf(f.x * lo[0], f.x * hi[0]) + fmaxf(f.y * lo[1], f.y * hi[1]) + fmaxf(f.z * lo[2], f.z * hi[2]) > f.w;
                }
                if (!__any_sync(FULL, on)) continue;
                unsigned olo = 0u, ohi = 0u;
                const int hw = open ? (vhi ? 64 - __clz(vhi) : 32 - __clz(vlo)) : 0;
                const int hmax = __reduce_max_sync(FULL, hw);
#pragma unroll 1
                for (int s0 = 0; s0 < hmax; s0 += 4) {
                    unsigned o4 = 0u;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const float4 v = C.V[s0 + q];
                        if (f_fma<float>(f.x, v.x, f_fma<float>(f.y, v.y, f_fma<float>(f.z, v.z, -f.w))) > 0.f) o4 |= 1u << q;
                    }
                    if (s0 < 32) olo |= o4 << s0;
                    else ohi |= o4 << (s0 - 32);
                }
                olo = on ? olo & vlo : 0u;
                ohi = on ? ohi & vhi : 0u;
#pragma unroll 1
                for (;;) {
                    const unsigned cm = gballot((olo | ohi) != 0u);
                    bool cut = open && !fail && !empty && cm != 0u;
                    if (!__any_sync(FULL, cut)) break;
                    const int src = gsh + (cut ? __ffs(cm) - 1 : 0);
                    unsigned rem0 = __shfl_sync(FULL, olo, src), rem1 = __shfl_sync(FULL, ohi, src);
                    if (cut && rem0 == vlo && rem1 == vhi) {  // nothing is left
                        empty = true;
                        cut = false;
                    }
                    unsigned w0, w1;
                    group_cut<G, true>(C, cut, src, rem0, rem1, f, 0u, vlo, vhi, np, nseq, fail, w0, w1);
                    __syncwarp();
                    olo &= ~rem0; ohi &= ~rem1;
                    if ((int)lane <= src || !cut) olo = ohi = 0u;
                    const bool later = on && cut && (int)lane > src;
                    unsigned m0 = cut ? w0 : 0u, m1 = cut ? w1 : 0u;
#pragma unroll 1
                    while (__any_sync(FULL, (m0 | m1) != 0u)) {
                        const int s = m0 ? __ffs(m0) - 1 : m1 ? 31 + __ffs(m1) : 0;
                        if (m0) m0 &= m0 - 1u; else m1 &= m1 - 1u;
                        const float4 v = C.V[s];
                        if (later && f_fma<float>(f.x, v.x, f_fma<float>(f.y, v.y, f_fma<float>(f.z, v.z, -f.w))) > 0.f) {
                            if (s < 32) olo |= 1u << s; else ohi |= 1u << (s - 32);
                        }
                    }
                }
            }
            // the volume from the edges: the edge a->b of a vertex leads to the vertex across it and bounds the face of
            // plane b, so a face's area is the sum of n.(w x w') / 2 over its edges, w relative to the mean vertex, and
            // the volume a third of offset times area
            const bool on = has && !fail && !empty;
            float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll 1
            for (int s = r; s < GNT; s += G)
                if (on && in_set(vlo, vhi, (uint32_t)s)) {
                    const float4 v = C.V[s];
                    sx += v.x; sy += v.y; sz += v.z;
                }
            const float im = 1.f / (float)max(1, __popc(vlo) + __popc(vhi));
            const float mx = gsum(sx) * im, my = gsum(sy) * im, mz = gsum(sz) * im;
            float vol = 0.f;
#pragma unroll 1
            for (int s = r; s < GNT; s += G)
                if (on && in_set(vlo, vhi, (uint32_t)s)) {
                    const float4 v = C.V[s];
                    const float ax = v.x - mx, ay = v.y - my, az = v.z - mz;
                    uint32_t id[3];
                    ids_of(v.w, id[0], id[1], id[2]);
                    const uint32_t ad = C.Ad[s];
#pragma unroll
                    for (int q = 0; q < 3; q++) {
                        const float4 o = C.V[(ad >> (8 * q)) & 63u];
                        const uint32_t y = id[q == 2 ? 0 : q + 1];
                        const float4 p = C.Pl[y];
                        const float bx = o.x - mx, by = o.y - my, bz = o.z - mz;
                        const float off = p.w - (p.x * mx + p.y * my + p.z * mz);
                        const float cr = p.x * (ay * bz - az * by) + p.y * (az * bx - ax * bz) + p.z * (ax * by - ay * bx);
                        vol += y < 6 ? off * cr : off * cr / (2.f * p.w);
                    }
                }
            vol = gsum(vol) / 6.f;  // (a sixth as a float is 3e-8 too large)
            if (r == 0 && has) {
                // a sliver's FP32 volume may come out slightly below zero; anything beyond 1e-5 of the box is a failure
                if (fail || (on && vol < -1e-5f * (hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2])))
                    push_retry(A, (int64_t)k, ent.y, ent.z, ent.w);
                else if (on && vol > 0.f) atomicAdd(&A.acc[vi], A.dens[k] * (double)vol);
            }
            __syncwarp();
        }
        if (!more && t1 >= total && idle) break;
    }
}

template <typename P, bool BIG>
void launch_voxels(const GridArgs& a, int sm_count, cudaStream_t s) {
    static int per_sm_dev[64] = {0};
    const size_t smem = 8 * sizeof(GCell) + sizeof(GridWarp);
    const int per_sm = blocks_per_sm(k_group_voxels<P, BIG>, 32, smem, per_sm_dev);
    k_group_voxels<P, BIG><<<(unsigned)(sm_count * per_sm), 32, smem, s>>>(a);
}
}  // namespace

int launch_clip_group(const ClipArgs& a, const GroupBuf& b, int dtype, int lanes, int sm_count, cudaStream_t s) {
    if (dtype == VT_F32) {
        if (lanes == 4) return a.sset ? launch_group<float4, 4, true>(a, b, sm_count, s) : launch_group<float4, 4, false>(a, b, sm_count, s);
        return a.sset ? launch_group<float4, 8, true>(a, b, sm_count, s) : launch_group<float4, 8, false>(a, b, sm_count, s);
    }
    if (lanes == 4) return a.sset ? launch_group<dpt4, 4, true>(a, b, sm_count, s) : launch_group<dpt4, 4, false>(a, b, sm_count, s);
    return a.sset ? launch_group<dpt4, 8, true>(a, b, sm_count, s) : launch_group<dpt4, 8, false>(a, b, sm_count, s);
}

int launch_grid_pairs(const GridArgs& a, int dtype, int sm_count, cudaStream_t s) {
    if (dtype == VT_F32) {
        launch_voxels<float4, false>(a, sm_count, s);
        launch_voxels<float4, true>(a, sm_count, s);
    } else {
        launch_voxels<dpt4, false>(a, sm_count, s);
        launch_voxels<dpt4, true>(a, sm_count, s);
    }
    return 2;
}

}  // namespace vt
