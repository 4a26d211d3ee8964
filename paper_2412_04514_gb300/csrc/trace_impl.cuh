// trace_impl.cuh -- stage 3 of the list schedule: whole cells by edge tracing.
//
// The cell of a generator is the intersection of the half-spaces of its walls
// and of the bisectors with its nearest generators (votess paper, Summary).
// Clipping plane by plane builds and discards about four vertices for every
// one that stays, and each cut is a chain of dependent topology updates. Here
// the final polyhedron of the whole list is found at once, vertex by vertex:
// from a vertex (a, b, c) the edge on planes a and b ends at the plane h that
// the ray along it meets first, which is the vertex (b, a, h). The midpoint to
// the nearest generator lies on the cell, so two such rays from it reach a
// first vertex, and every further vertex costs one ray. An edge whose other
// end was met already is closed by a search among the open ends instead of a
// ray, so a cell of V vertices takes V + 1 rays of one plane test per plane.
//
// Work split: 8 lanes build one cell, four cells of a warp in lockstep (every
// warp collective names all 32 lanes; a group that is done idles until the
// others are). Each lane holds every eighth plane in registers; a ray is NR
// plane tests per lane and a minimum over the 8 lanes. Wider groups repeat the
// per-ray bookkeeping on more lanes, narrower ones hold more of the planes and
// of shared memory per warp. Bound by instruction issue (3,000 warp
// instructions per cell of the first round, 3,400 with geometry, 9,100 in all
// against 14,900 of the clipper) and by instruction fetch; the FP64 form by the
// FP64 pipe (77% busy). 1M points on a GB300, cells and walks with neighbours
// against the clipper and its range lists: uniform 17.1 -> 7.1 ms, half in
// clumps 20.2 -> 10.7 ms in the FP32 form, 126 -> 20.5 and 141 -> 27.6 ms in the
// FP64 form.
//
// Certificate. The rays run in float32 and decide nothing by themselves: the
// vertices are solved again from their three planes, and the cell is accepted
// only when every vertex lies inside every other plane by more than the
// float32 error of that test (a bound that grows with the conditioning of the
// vertex) and every edge has both its ends. Such vertices are vertices of the
// exact polyhedron, and a set of them that is closed under its edges is all of
// them, so an accepted topology is the exact one. A cell that fails (vertices
// within round-off of a further plane, ill-conditioned or too many of them) is
// built again by other means, in the end by the plane-by-plane clipper with its
// FP64 rechecks. The bounds hold while squares of lengths are normal float32
// numbers: a cell with a generator or a vertex closer than 1e-18 to its own
// generator fails too, and one with a vertex whose products of three normals
// leave 1e-25..1e25 goes to the warp per cell, which solves it in FP64.
//
// Security radius. A cell whose 4 R^2 is within the list's reach is final.
// Otherwise its results are written all the same and a second kernel (a warp
// per cell) walks the generators beyond the list and within 2R, row by row of
// the grid: one that cuts no vertex changes nothing, so without a cutting
// generator the results stand. The other cells are built again from their
// faces and the nearest cutting generators, once more by groups of 8 lanes and
// then, with the cells that failed, by a warp per cell that rebuilds and walks
// until nothing cuts. That kernel holds more planes, vertices and open edges
// and solves more vertices in FP64; what its certificate refuses too goes to
// the plane-by-plane clipper.
#pragma once
#include "clip_impl.cuh"

namespace vt {

namespace {

constexpr unsigned TFULL = 0xffffffffu;
constexpr int TRACE_KEEP = 12;     // cutting generators handed to the next round
constexpr int PAD_PLANE = INT_MIN;

// A vertex is known to VERT_ERR |v|: float32 at the smallest |det| that the FP32
// form solves in float32 (UNIT_F64), rounding included. Whatever decides which
// generators can still cut a vertex allows for it: the true vertex v' has
// |v'| <= (1 + VERT_ERR) |v|, and the ball of its cutting generators, of radius
// |v'| around v', lies in the ball of (1 + 2 VERT_ERR) |v| around v. (Factors on
// squares; 1e-5 more covers the rounding of the comparisons.)
constexpr float UNIT_F64 = 1e-2f;
constexpr float VERT_ERR0 = 1e-6f, VERT_ERR1 = 1.5e-6f;  // VERT_ERR0 + VERT_ERR1 / |det|
constexpr float VERT_ERR = VERT_ERR0 + VERT_ERR1 / UNIT_F64;
constexpr float FAR_R2 = (1.0f + VERT_ERR) * (1.0f + VERT_ERR) + 1e-5f;
constexpr float FAR_BALL = 1.0f + 2.0f * VERT_ERR + 5e-6f;

// groups of TT lanes of a warp in lockstep
template <int TT>
struct Sub {
    int lane, gl, base, gi;
    __device__ __forceinline__ Sub()
    {
        lane = threadIdx.x & 31;
        gl = lane & (TT - 1);
        base = lane & ~(TT - 1);
        gi = lane / TT;
    }
    __device__ __forceinline__ unsigned ballot(bool p) const
    {
        const unsigned b = __ballot_sync(TFULL, p);
        return TT == 32 ? b : (b >> base) & ((1u << (TT & 31)) - 1u);
    }
    __device__ __forceinline__ bool any(bool p) const { return ballot(p) != 0; }
    template <typename V>
    __device__ __forceinline__ V bcast(V v, int src) const { return __shfl_sync(TFULL, v, src, TT); }
    __device__ __forceinline__ float max(float v) const
    {
#pragma unroll
        for (int o = TT / 2; o >= 1; o >>= 1) v = fmaxf(v, __shfl_xor_sync(TFULL, v, o));
        return v;
    }
    __device__ __forceinline__ int incl_scan(int v) const
    {
#pragma unroll
        for (int d = 1; d < TT; d <<= 1) {
            const int u = __shfl_up_sync(TFULL, v, d, TT);
            if (gl >= d) v += u;
        }
        return v;
    }
};

// reciprocal, square root and its reciprocal to 1e-6 or better, flushing
// denormals: the tests' margins cover them, no result is formed from them
__device__ __forceinline__ float rcp_fast(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_fast(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_fast(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// positions and planes in the arithmetic of the results. The FP32 form solves
// and integrates with the float planes; the FP64 form keeps double planes and
// positions beside the float ones that the tests use.
template <typename Real, int NP, int NV>
struct TraceReal {};
template <int NP, int NV>
struct TraceReal<double, NP, NV> {
    double pn[NP][3];  // n
    double ps[NP];     // b / |n|^2
    double v[NV][3];
};

// shared memory of a group: NP planes, NV vertices
template <typename Real, int NP, int NV>
struct alignas(16) TraceSmem : TraceReal<Real, NP, NV> {
    float4 pl[NP];       // n, b of n.x <= b
    float4 vp[NV];       // position; a bound of its error and that of a plane test, as a length
    int32_t src[NP];     // sorted index (with image code), -1..-6 walls, PAD_PLANE
    uint8_t vid[NV][4];  // planes (ccw from outside)
    // edges: planes a | b << 8, vertices s << 16 | t << 24; (a, b) follow one
    // another in vid[s], so s -> t runs ccw around b and t -> s around a
    uint32_t ed[3 * NV / 2];
    union {
        float nl[NP];    // |n| (until the vertices are solved)
        int32_t f[NP];   // the finish: each plane's area sum, then the faces' neighbour keys
    } u;
};
// stride of a group's block: the four groups of a warp read the same member
// at once (float4 broadcasts), so their blocks start 32 bytes apart modulo the
// 128 bytes of the banks
template <typename S>
constexpr size_t trace_stride()
{
    return (sizeof(S) + 95) / 128 * 128 + 32;
}

// FP64 position of the vertex of three planes (out of line: rarely needed)
template <bool PER>
__device__ VT_RARE bool solve_vertex64(int a, int b, int c, const float4* __restrict__ sorted, float4 pi,
                                       const GridDesc& grid, double& x, double& y, double& z)
{
    x = y = z = 0.0;
    return vertex64(plane64<PER>(a, sorted, pi, grid), plane64<PER>(b, sorted, pi, grid),
                    plane64<PER>(c, sorted, pi, grid), x, y, z);
}
// |det| of the unit normals of three planes of any scale
__device__ VT_RARE float unit_det(float4 p, float4 o, float4 h)
{
    const double bcx = (double)o.y * h.z - (double)o.z * h.y, bcy = (double)o.z * h.x - (double)o.x * h.z,
                 bcz = (double)o.x * h.y - (double)o.y * h.x;
    const double pp = (double)p.x * p.x + (double)p.y * p.y + (double)p.z * p.z,
                 oo = (double)o.x * o.x + (double)o.y * o.y + (double)o.z * o.z,
                 hh = (double)h.x * h.x + (double)h.y * h.y + (double)h.z * h.z;
    return (float)(fabs(p.x * bcx + p.y * bcy + p.z * bcz) / (sqrt(pp) * sqrt(oo) * sqrt(hh)));
}
// of the planes (n, b) that the ray v + t d meets at float keys of t below `below`, the
// first in FP64 (by a warp; out of line: rarely needed)
__device__ VT_RARE int hit_order64(const double (*pd)[4], const float* nl, int rows, double vx, double vy, double vz,
                                   double dx, double dy, double dz, float least, uint32_t below)
{
    const int lane = threadIdx.x & 31;
    double best = DBL_MAX;
    int plane = -1;
    for (int r = 0; r < rows; ++r) {
        const int p = r * 32 + lane;
        const double s = pd[p][3] - ((pd[p][0] * vx + pd[p][1] * vy) + pd[p][2] * vz);
        const double nd = (pd[p][0] * dx + pd[p][1] * dy) + pd[p][2] * dz;
        const bool near = (float)nd > least * nl[p] && __float_as_uint((float)s * rcp_fast((float)nd)) < below;
        const double t = near ? s / nd : DBL_MAX;
        if (t < best) {
            best = t;
            plane = p;
        }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        const double t = __shfl_xor_sync(TFULL, best, o);
        const int p = __shfl_xor_sync(TFULL, plane, o);
        if (t < best || (t == best && p < plane)) {
            best = t;
            plane = p;
        }
    }
    return plane;
}
// the low halves of a position in FP64 beside its float32 value
__device__ __forceinline__ float4 low_half(double x, double y, double z)
{
    return make_float4((float)(x - (double)(float)x), (float)(y - (double)(float)y), (float)(z - (double)(float)z), 0.0f);
}

// a set of planes
template <int W>
struct Faces {
    uint32_t w[W];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int i = 0; i < W; ++i) w[i] = 0;
    }
    __device__ __forceinline__ void add(int p)
    {
#pragma unroll
        for (int i = 0; i < W; ++i) w[i] |= p >> 5 == i ? 1u << (p & 31) : 0u;
    }
    __device__ __forceinline__ int count() const
    {
        int c = 0;
#pragma unroll
        for (int i = 0; i < W; ++i) c += __popc(w[i]);
        return c;
    }
    // the n-th (0-based) of them
    __device__ __forceinline__ int nth(int n) const
    {
        int at = 0;
        uint32_t x = w[0];
#pragma unroll
        for (int i = 1; i < W; ++i) {
            const int c = __popc(x);
            if (n >= c && at == 32 * (i - 1)) {
                n -= c;
                at = 32 * i;
                x = w[i];
            }
        }
        return at + nth_bit32(x, n);
    }
};

// mask of a group's open edge ends
template <int TT>
struct LiveMask {
    using T = uint32_t;
};
template <>
struct LiveMask<32> {
    using T = uint64_t;
};
__device__ __forceinline__ int lowest(uint32_t x) { return __ffs(x) - 1; }
__device__ __forceinline__ int lowest(uint64_t x) { return __ffsll((long long)x) - 1; }

// One cell per group of TT lanes: its planes (unit normals in registers, plane
// r * TT + lane in row r), then its polyhedron in shared memory. Every member
// is called by the whole warp; groups without work pass through.
template <typename Real, int TT, int NR, int NV, bool PER>
struct Tracer {
    static constexpr int NP = NR * TT;
    static constexpr bool F64 = sizeof(Real) == 8;
    static constexpr int NE = 3 * NV / 2;
    using S = TraceSmem<Real, NP, NV>;
    // smallest |det| of a vertex's three unit normals, above the rounding of the
    // rates of approach in float32, and in FP64. Both forms take the same for the
    // rays: the FP32 form solves such vertices in FP64 (UNIT_F64), and at 2e-4 the
    // sliver-cornered cells beside clumps, traced again with FP64 rays a warp each,
    // were the last to finish (500 points in clumps 0.63 -> 0.33 ms, 15,000 1.32 ->
    // 0.90 ms, periodic 2.80 -> 1.72 ms)
    static constexpr float UNIT_MIN = 2e-5f, UNIT_MIN64 = 1e-7f;
    // (below UNIT_F64 the FP32 form solves a vertex in FP64, about 1 in 3,000)
    static constexpr float UNIT_F64 = vt::UNIT_F64;
    static constexpr float REGULAR = 2e-6f;
    static constexpr double TIE = 1e-13;             // of |n| |v|: FP64 does not tell the plane from the vertex
    static constexpr int SR = 2;                     // registers of open edge ends per lane
    using Live = typename LiveMask<TT>::T;           // a bit per slot; the top bit takes the edges that closed
    static constexpr int TOP = 8 * sizeof(Live) - 1;
    static constexpr int SLOTS = SR * TT < TOP ? SR * TT : TOP;

    float nx[NR], ny[NR], nz[NR], nb[NR];
    int rows;               // rows of planes in use over the warp
    bool ok;
    int V, E;
    DevStatus* st;          // (the debug build's index checks)
    // indices that come from data: a plane, a vertex, an edge
    __device__ __forceinline__ int plane_ck(int p) const { return vt_ck(p, NP, CK_PLANE, st); }
    __device__ __forceinline__ int vertex_ck(int s) const { return vt_ck(s, NV, CK_SLOT, st); }
    __device__ __forceinline__ int edge_ck(int e) const { return vt_ck(e, NE, CK_EDGE, st); }
    float R2;               // max |v|^2
    Faces<(NP + 31) / 32> faces;  // the planes that are faces

    // squares below this lose digits in float32: a cell with such a vertex, or
    // whose first generator, the nearest of its lists, is so close, fails
    static constexpr float SQUARE_MIN = 1e-36f;
    static __device__ __forceinline__ bool in_range(const S& sm, int f0) { return sm.pl[f0].w >= 0.5f * SQUARE_MIN; }

    // plane row r of the lane from its source
    __device__ __forceinline__ void set_plane(S& sm, int r, int p, int src, float4 pi, const GridDesc& grid,
                                              const float4* __restrict__ sorted)
    {
        float x = 0.0f, y = 0.0f, z = 0.0f, b = 1.0f, len = 0.0f, inv = 0.0f;
        if (src >= 0) {
            const float3 o = img_off_t<PER>(pi, sorted[img_index_t<PER>(src)], img_code_t<PER>(src), grid);
            x = o.x;
            y = o.y;
            z = o.z;
            const float nn = x * x + y * y + z * z;
            b = 0.5f * nn;
            len = sqrt_fast(nn);
            inv = rsqrt_fast(nn);
        } else if (src != PAD_PLANE) {
            const int w = -src - 1, axis = w >> 1, upper = w & 1;
            const float one = upper ? 1.0f : -1.0f;
            x = axis == 0 ? one : 0.0f;
            y = axis == 1 ? one : 0.0f;
            z = axis == 2 ? one : 0.0f;
            const float pc = axis == 0 ? pi.x : (axis == 1 ? pi.y : pi.z);
            b = PER ? (float)(0.5 * ((double)grid.hi[axis] - (double)grid.lo[axis]))
                    : (upper ? grid.hi[axis] - pc : pc - grid.lo[axis]);
            len = inv = 1.0f;
        }
        nx[r] = x * inv;
        ny[r] = y * inv;
        nz[r] = z * inv;
        nb[r] = src != PAD_PLANE ? b * inv : FLT_MAX;
        sm.pl[p] = make_float4(x, y, z, b);
        sm.u.nl[p] = len;
        sm.src[p] = src;
        if constexpr (F64) {
            if (src != PAD_PLANE) {
                const P64 d = plane64<PER>(src, sorted, pi, grid);
                sm.pn[p][0] = d.x;
                sm.pn[p][1] = d.y;
                sm.pn[p][2] = d.z;
                sm.ps[p] = src >= 0 ? 0.5 : d.b;  // b / |n|^2
            }
        }
    }

    template <int N>
    __device__ __forceinline__ uint32_t hit_rows(float vx, float vy, float vz, float dx, float dy, float dz,
                                                 float least) const
    {
        uint32_t key = 0xffffffffu;
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const float s = fmaf(-nx[r], vx, fmaf(-ny[r], vy, fmaf(-nz[r], vz, nb[r])));
            const float nd = fmaf(nx[r], dx, fmaf(ny[r], dy, nz[r] * dz));
            const uint32_t k = (__float_as_uint(s * rcp_fast(nd)) & ~63u) | (uint32_t)(r * TT);
            key = nd > least ? ::min(key, k) : key;
        }
        return key;
    }
    // the ray v + t d against the planes (unit normals): the first plane met, -1
    // when none is. A plane counts when the ray closes in on it faster than
    // `least`, which leaves out the planes that hold the ray (their rate is
    // round-off) together with those whose vertex would be too ill-conditioned.
    // Groups of 8 lanes carry the plane index in the low six bits of t, which
    // orders hits that agree to 8e-6 by index: the certificate refuses the wrong
    // ones. A warp per cell compares all of t. Two unrolled forms of the former:
    // the lists fill all rows, most later rounds three.
    __device__ __forceinline__ int first_hit(const Sub<TT>& G, float vx, float vy, float vz, float dx, float dy, float dz,
                                             float least) const
    {
        if constexpr (TT == 32) {
            uint32_t key = 0xffffffffu;
            int row = 0;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const float s = fmaf(-nx[r], vx, fmaf(-ny[r], vy, fmaf(-nz[r], vz, nb[r])));
                const float nd = fmaf(nx[r], dx, fmaf(ny[r], dy, nz[r] * dz));
                const uint32_t k = __float_as_uint(s * rcp_fast(nd));
                const bool take = nd > least && k < key;
                key = take ? k : key;
                row = take ? r : row;
            }
            const uint32_t first = __reduce_min_sync(TFULL, key);
            const int lane = __ffs(__ballot_sync(TFULL, key == first)) - 1;
            row = __shfl_sync(TFULL, row, lane);
            return first < 0x7f800000u ? row * TT + lane : -1;
        } else {
            uint32_t key;
            if (NR > 3 && rows <= 3) key = hit_rows<(NR > 3 ? 3 : NR)>(vx, vy, vz, dx, dy, dz, least);
            else key = hit_rows<NR>(vx, vy, vz, dx, dy, dz, least);
            key |= (uint32_t)G.gl;
#pragma unroll
            for (int o = TT / 2; o >= 1; o >>= 1) key = ::min(key, __shfl_xor_sync(TFULL, key, o));
            return key < 0x7f800000u ? (int)(key & 63u) : -1;
        }
    }

    // the first plane met in FP64 (a warp per cell, its planes (n, b) in pd): for
    // cells whose far walls leave float32 positions too coarse for the near planes.
    // The quotients are float32; planes whose quotients agree to 64 roundings (4e-6)
    // are put in order in FP64. By the float32 order alone a few cells of every
    // million, and 28 of 125,000 of a lattice moved by 1e-3 of its spacing, were
    // refused: each costs the call a list and a range pass (1M half in clumps, FP64
    // form 30.3 -> 30.1 ms, 120,000 2.47 -> 2.43)
    __device__ __forceinline__ int first_hit64(const S& sm, const double (*pd)[4], double vx, double vy, double vz,
                                               double dx, double dy, double dz, float least) const
    {
        const int lane = threadIdx.x & 31;
        uint32_t key = 0xffffffffu, next = 0xffffffffu;
        int row = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int p = r * TT + lane;
            const double* h = pd[p];
            const float s = (float)(h[3] - ((h[0] * vx + h[1] * vy) + h[2] * vz));
            const float nd = (float)((h[0] * dx + h[1] * dy) + h[2] * dz);
            const uint32_t k = __float_as_uint(s * rcp_fast(nd));
            const bool meets = nd > least * sm.u.nl[p], take = meets && k < key;  // (no plane: nd = 0)
            next = take ? key : (meets && k < next ? k : next);
            key = take ? k : key;
            row = take ? r : row;
        }
        const uint32_t first = __reduce_min_sync(TFULL, key);
        const int from = __ffs(__ballot_sync(TFULL, key == first)) - 1;
        row = __shfl_sync(TFULL, row, from);
        // another plane within the rounding of these quotients: their order in FP64
        if (first < 0x7f800000u && __any_sync(TFULL, next < first + 64u || (key < first + 64u && lane != from)))
            return hit_order64(pd, sm.u.nl, NR, vx, vy, vz, dx, dy, dz, least, first + 64u);
        return first < 0x7f800000u ? row * TT + from : -1;
    }

    // vertices (as triples of planes) and edges, one ray per vertex. f0: the
    // plane of the nearest generator; on: the group has a cell. W: the rays'
    // arithmetic (double: a warp per cell, its planes in pd; lo holds the low
    // halves of the positions)
    template <typename W>
    __device__ __forceinline__ void trace(const Sub<TT>& G, S& sm, bool on, int f0, const double (*pd)[4], float4* lo)
    {
        constexpr bool DBL = sizeof(W) == 8;
        constexpr float LEAST = DBL ? UNIT_MIN64 : UNIT_MIN;
        const int gl = G.gl;
        ok = on;
        V = 1;
        E = 0;
        int o[SR];  // open edge ends (an edge of ed without its second vertex; -1: free)
#pragma unroll
        for (int i = 0; i < SR; ++i) o[i] = -1;
        auto plane = [&](int p, W& x, W& y, W& z, W& b) {
            if constexpr (DBL) {
                x = pd[p][0];
                y = pd[p][1];
                z = pd[p][2];
                b = pd[p][3];
            } else {
                const float4 h = sm.pl[p];
                x = h.x;
                y = h.y;
                z = h.z;
                b = h.w;
            }
        };
        auto hit_of = [&](W vx, W vy, W vz, W dx, W dy, W dz, float least) {
            if constexpr (DBL) return first_hit64(sm, pd, vx, vy, vz, dx, dy, dz, least);
            else return first_hit(G, vx, vy, vz, dx, dy, dz, least);
        };
        // v + t d on plane h
        auto advance = [&](W& vx, W& vy, W& vz, W dx, W dy, W dz, int h) {
            W hx, hy, hz, hb;
            plane(h, hx, hy, hz, hb);
            const W s = hb - (hx * vx + hy * vy + hz * vz), nd = hx * dx + hy * dy + hz * dz;
            W t;
            if constexpr (DBL) {  // (one Newton step from float32: 1e-13)
                const double r = rcp_fast((float)nd);
                t = s * r;
                t += (s - t * nd) * r;
            } else {
                t = s * rcp_fast(nd);
            }
            vx += t * dx;
            vy += t * dy;
            vz += t * dz;
        };
        auto put = [&](int s, W x, W y, W z) {
            sm.vp[s] = make_float4((float)x, (float)y, (float)z, 0.0f);
            if constexpr (DBL) lo[s] = low_half(x, y, z);
        };
        {
            W n0x, n0y, n0z, n0b;
            plane(f0, n0x, n0y, n0z, n0b);
            W vx = (W)0.5 * n0x, vy = (W)0.5 * n0y, vz = (W)0.5 * n0z;
            // a direction in plane f0: n0 x the axis it is least along
            const W ax = n0x < 0 ? -n0x : n0x, ay = n0y < 0 ? -n0y : n0y, az = n0z < 0 ? -n0z : n0z;
            W dx, dy, dz;
            if (ax <= ay && ax <= az) { dx = 0; dy = n0z; dz = -n0y; }
            else if (ay <= az) { dx = -n0z; dy = 0; dz = n0x; }
            else { dx = n0y; dy = -n0x; dz = 0; }
            int f1 = f0, h = f0;
#pragma unroll 1
            for (int e = 0; e < 2; ++e) {
                // (the second ray runs along f0 and f1: n0 x n1 ends at (f0, f1, h))
                const int hit = hit_of(vx, vy, vz, dx, dy, dz,
                                       e == 0 ? 1e-3f * sm.u.nl[f0] : LEAST * sm.u.nl[f0] * sm.u.nl[f1]);
                ok = ok && hit >= 0;
                h = plane_ck(ok ? hit : f0);
                advance(vx, vy, vz, dx, dy, dz, h);
                if (e == 0) {
                    f1 = h;
                    W hx, hy, hz, hb;
                    plane(h, hx, hy, hz, hb);
                    dx = n0y * hz - n0z * hy;
                    dy = n0z * hx - n0x * hz;
                    dz = n0x * hy - n0y * hx;
                }
            }
            if (gl == 0) {
                put(0, vx, vy, vz);
                *reinterpret_cast<uint32_t*>(sm.vid[0]) = (uint32_t)f0 | ((uint32_t)f1 << 8) | ((uint32_t)h << 16);
            }
            if (gl == 0) o[0] = f0 | (f1 << 8);
            if (gl == 1) o[0] = f1 | (h << 8);
            if (gl == 2) o[0] = h | (f0 << 8);
        }
        Live live = 7u;
        __syncwarp();
        bool run = ok;
#pragma unroll 1
        while (__any_sync(TFULL, run)) {
            // the lowest slot: new ends take the lowest free ones, so the newest go
            // first (oldest first leaves more ends open: 1.7% of the cells of
            // uniform points ran out of 16 slots, against 0.4%)
            const int slot = lowest(live);
            const int got = G.bcast(slot < TT ? o[0] : o[1], slot & (TT - 1));
#pragma unroll
            for (int i = 0; i < SR; ++i) o[i] = gl + i * TT == slot ? -1 : o[i];
            const int ent = run ? got : 0;
            const int a = plane_ck(ent & 0xff), b = plane_ck((ent >> 8) & 0xff), w = vertex_ck(ent >> 16);
            W vx, vy, vz, ax, ay, az, bx, by, bz, unused;
            {
                const float4 v = sm.vp[w];
                vx = v.x;
                vy = v.y;
                vz = v.z;
                if constexpr (DBL) {
                    vx += (double)lo[w].x;
                    vy += (double)lo[w].y;
                    vz += (double)lo[w].z;
                }
            }
            plane(a, ax, ay, az, unused);
            plane(b, bx, by, bz, unused);
            // the edge on a and b leaves (a, b, c) along n_b x n_a
            const W dx = by * az - bz * ay, dy = bz * ax - bx * az, dz = bx * ay - by * ax;
            const int hit = hit_of(vx, vy, vz, dx, dy, dz, LEAST * sm.u.nl[a] * sm.u.nl[b]);
            if (hit < 0 || V >= NV || E > NE - 3) {
                ok = ok && !run;
                run = false;
            }
            const int h = plane_ck(run ? hit : 0);
            advance(vx, vy, vz, dx, dy, dz, h);
            // the vertex (b, a, h): its other two edges, (a, h) and (h, b), close
            // against an open end of the same edge, (h, a) or (b, h), or stay open
            const int k1 = run ? h | (a << 8) : 0xfffe, k2 = run ? b | (h << 8) : 0xfffe;
            bool m1 = false, m2 = false;
#pragma unroll
            for (int i = 0; i < SR; ++i) {
                m1 = m1 || (o[i] & 0xffff) == k1;
                m2 = m2 || (o[i] & 0xffff) == k2;
            }
            const bool c1 = G.any(m1), c2 = G.any(m2);
#pragma unroll
            for (int i = 0; i < SR; ++i) {
                const int k = o[i] & 0xffff;
                if (k == k1 || k == k2) {
                    sm.ed[edge_ck(E + (k == k1 ? 1 : 1 + c1))] = (uint32_t)o[i] | ((uint32_t)V << 24);
                    o[i] = -1;
                }
            }
            live = (Live)G.ballot(o[0] >= 0) | ((Live)G.ballot(o[1] >= 0) << TT);
            if (run) {
                if (gl == 0) {
                    put(vertex_ck(V), vx, vy, vz);
                    *reinterpret_cast<uint32_t*>(sm.vid[V]) = (uint32_t)b | ((uint32_t)a << 8) | ((uint32_t)h << 16);
                    sm.ed[edge_ck(E)] = (uint32_t)ent | ((uint32_t)V << 24);
                }
                // the lowest free slots take what stays open (an edge that closed: no slot)
                const Live free1 = ~live, free2 = c1 ? free1 : free1 & (free1 - 1u);
                const int s1 = c1 ? -1 : lowest(free1), s2 = c2 ? -1 : lowest(free2);
#pragma unroll
                for (int i = 0; i < SR; ++i) {
                    const int at = gl + i * TT;
                    o[i] = at == s1 ? a | (h << 8) | (V << 16) : (at == s2 ? h | (b << 8) | (V << 16) : o[i]);
                }
                if ((!c1 && s1 >= SLOTS) || (!c2 && (unsigned)s2 >= (unsigned)SLOTS)) {
                    ok = run = false;
                    E = NE;  // (see outgrown)
                }
                live = (live | ((Live)1 << (s1 & TOP)) | ((Live)1 << (s2 & TOP))) & (((Live)1 << SLOTS) - 1u);
                E += 1 + c1 + c2;
                ++V;
                run = run && live != 0;
            }
            __syncwarp();
        }
    }

    // whether the polyhedron that failed had more vertices or open edges than there are places
    __device__ __forceinline__ bool outgrown() const { return V >= NV || E > NE - 3; }

    // the vertices from their planes (in the arithmetic of the form), R, the faces
    __device__ __forceinline__ void solve(const Sub<TT>& G, S& sm, float4 pi, const GridDesc& grid,
                                          const float4* __restrict__ sorted, float unit_f64, float unit_min,
                                          float4* lo = nullptr)
    {
        R2 = 0.0f;
        faces.clear();
#pragma unroll 1
        for (int s = G.gl; s < V; s += TT) {
            const uint32_t ids = *reinterpret_cast<const uint32_t*>(sm.vid[s]);
            const int a = plane_ck(ids & 0xff), b = plane_ck((ids >> 8) & 0xff), c = plane_ck((ids >> 16) & 0xff);
            faces.add(a);
            faces.add(b);
            faces.add(c);
            const float4 p = sm.pl[a], o = sm.pl[b], h = sm.pl[c];
            const float bcx = o.y * h.z - o.z * h.y, bcy = o.z * h.x - o.x * h.z, bcz = o.x * h.y - o.y * h.x;
            const float det = p.x * bcx + p.y * bcy + p.z * bcz;
            // |det| of the unit normals: the vertex moves by (rounding) / this
            const float len = sm.u.nl[a] * sm.u.nl[b] * sm.u.nl[c];
            float unit = fabsf(det) * rcp_fast(len);
            // terms of the determinant or of the position leave float32's range (at
            // unit >= UNIT_F64): for the warp per cell, which solves them in FP64
            const bool far_scale = __float_as_uint(len) - __float_as_uint(1e-25f) >
                                   __float_as_uint(1e25f) - __float_as_uint(1e-25f);
            if (TT == 32 && far_scale) unit = unit_det(p, o, h);
            if (!(unit > unit_min) || (TT < 32 && far_scale)) ok = false;
            float x, y, z, err;
            if constexpr (F64) {
                const double ax = sm.pn[a][0], ay = sm.pn[a][1], az = sm.pn[a][2];
                const double bx = sm.pn[b][0], by = sm.pn[b][1], bz = sm.pn[b][2];
                const double cx = sm.pn[c][0], cy = sm.pn[c][1], cz = sm.pn[c][2];
                const double ab = sm.ps[a] * (sm.src[a] < 0 ? 1.0 : (ax * ax + ay * ay) + az * az);
                const double bb = sm.ps[b] * (sm.src[b] < 0 ? 1.0 : (bx * bx + by * by) + bz * bz);
                const double cb = sm.ps[c] * (sm.src[c] < 0 ? 1.0 : (cx * cx + cy * cy) + cz * cz);
                double dx = 0, dy = 0, dz = 0;
                if (!solve3<double>(ax, ay, az, ab, bx, by, bz, bb, cx, cy, cz, cb, dx, dy, dz)) ok = false;
                sm.v[s][0] = dx;
                sm.v[s][1] = dy;
                sm.v[s][2] = dz;
                x = (float)dx;
                y = (float)dy;
                z = (float)dz;
                err = VERT_ERR0;  // float rounding of the position, of the plane and of the test
            } else {
                const float cax = h.y * p.z - h.z * p.y, cay = h.z * p.x - h.x * p.z, caz = h.x * p.y - h.y * p.x;
                const float abx = p.y * o.z - p.z * o.y, aby = p.z * o.x - p.x * o.z, abz = p.x * o.y - p.y * o.x;
                const float inv = rcp(det);
                x = (p.w * bcx + o.w * cax + h.w * abx) * inv;
                y = (p.w * bcy + o.w * cay + h.w * aby) * inv;
                z = (p.w * bcz + o.w * caz + h.w * abz) * inv;
                err = VERT_ERR0 + VERT_ERR1 * rcp_fast(unit);
                if (unit < unit_f64 || (TT == 32 && far_scale)) {  // ill-conditioned: float32 would lose digits
                    double dx, dy, dz;
                    if (!solve_vertex64<PER>(sm.src[a], sm.src[b], sm.src[c], sorted, pi, grid, dx, dy, dz)) ok = false;
                    x = (float)dx;
                    y = (float)dy;
                    z = (float)dz;
                    if (lo) lo[s] = low_half(dx, dy, dz);
                    err = VERT_ERR0;
                }
            }
            const float d = x * x + y * y + z * z;
            if (__float_as_uint(d) - __float_as_uint(SQUARE_MIN) >= 0x7f800000u - __float_as_uint(SQUARE_MIN)) ok = false;
            R2 = fmaxf(R2, d);
            sm.vp[s] = make_float4(x, y, z, TT < 32 && far_scale ? -INFINITY : err * sqrt_fast(d));
        }
        R2 = G.max(R2);
#pragma unroll
        for (int i = 0; i < (NP + 31) / 32; ++i)
#pragma unroll
            for (int o = TT / 2; o >= 1; o >>= 1) faces.w[i] |= __shfl_xor_sync(TFULL, faces.w[i], o);
        __syncwarp();
    }

    // the cell's listed generators within 2R
    __device__ __forceinline__ int listed_within(const Sub<TT>& G, const S& sm) const
    {
        int c = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int p = r * TT + G.gl;
            c += sm.src[p] >= 0 && sm.pl[p].w < 2.0f * R2 ? 1 : 0;
        }
        return G.bcast(G.incl_scan(c), TT - 1);
    }
    // planes of the lane's first N rows closer than thr to v (or behind it)
    template <int N>
    __device__ __forceinline__ int near_rows(float4 v, float thr) const
    {
        int near = 0;
#pragma unroll
        for (int r = 0; r < N; ++r)
            near += fmaf(-nx[r], v.x, fmaf(-ny[r], v.y, fmaf(-nz[r], v.z, nb[r]))) < thr ? 1 : 0;
        return near;
    }
    // every vertex clearly inside all planes but its three, every edge closed
    __device__ __forceinline__ void certify(const Sub<TT>& G, const S& sm)
    {
        int near = 0;
        const int vmax = __reduce_max_sync(TFULL, ok ? V : 0);
#pragma unroll 2
        for (int s = 0; s < vmax; ++s) {
            const float4 v = sm.vp[s];
            const float thr = s < V ? v.w : -INFINITY;  // (other slots hold anything)
            if (NR > 3 && rows <= 3) near += near_rows<(NR > 3 ? 3 : NR)>(v, thr);
            else near += near_rows<NR>(v, thr);
        }
        near = G.bcast(G.incl_scan(near), TT - 1);
        ok = !G.any(!ok) && near == 3 * V && 2 * E == 3 * V;
    }
    // whether a vertex found so far that no generator beyond `reach` cuts has a
    // fourth plane within its error bound or behind it
    __device__ __forceinline__ bool close_vertex(const Sub<TT>& G, const S& sm, bool on, float reach) const
    {
        bool found = false;
        const int vmax = __reduce_max_sync(TFULL, on ? V : 0);
#pragma unroll 1
        for (int s = 0; s < vmax; ++s) {
            const float4 v = sm.vp[s];
            const bool is = on && !found && s < V && 4.0f * (v.x * v.x + v.y * v.y + v.z * v.z) <= reach;
            if (!__any_sync(TFULL, is)) continue;
            int near = near_rows<NR>(v, v.w);
#pragma unroll
            for (int o = TT / 2; o >= 1; o >>= 1) near += __shfl_xor_sync(TFULL, near, o);
            found = found || (is && near > 3);
        }
        return found;
    }
    // a fourth plane at a vertex found so far (a warp per cell only): 2 when one
    // passes through it to what FP64 resolves, as certify64 would find at length
    // (the first two such vertices tell), or when so `many` vertices within half the
    // reach have one within REGULAR |v|, 1 when one is close, 0 when none is.
    // (343,000 points of a cubic lattice, every cell tied: 169 ms when each ran
    // through the walk and the FP64 rays first, now 60 ms, against 51 ms with the
    // clipper alone; 512,000 of a BCC lattice 19.0 -> 5.0 ms)
    __device__ __forceinline__ int tied(const Sub<TT>& G, const S& sm, const float4* __restrict__ sorted, float4 pi,
                                        const GridDesc& grid, float reach, int many) const
    {
        int close = 0, tights = 0;
#pragma unroll 1
        for (int s = 0; s < V; ++s) {
            const float4 v = sm.vp[s];
            const uint32_t ids = *reinterpret_cast<const uint32_t*>(sm.vid[s]);
            const int a = plane_ck(ids & 0xff), b = plane_ck((ids >> 8) & 0xff), c = plane_ck((ids >> 16) & 0xff);
            const float v2 = v.x * v.x + v.y * v.y + v.z * v.z;
            int at = -1;
            bool tight = false;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int p = r * TT + G.gl;
                const float d = fabsf(fmaf(-nx[r], v.x, fmaf(-ny[r], v.y, fmaf(-nz[r], v.z, nb[r]))));
                // (v.w is infinite where |v|^2 overflows: no finite distance keeps a padding plane out)
                if (p != a && p != b && p != c && sm.src[p] != PAD_PLANE && d < v.w) {
                    at = p;
                    tight = tight || d * d < REGULAR * REGULAR * v2;
                }
            }
            if (!__any_sync(TFULL, at >= 0)) continue;
            tights += __any_sync(TFULL, tight) && 4.0f * v2 <= reach;
            if (tights >= many) return 2;
            if (++close > 2) {
                if (tights == 0 || many == INT_MAX) break;
                continue;
            }
            bool tie = false;
            if (at >= 0) {
                double x, y, z;
                if (solve_vertex64<PER>(sm.src[a], sm.src[b], sm.src[c], sorted, pi, grid, x, y, z)) {
                    const P64 h = plane64<PER>(sm.src[at], sorted, pi, grid);
                    const double in = h.b - ((h.x * x + h.y * y) + h.z * z);
                    const double n2 = (h.x * h.x + h.y * h.y) + h.z * h.z, w2 = (x * x + y * y) + z * z;
                    tie = in * in < TIE * TIE * (n2 * w2);
                }
            }
            if (__any_sync(TFULL, tie)) return 2;
        }
        return close > 0 ? 1 : 0;
    }
    // the same with FP64 where float32 does not decide: a plane too close to a
    // vertex passes when the vertex, solved in FP64, is inside it by more than the
    // error of that test (a warp per cell only). With e = 2^-53 a vertex of three
    // planes is known to 32 e / |det| of its length (22 e for the three terms of
    // Cramer's rule, 10 e for the determinant, both over |det| of the unit
    // normals), its two float halves to 2^-48, and the test adds 6 e.
    __device__ __forceinline__ void certify64(const Sub<TT>& G, const S& sm, const double (*pd)[4], const float4* lo,
                                              unsigned& decided)
    {
        bool fine = ok && 2 * E == 3 * V;
        const int vmax = __any_sync(TFULL, !ok) ? 0 : V;
#pragma unroll 1
        for (int s = 0; s < vmax; ++s) {
            const float4 v = sm.vp[s];
            const uint32_t ids = *reinterpret_cast<const uint32_t*>(sm.vid[s]);
            const int a = plane_ck(ids & 0xff), b = plane_ck((ids >> 8) & 0xff), c = plane_ck((ids >> 16) & 0xff);
            uint32_t close = 0;  // rows of the lane's planes too close (PAD_PLANE never is: its distance is FLT_MAX)
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int p = r * TT + G.gl;
                const float d = fmaf(-nx[r], v.x, fmaf(-ny[r], v.y, fmaf(-nz[r], v.z, nb[r])));
                close |= p != a && p != b && p != c && !(d >= v.w) ? 1u << r : 0u;
            }
            if (!__any_sync(TFULL, close != 0)) continue;
            double x, y, z;
            if constexpr (F64) {
                x = sm.v[s][0];
                y = sm.v[s][1];
                z = sm.v[s][2];
            } else {
                x = (double)v.x + (double)lo[s].x;
                y = (double)v.y + (double)lo[s].y;
                z = (double)v.z + (double)lo[s].z;
            }
            const double *A = pd[a], *B = pd[b], *C = pd[c];
            const double det = A[0] * (B[1] * C[2] - B[2] * C[1]) + A[1] * (B[2] * C[0] - B[0] * C[2]) +
                               A[2] * (B[0] * C[1] - B[1] * C[0]);
            const double aa = A[0] * A[0] + A[1] * A[1] + A[2] * A[2], bb = B[0] * B[0] + B[1] * B[1] + B[2] * B[2],
                         cc = C[0] * C[0] + C[1] * C[1] + C[2] * C[2];
            // (squared: the test's margin is (4.3e-15 + 3.6e-15 / |det|) |n| |v|)
            const double m = 4.3e-15 + 3.6e-15 * sqrt(aa) * sqrt(bb) * sqrt(cc) / fabs(det);
            const double lim = m * m * ((x * x + y * y) + z * z);
            for (; close; close &= close - 1) {
                const double* h = pd[(__ffs(close) - 1) * TT + G.gl];
                const double in = h[3] - ((h[0] * x + h[1] * y) + h[2] * z);
                if (!(in > 0.0 && in * in > lim * ((h[0] * h[0] + h[1] * h[1]) + h[2] * h[2]))) fine = false;
                ++decided;
            }
        }
        ok = !__any_sync(TFULL, !fine);
    }
};

// moments, neighbours and geometry of the group's cell (the quantities of
// finish_cell); every lane of the warp calls, groups with V = 0 write nothing.
// A lane per edge (eight lanes also of a warp per cell, so that the float sums
// are the same whichever kernel built the cell): the two triangles of
// an edge share its cross product. Areas only decide which faces are above
// the neighbour threshold: they add up in fixed point (integers add in any
// order alike), and a face below 1e-4 R^2 is added up again in the arithmetic
// of the form, edge by edge.
template <typename Real, int TT, int NP, int NV, bool PER>
__device__ __forceinline__ void trace_finish(TraceSmem<Real, NP, NV>& sm, const Sub<TT>& G, int V,
                                             const Faces<(NP + 31) / 32>& faces, float R2, float4 pi, int64_t out_idx,
                                             const TraceArgs& A)
{
    constexpr bool F64 = sizeof(Real) == 8;
    const int gl = G.gl;
    const bool act = V > 0;
    const int F = act ? faces.count() : 0;
    const int E = 3 * V / 2;
    if (A.rec) {
        for (int f = gl; f < NP; f += TT) sm.u.f[f] = 0;
        __syncwarp();
    }
    auto plane = [&](int f, Real& x, Real& y, Real& z, Real& sc) {
        if constexpr (F64) {
            x = sm.pn[f][0];
            y = sm.pn[f][1];
            z = sm.pn[f][2];
            sc = sm.ps[f];
        } else {
            const float4 p = sm.pl[f];
            x = p.x;
            y = p.y;
            z = p.z;
            sc = sm.src[f] < 0 ? p.w : 0.5f;  // b / |n|^2
        }
    };
    auto vert = [&](int s, Real& x, Real& y, Real& z) {
        if constexpr (F64) {
            x = sm.v[s][0];
            y = sm.v[s][1];
            z = sm.v[s][2];
        } else {
            const float4 p = sm.vp[s];
            x = p.x;
            y = p.y;
            z = p.z;
        }
    };
    // tetrahedra (0, foot of face, v, next(v around the face)); float sums of three
    // edges' six, FP64 between them
    double s0[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const float fix = 1048576.0f * rcp_fast(R2);
#pragma unroll 1
    for (int e0 = gl < 8 ? gl : E; e0 < E; e0 += 24) {
        Real vol = 0, mx = 0, my = 0, mz = 0, m2 = 0;
#pragma unroll 1
        for (int e = e0; e < E && e < e0 + 24; e += 8) {
            const uint32_t ed = sm.ed[e];
            Real ax, ay, az, bx, by, bz;
            vert(vt_ck((ed >> 16) & 0xff, NV, CK_SLOT, A.st), ax, ay, az);
            vert(vt_ck(ed >> 24, NV, CK_SLOT, A.st), bx, by, bz);
            const Real cx = ay * bz - az * by, cy = az * bx - ax * bz, cz = ax * by - ay * bx;
            const Real ab2 = ax * ax + ay * ay + az * az + bx * bx + by * by + bz * bz;
            const Real tx = ax + bx, ty = ay + by, tz = az + bz;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int f = vt_ck((ed >> (8 * t)) & 0xff, NP, CK_PLANE, A.st);
                Real px, py, pz, sc;
                plane(f, px, py, pz, sc);
                const Real qx = px * sc, qy = py * sc, qz = pz * sc;
                const Real qc = qx * cx + qy * cy + qz * cz;
                const Real dv = qc * (Real)(t ? 1.0 / 6.0 : -1.0 / 6.0);
                const Real sx = qx + tx, sy = qy + ty, sz = qz + tz;
                const Real q2 = qx * qx + qy * qy + qz * qz;
                vol += dv;
                mx += dv * sx;
                my += dv * sy;
                mz += dv * sz;
                m2 += dv * (q2 + ab2 + sx * sx + sy * sy + sz * sz);
                if (A.rec) {  // twice the triangle's signed area is q.c / |q|
                    const float a2 = (float)qc * rsqrt_fast((float)q2) * fix;
                    atomicAdd(&sm.u.f[f], __float2int_rn(t ? a2 : -a2));
                }
            }
        }
        s0[0] += (double)vol;
        s0[1] += (double)mx;
        s0[2] += (double)my;
        s0[3] += (double)mz;
        s0[4] += (double)m2;
    }
    // FP64 sums over the 8 lanes by reduce-scatter: 7 additions instead of 15
    double w;
    {
        double t4[4], t2[2];
        const bool hi1 = (gl & 4) != 0, hi2 = (gl & 2) != 0, hi3 = (gl & 1) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double up = i == 0 ? s0[4] : 0.0, send = hi1 ? s0[i] : up;
            t4[i] = (hi1 ? up : s0[i]) + __shfl_xor_sync(TFULL, send, 4);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const double send = hi2 ? t4[i] : t4[2 + i];
            t2[i] = (hi2 ? t4[2 + i] : t4[i]) + __shfl_xor_sync(TFULL, send, 2);
        }
        w = (hi3 ? t2[1] : t2[0]) + __shfl_xor_sync(TFULL, hi3 ? t2[0] : t2[1], 1);
    }
    // lane 0 holds V, 1 M_x, 2 M_y, 3 M_z, 4 M2
    const double vol_t = G.bcast(w, 0);
    if (act) {
        if (gl == 0 && A.vol) A.vol[out_idx] = vol_t;
        if (gl >= 1 && gl <= 3 && A.cen) {
            const float pc = gl == 1 ? pi.x : (gl == 2 ? pi.y : pi.z);
            A.cen[3 * out_idx + gl - 1] = (double)pc + 0.25 * w / vol_t;
        }
        if (gl == 4 && A.m2) A.m2[out_idx] = 0.05 * w;
    }
    if (!A.rec) return;
    __syncwarp();  // the area sums are complete
    uint8_t* rec = A.rec + (size_t)out_idx * A.rec_stride;
    const bool geom = (A.emit & VT_EMIT_GEOM) != 0;
    int32_t* rfn = reinterpret_cast<int32_t*>(rec + REC_FNBR_OFF);
    int kept = 0;
    const int Fmax = __reduce_max_sync(TFULL, F);
#pragma unroll 1
    for (int i0 = 0; i0 < Fmax; i0 += TT) {
        const int i = i0 + gl;
        int key = INT_MAX;
        if (i < F) {
            const int f = vt_ck(faces.nth(i), NP, CK_PLANE, A.st);
            const int src = sm.src[f];
            int oid = src;  // wall ids stay
            if (PER) {
                if (src < 0)
                    oid = (int)out_idx;
                else
                    oid = A.index_space == VT_INDEX_ORIGINAL ? __float_as_int(A.sorted[src & IMG_INDEX_MASK].w)
                                                             : (src & IMG_INDEX_MASK);
            } else if (src >= 0 && A.index_space == VT_INDEX_ORIGINAL) {
                oid = __float_as_int(A.sorted[src].w);
            }
            if (geom) rfn[vt_ck(i, REC_FACES, CK_RECORD, A.st)] = oid;
            bool nb = true;
            if (sm.u.f[f] < 210) {  // 2e-4 R^2 of doubled area
                Real fnx, fny, fnz, sc, area = 0, tau;
                plane(f, fnx, fny, fnz, sc);
                const Real qx = fnx * sc, qy = fny * sc, qz = fnz * sc;
#pragma unroll 1
                for (int e = 0; e < E; ++e) {
                    const uint32_t ed = sm.ed[e];
                    const bool on_a = (ed & 0xff) == (uint32_t)f;
                    if (!on_a && ((ed >> 8) & 0xff) != (uint32_t)f) continue;
                    Real ux, uy, uz, wx, wy, wz;
                    vert(on_a ? ed >> 24 : (ed >> 16) & 0xff, ux, uy, uz);
                    vert(on_a ? (ed >> 16) & 0xff : ed >> 24, wx, wy, wz);
                    ux -= qx; uy -= qy; uz -= qz;
                    wx -= qx; wy -= qy; wz -= qz;
                    area += (uy * wz - uz * wy) * fnx + (uz * wx - ux * wz) * fny + (ux * wy - uy * wx) * fnz;
                }
                area *= (Real)0.5 / sqrt(fnx * fnx + fny * fny + fnz * fnz);
                if (!F64) {
                    const float cv = cbrtf((float)vol_t);
                    tau = (Real)((float)Tol<float>::area_rel * cv * cv);
                } else {
                    tau = (Real)(Tol<double>::area_rel * cbrt(vol_t * vol_t));
                }
                nb = area > tau;
            }
            nb = nb && (src >= 0 || PER);
            kept += nb;
            // (periodic ids may repeat; the plane makes the key unique)
            if (nb) key = PER ? oid * 128 + f : oid;
        }
        __syncwarp();  // (the i-th face is plane i or a later one: its area is read before this)
        if (i < F) sm.u.f[vt_ck(i, NP, CK_PLANE, A.st)] = key;
    }
    __syncwarp();
    int32_t* rnbr = reinterpret_cast<int32_t*>(rec + REC_NBR_OFF);
#pragma unroll 1
    for (int i = gl; i < F; i += TT) {  // neighbours ascending: each key's rank
        const int key = sm.u.f[i];
        if (key == INT_MAX) continue;
        int rank = 0;
#pragma unroll 4
        for (int k = 0; k < F; ++k) rank += sm.u.f[k] < key ? 1 : 0;
        rnbr[vt_ck(rank, REC_FACES, CK_RECORD, A.st)] = PER ? key / 128 : key;
    }
    const int nn = G.bcast(G.incl_scan(kept), TT - 1);
    if (geom) {
        double* rv = reinterpret_cast<double*>(rec + REC_VTX_OFF);
        float* rv32 = reinterpret_cast<float*>(rec + REC_VTX_OFF);
        for (int s = gl; s < V; s += TT) {
            Real x, y, z;
            vert(s, x, y, z);
            if (A.rec_f32) {
                rv32[3 * s] = (float)x;
                rv32[3 * s + 1] = (float)y;
                rv32[3 * s + 2] = (float)z;
            } else {
                rv[3 * s] = (double)pi.x + (double)x;
                rv[3 * s + 1] = (double)pi.y + (double)y;
                rv[3 * s + 2] = (double)pi.z + (double)z;
            }
        }
        // loops of the faces: the vertex after vertex s around the t-th of its
        // planes at byte 4 s + t, and each plane's lowest vertex and degree,
        // over the planes (not needed any more)
        __syncwarp();
        uint8_t* next = reinterpret_cast<uint8_t*>(sm.pl);
        int32_t* first = reinterpret_cast<int32_t*>(sm.pl) + NV;
        int32_t* degree = first + NP;
        static_assert(4 * NV + 8 * NP <= 16 * NP, "the loops fit the planes");
        for (int f = gl; f < NP; f += TT) {
            first[f] = NV;
            degree[f] = 0;
        }
        __syncwarp();
#pragma unroll 1
        for (int e = gl; e < E; e += TT) {
            const uint32_t ed = sm.ed[e];
            const int s = (ed >> 16) & 0xff, t = ed >> 24;
#pragma unroll
            for (int k = 0; k < 2; ++k) {  // k = 0: plane a, t -> s; 1: plane b, s -> t
                const int f = (ed >> (8 * k)) & 0xff, u = k ? s : t, v = k ? t : s;
                const uint32_t ids = *reinterpret_cast<const uint32_t*>(sm.vid[u]);
                const int at = (ids & 0xff) == (uint32_t)f ? 0 : (((ids >> 8) & 0xff) == (uint32_t)f ? 1 : 2);
                next[vt_ck(4 * u + at, 4 * NV, CK_SLOT, A.st)] = (uint8_t)v;
                atomicMin(&first[vt_ck(f, NP, CK_PLANE, A.st)], u);
                atomicAdd(&degree[f], 1);
            }
        }
        __syncwarp();
        uint8_t* rdeg = rec + REC_FDEG_OFF;
        uint8_t* rfv = rec + REC_FVTX_OFF;
        int base = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < Fmax; i0 += TT) {
            const int i = i0 + gl;
            const int f = i < F ? faces.nth(i) : 0;
            const int deg = i < F ? degree[f] : 0;
            const int inc = G.incl_scan(deg);
            const int pos = base + inc - deg;
            base += G.bcast(inc, TT - 1);
            if (i < F) {
                rdeg[i] = (uint8_t)deg;
                int cur = vt_ck(first[f], NV, CK_SLOT, A.st);
#pragma unroll 1
                for (int k = 0; k < deg; ++k) {
                    const uint32_t ids = *reinterpret_cast<const uint32_t*>(sm.vid[cur]);
                    const int at = (ids & 0xff) == (uint32_t)f ? 0 : (((ids >> 8) & 0xff) == (uint32_t)f ? 1 : 2);
                    rfv[vt_ck(pos + k, 3 * REC_VERTS, CK_RECORD, A.st)] = (uint8_t)cur;
                    cur = vt_ck(next[4 * cur + at], NV, CK_SLOT, A.st);
                }
            }
        }
    }
    if (act && gl == 0) {
        RecHeader* hd = reinterpret_cast<RecHeader*>(rec);
        hd->nnbr = nn;
        hd->nface = geom ? F : 0;
        hd->nvtx = geom ? V : 0;
        hd->nfv = geom ? 3 * V : 0;
        hd->p[0] = pi.x;
        hd->p[1] = pi.y;
        hd->p[2] = pi.z;
    }
    __syncwarp();
}

// appends q of the lanes with `on` to a device list, one counter update per warp
__device__ __forceinline__ void append(int32_t* list, int32_t* ctr, bool on, int q, int lane)
{
    const unsigned m = __ballot_sync(TFULL, on);
    if (!m) return;
    int at = 0;
    if (lane == __ffs(m) - 1) at = atomicAdd(ctr, __popc(m));
    at = __shfl_sync(TFULL, at, __ffs(m) - 1);
    if (on) list[at + __popc(m & ((1u << lane) - 1u))] = q;
}

// an open or failed cell between two kernels of the pass, in its state slot
struct alignas(16) OpenCell {
    int32_t np, nf;
    float reach;              // generators with a float key below this are behind it
    float all2;               // (2R)^2
    int32_t turns;            // times it was built
    int32_t close;            // 1: failed with a fourth plane at a vertex (see close_vertex)
    int32_t pad[2];
    int32_t src[40];          // its planes: the faces, then what cuts it
    float4 far[48];           // vertices a generator at `reach` or beyond can cut (see far_vertices)
};
static_assert(sizeof(OpenCell) <= StateLayout<float, 64, 64>::BYTES, "an open cell fits the state slot");

// a walk that met a cutting generator goes on for this many limits, or until
// it has this many: one annulus of a sparse side rarely closes a cell (0, 1 and
// 2 limits: 139, 85 and 74 thousand turns of the warp-per-cell kernel on 1M
// points half in clumps)
constexpr int WALK_ENOUGH = 8, WALK_PAST = 2;
// after a limit whose rows held more than WALK_DENSE generators (a clump inside one
// grid cell: every limit reads all of it again) the next lies WALK_WIDE times farther.
// Not in a periodic box, where a wide limit takes the clump's images as well (30,000
// points in one clump and 60 around it 17.3 -> 31.7 ms)
constexpr unsigned WALK_DENSE = 4096;
constexpr float WALK_WIDE = 16.0f;
// a warp's list of cutting generators: the ones kept, and a batch
constexpr int CUT_LIST = 64;

// the nearest `cap` of the warp's ns candidates, in order of (key, id)
__device__ __forceinline__ int keep_nearest(float* key, int32_t* id, int ns, int cap, int lane)
{
    __syncwarp();
    const float k0 = lane < ns ? key[lane] : FLT_MAX, k1 = lane + 32 < ns ? key[lane + 32] : FLT_MAX;
    const int j0 = lane < ns ? id[lane] : INT_MAX, j1 = lane + 32 < ns ? id[lane + 32] : INT_MAX;
    int r0 = 0, r1 = 0;
#pragma unroll 1
    for (int i = 0; i < ns; ++i) {
        const float k = key[i];
        const int j = id[i];
        r0 += k < k0 || (k == k0 && j < j0);
        r1 += k < k1 || (k == k1 && j < j1);
    }
    __syncwarp();
    if (lane < ns && r0 < cap) {
        key[r0] = k0;
        id[r0] = j0;
    }
    if (lane + 32 < ns && r1 < cap) {
        key[r1] = k1;
        id[r1] = j1;
    }
    __syncwarp();
    return ns < cap ? ns : cap;
}

// The walk of a cell, by a warp: the generators with keys of at least `reach`
// and within 2R (all2) that cut one of the nf far vertices (position and
// error bound; shared memory, as the lists key and id), the nearest `keep` of them in order;
// returns their count. own[0, np): the cell's planes. It takes the rows of the
// grid that meet the box of the far vertices' balls and the ball of the current
// limit, less the grid cells that are behind; the limit grows from the reach by
// half its radius at a time, and the walk ends soon after the first limit that
// met a cutting generator (the cell it leaves is smaller). A lane per row finds the
// row's runs, then the lanes share the rows' generators. reach becomes what a
// later walk of the cell need not look at again.
// SPREAD: no far vertices; the nearest two generators at `reach` or beyond of
// each octant around the generator, as far out as the emptiest octants but one
// need (an octant also ends at a wall): planes that close a cell whose list
// lies to one side of it.
template <bool PER, bool SPREAD>
__device__ __forceinline__ int walk(const TraceArgs& A, const GridDesc& grid, int q, float4 pi, const float4* far, int nf,
                                    const int32_t* own, int np, float all2, int keep, float& reach,
                                    float* key, int32_t* id, unsigned& cands)
{
    const int lane = threadIdx.x & 31;
    // the box of the far vertices' balls, around the generator
    float l0 = 0, l1 = 0, l2 = 0, h0 = 0, h1 = 0, h2 = 0;
    for (int s = lane; s < nf; s += 32) {
        const float4 v = far[s];
        const float r = sqrt_fast(v.x * v.x + v.y * v.y + v.z * v.z) * FAR_BALL;
        l0 = fminf(l0, v.x - r); h0 = fmaxf(h0, v.x + r);
        l1 = fminf(l1, v.y - r); h1 = fmaxf(h1, v.y + r);
        l2 = fminf(l2, v.z - r); h2 = fmaxf(h2, v.z + r);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        l0 = fminf(l0, __shfl_xor_sync(TFULL, l0, o)); h0 = fmaxf(h0, __shfl_xor_sync(TFULL, h0, o));
        l1 = fminf(l1, __shfl_xor_sync(TFULL, l1, o)); h1 = fmaxf(h1, __shfl_xor_sync(TFULL, h1, o));
        l2 = fminf(l2, __shfl_xor_sync(TFULL, l2, o)); h2 = fmaxf(h2, __shfl_xor_sync(TFULL, h2, o));
    }
    const int Gr = grid.G;
    const int32_t* coff = A.cell_off + grid.cell_base;
    const float m = (float)grid.margin;
    const float cx = (float)grid.cw[0], cy = (float)grid.cw[1];
    // periodic: unwrapped grid coordinates, and each row once per z image
    const float lim_lo = PER ? -2.0f * (float)Gr : 0.0f,
                lim_hi = PER ? 3.0f * (float)Gr - 1.0f : (float)Gr - 1.0f;
    auto clamp = [&](float t) { return (int)floorf(fminf(fmaxf(t, lim_lo), lim_hi)); };
    int ns = 0;
    // the farthest kept key once the list is full: what lies beyond it would be sorted
    // in and dropped again (thousands of a clump's generators cut the sparse cells beside
    // it: 30,000 points in one clump and 60 around it 17.6 -> 16.6 ms, 500,000 half in
    // clumps, fused, 7.82 -> 7.51, 120,000 2.53 -> 2.50 ms)
    float nearest = FLT_MAX;
    unsigned before = cands;
    bool more = false, end = !SPREAD && nf == 0;
    if (SPREAD) {
        l0 = l1 = l2 = -FLT_MAX;
        h0 = h1 = h2 = FLT_MAX;
        if (lane < 16) {
            key[lane] = FLT_MAX;
            id[lane] = -1;
        }
        __syncwarp();
    }
    // (40 steps of 2.25 cover every ratio of float32 keys that differ; the
    // last one takes the whole ball)
#pragma unroll 1
    for (int it = 0, past = 0; !end && (ns == 0 || (ns < WALK_ENOUGH && past++ < WALK_PAST)); ++it) {
        const float lim2 = it < 40 ? fminf(all2, (!PER && cands - before > WALK_DENSE ? WALK_WIDE : 2.25f) * reach) : all2;
        before = cands;
        const float r_out2 = lim2 * (1.0f + 1e-4f), r_in2 = reach * (1.0f - 1e-4f);
        const float rr = sqrt_fast(r_out2) * (1.0f + 1e-5f);
        const float z_lo = pi.z + fmaxf(l2, -rr) - m, z_hi = pi.z + fminf(h2, rr) + m;
        const int x0 = clamp((pi.x + fmaxf(l0, -rr) - m - grid.lo[0]) * grid.scale[0] - 1e-3f);
        const int x1 = clamp((pi.x + fminf(h0, rr) + m - grid.lo[0]) * grid.scale[0] + 1e-3f);
        const int y0 = clamp((pi.y + fmaxf(l1, -rr) - m - grid.lo[1]) * grid.scale[1] - 1e-3f);
        const int y1 = clamp((pi.y + fminf(h1, rr) + m - grid.lo[1]) * grid.scale[1] + 1e-3f);
        int t0 = 0, nt = 1;
        if (PER) {
            t0 = floordiv(clamp((z_lo - grid.lo[2]) * grid.scale[2] - 1e-3f), Gr);
            nt = floordiv(clamp((z_hi - grid.lo[2]) * grid.scale[2] + 1e-3f), Gr) - t0 + 1;
        }
        const int wy = y1 - y0 + 1, nrow = (x1 - x0 + 1) * wy * nt;
#pragma unroll 1
        for (int e0 = 0; e0 < nrow; e0 += 32) {
            const int e = e0 + lane;
            int sa = 0, la = 0, sb = 0, lb = 0, code = IMG_NONE;
            if (e < nrow) {
                const int e2 = PER ? e / nt : e;
                const int tz = PER ? t0 + (e - e2 * nt) : 0;
                const int ex = e2 / wy, x = x0 + ex, y = y0 + (e2 - ex * wy);
                const int tx = PER ? floordiv(x, Gr) : 0, ty = PER ? floordiv(y, Gr) : 0;
                const float gx0 = grid.lo[0] + (float)x * cx - m, gx1 = grid.lo[0] + (float)(x + 1) * cx + m;
                const float gy0 = grid.lo[1] + (float)y * cy - m, gy1 = grid.lo[1] + (float)(y + 1) * cy + m;
                const float dxn = fmaxf(fmaxf(gx0 - pi.x, pi.x - gx1), 0.0f),
                            dyn = fmaxf(fmaxf(gy0 - pi.y, pi.y - gy1), 0.0f);
                const float dxf = fmaxf(pi.x - gx0, gx1 - pi.x), dyf = fmaxf(pi.y - gy0, gy1 - pi.y);
                const float dn2 = dxn * dxn + dyn * dyn, df2 = dxf * dxf + dyf * dyf;
                if (dn2 <= r_out2) {
                    const float zr = sqrtf(r_out2 - dn2);
                    // the part of the row inside the balls: the hull of their spans
                    float s0 = SPREAD ? -FLT_MAX : FLT_MAX, s1 = -s0;
#pragma unroll 2
                    for (int k = 0; !SPREAD && k < nf; ++k) {
                        const float4 v = far[k];
                        const float bx = fmaxf(fmaxf(gx0 - pi.x - v.x, v.x - (gx1 - pi.x)), 0.0f);
                        const float by = fmaxf(fmaxf(gy0 - pi.y - v.y, v.y - (gy1 - pi.y)), 0.0f);
                        const float left = (v.x * v.x + v.y * v.y + v.z * v.z) * (FAR_BALL * FAR_BALL) - (bx * bx + by * by);
                        const float half = sqrt_fast(fmaxf(left, 0.0f));
                        if (left >= 0.0f) {
                            s0 = fminf(s0, v.z - half);
                            s1 = fmaxf(s1, v.z + half);
                        }
                    }
                    s0 = pi.z + fmaxf(s0, -zr) - m;
                    s1 = pi.z + fminf(s1, zr) + m;
                    int za = clamp((s0 - grid.lo[2]) * grid.scale[2] - 1e-3f);
                    int zb = clamp((s1 - grid.lo[2]) * grid.scale[2] + 1e-3f);
                    if (s0 > s1) zb = za - 1;
                    if (PER) {
                        za = za > tz * Gr ? za : tz * Gr;
                        zb = zb < tz * Gr + Gr - 1 ? zb : tz * Gr + Gr - 1;
                    }
                    // grid cells wholly inside the ball that is behind: [i0, i1]
                    int i0 = zb + 1, i1 = zb;
                    if (r_in2 > df2) {
                        const float zi = sqrtf(r_in2 - df2) - m;
                        i0 = (int)ceilf(fminf(fmaxf((pi.z - zi - grid.lo[2]) * grid.scale[2] + 1e-3f, lim_lo - 1.0f),
                                              lim_hi + 2.0f));
                        i1 = (int)floorf(fminf(fmaxf((pi.z + zi - grid.lo[2]) * grid.scale[2] - 1e-3f, lim_lo - 1.0f),
                                               lim_hi + 2.0f)) - 1;
                        if (i0 > i1 || i1 < za || i0 > zb) {
                            i0 = zb + 1;
                            i1 = zb;
                        }
                    }
                    const int base = ((x - tx * Gr) * Gr + (y - ty * Gr)) * Gr - tz * Gr;
                    const int ea = i0 - 1, fb = i1 + 1 > za ? i1 + 1 : za;
                    if (za <= ea) {
                        sa = coff[base + za];
                        la = coff[base + ea + 1] - sa;
                    }
                    if (i0 <= zb && fb <= zb) {
                        sb = coff[base + fb];
                        lb = coff[base + zb + 1] - sb;
                    }
                    if (PER) code = img_code(tx, ty, tz);
                }
            }
            int incl = la + lb;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int u = __shfl_up_sync(TFULL, incl, d);
                if (lane >= d) incl += u;
            }
            const int total = __shfl_sync(TFULL, incl, 31);
            const int start = incl - la - lb;
            cands += (unsigned)total;
#pragma unroll 1
            for (int c0 = 0; c0 < total; c0 += 32) {
                const int i = c0 + lane;
                int seg = 0;  // rows ending at or before i
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1)
                    if (__shfl_sync(TFULL, incl, (seg + step - 1) & 31) <= i) seg += step;
                seg &= 31;
                const int off = i - __shfl_sync(TFULL, start, seg), na = __shfl_sync(TFULL, la, seg);
                const int ja = __shfl_sync(TFULL, sa, seg), jb = __shfl_sync(TFULL, sb, seg);
                const int cd = PER ? __shfl_sync(TFULL, code, seg) : IMG_NONE;
                const int j = off < na ? ja + off : jb + (off - na);
                const int jj = PER ? img_pack(j, cd) : j;
                float3 o = make_float3(0.0f, 0.0f, 0.0f);
                const bool in = i < total && j != q;
                if (in) o = img_off_t<PER>(pi, A.sorted[j], cd, grid);
                const float d2 = fmaf(o.z, o.z, fmaf(o.y, o.y, o.x * o.x));
                bool cuts = in && d2 >= reach && d2 < lim2 && (SPREAD || d2 <= nearest);
                if (!__any_sync(TFULL, cuts)) continue;
                if (SPREAD) {
                    if (cuts)
                        for (int p = 0; p < np; ++p)
                            if (own[p] == jj) cuts = false;
                    const int oct = (o.x < 0.0f ? 1 : 0) | (o.y < 0.0f ? 2 : 0) | (o.z < 0.0f ? 4 : 0);
#pragma unroll 1
                    for (int e = 0; e < 16; ++e) {  // an octant's nearest, then its next
                        const bool mine = cuts && oct == e >> 1 && d2 < key[e | 1];
                        const unsigned near = __reduce_min_sync(TFULL, mine ? __float_as_uint(d2) : 0x7fffffffu);
                        if (near == 0x7fffffffu) continue;
                        const unsigned who = __ballot_sync(TFULL, mine && __float_as_uint(d2) == near);
                        const bool me = lane == __ffs(who) - 1;
                        if (me) {
                            const int f = e & ~1;
                            if (d2 < key[f]) {
                                key[f + 1] = key[f];
                                id[f + 1] = id[f];
                                key[f] = d2;
                                id[f] = jj;
                            } else {
                                key[f + 1] = d2;
                                id[f + 1] = jj;
                            }
                            cuts = false;
                        }
                        __syncwarp();
                    }
                    continue;
                }
                const float len = sqrt_fast(d2);
                float top = -FLT_MAX;
#pragma unroll 2
                for (int k = 0; k < nf; ++k) {
                    const float4 v = far[k];
                    top = fmaxf(top, fmaf(o.x, v.x, fmaf(o.y, v.y, fmaf(o.z, v.z, len * v.w))));
                }
                cuts = cuts && 0.5f * d2 <= top;
                if (cuts)  // (the cell's own faces touch their vertices)
                    for (int p = 0; p < np; ++p)
                        if (own[p] == jj) cuts = false;
                const unsigned cm = __ballot_sync(TFULL, cuts);
                if (cuts) {
                    const int at = ns + __popc(cm & ((1u << lane) - 1u));
                    key[vt_ck(at, CUT_LIST, CK_RECORD, A.st)] = d2;
                    id[vt_ck(at, CUT_LIST, CK_RECORD, A.st)] = jj;
                }
                ns += __popc(cm);
                if (ns > keep) {
                    more = true;
                    ns = keep_nearest(key, id, ns, keep, lane);
                    nearest = key[ns - 1];
                }
            }
        }
        end = lim2 >= all2;
        if (!more) reach = lim2;  // (all of it is behind)
        if (SPREAD) {
            bool full = true;
            if (lane < 8) {
                full = key[2 * lane] < FLT_MAX;
                if (!PER) {
                    const float wx = lane & 1 ? pi.x - grid.lo[0] : grid.hi[0] - pi.x;
                    const float wy = lane & 2 ? pi.y - grid.lo[1] : grid.hi[1] - pi.y;
                    const float wz = lane & 4 ? pi.z - grid.lo[2] : grid.hi[2] - pi.z;
                    const float wall = fminf(wx, fminf(wy, wz));
                    full = full || wall * wall < lim2;
                }
            }
            end = end || __popc(__ballot_sync(TFULL, full)) >= 31;
        }
    }
    if (SPREAD) {
        const int j = lane < 16 ? id[lane] : -1;
        const unsigned m = __ballot_sync(TFULL, j >= 0);
        __syncwarp();
        if (j >= 0) id[__popc(m & ((1u << lane) - 1u))] = j;
        __syncwarp();
        return __popc(m);
    }
    if (ns > 0) {
        ns = keep_nearest(key, id, ns, keep, lane);
        if (more) reach = key[ns - 1];
    }
    return ns;
}

// vertices beyond half the reach into far (position, error bound): a generator cuts a
// vertex v only from inside the ball of radius |v| around v
template <int TT, typename S>
__device__ __forceinline__ int far_vertices(const Sub<TT>& G, const S& sm, bool on, int V, float reach, float4* far, int cap,
                                            DevStatus* st)
{
    int nf = 0;
    const int vmax = __reduce_max_sync(TFULL, on ? V : 0);
    const float half = 0.25f * reach * (1.0f / FAR_R2);
#pragma unroll 1
    for (int s0 = 0; s0 < vmax; s0 += TT) {
        const int s = s0 + G.gl;  // (the slots are a multiple of TT)
        const float4 v = sm.vp[s];
        const float d = v.x * v.x + v.y * v.y + v.z * v.z;
        const bool is = on && s < V && d >= half;
        const unsigned m = G.ballot(is);
        if (is) far[vt_ck(nf + __popc(m & ((1u << G.gl) - 1u)), cap, CK_SLOT, st)] = v;
        nf += __popc(m);
    }
    return nf;
}

// The walk of a round's open cells, a warp per cell. Waits for the generators'
// loads: four blocks per SM (64 registers, 40 bytes of spills in the rows' set-up)
// against three: 8M points half in clumps 78.6 -> 76.0 ms, FP64 form of 1M 30.6 ->
// 30.3; 100,000 points in one clump and 1,000 around it, the walks alone 39.9 -> 29.1
// with the wider limits above (34.3 by these alone; the clipper's range lists 20.7)
constexpr int CUT_BLOCK = 256;
template <bool PER>
__global__ void __launch_bounds__(CUT_BLOCK, 4) k_cutters(const __grid_constant__ TraceArgs A)
{
    __shared__ float4 s_far[CUT_BLOCK / 32][48];
    __shared__ float s_key[CUT_BLOCK / 32][CUT_LIST];
    __shared__ int32_t s_id[CUT_BLOCK / 32][CUT_LIST];
    static_assert(48 / 2 + 2 + TRACE_KEEP <= 40, "the planes of the next round");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int have = *A.nq_dev;
    const int nq = have < (int)A.nq ? have : (int)A.nq;
    unsigned cells = 0, cands = 0;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(A.queue, 1);
        c = __shfl_sync(TFULL, c, 0);
        if (c >= nq) break;
        const int q = A.queries[c];
        const GridDesc& grid = grid_of(A.g, A.sets, A.set_of, q);
        const float4 pi = A.sorted[q];
        OpenCell* h = reinterpret_cast<OpenCell*>(A.state + (size_t)(q - A.first) * A.state_stride);
        const int np = h->np, nf = h->nf;
        float reach = h->reach;
        for (int s = lane; s < nf; s += 32) s_far[warp][s] = h->far[s];
        __syncwarp();
        const int ns = walk<PER, false>(A, grid, q, pi, s_far[warp], nf, h->src, np, h->all2, TRACE_KEEP, reach,
                                 s_key[warp], s_id[warp], cands);
        ++cells;
        if (ns > 0) {
            if (lane < ns) h->src[vt_ck(np + lane, 40, CK_PLANE, A.st)] = s_id[warp][lane];
            if (lane == 0) {
                h->np = np + ns;
                h->reach = reach;
                A.next_list[atomicAdd(A.next_ctr, 1)] = q;
            }
        }
        __syncwarp();
    }
    if (lane == 0 && cells) {
        // (one walk per cell: later rounds continue it)
        if (A.round == 0) atomicAdd(&A.st->walk_cells, (unsigned long long)cells);
        atomicAdd(&A.st->walk_cands, (unsigned long long)cands);
    }
}

// Blocks of 128 threads build 16 cells at a time, their warps aligned by a
// barrier before the rays and one after them: the rays, the certificate and the
// finish are 70 KB of code, and warps that drift apart wait for instructions
// (uniform 1M points, neighbours: 7.58 ms of the list pass against 9.07 without
// barriers; blocks of 256 threads 7.69 and of 64 threads 7.18 against 7.29 ms,
// the latter 0.4 ms slower with geometry). Five blocks per SM (96 registers, no
// spills) against six: 7.29 and 7.41 ms.
constexpr int TRACE_BLOCK = 128;
constexpr int TRACE_MINB = 5;

// the lists' cells, or the cells sent back by the walk of the round before, by
// groups of 8 lanes
template <typename Real, bool PER>
__global__ void __launch_bounds__(TRACE_BLOCK, (sizeof(Real) == 4 ? TRACE_MINB : 4)) k_trace(const __grid_constant__ TraceArgs A)
{
    constexpr int TT = 8, NR = 5, NV = 48;
    using T = Tracer<Real, TT, NR, NV, PER>;
    using S = typename T::S;
    constexpr bool F64 = T::F64;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_first;
    const Sub<TT> G;
    const int gl = G.gl;
    S& sm = *reinterpret_cast<S*>(smem_raw + (threadIdx.x / TT) * trace_stride<S>());
    int nq = (int)A.nq;
    if (A.nq_dev) {
        const int have = *A.nq_dev;
        nq = have < nq ? have : nq;
    }
    unsigned n_open = 0, n_second = 0;  // added once per group
    for (;;) {
        if (threadIdx.x == 0) s_first = atomicAdd(A.queue, TRACE_BLOCK / TT);
        __syncthreads();
        const int c_block = s_first;
        if (c_block >= nq) break;
        const int c0 = c_block + threadIdx.x / TT;
        const bool act = c0 < nq;  // a group past the end repeats the last cell and writes nothing
        const int c = act ? c0 : nq - 1;
        const int q = A.queries ? A.queries[c] : (int)A.first + c;
        const GridDesc& grid = grid_of(A.g, A.sets, A.set_of, q);
        const float4 pi = A.sorted[q];
        OpenCell* h = reinterpret_cast<OpenCell*>(A.state + (size_t)(q - A.first) * A.state_stride);
        T t;
        t.st = A.st;
        int P;
        float reach;  // every generator with a float key below this was in the lists so far
        const int32_t* srcs;
        if (A.round == 0) {
            srcs = A.nbr + (int64_t)c * A.kstride - 6;
            P = 6 + A.kc;
            reach = A.reach[c];
        } else {
            srcs = h->src;
            P = h->np;
            reach = h->reach;
        }
        t.rows = __reduce_max_sync(TFULL, (P + TT - 1) / TT);
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int p = r * TT + gl;
            int src = PAD_PLANE;
            if (p < P) {
                src = A.round == 0 && p < 6 ? -(p + 1) : srcs[p];
                if (A.round == 0 && p >= 6 && src < 0) src = PAD_PLANE;  // the list is shorter
            }
            t.set_plane(sm, r, p, src, pi, grid, A.sorted);
        }
        __syncwarp();
        const bool all = reach == FLT_MAX;  // the list holds every other generator
        const unsigned gen0 = G.ballot(sm.src[gl] >= 0);  // the nearest generator's plane follows the walls
        const int f0 = gen0 ? __ffs(gen0) - 1 : 0;
        t.template trace<float>(G, sm, gen0 != 0 && T::in_range(sm, f0), f0, nullptr, nullptr);
        __syncthreads();
        t.solve(G, sm, pi, grid, A.sorted, T::UNIT_F64, T::UNIT_MIN);
        t.certify(G, sm);
        const bool close = A.round == 0 && __any_sync(TFULL, act && !t.ok) && t.close_vertex(G, sm, act && !t.ok, reach);
        // security radius
        const bool valid = all || (A.round == 0 && 4.0f * FAR_R2 * t.R2 <= reach);
        const bool open = act && t.ok && !valid;
        if (A.round == 0) {
            const int within = t.listed_within(G, sm);
            if (act && t.ok && gl == 0) {
                n_open += open;
                n_second += A.k_first > 0 && within > A.k_first;
            }
        }
        // the results of an open cell stand unless a generator beyond the list
        // turns out to cut it
        const int64_t out_idx = A.index_space == VT_INDEX_ORIGINAL ? (int64_t)__float_as_int(pi.w) : (int64_t)q;
        trace_finish<Real, TT, T::NP, NV, PER>(sm, G, act && t.ok ? t.V : 0, t.faces, t.R2, pi, out_idx, A);
        const bool failed = act && !t.ok;
        if (!__any_sync(TFULL, open || failed)) continue;
        if (failed && gl == 0 && t.outgrown()) atomicAdd(&A.st->capacity_events, 1ull);
        append(A.open_list, A.open_ctr, open && gl == 0, q, G.lane);
        append(A.tail_list, A.tail_ctr, failed && gl == 0, q, G.lane);
        const unsigned closes = __ballot_sync(TFULL, gl == 0 && close);
        if (closes && G.lane == 0) atomicAdd(A.close_ctr, __popc(closes));
        // its faces, or all planes of a failed one
        const int F = t.faces.count();
        if (open)
            for (int i = gl; i < F; i += TT) h->src[vt_ck(i, 40, CK_PLANE, A.st)] = sm.src[t.plane_ck(t.faces.nth(i))];
        if (failed && A.round == 0)
            for (int p = gl; p < P; p += TT) h->src[p] = sm.src[p];
        const int nf = far_vertices<TT>(G, sm, open, t.V, reach, h->far, NV, A.st);
        if ((open || failed) && gl == 0) {
            h->np = open ? F : P;
            h->nf = nf;
            h->turns = A.round + (open ? 1 : 0);
            h->close = close;
            h->reach = reach;
            h->all2 = 4.0f * FAR_R2 * t.R2;
        }
        __syncwarp();
    }
    if (gl == 0 && n_open) atomicAdd(&A.st->n_open, (int)n_open);
    if (gl == 0 && n_second) atomicAdd(&A.st->n_second, (int)n_second);
}

// Whole cells by a warp each: traced, walked, and traced again with what cut
// them until nothing does. The cells that k_trace failed or that are still cut
// after its rounds, and every cell of a small call, whose time is the latency
// of one cell: one launch where the rounds take five, and rays over three rows
// of 32 planes instead of five of 8. A cell comes out the same bit for bit from
// either kernel.
constexpr int TAIL_BLOCK = 128;
constexpr int TAIL_TURNS = 64;
// close vertices of a cell in a call whose cells all run here, with no count to go by, from
// which it is taken as one of a lattice (one degenerate vertex of a generic cloud gives at
// most three; from 8 on, rare cells of filaments went to the clipper that it cannot
// validate): 8,000 points moved by 1e-5, 2.5 -> 1.6 ms
constexpr int MANY_CLOSE = 10;
constexpr int TAIL_KEEP = 32;  // cutting generators taken at once from the third turn on
template <typename Real, bool PER>
struct TailSmem {
    typename Tracer<Real, 32, 3, 128, PER>::S t;
    double pd[96][4];  // planes in FP64, when float32 does not settle a cell
    float4 far[128];   // far vertices; before that the low halves of FP64 positions
    int32_t src[96];
    float key[CUT_LIST];
    int32_t id[CUT_LIST];
};
template <typename Real, bool PER>
__global__ void __launch_bounds__(TAIL_BLOCK, 4) k_trace_tail(const __grid_constant__ TraceArgs A)
{
    constexpr int TT = 32, NR = 3, NV = 128;
    using T = Tracer<Real, TT, NR, NV, PER>;
    constexpr bool F64 = T::F64;
    static_assert(REC_FACES + TAIL_KEEP <= T::NP && NV <= REC_VERTS && TAIL_KEEP + 32 <= CUT_LIST, "capacities");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Sub<TT> G;
    const int lane = G.lane;
    TailSmem<Real, PER>& m = reinterpret_cast<TailSmem<Real, PER>*>(smem_raw)[threadIdx.x / 32];
    int nq = (int)A.nq;
    if (A.nq_dev) {
        const int have = *A.nq_dev;
        nq = have < nq ? have : nq;
    }
    int begin = 0;
    if (A.from_dev) begin = ::max(*A.from_dev, A.from);
    unsigned walks = 0, cands = 0, n_open = 0, n_second = 0, rechecks = 0;
    // so many cells of the call have close vertices (a lattice whose points moved
    // little): the clipper is faster than FP64 rays. 125,000 points of a cubic lattice
    // moved by 1e-5 of the spacing: 24.6 -> 8.5 ms (clipper alone 7.8), FP64 form 30.9 ->
    // 17.8 (16.7); by 1e-4 9.0 -> 3.8 (3.0), 11.6 -> 9.9 (14.0). Such cells are 0.02 to
    // 0.1% of uniform and clumped clouds, 1.4% and 0.4% (FP64) of that lattice moved by
    // 1e-2, 12 and 4% by 1e-3, 75 and 44% by 1e-4: the line lies at 1/16 in the FP32
    // form and at 1/4 in the FP64 form, whose clipper takes five times as long.
    const bool regular = A.round > 0 && *A.close_ctr > A.close_max;
    for (;;) {
        int c = 0;
        if (lane == 0) c = begin + atomicAdd(A.queue, 1);
        c = __shfl_sync(TFULL, c, 0);
        if (c >= nq) break;
        const int q = A.queries ? A.queries[c] : (int)A.first + c;
        const GridDesc& grid = grid_of(A.g, A.sets, A.set_of, q);
        const float4 pi = A.sorted[q];
        const OpenCell* h = reinterpret_cast<const OpenCell*>(A.state + (size_t)(A.kept ? c : q - A.first) * A.state_stride);
        if (regular && h->close) {
            if (lane == 0) A.slow_list[atomicAdd(A.slow_ctr, 1)] = q;
            continue;
        }
        int P;
        float reach;
        if (A.round == 0) {
            P = 6 + A.kc;
            reach = A.reach[c];
            for (int p = lane; p < P; p += TT) {
                const int src = p < 6 ? -(p + 1) : A.nbr[(int64_t)c * A.kstride + p - 6];
                m.src[p] = p >= 6 && src < 0 ? PAD_PLANE : src;
            }
        } else {
            P = h->np;
            reach = h->reach;
            for (int p = lane; p < P; p += TT) m.src[p] = h->src[p];
        }
        const bool all = reach == FLT_MAX;
        __syncwarp();
        T t;
        t.st = A.st;
        t.rows = NR;
        bool done = false, spread = false;
        // (every turn adds a generator that cuts. Cells of filaments take tens of turns, and
        // the clipper cannot validate all of those: of 9,000 points 56 cells stayed
        // unvalidated with 16 turns, 54 with 64 or 200. What has not ended after 64 is a
        // cell whose planes all pass within round-off of one point: 5,000 points of a
        // sphere 268 ms FP32 and 157 FP64 with 200 turns, 183 and 76 with 64, 134 and 31
        // with 16, 137 and 35 by the clipper alone)
#pragma unroll 1
        for (int turn = A.round == 0 ? 0 : h->turns; turn < TAIL_TURNS && !done; ++turn) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const int p = r * TT + lane;
                t.set_plane(m.t, r, p, p < P ? m.src[p] : PAD_PLANE, pi, grid, A.sorted);
            }
            __syncwarp();
            const unsigned gen0 = G.ballot(m.t.src[lane] >= 0);
            const int f0 = gen0 ? __ffs(gen0) - 1 : 0;
            if (!T::in_range(m.t, f0)) break;
            t.template trace<float>(G, m.t, gen0 != 0, f0, nullptr, nullptr);
            const bool traced = t.ok;
            t.solve(G, m.t, pi, grid, A.sorted, T::UNIT_F64, T::UNIT_MIN);
            t.certify(G, m.t);
            const int tied = t.ok ? 0 : t.tied(G, m.t, A.sorted, pi, grid, reach, A.round == 0 ? MANY_CLOSE : INT_MAX);
            if (tied == 2) break;  // degenerate: nothing the rest of the turn could certify
            if (turn == 0 && !t.ok && !all && !spread && !(traced && tied)) {
                // most often a list to one side of its generator
                spread = true;
                float r = reach;
                const float lx = grid.hi[0] - grid.lo[0], ly = grid.hi[1] - grid.lo[1], lz = grid.hi[2] - grid.lo[2];
                const int ns = walk<PER, true>(A, grid, q, pi, nullptr, 0, m.t.src, P, 1.01f * (lx * lx + ly * ly + lz * lz),
                                               0, r, m.key, m.id, cands);
                if (lane < ns) m.src[t.plane_ck(P + lane)] = m.id[lane];
                P += ns;
                --turn;
                __syncwarp();
                continue;
            }
            if (!t.ok) {
                // what float32 does not settle: every vertex and every close
                // decision in FP64, then the rays as well
                for (int p = lane; p < T::NP; p += TT) {
                    P64 d = {0.0, 0.0, 0.0, 1.0};
                    if (m.t.src[p] != PAD_PLANE) d = plane64<PER>(m.t.src[p], A.sorted, pi, grid);
                    m.pd[p][0] = d.x;
                    m.pd[p][1] = d.y;
                    m.pd[p][2] = d.z;
                    m.pd[p][3] = d.b;
                }
                __syncwarp();
            }
#pragma unroll 1
            for (int again = traced ? 0 : 1; again < 2 && !t.ok; ++again) {
                if (again == 1) {
                    if (!F64 && lane == 0) atomicAdd(&A.st->precision_events, 1ull);
                    t.template trace<double>(G, m.t, gen0 != 0, f0, m.pd, m.far);
                } else {
                    t.ok = true;
                }
                t.solve(G, m.t, pi, grid, A.sorted, 2.0f, again == 0 ? T::UNIT_MIN : -1.0f, m.far);
                t.certify64(G, m.t, m.pd, m.far, rechecks);
            }
            if (!t.ok || t.faces.count() > REC_FACES) break;
            bool valid = all;
            if (turn == 0) {
                valid = all || 4.0f * FAR_R2 * t.R2 <= reach;
                n_open += !valid;
                n_second += A.k_first > 0 && t.listed_within(G, m.t) > A.k_first;
                walks += !valid;
            }
            const float all2 = 4.0f * FAR_R2 * t.R2;
            if (!valid && all2 > reach) {
                const int F = t.faces.count();
                const int nf = far_vertices<TT>(G, m.t, true, t.V, reach, m.far, NV, A.st);
                __syncwarp();
                const int ns = walk<PER, false>(A, grid, q, pi, m.far, nf, m.t.src, P, all2,
                                         turn < TRACE_ROUNDS ? TRACE_KEEP : TAIL_KEEP, reach, m.key, m.id, cands);
                if (ns > 0) {
                    __syncwarp();
                    for (int i = lane; i < F; i += TT) m.src[i] = m.t.src[t.plane_ck(t.faces.nth(i))];
                    if (lane < ns) m.src[t.plane_ck(F + lane)] = m.id[lane];
                    P = F + ns;
                    __syncwarp();
                    continue;
                }
            }
            done = true;
        }
        const int64_t out_idx = A.index_space == VT_INDEX_ORIGINAL ? (int64_t)__float_as_int(pi.w) : (int64_t)q;
        if (done)
            trace_finish<Real, TT, T::NP, NV, PER>(m.t, G, t.V, t.faces, t.R2, pi, out_idx, A);
        else if (lane == 0) {
            A.slow_list[atomicAdd(A.slow_ctr, 1)] = q;
            if (!t.ok && t.outgrown()) atomicAdd(&A.st->capacity_events, 1ull);
        }
        __syncwarp();
    }
    if (!F64) rechecks = __reduce_add_sync(TFULL, rechecks);
    if (lane == 0) {
        if (!F64 && rechecks) atomicAdd(&A.st->fp64_rechecks, (unsigned long long)rechecks);
        if (walks) atomicAdd(&A.st->walk_cells, (unsigned long long)walks);
        if (cands) atomicAdd(&A.st->walk_cands, (unsigned long long)cands);
        if (n_open) atomicAdd(&A.st->n_open, (int)n_open);
        if (n_second) atomicAdd(&A.st->n_second, (int)n_second);
    }
}

// the state slots of the tail cells a part added, from its slots (A.state) to
// the kept ones (by place in the tail list, the first cap)
__global__ void __launch_bounds__(256) k_keep_tail(const __grid_constant__ TraceArgs A, const int32_t* __restrict__ before,
                                                   uint8_t* __restrict__ kept, int cap)
{
    constexpr int W = (int)(sizeof(OpenCell) + 15) / 16;
    const int i0 = *before, have = *A.tail_ctr, i1 = have < cap ? have : cap;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)(i1 - i0) * W;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int i = i0 + (int)(t / W), w = (int)(t % W);
        const int q = A.tail_list[i];
        reinterpret_cast<uint4*>(kept + (size_t)i * A.state_stride)[w] =
            reinterpret_cast<const uint4*>(A.state + (size_t)(q - A.first) * A.state_stride)[w];
    }
}

// as many blocks as are resident at once (they take cells from the queue)
template <typename K>
cudaError_t resident_blocks(K kern, int block, size_t smem, int64_t cells, int per_block, unsigned& blocks)
{
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int dev = 0, sms = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, smem);
    if (e != cudaSuccess) return e;
    const int64_t want = (cells + per_block - 1) / per_block, resident = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    blocks = (unsigned)(want < resident ? (want > 0 ? want : 1) : resident);
    return cudaSuccess;
}

template <typename Real>
cudaError_t launch_trace_t(const TraceArgs& a, cudaStream_t s)
{
    unsigned blocks = 1;
    if (a.tail) {
        auto kern = a.g.periodic ? k_trace_tail<Real, true> : k_trace_tail<Real, false>;
        const size_t smem = sizeof(TailSmem<Real, false>) * (TAIL_BLOCK / 32);
        const cudaError_t e = resident_blocks(kern, TAIL_BLOCK, smem, a.nq, TAIL_BLOCK / 32, blocks);
        if (e != cudaSuccess) return e;
        kern<<<blocks, TAIL_BLOCK, smem, s>>>(a);
    } else {
        auto kern = a.g.periodic ? k_trace<Real, true> : k_trace<Real, false>;
        const size_t smem = trace_stride<typename Tracer<Real, 8, 5, 48, false>::S>() * (TRACE_BLOCK / 8);
        const cudaError_t e = resident_blocks(kern, TRACE_BLOCK, smem, a.nq, TRACE_BLOCK / 8, blocks);
        if (e != cudaSuccess) return e;
        kern<<<blocks, TRACE_BLOCK, smem, s>>>(a);
    }
    count_launch();
    return cudaGetLastError();
}

}  // namespace

}  // namespace vt
