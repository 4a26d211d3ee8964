// adjoint.cu -- gradient of the per-cell moments (volume V_i, centroid c_i,
// second moment M2_i = integral over C_i of |x - p_i|^2) with respect to
// the generators, for Lloyd relaxation and other losses of the cells.
//
// For upstream gradients (gV_i, gC_i, gM_i) cell i carries the density
//     h_i(x) = gV_i + gC_i . (x - c_i) / V_i + gM_i |x - p_i|^2
// and grad_k = 2 gM_k V_k (p_k - c_k)                                (interior)
//            + sum over faces f of cell k, neighbour j, d = |p_j - p_k|:
//                (1/d) integral_f h_k(x) (x - p_k) dA               (face of k moves with p_k)
//              + (1/d) integral_f h_j(x) (p_k - x) dA               (face of j moves with p_k)
// (a face on the bisector moves along its normal with speed (x - p_k).dp_k / d
// seen from cell k and (p_k - x).dp_k / d seen from cell j; walls are fixed).
//
// Everything is integrated in the frame of p_k (y = x - p_k). On the shared
// face |x - p_j| = |x - p_k| = |y|, so both densities read a + b.y + g |y|^2
// there (each density's constant absorbs b.(p_k - c)), and one set of face
// moments -- M1, M2, Q1 of y, y y^T, |y|^2 y -- serves both.
// The moments are exact sums over the face's triangle fan: with S = A + B + C,
// the integrals over a triangle of y, y y^T and |y|^2 y are the area times
//   S / 3,  (S S^T + sum v v^T) / 12  and
//   (S (|S|^2 + sum |v|^2) + 2 sum v (v.S + |v|^2)) / 60   (sums over A, B, C),
// half the operations of a 7-point rule. Gather form: 8 lanes per cell, a lane
// per face, sum every contribution to the cell's own generator (deterministic,
// no atomics). The face integrals run in the precision of the tessellation
// (float32 for the FP32 form: the FP64 rate of the part is 1/64 of float32; the
// local frame keeps the values small), the sums over a cell's faces and across the
// lanes as in FP64 (FaceSum).
//
// Bound by the FP64 pipe even in the FP32 form (positions and centroids become
// differences from the generator in FP64): a warp per cell converted every
// vertex once per face and triangle and added over 32 lanes; here the cell's
// vertices are converted once into shared memory and four cells share an
// instruction (54 FP64 instructions per cell, the pipe 88% busy). 1M cells half
// in clumps: 7.38 -> 3.40 ms.
//
// Periodic box: the neighbour across a face is an image p_j + t L. The face
// lies on the bisector of p_k and that image, so the image is the reflection
// of p_k across the face's plane; t is that reflection minus p_j over L,
// rounded (the plane comes from the face's own vertices: its area vector
// and its first vertex). Cell j's density is then read through the same
// image (its centroid shifted by t L).
#include "vt_internal.cuh"

namespace vt {

namespace {

template <typename Real>
struct Dens {
    Real a, bx, by, bz, g;  // h(y) = a + b.y + g |y|^2 in the frame of p_k
};

// density of cell i written in the frame of the point (px, py, pz)
template <typename Real>
__device__ __forceinline__ Dens<Real> density(int i, double px, double py, double pz, const double* vol,
                                              const double* cen, const double* gV, const double* gC, const double* gM)
{
    Dens<Real> d;
    d.g = gM ? (Real)gM[i] : (Real)0;
    d.bx = d.by = d.bz = (Real)0;
    d.a = gV ? (Real)gV[i] : (Real)0;
    if (gC) {  // gV + b.(x - c) with x = y + p, b = gC / V
        const Real V = (Real)vol[i];  // (divided, not times a reciprocal: one rounding; 1M cells, FP64: 30.1 -> 30.8 ms)
        d.bx = (Real)gC[3 * i] / V;
        d.by = (Real)gC[3 * i + 1] / V;
        d.bz = (Real)gC[3 * i + 2] / V;
        d.a += d.bx * (Real)(px - cen[3 * i]) + d.by * (Real)(py - cen[3 * i + 1]) +
               d.bz * (Real)(pz - cen[3 * i + 2]);
    }
    return d;
}

// integral over the face of h y, from the face moments
template <typename Real>
__device__ __forceinline__ void face_term(const Dens<Real>& h, const Real* M1, const Real* M2, const Real* Q1,
                                          Real* out)
{
    out[0] = h.a * M1[0] + M2[0] * h.bx + M2[1] * h.by + M2[2] * h.bz + h.g * Q1[0];
    out[1] = h.a * M1[1] + M2[1] * h.bx + M2[3] * h.by + M2[4] * h.bz + h.g * Q1[1];
    out[2] = h.a * M1[2] + M2[2] * h.bx + M2[4] * h.by + M2[5] * h.bz + h.g * Q1[2];
}

// A sum over faces: in float32 with the rounding of every addition kept beside it
// (Knuth's two-sum), so that only the faces' own terms round in float32, as if
// they were added in FP64. The FP64 pipe bounds this kernel: FP64 additions would
// be 6 more of its instructions per face, this is 18 float32 ones. 1M cells half
// in clumps, whole backward pass: 3.81 ms with plain float32 sums, 3.89 so.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
template <typename Real>
struct FaceSum {
    Real s = 0, r = 0;
    __device__ __forceinline__ void add(Real x)
    {
        const Real t = add_rn(s, x);
        if (sizeof(Real) == 4) {
            const Real b = add_rn(t, -s);
            r = add_rn(r, add_rn(add_rn(s, -add_rn(t, -b)), add_rn(x, -b)));
        }
        s = t;
    }
    __device__ __forceinline__ double sum() const { return sizeof(Real) == 4 ? (double)s + (double)r : (double)s; }
};

constexpr int ADJ_BLOCK = 128;
constexpr int ADJ_T = 8;        // lanes per cell
constexpr int ADJ_V = 64;       // vertices of a cell kept in shared memory
template <typename Real, bool PER>
__global__ void __launch_bounds__(ADJ_BLOCK) k_adjoint(const float* __restrict__ pts, int64_t n,
                                                 const double* __restrict__ vol, const double* __restrict__ cen,
                                                 const int64_t* __restrict__ vtx_off, const double* __restrict__ vtx,
                                                 const int64_t* __restrict__ face_off,
                                                 const int32_t* __restrict__ face_nbr,
                                                 const int64_t* __restrict__ face_vtx_off,
                                                 const int32_t* __restrict__ face_vtx, const double* __restrict__ gV,
                                                 const double* __restrict__ gC, const double* __restrict__ gM,
                                                 double* __restrict__ grad, const __grid_constant__ GridDesc box)
{
    __shared__ Real s_v[ADJ_BLOCK / ADJ_T][3][ADJ_V];
    const double Lx = (double)box.hi[0] - (double)box.lo[0], Ly = (double)box.hi[1] - (double)box.lo[1],
                 Lz = (double)box.hi[2] - (double)box.lo[2];
    const int gl = threadIdx.x & (ADJ_T - 1);
    Real(*sv)[ADJ_V] = s_v[threadIdx.x / ADJ_T];
    const int64_t per_grid = (int64_t)gridDim.x * (ADJ_BLOCK / ADJ_T);
    // (whole warps step together: a group past the end repeats the last cell)
    const int64_t first = (int64_t)blockIdx.x * (ADJ_BLOCK / ADJ_T) + threadIdx.x / ADJ_T;
    for (int64_t c = first; c - threadIdx.x / ADJ_T % (32 / ADJ_T) < n; c += per_grid) {
        const int64_t k = c < n ? c : n - 1;
        const float fx = pts[3 * k], fy = pts[3 * k + 1], fz = pts[3 * k + 2];
        const double px = fx, py = fy, pz = fz;
        const Dens<Real> hk = density<Real>((int)k, px, py, pz, vol, cen, gV, gC, gM);
        const double* V = vtx + 3 * vtx_off[k];
        const int nv = (int)(vtx_off[k + 1] - vtx_off[k]);
        // the cell's vertices in the frame of p_k
        __syncwarp();
        for (int s = gl; s < nv && s < ADJ_V; s += ADJ_T) {
            sv[0][s] = (Real)(V[3 * s] - px);
            sv[1][s] = (Real)(V[3 * s + 1] - py);
            sv[2][s] = (Real)(V[3 * s + 2] - pz);
        }
        __syncwarp();
        auto vert = [&](int s, Real& x, Real& y, Real& z) {
            if (s < ADJ_V) {
                x = sv[0][s];
                y = sv[1][s];
                z = sv[2][s];
            } else {
                x = (Real)(V[3 * s] - px);
                y = (Real)(V[3 * s + 1] - py);
                z = (Real)(V[3 * s + 2] - pz);
            }
        };
        FaceSum<Real> gx, gy, gz;
        const int64_t f0 = face_off[k], f1 = face_off[k + 1];
        for (int64_t f = f0 + gl; f < f1; f += ADJ_T) {
            const int j = face_nbr[f];
            if (j < 0) continue;  // walls do not move
            // area-weighted sums of S, of S S^T + sum v v^T and of the cubic term
            Real M1[3] = {0, 0, 0}, M2[6] = {0, 0, 0, 0, 0, 0}, Q1[3] = {0, 0, 0};
            const int32_t* loop = face_vtx + face_vtx_off[f];
            const int deg = (int)(face_vtx_off[f + 1] - face_vtx_off[f]);
            Real A[3], B[3];
            vert(loop[0], A[0], A[1], A[2]);
            vert(loop[1], B[0], B[1], B[2]);
            const Real aa = A[0] * A[0] + A[1] * A[1] + A[2] * A[2];
            Real bb = B[0] * B[0] + B[1] * B[1] + B[2] * B[2];
            Real sx = 0, sy = 0, sz = 0;  // twice the face's area vector (outward)
            for (int t = 1; t + 1 < deg; ++t) {
                Real C[3];
                vert(loop[t + 1], C[0], C[1], C[2]);
                const Real ux = B[0] - A[0], uy = B[1] - A[1], uz = B[2] - A[2];
                const Real vx = C[0] - A[0], vy = C[1] - A[1], vz = C[2] - A[2];
                const Real cx = uy * vz - uz * vy, cy = uz * vx - ux * vz, cz = ux * vy - uy * vx;
                const Real area = sqrt(cx * cx + cy * cy + cz * cz);  // (twice)
                sx += cx;
                sy += cy;
                sz += cz;
                const Real x = A[0] + B[0] + C[0], y = A[1] + B[1] + C[1], z = A[2] + B[2] + C[2];
                const Real cc = C[0] * C[0] + C[1] * C[1] + C[2] * C[2];
                M1[0] += area * x;
                M1[1] += area * y;
                M1[2] += area * z;
                M2[0] += area * (x * x + A[0] * A[0] + B[0] * B[0] + C[0] * C[0]);
                M2[1] += area * (x * y + A[0] * A[1] + B[0] * B[1] + C[0] * C[1]);
                M2[2] += area * (x * z + A[0] * A[2] + B[0] * B[2] + C[0] * C[2]);
                M2[3] += area * (y * y + A[1] * A[1] + B[1] * B[1] + C[1] * C[1]);
                M2[4] += area * (y * z + A[1] * A[2] + B[1] * B[2] + C[1] * C[2]);
                M2[5] += area * (z * z + A[2] * A[2] + B[2] * B[2] + C[2] * C[2]);
                const Real w = x * x + y * y + z * z + aa + bb + cc;
                const Real wa = (Real)2 * (A[0] * x + A[1] * y + A[2] * z + aa);
                const Real wb = (Real)2 * (B[0] * x + B[1] * y + B[2] * z + bb);
                const Real wc = (Real)2 * (C[0] * x + C[1] * y + C[2] * z + cc);
                Q1[0] += area * (w * x + wa * A[0] + wb * B[0] + wc * C[0]);
                Q1[1] += area * (w * y + wa * A[1] + wb * B[1] + wc * C[1]);
                Q1[2] += area * (w * z + wa * A[2] + wb * B[2] + wc * C[2]);
                B[0] = C[0];
                B[1] = C[1];
                B[2] = C[2];
                bb = cc;
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                M1[i] *= (Real)(1.0 / 6.0);
                Q1[i] *= (Real)(1.0 / 120.0);
            }
#pragma unroll
            for (int i = 0; i < 6; ++i) M2[i] *= (Real)(1.0 / 24.0);
            double ox = 0.0, oy = 0.0, oz = 0.0;  // t L of the image across the face
            if (PER) {
                // reflection of p_k across the face plane: 2 (n.A) n, n the unit normal
                const double sn = sqrt((double)sx * sx + (double)sy * sy + (double)sz * sz);
                if (sn > 0.0) {
                    const double nx = sx / sn, ny = sy / sn, nz = sz / sn;
                    const double h2 = 2.0 * (nx * (double)A[0] + ny * (double)A[1] + nz * (double)A[2]);
                    ox = rint((px + h2 * nx - (double)pts[3 * (int64_t)j]) / Lx) * Lx;
                    oy = rint((py + h2 * ny - (double)pts[3 * (int64_t)j + 1]) / Ly) * Ly;
                    oz = rint((pz + h2 * nz - (double)pts[3 * (int64_t)j + 2]) / Lz) * Lz;
                }
            }
            const float qx = pts[3 * (int64_t)j], qy = pts[3 * (int64_t)j + 1], qz = pts[3 * (int64_t)j + 2];
            Real dx, dy, dz;
            if (PER) {
                dx = (Real)(((double)qx - px) + ox);
                dy = (Real)(((double)qy - py) + oy);
                dz = (Real)(((double)qz - pz) + oz);
            } else {  // (the difference of two floats rounds the same in float32)
                dx = (Real)qx - (Real)fx;
                dy = (Real)qy - (Real)fy;
                dz = (Real)qz - (Real)fz;
            }
            const Real inv_d = (Real)1 / sqrt(dx * dx + dy * dy + dz * dz);
            // cell j seen through its image: its density in the frame of p_k - t L
            const Dens<Real> hj = PER ? density<Real>(j, px - ox, py - oy, pz - oz, vol, cen, gV, gC, gM)
                                      : density<Real>(j, px, py, pz, vol, cen, gV, gC, gM);
            Real own[3], nbr[3];
            face_term(hk, M1, M2, Q1, own);  // integral of h_k y
            face_term(hj, M1, M2, Q1, nbr);  // integral of h_j y
            gx.add((own[0] - nbr[0]) * inv_d);
            gy.add((own[1] - nbr[1]) * inv_d);
            gz.add((own[2] - nbr[2]) * inv_d);
        }
        // FP64 sums over the 8 lanes by reduce-scatter: lanes 0, 2 and 4 end with
        // the x, y and z components
        const bool hi1 = (gl & 4) != 0, hi2 = (gl & 2) != 0;
        const double dx = gx.sum(), dy = gy.sum(), dz = gz.sum();
        const double p0 = (hi1 ? dz : dx) + __shfl_xor_sync(0xffffffffu, hi1 ? dx : dz, 4);
        const double p1 = (hi1 ? 0.0 : dy) + __shfl_xor_sync(0xffffffffu, hi1 ? dy : 0.0, 4);
        double w = (hi2 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, hi2 ? p0 : p1, 2);
        w += __shfl_xor_sync(0xffffffffu, w, 1);
        if (c < n && (gl == 0 || gl == 2 || gl == 4)) {
            const int a = gl >> 1;
            const double s = 2.0 * (gM ? gM[k] : 0.0) * vol[k];  // interior term of M2: 2 gM V (p - c)
            grad[3 * k + a] = w + s * ((a == 0 ? px : (a == 1 ? py : pz)) - cen[3 * k + a]);
        }
    }
}

// Lloyd's update written as a gradient step on the energy sum_i M2_i:
// p <- p - g / (2 V) with g = d(sum M2)/dp = 2 V (p - c), which lands on the
// centroid (Lloyd 1982), in FP64 and rounded once to float32. In a periodic
// box the new point is moved by whole periods into [lo, hi) (in FP64 from the
// rounded value, rounded again; a value that rounds onto hi belongs at lo);
// in a walled box a value that rounds onto hi is moved to the largest float
// below it, so the next tessellation gets a valid point.
__global__ void k_lloyd_step(const float* __restrict__ pts, int64_t n, const double* __restrict__ grad,
                             const double* __restrict__ vol, GridDesc g, float* __restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = i / 3;
        const int a = (int)(i - 3 * k);
        const double lo = (double)g.lo[a], hi = (double)g.hi[a];
        float x = (float)((double)pts[i] - grad[i] / (2.0 * vol[k]));
        if (g.periodic) {
            const double L = hi - lo, xd = (double)x;
            x = (float)(xd - floor((xd - lo) / L) * L);
            if (x >= g.hi[a]) x = g.lo[a];
        } else if (x >= g.hi[a]) {
            x = nextafterf(g.hi[a], g.lo[a]);
        }
        out[i] = x;
    }
}

}  // namespace

cudaError_t launch_lloyd_step(const float* pts, int64_t n, const double* grad, const double* vol, const GridDesc& g,
                              float* out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (3 * n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_lloyd_step<<<(unsigned)blocks, 256, 0, s>>>(pts, n, grad, vol, g, out);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_adjoint(const float* pts, int64_t n, const vt_cells_out& c, const double* gV, const double* gC,
                           const double* gM, double* grad, int precision, const GridDesc& g, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n + ADJ_BLOCK / ADJ_T - 1) / (ADJ_BLOCK / ADJ_T);
    if (blocks > 152 * 64) blocks = 152 * 64;
    auto kern = precision == VT_FP64 ? (g.periodic ? k_adjoint<double, true> : k_adjoint<double, false>)
                                     : (g.periodic ? k_adjoint<float, true> : k_adjoint<float, false>);
    kern<<<(unsigned)blocks, ADJ_BLOCK, 0, s>>>(pts, n, c.vol, c.cen, c.vtx_off, c.vtx, c.face_off, c.face_nbr,
                                                c.face_vtx_off, c.face_vtx, gV, gC, gM, grad, g);
    count_launch();
    return cudaGetLastError();
}

}  // namespace vt
