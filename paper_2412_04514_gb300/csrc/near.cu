// near.cu -- neighbour lists of the traced pass: the generators near each
// generator, unordered.
//
// The edge tracing (trace_impl.cuh) needs a set of close generators, its
// nearest first, and a reach: every generator with a float key below it is in
// the list. It needs no order, so nothing is sorted. A warp per generator
// estimates the radius that holds about NEAR_AIM generators from the 3^3 grid
// cells around it, takes the rows of the grid that meet that ball (a lane per
// row finds its run, then the lanes share the runs' generators), and collects
// those inside. A clump that overfills the buffer lowers the limit to the key
// that keeps a list's length, found by bisection on the key bits with two
// ballots a step; a void that leaves fewer than five eighths of a list starts
// over with a larger radius.
//
// Bound by instruction issue (109 generators read per query of uniform points,
// 324 where half the points lie in clumps). A sorted list (knn.cu) costs 2,650
// warp instructions per query of uniform points, most of them bitonic sorts
// and three rounds of shell set-up. 1M points: uniform 2.86 -> 0.92 ms, half in
// clumps 3.73 -> 1.68 ms, FP64 form 5.42 -> 1.69 ms (the lists' exact FP64 keys
// are not needed either: 2R against the reach is decided with a margin, and
// closer calls go to the walk). A list one short of the 32 asked for costs a
// bisection step less and leaves 1% more cells to the walk: 7.53 ms for lists
// and cells together, as with 32 exactly (7.49); three short 7.72 ms.
#include <float.h>

#include "vt_internal.cuh"

namespace vt {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int NEAR_BLOCK = 128;
constexpr int NEAR_BUF = 96;     // collected generators: 64 and a batch
constexpr float NEAR_AIM = 38.0f;  // (34: 0.04 ms less here, 0.15 ms more in the cells at 1M)
constexpr int NEAR_TURNS = 48;

// A limit below which k - 1 or k of the warp's cnt (at most 96) keys
// lie, as far as ties allow, never more than k; the keys are float bits
__device__ __forceinline__ unsigned limit_of(const float* key, int cnt, unsigned hi, int k, int lane)
{
    const unsigned a = lane < cnt ? __float_as_uint(key[lane]) : 0xffffffffu;
    const unsigned b = lane + 32 < cnt ? __float_as_uint(key[lane + 32]) : 0xffffffffu;
    const unsigned c = lane + 64 < cnt ? __float_as_uint(key[lane + 64]) : 0xffffffffu;
    unsigned lo = 0u, mid = __float_as_uint(0.7f * __uint_as_float(hi));
#pragma unroll 1
    while (hi - lo > 1u) {
        const int n = __popc(__ballot_sync(FULL, a < mid)) + __popc(__ballot_sync(FULL, b < mid)) +
                      __popc(__ballot_sync(FULL, c < mid));
        if (n > k) {
            hi = mid;
        } else {
            lo = mid;
            if (n >= k - 1) break;
        }
        mid = lo ? lo + (hi - lo) / 2u : __float_as_uint(0.5f * __uint_as_float(hi));
        if (mid <= lo || mid >= hi) mid = lo + (hi - lo) / 2u;
    }
    return lo;
}

// keeps the keys below the limit, in order; returns their count
__device__ __forceinline__ int keep_below(float* key, int32_t* id, int cnt, float lim, int lane)
{
    int out = 0;
#pragma unroll 1
    for (int i0 = 0; i0 < cnt; i0 += 32) {
        const float d = i0 + lane < cnt ? key[i0 + lane] : FLT_MAX;
        const int j = i0 + lane < cnt ? id[i0 + lane] : -1;
        const bool in = d < lim;
        const unsigned m = __ballot_sync(FULL, in);
        __syncwarp();
        if (in) {
            key[out + __popc(m & ((1u << lane) - 1u))] = d;
            id[out + __popc(m & ((1u << lane) - 1u))] = j;
        }
        out += __popc(m);
        __syncwarp();
    }
    return out;
}

template <bool PER>
__global__ void __launch_bounds__(NEAR_BLOCK) k_near(const float4* __restrict__ sorted,
                                                     const int32_t* __restrict__ cell_off0,
                                                     const __grid_constant__ GridDesc g0,
                                                     const GridDesc* __restrict__ sets,
                                                     const int32_t* __restrict__ set_of, int first, int n, int k,
                                                     int kstride,
                                                     int32_t* __restrict__ nbr, float* __restrict__ reach_out,
                                                     DevStatus* st, int32_t* __restrict__ queue)
{
    __shared__ float s_key[NEAR_BLOCK / 32][NEAR_BUF];
    __shared__ int32_t s_id[NEAR_BLOCK / 32][NEAR_BUF];
    const int lane = threadIdx.x & 31;
    float* key = s_key[threadIdx.x >> 5];
    int32_t* id = s_id[threadIdx.x >> 5];
    unsigned long long evals = 0, answered = 0;
    for (;;) {
        int c = 0;
        if (lane == 0) c = atomicAdd(queue, 1);
        c = __shfl_sync(FULL, c, 0);
        if (c >= n) break;
        const int q = first + c;
        ++answered;
        const float4 pq = sorted[q];
        const GridDesc& g = grid_of(g0, sets, set_of, q);
        const int G = g.G;
        const int32_t* coff = cell_off0 + g.cell_base;
        const int ix = cell_coord(pq.x, g.lo[0], g.scale[0], G), iy = cell_coord(pq.y, g.lo[1], g.scale[1], G),
                  iz = cell_coord(pq.z, g.lo[2], g.scale[2], G);
        const float m = (float)g.margin;
        const float cx = (float)g.cw[0], cy = (float)g.cw[1], cz = (float)g.cw[2];
        const float lx = g.hi[0] - g.lo[0], ly = g.hi[1] - g.lo[1], lz = g.hi[2] - g.lo[2];
        // the farthest a generator can be (periodic: can be and still cut)
        const float far2 = (lx * lx + ly * ly + lz * lz) * (1.0f + 1e-3f);
        float aim2;  // squared radius of the ball
        {
            int have = 0, cells = 0;
            const int x = ix + lane / 3 - 1, y = iy + lane % 3 - 1;
            if (lane < 9 && x >= 0 && x < G && y >= 0 && y < G) {
                const int z0 = iz > 0 ? iz - 1 : 0, z1 = iz < G - 1 ? iz + 1 : G - 1;
                const int base = (x * G + y) * G;
                have = coff[base + z1 + 1] - coff[base + z0];
                cells = z1 - z0 + 1;
            }
            have = __reduce_add_sync(FULL, have);
            cells = __reduce_add_sync(FULL, cells);
            const float r = cbrtf(NEAR_AIM * 0.2387324f * (float)cells / (float)(have > 0 ? have : 1)) * cbrtf(cx) *
                            cbrtf(cy) * cbrtf(cz);
            aim2 = r * r;
        }
        int cnt = 0;
        float lim = 0.0f;
        bool all = false, dup = false;
        // (NEAR_TURNS is never reached by a radius that grows from a normal number)
#pragma unroll 1
        for (int turn = 0;; ++turn) {
            const bool whole = !(aim2 < far2) || turn >= NEAR_TURNS;
            if (whole) aim2 = far2;
            cnt = 0;
            lim = aim2;
            const float rr = sqrtf(aim2 * (1.0f + 1e-4f));
            // periodic: unwrapped grid coordinates, and each row once per z image
            const float lim_lo = PER ? -2.0f * (float)G : 0.0f, lim_hi = PER ? 3.0f * (float)G - 1.0f : (float)G - 1.0f;
            auto clamp = [&](float t) { return (int)floorf(fminf(fmaxf(t, lim_lo), lim_hi)); };
            const int x0 = clamp((pq.x - rr - m - g.lo[0]) * g.scale[0] - 1e-3f);
            const int x1 = clamp((pq.x + rr + m - g.lo[0]) * g.scale[0] + 1e-3f);
            const int y0 = clamp((pq.y - rr - m - g.lo[1]) * g.scale[1] - 1e-3f);
            const int y1 = clamp((pq.y + rr + m - g.lo[1]) * g.scale[1] + 1e-3f);
            int t0 = 0, nt = 1;
            if (PER) {
                t0 = floordiv(clamp((pq.z - rr - m - g.lo[2]) * g.scale[2] - 1e-3f), G);
                nt = floordiv(clamp((pq.z + rr + m - g.lo[2]) * g.scale[2] + 1e-3f), G) - t0 + 1;
            }
            const int wy = y1 - y0 + 1, nrow = (x1 - x0 + 1) * wy * nt;
#pragma unroll 1
            for (int e0 = 0; e0 < nrow; e0 += 32) {
                const int e = e0 + lane;
                int sa = 0, len = 0, code = IMG_NONE;
                if (e < nrow) {
                    const int e2 = PER ? e / nt : e;
                    const int tz = PER ? t0 + (e - e2 * nt) : 0;
                    const int ex = e2 / wy, x = x0 + ex, y = y0 + (e2 - ex * wy);
                    const int tx = PER ? floordiv(x, G) : 0, ty = PER ? floordiv(y, G) : 0;
                    const float gx0 = g.lo[0] + (float)x * cx - m, gx1 = g.lo[0] + (float)(x + 1) * cx + m;
                    const float gy0 = g.lo[1] + (float)y * cy - m, gy1 = g.lo[1] + (float)(y + 1) * cy + m;
                    const float dx = fmaxf(fmaxf(gx0 - pq.x, pq.x - gx1), 0.0f), dy = fmaxf(fmaxf(gy0 - pq.y, pq.y - gy1), 0.0f);
                    const float left = aim2 * (1.0f + 1e-4f) - (dx * dx + dy * dy);
                    if (left >= 0.0f) {
                        const float zr = sqrtf(left) + m;
                        int za = clamp((pq.z - zr - g.lo[2]) * g.scale[2] - 1e-3f);
                        int zb = clamp((pq.z + zr - g.lo[2]) * g.scale[2] + 1e-3f);
                        if (PER) {
                            za = za > tz * G ? za : tz * G;
                            zb = zb < tz * G + G - 1 ? zb : tz * G + G - 1;
                        }
                        if (za <= zb) {
                            const int base = ((x - tx * G) * G + (y - ty * G)) * G - tz * G;
                            sa = coff[base + za];
                            len = coff[base + zb + 1] - sa;
                        }
                        if (PER) code = img_code(tx, ty, tz);
                    }
                }
                int incl = len;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int u = __shfl_up_sync(FULL, incl, d);
                    if (lane >= d) incl += u;
                }
                const int total = __shfl_sync(FULL, incl, 31);
                const int start = incl - len;
                evals += (unsigned)total;
#pragma unroll 1
                for (int c0 = 0; c0 < total; c0 += 32) {
                    const int i = c0 + lane;
                    int seg = 0;  // rows ending at or before i
#pragma unroll
                    for (int step = 16; step >= 1; step >>= 1)
                        if (__shfl_sync(FULL, incl, (seg + step - 1) & 31) <= i) seg += step;
                    const int j = __shfl_sync(FULL, sa, seg & 31) + (i - __shfl_sync(FULL, start, seg & 31));
                    const int cd = PER ? __shfl_sync(FULL, code, seg & 31) : IMG_NONE;
                    bool in = i < total && j != q;
                    float d2 = 0.0f;
                    if (in) {
                        const float4 pc = sorted[j];
                        d2 = key_f32(img_off_t<PER>(pq, pc, cd, g));
                        if (cd == IMG_NONE && pc.x == pq.x && pc.y == pq.y && pc.z == pq.z) dup = true;
                        in = d2 < lim;
                    }
                    const unsigned mask = __ballot_sync(FULL, in);
                    if (!mask) continue;
                    if (in) {
                        const int at = cnt + __popc(mask & ((1u << lane) - 1u));
                        key[vt_ck(at, NEAR_BUF, CK_RECORD, st)] = d2;
                        id[vt_ck(at, NEAR_BUF, CK_RECORD, st)] = PER ? img_pack(j, cd) : j;
                    }
                    cnt += __popc(mask);
                    __syncwarp();
                    if (cnt > 64) {
                        lim = __uint_as_float(limit_of(key, cnt, __float_as_uint(lim), k, lane));
                        cnt = keep_below(key, id, cnt, lim, lane);
                    }
                }
            }
            all = whole && lim == aim2;
            if (!PER && cnt == (int)g.npts - 1) all = true;
            if (all || 8 * cnt >= 5 * k || lim < aim2) break;
            aim2 *= cnt < k / 4 ? 3.0f : 1.7f;
        }
        if (cnt > k) {
            all = false;
            lim = __uint_as_float(limit_of(key, cnt, __float_as_uint(lim), k, lane));
            cnt = keep_below(key, id, cnt, lim, lane);
        }
        if (__any_sync(FULL, dup) && lane == 0) atomicExch((int*)&st->duplicate, 1);
        // the nearest first
        const unsigned ka = lane < cnt ? __float_as_uint(key[lane]) : 0xffffffffu;
        const unsigned kb = lane + 32 < cnt ? __float_as_uint(key[lane + 32]) : 0xffffffffu;
        const unsigned best = __reduce_min_sync(FULL, ::min(ka, kb));
        const unsigned ma = __ballot_sync(FULL, ka == best), mb = __ballot_sync(FULL, kb == best);
        const int at = ma ? __ffs(ma) - 1 : 32 + __ffs(mb) - 1;
        int32_t* out = nbr + (int64_t)c * kstride;
        for (int i = lane; i < k; i += 32) {
            const int from = i == 0 ? at : (i == at ? 0 : i);
            out[i] = i < cnt ? id[vt_ck(from, NEAR_BUF, CK_RECORD, st)] : -1;
        }
        if (lane == 0) reach_out[c] = all ? FLT_MAX : lim;
        __syncwarp();
    }
    if (lane == 0 && answered) {
        atomicAdd(&st->knn_evals, evals);
        atomicAdd(&st->knn_queries, answered);
    }
}

}  // namespace

cudaError_t launch_near(const float4* sorted, const int32_t* cell_off, const GridDesc& g, const GridDesc* sets,
                        const int32_t* set_of, int64_t first, int64_t n, int k, int kstride, int32_t* nbr, float* reach,
                        DevStatus* st, int32_t* queue, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (k < 1 || k > 64) return cudaErrorInvalidValue;
    auto kern = g.periodic ? k_near<true> : k_near<false>;
    // as many blocks as are resident at once (their warps take generators from the counter)
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NEAR_BLOCK, 0);
    if (e == cudaSuccess) e = cudaMemsetAsync(queue, 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    int64_t blocks = (n + NEAR_BLOCK / 32 - 1) / (NEAR_BLOCK / 32);
    const int64_t resident = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    if (blocks > resident) blocks = resident;
    kern<<<(unsigned)blocks, NEAR_BLOCK, 0, s>>>(sorted, cell_off, g, sets, set_of, (int)first, (int)n, k, kstride, nbr,
                                                 reach, st, queue);
    count_launch();
    return cudaGetLastError();
}

}  // namespace vt
