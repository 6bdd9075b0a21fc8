// Pair passes of large, spatially ordered lists, tile by tile (sm_103a).
//
// A list ordered in space (order_kernels.cu) is cut into tiles of 32 particles; a warp takes
// 64 receivers (two tiles, two particles a lane) against the tiles of its share of the sources
// and first looks at each pair of groups through their bounding boxes.
//
// Time-step pass (Sec. 4).  A minimum needs only the pairs that can set it: for most tiles the
// distance of the boxes alone bounds every criterion of every pair from below above the
// receivers' present minima, and the tile is passed over.  The result is the minimum over the
// same FP32 pair values as in the one-sided and the symmetric pass, so the same bits.
// With the sort of the list, Plummer spheres: 65536 particles 3.76 -> 1.06 ms, 40603 1.61 -> 0.52
// ms, 262144 53 -> 7.1 ms (before: the symmetric pass over all pairs).  What is left is latency:
// the judging of items issues about 0.4 of the time.
#include "pair_bodies.cuh"

namespace frost {
namespace {

using namespace dev;

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kInf = 0x7f800000u;

__device__ __forceinline__ float warp_min(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

__device__ __forceinline__ float warp_max(float v)
{
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// The box of a tile, rounded outwards, and what else bounds its pairs
struct TileHead {
    float4 lo;  // {x, y, z, max G m}
    float4 hi;  // {x, y, z, max |v|}
    float4 vc;  // {centre of the velocities, largest |v - centre|}
};

// A lower bound on the squared distance of two boxes
__device__ __forceinline__ float box_gap2(const float4 alo, const float4 ahi, const float4 blo, const float4 bhi)
{
    const float gx = fmaxf(0.f, fmaxf(__fsub_rd(blo.x, ahi.x), __fsub_rd(alo.x, bhi.x)));
    const float gy = fmaxf(0.f, fmaxf(__fsub_rd(blo.y, ahi.y), __fsub_rd(alo.y, bhi.y)));
    const float gz = fmaxf(0.f, fmaxf(__fsub_rd(blo.z, ahi.z), __fsub_rd(alo.z, bhi.z)));
    return __fmaf_rd(gx, gx, __fmaf_rd(gy, gy, __fmul_rd(gz, gz)));
}

// ------------------------------------------------------------------------------------
// time-step pass
// ------------------------------------------------------------------------------------
// Records as launch_pack_tstep_mixed makes them, the x velocities of every tile in ascending
// order (+inf past the end), and the tiles' heads; one tile a warp
__global__ void __launch_bounds__(128) k_tile_pack_tstep(const int32_t *__restrict__ list, int n,
                                                         const double *__restrict__ x, const double *__restrict__ v,
                                                         const double *__restrict__ m, int N, double G,
                                                         float4 *__restrict__ rec, float *__restrict__ vx,
                                                         TileHead *__restrict__ head, unsigned *__restrict__ best)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    if ((k & ~31) >= n) return;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    float vlo[3] = {INFINITY, INFINITY, INFINITY}, vhi[3] = {-INFINITY, -INFINITY, -INFINITY};
    float gm = 0.f, vv = 0.f, sx = INFINITY;
    float4 pv = make_float4(0.f, 0.f, 0.f, 0.f);
    if (k < n) {
        const int i = list ? list[k] : k;
        pack_tstep_mixed_one(k, list, n, x, v, m, N, G, rec);
        best[k] = kInf;
        for (int q = 0; q < 3; ++q) {
            const double p = x[(size_t)q * N + i];
            lo[q] = __double2float_rd(p);
            hi[q] = __double2float_ru(p);
        }
        pv = rec[2 * n + k];
        vlo[0] = vhi[0] = sx = pv.x;
        vlo[1] = vhi[1] = pv.y;
        vlo[2] = vhi[2] = pv.z;
        gm = pv.w;
        vv = sqrtf(fmaf(pv.x, pv.x, fmaf(pv.y, pv.y, pv.z * pv.z)));
    }
    TileHead h;
    float c[3];
    for (int q = 0; q < 3; ++q) {
        lo[q] = warp_min(lo[q]);
        hi[q] = warp_max(hi[q]);
        // a receiver's rounded position may be this far off beside the box
        const float pad = 2.4e-7f * fmaxf(fabsf(lo[q]), fabsf(hi[q]));
        lo[q] -= pad;
        hi[q] += pad;
        c[q] = 0.5f * (warp_min(vlo[q]) + warp_max(vhi[q]));
    }
    const float dx = pv.x - c[0], dy = pv.y - c[1], dz = pv.z - c[2];
    const float vr = warp_max(k < n ? sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz))) : 0.f);
    h.lo = make_float4(lo[0], lo[1], lo[2], warp_max(gm));
    h.hi = make_float4(hi[0], hi[1], hi[2], warp_max(vv));
    h.vc = make_float4(c[0], c[1], c[2], vr);
    if (lane == 0) head[k >> 5] = h;
    // bitonic sort over the lanes
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int o = size >> 1; o > 0; o >>= 1) {
            const float u = __shfl_xor_sync(kFull, sx, o);
            const bool up = (lane & size) == 0, low = (lane & o) == 0;
            sx = (up == low) ? fminf(sx, u) : fmaxf(sx, u);
        }
    vx[k] = sx;
}

// the warp's 64 receivers as the lanes of the packed loop
template <int SYM>
struct TstepGroup {
    TstepX2I P;
    TstepMixedI<2> I;
    int ipos[2];
    float best[2], minr2[2], bnd[2], ce[2];
};

template <int SYM>
__device__ __forceinline__ void tstep_group(TstepGroup<SYM> &W, const float4 *__restrict__ rec, int n, int g)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = g * 64 + k * 32 + lane;
        W.ipos[k] = i;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 a = make_float4(0.f, 0.f, 0.f, 1.f), b = zero4, c = a;
        if (i < n) {
            a = rec[i];
            b = rec[n + i];
            c = rec[2 * n + i];
        }
        W.I.xh[k] = a.x; W.I.yh[k] = a.y; W.I.zh[k] = a.z;
        W.I.xl[k] = b.x; W.I.yl[k] = b.y; W.I.zl[k] = b.z;
        W.I.vx[k] = c.x; W.I.vy[k] = c.y; W.I.vz[k] = c.z; W.I.gm[k] = c.w;
        W.best[k] = W.minr2[k] = W.bnd[k] = W.ce[k] = INFINITY;
    }
    const TstepMixedI<2> &I = W.I;
    W.P.nxh = make_float2(-I.xh[0], -I.xh[1]);
    W.P.nyh = make_float2(-I.yh[0], -I.yh[1]);
    W.P.nzh = make_float2(-I.zh[0], -I.zh[1]);
    W.P.nxl = make_float2(-I.xl[0], -I.xl[1]);
    W.P.nyl = make_float2(-I.yl[0], -I.yl[1]);
    W.P.nzl = make_float2(-I.zl[0], -I.zl[1]);
    W.P.nvx = make_float2(-I.vx[0], -I.vx[1]);
    W.P.nvy = make_float2(-I.vy[0], -I.vy[1]);
    W.P.nvz = make_float2(-I.vz[0], -I.vz[1]);
    W.P.gm = make_float2(I.gm[0], I.gm[1]);
}

struct TstepTile {
    float4 A[32], B[32], C[32], V0[32], V1[32];
};

// stage tile t (duplicated for the packed loop); returns its number of sources
__device__ __forceinline__ int tstep_stage(TstepTile &s, const float4 *__restrict__ rec, int n, int t)
{
    const int lane = threadIdx.x & 31, j = t * 32 + lane;
    __syncwarp();
    if (j < n) {
        const float4 a = rec[j], b = rec[n + j], v = rec[2 * n + j];
        s.A[lane] = make_float4(a.x, a.x, a.y, a.y);
        s.B[lane] = make_float4(a.z, a.z, b.x, b.x);
        s.C[lane] = make_float4(b.y, b.y, b.z, b.z);
        s.V0[lane] = make_float4(v.x, v.x, v.y, v.y);
        s.V1[lane] = make_float4(v.z, v.z, v.w, v.w);
    }
    __syncwarp();
    return min(32, n - t * 32);
}

// every pair of the warp's receivers with tile t, which holds none of them
template <int SYM>
__device__ __forceinline__ void tstep_tile(TstepGroup<SYM> &W, TstepTile &s, const float4 *__restrict__ rec, int n,
                                           int t, float eta, float eta15)
{
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const int cnt = tstep_stage(s, rec, n, t);
    int jj = 0;
    for (; jj + 4 <= cnt; jj += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            tstep_x2_j<SYM>(s.A[jj + u], s.B[jj + u], s.C[jj + u], s.V0[jj + u], s.V1[jj + u], zero4, zero4, W.P, eta,
                            eta15, W.best, W.minr2, W.bnd, W.ce);
    }
    for (; jj < cnt; ++jj)
        tstep_x2_j<SYM>(s.A[jj], s.B[jj], s.C[jj], s.V0[jj], s.V1[jj], zero4, zero4, W.P, eta, eta15, W.best, W.minr2,
                        W.bnd, W.ce);
}

// First pass: the pairs of each 64 receivers among themselves (blockIdx.y = 0) and with the
// SEED_TILES tiles before and after them in the list taken as a ring (blockIdx.y > 0, two of them
// a warp), mostly their neighbours in space: minima near the final ones, by which the second
// pass judges the other tiles.
constexpr int SEED_TILES = 4;
template <int SYM>
__global__ void __launch_bounds__(32) k_tstep_tile_seed(const float4 *__restrict__ rec, int n, float eta,
                                                        unsigned *__restrict__ best, int *__restrict__ err)
{
    __shared__ TstepTile s;
    const int g = blockIdx.x, ntiles = (n + 31) / 32;
    const float eta15 = 1.5f * eta;
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    TstepGroup<SYM> W;
    tstep_group(W, rec, n, g);
    const int own = min(2, ntiles - 2 * g);
    if (blockIdx.y == 0) {
        for (int t = 2 * g; t < 2 * g + own; ++t) {
            const int cnt = tstep_stage(s, rec, n, t);
            for (int jj = 0; jj < cnt; ++jj) {
                const float4 a = s.A[jj], b = s.B[jj], c = s.C[jj], v0 = s.V0[jj], v1 = s.V1[jj];
                const float4 J0 = make_float4(a.x, a.z, b.x, 0.f);
                const float4 J1 = make_float4(b.z, c.x, c.z, 0.f);
                const float4 JV = make_float4(v0.x, v0.z, v1.x, v1.z);
                tstep_mixed_j<2, SYM, true>(J0, J1, JV, zero4, W.I, eta, eta15, t * 32 + jj, W.ipos, W.best, W.minr2);
            }
        }
        // the last group may hold one tile only: its second is the ring's first
        if (own < 2) tstep_tile(W, s, rec, n, 0, eta, eta15);
    } else {
        const int o = blockIdx.y;  // 1 .. SEED_TILES
        tstep_tile(W, s, rec, n, (2 * g - o + ntiles) % ntiles, eta, eta15);
        tstep_tile(W, s, rec, n, (2 * g + 1 + o) % ntiles, eta, eta15);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (W.ipos[k] >= n) continue;
        // non-negative floats order as their bit patterns
        atomicMin(&best[W.ipos[k]], __float_as_uint(W.best[k]));
        if (W.minr2[k] == 0.f) atomicOr(err, ERR_COINCIDENT);
    }
}

// The bounds of the second pass.  With D a lower bound on the distance, V and M upper bounds on
// |v_ij| and G (m_i + m_j), B the receiver's bound, and u = v/r, w = G M / r^3 of a pair: every
// symmetrisation factor obeys 1 / s(d) <= h(|d|), h(d) = (1 + sqrt(1 + d^2) + d) / 2 (the harmonic
// factor of d < 0; arithmetic 1 + |d|/2 or d/2, none 1), h' <= 1, and |d_ff| <= 1.5 eta u t_ff,
// |d_fb| <= eta (1 + w / u^2).  So, with c = 1.5 eta,
//   1 / (t_ff s) <= (sqrt(w) + sqrt(w + (c u)^2) + c u) / 2,   1 / (t_fb s) <= h(eta) u + eta w / u.
// No pair can lower the minimum if (1) B times the first, at w = M / D^3 and u = V / D, is below
// 1, (2) B h(eta) V / D < 0.9 and (3) B eta w / u < 0.1, that is v > 10 B eta M / D^2, which fails
// only for a pair almost at rest relative to each other.  The margins of 1 % cover the FP32
// evaluation of the bounds and of the criteria.
// Returns (1) and (2); thr: the speed of (3).  heta: h(eta).
__device__ __forceinline__ bool tstep_far(float D2, float V, float M, float B, float eta, float heta, float &thr)
{
    const float iD = rsqrtf(D2), u = V * iD, m2 = M * iD * iD, w = m2 * iD, cu = 1.5f * eta * u;
    const float c1 = 0.5f * B * (sqrtf(w) + sqrtf(fmaf(cu, cu, w)) + cu);
    thr = 10.2f * B * eta * m2;
    return (D2 > 0.f) && (c1 < 0.98f) && (B * heta * u < 0.88f) && (thr < INFINITY);
}

constexpr int TQ = 128;  // queue of (receiver, tile) items

// Second pass: the other tiles of the ring, outwards, every nsplit-th one.  A tile is judged
// first as a whole (box against box, 32 tiles at once over the lanes), then, where that does
// not settle it, by every receiver on its own (point against box, its own bound and velocity:
// 0.8 % of the (receiver, tile) items of a 40960-body Plummer sphere remain, where whole tiles
// leave 38 %).  Condition (3) is tested on v_x alone, by bisection in the tile's ordered v_x.
// What remains is queued and evaluated with a source a lane.
template <int SYM>
__global__ void __launch_bounds__(32) k_tstep_tile(const float4 *__restrict__ rec, const float *__restrict__ vx,
                                                   const TileHead *__restrict__ head, int n, int nsplit, float eta,
                                                   unsigned *__restrict__ best, int *__restrict__ err)
{
    __shared__ float s_vx[32];
    __shared__ float4 s_x[64], s_l[64], s_v[64];
    __shared__ float s_best[64];
    __shared__ int s_q[TQ];
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int g = blockIdx.x, ntiles = (n + 31) / 32;
    const float eta15 = 1.5f * eta;
    const float heta = 0.5f * (1.f + sqrtf(fmaf(eta, eta, 1.f)) + eta);
    float px[2], py[2], pz[2], ux[2], uy[2], uz[2], gm[2], first[2];
    bool live[2], hit = false;
    float bmax = 0.f;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = g * 64 + k * 32 + lane;
        live[k] = i < n;
        const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = live[k] ? rec[i] : zero4, b = live[k] ? rec[n + i] : zero4, c = live[k] ? rec[2 * n + i] : zero4;
        first[k] = live[k] ? __uint_as_float(best[i]) : 0.f;
        px[k] = a.x; py[k] = a.y; pz[k] = a.z;
        ux[k] = c.x; uy[k] = c.y; uz[k] = c.z;
        gm[k] = c.w;
        s_x[k * 32 + lane] = a;
        s_l[k * 32 + lane] = b;
        s_v[k * 32 + lane] = c;
        s_best[k * 32 + lane] = first[k];
        bmax = fmaxf(bmax, first[k]);
    }
    bmax = 1.011f * warp_max(bmax);
    __syncwarp();
    TileHead I = head[2 * g];
    if (2 * g + 1 < ntiles) {
        const TileHead h = head[2 * g + 1];
        I.lo = make_float4(fminf(I.lo.x, h.lo.x), fminf(I.lo.y, h.lo.y), fminf(I.lo.z, h.lo.z), fmaxf(I.lo.w, h.lo.w));
        I.hi = make_float4(fmaxf(I.hi.x, h.hi.x), fmaxf(I.hi.y, h.hi.y), fmaxf(I.hi.z, h.hi.z), fmaxf(I.hi.w, h.hi.w));
    }
    int nq = 0;
    // the queued items, two at a time, a source a lane
    auto drain = [&]() {
        __syncwarp();
        for (int q = 0; q < nq; q += 2) {
            const int it[2] = {s_q[q], s_q[min(q + 1, nq - 1)]};
            float bq[2][1], mq[2][1];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int r = it[e] & 63, j = (it[e] >> 6) * 32 + lane;
                const bool in = j < n;
                const int jj = in ? j : n - 1;
                const float4 xi = s_x[r], li = s_l[r], vi = s_v[r];
                TstepMixedI<1> R;
                R.xh[0] = xi.x; R.yh[0] = xi.y; R.zh[0] = xi.z;
                R.xl[0] = li.x; R.yl[0] = li.y; R.zl[0] = li.z;
                R.vx[0] = vi.x; R.vy[0] = vi.y; R.vz[0] = vi.z; R.gm[0] = vi.w;
                bq[e][0] = s_best[r];
                mq[e][0] = INFINITY;
                // a lane past the end of the list is masked as a self pair
                const int ipos[1] = {in ? -1 : 0};
                tstep_mixed_j<1, SYM, true>(rec[jj], rec[n + jj], rec[2 * n + jj],
                                            make_float4(0.f, 0.f, 0.f, 0.f), R, eta, eta15, 0, ipos, bq[e], mq[e]);
                hit = hit || mq[e][0] == 0.f;
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float b = warp_min(bq[e][0]);
                if (lane == 0 && b < s_best[it[e] & 63]) s_best[it[e] & 63] = b;
                __syncwarp();
            }
        }
        nq = 0;
    };
    const int nrest = max(0, ntiles - 2 - 2 * SEED_TILES);
    for (int q0 = blockIdx.y; q0 < nrest; q0 += 32 * nsplit) {
        // this lane's tile of the batch, outwards from the seeds
        const int q = q0 + lane * nsplit;
        const bool have = q < nrest;
        const int off = (q & 1) ? -(q >> 1) - 1 - SEED_TILES : (q >> 1) + 2 + SEED_TILES;
        const int mine = have ? (2 * g + off + ntiles) % ntiles : 0;
        bool whole = false;
        float wthr = 0.f;
        if (have) {
            const TileHead J = head[mine];
            whole = tstep_far(box_gap2(I.lo, I.hi, J.lo, J.hi), I.hi.w + J.hi.w, I.lo.w + J.lo.w, bmax, eta, heta, wthr);
        }
        const unsigned wmask = __ballot_sync(kFull, whole);
        const int cnt = min(32, (nrest - q0 + nsplit - 1) / nsplit);
        int t = __shfl_sync(kFull, mine, 0);
        float next = vx[t * 32 + lane];
        for (int b = 0; b < cnt; ++b) {
            const int cur = t;
            __syncwarp();
            s_vx[lane] = next;
            __syncwarp();
            if (b + 1 < cnt) {
                t = __shfl_sync(kFull, mine, b + 1);
                next = vx[t * 32 + lane];
            }
            float thr[2];
            bool todo[2];
            thr[0] = thr[1] = __shfl_sync(kFull, wthr, b);
            todo[0] = todo[1] = false;
            if (!((wmask >> b) & 1u)) {
                const TileHead J = head[cur];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float gx = fmaxf(0.f, fmaxf(J.lo.x - px[k], px[k] - J.hi.x));
                    const float gy = fmaxf(0.f, fmaxf(J.lo.y - py[k], py[k] - J.hi.y));
                    const float gz = fmaxf(0.f, fmaxf(J.lo.z - pz[k], pz[k] - J.hi.z));
                    const float wx = J.vc.x - ux[k], wy = J.vc.y - uy[k], wz = J.vc.z - uz[k];
                    const float V = sqrtf(fmaf(wx, wx, fmaf(wy, wy, wz * wz))) + J.vc.w;
                    todo[k] = !tstep_far(fmaf(gx, gx, fmaf(gy, gy, gz * gz)), V, gm[k] + J.lo.w,
                                         1.011f * s_best[k * 32 + lane], eta, heta, thr[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                int p = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (s_vx[p + o - 1] < ux[k]) p += o;
                const float gap = fminf(fabsf(s_vx[p] - ux[k]), fabsf(s_vx[max(p - 1, 0)] - ux[k]));
                todo[k] = live[k] && (todo[k] || !(gap > thr[k]));
                const unsigned mask = __ballot_sync(kFull, todo[k]);
                if (todo[k]) s_q[nq + __popc(mask & below)] = (cur << 6) | (k * 32 + lane);
                nq += __popc(mask);
            }
            if (nq > TQ - 64) drain();
        }
        drain();
        // what the other splits of the group have found since
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (live[k])
                s_best[k * 32 + lane] = fminf(s_best[k * 32 + lane], __uint_as_float(best[g * 64 + k * 32 + lane]));
        __syncwarp();
        bmax = 1.011f * warp_max(fmaxf(s_best[lane], s_best[lane + 32]));
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float b = s_best[k * 32 + lane];
        if (live[k] && b < first[k]) atomicMin(&best[g * 64 + k * 32 + lane], __float_as_uint(b));
    }
    if (hit) atomicOr(err, ERR_COINCIDENT);
}

// tau[pos[i]] = eta best[i]
__global__ void k_finalize_tau_tile(const unsigned *__restrict__ best, int n, double eta, const int32_t *__restrict__ pos,
                                    double *__restrict__ tau, int *__restrict__ err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double t = eta * (double)__uint_as_float(best[i]);
    if (!(t > 0.0)) atomicOr(err, ERR_NONFINITE);
    tau[pos ? pos[i] : i] = t;
}

}  // namespace

void launch_tstep_tile(cudaStream_t s, const int32_t *list, int n, const double *x, const double *v, const double *m,
                       int N, double G, double eta, int sym, int n_sm, void *rec, unsigned *best, const int32_t *pos,
                       double *tau, int *err)
{
    const int ntiles = (n + 31) / 32, ngroups = (n + 63) / 64;
    float4 *r = (float4 *)rec;
    float *vx = (float *)(r + (size_t)3 * n);
    TileHead *head = (TileHead *)(r + (size_t)3 * n + 8 * ntiles);
    // about 24 resident warps an SM, four rounds of them, each warp a batch of 32 tiles at least
    const int nsplit = std::max(1, std::min((ntiles + 31) / 32, (4 * 24 * n_sm + ngroups - 1) / ngroups));
    k_tile_pack_tstep<<<(n + 127) / 128, 128, 0, s>>>(list, n, x, v, m, N, G, r, vx, head, best);
    const dim3 seeds(ngroups, 1 + SEED_TILES), grid(ngroups, nsplit);
#define FROST_TSTEP_TILE_CASE(SYMV)                                                             \
    {                                                                                           \
        k_tstep_tile_seed<SYMV><<<seeds, 32, 0, s>>>(r, n, (float)eta, best, err);              \
        k_tstep_tile<SYMV><<<grid, 32, 0, s>>>(r, vx, head, n, nsplit, (float)eta, best, err);  \
    }
    switch (sym) {
    case 0: FROST_TSTEP_TILE_CASE(0) break;
    case 1: FROST_TSTEP_TILE_CASE(1) break;
    default: FROST_TSTEP_TILE_CASE(2) break;
    }
#undef FROST_TSTEP_TILE_CASE
    k_finalize_tau_tile<<<(n + 255) / 256, 256, 0, s>>>(best, n, eta, pos, tau, err);
}

}  // namespace frost
