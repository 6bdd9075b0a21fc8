// Mixed-precision Newtonian and gradient passes of a spatially ordered list, tile by tile
// (sm_103a).  A warp takes 64 receivers (two a lane) against its share of the sources' tiles of
// 64 and treats a tile by the distance of its box from the receivers' box.
//
// What bounds these passes is FP32 issue, and half of it went into separations: from absolute
// float-float positions a component costs three additions (five from the gradient's
// three-part split), because the difference of two positions of size |x| has to be good to
// 2^-24 of a distance that may be far smaller.  Here a tile's positions are kept relative to its
// own centre c_J (hi + lo, 48 bits of an offset of at most the tile's radius R_J), and a
// receiver's offset X = x_i - c_J is formed once a tile, in double-float, for 64 pairs:
//   far tile (box distance D >= R_J / 5): dx = (x'_j - X_lo) - X_hi, x'_j rounded to FP32: two
//     additions, and below 2^-25 (|dx| + 2 R_J) in error.  (The low part first: added last, or to
//     a high difference that is already on the grid of dx, it is lost, the same way for every
//     source of the tile, and such errors add up.  One addition of a rounding of X, four
//     roundings in turn whose mean is right, scatter so much that g was off by 1.13 times the
//     one-sided pass's error at the 99.9th percentile; now 0.78.)
//   near tile: dx = (x'_j,hi - X_hi) + (x'_j,lo - X_lo), three additions as before.
// The gradient's a_j - a_i works alike against a tile's mean acceleration.  The plain Newtonian
// pass, whose error is the MUFU rsqrt's, does take the four roundings of X.
// A tile's terms, which all point the same way, are summed in eight partial sums of 8 and these by
// twos and fours before the compensated sum: as one of 16 each, two added, they left a with 1.14
// times the one-sided pass's error at the 99.9th percentile (which folds every 16), now 0.95.
//
// Dominant terms (above 1/16 of max_j m_j / r^3, of the prepass) are kept out of the FP32 sums
// and summed in double-float as in the other mixed passes.  In an ordered list they sit in the
// few tiles around the receiver, so a receiver has more slots a split.  A tile is searched for
// them unless its heaviest mass at its box stays below every receiver's threshold.
// The prepass itself looks only at tiles whose box can hold a larger m_j / r^3.
//
// Pairs of sources are the two lanes of packed f32x2 instructions (tiles are structures of
// arrays, so a pair loads as it lies; the receivers' operands are duplicated in registers).
// What a tile costs beside its pairs (offsets, roundings, folds: about 250 instructions) is why it
// holds 64 sources: with 32 it was 45 % of the instructions executed.
#include "pair_bodies.cuh"
#include "tile_bounds.cuh"

namespace frost {
namespace {

using namespace dev;

constexpr unsigned kFull = 0xffffffffu;
constexpr int TJ = TILE_N;            // particles a tile: the 64 receivers of a warp are one, too
static_assert(TJ == 64, "two particles a lane");
constexpr int TB = TJ / 4;            // 16-byte pieces of a row
constexpr float kFarRadius = 0.2f;    // far: box distance of at least this many source radii
constexpr int SLOTS = 16;             // dominant terms a receiver and split (see Slots)
constexpr float kFar = 1.0e15f;       // offset of the stand-ins past the end (mass 0)

// rows of 64 floats of a tile: positions {x, y, z, m}, {low parts of x, y, z, m}, m^(-2/3)
enum { P_X, P_Y, P_Z, P_M, P_XL, P_YL, P_ZL, P_ML, P_MQ, P_ROWS };
// gradient: {x, y, z, m}, {ax, ay, az}, low parts of both
enum { G_X, G_Y, G_Z, G_M, G_AX, G_AY, G_AZ, G_XL, G_YL, G_ZL, G_AXL, G_AYL, G_AZL, G_ROWS };
static_assert(P_ROWS == TILE_POS_ROWS && G_ROWS == TILE_GRAD_ROWS, "record sizes in frost_internal.cuh");

struct Head {
    float4 c;  // {centre, radius}
    float4 h;  // {largest |offset from the centre| by component, smallest m^(-2/3)}
    float4 a;  // {mean acceleration of the sources that count, 0} (gradient)
};
static_assert(sizeof(Head) == TILE_HEAD_BYTES, "head size in frost_internal.cuh");

__device__ __forceinline__ const Head *heads(const float *rec, int n, int rows)
{
    return (const Head *)(rec + (size_t)((n + TJ - 1) / TJ) * rows * TJ);
}

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
__device__ __forceinline__ float warp_sum(float v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// the squared distance of two boxes, from below
__device__ __forceinline__ float box_gap2(const float4 ca, const float4 ha, const float4 cb, const float4 hb)
{
    return gap2(axis_gap(ca.x - cb.x, ha.x + hb.x), axis_gap(ca.y - cb.y, ha.y + hb.y), axis_gap(ca.z - cb.z, ha.z + hb.z));
}

// ------------------------------------------------------------------------------------
// records
// ------------------------------------------------------------------------------------
// One tile a warp, two particles a lane.  GRAD: gradient records with the accelerations acc
// ([3][n] by list position) and the hot sources' masses zeroed; else position records, after a
// drift by dt v if v is given (the roundings of launch_drift).
template <bool GRAD>
__global__ void __launch_bounds__(128) k_tile_pack(const int32_t *__restrict__ list, int n, double *__restrict__ x,
                                                   const double *__restrict__ v, double dt,
                                                   const double *__restrict__ m, int N, const double *__restrict__ acc,
                                                   const uint32_t *__restrict__ hot, float *__restrict__ rec)
{
    constexpr int ROWS = GRAD ? G_ROWS : P_ROWS;
    const int tile = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (tile * TJ >= n) return;
    double p[2][3], mass[2];
    bool live[2];
    float *t = rec + (size_t)tile * ROWS * TJ + lane;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int k = tile * TJ + e * 32 + lane;
        live[e] = k < n;
        mass[e] = p[e][0] = p[e][1] = p[e][2] = 0.0;
        if (!live[e]) continue;
        const int i = list ? list[k] : k;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            p[e][q] = x[(size_t)q * N + i];
            if (!GRAD && v) {
                p[e][q] = __dadd_rn(p[e][q], __dmul_rn(dt, v[(size_t)q * N + i]));
                x[(size_t)q * N + i] = p[e][q];
            }
        }
        mass[e] = m[i];
    }
    float half[3], c[3], r2[2] = {0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float p0 = (float)p[0][q], p1 = (float)p[1][q];
        const float lo = warp_min(fminf(live[0] ? p0 : INFINITY, live[1] ? p1 : INFINITY));
        const float hi = warp_max(fmaxf(live[0] ? p0 : -INFINITY, live[1] ? p1 : -INFINITY));
        c[q] = 0.5f * lo + 0.5f * hi;
        float far = 0.f;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const double d = live[e] ? p[e][q] - (double)c[q] : (double)kFar;
            const float h = (float)d;
            t[((GRAD ? G_X : P_X) + q) * TJ + e * 32] = h;
            t[((GRAD ? G_XL : P_XL) + q) * TJ + e * 32] = live[e] ? (float)(d - (double)h) : 0.f;
            if (live[e]) {
                r2[e] = fmaf(h, h, r2[e]);
                far = fmaxf(far, fabsf(h));
            }
        }
        half[q] = warp_max(far);
    }
    Head h;
    float mq = INFINITY;
    h.a = make_float4(0.f, 0.f, 0.f, 0.f);
    bool cold[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int k = tile * TJ + e * 32 + lane;
        const float mf = (float)mass[e];
        const float q = (live[e] && mf > 0.f) ? exp2f(-0.6666667f * log2f(mf)) : INFINITY;
        mq = fminf(mq, q);
        cold[e] = live[e] && !(GRAD && hot && ((hot[k >> 5] >> (k & 31)) & 1u));
        if (GRAD) {
            t[G_M * TJ + e * 32] = cold[e] ? mf : 0.f;
        } else {
            t[P_M * TJ + e * 32] = mf;
            t[P_ML * TJ + e * 32] = (float)(mass[e] - (double)mf);
            t[P_MQ * TJ + e * 32] = q;
        }
    }
    if (GRAD) {
        const float share = 1.f / fmaxf(1.f, (float)(__popc(__ballot_sync(kFull, cold[0])) + __popc(__ballot_sync(kFull, cold[1]))));
        float ac[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            double a[2];
            float sum = 0.f;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                a[e] = live[e] ? acc[(size_t)q * n + tile * TJ + e * 32 + lane] : 0.0;
                if (cold[e]) sum += (float)a[e];
            }
            ac[q] = share * warp_sum(sum);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const double d = live[e] ? a[e] - (double)ac[q] : 0.0;
                const float ah = (float)d;
                t[(G_AX + q) * TJ + e * 32] = ah;
                t[(G_AXL + q) * TJ + e * 32] = (float)(d - (double)ah);
            }
        }
        h.a = make_float4(ac[0], ac[1], ac[2], 0.f);
    }
    h.c = make_float4(c[0], c[1], c[2], 1.00001f * sqrtf(warp_max(fmaxf(r2[0], r2[1]))));
    h.h = make_float4(half[0], half[1], half[2], warp_min(mq));
    if (lane == 0) ((Head *)heads(rec, n, ROWS))[tile] = h;
}

// ------------------------------------------------------------------------------------
// receivers
// ------------------------------------------------------------------------------------
// The 64 receivers of a warp (one tile of their list), in shared memory: a lane reads its two once
// a tile; in registers they cost a quarter of the resident warps.  Offsets from their tile's
// centre as {hi, lo} by component, and the sums.
struct Group {
    Head head;
    float xh[3][TJ], xl[3][TJ];
    float2 H[3][TJ], L[3][TJ];
};

// receiver k of this lane: its index among the 64
__device__ __forceinline__ int slot_of(int k) { return k * 32 + (threadIdx.x & 31); }

__device__ __forceinline__ void load_group(Group &W, const float *__restrict__ rec, int n, int rows, int xlrow, int g)
{
    if ((threadIdx.x & 31) == 0) W.head = heads(rec, n, rows)[g];
    const float *t = rec + (size_t)g * rows * TJ;
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            W.xh[q][slot_of(k)] = t[q * TJ + slot_of(k)];
            W.xl[q][slot_of(k)] = t[(xlrow + q) * TJ + slot_of(k)];
            W.H[q][slot_of(k)] = W.L[q][slot_of(k)] = make_float2(0.f, 0.f);
        }
    __syncwarp();
}

// the receivers' offsets from the centre of a source tile: X = {h, l}
__device__ __forceinline__ void offsets(const Group &W, const float4 c, float (&h)[2][3], float (&l)[2][3])
{
    const float rc[3] = {W.head.c.x, W.head.c.y, W.head.c.z}, jc[3] = {c.x, c.y, c.z};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        float s, e;
        df::two_sum(rc[q], -jc[q], s, e);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float p, r;
            df::two_sum(s, W.xh[q][slot_of(k)], p, r);
            h[k][q] = p;
            l[k][q] = __fadd_rn(r, __fadd_rn(e, W.xl[q][slot_of(k)]));
        }
    }
}

// FP32 sums of a tile (one per lane of the packed arithmetic) into the receivers' compensated
// ones, lane by lane: fold2 in packed form
__device__ __forceinline__ void fold_group(Group &W, int k, float2 x, float2 y, float2 z)
{
    const float2 v[3] = {x, y, z}, minus = make_float2(-1.f, -1.f);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float2 h = W.H[q][slot_of(k)], p = v[q];
        const float2 s = __fadd2_rn(h, p);
        const float2 bb = __ffma2_rn(h, minus, s);
        const float2 e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, minus, s), minus, h), __ffma2_rn(bb, minus, p));
        W.H[q][slot_of(k)] = s;
        W.L[q][slot_of(k)] = __fadd2_rn(W.L[q][slot_of(k)], e);
    }
}

__device__ __forceinline__ double group_total(const Group &W, int q, int r)
{
    return ((double)W.H[q][r].x + (double)W.L[q][r].x) + ((double)W.H[q][r].y + (double)W.L[q][r].y);
}

// the squared distance of this lane's receiver k from a tile's box, from below
__device__ __forceinline__ float point_gap2(const Group &W, int k, const float4 c, const float4 h)
{
    const int r = slot_of(k);
    return gap2(point_axis_gap(W.head.c.x - c.x, W.xh[0][r], h.x), point_axis_gap(W.head.c.y - c.y, W.xh[1][r], h.y),
                point_axis_gap(W.head.c.z - c.z, W.xh[2][r], h.z));
}

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
// four roundings of h + l (negated, for four sources at a time) whose mean is right to an eighth
// of a unit: each takes up what the ones before it left
__device__ __forceinline__ void four_roundings(float h, float l, float2 (&out)[2])
{
    const float a0 = __fadd_rn(h, l);
    const float rest = __fadd_rn(__fsub_rn(h, a0), l);
    const float a1 = __fadd_rn(a0, 2.f * rest);
    const float r1 = __fadd_rn(rest, __fsub_rn(2.f * rest, __fsub_rn(a1, a0)));
    const float a2 = __fadd_rn(a0, r1);
    const float a3 = __fadd_rn(a0, __fadd_rn(rest, __fsub_rn(r1, __fsub_rn(a2, a0))));
    out[0] = make_float2(-a0, -a1);
    out[1] = make_float2(-a2, -a3);
}

// a separation in a far tile: x'_j less the receiver's low part, then less its high part (LOW),
// or x'_j less one of four roundings
template <bool LOW>
__device__ __forceinline__ float2 far_sep(float2 x, const float2 (&n)[2], int u)
{
    return LOW ? __fadd2_rn(__fadd2_rn(x, n[1]), n[0]) : __fadd2_rn(x, n[u]);
}

// the negated receiver offset h + l for a searched tile, the part that goes with the sources' high
// parts first: in a far tile (single) the low one
__device__ __forceinline__ void searched_offset(bool single, float h, float l, float2 &nh, float2 &nl)
{
    nh = dup(single ? -l : -h);
    nl = dup(single ? -h : -l);
}

__device__ __forceinline__ float2 half_of(const float4 v, int u) { return u ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }

// ------------------------------------------------------------------------------------
// prepass: wmax[i] = max_j m_j / r^3 = (min_j r^2 m_j^(-2/3))^(-3/2)
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void wmax_tile(const Group &W, int g, const float *__restrict__ jrec, const Head &J, int t,
                                          bool diag, float eps2, float4 (*s)[TB], float (&q)[2])
{
    const int lane = threadIdx.x & 31;
    const float4 *tr = (const float4 *)(jrec + (size_t)t * P_ROWS * TJ);
    __syncwarp();
    // rows x, y, z and m^(-2/3), then the low parts
    if (lane < TB) {
#pragma unroll
        for (int r = 0; r < 3; ++r) s[r][lane] = tr[(P_X + r) * TB + lane];
        s[3][lane] = tr[P_MQ * TB + lane];
    } else {
#pragma unroll
        for (int r = 0; r < 3; ++r) s[4 + r][lane - TB] = tr[(P_XL + r) * TB + lane - TB];
    }
    __syncwarp();
    float xh[2][3], xl[2][3];
    offsets(W, J.c, xh, xl);
#pragma unroll 2
    for (int b = 0; b < TB; ++b) {
        const float4 X = s[0][b], Y = s[1][b], Z = s[2][b], M = s[3][b], XL = s[4][b], YL = s[5][b], ZL = s[6][b];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float2 r[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float2 x = half_of(X, u), y = half_of(Y, u);
                const float2 z = half_of(Z, u), mm = half_of(M, u);
                const float2 xx = half_of(XL, u), yy = half_of(YL, u);
                const float2 zz = half_of(ZL, u);
                const float2 dx = __fadd2_rn(__fadd2_rn(x, dup(-xh[k][0])), __fadd2_rn(xx, dup(-xl[k][0])));
                const float2 dy = __fadd2_rn(__fadd2_rn(y, dup(-xh[k][1])), __fadd2_rn(yy, dup(-xl[k][1])));
                const float2 dz = __fadd2_rn(__fadd2_rn(z, dup(-xh[k][2])), __fadd2_rn(zz, dup(-xl[k][2])));
                r[u] = __fmul2_rn(__ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, dup(eps2)))), mm);
            }
            if (diag) {
                const int j = t * TJ + 4 * b, i = g * TJ + slot_of(k);
                if (j == i) r[0].x = INFINITY;
                if (j + 1 == i) r[0].y = INFINITY;
                if (j + 2 == i) r[1].x = INFINITY;
                if (j + 3 == i) r[1].y = INFINITY;
            }
            q[k] = fminf(q[k], fminf(fminf(r[0].x, r[0].y), fminf(r[1].x, r[1].y)));
        }
    }
}

__global__ void __launch_bounds__(32) k_wmax_tile(const float *__restrict__ rec, int n, int nsplit, float eps2,
                                                  float *__restrict__ wmax)
{
    __shared__ float4 s[7][TB];
    __shared__ Group W;
    const int lane = threadIdx.x & 31, g = blockIdx.x, ntiles = (n + TJ - 1) / TJ;
    const Head *jh = heads(rec, n, P_ROWS);
    load_group(W, rec, n, P_ROWS, P_XL, g);
    float q[2] = {INFINITY, INFINITY};
    // first the tile whose centre is nearest (the receivers' own, if it is in this split)
    float best = INFINITY;
    int first = -1;
    for (int t = blockIdx.y + lane * nsplit; t < ntiles; t += 32 * nsplit) {
        const float4 c = jh[t].c;
        const float x = c.x - W.head.c.x, y = c.y - W.head.c.y, z = c.z - W.head.c.z;
        const float d = fmaf(x, x, fmaf(y, y, z * z));
        if (d < best) {
            best = d;
            first = t;
        }
    }
    {
        const float d = warp_min(best);
        const unsigned mask = __ballot_sync(kFull, best == d && first >= 0);
        if (!mask) return;
        first = __shfl_sync(kFull, first, __ffs(mask) - 1);
        wmax_tile(W, g, rec, jh[first], first, first == g, eps2, s, q);
    }
    // then those that can still hold a larger m_j / r^3 for some receiver: box against box, then
    // every receiver against the box (a few receivers far from the others stretch the group's box
    // and bound, and it would look into 11 instead of 1 % of a 65536-body sphere's tiles)
    for (int t0 = blockIdx.y; t0 < ntiles; t0 += 32 * nsplit) {
        const int t = t0 + lane * nsplit;
        const float qmax = 1.0001f * warp_max(fmaxf(g * TJ + slot_of(0) < n ? q[0] : 0.f, g * TJ + slot_of(1) < n ? q[1] : 0.f));
        bool near = false;
        if (t < ntiles && t != first) {
            const float4 c = jh[t].c, h = jh[t].h;
            near = !((box_gap2(W.head.c, W.head.h, c, h) + eps2) * h.w > qmax);
        }
        for (unsigned mask = __ballot_sync(kFull, near); mask; mask &= mask - 1) {
            const int tt = t0 + (__ffs(mask) - 1) * nsplit;
            const Head J = jh[tt];
            bool any = false;
#pragma unroll
            for (int k = 0; k < 2; ++k)
                any = any || (g * TJ + slot_of(k) < n && !((point_gap2(W, k, J.c, J.h) + eps2) * J.h.w > 1.0001f * q[k]));
            if (__any_sync(kFull, any)) wmax_tile(W, g, rec, J, tt, tt == g, eps2, s, q);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float y = rsqrtf(q[k]);
        // non-negative floats order as their bit patterns
        const int i = g * TJ + slot_of(k);
        if (i < n) atomicMax((int *)&wmax[i], __float_as_int(y * y * y));
    }
}

// The next 32 tiles of a split.  A tile is far from a receiver at distance d >= kFarRadius R_J of
// its box.  fm: far from every receiver and, with HEAVY, without a dominant term to look for: its
// heaviest mass at d stays below the receiver's threshold, d^2 m^(-2/3) > qk (qk = 0 for a
// receiver without a free slot).  sm: the others, to be searched for dominant terms; lm: those
// of sm that are far, which take single separations all the same.  Box against box with the
// largest qk (qthr) first, then, where that does not settle it, receiver by receiver.
// (Distance alone does not clear a tile: with a body of half the mass at the centre of a Plummer
// sphere, tiles left unsearched from R_J on made the median error of a 17 times, of g 19 times
// larger.)
template <bool HEAVY>
__device__ __forceinline__ void judge_tiles(const Group &W, const Head *__restrict__ jh, int ntiles, int t0, int nsplit,
                                            int own, bool live0, bool live1, float qthr, const float (&qk)[2], unsigned &fm,
                                            unsigned &sm, unsigned &lm)
{
    const int t = t0 + (threadIdx.x & 31) * nsplit;
    bool far = false;
    if (t < ntiles && t != own) {
        const float4 c = jh[t].c, h = jh[t].h;
        const float d2 = box_gap2(W.head.c, W.head.h, c, h);
        far = d2 > 0.f && d2 >= (kFarRadius * kFarRadius) * (c.w * c.w) && (!HEAVY || d2 * h.w > qthr);
    }
    fm = __ballot_sync(kFull, far);
    sm = lm = 0u;
    for (unsigned um = __ballot_sync(kFull, t < ntiles && !far); um; um &= um - 1) {
        const int b = __ffs(um) - 1, tt = t0 + b * nsplit;
        const float4 c = jh[tt].c, h = jh[tt].h;
        const float D2 = (kFarRadius * kFarRadius) * (c.w * c.w);
        const float d0 = point_gap2(W, 0, c, h), d1 = point_gap2(W, 1, c, h);
        const bool sep = ((d0 > 0.f && d0 >= D2) || !live0) && ((d1 > 0.f && d1 >= D2) || !live1);
        const bool light = !HEAVY || ((d0 * h.w > qk[0] || !live0) && (d1 * h.w > qk[1] || !live1));
        if (tt == own || !__all_sync(kFull, sep)) {
            sm |= 1u << b;
        } else if (HEAVY && !__all_sync(kFull, light)) {
            sm |= 1u << b;
            lm |= 1u << b;
        } else {
            fm |= 1u << b;
        }
    }
}

// whether a receiver with a free slot may find a dominant term in the tile: a far tile is searched
// only then (halo receivers, for which the whole core is within a factor 16 of the largest
// term, fill their slots in a tile or two: acc+gradient of 65536 particles 8.13 -> 7.94 ms)
__device__ __forceinline__ bool worth_search(const Group &W, const float4 c, const float4 h, bool live0, bool live1,
                                             const float (&qk)[2], const int (&cnt)[2])
{
    const bool n0 = live0 && cnt[0] < SLOTS && !(point_gap2(W, 0, c, h) * h.w > qk[0]);
    const bool n1 = live1 && cnt[1] < SLOTS && !(point_gap2(W, 1, c, h) * h.w > qk[1]);
    return __any_sync(kFull, n0 || n1);
}

// ------------------------------------------------------------------------------------
// dominant terms
// ------------------------------------------------------------------------------------
// A lane's slots: up to SLOTS source indices per receiver and split, and the double-float sums of
// their terms (with the terms beyond the FP32 range apart in FP64).  In local memory: they are
// touched a few times per receiver and split.  The limit is for receivers far out in the halo,
// for which thousands of sources are within a factor 16 of the nearest: their warps, without
// it, made the 65536-body passes a third longer.  (16, 32 and 64 slots: acc+gradient 7.98, 8.01
// and 8.06 ms, the same errors within 2 %.)
struct Slots {
    int j[2][SLOTS];
    float sum[2][6];
    double wide[2][3];
};

__device__ __forceinline__ void slots_clear(Slots &S)
{
    for (int k = 0; k < 2; ++k)
        for (int q = 0; q < 6; ++q) {
            S.sum[k][q] = 0.f;
            if (q < 3) S.wide[k][q] = 0.0;
        }
}

__device__ __forceinline__ void slots_add(Slots &S, int k, const DF3 &t)
{
    DF3 a;
    a.x.h = S.sum[k][0]; a.x.l = S.sum[k][1];
    a.y.h = S.sum[k][2]; a.y.l = S.sum[k][3];
    a.z.h = S.sum[k][4]; a.z.l = S.sum[k][5];
    df3_add(a, t);
    S.sum[k][0] = a.x.h; S.sum[k][1] = a.x.l;
    S.sum[k][2] = a.y.h; S.sum[k][3] = a.y.l;
    S.sum[k][4] = a.z.h; S.sum[k][5] = a.z.l;
}

__device__ __forceinline__ double slots_total(const Slots &S, int k, int q)
{
    return ((double)S.sum[k][2 * q] + (double)S.sum[k][2 * q + 1]) + S.wide[k][q];
}

// x_j - x_i in double-float from the two particles' own records (offsets {h, l} from their tiles'
// centres): every operation is antisymmetric, so the terms of the two partners of a tight pair
// cancel in the other particles' sums as exactly as their masses allow
__device__ __forceinline__ df::dfloat tile_sep(float jc, float jh, float jl, float ic, float ih, float il)
{
    df::dfloat c, a, b;
    df::two_sum(jc, -ic, c.h, c.l);
    a.h = jh;
    a.l = jl;
    b.h = ih;
    b.l = il;
    return df::add(c, df::sub(a, b));
}

// evaluates the slots of a lane's receiver k (n of them)
__device__ __noinline__ void acc_flush(Slots &S, const float *__restrict__ rec, const Head *__restrict__ hd, int i, int k,
                                       int n, double eps2d)
{
    if (n == 0) return;
    const float *ti = rec + (size_t)(i / TJ) * P_ROWS * TJ + i % TJ;
    const float4 ci = hd[i / TJ].c;
    using df::dfloat;
    const dfloat e2 = df::from_double(eps2d);
    for (int s = 0; s < n; ++s) {
        const int j = S.j[k][s];
        const float *t = rec + (size_t)(j / TJ) * P_ROWS * TJ + j % TJ;
        const float4 c = hd[j / TJ].c;
        const dfloat dx = tile_sep(c.x, t[P_X * TJ], t[P_XL * TJ], ci.x, ti[P_X * TJ], ti[P_XL * TJ]);
        const dfloat dy = tile_sep(c.y, t[P_Y * TJ], t[P_YL * TJ], ci.y, ti[P_Y * TJ], ti[P_YL * TJ]);
        const dfloat dz = tile_sep(c.z, t[P_Z * TJ], t[P_ZL * TJ], ci.z, ti[P_Z * TJ], ti[P_ZL * TJ]);
        const dfloat r2 = df::add(df::add(df::mul(dx, dx), df::mul(dy, dy)), df::add(df::mul(dz, dz), e2));
        const dfloat ri = df::rsqrt(r2);
        dfloat m;
        m.h = t[P_M * TJ];
        m.l = t[P_ML * TJ];
        const dfloat w = df::mul(df::mul(df::mul(ri, ri), ri), m);
        DF3 u;
        u.x = df::mul(w, dx);
        u.y = df::mul(w, dy);
        u.z = df::mul(w, dz);
        if (df3_finite(u)) {
            slots_add(S, k, u);
        } else {
            // beyond the FP32 range (r^-3 above ~3e38): FP64 from the same parts
            const double X = df::to_double(dx), Y = df::to_double(dy), Z = df::to_double(dz);
            const double ri64 = 1.0 / sqrt(X * X + Y * Y + Z * Z + eps2d);
            const double w64 = ((double)m.h + (double)m.l) * ri64 * ri64 * ri64;
            S.wide[k][0] += w64 * X;
            S.wide[k][1] += w64 * Y;
            S.wide[k][2] += w64 * Z;
        }
    }
}

// ------------------------------------------------------------------------------------
// Newtonian pass
// ------------------------------------------------------------------------------------
// m_j r^-3 of a pair of sources; REFINE: with the first-order correction of the MUFU rsqrt,
// (r2 y^2)^(-3/2) = 1 - 3/2 (r2 y^2 - 1)
template <bool REFINE>
__device__ __forceinline__ float2 pair_weight(float2 r2, float2 m)
{
    const float2 y = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    const float2 y2 = __fmul2_rn(y, y);
    const float2 w = __fmul2_rn(__fmul2_rn(m, y), y2);
    if (!REFINE) return w;
    const float2 e = __ffma2_rn(r2, y2, dup(-1.f));
    return __ffma2_rn(__fmul2_rn(w, e), dup(-1.5f), w);
}

// ACC: the variant that feeds a gradient (refined rsqrt, folds of every tile, dominant terms in
// double-float by wmax).  Bound by the FP32 pipe (about 80 % of its cycles): 12 packed
// operations a pair of far pairs (18 with ACC) and about 250 instructions a tile.  All 65536
// particles of a Plummer sphere, with the sort: plain 2.50 -> 2.12 ms (1.97 with one rounding a
// tile); ACC with its prepass 4.50 -> 2.98 ms (2.72 with one of four roundings and sums of 16).
// 12 resident warps an SM without spills beat 16 to 20 with fewer registers.
template <bool ACC>
__global__ void __launch_bounds__(32, ACC ? 13 : 12) k_acc_tile(const float *__restrict__ rec, int n, int nsplit,
                                                                      float eps2, double eps2d,
                                                                      const float *__restrict__ wmax,
                                                                      double *__restrict__ part)
{
    __shared__ float4 s[8][TB];
    __shared__ Group W;
    Slots S;
    const int lane = threadIdx.x & 31, g = blockIdx.x, ntiles = (n + TJ - 1) / TJ;
    const Head *jh = heads(rec, n, P_ROWS);
    load_group(W, rec, n, P_ROWS, P_XL, g);
    const bool live0 = g * TJ + slot_of(0) < n, live1 = g * TJ + slot_of(1) < n;
    float thr[2] = {INFINITY, INFINITY}, qk[2] = {0.f, 0.f};
    int cnt[2] = {0, 0};
    if (ACC) {
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (g * TJ + slot_of(k) < n) thr[k] = SLOT_FRACTION * wmax[g * TJ + slot_of(k)];
        // r^2 m^(-2/3) at the threshold: a pair above it is below the threshold
#pragma unroll
        for (int k = 0; k < 2; ++k) qk[k] = 1.0001f * exp2f(-0.6666667f * log2f(thr[k]));
        slots_clear(S);
    }
    const float2 e2 = dup(eps2);
    for (int t0 = blockIdx.y; t0 < ntiles; t0 += 32 * nsplit) {
        unsigned fm, sm, lm;
        const float qf[2] = {cnt[0] < SLOTS ? qk[0] : 0.f, cnt[1] < SLOTS ? qk[1] : 0.f};
        judge_tiles<ACC>(W, jh, ntiles, t0, nsplit, g, live0, live1, ACC ? warp_max(fmaxf(qf[0], qf[1])) : 0.f, qf, fm, sm, lm);
        // the next tile's rows wait in registers: 64 pieces of the far rows, 128 of all
        auto next_bit = [&]() { return __ffs(fm ? fm : sm) - 1; };
        float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0, n3 = n0;
        auto fetch = [&]() {
            const float4 *tr = (const float4 *)(rec + (size_t)(t0 + next_bit() * nsplit) * P_ROWS * TJ);
            n0 = tr[lane];
            n1 = tr[32 + lane];
            if (!fm) {
                n2 = tr[64 + lane];
                n3 = tr[96 + lane];
            }
        };
        if (fm | sm) fetch();
        while (fm | sm) {
            const bool isfar = fm != 0u;
            const bool single = (lm >> next_bit()) & 1u;
            const int t = t0 + next_bit() * nsplit;
            if (fm) fm &= fm - 1;
            else sm &= sm - 1;
            const float4 c = jh[t].c;
            float4 *sf = &s[0][0];
            __syncwarp();
            sf[lane] = n0;
            sf[32 + lane] = n1;
            if (!isfar) {
                sf[64 + lane] = n2;
                sf[96 + lane] = n3;
            }
            __syncwarp();
            if (fm | sm) fetch();
            float xh[2][3], xl[2][3];
            offsets(W, c, xh, xl);
            // ACC: eight partial sums of eight a component and tile (two accumulators of two lanes
            // for each half)
            constexpr int NU = ACC ? 2 : 1, STEP = ACC ? TB / 2 : TB;
            float2 ax[2][NU], ay[2][NU], az[2][NU], sum[2][3];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                sum[k][0] = sum[k][1] = sum[k][2] = dup(0.f);
#pragma unroll
                for (int u = 0; u < NU; ++u) ax[k][u] = ay[k][u] = az[k][u] = dup(0.f);
            }
            auto take = [&]() {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    sum[k][0] = __fadd2_rn(sum[k][0], NU > 1 ? __fadd2_rn(ax[k][0], ax[k][NU - 1]) : ax[k][0]);
                    sum[k][1] = __fadd2_rn(sum[k][1], NU > 1 ? __fadd2_rn(ay[k][0], ay[k][NU - 1]) : ay[k][0]);
                    sum[k][2] = __fadd2_rn(sum[k][2], NU > 1 ? __fadd2_rn(az[k][0], az[k][NU - 1]) : az[k][0]);
#pragma unroll
                    for (int u = 0; u < NU; ++u) ax[k][u] = ay[k][u] = az[k][u] = dup(0.f);
                }
            };
            if (isfar || (ACC && single && !worth_search(W, c, jh[t].h, live0, live1, qk, cnt))) {
                // ACC: {-high part, -low part}; else four roundings (an addition a component less,
                // with an error of a below that of the MUFU rsqrt; one rounding for all
                // sources had a median error 2 % above the one-sided pass's, four 5 % below it)
                float2 nx[2][3][2];
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (ACC) {
                            nx[k][q][0] = dup(-xh[k][q]);
                            nx[k][q][1] = dup(-xl[k][q]);
                        } else {
                            four_roundings(xh[k][q], xl[k][q], nx[k][q]);
                        }
                    }
#pragma unroll 1
                for (int b0 = 0; b0 < TB; b0 += STEP) {
#pragma unroll 2
                    for (int b = b0; b < b0 + STEP; ++b) {
                        const float4 X = s[P_X][b], Y = s[P_Y][b], Z = s[P_Z][b], M = s[P_M][b];
#pragma unroll
                        for (int k = 0; k < 2; ++k)
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                const float2 dx = far_sep<ACC>(half_of(X, u), nx[k][0], u);
                                const float2 dy = far_sep<ACC>(half_of(Y, u), nx[k][1], u);
                                const float2 dz = far_sep<ACC>(half_of(Z, u), nx[k][2], u);
                                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
                                const float2 w = pair_weight<ACC>(r2, half_of(M, u));
                                ax[k][u % NU] = __ffma2_rn(w, dx, ax[k][u % NU]);
                                ay[k][u % NU] = __ffma2_rn(w, dy, ay[k][u % NU]);
                                az[k][u % NU] = __ffma2_rn(w, dz, az[k][u % NU]);
                            }
                    }
                    take();
                }
            } else {
                const bool diag = t == g;
                float2 nx[2][3], nl[2][3];
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int q = 0; q < 3; ++q) searched_offset(single, xh[k][q], xl[k][q], nx[k][q], nl[k][q]);
#pragma unroll 1
                for (int b = 0; b < TB; ++b) {
                    const float4 X = s[P_X][b], Y = s[P_Y][b], Z = s[P_Z][b], M = s[P_M][b];
                    const float4 XL = s[P_XL][b], YL = s[P_YL][b], ZL = s[P_ZL][b];
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float2 dx = __fadd2_rn(__fadd2_rn(half_of(X, u), nx[k][0]),
                                                         __fadd2_rn(half_of(XL, u), nl[k][0]));
                            const float2 dy = __fadd2_rn(__fadd2_rn(half_of(Y, u), nx[k][1]),
                                                         __fadd2_rn(half_of(YL, u), nl[k][1]));
                            const float2 dz = __fadd2_rn(__fadd2_rn(half_of(Z, u), nx[k][2]),
                                                         __fadd2_rn(half_of(ZL, u), nl[k][2]));
                            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
                            float2 w = pair_weight<ACC>(r2, half_of(M, u));
                            const int j = t * TJ + 4 * b + 2 * u;
                            if (diag) {
                                if (j == g * TJ + slot_of(k)) w.x = 0.f;
                                if (j + 1 == g * TJ + slot_of(k)) w.y = 0.f;
                            }
                            if (ACC && __any_sync(kFull, w.x > thr[k] || w.y > thr[k])) {
                                if (w.x > thr[k] && cnt[k] < SLOTS) {
                                    S.j[k][cnt[k]++] = j;
                                    w.x = 0.f;
                                }
                                if (w.y > thr[k] && cnt[k] < SLOTS) {
                                    S.j[k][cnt[k]++] = j + 1;
                                    w.y = 0.f;
                                }
                            }
                            ax[k][u % NU] = __ffma2_rn(w, dx, ax[k][u % NU]);
                            ay[k][u % NU] = __ffma2_rn(w, dy, ay[k][u % NU]);
                            az[k][u % NU] = __ffma2_rn(w, dz, az[k][u % NU]);
                        }
                    if ((b + 1) % STEP == 0) take();
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) fold_group(W, k, sum[k][0], sum[k][1], sum[k][2]);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int r = slot_of(k);
        if (ACC) acc_flush(S, rec, jh, g * TJ + slot_of(k), k, cnt[k], eps2d);
        if (g * TJ + r >= n) continue;
        double *p = part + (size_t)blockIdx.y * 3 * n + g * TJ + r;
        for (int q = 0; q < 3; ++q) {
            double v = group_total(W, q, r);
            if (ACC) v += slots_total(S, k, q);
            p[(size_t)q * n] = v;
        }
    }
}

// ------------------------------------------------------------------------------------
// gradient pass
// ------------------------------------------------------------------------------------
// the receivers' accelerations less their tile's mean
struct GroupA {
    float h[3][TJ], l[3][TJ];
};

__device__ __noinline__ void grad_flush(Slots &S, const float *__restrict__ rec, const Head *__restrict__ hd, int i, int k,
                                        int n, double eps2d)
{
    if (n == 0) return;
    const float *ti = rec + (size_t)(i / TJ) * G_ROWS * TJ + i % TJ;
    const float4 ci = hd[i / TJ].c, ai = hd[i / TJ].a;
    using df::dfloat;
    const dfloat e2 = df::from_double(eps2d);
    for (int s = 0; s < n; ++s) {
        const int j = S.j[k][s];
        const float *t = rec + (size_t)(j / TJ) * G_ROWS * TJ + j % TJ;
        const float4 c = hd[j / TJ].c, a = hd[j / TJ].a;
        const dfloat dx = tile_sep(c.x, t[G_X * TJ], t[G_XL * TJ], ci.x, ti[G_X * TJ], ti[G_XL * TJ]);
        const dfloat dy = tile_sep(c.y, t[G_Y * TJ], t[G_YL * TJ], ci.y, ti[G_Y * TJ], ti[G_YL * TJ]);
        const dfloat dz = tile_sep(c.z, t[G_Z * TJ], t[G_ZL * TJ], ci.z, ti[G_Z * TJ], ti[G_ZL * TJ]);
        const dfloat Ax = tile_sep(a.x, t[G_AX * TJ], t[G_AXL * TJ], ai.x, ti[G_AX * TJ], ti[G_AXL * TJ]);
        const dfloat Ay = tile_sep(a.y, t[G_AY * TJ], t[G_AYL * TJ], ai.y, ti[G_AY * TJ], ti[G_AYL * TJ]);
        const dfloat Az = tile_sep(a.z, t[G_AZ * TJ], t[G_AZL * TJ], ai.z, ti[G_AZ * TJ], ti[G_AZL * TJ]);
        const dfloat r2 = df::add(df::add(df::mul(dx, dx), df::mul(dy, dy)), df::add(df::mul(dz, dz), e2));
        const dfloat ri = df::rsqrt(r2);
        const dfloat ri2 = df::mul(ri, ri);
        const float m = t[G_M * TJ];
        const dfloat w = df::mul_f(df::mul(ri2, ri), m);
        const dfloat xa = df::add(df::add(df::mul(dx, Ax), df::mul(dy, Ay)), df::mul(dz, Az));
        const dfloat t3 = df::mul(df::mul_f(xa, 3.f), ri2);
        DF3 u;
        u.x = df::mul(w, df::sub(Ax, df::mul(t3, dx)));
        u.y = df::mul(w, df::sub(Ay, df::mul(t3, dy)));
        u.z = df::mul(w, df::sub(Az, df::mul(t3, dz)));
        if (df3_finite(u)) {
            slots_add(S, k, u);
        } else {
            const double X = df::to_double(dx), Y = df::to_double(dy), Z = df::to_double(dz);
            const double P = df::to_double(Ax), Q = df::to_double(Ay), R = df::to_double(Az);
            const double ri64 = 1.0 / sqrt(X * X + Y * Y + Z * Z + eps2d);
            const double w64 = (double)m * ri64 * ri64 * ri64;
            const double t64 = 3.0 * (X * P + Y * Q + Z * R) * ri64 * ri64;
            S.wide[k][0] += w64 * (P - t64 * X);
            S.wide[k][1] += w64 * (Q - t64 * Y);
            S.wide[k][2] += w64 * (R - t64 * Z);
        }
    }
}

// the pair term from a separation and a difference of accelerations; w: m_j r^-3 on return
__device__ __forceinline__ void grad_weight(float2 r2, float2 m, float2 &w, float2 &ri2)
{
    float2 y = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
    // one Newton-Raphson step, y <- y (3/2 - r2 y^2 / 2)
    const float2 nhy = __fmul2_rn(__fmul2_rn(dup(-0.5f), r2), y);
    y = __ffma2_rn(y, __ffma2_rn(nhy, y, dup(0.5f)), y);
    ri2 = __fmul2_rn(y, y);
    w = __fmul2_rn(__fmul2_rn(m, y), ri2);
}

// 33 packed operations a pair of far pairs (47 in the pass on absolute three-part positions), the
// FP32 pipe 84 % busy.  65536 particles: 6.35 -> 4.71 ms (4.42 with 27, one of four roundings a
// separation).  The registers of 10 warps an SM hold the loop without spills.
__global__ void __launch_bounds__(32, 10) k_grad_tile(const float *__restrict__ rec, int n, int nsplit, double eps2d,
                                                      const float *__restrict__ wmax, double *__restrict__ part)
{
    __shared__ float4 s[G_ROWS][TB];
    __shared__ Group W;
    __shared__ GroupA A;
    Slots S;
    const int lane = threadIdx.x & 31, g = blockIdx.x, ntiles = (n + TJ - 1) / TJ;
    const Head *jh = heads(rec, n, G_ROWS);
    load_group(W, rec, n, G_ROWS, G_XL, g);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            A.h[q][slot_of(k)] = rec[((size_t)g * G_ROWS + G_AX + q) * TJ + slot_of(k)];
            A.l[q][slot_of(k)] = rec[((size_t)g * G_ROWS + G_AXL + q) * TJ + slot_of(k)];
        }
    const bool live0 = g * TJ + slot_of(0) < n, live1 = g * TJ + slot_of(1) < n;
    float thr[2] = {INFINITY, INFINITY};
    int cnt[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (g * TJ + slot_of(k) < n) thr[k] = SLOT_FRACTION * wmax[g * TJ + slot_of(k)];
    float qk[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) qk[k] = 1.0001f * exp2f(-0.6666667f * log2f(thr[k]));
    slots_clear(S);
    const float2 e2 = dup((float)eps2d);
    for (int t0 = blockIdx.y; t0 < ntiles; t0 += 32 * nsplit) {
        unsigned fm, sm, lm;
        const float qf[2] = {cnt[0] < SLOTS ? qk[0] : 0.f, cnt[1] < SLOTS ? qk[1] : 0.f};
        judge_tiles<true>(W, jh, ntiles, t0, nsplit, g, live0, live1, warp_max(fmaxf(qf[0], qf[1])), qf, fm, sm, lm);
        auto next_bit = [&]() { return __ffs(fm ? fm : sm) - 1; };
        // the next tile's far rows wait in registers, 112 of its 208 pieces
        float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0, n3 = n0;
        auto fetch = [&]() {
            const float4 *tr = (const float4 *)(rec + (size_t)(t0 + next_bit() * nsplit) * G_ROWS * TJ);
            n0 = tr[lane];
            n1 = tr[32 + lane];
            n2 = tr[64 + lane];
            n3 = tr[96 + lane];
        };
        if (fm | sm) fetch();
        while (fm | sm) {
            const bool isfar = fm != 0u;
            const bool single = (lm >> next_bit()) & 1u;
            const int t = t0 + next_bit() * nsplit;
            if (fm) fm &= fm - 1;
            else sm &= sm - 1;
            const float4 c = jh[t].c, a = jh[t].a;
            float4 *sf = &s[0][0];
            __syncwarp();
            sf[lane] = n0;
            sf[32 + lane] = n1;
            sf[64 + lane] = n2;
            sf[96 + lane] = n3;
            if (!isfar) {
                const float4 *tr = (const float4 *)(rec + (size_t)t * G_ROWS * TJ);
                sf[128 + lane] = tr[128 + lane];
                sf[160 + lane] = tr[160 + lane];
                if (lane < 16) sf[192 + lane] = tr[192 + lane];
            }
            __syncwarp();
            if (fm | sm) fetch();
            float xh[2][3], xl[2][3];
            offsets(W, c, xh, xl);
            // the receivers' accelerations less the tile's mean
            float Ah[2][3], Al[2][3];
            {
                const float rc[3] = {W.head.a.x, W.head.a.y, W.head.a.z}, jc[3] = {a.x, a.y, a.z};
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    float p, e;
                    df::two_sum(rc[q], -jc[q], p, e);
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float r;
                        df::two_sum(p, A.h[q][slot_of(k)], Ah[k][q], r);
                        Al[k][q] = __fadd_rn(r, __fadd_rn(e, A.l[q][slot_of(k)]));
                    }
                }
            }
            // eight partial sums of eight a component and tile
            constexpr int STEP = TB / 2;
            float2 gx[2][2], gy[2][2], gz[2][2], sum[2][3];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                sum[k][0] = sum[k][1] = sum[k][2] = dup(0.f);
#pragma unroll
                for (int u = 0; u < 2; ++u) gx[k][u] = gy[k][u] = gz[k][u] = dup(0.f);
            }
            auto take = [&]() {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    sum[k][0] = __fadd2_rn(sum[k][0], __fadd2_rn(gx[k][0], gx[k][1]));
                    sum[k][1] = __fadd2_rn(sum[k][1], __fadd2_rn(gy[k][0], gy[k][1]));
                    sum[k][2] = __fadd2_rn(sum[k][2], __fadd2_rn(gz[k][0], gz[k][1]));
#pragma unroll
                    for (int u = 0; u < 2; ++u) gx[k][u] = gy[k][u] = gz[k][u] = dup(0.f);
                }
            };
            if (isfar || (single && !worth_search(W, c, jh[t].h, live0, live1, qk, cnt))) {
                float2 nx[2][3][2], na[2][3][2];
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        nx[k][q][0] = dup(-xh[k][q]);
                        nx[k][q][1] = dup(-xl[k][q]);
                        na[k][q][0] = dup(-Ah[k][q]);
                        na[k][q][1] = dup(-Al[k][q]);
                    }
#pragma unroll 1
                for (int b0 = 0; b0 < TB; b0 += STEP) {
#pragma unroll 2
                    for (int b = b0; b < b0 + STEP; ++b) {
                        const float4 X = s[G_X][b], Y = s[G_Y][b], Z = s[G_Z][b], M = s[G_M][b];
                        const float4 P = s[G_AX][b], Q = s[G_AY][b], R = s[G_AZ][b];
#pragma unroll
                        for (int k = 0; k < 2; ++k)
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                const float2 dx = far_sep<true>(half_of(X, u), nx[k][0], u);
                                const float2 dy = far_sep<true>(half_of(Y, u), nx[k][1], u);
                                const float2 dz = far_sep<true>(half_of(Z, u), nx[k][2], u);
                                const float2 Ax = far_sep<true>(half_of(P, u), na[k][0], u);
                                const float2 Ay = far_sep<true>(half_of(Q, u), na[k][1], u);
                                const float2 Az = far_sep<true>(half_of(R, u), na[k][2], u);
                                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
                                float2 w, ri2;
                                grad_weight(r2, half_of(M, u), w, ri2);
                                const float2 xa = __ffma2_rn(dx, Ax, __ffma2_rn(dy, Ay, __fmul2_rn(dz, Az)));
                                const float2 nt3 = __fmul2_rn(__fmul2_rn(dup(-3.f), xa), ri2);
                                gx[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dx, Ax), gx[k][u]);
                                gy[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dy, Ay), gy[k][u]);
                                gz[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dz, Az), gz[k][u]);
                            }
                    }
                    take();
                }
            } else {
                const bool diag = t == g;
                float2 nx[2][3], nl[2][3], na[2][3], ma[2][3];
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        searched_offset(single, xh[k][q], xl[k][q], nx[k][q], nl[k][q]);
                        searched_offset(single, Ah[k][q], Al[k][q], na[k][q], ma[k][q]);
                    }
#pragma unroll 1
                for (int b = 0; b < TB; ++b) {
                    const float4 X = s[G_X][b], Y = s[G_Y][b], Z = s[G_Z][b], M = s[G_M][b];
                    const float4 P = s[G_AX][b], Q = s[G_AY][b], R = s[G_AZ][b];
                    const float4 XL = s[G_XL][b], YL = s[G_YL][b], ZL = s[G_ZL][b];
                    const float4 PL = s[G_AXL][b], QL = s[G_AYL][b], RL = s[G_AZL][b];
#pragma unroll
                    for (int k = 0; k < 2; ++k)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float2 dx = __fadd2_rn(__fadd2_rn(half_of(X, u), nx[k][0]), __fadd2_rn(half_of(XL, u), nl[k][0]));
                            const float2 dy = __fadd2_rn(__fadd2_rn(half_of(Y, u), nx[k][1]), __fadd2_rn(half_of(YL, u), nl[k][1]));
                            const float2 dz = __fadd2_rn(__fadd2_rn(half_of(Z, u), nx[k][2]), __fadd2_rn(half_of(ZL, u), nl[k][2]));
                            const float2 Ax = __fadd2_rn(__fadd2_rn(half_of(P, u), na[k][0]), __fadd2_rn(half_of(PL, u), ma[k][0]));
                            const float2 Ay = __fadd2_rn(__fadd2_rn(half_of(Q, u), na[k][1]), __fadd2_rn(half_of(QL, u), ma[k][1]));
                            const float2 Az = __fadd2_rn(__fadd2_rn(half_of(R, u), na[k][2]), __fadd2_rn(half_of(RL, u), ma[k][2]));
                            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
                            float2 w, ri2;
                            grad_weight(r2, half_of(M, u), w, ri2);
                            const int j = t * TJ + 4 * b + 2 * u;
                            if (diag) {
                                // the self pair: no weight, and no NaN of its 0 x infinity
                                if (j == g * TJ + slot_of(k)) w.x = ri2.x = 0.f;
                                if (j + 1 == g * TJ + slot_of(k)) w.y = ri2.y = 0.f;
                            }
                            if (__any_sync(kFull, w.x > thr[k] || w.y > thr[k])) {
                                if (w.x > thr[k] && cnt[k] < SLOTS) {
                                    S.j[k][cnt[k]++] = j;
                                    w.x = 0.f;
                                }
                                if (w.y > thr[k] && cnt[k] < SLOTS) {
                                    S.j[k][cnt[k]++] = j + 1;
                                    w.y = 0.f;
                                }
                            }
                            const float2 xa = __ffma2_rn(dx, Ax, __ffma2_rn(dy, Ay, __fmul2_rn(dz, Az)));
                            const float2 nt3 = __fmul2_rn(__fmul2_rn(dup(-3.f), xa), ri2);
                            gx[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dx, Ax), gx[k][u]);
                            gy[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dy, Ay), gy[k][u]);
                            gz[k][u] = __ffma2_rn(w, __ffma2_rn(nt3, dz, Az), gz[k][u]);
                        }
                    if ((b + 1) % STEP == 0) take();
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) fold_group(W, k, sum[k][0], sum[k][1], sum[k][2]);
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int r = slot_of(k);
        grad_flush(S, rec, jh, g * TJ + slot_of(k), k, cnt[k], eps2d);
        if (g * TJ + r >= n) continue;
        double *p = part + (size_t)blockIdx.y * 3 * n + g * TJ + r;
        for (int q = 0; q < 3; ++q)
            p[(size_t)q * n] = group_total(W, q, r) + slots_total(S, k, q);
    }
}

// ------------------------------------------------------------------------------------
// potential
// ------------------------------------------------------------------------------------
// phi_i = sum over the particles after i in the list of m_j / sqrt(r^2 + eps^2), in double-float
// like k_potential_df, whose operations are for the most part the exact separation from
// three-part absolute positions (81 of 143 a pair).  Against a tile's centre a far pair's
// separation is good to 2^-48 of the tile's radius, below 2^-45 of the distance, for 24.
// The double-float sums run over a tile's 64 terms and are added up in FP64.  (Where a close pair's
// term H leads, every later addition leaves up to half a unit of H to the low sum, an FP32 sum,
// whose own rounding grows as their number: over the 512 terms of a split U of 20001 stars with
// hard binaries was 9e-15 off (rms of 16 systems), over the 128 of k_potential_df 1.4e-15.)
// Scalar FP32 throughput bounds it: 65536 particles 10.8 ms on every pair's absolute positions, 7.5 so.
__global__ void __launch_bounds__(32) k_potential_tile(const int32_t *__restrict__ list, const float *__restrict__ rec,
                                                       const float4 *__restrict__ abs, int n, int nsplit, double eps2,
                                                       double *__restrict__ part)
{
    __shared__ float4 s[8][TB];
    __shared__ Group W;
    const int lane = threadIdx.x & 31, g = blockIdx.x, ntiles = (n + TJ - 1) / TJ;
    const Head *jh = heads(rec, n, P_ROWS);
    load_group(W, rec, n, P_ROWS, P_XL, g);
    const df::dfloat e2 = df::from_double(eps2);
    double sum[2] = {0.0, 0.0};
    for (int t = g + blockIdx.y; t < ntiles; t += nsplit) {
        float H[2] = {0.f, 0.f}, L[2] = {0.f, 0.f};
        const float4 c = jh[t].c, h = jh[t].h;
        const float d2 = box_gap2(W.head.c, W.head.h, c, h);
        if (t != g && d2 > 0.f && d2 >= (kFarRadius * kFarRadius) * c.w * c.w) {
            const float4 *tr = (const float4 *)(rec + (size_t)t * P_ROWS * TJ);
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 4; ++q) (&s[0][0])[32 * q + lane] = tr[32 * q + lane];
            __syncwarp();
            float xh[2][3], xl[2][3];
            offsets(W, c, xh, xl);
#pragma unroll 1
            for (int b = 0; b < TB; ++b) {
                float J[8][4];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float4 v = s[r][b];
                    J[r][0] = v.x; J[r][1] = v.y; J[r][2] = v.z; J[r][3] = v.w;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        float d[3], e[3], w, we;
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            df::two_sum(J[P_X + q][u], -xh[k][q], d[q], e[q]);
                            e[q] = __fadd_rn(e[q], __fsub_rn(J[P_XL + q][u], xl[k][q]));
                        }
                        df::mass_over_r(d[0], e[0], d[1], e[1], d[2], e[2], e2.h, e2.l, J[P_M][u], J[P_ML][u], w, we);
                        float r;
                        df::two_sum(H[k], w, H[k], r);
                        L[k] += r + we;
                    }
            }
        } else {
            const int cnt = min(TJ, n - t * TJ);
            float4 I0[2], I1[2], I2[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int i = min(g * TJ + slot_of(k), n - 1);
                I0[k] = abs[i];
                I1[k] = abs[n + i];
                I2[k] = abs[2 * n + i];
            }
#pragma unroll 2
            for (int jj = 0; jj < cnt; ++jj) {
                const int j = t * TJ + jj;
                const float4 J0 = abs[j], J1 = abs[n + j], J2 = abs[2 * n + j];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const df::dfloat dx = df::sep(J0.x, J1.x, J2.x, I0[k].x, I1[k].x, I2[k].x);
                    const df::dfloat dy = df::sep(J0.y, J1.y, J2.y, I0[k].y, I1[k].y, I2[k].y);
                    const df::dfloat dz = df::sep(J0.z, J1.z, J2.z, I0[k].z, I1[k].z, I2[k].z);
                    float w, we;
                    df::mass_over_r(dx.h, dx.l, dy.h, dy.l, dz.h, dz.l, e2.h, e2.l, J0.w, J1.w, w, we);
                    if (j > g * TJ + slot_of(k)) {
                        float r;
                        df::two_sum(H[k], w, H[k], r);
                        L[k] += r + we;
                    }
                }
            }
        }
        // the low parts of more terms in one FP32 sum lose what a close pair's term needs
#pragma unroll
        for (int k = 0; k < 2; ++k) sum[k] += f2d(H[k]) + f2d(L[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = g * TJ + slot_of(k);
        if (i < n) part[(size_t)blockIdx.y * n + list[i]] = sum[k];
    }
}

}  // namespace

int potential_tile_splits(int n, int n_sm, size_t part_elems)
{
    const long long ngroups = (n + TJ - 1) / TJ;
    // rows of the triangle get shorter: sixteen rounds of about 16 resident warps an SM
    const long long ns = std::min((16LL * 16 * n_sm + ngroups - 1) / ngroups, (ngroups + 7) / 8);
    return (int)std::max<long long>(1, std::min<long long>(ns, (long long)(part_elems / (size_t)n)));
}

void launch_potential_tile(cudaStream_t s, const int32_t *list, const void *rec, const float4 *abs, int n, double eps2,
                           int nsplit, double *part)
{
    k_potential_tile<<<dim3((n + TJ - 1) / TJ, nsplit), 32, 0, s>>>(list, (const float *)rec, abs, n, nsplit, eps2, part);
}

int tile_splits(int n, int n_sm, size_t part_elems)
{
    const long long ntiles = (n + TJ - 1) / TJ;
    // eight rounds of about 20 resident warps an SM, each warp 16 tiles at least (its slots, a few
    // double-float terms a lane whatever it sees, cost as much as several tiles: with 4 tiles a
    // warp a 65536-body step took 55.4 ms, with 16 52.3), the partials within their buffer
    long long ns = std::min((8LL * 20 * n_sm + ntiles - 1) / ntiles, (ntiles + 15) / 16);
    ns = std::min<long long>(ns, (long long)(part_elems / (3 * (size_t)n)));
    return (int)std::max<long long>(1, ns);
}

void launch_tile_pack_pos(cudaStream_t s, const int32_t *list, int n, double *x, const double *v, double dt,
                          const double *m, int N, void *rec)
{
    if (n <= 0) return;
    k_tile_pack<false><<<(n + 4 * TJ - 1) / (4 * TJ), 128, 0, s>>>(list, n, x, v, dt, m, N, nullptr, nullptr, (float *)rec);
}

void launch_tile_pack_grad(cudaStream_t s, const int32_t *list, int n, const double *x, const double *m, int N,
                           const double *acc, const uint32_t *hot, void *rec)
{
    if (n <= 0) return;
    k_tile_pack<true><<<(n + 4 * TJ - 1) / (4 * TJ), 128, 0, s>>>(list, n, const_cast<double *>(x), nullptr, 0.0, m, N, acc, hot,
                                                      (float *)rec);
}

void launch_wmax_tile(cudaStream_t s, const TileArgs &a, int n_sm, float *wmax)
{
    cudaMemsetAsync(wmax, 0, sizeof(float) * a.n, s);
    const int ntiles = (a.n + TJ - 1) / TJ;
    // few tiles are looked into, so a group is split only to fill the SMs
    const int ns = std::max(1, std::min((ntiles + 31) / 32, (16 * n_sm + ntiles - 1) / ntiles));
    k_wmax_tile<<<dim3(ntiles, ns), 32, 0, s>>>((const float *)a.rec, a.n, ns, (float)a.eps2, wmax);
}

void launch_acc_tile(cudaStream_t s, const TileArgs &a, const float *wmax)
{
    const dim3 grid((a.n + TJ - 1) / TJ, a.nsplit);
    if (wmax)
        k_acc_tile<true><<<grid, 32, 0, s>>>((const float *)a.rec, a.n, a.nsplit, (float)a.eps2, a.eps2, wmax, a.part);
    else
        k_acc_tile<false><<<grid, 32, 0, s>>>((const float *)a.rec, a.n, a.nsplit, (float)a.eps2, a.eps2, nullptr, a.part);
}

void launch_grad_tile(cudaStream_t s, const TileArgs &a, const float *wmax)
{
    k_grad_tile<<<dim3((a.n + TJ - 1) / TJ, a.nsplit), 32, 0, s>>>((const float *)a.rec, a.n, a.nsplit, a.eps2, wmax, a.part);
}

}  // namespace frost
