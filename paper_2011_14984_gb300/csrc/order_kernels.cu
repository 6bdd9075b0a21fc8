// Spatial order of an index list for the tile kernels (tile_kernels.cu) on sm_103a.
//
// The tile kernels group 64 receivers and 32 sources at a time and treat a pair of groups by
// their boxes, so a list whose neighbours in the list are neighbours in space makes most pairs
// of groups well separated.  The order is that of a Hilbert curve over a 128^3 grid of
// companded coordinates u = d / (s + |d|), d the offset from the componentwise median and s
// the median |d| of the component (both of a strided sample of 128 members): a star cluster's
// core and halo then get cells of about equal occupancy.  Only the speed of the passes depends
// on how well the order fits; the boxes are those of the actual members.
//
// 21-bit keys are sorted by two stable counting passes (11 and 10 bits; an LSD radix sort):
// per pass a histogram per block and a scatter whose ranks are fixed by position, so the order
// is a function of the positions and the list alone.  Bound by launches and latency, not
// bytes (12 B per member and pass): four launches, about 60 us for 40603 members (a scan kernel
// between the passes and medians over 256 samples in FP64 took it to 350).  Hilbert rather than
// Morton order and companded per coordinate rather than by radius: of the 64 x 32 pairs of
// groups of a 65536-body Plummer sphere 64 % (Morton 53 %) have their boxes further than two
// group radii from the group's centre, and 81 % (64 % companded by radius) are further apart
// than half a group radius.
#include "frost_internal.cuh"

#include <cmath>

namespace frost {
namespace {

constexpr int OB = 256;                 // threads a block
constexpr int OW = OB / 32;
constexpr int OPT = 8;                  // entries a thread
constexpr int OCHUNK = OB * OPT;        // entries a block
constexpr int LOW_BITS = 11, HIGH_BITS = 10;
constexpr int GRID_BITS = 7;            // cells per dimension: 2^7
static_assert(3 * GRID_BITS == LOW_BITS + HIGH_BITS, "key digits");
constexpr int SAMPLE = 128;
static_assert(OCHUNK == ORDER_CHUNK && (1 << LOW_BITS) == ORDER_DIGITS, "workspace sizes in frost_internal.cuh");

// The medians of three components of SAMPLE values, one per thread (by counting ranks, ties by
// thread index; four values a load, since the loop is bound by the latency of its loads)
__device__ void sample_medians(const float (&v)[3], float4 (*s_val)[SAMPLE / 4], float *s_med, float (&med)[3])
{
    const int t = threadIdx.x;
    __syncthreads();
    if (t < SAMPLE)
#pragma unroll
        for (int c = 0; c < 3; ++c) ((float *)s_val[c])[t] = v[c];
    __syncthreads();
    int rank[3] = {0, 0, 0};
#pragma unroll 4
    for (int q = 0; q < SAMPLE / 4 && t < SAMPLE; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 u = s_val[c][q];
            const int k = 4 * q;
            rank[c] += (u.x < v[c] || (u.x == v[c] && k < t)) + (u.y < v[c] || (u.y == v[c] && k + 1 < t)) +
                       (u.z < v[c] || (u.z == v[c] && k + 2 < t)) + (u.w < v[c] || (u.w == v[c] && k + 3 < t));
        }
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (t < SAMPLE && rank[c] == SAMPLE / 2) s_med[c] = v[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) med[c] = s_med[c];
}

// Hilbert index of a cell (Skilling's transposed form, AIP Conf. Proc. 707, 381 (2004))
__device__ __forceinline__ unsigned hilbert_key(unsigned x, unsigned y, unsigned z)
{
    unsigned X[3] = {x, y, z};
#pragma unroll
    for (unsigned Q = 1u << (GRID_BITS - 1); Q > 1; Q >>= 1) {
        const unsigned P = Q - 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (X[i] & Q) {
                X[0] ^= P;
            } else {
                const unsigned t = (X[0] ^ X[i]) & P;
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];
    X[2] ^= X[1];
    unsigned t = 0;
#pragma unroll
    for (unsigned Q = 1u << (GRID_BITS - 1); Q > 1; Q >>= 1)
        if (X[2] & Q) t ^= Q - 1;
    unsigned key = 0;
#pragma unroll
    for (int b = GRID_BITS - 1; b >= 0; --b)
#pragma unroll
        for (int i = 0; i < 3; ++i) key = (key << 1) | (((X[i] ^ t) >> b) & 1u);
    return key;
}

// Stable ranks of the block's entries by digit: warp w owns the entries [256 w, 256 (w + 1)) of
// the chunk, 32 consecutive ones a round.  rank[q]: the entries before this one in its warp
// with the same digit; s_cnt[w][d]: the warp's entries with digit d.
template <int BITS>
__device__ __forceinline__ void warp_ranks(const unsigned (&digit)[OPT], const bool (&live)[OPT], uint16_t *cnt,
                                           int (&rank)[OPT])
{
    const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < OPT; ++q) {
        const unsigned key = live[q] ? digit[q] : 0xffffffffu;
        const unsigned same = __match_any_sync(0xffffffffu, key);
        int base = 0;
        if (live[q]) base = cnt[digit[q]];
        __syncwarp();
        rank[q] = base + __popc(same & below);
        if (live[q] && (same & below) == 0u) cnt[digit[q]] = (uint16_t)(base + __popc(same));
        __syncwarp();
    }
}

// keys of the list and the histogram of their low digits per block
__global__ void __launch_bounds__(OB) k_order_keys(const int32_t *__restrict__ list, int n, const double *__restrict__ x,
                                                   int N, unsigned *__restrict__ key, int *__restrict__ hist)
{
    __shared__ float4 s_val[3][SAMPLE / 4];
    __shared__ float s_med[3];
    __shared__ int s_hist[1 << LOW_BITS];
    const int tid = threadIdx.x;
    float c[3], s[3];
    {
        const int k = (int)((long long)(tid % SAMPLE) * n / SAMPLE);
        const int i = list ? list[k] : k;
        const float v[3] = {(float)x[i], (float)x[(size_t)N + i], (float)x[(size_t)2 * N + i]};
        sample_medians(v, s_val, s_med, c);
        const float d[3] = {fabsf(v[0] - c[0]), fabsf(v[1] - c[1]), fabsf(v[2] - c[2])};
        sample_medians(d, s_val, s_med, s);
    }
    for (int d = tid; d < (1 << LOW_BITS); d += OB) s_hist[d] = 0;
    __syncthreads();
    for (int q = 0; q < OPT; ++q) {
        const int k = blockIdx.x * OCHUNK + q * OB + tid;
        if (k >= n) break;
        const int i = list ? list[k] : k;
        unsigned cell[3];
        for (int e = 0; e < 3; ++e) {
            const float d = (float)x[(size_t)e * N + i] - c[e];
            const float u = d / (s[e] + fabsf(d) + 1e-30f);
            cell[e] = (unsigned)min((1 << GRID_BITS) - 1, max(0, (int)((u + 1.f) * (0.5f * (1 << GRID_BITS)))));
        }
        const unsigned key_k = hilbert_key(cell[0], cell[1], cell[2]);
        key[k] = key_k;
        atomicAdd(&s_hist[key_k & ((1u << LOW_BITS) - 1u)], 1);
    }
    __syncthreads();
    for (int d = tid; d < (1 << LOW_BITS); d += OB) hist[((size_t)blockIdx.x << LOW_BITS) + d] = s_hist[d];
}

// histogram of the high digits of the keys after the first pass
__global__ void __launch_bounds__(OB) k_order_hist(const unsigned *__restrict__ key, int n, int *__restrict__ hist)
{
    __shared__ int s_hist[1 << HIGH_BITS];
    const int tid = threadIdx.x;
    for (int d = tid; d < (1 << HIGH_BITS); d += OB) s_hist[d] = 0;
    __syncthreads();
    for (int q = 0; q < OPT; ++q) {
        const int k = blockIdx.x * OCHUNK + q * OB + tid;
        if (k < n) atomicAdd(&s_hist[key[k] >> LOW_BITS], 1);
    }
    __syncthreads();
    for (int d = tid; d < (1 << HIGH_BITS); d += OB) hist[((size_t)blockIdx.x << HIGH_BITS) + d] = s_hist[d];
}

// one stable counting pass: entry k goes behind all entries of lower digits, those of its digit
// in earlier blocks (every block sums the histograms hist[block][digit] itself: a scan kernel
// in between cost as much as the pass) and those before it in its block.  FIRST: payload k
// itself, keys carried on; else payload pos_in, and the sorted list is written
template <int BITS, bool FIRST>
__global__ void __launch_bounds__(OB) k_order_scatter(const unsigned *__restrict__ key, const int32_t *__restrict__ pos_in,
                                                      const int32_t *__restrict__ list, int n,
                                                      const int *__restrict__ hist, unsigned *__restrict__ key_out,
                                                      int32_t *__restrict__ pos_out, int32_t *__restrict__ list_out)
{
    extern __shared__ uint16_t s_cnt[];  // [OW][1 << BITS]
    constexpr int D = 1 << BITS, DPT = D / OB;
    __shared__ int s_base[D];
    __shared__ int s_w[OW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // s_base[d]: the entries of lower digits, and those of digit d in earlier blocks
    {
        int tot[DPT], before[DPT];
#pragma unroll
        for (int e = 0; e < DPT; ++e) tot[e] = before[e] = 0;
        for (int b = 0; b < (int)gridDim.x; ++b)
#pragma unroll
            for (int e = 0; e < DPT; ++e) {
                const int c = hist[(size_t)b * D + e * OB + tid];
                tot[e] += c;
                if (b < (int)blockIdx.x) before[e] += c;
            }
        // scan of the totals, OB digits at a time
        int carry = 0;
#pragma unroll
        for (int e = 0; e < DPT; ++e) {
            int inc = tot[e];
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += u;
            }
            __syncthreads();
            if (lane == 31) s_w[warp] = inc;
            __syncthreads();
            int pre = carry;
#pragma unroll
            for (int w = 0; w < OW; ++w) {
                if (w < warp) pre += s_w[w];
                carry += s_w[w];
            }
            s_base[e * OB + tid] = pre + inc - tot[e] + before[e];
        }
    }
    for (int d = tid; d < OW * D; d += OB) s_cnt[d] = 0;
    __syncthreads();
    unsigned kk[OPT], digit[OPT];
    bool live[OPT];
    int rank[OPT];
    const int k0 = blockIdx.x * OCHUNK + warp * (32 * OPT) + lane;
#pragma unroll
    for (int q = 0; q < OPT; ++q) {
        const int k = k0 + 32 * q;
        live[q] = k < n;
        kk[q] = live[q] ? key[k] : 0u;
        digit[q] = FIRST ? (kk[q] & (D - 1)) : (kk[q] >> LOW_BITS);
    }
    warp_ranks<BITS>(digit, live, s_cnt + warp * D, rank);
    __syncthreads();
    // exclusive sums over the warps, per digit
    for (int d = tid; d < D; d += OB) {
        int at = 0;
        for (int w = 0; w < OW; ++w) {
            const int c = s_cnt[w * D + d];
            s_cnt[w * D + d] = (uint16_t)at;
            at += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < OPT; ++q) {
        if (!live[q]) continue;
        const int k = k0 + 32 * q;
        const int at = s_base[digit[q]] + s_cnt[warp * D + digit[q]] + rank[q];
        if (FIRST) {
            key_out[at] = kk[q];
            pos_out[at] = k;
        } else {
            const int p = pos_in[k];
            pos_out[at] = p;
            list_out[at] = list ? list[p] : p;
        }
    }
}

}  // namespace

void launch_spatial_order(cudaStream_t s, const int32_t *list, int n, const double *x, int N, const OrderWork &w,
                          int32_t *pos, int32_t *sorted)
{
    if (n <= 0) return;
    const int nb = order_blocks(n);
    k_order_keys<<<nb, OB, 0, s>>>(list, n, x, N, w.key, w.hist);
    k_order_scatter<LOW_BITS, true><<<nb, OB, OW * sizeof(uint16_t) << LOW_BITS, s>>>(w.key, nullptr, list, n, w.hist,
                                                                                     w.key2, w.pos2, nullptr);
    k_order_hist<<<nb, OB, 0, s>>>(w.key2, n, w.hist);
    k_order_scatter<HIGH_BITS, false><<<nb, OB, OW * sizeof(uint16_t) << HIGH_BITS, s>>>(w.key2, w.pos2, list, n, w.hist,
                                                                                        nullptr, pos, sorted);
}

}  // namespace frost
