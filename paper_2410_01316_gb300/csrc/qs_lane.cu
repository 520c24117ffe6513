// Grid stages with one slice per lane (arXiv 2410.01316, App. C Step 3, eq.
// 1d_sum_fourier): the spread, the filter and the interpolation of large
// problems.  A warp holds 32 slices, lane l slice 32 g + l, and walks over
// points; the grids of the 32 slices lie interleaved in shared memory, cell c
// of lane l at [c][l], so that every tap of every point is one conflict-free
// access whatever the points' order and spread.  (With one slice per CTA and
// one point per lane the taps of a warp fall on random banks: 2.6 wavefronts
// an access, measured, against 1.0 here for loads and integer atomics alike.)
// The points are the same for all lanes, so up to d = 64 the FP32 forms take
// the projection as d FMAs per point and lane from broadcast coordinates and
// registers, and nothing goes through HBM; the tensor-core forms write their projections
// slice-interleaved (U[g][n][32]), one coalesced row per point and warp.
//
// Only a window of each slice's grid is kept in shared memory, placed per
// slice by a sample of the points.  A narrow one holds polynomials (spread:
// K moments per bin; interpolation: K coefficients per bin), which cost K
// products per point; a wide one plain cells, W taps of K/2 + 1 FMAs.  A point
// outside its window takes the slow way, directly on the grid in global
// memory, so the window only ever decides the speed.  Where the sample spans
// more than the shared memory holds, the points are walked once per window.
//
// No unit is full: 2.0 to 3.0 of 4 warp instructions a clock, the load / store
// pipe at 36 to 71 %, FP32 at 28 to 40 %.  Warp instructions per 32 point-slices,
// projection included where it is done here: spread 53 (moments, U read) to 92
// (cells, d = 16), interpolation 47 (polynomials, U read; 10 of them the compensated
// sums) to 74 (derivative, d = 16).
// Kernel times against the kernels with one point per lane (us):
//   spread         d = 784, 6e4 points, P = 2048, G = 2048    822 (one kernel with the filter) -> 215 + 34
//                  d = 64, 2e5, P = 1024, G = 4096            814 -> 537 + 39
//                  d = 30, 9.6e5, P = 1280, G = 256           7590 + 2123 (projection) -> 3608 + 8
//                  d = 16, 2e5, P = 1024, G = 2048            740 and a projection (316 with that of y) -> 712 + 20
//   interpolation  d = 784  344 -> 203   d = 64  867 -> 525   d = 30  3180 + 2129 -> 3143
#include <cuda_bf16.h>
#include <float.h>
#include <limits.h>
#include <math.h>

#include "qs_device.cuh"
#include "qs_internal.cuh"

using namespace qsdev;

namespace {

constexpr int W = QS_LANE_W;
constexpr int HW = W / 2;
constexpr int K = qs_moment_count(W);
constexpr int T4 = qs_tap_terms(W);
static_assert(K == 2 * T4, "one moment per polynomial coefficient");
constexpr int SUB = 8;       // points of a warp's staging block
constexpr int NSAMPLE = 256; // points of the sample that places the window

// x + MAGIC is x rounded to the nearest integer in the low mantissa bits for
// |x| < 2^22: one FP32 addition instead of a conversion, of which an SM does
// 16 a clock (measured: 2.0 clocks per warp) against 128 additions.
constexpr float MAGIC = 12582912.0f;
constexpr int MAGIC_BITS = 0x4B400000;

// Threads per CTA (one CTA per SM).  A lane holds its slice's direction and
// the window's 32 coefficients in registers: as FP32x2 pairs a point's taps
// are then 12 packed and 8 scalar FMAs, against 32 FMAs each behind a load of
// its coefficient from the constant bank when they are left there.
__host__ __device__ constexpr int spread_threads(int D) { return D == 0 ? 768 : (D <= 16 ? 512 : 384); }
__host__ __device__ constexpr int interp_threads(int D) { return D <= 16 ? 512 : 384; }
// Slices a lane can hold: two where a point's coordinates are many enough that reading them once for both
// pays (a 16-byte broadcast takes the shared memory 2 clocks, as many as two taps) and the registers hold
// both directions.  Their windows have to fit side by side, so it is decided per group of 64 slices, on the
// spans that the sample finds.  d = 30, 2 x 9.6e5 points, P = 1280: spread 4.02 -> 3.49 ms, interpolation
// 4.70 -> 3.41 ms; at d = 16 two thirds of the sums are slower with it (windows that only fit singly double
// the clearing and adding up), at d = 48 the second direction spills (1.55 -> 1.62 ms).
__host__ __device__ constexpr int lane_slices(int D) { return D == 32 ? 2 : 1; }
// Each warp stages its points two blocks of SUB at a time: coordinates (row
// stride D, zeros past d), or projections of the 32 slices (D = 0).
__host__ __device__ constexpr int lane_stride(int D) { return D > 0 ? D : 32; }
__host__ __device__ constexpr int lane_ring_floats(int D) { return 2 * SUB * lane_stride(D); }
__host__ __device__ constexpr int lane_ring_bytes(int D, int threads) { return threads / 32 * lane_ring_floats(D) * 4; }

// Two FP32 numbers in a 64-bit register: packed arithmetic takes aligned
// register pairs, which 64-bit operands are without moves.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <int B>
__device__ __forceinline__ void cp_async_small(void* smem, const void* gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem),
                 "n"(B)
                 : "memory");
}

// Widest copy (floats) that keeps to the rows of d coordinates at x.
__device__ __forceinline__ int copy_width(const float* x, int d)
{
    const unsigned a = (unsigned)(reinterpret_cast<uintptr_t>(x) >> 2) | (unsigned)d;
    return (a & 3) == 0 ? 4 : ((a & 1) == 0 ? 2 : 1);
}

// Copy the `cnt` rows of d coordinates at src to dst with row stride D (the
// tail of a row stays zero), `width` floats at a time; inv = 65536 / d + 1:
// e inv >> 16 is the exact row of element e < 512.
template <int D>
__device__ __forceinline__ void stage_points(float* dst, const float* __restrict__ src, int cnt, int d, int width,
                                             unsigned inv, int lane)
{
    const int tot = cnt * d;
    if (d == D && width == 4) {
        for (int e = 4 * lane; e < tot; e += 128) cp_async16(dst + e, src + e);
        return;
    }
    for (int e = width * lane; e < tot; e += 32 * width) {
        const int r = (int)(((unsigned)e * inv) >> 16);
        float* o = dst + r * D + (e - r * d);
        if (width == 4) cp_async16(o, src + e);
        else if (width == 2) cp_async_small<8>(o, src + e);
        else cp_async_small<4>(o, src + e);
    }
}

// The projections of SUB points (8 rows of 32 slices, contiguous): two 16-byte copies per lane.
__device__ __forceinline__ void stage_rows(float* dst, const float* __restrict__ src, int lane)
{
    cp_async16(dst + 4 * lane, src + 4 * lane);
    cp_async16(dst + 128 + 4 * lane, src + 128 + 4 * lane);
}

// The lane's direction: coordinates 2 j, 2 j + 1 (0 past d, and in the lanes past P).
template <int D>
struct Direction {
    f32x2 c[D > 0 ? D / 2 : 1];
};

// The directions of the group's slices, lane l's at p0 + 32 h + l, by way of shared memory: read by every
// lane from global memory they would cost each warp 32 lines per coordinate (12 us of a CTA of 12 warps at
// d = 30).  scratch: 32 SL (D + 1) floats.  Begins and ends with a barrier.
template <int D, int SL>
__device__ __forceinline__ void share_xi(const qs_launch& L, int p0, Direction<D>* xi, float* scratch)
{
    if constexpr (D > 0) {
        const int lane = threadIdx.x & 31, d = L.d, rows = min(32 * SL, L.P - p0);
        const float* src = L.xi_s + (size_t)p0 * d;
        __syncthreads();
        for (int e = threadIdx.x; e < 32 * SL * d; e += blockDim.x) {
            const int r = e / d;
            scratch[r * (D + 1) + (e - r * d)] = r < rows ? __ldg(&src[e]) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < SL; ++h) {
            const float* row = scratch + (32 * h + lane) * (D + 1);
#pragma unroll
            for (int j = 0; j < D; j += 2) xi[h].c[j / 2] = pack2(j < d ? row[j] : 0.0f, j + 1 < d ? row[j + 1] : 0.0f);
        }
        __syncthreads();
    }
}

// Grid coordinates of the staged point at r on the lane's slices: FP32 products summed in four strands
// (coordinates mod 4), added at the end.
template <int D, int SL>
__device__ __forceinline__ void ring_u(const float* r, const Direction<D>* xi, int lane, float (&u)[SL])
{
    if constexpr (D > 0) {
        f32x2 a[SL], b[SL];
#pragma unroll
        for (int j = 0; j < D; j += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(r + j);
#pragma unroll
            for (int h = 0; h < SL; ++h) {
                a[h] = j == 0 ? mul2(xi[h].c[0], v.x) : fma2(xi[h].c[j / 2], v.x, a[h]);
                b[h] = j == 0 ? mul2(xi[h].c[1], v.y) : fma2(xi[h].c[j / 2 + 1], v.y, b[h]);
            }
        }
#pragma unroll
        for (int h = 0; h < SL; ++h) {
            const float2 t = unpack2(add2(a[h], b[h]));
            u[h] = t.x + t.y;
        }
    } else {
        u[0] = r[lane];
    }
}

// First tap cell l0 = rint(u - m + 1/2) as the low bits of the float
// l0 + MAGIC, and s = u - l0 - (m - 1/2) in [-1/2, 1/2].  A NaN, an infinity
// or a |u| beyond 2^22 gives bits outside every window.
__device__ __forceinline__ unsigned first_cell(float u, float& s)
{
    const float a = __fadd_rn(u, -((float)HW - 0.5f));
    const float k = __fadd_rn(a, MAGIC);
    s = __fadd_rn(a, -__fadd_rn(k, -MAGIC));
    return __float_as_uint(k);
}

// The even and odd tap polynomials' coefficients side by side.
struct Coeffs {
    f32x2 c[HW][T4];
};

// From the launch parameters into shared memory once per CTA, from there into
// registers by volatile loads: taken from the parameters directly, the pairs
// are put together anew by two moves ahead of every packed FMA (measured: 26
// moves per point).
__device__ __forceinline__ void share_coeffs(const qs_window& win, f32x2* sm)
{
    for (int i = threadIdx.x; i < HW * T4; i += blockDim.x) sm[i] = pack2(win.e[i / T4][i % T4], win.o[i / T4][i % T4]);
}

__device__ __forceinline__ void load_coeffs(const f32x2* sm, Coeffs& k)
{
#pragma unroll
    for (int i = 0; i < HW * T4; ++i) k.c[i / T4][i % T4] = *(volatile const f32x2*)&sm[i];
}

// The taps of qs_taps, rounded as there.
__device__ __forceinline__ void taps_of(const Coeffs& k, float s, float (&tap)[W])
{
    const f32x2 s2 = pack2(s * s, s * s);
#pragma unroll
    for (int j = 0; j < HW; ++j) {
        f32x2 p = k.c[j][T4 - 1];
#pragma unroll
        for (int i = T4 - 2; i >= 0; --i) p = fma2(p, s2, k.c[j][i]);
        const float2 q = unpack2(p);
        tap[j] = fmaf(s, q.y, q.x);
        tap[W - 1 - j] = fmaf(-s, q.y, q.x);
    }
}

// Bins whose points all satisfy |u| <= G/2: l0 in [-G/2 - (m - 1), G/2 - m],
// G of them.  Windows stay inside, so that the slow way sees every other point.
__device__ __forceinline__ int lowest_bin(int G) { return -(G >> 1) - (HW - 1); }

// A number in [0, 2^32) for point or sample i (the finaliser of MurmurHash3).
__device__ __forceinline__ uint32_t point_hash(uint32_t i)
{
    i = (i + 1) * 0x9E3779B9u;
    i = (i ^ (i >> 16)) * 0x85EBCA6Bu;
    i = (i ^ (i >> 13)) * 0xC2B2AE35u;
    return i ^ (i >> 16);
}

// The bins of a sample of the points n0 .. n1 - 1, one at a hashed place of each
// of NSAMPLE equal ranges (evenly spaced ones would see one cluster only of
// points that take turns between clusters, and every other point would go the
// slow way: 3453 against 545 us for 2 x 2e5 points, d = 16, P = 512), into lohi:
// [h][0..31] smallest, [h][32..63] largest of each lane's slice h.  scratch:
// NSAMPLE x D floats (the window itself, not yet in use).  All loads are issued
// before the first is used: the sample costs one trip to memory.  Ends with a
// barrier.
template <int D, int NT, int SL>
__device__ __forceinline__ void sample_bins(const qs_launch& L, const float* __restrict__ x, int g, int64_t n0,
                                            int64_t n1, const Direction<D>* xi, float* scratch, int* lohi)
{
    constexpr int NW = NT / 32, PER = (NSAMPLE + NW - 1) / NW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ns = (int)min(n1 - n0, (int64_t)NSAMPLE);
    const uint32_t gap = n1 - n0 > NSAMPLE ? (uint32_t)((uint64_t)(n1 - n0) / NSAMPLE) : 1u;  // a shift; points < 2^31
    auto at = [&](int i) { return n0 + (int64_t)i * gap + __umulhi(point_hash((uint32_t)i), gap); };
    float us[D > 0 ? 1 : PER];
    if constexpr (D > 0) {
        for (int e = threadIdx.x; e < ns * D; e += blockDim.x) {
            const int i = e / D, j = e % D;
            if (j < L.d) cp_async_small<4>(scratch + e, x + (size_t)at(i) * L.d + j);
            else scratch[e] = 0.0f;
        }
        cp_async_commit();
        cp_async_wait<0>();
    } else {
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int i = warp + k * NW;
            us[k] = i < ns ? __ldcg(&L.U[((size_t)g * L.ldU + at(i)) * 32 + lane]) : 0.0f;
        }
    }
    if (threadIdx.x < 64 * SL) lohi[threadIdx.x] = (threadIdx.x & 32) ? INT_MIN : INT_MAX;
    __syncthreads();
    int lo[SL], hi[SL];
#pragma unroll
    for (int h = 0; h < SL; ++h) {
        lo[h] = INT_MAX;
        hi[h] = INT_MIN;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = warp + k * NW;
        if (i >= ns) break;
        float v[SL];
        if constexpr (D > 0) ring_u<D, SL>(scratch + i * D, xi, lane, v);
        else v[0] = us[k];
#pragma unroll
        for (int h = 0; h < SL; ++h) {
            if (!(fabsf(v[h]) <= L.half_G)) continue;
            float s;
            const int l0 = (int)(first_cell(v[h], s) - (unsigned)MAGIC_BITS);
            lo[h] = min(lo[h], l0);
            hi[h] = max(hi[h], l0);
        }
    }
#pragma unroll
    for (int h = 0; h < SL; ++h) {
        atomicMin(&lohi[64 * h + lane], lo[h]);
        atomicMax(&lohi[64 * h + 32 + lane], hi[h]);
    }
    __syncthreads();
}

// A CTA's range of the `total` units of work, `group` in each slice group: an equal share of them all, or
// (per_group > 0) of one group among per_group CTAs.
__device__ __forceinline__ void cta_range(int64_t total, int64_t group, int per_group, int64_t& b0, int64_t& b1)
{
    if (per_group > 0) {
        const int g = blockIdx.x / per_group, j = blockIdx.x % per_group;
        b0 = g * group + j * group / per_group;
        b1 = g * group + (j + 1) * group / per_group;
    } else {
        b0 = (int64_t)blockIdx.x * total / gridDim.x;
        b1 = (int64_t)(blockIdx.x + 1) * total / gridDim.x;
    }
}

// Sampled bins -> the window: its width (bins, the same for all lanes) and the
// lane's first bin.  The sample's span is widened by half (256 normal
// samples reach 2.8 standard deviations, the window then 4.2).
struct Window {
    int nbt;   // bins covered, all walks together
    int nb;    // bins of one walk
    int walks;
    bool poly; // polynomials per bin, else cells
};

__device__ __forceinline__ int sampled_need(const int* lohi, int G, int lane)
{
    const int lo = lohi[lane], hi = lohi[32 + lane];
    const int span = lo > hi ? 1 : hi - lo + 1;
    return min(G, __reduce_max_sync(0xffffffffu, span + 2 * (span >> 2) + 8));
}

__device__ __forceinline__ int window_base(const int* lohi, int G, int lane, int nbt)
{
    int lo = lohi[lane], hi = lohi[32 + lane];
    if (lo > hi) lo = hi = 0;
    const int l = lowest_bin(G);
    return max(l, min(((lo + hi) >> 1) - (nbt >> 1), l + G - nbt));
}

// cap_poly / cap_cells: bins that fit as polynomials / as cells.
__device__ __forceinline__ Window place_window(int need, int cap_poly, int cap_cells, bool one_walk)
{
    Window v;
    v.poly = need <= cap_poly;
    v.walks = 1;
    v.nbt = need;
    if (!v.poly) {
        // a little less margin rather than another walk
        if (need > cap_cells && (one_walk || need <= cap_cells + (cap_cells >> 2))) v.nbt = cap_cells;
        v.walks = (v.nbt + cap_cells - 1) / cap_cells;
    }
    v.nb = (v.nbt + v.walks - 1) / v.walks;
    return v;
}

// ---------------------------------------------------------------------------
// Weight bound and cleared grids.  out[0] = 2^30 / B, out[1] = its inverse,
// out[2] = max|w| out[0]; B = sum |w| in a fixed order: block partials, then
// the last block adds them in block order.  ws[0 .. 2 blocks): the partials,
// ticket: zero before the first call, left zero.  The grids are cleared here
// because a launch of its own would cost as much as the clearing.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) lane_prep_kernel(const float* __restrict__ w, int64_t N, float* out, float* ws,
                                                         unsigned int* ticket, unsigned int* flag,
                                                         float4* __restrict__ grid4, int64_t n4)
{
    __shared__ float red[64];
    __shared__ bool last;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    float acc = 0.0f, mx = 0.0f;
    bool bad = false;
    if (w) {
        for (int64_t n = tid; n < N; n += 4 * step) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = n + k * step < N ? fabsf(__ldg(&w[n + k * step])) : 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                acc += v[k];
                mx = fmaxf(mx, v[k]);
            }
        }
    }
    for (int64_t i = tid; i < n4; i += step) grid4[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = acc;
        red[32 + (threadIdx.x >> 5)] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        acc = 0.0f;
        mx = 0.0f;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            acc += red[i];
            mx = fmaxf(mx, red[32 + i]);
        }
        ws[2 * blockIdx.x] = acc;
        ws[2 * blockIdx.x + 1] = mx;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (last) {
            __threadfence();
            float B = 0.0f, M = 0.0f;
            for (int i = 0; i < (int)gridDim.x; ++i) {
                B += __ldcg(&ws[2 * i]);
                M = fmaxf(M, __ldcg(&ws[2 * i + 1]));
            }
            if (!w) {
                B = (float)N;
                M = 1.0f;
            }
            float scale = 0.0f, inv = 0.0f;
            if (!isfinite(B)) {
                bad = true;
            } else if (B > 0.0f) {
                scale = 1073741824.0f / B;
                inv = B / 1073741824.0f;
                if (!isfinite(scale)) scale = inv = 0.0f;  // B below 2^-98: all weights negligible
            }
            if (bad) atomicOr(flag, QS_FLAG_NONFINITE);
            out[0] = scale;
            out[1] = inv;
            out[2] = M * scale;
            out[3] = bad ? 1.0f : 0.0f;
            *ticket = 0u;
        }
    }
}

// ---------------------------------------------------------------------------
// Spread.  The (slice group, block of 8 points) pairs are cut into one
// contiguous range per CTA, so every SM gets the same number of points and a
// CTA changes its group (clears, places and adds up a window) once or twice.
// The windows are integers and are added to the grids in global memory by
// integer atomics, so the order in which CTAs finish does not matter.  A
// window holds only the CTA's share of the weights, so its fixed-point scale
// is finer than the grid's by the largest power of two 2^k for which that
// share still fits 2^30; the sum of a cell is rounded to the grid's scale when
// it is added.  With plain cells that matters: every contribution is rounded
// once, and taps below half a unit would always vanish.
// ---------------------------------------------------------------------------
constexpr int MAX_SHIFT = 10;

// q / 2^k to the nearest integer, ties to even.
__device__ __forceinline__ int shift_rn(int q, int k)
{
    return k == 0 ? q : (q + (1 << (k - 1)) - 1 + ((q >> k) & 1)) >> k;
}

// Bits by which the scale of a window may exceed the grid's: sum of |w| over the points, as a share of
// 2^30 / scale.  red: a float per warp.  Ends with a barrier.
__device__ __forceinline__ int finer_bits(const float* __restrict__ w, int64_t n0, int64_t n1, float scale, float* red)
{
    float acc = 0.0f;
    if (w) {
        for (int64_t n = n0 + threadIdx.x; n < n1; n += 4 * blockDim.x) {
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = n + k * blockDim.x < n1 ? fabsf(__ldg(&w[n + k * blockDim.x])) : 0.0f;
            acc += (v[0] + v[1]) + (v[2] + v[3]);
        }
    } else if (threadIdx.x == 0) {
        acc = (float)(n1 - n0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    float share = 0.0f;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) share += red[i];
    share *= scale;
    int k = 0;
    while (k < MAX_SHIFT && share > 0.0f && share * (float)(2 << k) <= 1073741824.0f && scale * (float)(2 << k) < 1e38f) ++k;
    return k;
}

// A point outside its window: validated, W atomics on the grid itself.
__device__ __noinline__ void spread_outside(const qs_launch& L, float u, float ws, int* row)
{
    u = qs_check_u(u, L.half_G, L.flag);
    int l0;
    float tap[W];
    qs_taps<W>(u, L.win, l0, tap);
    const int mask = L.G - 1;
#pragma unroll
    for (int j = 0; j < W; ++j) atomicAdd(&row[(l0 + j) & mask], __float2int_rn(ws * tap[j]));
}

// Dither of point n, in [-1/2, 1/2): the outermost taps fall to 1e-8 of a weight, below half a unit of a window of
// cells, and would always round to zero; of many equal weights the sum would miss them (2e5 sources, d = 3, P = 300,
// G = 2048: 5.4e-7 of it; 5.6e-8 is left).  Added ahead of the rounding it keeps their mean, for one shuffle and two
// additions per point (1 to 1.6 % of sums at d = 16, 30 and 64).  The inner taps stay above 1e-3 of a weight, where the
// remainders are spread evenly.
__device__ __forceinline__ float tap_dither(uint32_t n) { return (float)(int)point_hash(n) * 0x1p-32f; }

// One point into the lane's column `col` of the window; returns its bin.  A
// point outside goes to a bin behind the window (`dump`) that nobody reads, so
// that no branch breaks the interleaving of several points.  FAST: max |w
// scale| < 2^21.  A weight of zero adds nothing: |dither| rounds to zero.
template <bool POLY, bool FAST>
__device__ __forceinline__ unsigned spread_one(float u, float ws, float dither, unsigned first, unsigned nb,
                                               unsigned dump, int* col, const Coeffs& cf)
{
    float s;
    const unsigned rel = first_cell(u, s) - first;
    const unsigned at = rel < nb ? rel : dump;
    if constexpr (POLY) {
        // moments w t^k, t = 2s; 0 and 1 as w (1 + t)/2 and w (1 - t)/2 (equal
        // weights would otherwise all round the same way)
        const float t = 2.0f * s, hw = 0.5f * ws, t2 = t * t, w2 = ws * t2;
        int* c = col + at * (K * 32);
        f32x2 v = fma2(pack2(hw, -hw), pack2(t, t), pack2(hw, hw));
        const f32x2 step = pack2(t2, t2), magic = pack2(MAGIC, MAGIC);
#pragma unroll
        for (int k = 0; k < K; k += 2) {
            if (k == 2) v = pack2(w2, w2 * t);
            else if (k > 2) v = mul2(v, step);
            if constexpr (FAST) {
                const float2 q = unpack2(add2(v, magic));
                atomicAdd(&c[k * 32], __float_as_int(q.x) - MAGIC_BITS);
                atomicAdd(&c[k * 32 + 32], __float_as_int(q.y) - MAGIC_BITS);
            } else {
                const float2 q = unpack2(v);
                atomicAdd(&c[k * 32], __float2int_rn(q.x));
                atomicAdd(&c[k * 32 + 32], __float2int_rn(q.y));
            }
        }
    } else {
        float tap[W];
        taps_of(cf, s, tap);
        int* c = col + at * 32;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const bool edge = j == 0 || j == W - 1;
            const float v = edge ? fmaf(tap[j], ws, dither) : ws * tap[j];
            const int q = !FAST ? __float2int_rn(v)
                                : __float_as_int(edge ? __fadd_rn(v, MAGIC) : fmaf(tap[j], ws, MAGIC)) - MAGIC_BITS;
            atomicAdd(&c[j * 32], q);
        }
    }
    return rel;
}

// The points n0 .. n0 + cnt - 1 into the windows of one walk, `cols` and `wstride` ints apart.
template <int D, int SL, bool POLY, bool FAST>
__device__ __forceinline__ void spread_walk(const qs_launch& L, const float* __restrict__ x,
                                            const float* __restrict__ w, float wscale, float scale, int g, int64_t n0,
                                            int cnt, const Direction<D>* xi, float* ring, int* cols, int wstride,
                                            const Window& v, const int (&base)[SL], int walk, int* Hi, int p,
                                            const f32x2* coef)
{
    constexpr int RS = lane_stride(D), STEP = spread_threads(D) / 32 * SUB;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned first[SL];
#pragma unroll
    for (int h = 0; h < SL; ++h) first[h] = (unsigned)(MAGIC_BITS + base[h] + walk * v.nb);
    const unsigned nb = (unsigned)min(v.nb, v.nbt - walk * v.nb);
    const unsigned dump = POLY ? nb : nb + (W - 1);
    Coeffs cf;
    if (!POLY) load_coeffs(coef, cf);
    const int d = D > 0 ? L.d : 32;
    const int width = D > 0 ? copy_width(x, d) : 4;
    const unsigned inv = 65536u / (unsigned)d + 1u;
    const float* src = D > 0 ? x + (size_t)n0 * d : L.U + ((size_t)g * L.ldU + n0) * 32;
    const float* wsrc = w ? w + n0 : nullptr;
    auto fetch = [&](int b, int buf) {
        if (b < cnt) {
            if constexpr (D > 0) stage_points<D>(ring + buf, src + (size_t)b * d, min(SUB, cnt - b), d, width, inv, lane);
            else stage_rows(ring + buf, src + (size_t)b * 32, lane);
        }
        cp_async_commit();
    };
    auto dither = [&](int b) { return POLY ? 0.0f : tap_dither((uint32_t)(n0 + b + (lane & (SUB - 1)))); };
    auto weight = [&](int b) { return (lane < SUB && b + lane < cnt) ? (wsrc ? __ldg(&wsrc[b + lane]) * wscale : wscale) : 0.0f; };
    fetch(warp * SUB, 0);
    float wn = weight(warp * SUB);
    int buf = 0;
    for (int b = warp * SUB; b < cnt; b += STEP, buf ^= SUB * RS) {
        fetch(b + STEP, buf ^ (SUB * RS));
        const float wk = wn, dk = dither(b);
        wn = weight(b + STEP);
        cp_async_wait<1>();
        __syncwarp();
        const float* r = ring + buf;
        unsigned worst = 0;
#pragma unroll
        for (int i = 0; i < SUB; ++i) {
            float u[SL];
            ring_u<D, SL>(r + i * RS, xi, lane, u);
            const float ws = __shfl_sync(0xffffffffu, wk, i);
            const float di = POLY ? 0.0f : __shfl_sync(0xffffffffu, dk, i);
#pragma unroll
            for (int h = 0; h < SL; ++h)
                worst = max(worst, spread_one<POLY, FAST>(u[h], ws, di, first[h], nb, dump, cols + h * wstride, cf));
        }
        if (worst >= nb && walk == 0) {
            // points past the last have weight 0 and whatever the ring held: not looked at
            for (int i = 0; i < SUB && b + i < cnt; ++i) {
                float u[SL], s;
                ring_u<D, SL>(r + i * RS, xi, lane, u);
#pragma unroll
                for (int h = 0; h < SL; ++h)
                    if (first_cell(u[h], s) - (unsigned)(MAGIC_BITS + base[h]) >= (unsigned)v.nbt)
                        spread_outside(L, u[h], (wsrc ? __ldg(&wsrc[b + i]) : 1.0f) * scale,
                                       Hi + (size_t)min(p + 32 * h, L.P - 1) * L.G);
            }
        }
        __syncwarp();  // this stage is refilled by the next step
    }
    cp_async_wait<0>();
}

// Points per window of plain cells: a weight is then at least 2^16 units (of equal weights), so that all taps
// but the outermost are many units (a single window over 1e6 points would lose those below 4e-4 and with
// them 1.4e-5 of the sum); adding a window up takes about 1 % of the time of 16384 points.
constexpr int CELL_POINTS = 16384;

// Window of plain cells -> grid rows.  A warp takes 32 cells of the 32 slices at a time and transposes them
// by exchanges between lanes, so that its atomics fall on consecutive cells of one slice (one 128-byte
// row of the grid instead of 32 scattered words).
__device__ __forceinline__ void add_cells(const int* win, int cells, int at, int finer, int p0, int P, int G,
                                          int* __restrict__ Hi)
{
    const int lane = threadIdx.x & 31, mask = G - 1;
    for (int c0 = (threadIdx.x >> 5) * 32; c0 < cells; c0 += blockDim.x) {
        int r[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = c0 + i < cells ? win[(c0 + i) * 32 + lane] : 0;
#pragma unroll
        for (int b = 16; b > 0; b >>= 1)
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if ((i & b) == 0) {
                    const bool up = lane & b;
                    const int other = __shfl_xor_sync(0xffffffffu, up ? r[i] : r[i | b], b);
                    if (up) r[i] = other;
                    else r[i | b] = other;
                }
        // r[i]: cell c0 + lane of slice p0 + i
#pragma unroll
        for (int i = 0; i < 32; ++i) {
            const int first = __shfl_sync(0xffffffffu, at, i) + c0 + lane;
            const int q = shift_rn(r[i], finer);
            if (q && p0 + i < P) atomicAdd(&Hi[(size_t)(p0 + i) * G + (first & mask)], q);
        }
    }
}

// Window of moments -> grid row of the lane: cell c = sum_j V_{c-j, j}, V_bj = sum_k a_jk M_bk; each warp
// takes a run of bins and slides the W open cells along.
template <int D>
__device__ __forceinline__ void add_moments(const qs_launch& L, const int* col, int nb, int at, int finer, int* row)
{
    constexpr int NW = spread_threads(D) / 32;
    const int warp = threadIdx.x >> 5, mask = L.G - 1;
    const int r0 = warp * nb / NW, r1 = (warp + 1) * nb / NW;
    if (r0 >= r1) return;
    const float unit = 1.0f / (float)(1 << finer);
    float acc[W];
#pragma unroll
    for (int j = 0; j < W; ++j) acc[j] = 0.0f;
    for (int r = r0; r < r1 + W - 1; ++r) {
        if (r < r1) {
            const int* mk = col + r * (K * 32);
            float mh[K];
            const int m0 = mk[0], m1 = mk[32];
            mh[0] = (float)(m0 + m1);
            mh[1] = (float)(m0 - m1);
#pragma unroll
            for (int k = 2; k < K; ++k) mh[k] = (float)mk[k * 32];
            // mirrored taps share the even and odd parts
#pragma unroll
            for (int j = 0; j < HW; ++j) {
                float e = 0.0f, o = 0.0f;
#pragma unroll
                for (int k = 0; k < K; k += 2) {
                    e = fmaf(L.atab[j * K + k], mh[k], e);
                    o = fmaf(L.atab[j * K + k + 1], mh[k + 1], o);
                }
                acc[j] += e + o;
                acc[W - 1 - j] += e - o;
            }
        }
        const int q = __float2int_rn(acc[0] * unit);
        if (q && row) atomicAdd(&row[(at + r) & mask], q);
#pragma unroll
        for (int j = 0; j + 1 < W; ++j) acc[j] = acc[j + 1];
        acc[W - 1] = 0.0f;
    }
}

// Everything about one CTA's share of a group's points that does not depend on the group.
struct SpreadShare {
    const float* x;
    const float* w;
    int* Hi;
    int* win;
    float* ring;
    float* red;
    const f32x2* coef;
    float scale, wmax;
};

// The points n0 .. n1 - 1 onto SL slices per lane, the first at p.
template <int D, int SL>
__device__ __forceinline__ void spread_slices(const qs_launch& L, const SpreadShare& c, int g, int p, int64_t n0,
                                              int64_t n1, const Direction<D>* xi, const Window& v,
                                              const int (&base)[SL])
{
    const int lane = threadIdx.x & 31;
    int* col = c.win + lane;
    const int64_t most = v.poly ? n1 - n0 : (int64_t)CELL_POINTS;
    for (int64_t m0 = n0; m0 < n1; m0 += most) {
        const int cnt = (int)min(most, n1 - m0);
        const int finer = finer_bits(c.w, m0, m0 + cnt, c.scale, c.red);
        const float ws = c.scale * (float)(1 << finer);
        const bool fast = c.wmax * (float)(1 << finer) < 2097152.0f;
        for (int walk = 0; walk < v.walks; ++walk) {
            const int nb = min(v.nb, v.nbt - walk * v.nb);
            // per slice: the window, and behind it the bin that nobody reads
            const int rows = v.poly ? nb * K : nb + W - 1, stride = (v.poly ? (nb + 1) * K : nb + 2 * W - 1) * 32;
            __syncthreads();
#pragma unroll
            for (int h = 0; h < SL; ++h)
                for (int i = threadIdx.x; i < rows * 8; i += blockDim.x)
                    reinterpret_cast<int4*>(c.win + h * stride)[i] = make_int4(0, 0, 0, 0);
            __syncthreads();
            if (v.poly) {
                if (fast) spread_walk<D, SL, true, true>(L, c.x, c.w, ws, c.scale, g, m0, cnt, xi, c.ring, col, stride, v, base, walk, c.Hi, p, c.coef);
                else spread_walk<D, SL, true, false>(L, c.x, c.w, ws, c.scale, g, m0, cnt, xi, c.ring, col, stride, v, base, walk, c.Hi, p, c.coef);
            } else {
                if (fast) spread_walk<D, SL, false, true>(L, c.x, c.w, ws, c.scale, g, m0, cnt, xi, c.ring, col, stride, v, base, walk, c.Hi, p, c.coef);
                else spread_walk<D, SL, false, false>(L, c.x, c.w, ws, c.scale, g, m0, cnt, xi, c.ring, col, stride, v, base, walk, c.Hi, p, c.coef);
            }
            __syncthreads();
#pragma unroll 1
            for (int h = 0; h < SL; ++h) {
                const int at = (SL > 1 && h ? base[SL - 1] : base[0]) + walk * v.nb, ph = p + 32 * h;
                if (v.poly) add_moments<D>(L, col + h * stride, nb, at, finer, ph < L.P ? c.Hi + (size_t)ph * L.G : nullptr);
                else add_cells(c.win + h * stride, nb + W - 1, at, finer, ph - lane, L.P, L.G, c.Hi);
            }
        }
    }
    __syncthreads();
}

template <int D>
__global__ void __launch_bounds__(spread_threads(D), 1)
    lane_spread_kernel(const __grid_constant__ qs_launch L, const float* __restrict__ x, const float* __restrict__ w,
                       int* __restrict__ Hi, int win_bytes, int per_group)
{
    constexpr int SL = lane_slices(D);
    extern __shared__ float4 smem4[];
    __shared__ int lohi[64 * SL];
    __shared__ f32x2 coef[HW * T4];
    __shared__ float red[32];
    share_coeffs(L.win, coef);  // read after the first barrier
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = L.G;
    if (__ldg(&L.wscale[3]) != 0.0f) return;  // non-finite weights: flagged, the grids stay zero
    SpreadShare c;
    c.x = x;
    c.w = w;
    c.Hi = Hi;
    c.win = reinterpret_cast<int*>(smem4);
    c.ring = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(smem4) + win_bytes) + warp * lane_ring_floats(D);
    c.red = red;
    c.coef = coef;
    c.scale = __ldg(&L.wscale[0]);
    c.wmax = __ldg(&L.wscale[2]);
    for (int i = lane; i < lane_ring_floats(D); i += 32) c.ring[i] = 0.0f;

    const int cap_poly = win_bytes / (K * 128) - 1, cap_cells = win_bytes / 128 - (2 * W - 1);
    const int64_t nsb = (L.N + SUB - 1) / SUB;
    int64_t b, b1;
    cta_range(nsb * ((L.P + 32 * SL - 1) / (32 * SL)), nsb, per_group, b, b1);
    while (b < b1) {
        const int g = (int)(b / nsb);
        const int64_t e = min(b1, (int64_t)(g + 1) * nsb);
        const int64_t n0 = (b - (int64_t)g * nsb) * SUB, n1 = min(L.N, (e - (int64_t)g * nsb) * SUB);
        b = e;
        const int p = 32 * SL * g + lane;
        Direction<D> xi[SL];
        share_xi<D, SL>(L, p - lane, xi, reinterpret_cast<float*>(c.win));
        sample_bins<D, spread_threads(D), SL>(L, x, g, 0, L.N, xi, reinterpret_cast<float*>(c.win), lohi);
        int need[SL];
#pragma unroll
        for (int h = 0; h < SL; ++h) need[h] = sampled_need(lohi + 64 * h, G, lane);
        if constexpr (SL == 2) {
            const int most = max(need[0], need[1]);
            const int cap_poly2 = win_bytes / 2 / (K * 128) - 1, cap_cells2 = win_bytes / 2 / 128 - (2 * W - 1);
            if (p - lane + 32 < L.P && most <= cap_cells2) {
                const Window v = place_window(most, cap_poly2, cap_cells2, false);
                const int base[2] = {window_base(lohi, G, lane, v.nbt), window_base(lohi + 64, G, lane, v.nbt)};
                spread_slices<D, 2>(L, c, g, p, n0, n1, xi, v, base);
                continue;
            }
        }
#pragma unroll 1
        for (int h = 0; h < SL && p - lane + 32 * h < L.P; ++h) {
            if (h) share_xi<D, 1>(L, p - lane + 32 * h, xi, reinterpret_cast<float*>(c.win));
            const Window v = place_window(h ? need[SL - 1] : need[0], cap_poly, cap_cells, false);
            const int base[1] = {window_base(lohi + 64 * h, G, lane, v.nbt)};
            spread_slices<D, 1>(L, c, g, p + 32 * h, n0, n1, xi, v, base);
        }
    }
}

// ---------------------------------------------------------------------------
// Filter: one CTA per slice, integer grid -> real FFT -> c_k / psi^2 ->
// inverse, in place.  MODE 0: plain into Hi.  1: derivative into Hi.  2: plain
// into Hi and derivative into H2.
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(256) lane_filter_kernel(const __grid_constant__ qs_launch L, float* __restrict__ Hi,
                                                          const float* __restrict__ Dd, float* __restrict__ H2)
{
    extern __shared__ float4 smem4[];
    float2* z = reinterpret_cast<float2*>(smem4);
    const int G = L.G, Gh = G >> 1, log2n = 31 - __clz(Gh);
    float2* z2 = z + Gh;
    const float inv = __ldg(&L.wscale[1]);
    float* row = Hi + (size_t)blockIdx.x * G;
    const int2* src = reinterpret_cast<const int2*>(row);
    for (int i = threadIdx.x; i < Gh; i += blockDim.x) {
        const int2 v = src[i];
        z[fft_sw(i)] = make_float2((float)v.x * inv, (float)v.y * inv);
    }
    __syncthreads();
    fft_inplace<false>(z, Gh, log2n, L.tw, G);
    if (MODE == 2) {
        real_filter<true>(z, z2, Gh, log2n, Dd, L.tw);
        __syncthreads();
    }
    if (MODE == 1) real_filter<true>(z, z, Gh, log2n, Dd, L.tw);
    else real_filter<false>(z, z, Gh, log2n, L.D, L.tw);
    __syncthreads();
    fft_inplace<true>(z, Gh, log2n, L.tw, G);
    fft_store(reinterpret_cast<const float*>(z), row, G, 0);
    if (MODE == 2) {
        fft_inplace<true>(z2, Gh, log2n, L.tw, G);
        fft_store(reinterpret_cast<const float*>(z2), H2 + (size_t)blockIdx.x * G, G, 0);
    }
}

// ---------------------------------------------------------------------------
// Interpolation.  The (slice group, block of 32 targets) pairs are cut into one
// contiguous range per CTA like the spread's: a CTA stages the windows of the
// filtered rows once or twice, and every SM gets the same number of targets.
// (A grid of target chunks x group ranges left 39 % of the SM time idle at
// 2e4 targets and 32 groups, and staged a window per group and chunk.)  The 32
// values of a target are added across the lanes as the targets go by -- pairs
// of targets over lane bit 0, pairs of pairs over bit 1, and so on, one to two
// shuffles per target in all -- after which lane l holds the group's sum of target
// l of the block.  Every addition is a TwoSum, its error goes along (2.5 to 5 % of
// a sum's time against plain additions; two sums side by side in packed
// arithmetic: 1 % less at d = 64 and 784, 2 % more at d = 30, not kept): hi to
// part[g][m] and lo to part[S + g][m] (without room for low parts, P > 2048 slices,
// hi + lo to part[g][m]); the reduction accumulates the groups the same way.
// ---------------------------------------------------------------------------
struct Sum {
    float hi, lo;  // the rounding errors of all additions so far in lo
};

__device__ __forceinline__ void add(Sum& a, Sum b)
{
    qs_two_sum(a.hi, a.lo, b.hi);
    a.lo += b.lo;
}

// LOW: the values have low parts.
template <int B, bool LOW = true>
__device__ __forceinline__ Sum fold(Sum a, Sum b, int lane)
{
    const bool up = (lane >> B) & 1;
    Sum keep = {up ? b.hi : a.hi, LOW ? (up ? b.lo : a.lo) : 0.0f}, other = {up ? a.hi : b.hi, 0.0f};
    other.hi = __shfl_xor_sync(0xffffffffu, other.hi, 1 << B);
    if (LOW) other.lo = __shfl_xor_sync(0xffffffffu, up ? a.lo : b.lo, 1 << B);
    add(keep, other);
    return keep;
}

// A target outside its window: validated, W taps from the row in global memory.
__device__ __noinline__ float interp_outside(const qs_launch& L, float u, const float* __restrict__ row)
{
    u = qs_check_u(u, L.half_G, L.flag);
    int l0;
    float tap[W];
    qs_taps<W>(u, L.win, l0, tap);
    const int mask = L.G - 1;
    float t = 0.0f;
#pragma unroll
    for (int j = 0; j < W; ++j) t = fmaf(__ldg(&row[(l0 + j) & mask]), tap[j], t);
    return t;
}

// Value at one target; outside its window (rel >= nb) the zeros behind it are read.
template <bool POLY>
__device__ __forceinline__ float interp_one(float u, unsigned first, unsigned nb, unsigned dump, const float* col,
                                            const Coeffs& cf, unsigned& rel)
{
    float s;
    rel = first_cell(u, s) - first;
    const unsigned at = rel < nb ? rel : dump;
    float v;
    if constexpr (POLY) {
        const float t = 2.0f * s;
        const float* c = col + at * (K * 32);
        v = c[(K - 1) * 32];
#pragma unroll
        for (int k = K - 2; k >= 0; --k) v = fmaf(v, t, c[k * 32]);
    } else {
        float tap[W];
        taps_of(cf, s, tap);
        const float* c = col + at * 32;
        v = 0.0f;
#pragma unroll
        for (int j = 0; j < W; ++j) v = fmaf(c[j * 32], tap[j], v);
    }
    return v;
}

// The targets m0 .. m0 + cnt - 1 against the windows of one walk: blocks of 32
// targets per warp, in steps of SUB.
template <int D, int SL, int OUT, bool POLY>
__device__ __forceinline__ void interp_walk(const qs_launch& L, const float* __restrict__ y, int g, int64_t m0,
                                            int cnt, const Direction<D>* xi, float* ring, const float* cols,
                                            int wstride, const Window& v, const int (&base)[SL], int walk,
                                            const float* H, int p, bool more, const f32x2* coef)
{
    constexpr int RS = lane_stride(D), NW = interp_threads(D) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned first[SL];
#pragma unroll
    for (int h = 0; h < SL; ++h) first[h] = (unsigned)(MAGIC_BITS + base[h] + walk * v.nb);
    const unsigned nb = (unsigned)min(v.nb, v.nbt - walk * v.nb);
    const unsigned dump = POLY ? nb : nb + (W - 1);
    Coeffs cf;
    if (!POLY) load_coeffs(coef, cf);
    const int d = D > 0 ? L.d : 32;
    const int width = D > 0 ? copy_width(y, d) : 4;
    const unsigned inv = 65536u / (unsigned)d + 1u;
    float* U = L.U + ((size_t)g * L.ldU + m0) * 32;
    const float* src = D > 0 ? y + (size_t)m0 * d : U;
    auto fetch = [&](int b, int buf) {
        if (b < cnt) {
            if constexpr (D > 0) stage_points<D>(ring + buf, src + (size_t)b * d, min(SUB, cnt - b), d, width, inv, lane);
            else stage_rows(ring + buf, src + (size_t)b * 32, lane);
        }
        cp_async_commit();
    };
    // OUT = 1, a value for the back-projection.  Unfused FP32: U[p][m].  Tensor-core forms: as three BF16
    // parts, high and middle in place of the projection (64 bytes each of the 128 of target m's 32
    // slices), low in Qlo, K-major operands of the back-projection GEMM.
    auto put = [&](int h, int m, float q, bool ok) {
        if (!ok || m >= cnt) return;
        if constexpr (D > 0) {
            if (p + 32 * h < L.P) L.U[(size_t)(p + 32 * h) * L.ldU + m0 + m] = q;
        } else {
            __nv_bfloat16* hm = reinterpret_cast<__nv_bfloat16*>(U + (size_t)m * 32);
            const __nv_bfloat16 hi = __float2bfloat16_rn(q);
            const float q1 = q - __bfloat162float(hi);
            const __nv_bfloat16 md = __float2bfloat16_rn(q1);
            hm[lane] = hi;
            hm[32 + lane] = md;
            reinterpret_cast<__nv_bfloat16*>(L.Qlo)[((size_t)g * L.ldU + m0 + m) * 32 + lane] =
                __float2bfloat16_rn(q1 - __bfloat162float(md));
        }
    };
    float* part = L.part + (size_t)g * L.M + m0;
    float* part_lo = L.no_low ? nullptr : part + (size_t)L.S * L.M;
    fetch(warp * 32, 0);
    Sum f3 = {0.0f, 0.0f}, f4 = f3, far = f3;
    int buf = 0;
    for (int b = warp * 32; b < ((cnt + 31) & ~31); buf ^= SUB * RS) {
        const int next = (b & 24) == 24 ? b - 24 + NW * 32 : b + SUB;
        fetch(next, buf ^ (SUB * RS));
        cp_async_wait<1>();
        __syncwarp();
        const float* r = ring + buf;
        Sum f[2];
        float all[OUT == 1 && D > 0 ? SL : 1][OUT == 1 && D > 0 ? SUB : 1];
        unsigned worst = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            Sum val[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = 4 * q + i;
                float u[SL];
                ring_u<D, SL>(r + j * RS, xi, lane, u);
#pragma unroll
                for (int h = 0; h < SL; ++h) {
                    unsigned rel;
                    const float t = interp_one<POLY>(u[h], first[h], nb, dump, cols + h * wstride, cf, rel);
                    worst = max(worst, rel);
                    if (h) add(val[i], Sum{t, 0.0f});
                    else val[i] = {t, 0.0f};
                    if constexpr (OUT == 1 && D > 0) all[h][j] = t;
                    else if (OUT == 1) put(h, b + j, t, rel < nb);
                }
            }
            if (OUT == 0) f[q] = fold<1>(fold<0, SL != 1>(val[0], val[1], lane), fold<0, SL != 1>(val[2], val[3], lane), lane);
        }
        if constexpr (OUT == 1 && D > 0) {
            // eight consecutive values of the lane's slice: one 32-byte sector (U's rows are padded to 128)
            if (worst < nb) {
#pragma unroll
                for (int h = 0; h < SL; ++h)
                    if (p + 32 * h < L.P) {
                        float4* o = reinterpret_cast<float4*>(L.U + (size_t)(p + 32 * h) * L.ldU + m0 + b);
                        o[0] = make_float4(all[h][0], all[h][1], all[h][2], all[h][3]);
                        o[1] = make_float4(all[h][4], all[h][5], all[h][6], all[h][7]);
                    }
            } else {
#pragma unroll
                for (int i = 0; i < SUB; ++i) {
                    float u[SL], s;
                    ring_u<D, SL>(r + i * RS, xi, lane, u);
#pragma unroll
                    for (int h = 0; h < SL; ++h) put(h, b + i, all[h][i], first_cell(u[h], s) - first[h] < nb);
                }
            }
        }
        if (walk == 0 && __any_sync(0xffffffffu, worst >= nb)) {
            for (int i = 0; i < SUB && b + i < cnt; ++i) {
                float u[SL], s;
                Sum t = {0.0f, 0.0f};
                ring_u<D, SL>(r + i * RS, xi, lane, u);
#pragma unroll
                for (int h = 0; h < SL; ++h)
                    if (first_cell(u[h], s) - (unsigned)(MAGIC_BITS + base[h]) >= (unsigned)v.nbt) {
                        const int ph = p + 32 * h;
                        const float q = interp_outside(L, u[h], H + (size_t)min(ph, L.P - 1) * L.G);
                        if (OUT == 1) put(h, b + i, q, true);
                        add(t, Sum{q, 0.0f});
                    }
                if (OUT == 0) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        add(t, Sum{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
                    if (lane == ((b + i) & 31)) far = t;
                }
            }
            __syncwarp();
        }
        if constexpr (OUT == 0) {
            Sum t = fold<2>(f[0], f[1], lane);
            if ((b & 8) == 0) {
                f3 = t;
            } else {
                t = fold<3>(f3, t, lane);
                if ((b & 16) == 0) {
                    f4 = t;
                } else {
                    t = fold<4>(f4, t, lane);
                    add(t, far);
                    far = {0.0f, 0.0f};
                    const int at = (b & ~31) + lane;
                    if (at < cnt) {
                        // `more`: the group's other slices, or another walk's targets, came before
                        if (more) add(t, Sum{part[at], part_lo ? part_lo[at] : 0.0f});
                        part[at] = part_lo ? t.hi : t.hi + t.lo;
                        if (part_lo) part_lo[at] = t.lo;
                    }
                }
            }
        }
        __syncwarp();  // this stage is refilled by the next step
        b = next;
    }
    cp_async_wait<0>();
}

// Bins that fit into `bytes` as polynomials (with the cells that they are formed from: n + W - 1, up to 3
// of alignment, and the zeros that points outside read) and as cells.
__device__ __forceinline__ int interp_cap_poly(int bytes) { return (bytes / 128 - (K + W)) / (K + 1); }
__device__ __forceinline__ int interp_cap_cells(int bytes) { return bytes / 128 - 2 * W; }

// The window of walk `walk` of the lane's row into win (`stride` rows of 32 in all); a barrier is the caller's.
template <int NT>
__device__ __forceinline__ void stage_cells(const qs_launch& L, const float* row, bool live, int b0, int nb, bool poly,
                                            float* win)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, mask = L.G - 1;
    constexpr int nw = NT / 32;
    // the cells b0 & ~3 .. of each lane's row, four at a time (rows are 16-byte aligned, G a multiple of 4)
    const int a0 = b0 & ~3, off = b0 - a0;
    const int n4 = (nb + W - 1 + 3 + 3) >> 2;
    // behind the window: the zeros that points outside read
    float* cells = poly ? win + (nb + 1) * K * 32 : win;
    float* zeros = win + (poly ? nb * K : nb + W - 1) * 32;
    for (int c0 = warp; c0 < n4; c0 += 4 * nw) {
        float4 t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = c0 + k * nw;
            t[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (c < n4 && live) t[k] = __ldcg(reinterpret_cast<const float4*>(row + ((a0 + 4 * c) & mask)));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // lanes with another alignment shift their cells; those before the first or after
            // the last bin's are dropped
            const float e[4] = {t[k].x, t[k].y, t[k].z, t[k].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 4 * (c0 + k * nw) + i - off;
                if (r >= 0 && r < nb + W - 1) cells[r * 32 + lane] = e[i];
            }
        }
    }
    for (int i = threadIdx.x; i < K * 32; i += blockDim.x) zeros[i] = 0.0f;
}

// The bins' polynomials from the staged cells.
template <int NT>
__device__ __forceinline__ void form_polynomials(const qs_launch& L, int nb, float* win)
{
    const int lane = threadIdx.x & 31;
    const float* cells = win + (nb + 1) * K * 32;
    for (int b = threadIdx.x >> 5; b < nb; b += NT / 32) {
        float r[W];
#pragma unroll
        for (int j = 0; j < W; ++j) r[j] = cells[(b + j) * 32 + lane];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            float q = 0.0f;
#pragma unroll
            for (int j = 0; j < W; ++j) q = fmaf(L.atab[j * K + k], r[j], q);
            win[(b * K + k) * 32 + lane] = q;
        }
    }
}

// The CTA's targets against SL slices per lane, the first at p.
template <int D, int SL, int OUT>
__device__ __forceinline__ void interp_slices(const qs_launch& L, const float* __restrict__ y, const float* H, int g,
                                              int p, int64_t m0, int64_t m1, const Direction<D>* xi, const Window& v,
                                              const int (&base)[SL], float* win, float* ring, bool more,
                                              const f32x2* coef)
{
    constexpr int NT = interp_threads(D);
    const int lane = threadIdx.x & 31;
    for (int walk = 0; walk < v.walks; ++walk) {
        const int nb = min(v.nb, v.nbt - walk * v.nb);
        const int stride = (v.poly ? (nb + 1) * K + nb + W - 1 : nb + 2 * W) * 32;
        __syncthreads();
#pragma unroll
        for (int h = 0; h < SL; ++h)
            stage_cells<NT>(L, H + (size_t)min(p + 32 * h, L.P - 1) * L.G, p + 32 * h < L.P, base[h] + walk * v.nb, nb,
                            v.poly, win + h * stride);
        __syncthreads();
        if (v.poly) {
#pragma unroll 1
            for (int h = 0; h < SL; ++h) form_polynomials<NT>(L, nb, win + h * stride);
            __syncthreads();
            interp_walk<D, SL, OUT, true>(L, y, g, m0, (int)(m1 - m0), xi, ring, win + lane, stride, v, base, walk, H, p, more || walk > 0, coef);
        } else {
            interp_walk<D, SL, OUT, false>(L, y, g, m0, (int)(m1 - m0), xi, ring, win + lane, stride, v, base, walk, H, p, more || walk > 0, coef);
        }
    }
    __syncthreads();  // the window is done with
}

template <int D, int OUT>
__global__ void __launch_bounds__(interp_threads(D), 1)
    lane_interp_kernel(const __grid_constant__ qs_launch L, const float* __restrict__ y, const float* __restrict__ H,
                       int win_bytes, int per_group)
{
    constexpr int SL = lane_slices(D);
    extern __shared__ float4 smem4[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(smem4);
    float* win = reinterpret_cast<float*>(smem4);
    __shared__ int lohi[64 * SL];
    __shared__ f32x2 coef[HW * T4];
    share_coeffs(L.win, coef);  // read after the first barrier
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* ring = reinterpret_cast<float*>(sm + win_bytes) + warp * lane_ring_floats(D);
    for (int i = lane; i < lane_ring_floats(D); i += 32) ring[i] = 0.0f;
    const int G = L.G;
    const int cap_poly = interp_cap_poly(win_bytes), cap_cells = interp_cap_cells(win_bytes);
    const int64_t nblk = (L.M + 31) / 32;
    int64_t b, b1;
    cta_range(nblk * ((L.P + 32 * SL - 1) / (32 * SL)), nblk, per_group, b, b1);
    while (b < b1) {
        const int g = (int)(b / nblk);
        const int64_t e = min(b1, (int64_t)(g + 1) * nblk);
        const int64_t m0 = (b - (int64_t)g * nblk) * 32, m1 = min(L.M, (e - (int64_t)g * nblk) * 32);
        b = e;
        const int p = 32 * SL * g + lane;
        Direction<D> xi[SL];
        share_xi<D, SL>(L, p - lane, xi, win);
        sample_bins<D, interp_threads(D), SL>(L, y, g, m0, m1, xi, win, lohi);
        int need[SL];
#pragma unroll
        for (int h = 0; h < SL; ++h) need[h] = sampled_need(lohi + 64 * h, G, lane);
        if constexpr (SL == 2) {
            const int most = max(need[0], need[1]);
            const int cap_poly2 = interp_cap_poly(win_bytes / 2), cap_cells2 = interp_cap_cells(win_bytes / 2);
            if (p - lane + 32 < L.P && most <= cap_cells2) {
                const Window v = place_window(most, cap_poly2, cap_cells2, false);
                const int base[2] = {window_base(lohi, G, lane, v.nbt), window_base(lohi + 64, G, lane, v.nbt)};
                interp_slices<D, 2, OUT>(L, y, H, g, p, m0, m1, xi, v, base, win, ring, false, coef);
                continue;
            }
        }
#pragma unroll 1
        for (int h = 0; h < SL && p - lane + 32 * h < L.P; ++h) {
            if (h) share_xi<D, 1>(L, p - lane + 32 * h, xi, win);
            // values written over their own projections allow one walk only
            const Window v = place_window(h ? need[SL - 1] : need[0], cap_poly, cap_cells, OUT == 1 && D == 0);
            const int base[1] = {window_base(lohi + 64 * h, G, lane, v.nbt)};
            interp_slices<D, 1, OUT>(L, y, H, g, p + 32 * h, m0, m1, xi, v, base, win, ring, h > 0, coef);
        }
    }
}

// Dynamic shared memory of a CTA: whole KB of the 227 that the kernels' static arrays leave (sampled bins of
// two slices per lane, coefficients, a float per warp).
constexpr int LANE_SMEM = 226 * 1024;
static_assert(LANE_SMEM + 64 * 2 * 4 + HW * T4 * 8 + 32 * 4 <= 227 * 1024, "static and dynamic shared memory of a CTA");

// How the work is cut: `group` units in each of `groups` slice groups, at least `least` per CTA; `visit` units
// cost as much as placing, clearing and adding up a window.  A range of equal shares crosses into a second
// group in some CTAs, which then set the time; whole CTAs per group leave some SMs out.
struct Cut {
    int ctas, per_group;
};

Cut cut_work(int64_t group, int64_t groups, int64_t least, double visit)
{
    const int64_t total = group * groups;
    int64_t n = (total + least - 1) / least;
    if (n > QS_LANE_CTAS) n = QS_LANE_CTAS;
    const int64_t k = n / groups;
    if (k < 1) return {(int)n, 0};
    const double equal = (double)total / n + (n % groups ? 2.0 : 1.0) * visit;
    const double whole = (double)((group + k - 1) / k) + visit;
    return whole < equal ? Cut{(int)(k * groups), (int)k} : Cut{(int)n, 0};
}

template <int D>
cudaError_t launch_spread_d(const qs_launch& L, const float* x, const float* w, int* Hi, cudaStream_t st)
{
    const int win = (LANE_SMEM - lane_ring_bytes(D, spread_threads(D))) & ~1023;
    cudaError_t e = cudaFuncSetAttribute(lane_spread_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, LANE_SMEM);
    if (e != cudaSuccess) return e;
    // at least 32 blocks of 8 points per CTA: fewer would not pay for its window, which costs about 100
    const Cut c = cut_work((L.N + SUB - 1) / SUB, (L.P + 32 * lane_slices(D) - 1) / (32 * lane_slices(D)), 32, 100.0);
    lane_spread_kernel<D><<<(unsigned)c.ctas, spread_threads(D), LANE_SMEM, st>>>(L, x, w, Hi, win, c.per_group);
    return cudaGetLastError();
}

template <int D, int OUT>
cudaError_t launch_interp_d(const qs_launch& L, const float* y, const float* H, cudaStream_t st)
{
    const int win = (LANE_SMEM - lane_ring_bytes(D, interp_threads(D))) & ~1023;
    cudaError_t e =
        cudaFuncSetAttribute(lane_interp_kernel<D, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, LANE_SMEM);
    if (e != cudaSuccess) return e;
    // at least 8 blocks of 32 targets per CTA, a window costs about 12
    const Cut c = cut_work((L.M + 31) / 32, (L.P + 32 * lane_slices(D) - 1) / (32 * lane_slices(D)), 8, 12.0);
    lane_interp_kernel<D, OUT><<<(unsigned)c.ctas, interp_threads(D), LANE_SMEM, st>>>(L, y, H, win, c.per_group);
    return cudaGetLastError();
}

}  // namespace

// Coordinates per lane of the FP32 forms' kernels, 0 for the projections in U.
static int lane_dims(int d, bool from_u)
{
    if (from_u) return 0;
    const int dims[] = {4, 8, 16, 32, 48, 64};
    for (int D : dims)
        if (d <= D) return D;
    return -1;
}

cudaError_t qs_launch_lane_prep(const qs_launch& L, const float* w, float* grid, cudaStream_t st)
{
    // wscale: 4 values, then the block partials and the ticket (QS_WSCALE_FLOATS in all)
    float* ws = L.wscale + 4;
    unsigned int* ticket = reinterpret_cast<unsigned int*>(ws + 2 * QS_PREP_BLOCKS);
    const int64_t n4 = (int64_t)L.P * L.G / 4, per = 1024 * 4;
    int64_t blocks = ((w ? L.N : 0) + per - 1) / per, zb = (n4 + per - 1) / per;
    if (zb > blocks) blocks = zb;
    if (blocks > QS_PREP_BLOCKS) blocks = QS_PREP_BLOCKS;
    if (blocks < 1) blocks = 1;
    lane_prep_kernel<<<(unsigned)blocks, 1024, 0, st>>>(w, L.N, L.wscale, ws, ticket, L.flag,
                                                        reinterpret_cast<float4*>(grid), n4);
    return cudaGetLastError();
}

cudaError_t qs_launch_lane_spread(const qs_launch& L, const float* x, const float* w, bool from_u, float* grid,
                                  cudaStream_t st)
{
    int* Hi = reinterpret_cast<int*>(grid);
    switch (lane_dims(L.d, from_u)) {
        case 0: return launch_spread_d<0>(L, x, w, Hi, st);
        case 4: return launch_spread_d<4>(L, x, w, Hi, st);
        case 8: return launch_spread_d<8>(L, x, w, Hi, st);
        case 16: return launch_spread_d<16>(L, x, w, Hi, st);
        case 32: return launch_spread_d<32>(L, x, w, Hi, st);
        case 48: return launch_spread_d<48>(L, x, w, Hi, st);
        case 64: return launch_spread_d<64>(L, x, w, Hi, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t qs_launch_lane_filter(const qs_launch& L, int mode, float* grid, const float* Dd, float* H2,
                                  cudaStream_t st)
{
    const size_t smem = (size_t)L.G * 4 * (mode == 2 ? 2 : 1);
    const int nt = L.G / 16 < 32 ? 32 : (L.G / 16 > 256 ? 256 : L.G / 16);  // a radix-8 butterfly per thread
    auto kern = mode == 0 ? lane_filter_kernel<0> : (mode == 1 ? lane_filter_kernel<1> : lane_filter_kernel<2>);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<L.P, nt, smem, st>>>(L, grid, Dd, H2);
    return cudaGetLastError();
}

cudaError_t qs_launch_lane_interp(const qs_launch& L, const float* y, bool from_u, const float* H, bool deriv,
                                  cudaStream_t st)
{
#define QS_LANE_INTERP(DD) (deriv ? launch_interp_d<DD, 1>(L, y, H, st) : launch_interp_d<DD, 0>(L, y, H, st))
    switch (lane_dims(L.d, from_u)) {
        case 0: return QS_LANE_INTERP(0);
        case 4: return QS_LANE_INTERP(4);
        case 8: return QS_LANE_INTERP(8);
        case 16: return QS_LANE_INTERP(16);
        case 32: return QS_LANE_INTERP(32);
        case 48: return QS_LANE_INTERP(48);
        case 64: return QS_LANE_INTERP(64);
        default: return cudaErrorInvalidValue;
    }
#undef QS_LANE_INTERP
}

// Slice groups of the interpolation, a partial sum of each target for each.
int qs_lane_groups(int P, int d, bool from_u)
{
    const int D = lane_dims(d, from_u), slices = 32 * (D < 0 ? 1 : lane_slices(D));
    return (P + slices - 1) / slices;
}
