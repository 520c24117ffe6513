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
__host__ __device__ constexpr int spread_threads(int D) { return D == 0 ? 768 : (D <= 32 ? 512 : 384); }
__host__ __device__ constexpr int interp_threads(int D) { return D <= 32 ? 512 : 384; }
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

template <int D>
__device__ __forceinline__ void load_xi(const qs_launch& L, int p, Direction<D>& xi)
{
    const float* src = L.xi_s + (size_t)p * L.d;
    auto at = [&](int j) { return (p < L.P && j < L.d) ? __ldg(&src[j]) : 0.0f; };
#pragma unroll
    for (int j = 0; j < D; j += 2) xi.c[j / 2] = pack2(at(j), at(j + 1));
}

// Grid coordinate of the staged point at r on the lane's slice: FP32 products summed in four strands
// (coordinates mod 4), added at the end.
template <int D>
__device__ __forceinline__ float ring_u(const float* r, const Direction<D>& xi, int lane)
{
    if constexpr (D > 0) {
        f32x2 a = 0, b = 0;
#pragma unroll
        for (int j = 0; j < D; j += 4) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(r + j);
            a = j == 0 ? mul2(xi.c[0], v.x) : fma2(xi.c[j / 2], v.x, a);
            b = j == 0 ? mul2(xi.c[1], v.y) : fma2(xi.c[j / 2 + 1], v.y, b);
        }
        const float2 t = unpack2(add2(a, b));
        return t.x + t.y;
    } else {
        return r[lane];
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

// The bins of a sample of the points n0 .. n1 - 1, spaced evenly, into lohi:
// [0..31] smallest, [32..63] largest of each lane.  scratch: NSAMPLE x D
// floats (the window itself, not yet in use).  All loads are issued before
// the first is used: the sample costs one trip to memory.  Ends with a barrier.
template <int D, int NT>
__device__ __forceinline__ void sample_bins(const qs_launch& L, const float* __restrict__ x, int g, int64_t n0,
                                            int64_t n1, const Direction<D>& xi, float* scratch, int* lohi)
{
    constexpr int NW = NT / 32, PER = (NSAMPLE + NW - 1) / NW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ns = (int)min(n1 - n0, (int64_t)NSAMPLE);
    const int64_t gap = n1 - n0 > NSAMPLE ? (int64_t)((uint64_t)(n1 - n0) / NSAMPLE) : 1;
    auto at = [&](int i) { return n0 + i * gap; };
    float u[PER];
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
            u[k] = i < ns ? __ldcg(&L.U[((size_t)g * L.ldU + at(i)) * 32 + lane]) : 0.0f;
        }
    }
    if (threadIdx.x < 64) lohi[threadIdx.x] = threadIdx.x < 32 ? INT_MAX : INT_MIN;
    __syncthreads();
    int lo = INT_MAX, hi = INT_MIN;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = warp + k * NW;
        if (i >= ns) break;
        const float v = D > 0 ? ring_u<D>(scratch + i * D, xi, lane) : u[k];
        if (!(fabsf(v) <= L.half_G)) continue;
        float s;
        const int l0 = (int)(first_cell(v, s) - (unsigned)MAGIC_BITS);
        lo = min(lo, l0);
        hi = max(hi, l0);
    }
    atomicMin(&lohi[lane], lo);
    atomicMax(&lohi[32 + lane], hi);
    __syncthreads();
}

// Sampled bins -> the window: its width (bins, the same for all lanes) and the
// lane's first bin.  The sample's span is widened by half (256 normal
// samples reach 2.8 standard deviations, the window then 4.2).
struct Window {
    int nbt;   // bins covered, all walks together
    int nb;    // bins of one walk
    int walks;
    bool poly; // polynomials per bin, else cells
    int base;  // the lane's first bin
};

// cap_poly / cap_cells: bins that fit as polynomials / as cells.
__device__ __forceinline__ Window place_window(const int* lohi, int G, int lane, int cap_poly, int cap_cells,
                                               bool one_walk)
{
    int lo = lohi[lane], hi = lohi[32 + lane];
    if (lo > hi) lo = hi = 0;
    const int span = hi - lo + 1;
    int need = __reduce_max_sync(0xffffffffu, span + 2 * (span >> 2) + 8);
    need = min(need, G);
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
    const int l = lowest_bin(G);
    v.base = max(l, min(((lo + hi) >> 1) - (v.nbt >> 1), l + G - v.nbt));
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
    while (k < MAX_SHIFT && share > 0.0f && share * (float)(2 << k) <= 1073741824.0f) ++k;
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

// One point into the lane's column `col` of the window; returns its bin.  A
// point outside goes to a bin behind the window (`dump`) that nobody reads, so
// that no branch breaks the interleaving of several points.  FAST: max |w
// scale| < 2^21.
template <bool POLY, bool FAST>
__device__ __forceinline__ unsigned spread_one(float u, float ws, unsigned first, unsigned nb,
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
            const int q = FAST ? __float_as_int(fmaf(tap[j], ws, MAGIC)) - MAGIC_BITS : __float2int_rn(ws * tap[j]);
            atomicAdd(&c[j * 32], q);
        }
    }
    return rel;
}

// The points n0 .. n0 + cnt - 1 into the window of one walk.
template <int D, bool POLY, bool FAST>
__device__ __forceinline__ void spread_walk(const qs_launch& L, const float* __restrict__ x,
                                            const float* __restrict__ w, float wscale, float scale, int g, int64_t n0, int cnt,
                                            const Direction<D>& xi, float* ring, int* col, const Window& v, int walk,
                                            int* row, const f32x2* coef)
{
    constexpr int RS = lane_stride(D), STEP = spread_threads(D) / 32 * SUB;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned first0 = (unsigned)(MAGIC_BITS + v.base), first = first0 + (unsigned)(walk * v.nb);
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
    auto weight = [&](int b) { return (lane < SUB && b + lane < cnt) ? (wsrc ? __ldg(&wsrc[b + lane]) * wscale : wscale) : 0.0f; };
    fetch(warp * SUB, 0);
    float wn = weight(warp * SUB);
    int buf = 0;
    for (int b = warp * SUB; b < cnt; b += STEP, buf ^= SUB * RS) {
        fetch(b + STEP, buf ^ (SUB * RS));
        const float wk = wn;
        wn = weight(b + STEP);
        cp_async_wait<1>();
        __syncwarp();
        const float* r = ring + buf;
        unsigned worst = 0;
#pragma unroll
        for (int i = 0; i < SUB; ++i)
            worst = max(worst, spread_one<POLY, FAST>(ring_u<D>(r + i * RS, xi, lane), __shfl_sync(0xffffffffu, wk, i),
                                                      first, nb, dump, col, cf));
        if (worst >= nb && walk == 0) {
            // points past the last have weight 0 and whatever the ring held: not looked at
            for (int i = 0; i < SUB && b + i < cnt; ++i) {
                float s;
                const float u = ring_u<D>(r + i * RS, xi, lane);
                if (first_cell(u, s) - first0 >= (unsigned)v.nbt)
                    spread_outside(L, u, (wsrc ? __ldg(&wsrc[b + i]) : 1.0f) * scale, row);
            }
        }
        __syncwarp();  // this stage is refilled by the next step
    }
    cp_async_wait<0>();
}

// Points per window of plain cells: a weight is then at least 2^16 units (of equal weights), so that the
// taps lost to rounding are below 2^-17 (a single window over 1e6 points loses those below 4e-4 and with
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

template <int D>
__global__ void __launch_bounds__(spread_threads(D), 1)
    lane_spread_kernel(const __grid_constant__ qs_launch L, const float* __restrict__ x, const float* __restrict__ w,
                       int* __restrict__ Hi, int win_bytes)
{
    extern __shared__ float4 smem4[];
    int* win = reinterpret_cast<int*>(smem4);
    __shared__ int lohi[64];
    __shared__ f32x2 coef[HW * T4];
    share_coeffs(L.win, coef);  // read after the first barrier
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int G = L.G;
    if (__ldg(&L.wscale[3]) != 0.0f) return;  // non-finite weights: flagged, the grids stay zero
    const float scale = __ldg(&L.wscale[0]);
    const float wmax = __ldg(&L.wscale[2]);
    __shared__ float red[32];
    float* ring = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(smem4) + win_bytes) +
                  warp * lane_ring_floats(D);
    for (int i = lane; i < lane_ring_floats(D); i += 32) ring[i] = 0.0f;

    const int64_t nsb = (L.N + SUB - 1) / SUB;
    const int64_t total = nsb * ((L.P + 31) / 32);
    const int64_t b0 = (int64_t)blockIdx.x * total / gridDim.x, b1 = (int64_t)(blockIdx.x + 1) * total / gridDim.x;
    for (int64_t b = b0; b < b1;) {
        const int g = (int)(b / nsb);
        const int64_t e = min(b1, (int64_t)(g + 1) * nsb);
        const int64_t n0 = (b - (int64_t)g * nsb) * SUB, n1 = min(L.N, (e - (int64_t)g * nsb) * SUB);
        b = e;
        const int p = 32 * g + lane;
        Direction<D> xi;
        load_xi<D>(L, p, xi);
        sample_bins<D, spread_threads(D)>(L, x, g, 0, L.N, xi, reinterpret_cast<float*>(win), lohi);
        const Window v = place_window(lohi, G, lane, win_bytes / (K * 128) - 1, win_bytes / 128 - (2 * W - 1), false);
        int* col = win + lane;
        int* row = Hi + (size_t)min(p, L.P - 1) * G;
        const int64_t most = v.poly ? n1 - n0 : (int64_t)CELL_POINTS;
        for (int64_t c = n0; c < n1; c += most) {
            const int cnt = (int)min(most, n1 - c);
            const int finer = finer_bits(w, c, c + cnt, scale, red);
            const float wscale = scale * (float)(1 << finer);
            const bool fast = wmax * (float)(1 << finer) < 2097152.0f;
            for (int walk = 0; walk < v.walks; ++walk) {
                const int nb = min(v.nb, v.nbt - walk * v.nb);
                const int rows = v.poly ? nb * K : nb + W - 1;
                __syncthreads();
                for (int i = threadIdx.x; i < rows * 8; i += blockDim.x)
                    reinterpret_cast<int4*>(win)[i] = make_int4(0, 0, 0, 0);
                __syncthreads();
                if (v.poly) {
                    if (fast) spread_walk<D, true, true>(L, x, w, wscale, scale, g, c, cnt, xi, ring, col, v, walk, row, coef);
                    else spread_walk<D, true, false>(L, x, w, wscale, scale, g, c, cnt, xi, ring, col, v, walk, row, coef);
                } else {
                    if (fast) spread_walk<D, false, true>(L, x, w, wscale, scale, g, c, cnt, xi, ring, col, v, walk, row, coef);
                    else spread_walk<D, false, false>(L, x, w, wscale, scale, g, c, cnt, xi, ring, col, v, walk, row, coef);
                }
                __syncthreads();
                const int at = v.base + walk * v.nb;
                if (v.poly) add_moments<D>(L, col, nb, at, finer, p < L.P ? row : nullptr);
                else add_cells(win, nb + W - 1, at, finer, 32 * g, L.P, G, Hi);
            }
        }
        __syncthreads();
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
// Interpolation.  CTA (chunk of L.lane_T targets, slice groups [s NG / S,
// (s + 1) NG / S)); per group it stages the windows of the 32 filtered rows
// and its warps walk over the targets, 32 slices at a time.  The 32 values of
// a target are added across the lanes as the targets go by -- pairs of targets
// over lane bit 0, pairs of pairs over bit 1, and so on, one shuffle per
// target in all -- after which lane l holds the group's sum of target l of the
// block; the groups' sums are accumulated by TwoSum in increasing order.
// ---------------------------------------------------------------------------
template <int B>
__device__ __forceinline__ float fold(float a, float b, int lane)
{
    const bool up = (lane >> B) & 1;
    const float keep = up ? b : a, send = up ? a : b;
    return keep + __shfl_xor_sync(0xffffffffu, send, 1 << B);
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

// The targets m0 .. m0 + cnt - 1 against the window of one walk: blocks of 32
// targets per warp, in steps of SUB.
template <int D, int OUT, bool POLY>
__device__ __forceinline__ void interp_walk(const qs_launch& L, const float* __restrict__ y, int g, int64_t m0,
                                            int cnt, const Direction<D>& xi, float* ring, const float* col,
                                            const Window& v, int walk, const float* row, float* acc, const f32x2* coef)
{
    constexpr int RS = lane_stride(D), NW = interp_threads(D) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned first0 = (unsigned)(MAGIC_BITS + v.base), first = first0 + (unsigned)(walk * v.nb);
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
    const int p = 32 * g + lane;
    auto put = [&](int m, float q, bool ok) {
        if (!ok || m >= cnt) return;
        if constexpr (D > 0) {
            if (p < L.P) L.U[(size_t)p * L.ldU + m0 + m] = q;
        } else {
            __nv_bfloat16* hm = reinterpret_cast<__nv_bfloat16*>(U + (size_t)m * 32);
            const __nv_bfloat16 h = __float2bfloat16_rn(q);
            const float q1 = q - __bfloat162float(h);
            const __nv_bfloat16 md = __float2bfloat16_rn(q1);
            hm[lane] = h;
            hm[32 + lane] = md;
            reinterpret_cast<__nv_bfloat16*>(L.Qlo)[((size_t)g * L.ldU + m0 + m) * 32 + lane] =
                __float2bfloat16_rn(q1 - __bfloat162float(md));
        }
    };
    fetch(warp * 32, 0);
    float f3 = 0.0f, f4 = 0.0f;
    int buf = 0;
    for (int b = warp * 32; b < ((cnt + 31) & ~31); buf ^= SUB * RS) {
        const int next = (b & 24) == 24 ? b - 24 + NW * 32 : b + SUB;
        fetch(next, buf ^ (SUB * RS));
        cp_async_wait<1>();
        __syncwarp();
        const float* r = ring + buf;
        float f[2], all[OUT == 1 && D > 0 ? SUB : 1];
        unsigned worst = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float val[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = 4 * h + i;
                unsigned rel;
                val[i] = interp_one<POLY>(ring_u<D>(r + j * RS, xi, lane), first, nb, dump, col, cf, rel);
                worst = max(worst, rel);
                if constexpr (OUT == 1 && D > 0) all[j] = val[i];
                else if (OUT == 1) put(b + j, val[i], rel < nb);
            }
            if (OUT == 0) f[h] = fold<1>(fold<0>(val[0], val[1], lane), fold<0>(val[2], val[3], lane), lane);
        }
        if constexpr (OUT == 1 && D > 0) {
            // eight consecutive values of the lane's slice: one 32-byte sector (U's rows are padded to 128)
            if (worst < nb) {
                if (p < L.P) {
                    float4* o = reinterpret_cast<float4*>(L.U + (size_t)p * L.ldU + m0 + b);
                    o[0] = make_float4(all[0], all[1], all[2], all[3]);
                    o[1] = make_float4(all[4], all[5], all[6], all[7]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < SUB; ++i) {
                    float s;
                    put(b + i, all[i], first_cell(ring_u<D>(r + i * RS, xi, lane), s) - first < nb);
                }
            }
        }
        if (walk == 0 && __any_sync(0xffffffffu, worst >= nb)) {
            for (int i = 0; i < SUB && b + i < cnt; ++i) {
                float s, t = 0.0f;
                const float u = ring_u<D>(r + i * RS, xi, lane);
                if (first_cell(u, s) - first0 >= (unsigned)v.nbt) {
                    t = interp_outside(L, u, row);
                    if (OUT == 1) put(b + i, t, true);
                }
                if (OUT == 0) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                    if (lane == 0) {
                        float hi = acc[b + i], lo = acc[L.lane_T + b + i];
                        qs_two_sum(hi, lo, t);
                        acc[b + i] = hi;
                        acc[L.lane_T + b + i] = lo;
                    }
                }
            }
            __syncwarp();
        }
        if constexpr (OUT == 0) {
            float t = fold<2>(f[0], f[1], lane);
            if ((b & 8) == 0) {
                f3 = t;
            } else {
                t = fold<3>(f3, t, lane);
                if ((b & 16) == 0) {
                    f4 = t;
                } else {
                    t = fold<4>(f4, t, lane);
                    const int at = (b & ~31) + lane;
                    float hi = acc[at], lo = acc[L.lane_T + at];
                    qs_two_sum(hi, lo, t);
                    acc[at] = hi;
                    acc[L.lane_T + at] = lo;
                }
            }
        }
        __syncwarp();  // this stage is refilled by the next step
        b = next;
    }
    cp_async_wait<0>();
}

template <int D, int OUT>
__global__ void __launch_bounds__(interp_threads(D), 1)
    lane_interp_kernel(const __grid_constant__ qs_launch L, const float* __restrict__ y, const float* __restrict__ H,
                       int win_bytes)
{
    extern __shared__ float4 smem4[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(smem4);
    float* win = reinterpret_cast<float*>(smem4);
    float* acc = reinterpret_cast<float*>(sm + win_bytes + lane_ring_bytes(D, interp_threads(D)));
    __shared__ int lohi[64];
    __shared__ f32x2 coef[HW * T4];
    share_coeffs(L.win, coef);  // read after the first barrier
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float* ring = reinterpret_cast<float*>(sm + win_bytes) + warp * lane_ring_floats(D);
    for (int i = lane; i < lane_ring_floats(D); i += 32) ring[i] = 0.0f;
    const int G = L.G, mask = G - 1;
    const int chunk = blockIdx.x / L.S, s = blockIdx.x % L.S;
    const int NG = (L.P + 31) / 32;
    const int g0 = (int)((int64_t)s * NG / L.S), g1 = (int)((int64_t)(s + 1) * NG / L.S);
    const int64_t m0 = L.m_base + (int64_t)chunk * L.lane_T, m1 = min(L.m_end, m0 + L.lane_T);
    if (OUT == 0)
        for (int i = threadIdx.x; i < 2 * L.lane_T; i += blockDim.x) acc[i] = 0.0f;
    for (int g = g0; g < g1; ++g) {
        const int p = 32 * g + lane;
        Direction<D> xi;
        load_xi<D>(L, p, xi);
        __syncthreads();  // the last group's window is done with
        sample_bins<D, interp_threads(D)>(L, y, g, m0, m1, xi, win, lohi);
        // polynomials of n bins also need their n + W - 1 cells (and up to 3 of alignment) while they
        // are formed; values written over their own projections allow one walk only
        const Window v = place_window(lohi, G, lane, (win_bytes / 128 - (K + W)) / (K + 1), win_bytes / 128 - 2 * W,
                                      OUT == 1 && D == 0);
        const float* row = H + (size_t)min(p, L.P - 1) * G;
        for (int walk = 0; walk < v.walks; ++walk) {
            const int nb = min(v.nb, v.nbt - walk * v.nb);
            const int b0 = v.base + walk * v.nb;
            // the cells b0 & ~3 .. of each lane's row, four at a time (rows are 16-byte aligned, G a multiple of 4)
            const int a0 = b0 & ~3, off = b0 - a0;
            const int n4 = (nb + W - 1 + 3 + 3) >> 2;
            // behind the window: the zeros that points outside read
            float* cells = v.poly ? win + (nb + 1) * K * 32 : win;
            float* zeros = win + (v.poly ? nb * K : nb + W - 1) * 32;
            __syncthreads();
            for (int c0 = warp; c0 < n4; c0 += 4 * nw) {
                float4 t[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = c0 + k * nw;
                    t[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (c < n4 && p < L.P) t[k] = __ldcg(reinterpret_cast<const float4*>(row + ((a0 + 4 * c) & mask)));
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
            __syncthreads();
            if (v.poly) {
                for (int b = warp; b < nb; b += nw) {
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
                __syncthreads();
                interp_walk<D, OUT, true>(L, y, g, m0, (int)(m1 - m0), xi, ring, win + lane, v, walk, row, acc, coef);
            } else {
                interp_walk<D, OUT, false>(L, y, g, m0, (int)(m1 - m0), xi, ring, win + lane, v, walk, row, acc, coef);
            }
        }
    }
    if (OUT == 0) {
        __syncthreads();
        for (int64_t m = m0 + threadIdx.x; m < m1; m += blockDim.x) {
            L.part[(size_t)s * L.M + m] = acc[m - m0];
            L.part[(size_t)(L.S + s) * L.M + m] = acc[L.lane_T + (m - m0)];
        }
    }
}

// Dynamic shared memory of a CTA: all that the static 256 bytes leave.
constexpr int LANE_SMEM = 226 * 1024;

template <int D>
cudaError_t launch_spread_d(const qs_launch& L, const float* x, const float* w, int* Hi, cudaStream_t st)
{
    const int win = (LANE_SMEM - lane_ring_bytes(D, spread_threads(D))) & ~1023;
    cudaError_t e = cudaFuncSetAttribute(lane_spread_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, LANE_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t total = (L.N + SUB - 1) / SUB * ((L.P + 31) / 32);
    // at least 32 blocks of 8 points per CTA: fewer would not pay for its window
    int64_t ctas = (total + 31) / 32;
    if (ctas > QS_LANE_CTAS) ctas = QS_LANE_CTAS;
    lane_spread_kernel<D><<<(unsigned)ctas, spread_threads(D), LANE_SMEM, st>>>(L, x, w, Hi, win);
    return cudaGetLastError();
}

template <int D, int OUT>
cudaError_t launch_interp_d(const qs_launch& L, const float* y, const float* H, cudaStream_t st)
{
    const int win = (LANE_SMEM - lane_ring_bytes(D, interp_threads(D)) - (OUT == 0 ? 8 * L.lane_T : 0)) & ~1023;
    cudaError_t e =
        cudaFuncSetAttribute(lane_interp_kernel<D, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, LANE_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t chunks = (L.m_end - L.m_base + L.lane_T - 1) / L.lane_T;
    if (chunks <= 0) return cudaSuccess;
    lane_interp_kernel<D, OUT><<<(unsigned)(chunks * L.S), interp_threads(D), LANE_SMEM, st>>>(L, y, H, win);
    return cudaGetLastError();
}

}  // namespace

// Coordinates per lane of the FP32 forms' kernels, 0 for the projections in U.
static int lane_dims(const qs_launch& L, bool from_u)
{
    if (from_u) return 0;
    const int dims[] = {4, 8, 16, 32, 48, 64};
    for (int D : dims)
        if (L.d <= D) return D;
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
    switch (lane_dims(L, from_u)) {
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
    switch (lane_dims(L, from_u)) {
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

// Targets per CTA and slice groups of the interpolation: the fewest rounds of
// (targets + the cost of staging a window, about 400 targets' worth) over the
// CTAs, from M and P only.
void qs_lane_shape(int64_t M, int P, int S_max, int* T, int* S)
{
    const int NG = (P + 31) / 32;
    double best = 1e300;
    for (int t = 256; t <= 4096; t = t < 1024 ? 2 * t : t + 1024) {
        const int64_t chunks = (M + t - 1) / t;
        for (int s = 1; s <= NG && s <= S_max; ++s) {
            const int64_t rounds = (chunks * s + QS_LANE_CTAS - 1) / QS_LANE_CTAS;
            const double cost = (double)rounds * ((NG + s - 1) / s) * (t + 400.0) + 2.0 * s;
            if (cost < best) {
                best = cost;
                *T = t;
                *S = s;
            }
        }
    }
}
