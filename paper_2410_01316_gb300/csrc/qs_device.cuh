// Device helpers shared by the grid kernels: the shared-memory real FFT and
// filter of a slice grid, and the cp.async staging of filtered rows.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace qsdev {

// ---------------------------------------------------------------------------
// Complex FFT of length n = G/2 in place in shared memory, n a power of two.
// Forward (e^{-2 pi i j / len}): decimation in frequency, natural order in,
// digit-reversed order out; inverse (e^{+...}): the same passes backwards,
// digit-reversed in, natural out, so that no pass reorders anything -- the
// spectrum is only ever touched by real_filter, which goes through
// fft_pos.  Both unnormalised.  tw[t] = e^{-2 pi i t / G}, t < G/2.
//
// The passes are bound by their barriers and shared-memory round trips, not
// by arithmetic, so each takes eight points per thread (radix 8, after one
// radix-2 or radix-4 pass when log2 n is no multiple of 3): ceil(log2 n / 3)
// passes instead of the log2 n of a radix-2 transform and no bit reversal.
// Element i lies at fft_sw(i): the XOR spreads the strides of 8 and 64
// elements of the last passes over the banks without padding.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ int fft_sw(int i) { return i ^ ((i >> 4) & 15); }

// Place of frequency k after the forward transform (before fft_sw).
__device__ __forceinline__ int fft_pos(int k, int log2n)
{
    const int r = log2n % 3;
    int len = (1 << log2n) >> r;
    int pos = (k & ((1 << r) - 1)) * len;
    k >>= r;
    while (len > 1) {
        len >>= 3;
        pos += (k & 7) * len;
        k >>= 3;
    }
    return pos;
}

template <bool INV>
__device__ __forceinline__ float2 fft_rot(float2 a)  // times -i, inverse: +i
{
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

template <bool INV>
__device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d)  // natural order in and out
{
    const float2 s0 = make_float2(a.x + c.x, a.y + c.y), d0 = make_float2(a.x - c.x, a.y - c.y);
    const float2 s1 = make_float2(b.x + d.x, b.y + d.y);
    const float2 d1 = fft_rot<INV>(make_float2(b.x - d.x, b.y - d.y));
    a = make_float2(s0.x + s1.x, s0.y + s1.y);
    b = make_float2(d0.x + d1.x, d0.y + d1.y);
    c = make_float2(s0.x - s1.x, s0.y - s1.y);
    d = make_float2(d0.x - d1.x, d0.y - d1.y);
}

template <bool INV, int R>
__device__ __forceinline__ void dft_r(float2 (&v)[R])
{
    if constexpr (R == 2) {
        const float2 t = make_float2(v[0].x - v[1].x, v[0].y - v[1].y);
        v[0] = make_float2(v[0].x + v[1].x, v[0].y + v[1].y);
        v[1] = t;
    } else if constexpr (R == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else {
        dft4<INV>(v[0], v[2], v[4], v[6]);
        dft4<INV>(v[1], v[3], v[5], v[7]);
        constexpr float h = 0.70710678118654752440f;
        const float2 e[4] = {v[0], v[2], v[4], v[6]};
        float2 o[4] = {v[1], v[3], v[5], v[7]};
        o[1] = INV ? make_float2(h * (o[1].x - o[1].y), h * (o[1].x + o[1].y))
                   : make_float2(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
        o[2] = fft_rot<INV>(o[2]);
        o[3] = INV ? make_float2(-h * (o[3].x + o[3].y), h * (o[3].x - o[3].y))
                   : make_float2(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = make_float2(e[k].x + o[k].x, e[k].y + o[k].y);
            v[k + 4] = make_float2(e[k].x - o[k].x, e[k].y - o[k].y);
        }
    }
}

// One pass over all blocks of `len` elements; ends with a barrier.
template <bool INV, int R>
__device__ __forceinline__ void fft_pass(float2* z, int n, int len, const float2* __restrict__ tw, int G)
{
    constexpr int LR = R == 2 ? 1 : (R == 4 ? 2 : 3);
    const int sub = len >> LR;
    const int ts = G / len;
    for (int b = threadIdx.x; b < (n >> LR); b += blockDim.x) {
        const int j = b & (sub - 1);
        const int base = ((b - j) << LR) + j;
        float2 v[R], w[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = z[fft_sw(base + q * sub)];
        if (sub > 1) {
            // w^q, all from the table (a product of two entries would round twice more); entry t + G/2 is minus entry t
#pragma unroll
            for (int q = 1; q < R; ++q) {
                const int t = q * j * ts, h = G >> 1;
                w[q] = __ldg(&tw[t & (h - 1)]);
                if (2 * q > R && t >= h) w[q] = make_float2(-w[q].x, -w[q].y);
            }
        }
        if (INV && sub > 1) {
#pragma unroll
            for (int q = 1; q < R; ++q) v[q] = cmul(v[q], make_float2(w[q].x, -w[q].y));
        }
        dft_r<INV, R>(v);
        if (!INV && sub > 1) {
#pragma unroll
            for (int q = 1; q < R; ++q) v[q] = cmul(v[q], w[q]);
        }
#pragma unroll
        for (int q = 0; q < R; ++q) z[fft_sw(base + q * sub)] = v[q];
    }
    __syncthreads();
}

// The barrier before the first pass is the caller's.
template <bool INV>
__device__ inline void fft_inplace(float2* z, int n, int log2n, const float2* __restrict__ tw, int G)
{
    const int r = log2n % 3;
    if (!INV) {
        if (r == 1) fft_pass<false, 2>(z, n, n, tw, G);
        else if (r == 2) fft_pass<false, 4>(z, n, n, tw, G);
        for (int len = n >> r; len > 1; len >>= 3) fft_pass<false, 8>(z, n, len, tw, G);
    } else {
        for (int len = 8; len <= (n >> r); len <<= 3) fft_pass<true, 8>(z, n, len, tw, G);
        if (r == 1) fft_pass<true, 2>(z, n, n, tw, G);
        else if (r == 2) fft_pass<true, 4>(z, n, n, tw, G);
    }
}

// Real-input FFT post-processing, filter by D, and pre-processing of the
// real-output inverse, all on the packed spectrum z (length Gh = G/2, in the
// forward transform's order):
//   z_j = g_{2j} + i g_{2j+1},  Z = FFT_Gh(z)
//   X_k = (Z_k + conj Z_{Gh-k})/2 + e^{-2 pi i k/G} (Z_k - conj Z_{Gh-k})/(2i)   (k = 0..Gh)
//   Y_k = D_k X_k
//   Z'_k = (Y_k + conj Y_{Gh-k}) + i e^{2 pi i k/G} (Y_k - conj Y_{Gh-k})       (k < Gh)
// so that IFFT_Gh(Z') interleaves the real sequence h_l = sum_k Y_k e^{2 pi i k l/G}.
// DERIV: the filter is i g_k with the real table g (derivative coefficients
// 2 pi i k c_k over psi^2), i.e. Y_k = i g_k X_k.
// zo: where Z' is written (z itself, or a second buffer).
template <bool DERIV>
__device__ inline void real_filter(const float2* z, float2* zo, int Gh, int log2n, const float* __restrict__ D,
                                   const float2* __restrict__ tw)
{
    for (int k = threadIdx.x; k <= (Gh >> 1); k += blockDim.x) {
        if (k == 0) {
            const float2 z0 = z[0];
            if (DERIV) {
                // g_0 = 0 and g_{Gh} = 0 (Gh > N_ft/2): the real parts at k = 0, Gh vanish
                zo[0] = make_float2(0.0f, 0.0f);
                continue;
            }
            const float y0 = __ldg(&D[0]) * (z0.x + z0.y);
            const float yh = __ldg(&D[Gh]) * (z0.x - z0.y);
            zo[0] = make_float2(y0 + yh, y0 - yh);
            continue;
        }
        const int k2 = Gh - k;
        const int i1 = fft_sw(fft_pos(k, log2n)), i2 = fft_sw(fft_pos(k2, log2n));
        const float2 zk = z[i1];
        const float2 zc = make_float2(z[i2].x, -z[i2].y);  // conj Z_{Gh-k}
        const float2 A = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y + zc.y));
        const float2 B = make_float2(0.5f * (zk.y - zc.y), -0.5f * (zk.x - zc.x));  // -i (Zk - Zc)/2
        const float2 t = __ldg(&tw[k]);
        const float2 tB = cmul(t, B);
        const float2 Xk = make_float2(A.x + tB.x, A.y + tB.y);
        const float2 Xk2 = make_float2(A.x - tB.x, -(A.y - tB.y));  // conj(A - t B)
        const float dk = __ldg(&D[k]);
        const float dk2 = __ldg(&D[k2]);
        const float2 Yk = DERIV ? make_float2(-dk * Xk.y, dk * Xk.x) : make_float2(dk * Xk.x, dk * Xk.y);
        const float2 Yk2 = DERIV ? make_float2(-dk2 * Xk2.y, dk2 * Xk2.x) : make_float2(dk2 * Xk2.x, dk2 * Xk2.y);
        const float2 tc = make_float2(t.x, -t.y);  // e^{+2 pi i k / G}
        // Z'_k = (Yk + conj Yk2) + i tc (Yk - conj Yk2)
        {
            const float2 sum = make_float2(Yk.x + Yk2.x, Yk.y - Yk2.y);
            const float2 dif = make_float2(Yk.x - Yk2.x, Yk.y + Yk2.y);
            const float2 r = cmul(tc, dif);
            zo[i1] = make_float2(sum.x - r.y, sum.y + r.x);
        }
        // Z'_{k2} = (Yk2 + conj Yk) + i (-t) (Yk2 - conj Yk)
        {
            const float2 sum = make_float2(Yk2.x + Yk.x, Yk2.y - Yk.y);
            const float2 dif = make_float2(Yk2.x - Yk.x, Yk2.y + Yk.y);
            const float2 r = cmul(make_float2(-t.x, -t.y), dif);
            zo[i2] = make_float2(sum.x - r.y, sum.y + r.x);
        }
    }
}

// Grid cell c of the real sequence in the transform's buffer.
__device__ __forceinline__ float& fft_cell(float* grid, int c) { return grid[2 * fft_sw(c >> 1) + (c & 1)]; }

// Copy the inverse transform's G cells to global memory: dst[c] = cell (c + shift) mod G, shift even.
__device__ __forceinline__ void fft_store(const float* grid, float* dst, int G, int shift)
{
    const float2* z = reinterpret_cast<const float2*>(grid);
    float2* out = reinterpret_cast<float2*>(dst);
    const int Gh = G >> 1, hs = shift >> 1;
    for (int i = threadIdx.x; i < Gh; i += blockDim.x) out[i] = z[fft_sw((i + hs) & (Gh - 1))];
}

constexpr int IT_THREADS = 256;
constexpr int ROW_PAD = 16;  // >= QS_MAX_W, keeps rows 64-byte aligned

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Copy the G-cell row `src` into `dst` followed by its first ROW_PAD cells.
__device__ __forceinline__ void stage_row(float* dst, const float* src, int G)
{
    const int n16 = (G + ROW_PAD) >> 2;
    for (int i = threadIdx.x; i < n16; i += blockDim.x) {
        const int c = (i << 2) < G ? (i << 2) : (i << 2) - G;
        cp_async16(dst + (i << 2), src + c);
    }
    cp_async_commit();
}


// ---------------------------------------------------------------------------
// One 128-slice x 128-point tile of the FP32 projection GEMM
//     U[p][n] = sum_j A[p][j] X[n][j]   (A = G tau Xi, X points, both K-major)
// by a CTA of 256 threads: 8-deep k slabs double-buffered in shared memory
// (`smem`: 2 x 8 x 256 floats = 16 KB), 8 x 8 outputs per thread.  Rows
// p >= P are not stored; columns n0..n0+127 are stored (U needs ldU >=
// round_up(N, 128)).
// ---------------------------------------------------------------------------
constexpr int GT_BM = 128;
constexpr int GT_BN = 128;
constexpr int GT_BK = 8;

template <bool VEC>
__device__ __forceinline__ void gemm_load_slab(const float* __restrict__ A, int P, const float* __restrict__ X,
                                               int64_t N, int d, int p0, int64_t n0, int k0, int lrow, int lk,
                                               float (&ra)[4], float (&rb)[4])
{
    const int gp = p0 + lrow;
    const int64_t gn = n0 + lrow;
    const int kk = k0 + lk;
    if (VEC && kk + 3 < d) {
        float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
        if (gp < P) va = __ldg(reinterpret_cast<const float4*>(A + (size_t)gp * d + kk));
        if (gn < N) vb = __ldg(reinterpret_cast<const float4*>(X + (size_t)gn * d + kk));
        ra[0] = va.x; ra[1] = va.y; ra[2] = va.z; ra[3] = va.w;
        rb[0] = vb.x; rb[1] = vb.y; rb[2] = vb.z; rb[3] = vb.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ra[i] = (gp < P && kk + i < d) ? __ldg(A + (size_t)gp * d + kk + i) : 0.0f;
            rb[i] = (gn < N && kk + i < d) ? __ldg(X + (size_t)gn * d + kk + i) : 0.0f;
        }
    }
}

template <bool VEC>
__device__ inline void gemm_tile_fp32(const float* __restrict__ X, int64_t N, int d, const float* __restrict__ A,
                                      int P, float* __restrict__ U, int64_t ldU, int p0, int64_t n0, float* smem)
{
    float(*As)[GT_BK][GT_BM] = reinterpret_cast<float(*)[GT_BK][GT_BM]>(smem);
    float(*Bs)[GT_BK][GT_BN] = reinterpret_cast<float(*)[GT_BK][GT_BN]>(smem + 2 * GT_BK * GT_BM);
    const int tid = threadIdx.x;
    const int tx = tid & 15;
    const int ty = tid >> 4;
    const int lrow = tid >> 1;
    const int lk = (tid & 1) * 4;

    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;

    float ra[4], rb[4];
    const int nk = (d + GT_BK - 1) / GT_BK;
    gemm_load_slab<VEC>(A, P, X, N, d, p0, n0, 0, lrow, lk, ra, rb);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        As[0][lk + i][lrow] = ra[i];
        Bs[0][lk + i][lrow] = rb[i];
    }
    __syncthreads();

    for (int kt = 0; kt < nk; ++kt) {
        const int cur = kt & 1;
        if (kt + 1 < nk) gemm_load_slab<VEC>(A, P, X, N, d, p0, n0, (kt + 1) * GT_BK, lrow, lk, ra, rb);
#pragma unroll
        for (int k = 0; k < GT_BK; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[cur][k][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[cur][k][64 + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[cur][k][tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Bs[cur][k][64 + tx * 4]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (kt + 1 < nk) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                As[cur ^ 1][lk + i][lrow] = ra[i];
                Bs[cur ^ 1][lk + i][lrow] = rb[i];
            }
        }
        __syncthreads();
    }

    // rows: p0 + ty*4 + i (i < 4) and p0 + 64 + ty*4 + (i - 4); columns likewise
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int p = p0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4));
        if (p >= P) continue;
        float* row = U + (size_t)p * ldU + n0;
        *reinterpret_cast<float4*>(row + tx * 4) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(row + 64 + tx * 4) = make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
}

}  // namespace qsdev
