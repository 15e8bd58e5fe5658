// Kernels of fmg_small.h, for one working type per translation unit.
//
// Level by level, a V-cycle below 128 cells per side is a chain of launches of
// a few microseconds each that move every array through global memory; a
// sample's levels up to 64 x 64 (faces, right-hand sides, iterates: 92 KB in
// FP32) fit in shared memory, so one CTA walks the whole chain with a CTA
// barrier between phases. The arithmetic of every cell is that of the
// per-level kernels (kb_rbgs_whole or, on sides it does not take, kb_gs;
// kb_resid_restrict, kb_prolong, kb_coarse_fixed or kb_coarse,
// kb_prolong_resid64, kb_resnorm_part): the same bits. The FP64 form, which takes
// these kernels for small calls only, sums F_t in the order of kb_qoi too.
#pragma once

#include <type_traits>

#include "fmg_small.h"
#include "ptx_async.cuh"

namespace mlqmc_small {
namespace {
using namespace mlqmc_dev;
using namespace mlqmc_ptx;

// sides whose per-level smoother is kb_gs and whose coarse solve is kb_coarse
template <int NC>
constexpr bool kPlain = NC != 4 && NC != 8;

template <int NC>
__device__ __forceinline__ void split(const Level& L, bool half, int q, int& y, int& x)
{
    if constexpr (!kPlain<NC>) {
        const int s = L.lg - (half ? 1 : 0);
        y = q >> s;
        x = q - (y << s);
    } else {
        y = static_cast<int>((half ? L.by_nc : L.by_n).div(static_cast<uint32_t>(q)));
        x = q - y * (half ? L.n >> 1 : L.n);
    }
}

// One half sweep from shared memory (FP64, and FP32 on sides without register
// blocks; both multiply by the level's stored 1/D). FIRST: u is zero on entry (the first colour of a correction:
// the other colour's values are not read, nothing has to be cleared).
template <typename T, int NC, bool FIRST>
__device__ __forceinline__ void half_sweep(const Level& L, T* S, int colour, bool ones)
{
    const int n = L.n, nc = n >> 1, XP = kx_pitch(n);
    T* su = S + L.oU;
    const T *skx = S + L.oKx, *sky = S + L.oKy, *sb = S + L.oB, *sd = S + L.oD;
    const T h2 = T(1) / (T(n) * T(n));
    for (int q = threadIdx.x; q < n * nc; q += blockDim.x) {
        int y, m;
        split<NC>(L, true, q, y, m);
        const int x = 2 * m + ((y + colour) & 1);
        const int c0 = y * n + x;
        const T* kr = skx + y * XP;
        T acc = h2;  // b = 1: no product
        if (!ones) acc = mul_rn(h2, sb[c0]);
        if constexpr (!FIRST)
            acc = gs_sum(acc, kr[x], x > 0 ? su[c0 - 1] : T(0), kr[x + 1], x < n - 1 ? su[c0 + 1] : T(0),
                         sky[c0], y > 0 ? su[c0 - n] : T(0), sky[c0 + n], y < n - 1 ? su[c0 + n] : T(0));
        su[c0] = acc * sd[c0];
    }
    __syncthreads();
}

// bc of level t-1: mean over the 4 children of b - A u (resid_restrict_cell's arithmetic).
template <typename T, int NC>
__device__ __forceinline__ void restrict_residual(const Level& F, const Level& C, T* S, bool ones)
{
    const int n = F.n, nc = n >> 1, XP = kx_pitch(n);
    const T *su = S + F.oU, *skx = S + F.oKx, *sky = S + F.oKy, *sb = S + F.oB;
    const T ih2 = T(n) * T(n);
    for (int q = threadIdx.x; q < nc * nc; q += blockDim.x) {
        int I2, I1;
        split<NC>(C, false, q, I2, I1);
        if constexpr (sizeof(T) == 8) {
            const int o = 2 * I2 * n + 2 * I1;
            const double qf = quad_flux(skx + 2 * I2 * XP + 2 * I1, sky + o, su + o, n, XP, I1 > 0, I1 < nc - 1, I2 > 0,
                                        I2 < nc - 1);
            const double sum = ones ? 4.0 : (sb[o] + sb[o + 1]) + (sb[o + n] + sb[o + n + 1]);
            S[C.oB + q] = 0.25 * fma(-ih2, qf, sum);
            continue;
        }
        T s = T(0);
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            const int x = 2 * I1 + (d & 1), y = 2 * I2 + (d >> 1);
            const int c0 = y * n + x;
            const T up = su[c0];
            const T* kr = skx + y * XP;
            const T a2 = flux_sum<T>(cell_head(d), kr[x], up - (x > 0 ? su[c0 - 1] : T(0)), kr[x + 1],
                                     up - (x < n - 1 ? su[c0 + 1] : T(0)), sky[c0], up - (y > 0 ? su[c0 - n] : T(0)),
                                     sky[c0 + n], up - (y < n - 1 ? su[c0 + n] : T(0)));
            s += fma(-ih2, a2, ones ? T(1) : sb[c0]);
        }
        S[C.oB + q] = T(0.25) * s;
    }
    __syncthreads();
}

// The 2 x 2 fine cells of every coarse parent from the parent's 3 x 3
// neighbourhood, odd reflection across the boundary: dst += P e, or dst = P e.
template <typename T, int NC, bool ADD>
__device__ __forceinline__ void interpolate(const Level& C, const T* se, T* dst)
{
    const int nc = C.n, n = 2 * nc;
    for (int q = threadIdx.x; q < nc * nc; q += blockDim.x) {
        int I2, I1;
        split<NC>(C, false, q, I2, I1);
        const bool lo1 = I1 == 0, hi1 = I1 == nc - 1, lo2 = I2 == 0, hi2 = I2 == nc - 1;
        T E[3][3];
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
                const bool ry = (dy < 0 && lo2) || (dy > 0 && hi2);
                const bool rx = (dx < 0 && lo1) || (dx > 0 && hi1);
                const T v = se[(I2 + (ry ? 0 : dy)) * nc + I1 + (rx ? 0 : dx)];
                E[dy + 1][dx + 1] = (ry != rx) ? -v : v;
            }
        }
        T* f = dst + (2 * I2) * n + 2 * I1;
        if constexpr (sizeof(T) == 8) {
            double v[2][2];
            prolong_quad64(E, v);
#pragma unroll
            for (int fy = 0; fy < 2; ++fy)
#pragma unroll
                for (int fx = 0; fx < 2; ++fx) {
                    if constexpr (ADD) f[fy * n + fx] += v[fy][fx];
                    else f[fy * n + fx] = v[fy][fx];
                }
        } else {
#pragma unroll
            for (int fy = 0; fy < 2; ++fy)
#pragma unroll
                for (int fx = 0; fx < 2; ++fx) {
                    const T v = fma(T(0.5625), E[1][1], fma(T(0.1875), E[1][2 * fx] + E[2 * fy][1], T(0.0625) * E[2 * fy][2 * fx]));
                    if constexpr (ADD) f[fy * n + fx] += v;
                    else f[fy * n + fx] = v;
                }
        }
    }
    __syncthreads();
}

// u_0 = A_0^-1 bc_0. FP32: one thread with the factor's columns (and rows) as
// padded vectors in shared memory, every solved row pushed into the pending
// sums of the next NC rows in registers: a row costs its nine products and a
// few wide loads, where lanes that hand values on pay a shuffle per row. FP64
// (a warp instruction costs ~70 cycles whatever its lanes): NC lanes, each
// with the pending value of one row. Oldest term first as in kb_coarse_fixed
// (kPlain FP32: newest first as in kb_coarse).
template <int NC>
struct CoarseGeom {
    static constexpr int N = NC * NC, W = (NC + 1 + 3) / 4 * 4;  // row pitch
    static constexpr int elems = 2 * N * W;  // rows L(r, r - e), then columns L(r + e, r), e = 0..NC
};

template <typename T, int NC>
__device__ __forceinline__ void coarse_solve(const T* ch, const T* b, T* x)
{
    using Gm = CoarseGeom<NC>;
    constexpr int N = Gm::N, W = Gm::W;
    const T* col = ch + N * W;
    const T h2 = T(1) / (T(NC) * T(NC));
    if constexpr (sizeof(T) == 4) {
        if (threadIdx.x == 0) {
            auto row9 = [](const float* p, float (&o)[W]) {
#pragma unroll
                for (int k = 0; k < W / 4; ++k) {
                    const float4 v = reinterpret_cast<const float4*>(p)[k];
                    o[4 * k] = v.x;
                    o[4 * k + 1] = v.y;
                    o[4 * k + 2] = v.z;
                    o[4 * k + 3] = v.w;
                }
            };
            if constexpr (!kPlain<NC>) {
                // push: a solved row updates the NC pending sums in registers
                // (independent products; only the next row's is on the chain).
                // The factor comes four rows ahead and x goes out four rows at
                // a time: a store between the loads would hold each of them back.
                constexpr int GR = 4;
                auto load = [&](const float* p, float (&o)[GR][W], int r) {
#pragma unroll
                    for (int k = 0; k < GR; ++k) row9(p + (r + k) * W, o[k]);
                };
                auto four = [](const float* p, float (&o)[GR]) {
                    const float4 v = *reinterpret_cast<const float4*>(p);
                    o[0] = v.x;
                    o[1] = v.y;
                    o[2] = v.z;
                    o[3] = v.w;
                };
                float acc[NC];  // row r + 1 .. r + NC at (row mod NC)
                float cur[GR][W], nxt[GR][W];
#pragma unroll
                for (int q = 0; q < NC; ++q) acc[q] = __fmul_rn(h2, b[q]);
                load(col, cur, 0);
                for (int r0 = 0; r0 < N; r0 += NC) {
#pragma unroll
                    for (int g = 0; g < NC; g += GR) {
                        const int r = r0 + g;
                        float nb[GR], xr[GR];  // the right-hand sides that enter, the rows solved
                        load(col, nxt, r + GR < N ? r + GR : r);
                        four(b + (r0 + NC < N ? r + NC : r), nb);
#pragma unroll
                        for (int k = 0; k < GR; ++k) {
                            const int a = g + k;
                            xr[k] = __fmul_rn(acc[a], cur[k][0]);
                            acc[a] = r0 + NC < N ? __fmul_rn(h2, nb[k]) : 0.0f;
#pragma unroll
                            for (int q = 1; q <= NC; ++q) acc[(a + q) % NC] = __fmaf_rn(-cur[k][q], xr[k], acc[(a + q) % NC]);
                        }
                        *reinterpret_cast<float4*>(x + r) = make_float4(xr[0], xr[1], xr[2], xr[3]);
#pragma unroll
                        for (int k = 0; k < GR; ++k)
#pragma unroll
                            for (int q = 0; q <= NC; ++q) cur[k][q] = nxt[k][q];
                    }
                }
                load(ch, cur, N - GR);
#pragma unroll
                for (int q = 0; q < NC; ++q) acc[q] = x[N - NC + q];
                for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
                    for (int g = NC - GR; g >= 0; g -= GR) {
                        const int r = r0 + g;
                        float nb[GR], xr[GR];
                        load(ch, nxt, r >= GR ? r - GR : 0);
                        four(x + (r0 > 0 ? r - NC : r), nb);
#pragma unroll
                        for (int k = GR - 1; k >= 0; --k) {
                            const int a = g + k;
                            xr[k] = __fmul_rn(acc[a], cur[k][0]);
                            acc[a] = r0 > 0 ? nb[k] : 0.0f;
#pragma unroll
                            for (int q = 1; q <= NC; ++q) acc[(a + NC - q) % NC] = __fmaf_rn(-cur[k][q], xr[k], acc[(a + NC - q) % NC]);
                        }
                        *reinterpret_cast<float4*>(x + r) = make_float4(xr[0], xr[1], xr[2], xr[3]);
#pragma unroll
                        for (int k = 0; k < GR; ++k)
#pragma unroll
                            for (int q = 0; q <= NC; ++q) cur[k][q] = nxt[k][q];
                    }
                }
            } else {
                // newest term first (as kb_coarse): the last NC values in a static window
                float win[NC];  // win[r mod NC]
#pragma unroll
                for (int q = 0; q < NC; ++q) win[q] = 0.0f;
                for (int r0 = 0; r0 < N; r0 += NC) {
#pragma unroll
                    for (int a = 0; a < NC; ++a) {
                        float l[W];
                        row9(ch + (r0 + a) * W, l);
                        float v = __fmul_rn(h2, b[r0 + a]);
#pragma unroll
                        for (int q = 1; q <= NC; ++q) v = __fmaf_rn(-l[q], win[(a + NC - q) % NC], v);
                        win[a] = __fmul_rn(v, l[0]);
                        x[r0 + a] = win[a];
                    }
                }
#pragma unroll
                for (int q = 0; q < NC; ++q) win[q] = 0.0f;
                for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
                    for (int a = NC - 1; a >= 0; --a) {
                        float l[W];
                        row9(col + (r0 + a) * W, l);
                        float v = x[r0 + a];
#pragma unroll
                        for (int q = 1; q <= NC; ++q) v = __fmaf_rn(-l[q], win[(a + q) % NC], v);
                        win[a] = __fmul_rn(v, l[0]);
                        x[r0 + a] = win[a];
                    }
                }
            }
        }
    } else {
        if (threadIdx.x < 32) {
            const int p = threadIdx.x < NC ? threadIdx.x : 0;
            const bool own = threadIdx.x < NC;
            double v = h2 * b[p];
            for (int r0 = 0; r0 < N; r0 += NC) {
#pragma unroll
                for (int a = 0; a < NC; ++a) {
                    const int r = r0 + a, e = p > a ? p - a : p - a + NC;  // the slot's row is r + e
                    const double xr = __shfl_sync(0xffffffffu, v, a) * col[r * W];
                    if (p == a) v = r + NC < N ? h2 * b[r + NC] : 0.0;
                    v = fma(-col[r * W + e], xr, v);
                    if (own && p == a) x[r] = xr;
                }
            }
            __syncwarp();
            v = x[N - NC + p];
            for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
                for (int a = NC - 1; a >= 0; --a) {
                    const int r = r0 + a, e = p < a ? a - p : a - p + NC;  // the slot's row is r - e
                    const double xr = __shfl_sync(0xffffffffu, v, a) * ch[r * W];
                    if (p == a) v = r - NC >= 0 ? x[r - NC] : 0.0;
                    v = fma(-ch[r * W + e], xr, v);
                    if (own && p == a) x[r] = xr;
                }
            }
        }
    }
    __syncthreads();
}

// Sweeps of a level from registers (FP32, N = 8, 16, 32, 64): a thread keeps an
// RB x RB block of cells (its u, b, faces and the reciprocal of the diagonal);
// left and right neighbours come by shuffles, the rows above and below through
// the level's u array with one barrier of the level's threads per half sweep.
// From shared memory alone a half sweep costs ten shared-memory wavefronts per
// 32 updates; this way about two, and the update itself is the rest. A row's
// store rewrites the other colour's unchanged values, and a reader uses only
// the colour just updated, so one buffer suffices.
template <int N>
struct Blk {
    static constexpr int RB = N >= 64 ? 4 : 2, TX = N / RB, NT = TX * TX;
};

template <int NT>
__device__ __forceinline__ void level_sync()
{
    if constexpr (NT <= 32) __syncwarp(NT == 32 ? 0xffffffffu : (1u << NT) - 1u);
    else asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

template <int N>
struct Visit {
    static constexpr int RB = Blk<N>::RB, TX = Blk<N>::TX, NT = Blk<N>::NT, XP = N + 4;
    static constexpr unsigned kMask = NT >= 32 ? 0xffffffffu : (1u << NT) - 1u;
    float u[RB][RB], b[RB][RB], kx[RB][RB + 1], ky[RB + 1][RB], rd[RB][RB];
    float up[RB], dn[RB];  // the rows above and below the block
    int tx, ty;
    float* su;

    // RB consecutive values of a row (16- or 8-byte aligned: every part of the plan and every row is)
    __device__ __forceinline__ void get_row(const float* p, float (&o)[RB]) const
    {
        if constexpr (RB == 4) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            o[0] = v.x;
            o[1] = v.y;
            o[2] = v.z;
            o[3] = v.w;
        } else {
            const float2 v = *reinterpret_cast<const float2*>(p);
            o[0] = v.x;
            o[1] = v.y;
        }
    }
    __device__ __forceinline__ void load(const Level& L, float* S)
    {
        tx = threadIdx.x % TX;
        ty = threadIdx.x / TX;
        su = S + L.oU;
        const float *skx = S + L.oKx, *sky = S + L.oKy, *sb = S + L.oB;
#pragma unroll
        for (int y = 0; y < RB; ++y) {
            float k[RB];
            get_row(skx + (ty * RB + y) * XP + tx * RB, k);
#pragma unroll
            for (int x = 0; x < RB; ++x) kx[y][x] = k[x];
            // the face after the block is the right neighbour's first
            const float nx = __shfl_down_sync(kMask, k[0], 1, TX < 32 ? TX : 32);
            kx[y][RB] = tx < TX - 1 ? nx : skx[(ty * RB + y) * XP + N];
            get_row(sb + (ty * RB + y) * N + tx * RB, b[y]);
        }
#pragma unroll
        for (int y = 0; y <= RB; ++y) get_row(sky + (ty * RB + y) * N + tx * RB, ky[y]);
#pragma unroll
        for (int y = 0; y < RB; ++y)
#pragma unroll
            for (int x = 0; x < RB; ++x)
                rd[y][x] = __fdividef(1.0f, kx[y][x] + kx[y][x + 1] + ky[y][x] + ky[y + 1][x]);
    }
    __device__ __forceinline__ void load_u()
    {
#pragma unroll
        for (int y = 0; y < RB; ++y) get_row(su + (ty * RB + y) * N + tx * RB, u[y]);
    }
    __device__ __forceinline__ void zero_u()
    {
#pragma unroll
        for (int y = 0; y < RB; ++y)
#pragma unroll
            for (int x = 0; x < RB; ++x) u[y][x] = 0.0f;
    }
    __device__ __forceinline__ void put_row(int y) const
    {
        float* d = su + (ty * RB + y) * N + tx * RB;
        if constexpr (RB == 4) *reinterpret_cast<float4*>(d) = make_float4(u[y][0], u[y][1], u[y][2], u[y][3]);
        else *reinterpret_cast<float2*>(d) = make_float2(u[y][0], u[y][1]);
    }
    // the block's first and last rows to the neighbours, theirs back
    __device__ __forceinline__ void exchange()
    {
        put_row(0);
        put_row(RB - 1);
        level_sync<NT>();
        float a[RB], d[RB];
        get_row(su + (ty > 0 ? ty * RB - 1 : 0) * N + tx * RB, a);
        get_row(su + (ty < TX - 1 ? ty * RB + RB : 0) * N + tx * RB, d);
#pragma unroll
        for (int x = 0; x < RB; ++x) {
            up[x] = ty > 0 ? a[x] : 0.0f;
            dn[x] = ty < TX - 1 ? d[x] : 0.0f;
        }
    }
    __device__ __forceinline__ float left(int y) const
    {
        const float v = __shfl_up_sync(kMask, u[y][RB - 1], 1, TX < 32 ? TX : 32);
        return tx > 0 ? v : 0.0f;
    }
    __device__ __forceinline__ float right(int y) const
    {
        const float v = __shfl_down_sync(kMask, u[y][0], 1, TX < 32 ? TX : 32);
        return tx < TX - 1 ? v : 0.0f;
    }
    // one half sweep from the current up, dn; colour 0: x + y even (RB even: the block's own parity)
    template <int COLOUR>
    __device__ __forceinline__ void half()
    {
        constexpr float h2 = 1.0f / (static_cast<float>(N) * N);
#pragma unroll
        for (int y = 0; y < RB; ++y) {
            const float l = (y & 1) == COLOUR ? left(y) : 0.0f;           // cell x = 0 has this colour
            const float r = ((RB - 1 + y) & 1) == COLOUR ? right(y) : 0.0f;  // cell x = RB - 1 has it
#pragma unroll
            for (int x = 0; x < RB; ++x) {
                if (((x + y) & 1) != COLOUR) continue;
                const float acc = gs_sum_b<float, (N > 8)>(h2, b[y][x], kx[y][x], x > 0 ? u[y][x > 0 ? x - 1 : 0] : l, kx[y][x + 1],
                                      x < RB - 1 ? u[y][x < RB - 1 ? x + 1 : 0] : r, ky[y][x],
                                      y > 0 ? u[y > 0 ? y - 1 : 0][x] : up[x], ky[y + 1][x],
                                      y < RB - 1 ? u[y < RB - 1 ? y + 1 : 0][x] : dn[x]);
                u[y][x] = acc * rd[y][x];
            }
        }
    }
    // sweeps starting with colour FIRST; on return up, dn are current
    template <int FIRST>
    __device__ __forceinline__ void sweeps(int n)
    {
        for (int k = 0; k < n; ++k) {
            half<FIRST>();
            exchange();
            half<1 - FIRST>();
            exchange();
        }
    }
    __device__ __forceinline__ void put_all() const
    {
#pragma unroll
        for (int y = 0; y < RB; ++y) put_row(y);
    }
};

// Pre-smoothing of a level and the restricted residual (bc of the level below).
template <int N>
__device__ __forceinline__ void visit_down(const Level& L, const Level& C, float* S, int nu, bool zero)
{
    using V = Visit<N>;
    constexpr int RB = V::RB;
    if (threadIdx.x < V::NT) {
        V v;
        v.load(L, S);
        if (zero) {
            v.zero_u();
#pragma unroll
            for (int x = 0; x < RB; ++x) v.up[x] = v.dn[x] = 0.0f;
        } else {
            v.load_u();
            v.exchange();
        }
        v.template sweeps<0>(nu);
        constexpr float ih2 = static_cast<float>(N) * N;
        float r[RB][RB];
#pragma unroll
        for (int y = 0; y < RB; ++y) {
            const float l = v.left(y), rt = v.right(y);
#pragma unroll
            for (int x = 0; x < RB; ++x) {
                const float c = v.u[y][x];
                const float a2 = flux_sum<float>(whole_head((x & 1) + 2 * (y & 1)), v.kx[y][x], c - (x > 0 ? v.u[y][x > 0 ? x - 1 : 0] : l),
                                                 v.kx[y][x + 1], c - (x < RB - 1 ? v.u[y][x < RB - 1 ? x + 1 : 0] : rt),
                                                 v.ky[y][x], c - (y > 0 ? v.u[y > 0 ? y - 1 : 0][x] : v.up[x]),
                                                 v.ky[y + 1][x], c - (y < RB - 1 ? v.u[y < RB - 1 ? y + 1 : 0][x] : v.dn[x]));
                r[y][x] = fmaf(-ih2, a2, v.b[y][x]);
            }
        }
#pragma unroll
        for (int y = 0; y < RB; y += 2)
#pragma unroll
            for (int x = 0; x < RB; x += 2)
                S[C.oB + (v.ty * RB + y) / 2 * (N / 2) + (v.tx * RB + x) / 2] =
                    0.25f * (((r[y][x] + r[y][x + 1]) + r[y + 1][x]) + r[y + 1][x + 1]);
        v.put_all();
    }
    __syncthreads();
}

// Coarse-grid correction P e of a level and its post-smoothing.
template <int N>
__device__ __forceinline__ void visit_up(const Level& L, const Level& C, float* S, int nu)
{
    using V = Visit<N>;
    constexpr int RB = V::RB, NCO = N / 2, CB = RB / 2;
    if (threadIdx.x < V::NT) {
        V v;
        v.load(L, S);
        v.load_u();
        const float* se = S + C.oU;
        float E[CB + 2][CB + 2];  // the parents and one coarse cell around them, odd reflection
#pragma unroll
        for (int dy = 0; dy < CB + 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < CB + 2; ++dx) {
                const int I2 = v.ty * CB + dy - 1, I1 = v.tx * CB + dx - 1;
                const bool ry = I2 < 0 || I2 >= NCO, rx = I1 < 0 || I1 >= NCO;
                const float e = se[(ry ? (I2 < 0 ? 0 : NCO - 1) : I2) * NCO + (rx ? (I1 < 0 ? 0 : NCO - 1) : I1)];
                E[dy][dx] = (ry != rx) ? -e : e;
            }
#pragma unroll
        for (int y = 0; y < RB; ++y)
#pragma unroll
            for (int x = 0; x < RB; ++x) {
                const int py = y / 2 + 1, px = x / 2 + 1, qy = py + ((y & 1) ? 1 : -1), qx = px + ((x & 1) ? 1 : -1);
                v.u[y][x] += fmaf(0.5625f, E[py][px], fmaf(0.1875f, E[py][qx] + E[qy][px], 0.0625f * E[qy][qx]));
            }
        v.exchange();
        v.template sweeps<1>(nu);
        v.put_all();
    }
    __syncthreads();
}

// V-cycle of levels t..0. zero: u_t is zero on entry; ones: the right-hand side of level t is 1.
// BIG: levels of 64 cells per side among them (their blocks of 4 x 4 cells take
// 127 registers a thread; without them a CTA needs half of that).
template <typename T, int NC, bool BIG>
__device__ __forceinline__ void vcycle(const Plan& P, T* S, int t, int nu1, int nu2, bool zero, bool ones)
{
    for (int l = t; l >= 1; --l) {
        const Level& F = P.lv[l];
        const bool z = zero || l < t, o = ones && l == t;
        if constexpr (sizeof(T) == 4 && !kPlain<NC>) {
            if constexpr (BIG) {
                if (F.n == 64) {
                    visit_down<64>(F, P.lv[l - 1], S, nu1, z);
                    continue;
                }
            }
            switch (F.n) {
            case 32: visit_down<32>(F, P.lv[l - 1], S, nu1, z); break;
            case 16: visit_down<16>(F, P.lv[l - 1], S, nu1, z); break;
            default: visit_down<8>(F, P.lv[l - 1], S, nu1, z); break;
            }
        } else {
            if (z) half_sweep<T, NC, true>(F, S, 0, o);
            else half_sweep<T, NC, false>(F, S, 0, o);
            for (int h = 1; h < 2 * nu1; ++h) half_sweep<T, NC, false>(F, S, h & 1, o);
            restrict_residual<T, NC>(F, P.lv[l - 1], S, o);
        }
    }
    coarse_solve<T, NC>(S + P.oChol, S + P.lv[0].oB, S + P.lv[0].oU);
    for (int l = 1; l <= t; ++l) {
        const Level& F = P.lv[l];
        const bool o = ones && l == t;
        if constexpr (sizeof(T) == 4 && !kPlain<NC>) {
            if constexpr (BIG) {
                if (F.n == 64) {
                    visit_up<64>(F, P.lv[l - 1], S, nu2);
                    continue;
                }
            }
            switch (F.n) {
            case 32: visit_up<32>(F, P.lv[l - 1], S, nu2); break;
            case 16: visit_up<16>(F, P.lv[l - 1], S, nu2); break;
            default: visit_up<8>(F, P.lv[l - 1], S, nu2); break;
            }
        } else {
            interpolate<T, NC, true>(P.lv[l - 1], S + P.lv[l - 1].oU, S + F.oU);
            for (int h = 0; h < 2 * nu2; ++h) half_sweep<T, NC, false>(F, S, (h + 1) & 1, o);
        }
    }
}

// Bring the levels' faces (and stored 1/D, and bc of the top level) and the
// level-0 factor into shared memory. False: a copy did not land in time (the
// status is set).
template <typename T, int NC>
__device__ __forceinline__ bool load_levels(const FmgArgs& A, const Plan& P, T* S, uint64_t* bar, int i, bool with_bc)
{
    constexpr int N = NC * NC;
    constexpr uint32_t es = sizeof(T);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t bytes = 0;
        for (int t = 1; t <= P.top; ++t) {
            const uint32_t n = static_cast<uint32_t>(P.lv[t].n);
            bytes += es * (n * static_cast<uint32_t>(kx_pitch(static_cast<int>(n))) + (n + 1) * n + (P.stored_d ? n * n : 0));
        }
        const uint32_t nt = static_cast<uint32_t>(P.lv[P.top].n);
        if (with_bc) bytes += es * nt * nt;
        mbar_arrive_tx(bar, bytes);
        for (int t = P.top; t >= 1; --t) {
            const Level& L = P.lv[t];
            const uint32_t n = static_cast<uint32_t>(L.n);
            if (with_bc && t == P.top) bulk_load(S + L.oB, at<T>(A.lv[t].bc, i), es * n * n, bar);
            bulk_load(S + L.oKx, at<T>(A.lv[t].kx, i), es * n * static_cast<uint32_t>(kx_pitch(L.n)), bar);
            bulk_load(S + L.oKy, at<T>(A.lv[t].ky, i), es * (n + 1) * n, bar);
            if (P.stored_d) bulk_load(S + L.oD, at<T>(A.lv[t].idiag, i), es * n * n, bar);
        }
    }
    // the factor: entry (r, e) = L(r, r - e) of sample i at (r (NC + 1) + e) stride + i, as
    // rows and as columns; entries left of column 0 and rows past N as zeros
    const T* fac = reinterpret_cast<const T*>(sizeof(T) == 4 ? A.chol32 : A.chol.base);
    constexpr int CW = CoarseGeom<NC>::W;
    T* ch = S + P.oChol;
#pragma unroll 4
    for (int q = threadIdx.x; q < N * CW; q += blockDim.x) {
        const int r = q / CW, e = q - r * CW;
        const T v = (e <= NC && e <= r) ? fac[static_cast<size_t>(r * (NC + 1) + e) * A.chol.stride + i] : T(0);
        ch[q] = v;
        if (e <= r) ch[N * CW + (r - e) * CW + e] = v;
        if (r + e >= N) ch[N * CW + q] = T(0);
    }
    if (!with_bc) {  // the FMG stages start from the level-0 solution
        const T* u0 = at<T>(A.lv[0].u, i);
        for (int q = threadIdx.x; q < N; q += blockDim.x) S[P.lv[0].oU + q] = u0[q];
    }
    const bool landed = mbar_wait(bar, 0, A.status, kStatusTimeout);
    if (!landed) {  // gave up: let the copies land before the CTA leaves
        const uint64_t t0 = now_ns();
        while (!mbar_test(bar, 0) && now_ns() - t0 < 1000000000ull) {
        }
    }
    return __syncthreads_and(landed ? 1 : 0) != 0;
}

template <typename T, int NC, bool BIG>
__global__ void __launch_bounds__(256, BIG ? 2 : 3) kb_small_vcycle(FmgArgs A, Plan P, int B)
{
    extern __shared__ __align__(128) unsigned char smraw[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smraw);
    T* S = reinterpret_cast<T*>(smraw + 128);
    const int i = blockIdx.x;
    if (A.active && !A.active[i]) return;  // uniform per CTA
    if (!load_levels<T, NC>(A, P, S, bar, i, true)) return;
    vcycle<T, NC, BIG>(P, S, P.top, A.nu1, A.nu2, true, false);
    const Level& L = P.lv[P.top];
    using V = typename std::conditional<sizeof(T) == 8, double2, float4>::type;  // 16-byte stores
    constexpr int VE = 16 / sizeof(T);
    V* g = reinterpret_cast<V*>(at<T>(A.lv[P.top].u, i));
    for (int q = threadIdx.x; q < L.n * L.n / VE; q += blockDim.x) g[q] = reinterpret_cast<const V*>(S + L.oU)[q];
}

// Sum of FP32 pairs h + l kept as three floats (TwoSum on h, TwoSum of its
// error and of l on the second, the rest on the third): below FP64 rounding
// for the few values a thread sums, without the FP64 pipe.
struct TripleSum {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float h, float l)
    {
        float e, f;
        two_sum32(a, h, a, e);
        two_sum32(b, e, b, f);
        c = __fadd_rn(c, f);
        two_sum32(b, l, b, f);
        c = __fadd_rn(c, f);
    }
    __device__ __forceinline__ double value() const { return widen(a) + (widen(b) + widen(c)); }
};

// Sum over the CTA, complete in thread 0 (ALL: in every thread), in a fixed
// order: shuffles inside the warps, then over the warps' sums.
template <bool ALL>
__device__ __forceinline__ double cta_sum(double v, double* red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int nw = blockDim.x >> 5;
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < nw ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    if constexpr (ALL) {
        if (threadIdx.x == 0) red[8] = v;
        __syncthreads();
        v = red[8];
    }
    return v;
}

// FMG stages 1..top of one sample per CTA: the interpolation of the level
// below, mu0 V-cycles, F_t. FP32 (mixed forms): the interpolant U and the
// residual r = 1 - A U in error-free pairs, the V-cycles on A e = r from zero,
// u = U + e; converged form: then FP64 residuals and corrections until the
// sample's norm is below the threshold. FP64: the V-cycles act on u.
template <typename T, int NC, bool CONV, bool BIG>
__global__ void __launch_bounds__(256, BIG ? 2 : 3) kb_small_stages(FmgArgs A, Plan P, Stages G)
{
    static_assert(!CONV || sizeof(T) == 4, "the converged FP64 form keeps its stages level by level");
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ double red[sizeof(T) == 8 ? 128 : 16];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smraw);
    T* S = reinterpret_cast<T*>(smraw + 128);
    const int i = G.i0 + blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    if (!load_levels<T, NC>(A, P, S, bar, i, false)) return;
    for (int t = 1; t <= P.top; ++t) {
        const Level& L = P.lv[t];
        const Level& C = P.lv[t - 1];
        const int n = L.n, nn = n * n, XP = kx_pitch(n);
        T* su = S + L.oU;
        double F;  // complete in thread 0
        const double inv = 1.0 / static_cast<double>(nn);  // exact where n0 is a power of two
        auto mean_of = [&](double sum) { return kPlain<NC> ? sum / static_cast<double>(nn) : sum * inv; };
        if constexpr (sizeof(T) == 8) {
            interpolate<T, NC, false>(C, S + C.oU, su);
            for (int m = 0; m < A.mu0; ++m) vcycle<T, NC, BIG>(P, S, t, A.nu1, A.nu2, false, true);
            if (A.qoi == MLQMC_QOI_MEAN) {
                F = mean_of(sum128_cta(su, nn, red));
            } else {
                const int m = n / 2;
                F = 0.25 * (su[(m - 1) * n + (m - 1)] + su[(m - 1) * n + m] + su[m * n + (m - 1)] + su[m * n + m]);
                __syncthreads();
            }
            if (G.keep || t == P.top) {
                double2* g = reinterpret_cast<double2*>(at<double>(A.lv[t].u, i));
                for (int q = tid; q < nn / 2; q += nt) g[q] = reinterpret_cast<const double2*>(su)[q];
            }
        } else {
            const float *skx = S + L.oKx, *sky = S + L.oKy;
            float* sb = S + L.oB;
            float* U = S + P.oW;                                  // fixed cycles
            double* u64 = reinterpret_cast<double*>(S + P.oW);    // converged form
            float* interp = CONV ? su : U;  // converged form: held in u until r is formed, then widened into u64
            interpolate<float, NC, false>(C, S + C.oU, interp);
            {
                const float ih2 = static_cast<float>(n) * static_cast<float>(n);  // exact
                for (int p = tid; p < nn; p += nt) {
                    int y, x;
                    split<NC>(L, false, p, y, x);
                    const float* kr = skx + y * XP;
                    const float kv[4] = {kr[x], kr[x + 1], sky[p], sky[p + n]};
                    const float uv[4] = {x > 0 ? interp[p - 1] : 0.0f, x < n - 1 ? interp[p + 1] : 0.0f,
                                         y > 0 ? interp[p - n] : 0.0f, y < n - 1 ? interp[p + n] : 0.0f};
                    sb[p] = resid_f32x2(kv, interp[p], uv, ih2);
                }
            }
            __syncthreads();
            if constexpr (CONV) {
                for (int p = tid; p < nn; p += nt) u64[p] = widen(interp[p]);
                __syncthreads();
            }
            for (int m = 0; m < A.mu0; ++m) vcycle<float, NC, BIG>(P, S, t, A.nu1, A.nu2, m == 0, false);
            if constexpr (CONV) {
                for (int p = tid; p < nn; p += nt) u64[p] += widen(su[p]);
                __syncthreads();
                const double ih2 = static_cast<double>(n) * n;
                for (int it = 0;; ++it) {
                    double acc = 0.0;
                    for (int p = tid; p < nn; p += nt) {
                        int y, x;
                        split<NC>(L, false, p, y, x);
                        const double r = fma(-ih2, apply_h2_64<float>(skx, sky, u64, n, x, y), 1.0);
                        sb[p] = narrow(r);
                        acc += r * r;
                    }
                    const double nr = sqrt(cta_sum<true>(acc, red));
                    const bool more = nr > G.thresh * n;  // the same value in every thread
                    if (tid == 0 && it > 0) atomicMax(G.iters + t, it);
                    if (!more) break;
                    if (it >= G.max_iter) {
                        if (tid == 0) atomicOr(A.status, kStatusNotConverged);
                        break;
                    }
                    for (int m = 0; m < A.mu0; ++m) vcycle<float, NC, BIG>(P, S, t, A.nu1, A.nu2, m == 0, false);
                    for (int p = tid; p < nn; p += nt) u64[p] += widen(su[p]);
                    __syncthreads();
                }
                double acc = 0.0;
                for (int p = tid; p < nn; p += nt) {
                    su[p] = narrow(u64[p]);
                    if (A.qoi == MLQMC_QOI_MEAN) acc += u64[p];
                    if (G.keep) at<double>(A.lv[t].u64, i)[p] = u64[p];
                }
                if (A.qoi == MLQMC_QOI_MEAN) {
                    F = mean_of(cta_sum<false>(acc, red));
                } else {
                    const int m = n / 2;
                    F = 0.25 * (u64[(m - 1) * n + (m - 1)] + u64[(m - 1) * n + m] + u64[m * n + (m - 1)] + u64[m * n + m]);
                    __syncthreads();
                }
            } else {
                // u = U + e exactly as the pair (h, l); h is the FP32 copy the next stage interpolates
                const int m = n / 2;
                const bool mean = A.qoi == MLQMC_QOI_MEAN;
                TripleSum ts;
                double c4 = 0.0;
                for (int p = tid; p < nn; p += nt) {
                    float h, l;
                    two_sum32(U[p], su[p], h, l);
                    su[p] = h;
                    if (mean) ts.add(h, l);
                    if (G.keep || !mean) {
                        const double v = widen(h) + widen(l);
                        if (G.keep) at<double>(A.lv[t].u64, i)[p] = v;
                        if (!mean) {
                            int y, x;
                            split<NC>(L, false, p, y, x);
                            if ((y == m || y == m - 1) && (x == m || x == m - 1)) c4 += v;
                        }
                    }
                }
                F = mean ? mean_of(cta_sum<false>(ts.value(), red)) : 0.25 * cta_sum<false>(c4, red);
            }
            if (t == P.top) {
                float4* g = reinterpret_cast<float4*>(at<float>(A.lv[t].u, i));
                for (int q = tid; q < nn / 4; q += nt) g[q] = reinterpret_cast<const float4*>(su)[q];
            }
        }
        if (tid == 0) A.F[static_cast<size_t>(i) * A.n_levels + t] = F;
        // su stays the level's solution until the next stage has interpolated it
    }
}

// Whether the kernels have a form with blocks of 4 x 4 cells (64 cells per side).
template <typename T, int NC>
constexpr bool kHasBig = sizeof(T) == 4 && !kPlain<NC>;

template <typename T, int NC, bool BIG>
bool attrs(int bytes)
{
    bool good = cudaFuncSetAttribute(kb_small_vcycle<T, NC, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
                cudaFuncSetAttribute(kb_small_stages<T, NC, false, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    if constexpr (sizeof(T) == 4)
        good = good && cudaFuncSetAttribute(kb_small_stages<T, NC, true, BIG>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    return good;
}

constexpr int kMaxSmem = 226 * 1024;  // and 1 KB of sums

template <typename T, int NC>
bool prepare_n0()
{
    if constexpr (kHasBig<T, NC>)
        if (!attrs<T, NC, true>(kMaxSmem)) return false;
    return attrs<T, NC, false>(kMaxSmem);
}

template <typename T>
bool prepare_all()
{
    return prepare_n0<T, 4>() && prepare_n0<T, 6>() && prepare_n0<T, 8>() && prepare_n0<T, 10>();
}

// f(NC, BIG) with both as compile-time constants.
template <typename T, typename Launch>
bool by_n0(int n0, bool big, Launch f)
{
    auto go = [&](auto nc) {
        if constexpr (kHasBig<T, decltype(nc)::value>) {
            if (big) {
                f(nc, std::true_type());
                return;
            }
        }
        f(nc, std::false_type());
    };
    switch (n0) {
    case 4: go(std::integral_constant<int, 4>()); break;
    case 6: go(std::integral_constant<int, 6>()); break;
    case 8: go(std::integral_constant<int, 8>()); break;
    case 10: go(std::integral_constant<int, 10>()); break;
    default: return false;
    }
    return cudaGetLastError() == cudaSuccess;
}

template <typename T>
bool vcycle_launch(const FmgArgs& A, const Plan& P, int B, cudaStream_t st)
{
    if (B <= 0) return true;
    return by_n0<T>(A.n0, P.lv[P.top].n == 64, [&](auto nc, auto big) {
        kb_small_vcycle<T, decltype(nc)::value, decltype(big)::value><<<B, P.threads, P.bytes, st>>>(A, P, B);
    });
}

template <typename T, bool CONV>
bool stages_launch(const FmgArgs& A, const Plan& P, const Stages& S, int count, cudaStream_t st)
{
    if (count <= 0) return true;
    return by_n0<T>(A.n0, P.lv[P.top].n == 64, [&](auto nc, auto big) {
        kb_small_stages<T, decltype(nc)::value, CONV, decltype(big)::value><<<count, P.threads, P.bytes, st>>>(A, P, S);
    });
}

}  // namespace
}  // namespace mlqmc_small
