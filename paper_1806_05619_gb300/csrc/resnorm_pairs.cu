// Refinement residual r = 1 - A u64 of a level and the sums of r^2 behind its
// norm (mixed forms refined to a tolerance).
//
// In FP64 a cell's residual is nine operations and four widened faces, with
// r^2 about thirteen slots of a pipe that takes one warp instruction in 64
// cycles: 1.6 ms for 64 samples of 1024 x 1024, whose 20 bytes per cell move
// in 0.2 ms. Only the differences u_P - u_Q need FP64 (u64 has all 53 bits, and
// neighbours cancel to its last ones); a difference is then a pair of FP32
// numbers to 2^-49 of itself, and fluxes, their sum, the residual and its square
// are FP32 error-free pairs (as resid_f32x2 does for FP32 iterates). Each
// difference belongs to a face and is formed once: a warp takes 128 columns,
// four cells per lane, and walks down eight rows with the fluxes of the row
// above in registers and the west fluxes of the next lane by shuffles, 2.4 FP64
// operations per cell in place of thirteen. Four samples x 16 shifts on 1024 x
// 1024 refined to 1e-10 (the step's 66 such passes on 128 x 128 and above): 45.5
// -> 29.5 ms for the step, 85 us per pass; one 256 x 256 sample 2.2 -> 2.0 ms,
// Algorithm 1 on seven levels 4.0 -> 3.4 ms. Now bounded by
// latency: on 64 samples of 512 x 512 the FP64 pipe is 53 % and the issue slots 45 %
// busy, DRAM 30 %, with 16 warps of 128 registers per SM.
//
// Error: a flux k d is off by at most 2^-47 |k d|; d is a difference of
// neighbours, u/d is at least n/8 for these solutions, so on the levels the
// kernel takes this stays below what u64's own rounding (2^-53 u) puts into
// the residual. Values outside FP32's comfortable range (a difference below
// 2^-74 or beyond 2^127, a residual above 1e15 or not finite) take FP64.
#include "resnorm_pairs.h"

#include <algorithm>
#include <cstdint>

using namespace mlqmc_dev;

namespace {

constexpr int kCols = 128, kWarps = 8;  // a warp's strip is kCols wide; a CTA stacks kWarps of them
constexpr uint32_t kAll = 0xffffffffu;

struct Pair {
    float h, l;
};

static __device__ __noinline__ Pair split_rare(double d)
{
    Pair p;
    p.h = __double2float_rn(d);
    p.l = fabsf(p.h) <= 3.0e38f ? __double2float_rn(d - static_cast<double>(p.h)) : 0.0f;
    return p;
}

// d = h + l: the 29 significand bits FP32 has no room for are rounded off h
// (half up) and make up l, exact but for l's own rounding (2^-49 |d|); bit
// operations only. Biased exponents 949..1150, where both parts are normal;
// anything else but zero takes the conversions.
__device__ __forceinline__ Pair split(double d)
{
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(d)), lo = static_cast<uint32_t>(__double2loint(d));
    const uint32_t e = (hi >> 20) & 0x7FFu;
    Pair p;
    if (e - 949u > 201u) {
        if (((hi << 1) | lo) == 0u) {
            p.h = p.l = 0.0f;
            return p;
        }
        return split_rare(d);
    }
    const uint32_t sgn = hi & 0x80000000u;
    const uint64_t m = ((static_cast<uint64_t>(hi) << 32) | lo) + 0x10000000ull;
    const uint32_t mag = __funnelshift_r(static_cast<uint32_t>(m), static_cast<uint32_t>(m >> 32), 29) - 0xC0000000u;
    p.h = __uint_as_float((mag & 0x7FFFFFFFu) | sgn);
    const int low = static_cast<int>(static_cast<uint32_t>(m) & 0x1FFFFFFFu) - 0x10000000;
    p.l = __uint_as_float(__float_as_uint(static_cast<float>(low) * __uint_as_float((e - 948u) << 23)) ^ sgn);
    return p;
}

// k (a - b) as a pair.
__device__ __forceinline__ Pair flux(float k, double a, double b)
{
    const Pair d = split(a - b);
    Pair f;
    f.h = __fmul_rn(k, d.h);
    f.l = __fmaf_rn(k, d.l, __fmaf_rn(k, d.h, -f.h));
    return f;
}

static __device__ __noinline__ double resid_rare(const FmgArgs* A, int t, int i, int i1, int i2)
{
    const Lv<float> L = view<float>(*A, t, i);
    return resid64_cell(L, static_cast<double>(L.n) * L.n, i1, i2);
}

struct Row {
    double u[4];
    float4 kx, ky;  // west faces of the row's cells; faces between it and the row above
};

__device__ __forceinline__ void load_u(const double* u, bool in, double (&v)[4])
{
    double2 a = make_double2(0.0, 0.0), b = a;
    if (in) {
        a = *reinterpret_cast<const double2*>(u);
        b = *reinterpret_cast<const double2*>(u + 2);
    }
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

__device__ __forceinline__ float4 load_f(const float* p, bool in)
{
    return in ? *reinterpret_cast<const float4*>(p) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// ROWS: rows of a warp's strip. Eight form the fluxes between strips once in
// eight rows; two keep the chain of a small level short (one 256 x 256 sample:
// 13.8 -> 6.2 us).
template <int ROWS>
__global__ void __launch_bounds__(32 * kWarps, 2) kb_resnorm_pairs(const __grid_constant__ FmgArgs A, int t, int B,
                                                                   int PX, int P, double* __restrict__ part,
                                                                   const int* __restrict__ active)
{
    __shared__ double red[48];
    const int n = A.lv[t].n, pitch = kx_pitch(n);
    const float c = static_cast<float>(n) * static_cast<float>(n);  // exact: n = coarse_cells 2^t
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int w = blockIdx.x; w < B * P; w += gridDim.x) {  // uniform per CTA: every thread reaches block_sum
        const int i = w / P, q = w - i * P;
        if (active && !active[i]) continue;
        const int x = (q % PX) * kCols + 4 * lane, y0 = ((q / PX) * kWarps + warp) * ROWS;
        const int y1 = min(y0 + ROWS, n);
        const bool in = x < n;                                // x and n multiples of 4: all four cells or none
        const bool east = in && (lane == 31 || x + 4 >= n);   // the strip's last cell owns its east face too
        const double* u = at<double>(A.lv[t].u64, i) + x;
        const float* kx = at<float>(A.lv[t].kx, i) + x;
        const float* ky = at<float>(A.lv[t].ky, i) + x;
        float* bc = at<float>(A.lv[t].bc, i) + x;
        PairSum ps;
        double wide = 0.0;
        if (y0 < y1) {
            Row cur, nxt;
            Pair south[4];  // fluxes of the faces below the row
            {
                double below[4];
                load_u(u + static_cast<ptrdiff_t>(y0 - 1) * n, in && y0 > 0, below);
                load_u(u + static_cast<ptrdiff_t>(y0) * n, in, cur.u);
                const float4 k0 = load_f(ky + static_cast<ptrdiff_t>(y0) * n, in);
                cur.kx = load_f(kx + static_cast<ptrdiff_t>(y0) * pitch, in);
                south[0] = flux(k0.x, cur.u[0], below[0]);
                south[1] = flux(k0.y, cur.u[1], below[1]);
                south[2] = flux(k0.z, cur.u[2], below[2]);
                south[3] = flux(k0.w, cur.u[3], below[3]);
            }
            load_u(u + static_cast<ptrdiff_t>(y0 + 1) * n, in && y0 + 1 < n, nxt.u);
            cur.ky = load_f(ky + static_cast<ptrdiff_t>(y0 + 1) * n, in);
#pragma unroll 2
            for (int y = y0; y < y1; ++y) {
                // the strip's edge values, and the next row ahead of its use
                double uw = 0.0, ue = 0.0;
                float ke = 0.0f;
                if (lane == 0 && x > 0) uw = u[static_cast<ptrdiff_t>(y) * n - 1];
                if (east) {
                    ke = kx[static_cast<ptrdiff_t>(y) * pitch + 4];
                    if (x + 4 < n) ue = u[static_cast<ptrdiff_t>(y) * n + 4];
                }
                double ahead[4];
                const bool more = y + 1 < y1;
                load_u(u + static_cast<ptrdiff_t>(y + 2) * n, in && more && y + 2 < n, ahead);
                nxt.ky = load_f(ky + static_cast<ptrdiff_t>(y + 2) * n, in && more);
                nxt.kx = load_f(kx + static_cast<ptrdiff_t>(y + 1) * pitch, in && more);

                const double ul = __shfl_up_sync(kAll, cur.u[3], 1);
                Pair fx[5];
                fx[0] = flux(cur.kx.x, cur.u[0], lane == 0 ? uw : ul);
                fx[1] = flux(cur.kx.y, cur.u[1], cur.u[0]);
                fx[2] = flux(cur.kx.z, cur.u[2], cur.u[1]);
                fx[3] = flux(cur.kx.w, cur.u[3], cur.u[2]);
                fx[4].h = __shfl_down_sync(kAll, fx[0].h, 1);
                fx[4].l = __shfl_down_sync(kAll, fx[0].l, 1);
                if (east) fx[4] = flux(ke, ue, cur.u[3]);
                const float kn[4] = {cur.ky.x, cur.ky.y, cur.ky.z, cur.ky.w};
                float r[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const Pair north = flux(kn[j], nxt.u[j], cur.u[j]);
                    // sum of the four outward differences, Sum2
                    float sh, sl, e;
                    two_sum32(fx[j].h, -fx[j + 1].h, sh, e);
                    sl = __fadd_rn(__fsub_rn(fx[j].l, fx[j + 1].l), e);
                    two_sum32(sh, south[j].h, sh, e);
                    sl = __fadd_rn(sl, __fadd_rn(e, south[j].l));
                    two_sum32(sh, -north.h, sh, e);
                    sl = __fadd_rn(sl, __fsub_rn(e, north.l));
                    south[j] = north;
                    // r = 1 - c s
                    const float ah = __fmul_rn(c, sh);
                    const float al = __fmaf_rn(c, sl, __fmaf_rn(c, sh, -ah));
                    float rh, re, b, rem;
                    two_sum32(1.0f, -ah, rh, re);
                    two_sum32(rh, __fsub_rn(re, al), b, rem);
                    if (!(fabsf(b) <= 1.0e15f) && in) {
                        const double v = resid_rare(&A, t, i, x + j, y);
                        b = narrow(v);
                        wide += v * v;
                    } else {
                        const float sq = __fmul_rn(b, b);
                        ps.add(sq, __fmaf_rn(2.0f * b, rem, __fmaf_rn(b, b, -sq)));
                    }
                    r[j] = b;
                }
                if (in) *reinterpret_cast<float4*>(bc + static_cast<ptrdiff_t>(y) * n) = make_float4(r[0], r[1], r[2], r[3]);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    cur.u[j] = nxt.u[j];
                    nxt.u[j] = ahead[j];
                }
                cur.kx = nxt.kx;
                cur.ky = nxt.ky;
            }
        }
        const double sum = block_sum(in ? ps.value() + wide : 0.0, red);
        if (threadIdx.x == 0) part[w] = sum;
    }
}

}  // namespace

namespace mlqmc_resnorm {

bool launch(const FmgArgs& A, int t, int n, int B, double* part, const int* active, int sm_count, cudaStream_t st)
{
    const int PX = (n + kCols - 1) / kCols, P = chunks(n);
    static_assert(kWarps == 8 && kCols == 128, "chunks()");
    const int grid = static_cast<int>(std::min<int64_t>(static_cast<int64_t>(B) * P, static_cast<int64_t>(sm_count) * 16));
    if (rows(n) == 2) kb_resnorm_pairs<2><<<grid, 32 * kWarps, 0, st>>>(A, t, B, PX, P, part, active);
    else kb_resnorm_pairs<8><<<grid, 32 * kWarps, 0, st>>>(A, t, B, PX, P, part, active);
    return cudaGetLastError() == cudaSuccess;
}

}  // namespace mlqmc_resnorm
