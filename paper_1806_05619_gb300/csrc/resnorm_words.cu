// Refinement residual r = 1 - A u64 of a level and the sums of r^2 behind its
// norm (mixed forms refined to a tolerance).
//
// In FP64 a cell's residual is nine operations and four widened faces, with
// r^2 about thirteen slots of a pipe that takes one warp instruction in 64
// cycles: 1.6 ms for 64 samples of 1024 x 1024, whose 20 bytes per cell move
// in 0.2 ms. Here only the differences u_P - u_Q are formed in FP64; their
// products with the faces, the sum over the faces, the scaling and the residual
// run in three FP32 words per number (flux_words.h), with no more error than the
// FP64 form: below 2^-62 of the fluxes beyond the differences' own rounding.
// (Two words left 2^-47 of them: the norm at the FP64 solution rose by a half on
// 32 x 32 and by a twentieth on 128 x 128, and a tolerance near it was missed.)
// Four samples x 16 shifts on 1024 x 1024 refined to 1e-10: 45.5 ms for the step
// with the FP64 form, 29.4 with two words, 30.7 with three.
// Each difference belongs to a face and is formed once: a warp takes 128
// columns, four cells per lane, and walks down its rows with the fluxes of the
// row above in registers and the west fluxes of the next lane by shuffles, 2.4
// FP64 operations per cell in place of thirteen.
//
// Values outside FP32's comfortable range take other routes: a difference below
// 2^-74 or from 2^128 on the conversion instructions, a residual above 1e15 or
// not finite FP64.
#include "resnorm_words.h"

#include <algorithm>
#include <cstdint>

#include "flux_words.h"

using namespace mlqmc_dev;
using mlqmc_words::flux;
using mlqmc_words::Words;

namespace {

constexpr int kCols = 128, kWarps = 8;  // a warp's strip is kCols wide; a CTA stacks kWarps of them
constexpr uint32_t kAll = 0xffffffffu;

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
__global__ void __launch_bounds__(32 * kWarps, 2) kb_resnorm_words(const __grid_constant__ FmgArgs A, int t, int B,
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
            Words south[4];  // fluxes of the faces below the row
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
                // the fluxes of the cell's west and east faces; the last cell's east one is the next lane's first
                const Words first = flux(cur.kx.x, cur.u[0], lane == 0 ? uw : ul);
                Words last;
                last.h = __shfl_down_sync(kAll, first.h, 1);
                last.m = __shfl_down_sync(kAll, first.m, 1);
                last.l = __shfl_down_sync(kAll, first.l, 1);
                if (east) last = flux(ke, ue, cur.u[3]);
                const float kn[4] = {cur.ky.x, cur.ky.y, cur.ky.z, cur.ky.w}, ki[3] = {cur.kx.y, cur.kx.z, cur.kx.w};
                Words west = first;
                float r[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const Words e = j < 3 ? flux(ki[j < 3 ? j : 0], cur.u[j < 3 ? j + 1 : 3], cur.u[j]) : last;
                    const Words north = flux(kn[j], nxt.u[j], cur.u[j]);
                    float b, rem;
                    mlqmc_words::residual(c, west, e, south[j], north, b, rem);
                    west = e;
                    south[j] = north;
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
    if (rows(n) == 2) kb_resnorm_words<2><<<grid, 32 * kWarps, 0, st>>>(A, t, B, PX, P, part, active);
    else kb_resnorm_words<8><<<grid, 32 * kWarps, 0, st>>>(A, t, B, PX, P, part, active);
    return cudaGetLastError() == cudaSuccess;
}

}  // namespace mlqmc_resnorm
