// Level 0 of the FMG: the band matrix and the FP64 factorisation and exact
// solve on several lanes per sample.
#pragma once

#include "fmg_device.cuh"

namespace mlqmc_dev {

template <typename T>
__device__ __forceinline__ T band_a(const T* kx, const T* ky, int n0, int r, int l)
{
    const int r1 = r % n0, r2 = r / n0;
    if (l == 1 && r1 > 0) return -kx[r2 * kx_pitch(n0) + r1];
    if (l == n0) return -ky[r2 * n0 + r1];
    return T(0);
}

// Diagonal of row j of h0^2 A_0: the sum of the cell's four faces.
template <typename T>
__device__ __forceinline__ double level0_diag(const T* kx, const T* ky, int n0, int j)
{
    const int j1 = j % n0, j2 = j / n0;
    return widen(kx[j2 * kx_pitch(n0) + j1]) + widen(kx[j2 * kx_pitch(n0) + j1 + 1]) + widen(ky[j2 * n0 + j1]) +
           widen(ky[(j2 + 1) * n0 + j1]);
}

// Level 0 for n0 = NC on several lanes per sample (LPR lanes for each of the
// NC rows of the working window, NC LPR lanes in all). On GB300 an FP64 warp
// instruction holds its SM sub-partition for about 70 cycles whatever its
// active lanes, so what a sample costs is its FP64 warp instructions, and one
// thread's ~4,700 of them take 0.2 ms however few samples a call has. Here
// column j updates the whole trailing window at once (right-looking): lane
// (p, g) keeps row r = p mod NC and its columns c = g mod LPR in registers
// (register c mod NC), the diagonal and the right-hand side ride along, and a
// column costs its reciprocal square root (5), one scaling and NC/LPR + 1 (or
// + 3, LPR = 1) updates. Registers whose column is already eliminated take
// part with stale values and are reset when their row is replaced; the
// finished column goes to shared memory (backward substitution, pushed the
// same way) and to the global factor. Sums take their oldest term first, as
// in kb_level0_fixed: the same bits.
template <int NC, int LPR>
struct L0Geom {
    static constexpr int TL = NC * LPR;      // lanes that work on a sample
    static constexpr int SEG = TL <= 4 ? 4 : (TL <= 8 ? 8 : (TL <= 16 ? 16 : 32));  // lanes that a sample occupies
    static constexpr int SPW = 32 / SEG;     // samples per warp
    static constexpr int N = NC * NC;
    static constexpr int oL = 0;             // column j of L below the diagonal: [j * NC + row mod NC]
    static constexpr int oR = oL + N * NC;   // 1 / L(j, j)
    static constexpr int oY = oR + N;        // forward values, then the solution
    static constexpr int oD = oY + N;        // diagonal sums of h0^2 A_0
    static constexpr int oA = oD + N;        // -L.kx: coupling of row r to r - 1, then of row r to r - NC
    static constexpr int per = oA + 2 * N;   // doubles per sample
    static constexpr size_t bytes = sizeof(double) * per * SPW;
};

// Called by a whole warp; `base`: its first sample, `only`: bits of the warp's
// samples to store (the others take part and leave nothing behind).
template <typename T, bool MX, int NC, int LPR>
__device__ void level0_warp(const FmgArgs& A, int B, int base, unsigned only)
{
    using Gm = L0Geom<NC, LPR>;
    constexpr int N = NC * NC, W = NC + 1, KR = (NC + LPR - 1) / LPR;
    static_assert(LPR == 1 || LPR == 4, "the diagonal and the right-hand side take two groups, the column a third");
    extern __shared__ double l0sh[];
    const int lane = threadIdx.x, team = lane / Gm::SEG, tl = lane - team * Gm::SEG;
    const int i = base + team;
    const bool live = i < B && ((only >> team) & 1u);
    const int si = i < B ? i : B - 1;  // lanes past B compute on sample B-1 and store nothing
    const bool work = tl < Gm::TL;    // NC = 6: lanes past the window stay idle but converged
    const int p = work ? tl / LPR : 0, g = work ? tl - p * LPR : 0;
    const int t0 = team * Gm::SEG;
    double* S = l0sh + static_cast<size_t>(team) * Gm::per;
    const size_t cs = A.chol.stride;
    double* fac = reinterpret_cast<double*>(A.chol.base);
    float* f32 = reinterpret_cast<float*>(A.chol32);
    const double h2 = 1.0 / (static_cast<double>(NC) * NC);
    const Lv<T> L0 = view<T>(A, 0, si);
    for (int r = tl; r < N; r += Gm::SEG) {
        S[Gm::oD + r] = level0_diag(L0.kx, L0.ky, NC, r);
        S[Gm::oA + 2 * r] = widen(band_a(L0.kx, L0.ky, NC, r, 1));
        S[Gm::oA + 2 * r + 1] = r >= NC ? widen(band_a(L0.kx, L0.ky, NC, r, NC)) : 0.0;
    }
    __syncwarp();
    // LPR = 4: group (p + 2) mod 4 of row slot p holds its diagonal, group (p + 1) mod 4 its
    // right-hand side: never the group of the column being eliminated when the slot is the pivot
    const int gd = LPR == 1 ? 0 : (p + 2) % LPR;
    double off[KR];  // column c of the lane's row, c mod NC = g + LPR k
    double X, V = 0.0;  // diagonal or right-hand side (LPR = 1: diagonal and right-hand side)
    auto reset = [&](int r) {  // row r enters the window
        const bool in = r < N;
        const int rr = in ? r : 0;
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            const int cm = g + LPR * k;
            double a = 0.0;
            if (cm == (r + NC - 1) % NC) a = S[Gm::oA + 2 * rr];
            if (cm == r % NC) a = S[Gm::oA + 2 * rr + 1];
            off[k] = in ? a : 0.0;
        }
        const double d = S[Gm::oD + rr];
        if constexpr (LPR == 1) {
            X = d;
            V = h2;
        } else {
            X = g == gd ? d : h2;
        }
    };
    reset(p);
    for (int j0 = 0; j0 < N; j0 += NC) {
#pragma unroll
        for (int sj = 0; sj < NC; ++sj) {
            const int j = j0 + sj;
            constexpr int L1 = LPR - 1;
            const int gc = sj & L1, kc = sj / LPR;        // group and register of the column being eliminated
            const int ld = LPR == 1 ? 0 : (sj + 2) % LPR, lv = LPR == 1 ? 0 : (sj + 1) % LPR;
            const double d = __shfl_sync(0xffffffffu, X, t0 + sj * LPR + ld);
            const double rl = rsqrt64(d);
            double yj;
            double Lm;
            if constexpr (LPR == 1) {
                const double vj = __shfl_sync(0xffffffffu, V, t0 + sj);
                if (p == sj) reset(j + NC);
                Lm = off[kc] * rl;
                yj = vj * rl;
            } else {
                const double xo = X;
                if (p == sj) reset(j + NC);
                Lm = ((p == sj && g == lv) ? xo : off[kc]) * rl;  // one multiplication: column j and y_j
                yj = __shfl_sync(0xffffffffu, Lm, t0 + sj * LPR + lv);
            }
            const double Lr = LPR == 1 ? Lm : __shfl_sync(0xffffffffu, Lm, t0 + p * LPR + gc);
#pragma unroll
            for (int k = 0; k < KR; ++k) {
                const int cm = g + LPR * k;  // row slot of column c
                if (LPR == 1 && cm == sj) continue;
                const double Lc = __shfl_sync(0xffffffffu, Lm, t0 + (cm < NC ? cm : 0) * LPR + gc);
                if (cm != sj) off[k] = fma(-Lr, Lc, off[k]);
            }
            if constexpr (LPR == 1) {
                X = fma(-Lr, Lr, X);
                V = fma(-Lr, yj, V);
            } else {
                X = fma(-Lr, g == gd ? Lr : yj, X);
            }
            if (work && g == gc) S[Gm::oL + j * NC + p] = Lr;
            if (tl == 0) {
                S[Gm::oR + j] = rl;
                S[Gm::oY + j] = yj;
            }
        }
    }
    __syncwarp();
    // the factor to global memory in one pass (inside the loop its address
    // arithmetic and, mixed forms, the rounding to FP32 sat on the critical path)
    if (live) {
        auto put = [&](int q, double v) {
            if constexpr (MX) f32[static_cast<size_t>(q) * cs + i] = narrow(v);
            else fac[static_cast<size_t>(q) * cs + i] = v;
        };
        for (int q = tl; q < N * NC; q += Gm::SEG) {  // column j, row slot q mod NC: row j + l
            const int j = q / NC, l = (q - j * NC + NC - j % NC) % NC;
            const int lr = l ? l : NC;
            if (j + lr < N) put((j + lr) * W + lr, S[Gm::oL + q]);
        }
        for (int j = tl; j < N; j += Gm::SEG) put(j * W, S[Gm::oR + j]);
    }
    __syncwarp();
    // backward substitution: lane p < NC (LPR lanes of a slot alike) keeps the
    // pending value of the row of slot p; row r's solution updates rows r-1..r-NC
    double v = S[Gm::oY + N - NC + p];
    for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
        for (int sr = NC - 1; sr >= 0; --sr) {
            const int r = r0 + sr;
            const int c = p < sr ? r0 + p : r0 + p - NC;  // the slot's row below r (slot sr: row r - NC enters)
            const double Lc = c >= 0 ? S[Gm::oL + c * NC + sr] : 0.0;
            const double xr = __shfl_sync(0xffffffffu, v, t0 + sr * LPR) * S[Gm::oR + r];
            if (p == sr) v = c >= 0 ? S[Gm::oY + c] : 0.0;
            v = fma(-Lc, xr, v);
            if (tl == 0) S[Gm::oY + r] = xr;
        }
    }
    __syncwarp();
    double* x = (MX || A.refine) ? L0.u64 : reinterpret_cast<double*>(L0.u);
    if (live)
        for (int r = tl; r < N; r += Gm::SEG) {
            x[r] = S[Gm::oY + r];
            if constexpr (MX) reinterpret_cast<float*>(L0.u)[r] = narrow(S[Gm::oY + r]);  // FP32 copy for the first FMG interpolation
        }
    double F0;
    if (A.qoi == MLQMC_QOI_MEAN) {
        constexpr int Q = Gm::SEG >= 16 ? 1 : 16 / Gm::SEG;  // partial sums per lane: c = tl + SEG q
        double s[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int c = (tl & 15) + Gm::SEG * q;
            s[q] = S[Gm::oY + c];
            for (int r = 16 + c; r < N; r += 16) s[q] += S[Gm::oY + r];
        }
#pragma unroll
        for (int w = Q / 2; w > 0; w >>= 1)
#pragma unroll
            for (int q = 0; q < w; ++q) s[q] += s[q + w];
        double acc = s[0];
#pragma unroll
        for (int w = Gm::SEG >= 16 ? 8 : Gm::SEG / 2; w > 0; w >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
        F0 = acc / static_cast<double>(N);
    } else {
        constexpr int m = NC / 2;
        const double* y = S + Gm::oY;
        F0 = 0.25 * (y[(m - 1) * NC + (m - 1)] + y[(m - 1) * NC + m] + y[m * NC + (m - 1)] + y[m * NC + m]);
    }
    if (live && tl == 0) A.F[static_cast<size_t>(i) * A.n_levels] = F0;
}

}  // namespace mlqmc_dev
