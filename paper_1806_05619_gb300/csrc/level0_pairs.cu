// Level 0 of the mixed forms: band Cholesky factor of h0^2 A_0 (kept in FP32
// for the V-cycles), exact FP64 solve with f = 1 and F_0, on several lanes per
// sample.
//
// In FP64 a column of the factorisation is nine or more warp instructions that
// each hold the sub-partition's pipe for about 70 cycles: at n0 = 8 40 us for one
// sample, 202 for 8,064, 556 for 32,256, and Algorithm 1's rounds wait for it (26,
// 115 and 390 us so). Here the factor, the
// forward and the backward substitution run in FP32 pairs (hi + lo, products and
// sums by error-free transformations, 2^-46 per operation): about 85 FP32
// instructions per column of 4 cycles each. Then r = h^2 - A x in FP64 and the
// correction A e = r with the pairs' leading parts, x += e, until e is below
// 2^-37 of the largest x. A correction leaves at most about 2^-24 times the
// condition number of the error before it, so the end of the steps is 2^-61 times
// the condition number away in the maximum norm, where an FP64 factor leaves 2^-53
// times; against 60-digit solutions (n0 = 4 and 8, independent cells with standard
// deviations of the exponent up to 12) the errors were those of the FP64 factor or
// smaller in the maximum norm, and as large as its own in the smallest components. The
// faces are FP32 numbers, so the matrix itself is exact in both. A sample whose
// corrections do not get there in four steps (a condition number near 2^24 and
// more, as of an island of high coefficient within a low one, or coefficients
// beyond what FP32's exponents hold beside each other) is redone in FP64.
#include "level0_pairs.h"

#include <algorithm>
#include <cstdint>

#include "level0_lanes.cuh"

using namespace mlqmc_dev;

namespace {

struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair mul(Pair a, Pair b)
{
    Pair p;
    p.h = __fmul_rn(a.h, b.h);
    p.l = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p.h)));
    return p;
}

// c - a b, normalised
__device__ __forceinline__ Pair fnma(Pair a, Pair b, Pair c)
{
    const Pair p = mul(a, b);
    float s, e;
    two_sum32(c.h, -p.h, s, e);
    e = __fadd_rn(e, __fsub_rn(c.l, p.l));
    Pair r;
    r.h = __fadd_rn(s, e);
    r.l = __fsub_rn(e, __fsub_rn(r.h, s));
    return r;
}

// 1/sqrt(d): the hardware's estimate y and one step of third order,
// y + y e (1/2 + 3/8 e) with e = 1 - d y^2 formed to 2^-47
__device__ __forceinline__ Pair rsqrt_pair(Pair d)
{
    const float y = rsqrtf(d.h);
    const float q = __fmul_rn(y, y), ql = __fmaf_rn(y, y, -q);
    const float p = __fmul_rn(d.h, q);
    const float pl = __fmaf_rn(d.l, q, __fmaf_rn(d.h, ql, __fmaf_rn(d.h, q, -p)));
    const float e = __fsub_rn(__fsub_rn(1.0f, p), pl);
    const float c = __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f));
    Pair r;
    r.h = __fadd_rn(y, c);
    r.l = __fsub_rn(c, __fsub_rn(r.h, y));
    return r;
}

__device__ __forceinline__ Pair shfl(Pair v, int src)
{
    return Pair{__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}

__device__ __forceinline__ Pair pair_of(double v)
{
    const float h = narrow(v);
    return Pair{h, narrow_rest(v, h)};
}

template <int NC, int LPR>
struct Geom {
    using FP64 = L0Geom<NC, LPR>;  // the same lanes
    static constexpr int N = NC * NC, SPW = FP64::SPW;
    static constexpr int oL = 0;             // pairs: column j of L below the diagonal, [j * NC + row mod NC]
    static constexpr int oR = oL + N * NC;   // 1 / L(j, j)
    static constexpr int oY = oR + N;        // forward values; the solution (double)
    static constexpr int oD = oY + N;        // diagonal of h0^2 A_0
    static constexpr int oA = oD + N;        // floats (a, b): coupling of row r to r - 1 and to r - NC
    static constexpr int oE = oA + N;        // floats: residual, forward values of the correction, correction
    static constexpr int per = oE + (N + 1) / 2;
    static constexpr size_t bytes = std::max(sizeof(Pair) * static_cast<size_t>(per) * SPW, FP64::bytes);
};

template <int NC, int LPR>
__global__ void __launch_bounds__(32) kb_level0_pairs(const __grid_constant__ FmgArgs A, int B)
{
    using G = Geom<NC, LPR>;
    using L0 = typename G::FP64;
    constexpr int N = NC * NC, W = NC + 1, KR = (NC + LPR - 1) / LPR, SEG = L0::SEG;
    extern __shared__ double l0sh[];
    const int lane = threadIdx.x, team = lane / SEG, tl = lane - team * SEG;
    const int i = blockIdx.x * G::SPW + team;
    const bool live = i < B;
    const int si = live ? i : B - 1;  // lanes past B compute on sample B-1 and store nothing
    const bool work = tl < L0::TL;    // NC = 6, 10: lanes past the window stay idle but converged
    const int p = work ? tl / LPR : 0, g = work ? tl - p * LPR : 0;
    const int t0 = team * SEG;
    Pair* S = reinterpret_cast<Pair*>(l0sh) + static_cast<size_t>(team) * G::per;
    float* Sa = reinterpret_cast<float*>(S + G::oA);
    float* Se = reinterpret_cast<float*>(S + G::oE);
    const size_t cs = A.chol.stride;
    float* f32 = reinterpret_cast<float*>(A.chol32);
    const double h2 = 1.0 / (static_cast<double>(NC) * NC);
    const Pair h2p = pair_of(h2), zero = {0.0f, 0.0f};
    const Lv<float> L = view<float>(A, 0, si);
    for (int r = tl; r < N; r += SEG) {
        S[G::oD + r] = pair_of(level0_diag(L.kx, L.ky, NC, r));
        Sa[2 * r] = band_a(L.kx, L.ky, NC, r, 1);
        Sa[2 * r + 1] = r >= NC ? band_a(L.kx, L.ky, NC, r, NC) : 0.0f;
    }
    __syncwarp();
    // the right-looking factorisation of level0_warp (its registers, groups and order), in pairs
    const int gd = LPR == 1 ? 0 : (p + 2) % LPR;
    Pair off[KR];
    Pair X, V = zero;
    auto reset = [&](int r) {  // row r enters the window
        const bool in = r < N;
        const int rr = in ? r : 0;
        const float a1 = Sa[2 * rr], an = Sa[2 * rr + 1];
#pragma unroll
        for (int k = 0; k < KR; ++k) {
            const int cm = g + LPR * k;
            float a = 0.0f;
            if (cm == (r + NC - 1) % NC) a = a1;
            if (cm == r % NC) a = an;
            off[k] = Pair{in ? a : 0.0f, 0.0f};
        }
        const Pair d = S[G::oD + rr];
        if constexpr (LPR == 1) {
            X = d;
            V = h2p;
        } else {
            X = g == gd ? d : h2p;
        }
    };
    reset(p);
    for (int j0 = 0; j0 < N; j0 += NC) {
#pragma unroll
        for (int sj = 0; sj < NC; ++sj) {
            const int j = j0 + sj;
            constexpr int L1 = LPR - 1;
            const int gc = sj & L1, kc = sj / LPR;
            const int ld = LPR == 1 ? 0 : (sj + 2) % LPR, lv = LPR == 1 ? 0 : (sj + 1) % LPR;
            const Pair rl = rsqrt_pair(shfl(X, t0 + sj * LPR + ld));
            Pair yj, Lm;
            if constexpr (LPR == 1) {
                const Pair vj = shfl(V, t0 + sj);
                if (p == sj) reset(j + NC);
                Lm = mul(off[kc], rl);
                yj = mul(vj, rl);
            } else {
                const Pair xo = X;
                if (p == sj) reset(j + NC);
                Lm = mul((p == sj && g == lv) ? xo : off[kc], rl);
                yj = shfl(Lm, t0 + sj * LPR + lv);
            }
            const Pair Lr = LPR == 1 ? Lm : shfl(Lm, t0 + p * LPR + gc);
#pragma unroll
            for (int k = 0; k < KR; ++k) {
                const int cm = g + LPR * k;
                if (LPR == 1 && cm == sj) continue;
                const Pair Lc = shfl(Lm, t0 + (cm < NC ? cm : 0) * LPR + gc);
                if (cm != sj) off[k] = fnma(Lr, Lc, off[k]);
            }
            if constexpr (LPR == 1) {
                X = fnma(Lr, Lr, X);
                V = fnma(Lr, yj, V);
            } else {
                X = fnma(Lr, g == gd ? Lr : yj, X);
            }
            if (work && g == gc) S[G::oL + j * NC + p] = Lr;
            if (tl == 0) {
                S[G::oR + j] = rl;
                S[G::oY + j] = yj;
            }
        }
    }
    __syncwarp();
    if (live) {  // the factor, FP32
        auto put = [&](int q, Pair v) { f32[static_cast<size_t>(q) * cs + i] = __fadd_rn(v.h, v.l); };
        for (int q = tl; q < N * NC; q += SEG) {  // column j, row slot q mod NC: row j + l
            const int j = q / NC, l = (q - j * NC + NC - j % NC) % NC;
            const int lr = l ? l : NC;
            if (j + lr < N) put((j + lr) * W + lr, S[G::oL + q]);
        }
        for (int j = tl; j < N; j += SEG) put(j * W, S[G::oR + j]);
    }
    {
        // backward substitution in pairs: slot p's lanes keep the pending value of its row
        Pair v = S[G::oY + N - NC + p];
        for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
            for (int sr = NC - 1; sr >= 0; --sr) {
                const int r = r0 + sr;
                const int c = p < sr ? r0 + p : r0 + p - NC;  // the slot's row below r (slot sr: row r - NC enters)
                const Pair Lc = c >= 0 ? S[G::oL + c * NC + sr] : zero;
                const Pair xr = mul(shfl(v, t0 + sr * LPR), S[G::oR + r]);
                if (p == sr) v = c >= 0 ? S[G::oY + c] : zero;
                v = fnma(Lc, xr, v);
                if (tl == 0) S[G::oY + r] = xr;
            }
        }
    }
    __syncwarp();
    double* x = reinterpret_cast<double*>(S + G::oY);
    for (int r = tl; r < N; r += SEG) {
        const Pair v = S[G::oY + r];
        x[r] = widen(v.h) + widen(v.l);
    }
    __syncwarp();
    // corrections until the next one would be below FP64's rounding
    bool done = false;
    for (int it = 0; it < 4; ++it) {
        for (int r = tl; r < N; r += SEG) {
            const Pair d = S[G::oD + r];
            double s = fma(-(widen(d.h) + widen(d.l)), x[r], h2);
            if (r >= 1) s = fma(-widen(Sa[2 * r]), x[r - 1], s);
            if (r >= NC) s = fma(-widen(Sa[2 * r + 1]), x[r - NC], s);
            if (r + 1 < N) s = fma(-widen(Sa[2 * r + 2]), x[r + 1], s);
            if (r + NC < N) s = fma(-widen(Sa[2 * (r + NC) + 1]), x[r + NC], s);
            Se[r] = narrow(s);
        }
        __syncwarp();
        float v = Se[p];
        for (int r0 = 0; r0 < N; r0 += NC) {
#pragma unroll
            for (int sr = 0; sr < NC; ++sr) {
                const int r = r0 + sr;
                const float e = __shfl_sync(0xffffffffu, v, t0 + sr * LPR) * S[G::oR + r].h;
                if (p == sr) v = r + NC < N ? Se[r + NC] : 0.0f;
                v = fmaf(-S[G::oL + r * NC + p].h, e, v);
                if (tl == 0) Se[r] = e;
            }
        }
        __syncwarp();
        v = Se[N - NC + p];
        for (int r0 = N - NC; r0 >= 0; r0 -= NC) {
#pragma unroll
            for (int sr = NC - 1; sr >= 0; --sr) {
                const int r = r0 + sr;
                const int c = p < sr ? r0 + p : r0 + p - NC;
                const float Lc = c >= 0 ? S[G::oL + c * NC + sr].h : 0.0f;
                const float e = __shfl_sync(0xffffffffu, v, t0 + sr * LPR) * S[G::oR + r].h;
                if (p == sr) v = c >= 0 ? Se[c] : 0.0f;
                v = fmaf(-Lc, e, v);
                if (tl == 0) Se[r] = e;
            }
        }
        __syncwarp();
        float em = 0.0f, xm = 0.0f;
        bool finite = true;
        for (int r = tl; r < N; r += SEG) {
            const float e = Se[r];
            if (!done) x[r] += widen(e);
            em = fmaxf(em, fabsf(e));
            finite = finite && e - e == 0.0f;  // fmaxf drops NaN
            xm = fmaxf(xm, fabsf(narrow(x[r])));
        }
#pragma unroll
        for (int o = SEG / 2; o > 0; o >>= 1) {
            em = fmaxf(em, __shfl_xor_sync(0xffffffffu, em, o));
            xm = fmaxf(xm, __shfl_xor_sync(0xffffffffu, xm, o));
        }
        constexpr unsigned kTeam = SEG == 32 ? 0xffffffffu : (1u << (SEG & 31)) - 1u;
        const bool all_finite = ((__ballot_sync(0xffffffffu, finite) >> t0) & kTeam) == kTeam;
        done = done || (all_finite && em <= 0x1p-37f * xm && xm <= 3.0e38f);
        __syncwarp();
        if (__all_sync(0xffffffffu, done)) break;
    }
    if (live && done) {
        for (int r = tl; r < N; r += SEG) {
            L.u64[r] = x[r];
            L.u[r] = narrow(x[r]);  // FP32 copy for the first FMG interpolation
        }
    }
    double F0;
    if (A.qoi == MLQMC_QOI_MEAN) {
        constexpr int Q = SEG >= 16 ? 1 : 16 / SEG;  // partial sums per lane: c = tl + SEG q
        double s[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int c = (tl & 15) + SEG * q;
            s[q] = x[c];
            for (int r = 16 + c; r < N; r += 16) s[q] += x[r];
        }
#pragma unroll
        for (int w = Q / 2; w > 0; w >>= 1)
#pragma unroll
            for (int q = 0; q < w; ++q) s[q] += s[q + w];
        double acc = s[0];
#pragma unroll
        for (int w = SEG >= 16 ? 8 : SEG / 2; w > 0; w >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
        F0 = acc / static_cast<double>(N);
    } else {
        constexpr int m = NC / 2;
        F0 = 0.25 * (x[(m - 1) * NC + (m - 1)] + x[(m - 1) * NC + m] + x[m * NC + (m - 1)] + x[m * NC + m]);
    }
    if (live && done && tl == 0) A.F[static_cast<size_t>(i) * A.n_levels] = F0;
    // samples left over: in FP64 (uniform per warp)
    const unsigned missing = __ballot_sync(0xffffffffu, live && !done && tl == 0);
    if (missing) {
        unsigned only = 0;
#pragma unroll
        for (int q = 0; q < G::SPW; ++q) only |= ((missing >> (q * SEG)) & 1u) << q;
        __syncwarp();
        level0_warp<float, true, NC, LPR>(A, B, blockIdx.x * G::SPW, only);
    }
}

// Calls with fewer samples take four lanes per window row, the shorter chain;
// one lane per row takes fewer instructions per sample. Microseconds of a call,
// four lanes / one: n0 = 8, 16 samples 26 / 45, 2,048: 42 / 48, 4,096: 66 / 57; n0 = 6,
// 16: 19 / 26, 2,048: 28 / 27, 4,096: 44 / 30; n0 = 4, 16: 8 / 14, 4,096: 11 / 14, 8,192: 20 / 16.
constexpr int four_lanes_below(int n0) { return n0 == 4 ? 6144 : n0 == 6 ? 2048 : 3072; }

template <int NC>
void go(const FmgArgs& A, int B, cudaStream_t st)
{
    if constexpr (4 * NC <= 32) {
        if (mlqmc_level0::four_lanes(NC, B)) {
            using G = Geom<NC, 4>;
            kb_level0_pairs<NC, 4><<<(B + G::SPW - 1) / G::SPW, 32, G::bytes, st>>>(A, B);
            return;
        }
    }
    using G = Geom<NC, 1>;
    kb_level0_pairs<NC, 1><<<(B + G::SPW - 1) / G::SPW, 32, G::bytes, st>>>(A, B);
}

}  // namespace

namespace mlqmc_level0 {

bool four_lanes(int n0, int B) { return 4 * n0 <= 32 && B < four_lanes_below(n0); }

bool launch(const FmgArgs& A, int n0, int B, cudaStream_t st)
{
    if (B <= 0 || !supported(n0)) return false;
    if (n0 == 4) go<4>(A, B, st);
    else if (n0 == 6) go<6>(A, B, st);
    else if (n0 == 8) go<8>(A, B, st);
    else go<10>(A, B, st);
    return cudaGetLastError() == cudaSuccess;
}

}  // namespace mlqmc_level0
