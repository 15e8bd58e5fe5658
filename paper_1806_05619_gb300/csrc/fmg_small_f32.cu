// Small-level FMG kernels of the mixed forms (fmg_small.cuh) and the
// shared-memory plan of both forms.
#include "fmg_small.cuh"

namespace mlqmc_small {

namespace {

bool power_of_two(int n) { return n > 0 && (n & (n - 1)) == 0; }

}  // namespace

Plan make_plan(int n0, int top, bool fp64, bool stages, bool conv)
{
    Plan P{};
    P.top = top;
    P.stored_d = (fp64 || !power_of_two(n0)) ? 1 : 0;
    const int es = fp64 ? 8 : 4;
    int o = 0;
    auto take = [&](int elems) {  // every part starts on a 16-byte boundary
        const int at = o;
        o += (elems + 3) / 4 * 4;
        return at;
    };
    for (int t = 0; t <= top; ++t) {
        Level& L = P.lv[t];
        L.n = n0 << t;
        for (L.lg = 0; (1 << L.lg) < L.n; ++L.lg) {
        }
        L.by_n = mlqmc_dev::FastDiv(static_cast<uint32_t>(L.n));
        L.by_nc = mlqmc_dev::FastDiv(static_cast<uint32_t>(L.n / 2));
        L.oU = take(L.n * L.n);
        L.oB = take(L.n * L.n);
        if (t == 0) continue;
        L.oKx = take(L.n * mlqmc_dev::kx_pitch(L.n));
        L.oKy = take((L.n + 1) * L.n);
        if (P.stored_d) L.oD = take(L.n * L.n);
    }
    P.oChol = take(2 * n0 * n0 * ((n0 + 1 + 3) / 4 * 4));  // CoarseGeom<n0>::elems
    const int nt = P.lv[top].n;
    if (stages && !fp64) P.oW = take(nt * nt * (conv ? 2 : 1));
    P.bytes = 128 + static_cast<size_t>(es) * static_cast<size_t>(o);
    P.threads = nt >= 32 ? 256 : (fp64 || !power_of_two(n0) ? 128 : 64);  // 16 x 16: blocks of 2 x 2 cells
    return P;
}

int top_level(int n0, int n_levels, bool fp64)
{
    if (!supported_n0(n0)) return 0;
    int top = 0;
    for (int t = 1; t < n_levels && t <= kMaxTop && (n0 << t) <= 64; ++t)
        if (make_plan(n0, t, fp64, true, true).bytes <= static_cast<size_t>(kMaxSmem)) top = t;
    return top;
}

bool prepare_f32() { return prepare_all<float>(); }

bool vcycle_f32(const mlqmc_dev::FmgArgs& A, const Plan& P, int B, cudaStream_t st)
{
    return vcycle_launch<float>(A, P, B, st);
}

bool stages_f32(const mlqmc_dev::FmgArgs& A, const Plan& P, const Stages& S, int count, cudaStream_t st)
{
    return S.thresh > 0.0 ? stages_launch<float, true>(A, P, S, count, st) : stages_launch<float, false>(A, P, S, count, st);
}

}  // namespace mlqmc_small
