// Launchers of the runtime-length forms, included by one .cu file per arithmetic.
#pragma once
#include "passes.cuh"
#include "passes_any.cuh"

namespace gsp {

// CTAs of a pass.  FP32: what fits on the SMs at once, each walking several tiles with one copy of
// the twiddles.  The others hold no copy and take one tile each (double-float, N = 162 and 200:
// z 479 and 950 us, against 551 and 1106 us when the CTAs walk the tiles).
template <typename Real, class K> int any_grid(K k, int threads, int smem, int ntiles) {
    return AnyTwiddles<Real>::kCopy ? persistent_blocks(k, threads, smem, ntiles) : ntiles;
}

// Whether launches of few tiles take the last x stage and the Hermitian split apart: the wider
// arithmetics, whose combined stage is a chain of a thousand instructions in a quarter of the
// threads (double-float N = 30 36.4 -> 32.1 us, N = 40 39.2 -> 35.0; N = 162, whose tiles fill the
// SMs, 867 -> 901 us).  The bits are the same.
template <typename Real> constexpr bool any_split_form() { return Types<Real>::W == 1; }

// Runs f.template operator()<MR>() with MR the largest radix the kernels are compiled for.
template <typename Real, class F> cudaError_t any_with_radix(int mr, F &&f) {
    if constexpr (any_max_radix(std::is_same<Real, DF>::value) > 10)
        if (mr > 10) return f.template operator()<12>();
    return f.template operator()<10>();
}

template <typename Real>
cudaError_t any_x(const DevicePlan &p, const PtrArray &rho, const PtrArray &u, int B, cudaStream_t s, bool fwd,
                  int rows, void *w1) {
    const int nx = p.n3[0], ny = p.n3[1], nz = p.n3[2];
    const AnyTile &t = p.any_tile[std::is_same<Real, DF>::value][0];
    if (!t.s.nst) return cudaErrorInvalidValue;
    const int rows_b = ny * nz, nrows = rows ? rows : B * rows_b;
    const AnyTw<Real> *tw = static_cast<const AnyTw<Real> *>(p.tw3[0]);
    Cx2<Real> *ws = static_cast<Cx2<Real> *>(w1 ? w1 : p.w1);
    const int TR = Types<Real>::W << t.lg, nt = (nrows + TR - 1) / TR;
    const bool few = any_is_few(t, p.sms, nt), split = few && any_split_form<Real>();
    const int smem = t.smem + any_tw_bytes<Real>(nx), T = few ? t.few : t.threads;
    const unsigned mul_half = (unsigned)((1ull << 32) / (unsigned)((split ? nx : t.s.P[t.s.nst - 1]) / 2 + 1) + 1);
    auto run = [&](auto kf, auto ki) {
        if (fwd) {
            GSP_CHECK(set_smem(kf, smem));
            GSP_CHECK(launch_pdl(kf, any_grid<Real>(kf, T, smem, nt), T, smem, s, rho, ws, tw, t.s, rows_b, nrows, p.Px, mul_half, t.lg, nt));
        } else {
            GSP_CHECK(set_smem(ki, smem));
            GSP_CHECK(launch_pdl(ki, any_grid<Real>(ki, T, smem, nt), T, smem, s, static_cast<const Cx2<Real> *>(ws), u, tw, t.s, rows_b,
                                 nrows, p.Px, mul_half, t.lg, nt));
        }
        return cudaGetLastError();
    };
    return any_with_radix<Real>(t.mr, [&]<int MR>() {
        if constexpr (any_split_form<Real>())
            if (split) return run(k_any_x_fwd<Real, MR, true>, k_any_x_inv<Real, MR, true>);
        return run(k_any_x_fwd<Real, MR, false>, k_any_x_inv<Real, MR, false>);
    });
}

template <typename Real>
cudaError_t any_y(const DevicePlan &p, int B, cudaStream_t s, bool fwd, int z0, int nzs) {
    const int nx = p.n3[0], ny = p.n3[1], nz = p.n3[2], L = 2 * ny;
    const int planes = nzs ? nzs : B * nz, ncols = nx + 1;
    const AnyTw<Real> *tw = static_cast<const AnyTw<Real> *>(p.tw3[1]);
    const long long w1p = (long long)ny * p.Px, w2p = (long long)L * p.Px;
    const AnyTile &t = p.any_tile[std::is_same<Real, DF>::value][1];
    if (!t.s.nst) return cudaErrorInvalidValue;
    const int TC = Types<Real>::W << t.lg, ntx = (ncols + TC - 1) / TC, nt = ntx * planes;
    const int smem = t.smem + any_tw_bytes<Real>(L), T = any_is_few(t, p.sms, nt) ? t.few : t.threads;
    return any_with_radix<Real>(t.mr, [&]<int MR>() {
        if (fwd) {
            GSP_CHECK(set_smem(k_any_col<Real, MR, true>, smem));
            GSP_CHECK(launch_pdl(k_any_col<Real, MR, true>, any_grid<Real>(k_any_col<Real, MR, true>, T, smem, nt), T, smem, s,
                                 static_cast<const Cx2<Real> *>(p.w1) + z0 * w1p, static_cast<Cx2<Real> *>(p.w2) + z0 * w2p,
                                 tw, t.s, ncols, ntx, p.Px, w1p, w2p, t.lg, nt));
        } else {
            GSP_CHECK(set_smem(k_any_col<Real, MR, false>, smem));
            GSP_CHECK(launch_pdl(k_any_col<Real, MR, false>, any_grid<Real>(k_any_col<Real, MR, false>, T, smem, nt), T, smem, s,
                                 static_cast<const Cx2<Real> *>(p.w3) + z0 * w2p, static_cast<Cx2<Real> *>(p.w1) + z0 * w1p,
                                 tw, t.s, ncols, ntx, p.Px, w2p, w1p, t.lg, nt));
        }
        return cudaGetLastError();
    });
}

// The z pass of lines ky0 <= ky < ky0 + nky (nky = 0: all 2 ny lines).  Runs on the tables of
// any plan: the compiled-length plans' symbol octant has the same layout as the box table
// and their twiddles W_{2N} are axis z's table.
template <typename Real>
cudaError_t any_z(const DevicePlan &p, int B, cudaStream_t s, double *tail, int ky0, int nky) {
    const int nx = p.n3[0], ny = p.n3[1];
    if (nky == 0) nky = 2 * ny;
    const AnyTw<Real> *tw = static_cast<const AnyTw<Real> *>(p.any ? p.tw3[2] : p.tw);
    const AnyTile &t = p.any_tile[std::is_same<Real, DF>::value][2];
    if (!t.s.nst) return cudaErrorInvalidValue;
    const int TC = Types<Real>::W << t.lg, ntx = (nx + 1 + TC - 1) / TC, nt = ntx * nky * B;
    const int smem = t.smem + any_tw_bytes<Real>(t.s.L), T = any_is_few(t, p.sms, nt) ? t.few : t.threads;
    return any_with_radix<Real>(t.mr, [&]<int MR>() {
        auto k = tail ? k_any_z<Real, MR, true> : k_any_z<Real, MR, false>;
        GSP_CHECK(set_smem(k, smem));
        GSP_CHECK(launch_pdl(k, any_grid<Real>(k, T, smem, nt), T, smem, s, static_cast<const Cx2<Real> *>(p.w2),
                             static_cast<Cx2<Real> *>(p.w3), static_cast<const Real *>(p.sym), tw, t.s, nx, ny, ntx, p.Px,
                             p.Ps, tail, ky0, nky, t.lg, nt));
        return cudaGetLastError();
    });
}

// One translation unit per pass and arithmetic (the double-float ones compile slowly).
#define GSP_INSTANTIATE_ANY_X(Real) \
    template cudaError_t any_x<Real>(const DevicePlan &, const PtrArray &, const PtrArray &, int, cudaStream_t, bool, int, void *);
#define GSP_INSTANTIATE_ANY_Y(Real) \
    template cudaError_t any_y<Real>(const DevicePlan &, int, cudaStream_t, bool, int, int);
#define GSP_INSTANTIATE_ANY_Z(Real) \
    template cudaError_t any_z<Real>(const DevicePlan &, int, cudaStream_t, double *, int, int);

}  // namespace gsp
