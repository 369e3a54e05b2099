// Test shim: the runtime-length forms' schedules and index arithmetic (csrc/any_sched.h) on the
// CPU.  Runs the in-place stages of one transform with plain DFTs in place of the radix
// butterflies.
#include <cmath>
#include <complex>
#include <vector>

#include "any_sched.h"

using cd = std::complex<double>;

// The transform of x (L values) into X in natural order.  Returns 0, or the number of the rule
// that failed: 1 schedule, 2 slot out of range or taken twice in a stage, 3 frequency of a
// butterfly's outputs, 4 slot of a frequency, 5 a radix above max_radix, or
// the last one above max_last.
extern "C" int shim_any_transform(int L, int max_radix, int max_last, int pad, const double *x, double *X) {
    const gsp::AnySched s = gsp::any_sched(L, max_radix, max_last, pad != 0);
    int prod = 1;
    for (int st = 0; st < s.nst; ++st) {
        if (s.r[st] > max_radix || (st + 1 == s.nst && s.r[st] > max_last)) return 5;
        prod *= s.r[st];
    }
    if (s.nst < 2 || prod != L || s.r[0] % 2 || s.slots < L) return 1;
    const double tau = 2.0 * std::acos(-1.0);
    std::vector<cd> v(s.slots);
    for (int j = 0; j < s.M[0]; ++j)
        for (int r = 0; r < s.r[0]; ++r) {
            const int n = j + r * s.M[0];
            v[gsp::any_lo_slot(s, 0, j) + r * s.S[0]] = cd(x[2 * n], x[2 * n + 1]);
        }
    for (int st = 0; st < s.nst; ++st) {
        const int R = s.r[st], nb = s.P[st] * s.M[st];
        std::vector<char> hit(s.slots, 0);
        for (int b = 0; b < nb; ++b) {
            const gsp::AnyBfly f = gsp::any_bfly(s, st, b);
            std::vector<cd> in(R), out(R);
            for (int r = 0; r < R; ++r) {
                const int a = f.slot + r * s.S[st];
                if (a < 0 || a >= s.slots || hit[a]) return 2;
                hit[a] = 1;
                in[r] = v[a];
            }
            for (int k = 0; k < R; ++k) {
                cd acc = 0;
                for (int r = 0; r < R; ++r) acc += in[r] * std::polar(1.0, -tau * (r * k % R) / R);
                const int e = st + 1 < s.nst ? f.lo * s.P[st] * k : 0;
                if (e >= L) return 3;
                out[k] = acc * std::polar(1.0, -tau * e / L);
            }
            for (int r = 0; r < R; ++r) {
                v[f.slot + r * s.S[st]] = out[r];
                if (st + 1 == s.nst && gsp::any_freq_slot(s, f.freq + r * nb) != f.slot + r * s.S[st]) return 3;
            }
        }
    }
    for (int k = 0; k < L; ++k) {
        const int a = gsp::any_freq_slot(s, k);
        if (a < 0 || a >= s.slots) return 4;
        X[2 * k] = v[a].real();
        X[2 * k + 1] = v[a].imag();
    }
    return 0;
}

// The schedule and the kernel's largest radix that the passes of length L take: 0, or 1 if a
// radix is above it, 2 if 12 is taken where 10 gives no more stages, 3 if a stage is wasted.
extern "C" int shim_any_radix_rule(int L, int max_radix, int max_last, int pad) {
    int mr = 0;
    const gsp::AnySched s = gsp::any_sched_of(L, max_radix, max_last, pad != 0, &mr);
    const gsp::AnySched a = gsp::any_sched(L, 10, std::min(max_last, 10), pad != 0);
    const gsp::AnySched b = gsp::any_sched(L, max_radix, max_last, pad != 0);
    for (int st = 0; st < s.nst; ++st)
        if (s.r[st] > mr) return 1;
    if (mr > 10 && s.nst >= a.nst) return 2;
    return s.nst == std::min(a.nst, b.nst) ? 0 : 3;
}

// The tile of a pass: lg, threads, few, few_ctas, bytes of shared memory with the twiddles, the weighted
// rounds over the butterflies (and, for rows, over the Hermitian split) with `threads` and with `few`.
// 0, or 1 if the schedule does not multiply up to L.
extern "C" int shim_any_tile(int L, int df, int f32, int rows, long long groups, int planes, int sms, int *out) {
    const gsp::AnyTile t = gsp::any_tile(L, gsp::any_max_radix(df != 0), f32 != 0, rows != 0, groups, planes, sms);
    int prod = 1;
    for (int st = 0; st < t.s.nst; ++st) prod *= t.s.r[st];
    if (t.s.nst < 2 || prod != L || t.smem != t.s.slots * t.pitch * 16) return 1;
    auto rounds = [&](int n) {
        int v = rows ? (((L / 2 + 1) << t.lg) + n - 1) / n * 2 : 0;
        for (int st = 0; st < t.s.nst; ++st) v += (((L / t.s.r[st]) << t.lg) + n - 1) / n * t.s.r[st];
        return v;
    };
    const int v[] = {t.lg, t.threads, t.few, t.few_ctas, t.smem + (f32 ? L * 8 + 8 : 0), rounds(t.threads), rounds(t.few)};
    std::copy(v, v + 7, out);
    return 0;
}
// Whether a launch of ntiles tiles of that pass takes `few`.
extern "C" int shim_any_is_few(int threads, int ctas, int sms, int ntiles) {
    gsp::AnyTile t{};
    t.few = threads;
    t.few_ctas = ctas;
    return gsp::any_is_few(t, sms, ntiles);
}
// The plane kernels' tile: whether a launch of `planes` planes on sms SMs runs them, threads, bytes of
// shared memory with the twiddles.  df: double-float arithmetic, else FP32 or FP64 by f32.
extern "C" int shim_plane_tile(int nx, int ny, int df, int f32, int sms, int planes, int *out) {
    const gsp::PlaneTile t = gsp::plane_tile(nx, ny, gsp::any_max_radix(df != 0), f32 ? 2 : 1, !f32 && !df);
    const int v[] = {gsp::plane_runs(t, sms, planes), t.threads, t.smem + (f32 ? (nx + 2 * ny) * 8 + 16 : 0)};
    std::copy(v, v + 3, out);
    return 0;
}
