// Radix schedules and index arithmetic of the runtime-length forms (passes_any.cuh), shared by
// host and device.
#pragma once
#include <algorithm>

#ifdef __CUDACC__
#define GSP_HD __host__ __device__
#else
#define GSP_HD
#endif

namespace gsp {

// Radix schedule of a runtime-length transform (the runtime-length pass forms): length L in
// nst stages of radices r[0..nst), r[0] even.  M[st] is the product of the later radices, P[st]
// of the earlier ones.  Digit st of a value's slot has stride S[st] (S[nst - 1] = 1), which is
// M[st], or with padding the next odd number from r[st + 1] S[st + 1] on; slots = r[0] S[0].
// mulM and mulR are the reciprocals floor(2^32 / d) + 1 of M[st] and r[st], so that
// e / d = umulhi(e, mul) exactly for e < 2^20.
constexpr int kAnyMaxStages = 8;
struct AnySched {
    int L;
    int nst;
    int slots;
    int r[kAnyMaxStages], M[kAnyMaxStages], P[kAnyMaxStages], S[kAnyMaxStages];
    unsigned mulM[kAnyMaxStages], mulR[kAnyMaxStages];
};
// The schedule of the even 5-smooth length L >= 4 with radices 2, 3, 4, 5, 6, 8, 9, 10 and 12
// up to max_radix: at least two and otherwise the fewest stages, among those the smallest sum
// of the radices.  First (its stage skips the padding's zeros) a 4 or an 8, whose zero-skipping
// forms have the fewest products to round, or the largest even radix; last the smallest of the
// others, at most max_last.  nst = 0 if there is none.
inline AnySched any_sched(int L, int max_radix, int max_last, bool pad) {
    static const int kRadix[] = {12, 10, 9, 8, 6, 5, 4, 3, 2};
    // Which of the n non-increasing radices goes first, or -1 if none can.
    auto first_of = [&](const int *f, int n) {
        const int i4 = (int)(std::find(f, f + n, 4) - f), i8 = (int)(std::find(f, f + n, 8) - f);
        const int even = (int)(std::find_if(f, f + n, [](int v) { return v % 2 == 0; }) - f);
        for (int i : {i4, i8, even})
            if (i < n && f[i == n - 1 ? n - 2 : n - 1] <= max_last) return i;
        return -1;
    };
    // Depth-first over non-increasing radices.
    int cur[kAnyMaxStages], best[kAnyMaxStages], nbest = 0, sbest = 0;
    auto search = [&](auto &&self, int m, int n, int from) -> void {
        if (m == 1) {
            if (n < 2 || (nbest && n > nbest)) return;
            int sum = 0;
            for (int i = 0; i < n; ++i) sum += cur[i];
            if (first_of(cur, n) >= 0 && (n < nbest || !nbest || sum < sbest)) {
                nbest = n;
                sbest = sum;
                std::copy(cur, cur + n, best);
            }
            return;
        }
        if (n == kAnyMaxStages) return;
        for (int i = from; i < 9; ++i)
            if (kRadix[i] <= max_radix && m % kRadix[i] == 0) {
                cur[n] = kRadix[i];
                self(self, m / kRadix[i], n + 1, i);
            }
    };
    search(search, L, 0, 0);
    AnySched s{};
    s.L = L;
    s.nst = nbest;
    if (nbest) {
        const int i = first_of(best, nbest);
        std::rotate(best, best + i, best + i + 1);
    }
    for (int st = nbest - 1; st >= 0; --st) {
        const bool last = st == nbest - 1;
        s.r[st] = best[st];
        s.M[st] = last ? 1 : s.M[st + 1] * s.r[st + 1];
        s.S[st] = last ? 1 : s.r[st + 1] * s.S[st + 1];
        if (pad && !last) s.S[st] |= 1;
        s.mulM[st] = s.M[st] == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)s.M[st] + 1);
        s.mulR[st] = (unsigned)((1ull << 32) / (unsigned)s.r[st] + 1);
    }
    for (int st = 0; st < nbest; ++st) s.P[st] = st == 0 ? 1 : s.P[st - 1] * s.r[st - 1];
    s.slots = nbest ? s.r[0] * s.S[0] : 0;
    return s;
}

// Largest radix, per arithmetic.  Double-float stops at 10: its butterflies are ten times longer
// in instructions, and the stages of a kernel should stay within the instruction cache.
constexpr int any_max_radix(bool df) { return df ? 10 : 12; }
// The schedule with radices up to 10, or up to max_radix where that takes a stage less; mr: the
// largest radix (10 or 12) the kernels that run it need.  Kernels without the radix-12 stages
// are 2 to 10% faster on the same schedule (FP32 solves: N = 400 2.81 and 2.78 ms, N = 162 242 and
// 234 us, N = 120 107 and 97 us), one more stage costs more (N = 60 25 and 33 us, N = 72 29 and
// 36 us).
inline AnySched any_sched_of(int L, int max_radix, int max_last, bool pad, int *mr) {
    const AnySched a = any_sched(L, 10, std::min(max_last, 10), pad);
    *mr = std::max(*mr, 10);
    if (max_radix == 10) return a;
    const AnySched b = any_sched(L, max_radix, max_last, pad);
    if (!b.nst || (a.nst && a.nst <= b.nst)) return a;
    *mr = max_radix;
    return b;
}
// Warps of an SM that their registers admit (80 in FP32, 128 otherwise).
constexpr int any_max_warps(bool f32) { return f32 ? 24 : 16; }
// Largest last radix of the x passes, whose last stage holds two butterflies.
constexpr int kAnyRowsLast = 8;

// Tile of a runtime-length pass: its schedule, 2^lg 16-byte groups, slots pitch groups apart,
// threads (few: where all tiles of a launch are resident at once, few_ctas to an SM), bytes of
// shared memory, largest radix of its kernel.
struct AnyTile {
    AnySched s;
    int lg, pitch, threads, few, few_ctas, smem, mr;
};
constexpr int kAnyThreads = 256;  // threads the kernels are compiled for
// Whether a launch of ntiles tiles lasts as long as one CTA: all tiles are resident at once, with at
// most three warps to a scheduler.  Then the threads with the fewest rounds over the butterflies
// serve it best, not those that fill an SM with CTAs (double-float solves: N = 36 39.4 -> 36.5 us,
// 40 42.0 -> 39.2, box 12 x 200 x 12 44.5 -> 40.2; with more warps it loses, FP64 N = 50 152.9 ->
// 154.0, where the rule leaves the threads as they are).
inline bool any_is_few(const AnyTile &t, int sms, int ntiles) {
    return ntiles <= sms * t.few_ctas && (long long)ntiles * t.few <= (long long)sms * 384;
}

// rows: an x pass (one more group of pitch, odd slot strides: conflict-free for neighbouring
// groups and for neighbouring samples alike); else a column pass (eight groups fill a 128-byte
// row, which a quarter-warp reads whole; four groups take odd strides instead).  Eight groups
// while three CTAs fit an SM, else four (FP32, solves: N = 240 590 us with eight, 605 us with
// four; N = 162 243 and 275 us; N = 400, where only two CTAs of eight fit, 2.86 and 2.83 ms).
// groups x planes: the 16-byte groups of one solve's pass (a tile stays within a plane).  Tiles of
// eight that leave half of the SMs idle are made of four where a stage of eight takes several rounds
// (box 400 x 12 x 12, double-float 54.4 -> 42.5 us; 400 x 20 x 20, FP32 31.8 -> 27.2 us).  In the
// wider arithmetics two groups where four leave room for one CTA of eight warps (the columns of
// N = 900 to 1000: double-float box 24 x 24 x 1000 213 -> 174 us, cube N = 1000 278 -> 253 ms, in
// FP64 828 -> 692 us for the box; FP32, whose columns are half as wide, loses at N = 900, 51 -> 61 ms).
// Threads: the multiple of 32 with the most threads of
// an SM at work, counting the share of thread slots that the rounds over the butterflies of
// each stage fill and the CTAs that shared memory and registers admit; few: see any_is_few.
inline AnyTile any_tile(int L, int max_radix, bool f32, bool rows, long long groups, int planes, int sms) {
    AnyTile t{};
    const int max_last = rows ? kAnyRowsLast : max_radix, max_warps = any_max_warps(f32);
    const AnySched wide = any_sched_of(L, max_radix, max_last, rows, &t.mr);
    bool eight = wide.slots * (rows ? 9 : 8) * 16 <= 70 * 1024;
    if (2 * ((groups + 7) / 8) * planes <= sms)
        for (int st = 0; st < wide.nst; ++st) eight = eight && L / wide.r[st] * 8 <= kAnyThreads;
    t.lg = eight ? 3 : 2;
    t.s = t.lg == 3 ? wide : any_sched_of(L, max_radix, max_last, true, &t.mr);
    if (!f32 && !rows && t.s.slots * (16 << t.lg) > 112 * 1024) t.lg = 1;
    t.pitch = (1 << t.lg) + (rows ? 1 : 0);
    t.smem = t.s.slots * t.pitch * 16;
    auto rounds_of = [&](int n) {
        int rounds = 0;
        for (int st = 0; st < t.s.nst; ++st) rounds += (((L / t.s.r[st]) << t.lg) + n - 1) / n * t.s.r[st];
        // the Hermitian split on its own, two values an item
        return rows ? rounds + (((L / 2 + 1) << t.lg) + n - 1) / n * 2 : rounds;
    };
    auto ctas_of = [&](int n) { return std::min(232448 / (t.smem + L * 16 + 1024), max_warps * 32 / n); };
    double best = 0.0;
    for (int n = kAnyThreads; n >= 64; n -= 32) {
        double slots = 0.0, used = 0.0;
        for (int st = 0; st < t.s.nst; ++st) {
            const int items = (L / t.s.r[st]) << t.lg;
            slots += (double)((items + n - 1) / n) * n * t.s.r[st];
            used += (double)items * t.s.r[st];
        }
        const double score = used / slots * ctas_of(n) * n;
        if (score > best * 1.02 || n == kAnyThreads) {
            best = score;
            t.threads = n;
        }
    }
    t.few = t.threads;
    for (int n = kAnyThreads; n >= 64; n -= 32) {
        const int less = rounds_of(n) - rounds_of(t.few);
        if (less < 0 || (less == 0 && t.few != t.threads)) t.few = n;
    }
    t.few_ctas = ctas_of(t.few);
    return t;
}

// Tile of the plane kernels (passes_plane.cuh): the x and y passes of one nx x ny plane in
// shared memory, gx row groups (pitch px) by sx.slots and gy column groups (pitch py) by sy.slots;
// w columns or rows per 16-byte group.  threads as for any_tile, over the stages of both axes.
struct PlaneTile {
    AnySched sx, sy;
    int gx, px, gy, py, threads, smem, mr;
    bool on, many;
};
constexpr int kPlaneThreads = 384;
// Largest plane: in FP32 two CTAs fit an SM (solves, separate passes against the plane kernels:
// 20^3 21.4 and 18.9 us, 60^3 27.2 and 25.5, 64 x 64 x 256 66 and 57, but 72^3 28.6 and 30.2); the
// wider arithmetics are bound by the longer chain of one CTA soon (double-float 10^3 24.3 and
// 20.8 us, 18^3 27.4 and 27.4, 20^3 25.9 and 28.5, 30^3 32.0 and 36.6).  Larger planes, up
// to plane_many, are worth a CTA each where they fill the SMs, no wave of them below nine tenths
// (many; FP64 24 x 24 x 600 413 and 395 us, but 20 x 20 x 240 112 and 122; double-float 20 x 20 x 300 45.8
// and 43.3, but 20 x 20 x 400 53.8 and 62.4 and 24 x 24 x 300 56.6 and 61.5).  Cubes whose passes are compiled for
// their length have kernels of their own (plane_n_size).
constexpr int plane_smem(bool f32) { return f32 ? 106 * 1024 : 18 * 1024; }
constexpr int plane_many(bool fp64) { return fp64 ? 48 * 1024 : 20 * 1024; }
// fp64: FP64 arithmetic.
inline PlaneTile plane_tile(int nx, int ny, int max_radix, int w, bool fp64) {
    PlaneTile t{};
    t.sx = any_sched_of(nx, max_radix, kAnyRowsLast, true, &t.mr);
    t.sy = any_sched_of(2 * ny, max_radix, max_radix, false, &t.mr);
    t.gx = ny / w;
    t.gy = (nx + w) / w;
    t.px = t.gx | 1;
    t.py = t.gy | 1;
    t.smem = 16 * (t.sx.slots * t.px + t.sy.slots * t.py);
    // The fewest rounds of butterflies per thread, weighted by their radix; among equals the
    // fewest threads.
    int best = 0;
    for (int n = kPlaneThreads; n >= 128; n -= 32) {
        int rounds = 0;
        for (const AnySched *s : {&t.sx, &t.sy})
            for (int st = 0; st < s->nst; ++st)
                rounds += (s->L / s->r[st] * (s == &t.sx ? t.gx : t.gy) + n - 1) / n * s->r[st];
        if (n == kPlaneThreads || rounds <= best) {
            best = rounds;
            t.threads = n;
        }
    }
    t.on = t.sx.nst && t.sy.nst && t.smem <= plane_smem(w == 2);
    t.many = w == 1 && t.sx.nst && t.sy.nst && t.smem <= plane_many(fp64);
    return t;
}
// Whether a launch of `planes` planes runs the plane kernels.
inline bool plane_runs(const PlaneTile &t, int sms, int planes) {
    if (t.on || !t.many) return t.on;
    const long long resident = (long long)sms * std::max(1, any_max_warps(false) * 32 / t.threads);
    return 10 * planes >= 9 * ((planes + resident - 1) / resident * resident);
}

// e / d by its reciprocal mul.
GSP_HD inline int rdiv(int e, unsigned mul) { return (int)(((unsigned long long)(unsigned)e * mul) >> 32); }

// Butterfly b < L / R of stage st: its first slot, the time index lo of its later digits and
// the frequency of its earlier digits.
struct AnyBfly {
    int slot, lo, freq;
};
GSP_HD inline int any_lo_slot(const AnySched &s, int st, int lo) {
    int a = 0;
    for (int u = st + 1; u < s.nst - 1; ++u) {
        const int q = rdiv(lo, s.mulM[u]);
        a += q * s.S[u];
        lo -= q * s.M[u];
    }
    return a + lo;
}
GSP_HD inline AnyBfly any_bfly(const AnySched &s, int st, int b) {
    AnyBfly f;
    int hi = b;
    f.lo = 0;
    f.slot = 0;
    f.freq = 0;
    if (st < s.nst - 1) {
        hi = rdiv(b, s.mulM[st]);
        f.lo = b - hi * s.M[st];
        f.slot = any_lo_slot(s, st, f.lo);
    }
    if (st > 0) {
        for (int u = st - 1; u >= 1; --u) {
            const int q = rdiv(hi, s.mulR[u]), d = hi - q * s.r[u];
            f.slot += d * s.S[u];
            f.freq += d * s.P[u];
            hi = q;
        }
        f.slot += hi * s.S[0];
        f.freq += hi;
    }
    return f;
}
// Slot of frequency k.
GSP_HD inline int any_freq_slot(const AnySched &s, int k) {
    int a = 0;
    for (int u = 0; u < s.nst - 1; ++u) {
        const int q = rdiv(k, s.mulR[u]);
        a += (k - q * s.r[u]) * s.S[u];
        k = q;
    }
    return a + k;
}

}  // namespace gsp
