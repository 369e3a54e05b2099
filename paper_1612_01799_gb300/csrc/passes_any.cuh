// Runtime-length forms of the five passes: any even N with N 5-smooth (4 <= N <= 1024)
// and boxes with a different number of points per axis (Sec. 2 standardised form, n_q
// points on axis q).  Same operations as the compiled-length forms of passes.cuh (K1 x
// forward, K2 y forward, K3 z fused with the symbol, K4 y inverse, K5 x inverse), with
// the transform lengths, radix schedules and grid dimensions as kernel arguments, so one
// instantiation per arithmetic serves every shape.
//
// A tile of transforms sits in shared memory in 16-byte groups (two neighbouring FP32
// columns, packed FP32x2, or one FP64 or double-float column).  A transform of length
// L = R_0 R_1 ... runs its radix stages in place, decimation in frequency: stage s takes the
// R_s values that differ in digit s of their slot, transforms them in registers and writes
// them back to the same slots times W^{j k}, so one block barrier separates two stages
// and no second buffer is needed.  After the last stage the frequency
// k_0 + R_0 (k_1 + R_1 (k_2 + ...)) sits in slot (k_0, k_1, ...): the rows of a column pass
// may leave in any order (each is its own segment of device memory), and the inverse is the
// adjoint, stage by stage in reverse order, so the z pass applies the symbol to the
// registers between the last forward and the first inverse stage.  The first stage reads
// its inputs from device memory and leaves out the zero half of the padding (the transform
// of R_0 / 2 values, R_0 even), the last one writes device memory.
//
// What bounds them (N = 200, FP32): instruction issue at 40 to 50% of its slots and latency with
// 20 to 24 warps on an SM (80 registers a thread); double-float issues 43% in the x passes and
// three quarters of its slots in z.  Two or three stages of radix 8 to 12 in place of five to
// seven of radix 2 to 5 with a ping-pong pair, the first stage's zeros left out, took the
// FP32 solve at N = 400 from 9.45 to 2.77 ms, N = 240 from 2.14 to 0.59 ms, the box 64 x 128 x
// 192 from 257 to 109 us and the double-float solve at N = 162 from 1.20 to 0.87 ms.
//
// Workspace layout (complex, the arithmetic's storage): w1 [b][z < nz][y < ny][kx < Px],
// w2 and w3 [b][z < nz][ky < 2 ny][kx < Px], Px = pitch of nx + 1; symbol
// [kz <= nz][ky <= ny][kx < Ps] (Ps = pitch of nx + 1), real, scaled by lambda^2 /
// (8 nx ny nz).
#pragma once

namespace gsp {

// Row r (< TR) of the tile starting at batch row r0: its density and its row in that density.
// rows_b >= TR, so a tile crosses at most one density boundary.
struct AnyRows {
    int b0;
    long long first;  // row of r0 within density b0
    long long left;   // rows of density b0 from r0 on
    __device__ AnyRows(long long r0, int rows_b) {
        b0 = (int)((unsigned)r0 / (unsigned)rows_b);  // r0 lies below the number of rows, an int
        first = r0 - (long long)b0 * rows_b;
        left = rows_b - first;
    }
    __device__ int density(int r) const { return r < left ? b0 : b0 + 1; }
    __device__ long long row(int r) const { return r < left ? first + r : r - left; }
};

// ---- 16-byte groups ----------------------------------------------------------------------------
__device__ __forceinline__ CV any_ld(const float4 *p, CV) {
    const float4 f = sm_ld(p);
    return {f2(f.x, f.y), f2(f.z, f.w)};
}
__device__ __forceinline__ void any_st(float4 *p, CV x) { sm_st(p, make_float4(x.re.x, x.re.y, x.im.x, x.im.y)); }
__device__ __forceinline__ CD any_ld(const float4 *p, CD) {
    const double2 f = sm_ld(reinterpret_cast<const double2 *>(p));
    return {f.x, f.y};
}
__device__ __forceinline__ void any_st(float4 *p, CD x) {
    sm_st(reinterpret_cast<double2 *>(p), make_double2(x.re, x.im));
}
__device__ __forceinline__ CDF any_ld(const float4 *p, CDF) {
    const float4 f = sm_ld(p);
    return {DF(f.x, f.y), DF(f.z, f.w)};
}
__device__ __forceinline__ void any_st(float4 *p, CDF x) {
    sm_st(p, make_float4(x.re.hi, x.re.lo, x.im.hi, x.im.lo));
}


// a times the table twiddle w (D < 0) or its conjugate (D > 0).
// FP32 negates by a packed product with -1 (one instruction, exact).
template <int D> __device__ __forceinline__ CV any_twmul(CV a, float2 w) {
    const float2 R = f2(w.x, w.x), I = f2(w.y, w.y), M = f2(-1.f, -1.f);
    if (D < 0) return {f2fma(f2mul(a.im, M), I, f2mul(a.re, R)), f2fma(a.re, I, f2mul(a.im, R))};
    return {f2fma(a.im, I, f2mul(a.re, R)), f2fma(f2mul(a.re, M), I, f2mul(a.im, R))};
}
template <int D> __device__ __forceinline__ CD any_twmul(CD a, double2 w) { return twmul<D>(a, w); }
template <int D> __device__ __forceinline__ CDF any_twmul(CDF a, float4 w) {
    // Renormalised: the stages of larger radix collect more in lo (rel-L2 error of a solve at
    // N = 100 and 162 over eight densities: 8.2e-15 and 8.2e-15 without, 6.0e-15 and 7.4e-15 with).
    return cnorm(twmul<D>(a, w));
}

// One row pair's worth of consecutive real sample pairs (x_2m, x_2m+1) as a group and back:
// rows a and b for FP32 (b unused elsewhere).
__device__ __forceinline__ CV any_pack(float2 a, float2 b, CV) { return {f2(a.x, b.x), f2(a.y, b.y)}; }
__device__ __forceinline__ CD any_pack(double2 a, double2, CD) { return {a.x, a.y}; }
__device__ __forceinline__ CDF any_pack(double2 a, double2, CDF) { return {DF(a.x), DF(a.y)}; }
__device__ __forceinline__ float2 any_ext(CV x, int i) { return i ? f2(x.re.y, x.im.y) : f2(x.re.x, x.im.x); }
__device__ __forceinline__ double2 any_ext(CD x, int) { return make_double2(x.re, x.im); }
__device__ __forceinline__ double2 any_ext(CDF x, int) { return c_ext(x); }
// The same for workspace values.
__device__ __forceinline__ CV any_wpack(float2 a, float2 b, CV) { return any_pack(a, b, CV{}); }
__device__ __forceinline__ CD any_wpack(double2 a, double2, CD) { return {a.x, a.y}; }
__device__ __forceinline__ CDF any_wpack(float4 a, float4, CDF) { return ws_c(a); }
__device__ __forceinline__ float2 any_ws(CV x, int i) { return any_ext(x, i); }
__device__ __forceinline__ double2 any_ws(CD x, int) { return make_double2(x.re, x.im); }
__device__ __forceinline__ float4 any_ws(CDF x, int) { return make_float4(x.re.hi, x.re.lo, x.im.hi, x.im.lo); }

__device__ __forceinline__ CV any_conj(CV a) { return {a.re, f2neg(a.im)}; }
__device__ __forceinline__ CD any_conj(CD a) { return {a.re, -a.im}; }
__device__ __forceinline__ CDF any_conj(CDF a) { return {a.re, -a.im}; }
__device__ __forceinline__ CV any_half(CV a) { return cscale(a, 0.5f); }
__device__ __forceinline__ CD any_half(CD a) { return cscale(a, 0.5); }
__device__ __forceinline__ CDF any_half(CDF a) {
    return {DF(0.5f * a.re.hi, 0.5f * a.re.lo), DF(0.5f * a.im.hi, 0.5f * a.im.lo)};
}

// ---- the radix stages ----------------------------------------------------------------------------
// exp(-2 pi i r / R) for r < R / 2, R in {4, 6, 8, 10, 12}.
__host__ __device__ constexpr double any_cos(int R, int r) {
    return r == 0 ? 1.0
         : 4 * r == R ? 0.0
         : R == 8 ? (r == 1 ? 0.70710678118654752440 : -0.70710678118654752440)
         : R == 10 ? (r == 1 ? 0.80901699437494742410 : r == 2 ? 0.30901699437494742410
                      : r == 3 ? -0.30901699437494742410 : -0.80901699437494742410)
         : R == 12 ? (r == 1 ? 0.86602540378443864676 : r == 2 ? 0.5 : r == 4 ? -0.5 : -0.86602540378443864676)
                   : (r == 1 ? 0.5 : -0.5);  // 6
}
__host__ __device__ constexpr double any_sin(int R, int r) {
    return r == 0 ? 0.0
         : 4 * r == R ? -1.0
         : R == 8 ? -0.70710678118654752440
         : R == 10 ? (r == 1 || r == 4 ? -0.58778525229247312917 : -0.95105651629515357212)
         : R == 12 ? (r == 1 || r == 5 ? -0.5 : -0.86602540378443864676)
                   : -0.86602540378443864676;  // 6
}
// Length-R DFT of v[0 .. R/2 - 1] (the rest zero): v[m] = X[2 m], v[R/2 + m] = X[2 m + 1].
template <int R, typename C> __device__ __forceinline__ void any_dft_half(C *v) {
    using Re = typename CxReal<C>::T;
    constexpr int H = R / 2;
#pragma unroll
    for (int r = 0; r < H; ++r) {
        if (r == 0) v[H] = v[0];
        else if (4 * r == R) v[H + r] = cmul_mi(v[r]);
        else if (R == 8 && r == 1) v[H + r] = cmul_w8<-1, 1>(v[r], (Re)any_cos(8, 1));
        else if (R == 8) v[H + r] = cmul_w8<-1, 3>(v[r], (Re)any_cos(8, 1));
        else v[H + r] = cmulk<-1>(v[r], (Re)any_cos(R, r), (Re)any_sin(R, r));
    }
    dft<H, -1>(v);
    dft<H, -1>(v + H);
}
// Its adjoint: y_r = IDFT_H(v[0..])[r] + conj(W_R^r) IDFT_H(v[H..])[r], r < H, in v[0 .. H - 1].
template <int R, typename C> __device__ __forceinline__ void any_dft_half_adj(C *v) {
    using Re = typename CxReal<C>::T;
    constexpr int H = R / 2;
    dft<H, 1>(v);
    dft<H, 1>(v + H);
#pragma unroll
    for (int r = 0; r < H; ++r) {
        if (r == 0) v[r] = cadd(v[r], v[H]);
        else if (4 * r == R) v[r] = add_rot<1>(v[r], v[H + r]);
        else if (R == 8 && r == 1) v[r] = cadd(v[r], cmul_w8<1, 1>(v[H + r], (Re)any_cos(8, 1)));
        else if (R == 8) v[r] = cadd(v[r], cmul_w8<1, 3>(v[H + r], (Re)any_cos(8, 1)));
        else v[r] = cadd(v[r], cmulk<1>(v[H + r], (Re)any_cos(R, r), (Re)any_sin(R, r)));
    }
}

// Runs f.template operator()<R>() for the radix R <= MR (10 or 12) of a stage: the even ones
// (first stages) and all of them.
template <int MR, typename F> __device__ __forceinline__ void any_radix_even(int R, F &&f) {
    switch (R) {
        case 2: f.template operator()<2>(); break;
        case 4: f.template operator()<4>(); break;
        case 6: f.template operator()<6>(); break;
        case 8: f.template operator()<8>(); break;
        default:
            if constexpr (MR > 10) {
                if (R == 12) {
                    f.template operator()<12>();
                    break;
                }
            }
            f.template operator()<10>();
    }
}
template <int MR, typename F> __device__ __forceinline__ void any_radix(int R, F &&f) {
    switch (R) {
        case 3: f.template operator()<3>(); break;
        case 5: f.template operator()<5>(); break;
        case 9: f.template operator()<9>(); break;
        default: any_radix_even<MR>(R, f);
    }
}

// The radices the last stage of the x passes may have (kAnyRowsLast).
template <typename F> __device__ __forceinline__ void any_radix_last(int R, F &&f) {
    switch (R) {
        case 2: f.template operator()<2>(); break;
        case 3: f.template operator()<3>(); break;
        case 4: f.template operator()<4>(); break;
        case 5: f.template operator()<5>(); break;
        case 6: f.template operator()<6>(); break;
        default: f.template operator()<8>(); break;
    }
}

// The twiddles W_L^e, e < L, of a transform of length L, from the plan's table tw of
// W_{L stride}.  FP32 copies them to shared memory at sm (once per CTA): a warp takes 4 or 8
// distinct ones per load, each a cache line of its own in the table (N = 240: z 334 -> 322 us,
// y inverse 135 -> 123 us).  The wider arithmetics read the table: there the copy costs more
// than it saves (double-float, N = 162: z 526 us with it, 471 us without).
template <typename Real> struct AnyTwiddles {
    const AnyTw<Real> *t;
    int stride;
    static constexpr bool kCopy = std::is_same<Real, float>::value;
    __device__ __forceinline__ AnyTwiddles(const AnyTw<Real> *__restrict__ tw, int L, int st, float4 *sm) {
        if constexpr (kCopy) {
            AnyTw<Real> *c = reinterpret_cast<AnyTw<Real> *>(sm);
            for (int e = threadIdx.x; e < L; e += blockDim.x) sm_st(c + e, __ldg(tw + e * st));
            t = c;
            stride = 1;
        } else {
            t = tw;
            stride = st;
        }
    }
    __device__ __forceinline__ AnyTw<Real> operator[](int e) const {
        if constexpr (kCopy) return sm_ld(t + e);
        else return __ldg(t + e * stride);
    }
};
// Bytes of shared memory of the copy.
template <typename Real> __host__ __device__ constexpr int any_tw_bytes(int L) {
    return AnyTwiddles<Real>::kCopy ? (L * (int)sizeof(AnyTw<Real>) + 15) / 16 * 16 : 0;
}

// Butterfly of a stage in the middle of a transform, in place over slots p[r * step], with the
// twiddles W_L^{e r} of the shared table tw.
template <int R, int D, typename C, typename Tw>
__device__ __forceinline__ void any_stage(float4 *p, int step, const Tw &tw, int e, C) {
    C v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = any_ld(p + r * step, C{});
    if constexpr (D > 0) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = any_twmul<1>(v[r], tw[r * e]);
    }
    dft<R, D>(v);
    if constexpr (D < 0) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = any_twmul<-1>(v[r], tw[r * e]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) any_st(p + r * step, v[r]);
}

// The middle stages st0 <= st < st1 of a tile of 2^lg groups (slot a of group g at buf[a * PG + g]),
// forward in ascending and inverse in descending order, each behind a block barrier.
// twstride: the table holds exp(-2 pi i e / (L twstride)).
template <typename Real, int MR, int D>
__device__ __forceinline__ void any_stages(float4 *buf, const AnySched &s, int lg, int PG, const AnyTwiddles<Real> &tw,
                                           int st0, int st1) {
    using C = typename Types<Real>::CC;
    const int g = threadIdx.x & ((1 << lg) - 1);
    for (int i = st0; i < st1; ++i) {
        const int st = D < 0 ? i : st0 + st1 - 1 - i;
        __syncthreads();
        const int R = s.r[st], nb = s.P[st] * s.M[st], step = s.S[st] * PG;
        any_radix<MR>(R, [&]<int RR>() {
            for (int b = threadIdx.x >> lg; b < nb; b += blockDim.x >> lg) {
                const AnyBfly f = any_bfly(s, st, b);
                float4 *p = buf + f.slot * PG + g;
                any_stage<RR, D>(p, step, tw, f.lo * s.P[st], C{});
            }
        });
    }
}

// The first forward stage of a column transform (time j + r M_0, r < R_0 / 2, loaded by
// ld(row)) and the last inverse stage (st(row, value) for the kept rows).
template <typename Real, int MR, class Ld>
__device__ __forceinline__ void any_first(float4 *buf, const AnySched &s, int lg, const AnyTwiddles<Real> &tw, Ld &&ld) {
    using C = typename Types<Real>::CC;
    const int g = threadIdx.x & ((1 << lg) - 1), M = s.M[0], step = s.S[0] << lg;
    any_radix_even<MR>(s.r[0], [&]<int R>() {
        constexpr int H = R / 2;
        for (int j = threadIdx.x >> lg; j < M; j += blockDim.x >> lg) {
            C v[R];
#pragma unroll
            for (int r = 0; r < H; ++r) v[r] = ld(j + r * M);
            any_dft_half<R>(v);
            float4 *p = buf + (any_lo_slot(s, 0, j) << lg) + g;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int k = i < H ? 2 * i : 2 * (i - H) + 1;
                any_st(p + k * step, k == 0 ? v[i] : any_twmul<-1>(v[i], tw[k * j]));
            }
        }
    });
}
template <typename Real, int MR, class St>
__device__ __forceinline__ void any_first_adj(const float4 *buf, const AnySched &s, int lg, const AnyTwiddles<Real> &tw, St &&st) {
    using C = typename Types<Real>::CC;
    const int g = threadIdx.x & ((1 << lg) - 1), M = s.M[0], step = s.S[0] << lg;
    __syncthreads();
    any_radix_even<MR>(s.r[0], [&]<int R>() {
        constexpr int H = R / 2;
        for (int j = threadIdx.x >> lg; j < M; j += blockDim.x >> lg) {
            const float4 *p = buf + (any_lo_slot(s, 0, j) << lg) + g;
            C v[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int k = i < H ? 2 * i : 2 * (i - H) + 1;
                v[i] = any_ld(p + k * step, C{});
                if (k > 0) v[i] = any_twmul<1>(v[i], tw[k * j]);
            }
            any_dft_half_adj<R>(v);
#pragma unroll
            for (int r = 0; r < H; ++r) st(j + r * M, v[r]);
        }
    });
}

// The last radix stage on its own, in place without twiddles, behind a block barrier; another one
// follows it.
template <typename Real, int D>
__device__ __forceinline__ void any_last(float4 *buf, const AnySched &s, int lg, int PG) {
    using C = typename Types<Real>::CC;
    const int g = threadIdx.x & ((1 << lg) - 1), last = s.nst - 1;
    __syncthreads();
    any_radix_last(s.r[last], [&]<int R>() {
        for (int b = threadIdx.x >> lg; b < s.P[last]; b += blockDim.x >> lg) {
            float4 *p = buf + any_bfly(s, last, b).slot * PG + g;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = any_ld(p + r * PG, C{});
            dft<R, D>(v);
#pragma unroll
            for (int r = 0; r < R; ++r) any_st(p + r * PG, v[r]);
        }
    });
    __syncthreads();
}

// Blocks per SM the kernels are compiled for.
template <typename Real> constexpr int kAnyMinBlocks = sizeof(typename Types<Real>::CS) == 8 ? 3 : 2;

// ---- K1: x forward ----------------------------------------------------------------------------
// Rows of nx = s.L reals (row g of the batch: density g / rows_b, row g % rows_b of it),
// NG = 2^lg groups per CTA (a group is two rows in FP32, one otherwise; slots NG + 1 groups apart, so that
// both the stages, with neighbouring groups in a warp, and the row-wise accesses, with
// neighbouring samples, are free of bank conflicts).  The padded length-2nx real DFT is the
// nx-point complex FFT of the (even, odd) sample pairs (pairs >= nx/2 zero) and the Hermitian
// split into the nx + 1 bins (twiddles W_{2nx}^k; the nx-point FFT reads the same table at
// stride 2).
template <typename Real, int MR, bool SPLIT>
__global__ void __launch_bounds__(kAnyThreads, kAnyMinBlocks<Real>)
k_any_x_fwd(const PtrArray rho, Cx2<Real> *__restrict__ out, const AnyTw<Real> *__restrict__ tw,
            const __grid_constant__ AnySched s, int rows_b, int nrows, int Px, unsigned mul_half, int lg, int ntiles) {
    using C = typename Types<Real>::CC;
    using X2 = Ext2<Real>;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4 *buf = reinterpret_cast<float4 *>(smraw);
    const int n = s.L, h = n / 2, M = s.M[0], NG = 1 << lg, PG = NG + 1, TR = NG * W;
    const AnyTwiddles<Real> ts(tw, n, 2, buf + s.slots * PG);
    griddep_wait();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();  // the table is written, the previous tile's reads of buf are done
        const long long r0 = (long long)t * TR;
        const int ng = (int)min((long long)NG, (nrows - r0) / W);
        const AnyRows rows(r0, rows_b);
        // Rows as they lie, times j + r M_0 of group g into their slots; missing rows as zeros.
        any_radix_even<MR>(s.r[0], [&]<int R>() {
            for (int e = threadIdx.x; e < NG * M; e += blockDim.x) {
                const int g = rdiv(e, s.mulM[0]), j = e - g * M;
                const bool ok = g < ng && dbg_index_ok(rows.row(W * g), rows_b);
                const X2 *src = ok ? reinterpret_cast<const X2 *>(rho.p[rows.density(W * g)]) + rows.row(W * g) * h : nullptr;
                C v[R / 2];
#pragma unroll
                for (int r = 0; r < R / 2; ++r) {
                    const int m = j + r * M;
                    if (ok) {
                        const X2 x = __ldg(src + m);
                        v[r] = any_pack(x, W == 2 ? __ldg(src + h + m) : x, C{});
                    } else {
                        v[r] = czero<C>();
                    }
                }
                float4 *p = buf + any_lo_slot(s, 0, j) * PG + g;
#pragma unroll
                for (int r = 0; r < R / 2; ++r) any_st(p + r * s.S[0] * PG, v[r]);
            }
        });
        __syncthreads();
        {
            const int g = threadIdx.x & (NG - 1), step = s.S[0] * PG;
            any_radix_even<MR>(s.r[0], [&]<int R>() {
                constexpr int H = R / 2;
                for (int j = threadIdx.x >> lg; j < M; j += blockDim.x >> lg) {
                    float4 *p = buf + any_lo_slot(s, 0, j) * PG + g;
                    C v[R];
#pragma unroll
                    for (int r = 0; r < H; ++r) v[r] = any_ld(p + r * step, C{});
                    any_dft_half<R>(v);
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int k = i < H ? 2 * i : 2 * (i - H) + 1;
                        any_st(p + k * step, k == 0 ? v[i] : any_twmul<-1>(v[i], ts[k * j]));
                    }
                }
            });
        }
        const int last = s.nst - 1, P = s.P[last], half = P / 2 + 1;
        any_stages<Real, MR, -1>(buf, s, lg, PG, ts, 1, last);
        if constexpr (SPLIT) {
            any_last<Real, -1>(buf, s, lg, PG);
            for (int e = threadIdx.x; e < ng * (h + 1); e += blockDim.x) {
                const int g = rdiv(e, mul_half), k = e - g * (h + 1);
                const C ck = any_ld(buf + any_freq_slot(s, k) * PG + g, C{});
                const C cn = any_conj(any_ld(buf + any_freq_slot(s, k ? n - k : 0) * PG + g, C{}));
                const C ev = any_half(cadd(ck, cn)), od = any_half(cmul_mi(csub(ck, cn)));
                const C wo = any_twmul<-1>(od, __ldg(tw + k));
                Cx2<Real> *dst = out + (r0 + g) * Px;
                dst[k] = any_ws(cadd(ev, wo), 0);
                if (2 * k != n) dst[n - k] = any_ws(any_conj(csub(ev, wo)), 0);
            }
        } else {
            __syncthreads();
            // The last stage with the split, neighbouring frequencies in a warp: butterfly f makes the
            // bins k = f + r P, its partner P - f the bins n - k.
            // X_k = Ev_k + W_{2n}^k Od_k, X_{n-k} = conj(Ev_k - W_{2n}^k Od_k), with Ev, Od the DFTs
            // of the even and odd samples from C_k and conj C_{n-k}.
            any_radix_last(s.r[last], [&]<int R>() {
                for (int e = threadIdx.x; e < ng * half; e += blockDim.x) {
                    const int g = rdiv(e, mul_half), f = e - g * half;
                    const bool own = f == 0 || 2 * f == P;  // n - k lies in butterfly f itself
                    C v[R], w[R];
                    const float4 *p = buf + any_freq_slot(s, f) * PG + g;
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = any_ld(p + r * PG, C{});
                    dft<R, -1>(v);
                    if (own) {
#pragma unroll
                        for (int r = 0; r < R; ++r) w[r] = f == 0 ? v[(r + 1) % R] : v[r];
                    } else {
                        p = buf + any_freq_slot(s, P - f) * PG + g;
#pragma unroll
                        for (int r = 0; r < R; ++r) w[r] = any_ld(p + r * PG, C{});
                        dft<R, -1>(w);
                    }
                    Cx2<Real> *dst = out + (r0 + W * g) * Px;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int k = f + r * P;
                        const C ck = v[r], cn = any_conj(w[R - 1 - r]);
                        const C ev = any_half(cadd(ck, cn)), od = any_half(cmul_mi(csub(ck, cn)));
                        const C wo = any_twmul<-1>(od, __ldg(tw + k));
                        const C lo = cadd(ev, wo), hi = any_conj(csub(ev, wo));
#pragma unroll
                        for (int i = 0; i < W; ++i) {
                            dst[(long long)i * Px + k] = any_ws(lo, i);
                            if (!own || k == 0) dst[(long long)i * Px + n - k] = any_ws(hi, i);
                        }
                    }
                }
            });
        }
    }
}

// ---- K5: x inverse ----------------------------------------------------------------------------
// The nx + 1 Hermitian bins of each row -> C_k = Ev_k + i Od_k (Ev_k = Y_k + conj Y_{n-k},
// Od_k = (Y_k - conj Y_{n-k}) W_{2n}^{-k}), the inverse nx-point FFT gives y_{2m} + i y_{2m+1};
// pairs m < nx/2 are kept (the crop).  Shared layout as in the forward.
template <typename Real, int MR, bool SPLIT>
__global__ void __launch_bounds__(kAnyThreads, kAnyMinBlocks<Real>)
k_any_x_inv(const Cx2<Real> *__restrict__ in, const PtrArray u, const AnyTw<Real> *__restrict__ tw,
            const __grid_constant__ AnySched s, int rows_b, int nrows, int Px, unsigned mul_half, int lg, int ntiles) {
    using C = typename Types<Real>::CC;
    using X2 = Ext2<Real>;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4 *buf = reinterpret_cast<float4 *>(smraw);
    const int n = s.L, h = n / 2, M = s.M[0], NG = 1 << lg, PG = NG + 1, TR = NG * W;
    const AnyTwiddles<Real> ts(tw, n, 2, buf + s.slots * PG);
    griddep_wait();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();  // the table is written, the previous tile's reads of buf are done
        const long long r0 = (long long)t * TR;
        const int ng = (int)min((long long)NG, (nrows - r0) / W);
        // The combination with the first stage of the inverse, as the forward's last one.
        const int last = s.nst - 1, P = s.P[last], half = P / 2 + 1;
        if constexpr (SPLIT) {
            for (int e = threadIdx.x; e < NG * (h + 1); e += blockDim.x) {
                const int g = rdiv(e, mul_half), k = e - g * (h + 1);
                const Cx2<Real> *src = in + (r0 + g) * Px;
                C yk = czero<C>(), yn = czero<C>();
                if (g < ng) {
                    yk = any_wpack(__ldg(src + k), __ldg(src + k), C{});
                    yn = any_wpack(__ldg(src + n - k), __ldg(src + n - k), C{});
                }
                if (k == 0) {  // Y_0 and Y_n are real, as below
                    yk.im = czero<C>().re;
                    yn.im = czero<C>().re;
                }
                const C cn = any_conj(yn), ev = cadd(yk, cn), od = any_twmul<1>(csub(yk, cn), __ldg(tw + k));
                any_st(buf + any_freq_slot(s, k) * PG + g, add_rot<1>(ev, od));
                if (k > 0 && 2 * k != n)
                    any_st(buf + any_freq_slot(s, n - k) * PG + g, add_rot<1>(any_conj(ev), any_conj(od)));
            }
            any_last<Real, 1>(buf, s, lg, PG);
        } else {
            any_radix_last(s.r[last], [&]<int R>() {
                for (int e = threadIdx.x; e < NG * half; e += blockDim.x) {
                    const int g = rdiv(e, mul_half), f = e - g * half;
                    const bool own = f == 0 || 2 * f == P;
                    const Cx2<Real> *src = in + (r0 + W * g) * Px;
                    C v[R], w[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int k = f + r * P;
                        v[r] = w[r] = czero<C>();
                        if (g < ng) {
                            v[r] = any_wpack(__ldg(src + k), __ldg(src + (W - 1) * Px + k), C{});
                            w[r] = any_wpack(__ldg(src + n - k), __ldg(src + (W - 1) * Px + n - k), C{});
                        }
                    }
                    if (f == 0) {  // Y_0 and Y_n are real: drop what rounding left in their imaginary parts
                        v[0].im = czero<C>().re;
                        w[0].im = czero<C>().re;
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const C cn = any_conj(w[r]), ev = cadd(v[r], cn);
                        const C od = any_twmul<1>(csub(v[r], cn), __ldg(tw + f + r * P));
                        v[r] = add_rot<1>(ev, od);
                        w[r] = add_rot<1>(any_conj(ev), any_conj(od));
                    }
                    dft<R, 1>(v);
                    float4 *p = buf + any_freq_slot(s, f) * PG + g;
#pragma unroll
                    for (int r = 0; r < R; ++r) any_st(p + r * PG, v[r]);
                    if (own) continue;
                    C x[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) x[r] = w[R - 1 - r];
                    dft<R, 1>(x);
                    p = buf + any_freq_slot(s, P - f) * PG + g;
#pragma unroll
                    for (int r = 0; r < R; ++r) any_st(p + r * PG, x[r]);
                }
            });
        }
        any_stages<Real, MR, 1>(buf, s, lg, PG, ts, 1, last);
        __syncthreads();
        {
            const int g = threadIdx.x & (NG - 1), step = s.S[0] * PG;
            any_radix_even<MR>(s.r[0], [&]<int R>() {
                constexpr int H = R / 2;
                for (int j = threadIdx.x >> lg; j < M; j += blockDim.x >> lg) {
                    float4 *p = buf + any_lo_slot(s, 0, j) * PG + g;
                    C v[R];
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        const int k = i < H ? 2 * i : 2 * (i - H) + 1;
                        v[i] = any_ld(p + k * step, C{});
                        if (k > 0) v[i] = any_twmul<1>(v[i], ts[k * j]);
                    }
                    any_dft_half_adj<R>(v);
#pragma unroll
                    for (int r = 0; r < H; ++r) any_st(p + r * step, v[r]);
                }
            });
        }
        __syncthreads();
        const AnyRows rows(r0, rows_b);
        any_radix_even<MR>(s.r[0], [&]<int R>() {
            for (int e = threadIdx.x; e < ng * M; e += blockDim.x) {
                const int g = rdiv(e, s.mulM[0]), j = e - g * M;
                if (!dbg_index_ok(rows.row(W * g), rows_b)) continue;
                X2 *dst = reinterpret_cast<X2 *>(const_cast<void *>(u.p[rows.density(W * g)])) + rows.row(W * g) * h + j;
                const float4 *p = buf + any_lo_slot(s, 0, j) * PG + g;
#pragma unroll
                for (int r = 0; r < R / 2; ++r) {
                    const C v = any_ld(p + r * s.S[0] * PG, C{});
#pragma unroll
                    for (int i = 0; i < W; ++i) dst[(long long)i * h + r * M] = any_ext(v, i);
                }
            }
        });
    }
}

// ---- K2 / K4: y passes --------------------------------------------------------------------------
// Tile (tx, plane): 2^lg groups of columns of one plane.  FWD: input rows < L/2 (the rest zero),
// all L rows stored; !FWD: all L input rows, rows < L/2 stored.
template <typename Real, int MR, bool FWD>
__global__ void __launch_bounds__(kAnyThreads, kAnyMinBlocks<Real>)
k_any_col(const Cx2<Real> *__restrict__ in, Cx2<Real> *__restrict__ out, const AnyTw<Real> *__restrict__ tw,
          const __grid_constant__ AnySched s, int ncols, int ntx, int Px, long long in_outer, long long out_outer, int lg, int ntiles) {
    using C = typename Types<Real>::CC;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4 *buf = reinterpret_cast<float4 *>(smraw);
    const int g = threadIdx.x & ((1 << lg) - 1);
    const AnyTwiddles<Real> ts(tw, s.L, 1, buf + (s.slots << lg));
    griddep_wait();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();  // the table is written, the previous tile's reads of buf are done
        const long long plane = t / ntx;
        const int col = (((int)(t - plane * ntx) << lg) + g) * W;
        const bool valid = col < ncols;
        const Cx2<Real> *src = in + plane * in_outer + (valid ? col : 0);
        Cx2<Real> *dst = out + plane * out_outer + (valid ? col : 0);
        const int last = s.nst - 1, nb = s.P[last], step = s.S[last];
        if constexpr (FWD) {
            any_first<Real, MR>(buf, s, lg, ts,
                                    [&](int row) { return valid ? ld_cc(src + (long long)row * Px) : czero<C>(); });
            any_stages<Real, MR, -1>(buf, s, lg, 1 << lg, ts, 1, last);
            __syncthreads();
            any_radix<MR>(s.r[last], [&]<int R>() {
                for (int b = threadIdx.x >> lg; b < nb; b += blockDim.x >> lg) {
                    const AnyBfly f = any_bfly(s, last, b);
                    C v[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = any_ld(buf + ((f.slot + r * step) << lg) + g, C{});
                    dft<R, -1>(v);
                    if (valid)
#pragma unroll
                        for (int r = 0; r < R; ++r) st_cc(dst + (long long)(f.freq + r * nb) * Px, v[r]);
                }
            });
        } else {
            any_radix<MR>(s.r[last], [&]<int R>() {
                for (int b = threadIdx.x >> lg; b < nb; b += blockDim.x >> lg) {
                    const AnyBfly f = any_bfly(s, last, b);
                    C v[R];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        v[r] = valid ? ld_cc(src + (long long)(f.freq + r * nb) * Px) : czero<C>();
                    dft<R, 1>(v);
#pragma unroll
                    for (int r = 0; r < R; ++r) any_st(buf + ((f.slot + r * step) << lg) + g, v[r]);
                }
            });
            any_stages<Real, MR, 1>(buf, s, lg, 1 << lg, ts, 1, last);
            any_first_adj<Real, MR>(buf, s, lg, ts, [&](int row, C x) {
                if (valid) st_cc(dst + (long long)row * Px, x);
            });
        }
    }
}

// ---- K3: z fused ------------------------------------------------------------------------------------
// Tile (tx, ky, b): 2^lg groups of columns kx of line ky of density b.  Forward length Lz = 2 nz
// (input z < nz), product with the symbol at (|kx|, |ky|, |kz|), inverse, z < nz stored.  With
// TAIL the forward spectrum's energy in the outer shell (|k_q| >= n_q - n_q / 8 on some axis)
// and its total energy go to its pair of tail (FP32 per thread, FP64 per tile, one atomic pair
// per tile).  The tiles cover the lines ky0 <= ky < ky0 + nky (all of them:
// ky0 = 0, nky = 2 ny, taken as ky and its mirror in turn, which read the same symbol rows; a
// rank's slab of lines in the slab decomposition of one solve).
template <typename Real, int MR, bool TAIL>
__global__ void __launch_bounds__(kAnyThreads, kAnyMinBlocks<Real>)
k_any_z(const Cx2<Real> *__restrict__ in, Cx2<Real> *__restrict__ out, const Real *__restrict__ sym,
        const AnyTw<Real> *__restrict__ tw, const __grid_constant__ AnySched s, int nx, int ny, int ntx, int Px, int Ps,
        double *__restrict__ tail, int ky0, int nky, int lg, int ntiles) {
    using C = typename Types<Real>::CC;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    float4 *buf = reinterpret_cast<float4 *>(smraw);
    const int Lz = s.L, nz = Lz / 2, Ly = 2 * ny;
    const int g = threadIdx.x & ((1 << lg) - 1);
    const AnyTwiddles<Real> ts(tw, s.L, 1, buf + (s.slots << lg));
    griddep_wait();
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        __syncthreads();  // the table is written, the previous tile's reads of buf are done
        const int line = t / ntx, bb = line / nky, li = line - bb * nky;
        const int ky = nky == Ly ? ((li & 1) ? Ly - ((li + 1) >> 1) : li >> 1) : ky0 + li;
        const int kya = ky <= ny ? ky : Ly - ky;
        const int col = (((t - line * ntx) << lg) + g) * W;
        const bool valid = col <= nx && dbg_index_ok(kya, ny + 1);
        const long long zs = (long long)Ly * Px;  // z stride of w2 and w3
        const long long base = ((long long)bb * nz * Ly + ky) * Px + (valid ? col : 0);
        const Real *srow = sym + (long long)kya * Ps + (valid ? col : 0);
        const long long splane = (long long)(ny + 1) * Ps;
        any_first<Real, MR>(buf, s, lg, ts, [&](int row) { return valid ? ld_cc(in + base + row * zs) : czero<C>(); });
        const int last = s.nst - 1, nb = s.P[last], step = s.S[last];
        any_stages<Real, MR, -1>(buf, s, lg, 1 << lg, ts, 1, last);
        __syncthreads();
        float eshell = 0.f, etot = 0.f;
        any_radix<MR>(s.r[last], [&]<int R>() {
            for (int b = threadIdx.x >> lg; b < nb; b += blockDim.x >> lg) {
                const AnyBfly f = any_bfly(s, last, b);
                float4 *p = buf + (f.slot << lg) + g;
                C v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = any_ld(p + ((r * step) << lg), C{});
                dft<R, -1>(v);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int k = f.freq + r * nb, kz = k <= nz ? k : Lz - k;
                    if constexpr (TAIL) {
                        const bool outer = kya >= ny - ny / 8 || kz >= nz - nz / 8;
                        auto add = [&](int kx, float en) {
                            const float e = kx > nx || !valid ? 0.f : (kx == 0 || kx == nx) ? en : 2.f * en;
                            etot += e;
                            if (outer || kx >= nx - nx / 8) eshell += e;
                        };
                        if constexpr (W == 2) {
                            const float2 en = cenergy(v[r]);
                            add(col, en.x);
                            add(col + 1, en.y);
                        } else {
                            add(col, cenergy(v[r]));
                        }
                    }
                    if (dbg_index_ok(kz, nz + 1)) v[r] = scale_sym(v[r], srow + kz * splane);
                }
                dft<R, 1>(v);
#pragma unroll
                for (int r = 0; r < R; ++r) any_st(p + ((r * step) << lg), v[r]);
            }
        });
        any_stages<Real, MR, 1>(buf, s, lg, 1 << lg, ts, 1, last);
        any_first_adj<Real, MR>(buf, s, lg, ts, [&](int row, C x) {
            if (valid) st_cc(out + base + row * zs, x);
        });
        if constexpr (TAIL) {
            double es = eshell, et = etot;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                es += __shfl_xor_sync(0xffffffffu, es, o);
                et += __shfl_xor_sync(0xffffffffu, et, o);
            }
            double *part = reinterpret_cast<double *>(buf);
            __syncthreads();  // the tile's last reads of buf are done
            if ((threadIdx.x & 31) == 0) {
                sm_st(part + 2 * (threadIdx.x >> 5), es);
                sm_st(part + 2 * (threadIdx.x >> 5) + 1, et);
            }
            __syncthreads();
            if (threadIdx.x < 2) {
                double sum = 0.0;
                for (unsigned w = 0; w < blockDim.x / 32; ++w) sum += sm_ld(part + 2 * w + threadIdx.x);
                atomicAdd(tail_pair(tail, bb) + threadIdx.x, sum);
            }
        }
    }
}

}  // namespace gsp
