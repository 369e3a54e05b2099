// The x and y passes of small planes in one kernel per direction, with runtime lengths.
//
// A CTA owns one z-plane: it brings the plane's rows into shared memory, transforms them (K1),
// leaves the Hermitian bins in the column layout of the y transform, transforms the columns
// (K2) and writes the y-spectrum; the inverse runs the adjoint steps back (K4, K5).  The x
// spectrum never leaves shared memory and a solve takes three launches instead of five.  The
// stages are those of passes_any.cuh on 16-byte groups: pairs of rows along x and pairs of
// columns along y in FP32, one row or column otherwise.
//
// What bounds them: latency.  A plane of 32 x 32 is a tenth of the arithmetic an SM does in the
// time of one launch; the kernels are a chain of five to seven block barriers.
#pragma once

namespace gsp {

// Groups of a tile along one axis: item e is butterfly e / G, group e mod G.
struct PlaneGroups {
    int G;
    unsigned mul;
    int pitch;
};
template <class F> __device__ __forceinline__ void plane_each(int nb, const PlaneGroups &q, F &&f) {
    for (int e = threadIdx.x; e < nb * q.G; e += blockDim.x) {
        const int b = rdiv(e, q.mul);
        f(b, e - b * q.G);
    }
}

// Middle stages st0 <= st < st1, each behind a block barrier.
template <typename Real, int MR, int D>
__device__ __forceinline__ void plane_stages(float4 *buf, const AnySched &s, const PlaneGroups &q,
                                             const AnyTwiddles<Real> &tw, int st0, int st1) {
    using C = typename Types<Real>::CC;
    for (int i = st0; i < st1; ++i) {
        const int st = D < 0 ? i : st0 + st1 - 1 - i;
        __syncthreads();
        any_radix<MR>(s.r[st], [&]<int R>() {
            plane_each(s.P[st] * s.M[st], q, [&](int b, int g) {
                const AnyBfly f = any_bfly(s, st, b);
                any_stage<R, D>(buf + f.slot * q.pitch + g, s.S[st] * q.pitch, tw, f.lo * s.P[st], C{});
            });
        });
    }
}
// First forward stage in place (times j + r M_0, r < R_0 / 2) and its adjoint.
template <typename Real, int MR, int D>
__device__ __forceinline__ void plane_first(float4 *buf, const AnySched &s, const PlaneGroups &q,
                                            const AnyTwiddles<Real> &tw) {
    using C = typename Types<Real>::CC;
    const int step = s.S[0] * q.pitch;
    __syncthreads();
    any_radix_even<MR>(s.r[0], [&]<int R>() {
        constexpr int H = R / 2;
        plane_each(s.M[0], q, [&](int j, int g) {
            float4 *p = buf + any_lo_slot(s, 0, j) * q.pitch + g;
            C v[R];
            if constexpr (D < 0) {
#pragma unroll
                for (int r = 0; r < H; ++r) v[r] = any_ld(p + r * step, C{});
                any_dft_half<R>(v);
            }
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int k = i < H ? 2 * i : 2 * (i - H) + 1;
                if constexpr (D < 0) {
                    any_st(p + k * step, k == 0 ? v[i] : any_twmul<-1>(v[i], tw[k * j]));
                } else {
                    v[i] = any_ld(p + k * step, C{});
                    if (k > 0) v[i] = any_twmul<1>(v[i], tw[k * j]);
                }
            }
            if constexpr (D > 0) {
                any_dft_half_adj<R>(v);
#pragma unroll
                for (int r = 0; r < H; ++r) any_st(p + r * step, v[r]);
            }
        });
    });
}

// Bin k of rows W g + i (slots a and b of the y buffer, in groups) as a row group.
__device__ __forceinline__ CV plane_ld(const float4 *yb, int a, int b, int k, CV) {
    const float *p = reinterpret_cast<const float *>(yb + a + (k >> 1)) + (k & 1);
    const float *q = reinterpret_cast<const float *>(yb + b + (k >> 1)) + (k & 1);
    return {f2(sm_ld(p), sm_ld(q)), f2(sm_ld(p + 2), sm_ld(q + 2))};
}
__device__ __forceinline__ void plane_st(float4 *yb, int a, int b, int k, CV x) {
    float *p = reinterpret_cast<float *>(yb + a + (k >> 1)) + (k & 1);
    float *q = reinterpret_cast<float *>(yb + b + (k >> 1)) + (k & 1);
    sm_st(p, x.re.x);
    sm_st(p + 2, x.im.x);
    sm_st(q, x.re.y);
    sm_st(q + 2, x.im.y);
}
template <typename C> __device__ __forceinline__ C plane_ld(const float4 *yb, int a, int, int k, C) {
    return any_ld(yb + a + k, C{});
}
template <typename C> __device__ __forceinline__ void plane_st(float4 *yb, int a, int, int k, C x) {
    any_st(yb + a + k, x);
}
// Slot of time index t < L / 2.
__device__ __forceinline__ int plane_time_slot(const AnySched &s, int t) {
    const int d = rdiv(t, s.mulM[0]);
    return d * s.S[0] + any_lo_slot(s, 0, t - d * s.M[0]);
}

// Schedules and groups of a plane: x (length nx, ny / W row groups), y (length 2 ny, the
// (nx + W) / W column groups that hold the nx + 1 bins).
struct PlaneArgs {
    AnySched sx, sy;
    PlaneGroups qx, qy;
    unsigned mul_half;  // reciprocal of sx.P[last] / 2 + 1
    int nz, Px;
};

template <typename Real> constexpr int kPlaneMinBlocks = sizeof(typename Types<Real>::CS) == 8 ? 2 : 1;

// ---- K1 + K2 --------------------------------------------------------------------------------------
template <typename Real, int MR>
__global__ void __launch_bounds__(kPlaneThreads, kPlaneMinBlocks<Real>)
k_plane_fwd(const PtrArray rho, Cx2<Real> *__restrict__ w2, const AnyTw<Real> *__restrict__ tw_x,
            const AnyTw<Real> *__restrict__ tw_y, const __grid_constant__ PlaneArgs a) {
    using C = typename Types<Real>::CC;
    using X2 = Ext2<Real>;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    const AnySched &sx = a.sx, &sy = a.sy;
    float4 *xb = reinterpret_cast<float4 *>(smraw), *yb = xb + sx.slots * a.qx.pitch, *tb = yb + sy.slots * a.qy.pitch;
    const int n = sx.L, h = n / 2, M = sx.M[0], ny = sy.L / 2;
    const AnyTwiddles<Real> tx(tw_x, n, 2, tb), ty(tw_y, sy.L, 1, tb + any_tw_bytes<Real>(n) / 16);
    griddep_wait();
    const int pl = blockIdx.x, b = pl / a.nz, z = pl - b * a.nz;
    const X2 *plane = reinterpret_cast<const X2 *>(rho.p[b]) + (long long)z * ny * h;
    any_radix_even<MR>(sx.r[0], [&]<int R>() {
        for (int e = threadIdx.x; e < a.qx.G * M; e += blockDim.x) {
            const int g = rdiv(e, sx.mulM[0]), j = e - g * M;
            const X2 *src = plane + (long long)W * g * h + j;
            C v[R / 2];
#pragma unroll
            for (int r = 0; r < R / 2; ++r) {
                const X2 x = __ldg(src + r * M);
                v[r] = any_pack(x, W == 2 ? __ldg(src + h + r * M) : x, C{});
            }
            float4 *p = xb + any_lo_slot(sx, 0, j) * a.qx.pitch + g;
#pragma unroll
            for (int r = 0; r < R / 2; ++r) any_st(p + r * sx.S[0] * a.qx.pitch, v[r]);
        }
    });
    plane_first<Real, MR, -1>(xb, sx, a.qx, tx);
    const int last = sx.nst - 1, P = sx.P[last], half = P / 2 + 1;
    plane_stages<Real, MR, -1>(xb, sx, a.qx, tx, 1, last);
    __syncthreads();
    // The last x stage with the Hermitian split (as in k_any_x_fwd), into the y buffer.
    any_radix_last(sx.r[last], [&]<int R>() {
        for (int e = threadIdx.x; e < a.qx.G * half; e += blockDim.x) {
            const int g = rdiv(e, a.mul_half), f = e - g * half;
            const bool own = f == 0 || 2 * f == P;
            C v[R], w[R];
            const float4 *p = xb + any_freq_slot(sx, f) * a.qx.pitch + g;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = any_ld(p + r * a.qx.pitch, C{});
            dft<R, -1>(v);
            if (own) {
#pragma unroll
                for (int r = 0; r < R; ++r) w[r] = f == 0 ? v[(r + 1) % R] : v[r];
            } else {
                p = xb + any_freq_slot(sx, P - f) * a.qx.pitch + g;
#pragma unroll
                for (int r = 0; r < R; ++r) w[r] = any_ld(p + r * a.qx.pitch, C{});
                dft<R, -1>(w);
            }
            const int s0 = plane_time_slot(sy, W * g) * a.qy.pitch;
            const int s1 = W == 2 ? plane_time_slot(sy, W * g + 1) * a.qy.pitch : s0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = f + r * P;
                const C ck = v[r], cn = any_conj(w[R - 1 - r]);
                const C ev = any_half(cadd(ck, cn)), od = any_half(cmul_mi(csub(ck, cn)));
                const C wo = any_twmul<-1>(od, __ldg(tw_x + k));
                plane_st(yb, s0, s1, k, cadd(ev, wo));
                if (!own || k == 0) plane_st(yb, s0, s1, n - k, any_conj(csub(ev, wo)));
                if (W == 2 && k == 0) plane_st(yb, s0, s1, n + 1, czero<C>());  // the last pair's second column
            }
        }
    });
    plane_first<Real, MR, -1>(yb, sy, a.qy, ty);
    const int lasty = sy.nst - 1, nb = sy.P[lasty];
    plane_stages<Real, MR, -1>(yb, sy, a.qy, ty, 1, lasty);
    __syncthreads();
    Cx2<Real> *dst = w2 + (long long)pl * sy.L * a.Px;
    any_radix<MR>(sy.r[lasty], [&]<int R>() {
        plane_each(nb, a.qy, [&](int bf, int g) {
            const AnyBfly f = any_bfly(sy, lasty, bf);
            const float4 *p = yb + f.slot * a.qy.pitch + g;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = any_ld(p + r * a.qy.pitch, C{});
            dft<R, -1>(v);
#pragma unroll
            for (int r = 0; r < R; ++r) st_cc(dst + (long long)(f.freq + r * nb) * a.Px + W * g, v[r]);
        });
    });
}

// ---- K4 + K5 --------------------------------------------------------------------------------------
template <typename Real, int MR>
__global__ void __launch_bounds__(kPlaneThreads, kPlaneMinBlocks<Real>)
k_plane_inv(const Cx2<Real> *__restrict__ w3, const PtrArray u, const AnyTw<Real> *__restrict__ tw_x,
            const AnyTw<Real> *__restrict__ tw_y, const __grid_constant__ PlaneArgs a) {
    using C = typename Types<Real>::CC;
    using X2 = Ext2<Real>;
    constexpr int W = Types<Real>::W;
    extern __shared__ __align__(16) unsigned char smraw[];
    const AnySched &sx = a.sx, &sy = a.sy;
    float4 *xb = reinterpret_cast<float4 *>(smraw), *yb = xb + sx.slots * a.qx.pitch, *tb = yb + sy.slots * a.qy.pitch;
    const int n = sx.L, h = n / 2, M = sx.M[0], ny = sy.L / 2;
    const AnyTwiddles<Real> tx(tw_x, n, 2, tb), ty(tw_y, sy.L, 1, tb + any_tw_bytes<Real>(n) / 16);
    griddep_wait();
    const int pl = blockIdx.x, b = pl / a.nz, z = pl - b * a.nz;
    const Cx2<Real> *src = w3 + (long long)pl * sy.L * a.Px;
    const int lasty = sy.nst - 1, nb = sy.P[lasty];
    any_radix<MR>(sy.r[lasty], [&]<int R>() {
        plane_each(nb, a.qy, [&](int bf, int g) {
            const AnyBfly f = any_bfly(sy, lasty, bf);
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = ld_cc(src + (long long)(f.freq + r * nb) * a.Px + W * g);
            dft<R, 1>(v);
            float4 *p = yb + f.slot * a.qy.pitch + g;
#pragma unroll
            for (int r = 0; r < R; ++r) any_st(p + r * a.qy.pitch, v[r]);
        });
    });
    plane_stages<Real, MR, 1>(yb, sy, a.qy, ty, 1, lasty);
    plane_first<Real, MR, 1>(yb, sy, a.qy, ty);
    __syncthreads();
    // The combination with the first stage of the x inverse (as in k_any_x_inv).
    const int last = sx.nst - 1, P = sx.P[last], half = P / 2 + 1;
    any_radix_last(sx.r[last], [&]<int R>() {
        for (int e = threadIdx.x; e < a.qx.G * half; e += blockDim.x) {
            const int g = rdiv(e, a.mul_half), f = e - g * half;
            const bool own = f == 0 || 2 * f == P;
            const int s0 = plane_time_slot(sy, W * g) * a.qy.pitch;
            const int s1 = W == 2 ? plane_time_slot(sy, W * g + 1) * a.qy.pitch : s0;
            C v[R], w[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int k = f + r * P;
                C yk = plane_ld(yb, s0, s1, k, C{}), yn = plane_ld(yb, s0, s1, n - k, C{});
                if (k == 0) {  // Y_0 and Y_n are real: drop what rounding left in their imaginary parts
                    yk.im = czero<C>().re;
                    yn.im = czero<C>().re;
                }
                const C cn = any_conj(yn), ev = cadd(yk, cn);
                const C od = any_twmul<1>(csub(yk, cn), __ldg(tw_x + k));
                v[r] = add_rot<1>(ev, od);
                w[R - 1 - r] = add_rot<1>(any_conj(ev), any_conj(od));
            }
            dft<R, 1>(v);
            float4 *p = xb + any_freq_slot(sx, f) * a.qx.pitch + g;
#pragma unroll
            for (int r = 0; r < R; ++r) any_st(p + r * a.qx.pitch, v[r]);
            if (own) continue;
            dft<R, 1>(w);
            p = xb + any_freq_slot(sx, P - f) * a.qx.pitch + g;
#pragma unroll
            for (int r = 0; r < R; ++r) any_st(p + r * a.qx.pitch, w[r]);
        }
    });
    plane_stages<Real, MR, 1>(xb, sx, a.qx, tx, 1, last);
    plane_first<Real, MR, 1>(xb, sx, a.qx, tx);
    __syncthreads();
    X2 *plane = reinterpret_cast<X2 *>(const_cast<void *>(u.p[b])) + (long long)z * ny * h;
    any_radix_even<MR>(sx.r[0], [&]<int R>() {
        for (int e = threadIdx.x; e < a.qx.G * M; e += blockDim.x) {
            const int g = rdiv(e, sx.mulM[0]), j = e - g * M;
            X2 *dst = plane + (long long)W * g * h + j;
            const float4 *p = xb + any_lo_slot(sx, 0, j) * a.qx.pitch + g;
#pragma unroll
            for (int r = 0; r < R / 2; ++r) {
                const C v = any_ld(p + r * sx.S[0] * a.qx.pitch, C{});
#pragma unroll
                for (int i = 0; i < W; ++i) dst[(long long)i * h + r * M] = any_ext(v, i);
            }
        }
    });
}

template <typename Real, int MR>
cudaError_t plane_run(const DevicePlan &p, const PtrArray &rho, const PtrArray &u, int B, cudaStream_t s, bool fwd) {
    const PlaneTile &t = p.plane[std::is_same<Real, DF>::value];
    auto groups = [](int G, int pitch) { return PlaneGroups{G, (unsigned)((1ull << 32) / (unsigned)G + 1), pitch}; };
    PlaneArgs a{t.sx, t.sy, groups(t.gx, t.px), groups(t.gy, t.py), 0u, p.n3[2], p.Px};
    a.mul_half = (unsigned)((1ull << 32) / (unsigned)(t.sx.P[t.sx.nst - 1] / 2 + 1) + 1);
    const AnyTw<Real> *tx = static_cast<const AnyTw<Real> *>(p.tw3[0]);
    const AnyTw<Real> *ty = static_cast<const AnyTw<Real> *>(p.tw3[1]);
    const int smem = t.smem + any_tw_bytes<Real>(t.sx.L) + any_tw_bytes<Real>(t.sy.L), planes = B * p.n3[2];
    if (fwd) {
        GSP_CHECK(set_smem(k_plane_fwd<Real, MR>, smem));
        GSP_CHECK(launch_pdl(k_plane_fwd<Real, MR>, planes, t.threads, smem, s, rho, static_cast<Cx2<Real> *>(p.w2), tx, ty, a));
    } else {
        GSP_CHECK(set_smem(k_plane_inv<Real, MR>, smem));
        GSP_CHECK(launch_pdl(k_plane_inv<Real, MR>, planes, t.threads, smem, s, static_cast<const Cx2<Real> *>(p.w3), u, tx, ty, a));
    }
    return cudaGetLastError();
}

template <typename Real>
cudaError_t plane_xy(const DevicePlan &p, const PtrArray &rho, const PtrArray &u, int B, cudaStream_t s, bool fwd) {
    const PlaneTile &t = p.plane[std::is_same<Real, DF>::value];
    return any_with_radix<Real>(t.mr, [&]<int MR>() { return plane_run<Real, MR>(p, rho, u, B, s, fwd); });
}

}  // namespace gsp
