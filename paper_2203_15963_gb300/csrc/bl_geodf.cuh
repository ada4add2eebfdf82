// Double-float Dormand-Prince geodesics (the fast form, and the work-ordered queue's prediction).
// Included by bl_kernels.cuh.
//
// What bounds it: instruction issue and dependent latency (57 % of the issue slots on one 256^2
// image with at most 12 resident warps an SM, which its 152 registers allow). sm_103a's packed FP32 instructions
// (fma/add/mul.f32x2) do two IEEE operations in one issue slot, so everything that is done alike
// for two components is packed: (x, y), (k_x, k_y) and (z, k_z) in the stage, error and midpoint
// sums, (x, y)-like pairs in the right-hand side. Each half of a packed operation is the scalar
// operation, and differences are taken as fma(b, -1, a), which rounds as a - b does: every result
// is bit-identical to the unpacked arithmetic (bl_df64.cuh). Double-precision instructions, 64
// cycles of a scheduler's FP64 share each, are kept out of the loop: comparisons on bit patterns,
// the segment length's quotient in FP32 (its double rounding through FP64 was innocuous: 53 >= 2 *
// 24 + 2 bits). Nine 256^2 images:
// 27.3 -> 22.7 ms, 1024^2 48.2 -> 39.7.
#pragma once

namespace bl {

// Two double-float values: the high words and the low words as packed pairs.
struct DFP {
    float2 h, l;
};
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ DFP df_dup(const df64& v) { return DFP{dup2(v.hi), dup2(v.lo)}; }
__device__ __forceinline__ DFP df_pair(const df64& a, const df64& b) {
    return DFP{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
}
__device__ __forceinline__ df64 df_first(const DFP& v) { return df64(v.h.x, v.l.x); }
__device__ __forceinline__ df64 df_second(const DFP& v) { return df64(v.h.y, v.l.y); }
__device__ __forceinline__ DFP df_swap(const DFP& v) {
    return DFP{make_float2(v.h.y, v.h.x), make_float2(v.l.y, v.l.x)};
}
__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(a, dup2(-1.0f)); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup2(-1.0f), a); }

// df_fast_two_sum, operator* and DFDot of bl_df64.cuh on pairs, operation for operation.
__device__ __forceinline__ DFP dfp_fast_two_sum(float2 a, float2 b) {
    const float2 s = __fadd2_rn(a, b);
    return DFP{s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ DFP dfp_mul(const DFP& x, const DFP& y) {
    const float2 p = __fmul2_rn(x.h, y.h);
    float2 lo = __ffma2_rn(x.h, y.h, neg2(p));
    lo = __ffma2_rn(x.h, y.l, lo);
    lo = __ffma2_rn(x.l, y.h, lo);
    return dfp_fast_two_sum(p, lo);
}
// df_mul_nn on pairs
__device__ __forceinline__ DFP dfp_mul_nn(const DFP& x, const DFP& y) {
    const float2 p = __fmul2_rn(x.h, y.h);
    float2 e = __ffma2_rn(x.h, y.h, neg2(p));
    e = __ffma2_rn(x.h, y.l, e);
    return DFP{p, __ffma2_rn(x.l, y.h, e)};
}
struct DFPDot {
    float2 s, c;
    __device__ __forceinline__ void first(const DFP& a, const DFP& x) {
        s = __fmul2_rn(a.h, x.h);
        c = __ffma2_rn(a.h, x.h, neg2(s));
        c = __ffma2_rn(a.h, x.l, c);
        c = __ffma2_rn(a.l, x.h, c);
    }
    // TwoSum of s and p, its error and the rest q into the low word
    __device__ __forceinline__ void two_sum(float2 p, float2 q) {
        const float2 t = __fadd2_rn(s, p);
        const float2 z = sub2(t, s);
        const float2 e = __fadd2_rn(sub2(s, sub2(t, z)), sub2(p, z));
        s = t;
        c = __fadd2_rn(c, __fadd2_rn(e, q));
    }
    __device__ __forceinline__ void add(const DFP& a, const DFP& x) {
        const float2 p = __fmul2_rn(a.h, x.h);
        float2 q = __ffma2_rn(a.h, x.h, neg2(p));
        q = __ffma2_rn(a.h, x.l, q);
        q = __ffma2_rn(a.l, x.h, q);
        two_sum(p, q);
    }
    __device__ __forceinline__ void add_term(const DFP& t) { two_sum(t.h, t.l); }
    __device__ __forceinline__ DFP get() const { return dfp_fast_two_sum(s, c); }
    __device__ __forceinline__ DFP axpy(const DFP& h, const DFP& y) const {
        const float2 p = __fmul2_rn(h.h, s);
        float2 q = __ffma2_rn(h.h, s, neg2(p));
        q = __ffma2_rn(h.h, c, q);
        q = __ffma2_rn(h.l, s, q);
        const float2 t = __fadd2_rn(y.h, p);
        const float2 z = sub2(t, y.h);
        const float2 e = __fadd2_rn(sub2(y.h, sub2(t, z)), sub2(p, z));
        return dfp_fast_two_sum(t, __fadd2_rn(__fadd2_rn(y.l, q), e));
    }
};

// State or derivative of a ray: x^t, then (x, y), (k_x, k_y), (z, k_z); k_t apart (constant).
struct StateDF {
    df64 t;
    DFP xy, kk, zk;
    __device__ __forceinline__ df64 get(int c) const {   // component c of (x^a, k_a), c != 4
        return c == 0 ? t : c == 1 ? df_first(xy) : c == 2 ? df_second(xy) : c == 3 ? df_first(zk)
             : c == 5 ? df_first(kk) : c == 6 ? df_second(kk) : df_second(zk);
    }
};

// Per-ray constants of the right-hand side.
struct RhsDF {
    df64 a, aa, m2;      // spin, its square, 2 M
    bool flat;
};

// Eq. (geodesic) in double-float, packed: the sums and products of geodesic_rhs64 (bl_geo64.cuh).
__device__ __forceinline__ df64 geodesic_rhs_df(const StateDF& S, const df64& kt, const RhsDF& C,
                                                StateDF& d) {
    const df64 x = df_first(S.xy), yy = df_second(S.xy), z = df_first(S.zk), kz = df_second(S.zk);
    const df64 a = C.a, aa = C.aa;
    const df64 q = g_dot3(x, x, yy, yy, z, z) - aa;
    const df64 aaz2 = g_mul_nn(aa, z) * z;
    const df64 D2 = g_fma(q, q, scale2(aaz2, 4.0f));
    const df64 iD = rsqrt(D2);
    const df64 r2 = scale2(g_fma(D2, iD, q), 0.5f);
    const df64 ir = rsqrt(r2);
    const df64 r = r2 * ir;
    const df64 s4 = g_fma(r2, r2, aaz2);
    const df64 P = r2 + aa;
    const df64 iPs = rcp(P * s4);
    const DFP inv = dfp_mul(df_pair(P, s4), df_dup(iPs));
    const df64 is4 = df_first(inv), iP = df_second(inv);
    // f = 2 M r^3 / s4 and d_z r = z P / (r D)
    const DFP fd = dfp_mul(dfp_mul_nn(dfp_mul_nn(df_pair(C.m2, z), df_pair(r, P)), df_pair(r2, ir)),
                           df_pair(is4, iD));
    const df64 f = C.flat ? df64(0.0f, 0.0f) : df_first(fd);
    const df64 drz = df_second(fd);
    const DFP rr = df_dup(r), ii = df_dup(iP);
    const DFP am = df_pair(a, -a);
    DFPDot D;
    // (l_x, l_y) = ((r x + a y), (r y - a x)) / P
    D.first(rr, S.xy);
    D.add(am, df_swap(S.xy));
    const DFP l = dfp_mul(D.get(), ii);
    // (l_z, k_z / r)
    const DFP lw = dfp_mul(S.zk, df_dup(ir));
    const df64 lz = df_first(lw), w = df_second(lw);
    // A = x k_x + y k_y, B = y k_x - x k_y
    const df64 kx = df_first(S.kk), ky = df_second(S.kk);
    D.first(S.xy, df_dup(kx));
    D.add(df_swap(S.xy), df_pair(ky, -ky));
    const DFP AB = D.get();
    const df64 A_ = df_first(AB), B_ = df_second(AB);
    const df64 Lxy = g_dot2(r, A_, a, B_) * iP;
    const df64 L = g_fma(lz, kz, Lxy - kt);
    const df64 fL = f * L;
    d.t = fL - kt;
    const df64 nfL = -fL;
    D.first(l, df_dup(nfL));
    D.add_term(S.kk);
    d.xy = D.get();
    const df64 dz = g_fma(lz, nfL, kz);
    // d_c r
    const df64 riD = r * iD;
    const DFP dr = dfp_mul(df_dup(riD), S.xy);
    // d_c L at fixed k, and d_c f: V and F1 / f together
    D.first(df_pair(g_fma(-scale2(r, 2.0f), Lxy, A_), df64(3.0f, 0.0f)), df_pair(iP, ir));
    D.add(df_pair(-w, -(scale2(r2, 4.0f) * r)), df_pair(lz, is4));
    const DFP VF = D.get();
    const df64 V = df_first(VF);
    D.first(rr, S.kk);
    D.add(df_swap(am), df_swap(S.kk));
    const DFP in = D.get();
    D.first(dr, df_dup(V));
    D.add(in, ii);
    const DFP Sxy = D.get();
    const df64 F1 = f * df_second(VF);
    const DFP df = dfp_mul(df_dup(F1), dr);
    // S_z = d_z r V + w and d_z f = F1 d_z r - 2 a^2 z f / s4
    D.first(df_pair(drz, F1), df_pair(V, drz));
    D.add_term(df_pair(w, -(g_mul_nn(g_mul_nn(scale2(aa, 2.0f), z), f) * is4)));
    const DFP Sd = D.get();
    const df64 Sz = df_first(Sd), dfz = df_second(Sd);
    const df64 halfL = scale2(L, 0.5f);
    D.first(df, df_dup(halfL));
    D.add(df_dup(f), Sxy);
    d.kk = dfp_mul(df_dup(L), D.get());
    d.zk = df_pair(dz, L * g_dot2(dfz, halfL, f, Sz));
    return r;
}

// Stage derivatives in dynamic shared memory, thread-fastest: three 16-byte pairs and one 8-byte
// x^t a stage (56 bytes, as 7 components).
struct KStoreDF {
    float4* p;
    float2* t;
    __device__ __forceinline__ void init(unsigned char* smem) {
        p = reinterpret_cast<float4*>(smem) + threadIdx.x;
        t = reinterpret_cast<float2*>(smem + 7 * 3 * 128 * sizeof(float4)) + threadIdx.x;
    }
    __device__ __forceinline__ DFP pair(int j, int k) const {
        const float4 v = p[(3 * j + k) * 128];
        return DFP{make_float2(v.x, v.y), make_float2(v.z, v.w)};
    }
    __device__ __forceinline__ df64 time(int j) const {
        const float2 v = t[j * 128];
        return df64(v.x, v.y);
    }
    __device__ __forceinline__ void put(int j, const StateDF& d) const {
        p[(3 * j) * 128] = make_float4(d.xy.h.x, d.xy.h.y, d.xy.l.x, d.xy.l.y);
        p[(3 * j + 1) * 128] = make_float4(d.kk.h.x, d.kk.h.y, d.kk.l.x, d.kk.l.y);
        p[(3 * j + 2) * 128] = make_float4(d.zk.h.x, d.zk.h.y, d.zk.l.x, d.zk.l.y);
        t[j * 128] = make_float2(d.t.hi, d.t.lo);
    }
    __device__ __forceinline__ StateDF get(int j) const {
        return StateDF{time(j), pair(j, 0), pair(j, 1), pair(j, 2)};
    }
};

// |h| < 1e-12 r in FP64, out of line (reached by rays whose step has all but underflowed).
__device__ __noinline__ bool below_step_limit(float ha, float r) {
    return (double)ha < 1e-12 * (double)r;
}

// The fast form's geodesics: state and stages in double-float, step control and records in FP32.
__device__ __forceinline__ void geodesic_df_body(const ImageDesc* __restrict__ imgs, int n_images,
                                                 int64_t ray_begin, int64_t ray_end,
                                                 RayHdr* __restrict__ hdr, RecordSink<float> sink,
                                                 int record, BlockSource bs,
                                                 const RayInit* __restrict__ init) {
    // rays [ray_begin, ray_end) of the batch form this wave; hdr, init and the chunk tables
    // are indexed by ray - ray_begin
    const int64_t re = wave_end(bs, ray_end);
    const int64_t total_rays = re > ray_begin ? re - ray_begin : 0;
    Counters* ctr = sink.ctr;
    bool active = false, exhausted = false;
    int64_t wray = 0, opix = 0;
    int q = 0, pi = 0, pj = 0;
    StateDF y;
    y.t = df64(0.0f, 0.0f);
    df64 kt(0.0f, 0.0f), h(0.0f, 0.0f);
    // K(0) = f(y); K(1..6) stage derivatives of the current attempt
    extern __shared__ __align__(16) unsigned char geo_smem[];
    KStoreDF K;
    K.init(geo_smem);
    double nnorm = 0.0;
    bool been_inside = false, prev_rej = false;
    int64_t attempts = 0, max_steps = 0;
    int32_t nrec = 0, status = 0;
    // radii compare with FP32 radii r: r < R exactly when r < R rounded up, r > R when r > R
    // rounded down
    float r_in_up = 0.0f, r_cam_up = 0.0f, r_cam_dn = 0.0f, r_grid_up = 0.0f;
    float tol_abs = 0.0f, tol_rel = 0.0f, ds_max = 0.0f;
    RhsDF C{df64(0.0f, 0.0f), df64(0.0f, 0.0f), df64(0.0f, 0.0f), false};
    float r_cur = 0.0f;     // r at y (of a ray's first point, which lies far out, rounded)
    bool near_grid = false; // r at y < r_max
    bool want_aux = false;  // auxiliary images: proper length and affine parameter
    double aux_len = 0.0, aux_lam = 0.0;

    // All 32 lanes stay in the loop until the whole warp is out of work, so the warp
    // reconverges every iteration and the attempt is issued once for all lanes that hold a
    // ray (lanes without one are masked).
    while (true) {
        const bool need = !active && !exhausted;
        const unsigned long long got = warp_refill(&ctr->next_ray_geo, need);
        if (need) {
            if ((int64_t)got >= total_rays) {
                exhausted = true;
            } else {
                wray = (int64_t)got;
                active = true;
            }
        }
        if (!__any_sync(0xffffffffu, active)) break;
        if (!active) continue;
        if (need) {   // a ray taken from the queue in this iteration: set it up
            setup_ray(imgs, n_images, bs, ray_begin + wray, q, opix, pi, pj);
            const ImageDesc& im = imgs[q];
            // the pixel's initial state, from ray_init_kernel (its FP64 set-up stays out of this
            // loop)
            const RayInit& ri = init[wray];
            y.t = df64(ri.y[0]);
            y.xy = df_pair(df64(ri.y[1]), df64(ri.y[2]));
            y.kk = df_pair(df64(ri.y[5]), df64(ri.y[6]));
            y.zk = df_pair(df64(ri.y[3]), df64(ri.y[7]));
            kt = df64(ri.y[4]);
            nnorm = ri.nnorm;
            C.a = df64(im.spin);
            C.aa = C.a * C.a;
            C.m2 = scale2(df64(im.mass), 2.0f);
            C.flat = im.flat != 0;
            r_cam_up = __double2float_ru(im.r_cam);
            r_cam_dn = __double2float_rd(im.r_cam);
            r_in_up = __double2float_ru(im.r_in_over_rhor * im.r_hor);
            r_grid_up = __double2float_ru(im.r_max);
            ds_max = (float)im.ds_max;
            tol_abs = (float)im.tol_abs;
            tol_rel = (float)im.tol_rel;
            max_steps = im.max_steps;
            want_aux = record && im.aux != nullptr;
            aux_len = aux_lam = 0.0;
            h = df64(-im.h0_frac * (im.r_cam - im.r_hor));
            prev_rej = false;
        }
        // ---- one Dormand-Prince attempt (Table tab:dp) ----
        // Rolled stage loop: one right-hand-side body run six times keeps the kernel small
        // enough for the instruction cache. K(0) holds f(y) (first same as last), K(s) the
        // stage derivatives; stage 6 is evaluated at the fifth-order solution y5. A ray's first
        // attempt starts at stage 0, which evaluates f(y) at the stage point y, so that the
        // set-up path needs no copy of the right-hand side.
        StateDF ys;
        float r5 = 0.0f;
#pragma unroll 1
        for (int st = need ? 0 : 1; st < 7; ++st) {
            if (st == 0) {
                ys = y;
            } else {
                // earlier stages outer (rolled), components inner: each coefficient is read
                // once per stage term; every component keeps its order of operations
                DFPDot a0, a1, a2;
                {
                    const DFP cc = df_dup(DPCoef<df64>::a(st, 0));
                    a0.first(cc, K.pair(0, 0));
                    a1.first(cc, K.pair(0, 1));
                    a2.first(cc, K.pair(0, 2));
                }
                // the last row's second coefficient (b_2 of the fifth-order weights) is zero
#pragma unroll 1
                for (int j = st == 6 ? 2 : 1; j < st; ++j) {
                    const DFP cc = df_dup(DPCoef<df64>::a(st, j));
                    a0.add(cc, K.pair(j, 0));
                    a1.add(cc, K.pair(j, 1));
                    a2.add(cc, K.pair(j, 2));
                }
                const DFP hh = df_dup(h);
                ys.xy = a0.axpy(hh, y.xy);
                ys.kk = a1.axpy(hh, y.kk);
                ys.zk = a2.axpy(hh, y.zk);
            }
            StateDF fs;
            const df64 rr = geodesic_rhs_df(ys, kt, C, fs);
            K.put(st, fs);
            if (st == 0) {
                const double r0 = df_to_double(rr);
                been_inside = r0 < imgs[q].r_cam;
                near_grid = r0 < imgs[q].r_max;
                r_cur = rr.hi + rr.lo;
            }
            r5 = rr.hi + rr.lo;
        }
        // x^t at the fifth-order solution (the right-hand side does not read it)
        {
            DFDot at;
            at.first(DPCoef<df64>::a(6, 0), K.time(0));
#pragma unroll 1
            for (int j = 2; j < 6; ++j) at.add(DPCoef<df64>::a(6, j), K.time(j));
            ys.t = at.axpy(h, y.t);
        }
        const StateDF& y5 = ys;
        // Error norm eps = max_c |y5_c - y4_c| / (f_abs + f_rel max(|y_c|, |y5_c|)) with
        // y5 - y4 = h sum (b5 - b4) k, used in FP32 only: h_hi (s + c) (it only steers the step
        // size).
        const float hf = h.hi + h.lo;
        float eps;
        bool finite = true;
        {
            DFPDot a0, a1, a2;
            DFDot at;
            {
                const df64 c = DPCoef<df64>::e(0);
                const DFP cc = df_dup(c);
                a0.first(cc, K.pair(0, 0));
                a1.first(cc, K.pair(0, 1));
                a2.first(cc, K.pair(0, 2));
                at.first(c, K.time(0));
            }
#pragma unroll 1
            for (int j = 2; j < 7; ++j) {
                const df64 c = DPCoef<df64>::e(j);
                const DFP cc = df_dup(c);
                a0.add(cc, K.pair(j, 0));
                a1.add(cc, K.pair(j, 1));
                a2.add(cc, K.pair(j, 2));
                at.add(c, K.time(j));
            }
            const float2 e0 = __fmul2_rn(dup2(hf), __fadd2_rn(a0.s, a0.c));
            const float2 e1 = __fmul2_rn(dup2(hf), __fadd2_rn(a1.s, a1.c));
            const float2 e2 = __fmul2_rn(dup2(hf), __fadd2_rn(a2.s, a2.c));
            const float errf[8] = {hf * (at.s + at.c), e0.x, e0.y, e2.x, 0.0f, e1.x, e1.y, e2.y};
            float num = 0.0f, den = 1.0f;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c == 4) continue;   // (k_t: no difference)
                const df64 yc = y.get(c), zc = y5.get(c);
                const float yn = zc.hi + zc.lo;
                const float err = fabsf(errf[c]);
                const float sc = tol_abs + tol_rel * fmaxf(fabsf(yc.hi + yc.lo), fabsf(yn));
                finite = finite && isfinite(err) && isfinite(yn);
                if (err * den > num * sc) { num = err; den = sc; }
            }
            eps = num / den;
        }
        ++attempts;
        bool done = false;
        if (!finite) {
            status = BL_RAY_NAN;
            done = true;
        } else if (eps <= 1.0f) {
            // accepted: samples of this step (camera side first). The midpoint's increment
            // (h/2) sum_j b_mid,j k_j and the quartic coefficients are formed in FP32 from the
            // state; they move a record by about one FP32 ulp and leave the integration and
            // its step decisions untouched.
            if (record) {
                float ymf[8], incm[8];
                {
                    const float hh = 0.5f * hf;
                    float2 m0, m1, m2;
                    float mt;
                    auto sum = [](const DFP& v) { return __fadd2_rn(v.h, v.l); };
                    {
                        const float c = c_dpf.m[0].x;
                        const df64 t = K.time(0);
                        m0 = __fmul2_rn(dup2(c), sum(K.pair(0, 0)));
                        m1 = __fmul2_rn(dup2(c), sum(K.pair(0, 1)));
                        m2 = __fmul2_rn(dup2(c), sum(K.pair(0, 2)));
                        mt = c * (t.hi + t.lo);
                    }
#pragma unroll 1
                    for (int j = 2; j < 7; ++j) {
                        const float c = c_dpf.m[j].x;
                        const df64 t = K.time(j);
                        m0 = __ffma2_rn(dup2(c), sum(K.pair(j, 0)), m0);
                        m1 = __ffma2_rn(dup2(c), sum(K.pair(j, 1)), m1);
                        m2 = __ffma2_rn(dup2(c), sum(K.pair(j, 2)), m2);
                        mt = fmaf(c, t.hi + t.lo, mt);
                    }
                    const float acc[8] = {mt, m0.x, m0.y, m2.x, 0.0f, m1.x, m1.y, m2.y};
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const df64 yc = c == 4 ? kt : y.get(c);
                        incm[c] = hh * acc[c];
                        ymf[c] = yc.hi + (yc.lo + incm[c]);
                    }
                }
                float rmid, kt_up, fmid;
                {
                    KSGeom<float> Gm;
                    ks_geom<float>(ymf[1], ymf[2], ymf[3], imgs[q].f_c[kcSpin], imgs[q].f_c[kcMass],
                                   C.flat, Gm);
                    const float L = -ymf[4] + Gm.l[1] * ymf[5] + Gm.l[2] * ymf[6] + Gm.l[3] * ymf[7];
                    kt_up = -ymf[4] + Gm.f * L;
                    rmid = Gm.r;
                    fmid = Gm.f;
                }
                const float hl = fabsf(hf);
                if (want_aux) {
                    aux_lam += fabs((double)hf);
                    aux_len += fabs((double)hf) * fabs((double)kt_up) / sqrt(1.0 + (double)fmid);
                }
                int nsub = 1;
                if (near_grid || fminf(rmid, r5) < r_grid_up) {
                    // ds/dl = (g_pq k^p k^q)^1/2 = alpha |k^t| for a null ray
                    const float ds = hl * fabsf(kt_up) * rsqrtf(1.0f + fmid);
                    if (ds > ds_max) {
                        const float nd = ceilf(ds / ds_max);
                        nsub = nd > 4096.0f ? 4097 : (int)nd;
                    }
                }
                bool ok = true;
                if (nsub == 1) {
                    float yf[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const df64 yc = c == 4 ? kt : y.get(c);
                        yf[c] = yc.hi + yc.lo;
                    }
                    ok = append_record(sink, wray, nrec, ymf, yf, hl);
                } else {
                    // the quartic through y0, y1, h f0, h f1 and y_mid (Shampine 1986), in FP32
                    // about y0 (y_mid - y0 is the midpoint increment)
                    float y0f[8], d0f[8], c2f[8], c3f[8], c4f[8];
                    const StateDF f0 = K.get(0), f6 = K.get(6);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        if (c == 4) {
                            y0f[c] = d0f[c] = c2f[c] = c3f[c] = c4f[c] = 0.0f;   // not recorded
                            continue;
                        }
                        const df64 yc = y.get(c), zc = y5.get(c), k0 = f0.get(c), k6 = f6.get(c);
                        const df64 dy = zc - yc;
                        const float d0 = hf * (k0.hi + k0.lo);
                        const float D1 = (dy.hi + dy.lo) - d0;
                        const float D2 = hf * (k6.hi + k6.lo) - d0;
                        const float D3 = incm[c] - 0.5f * d0;
                        y0f[c] = yc.hi + yc.lo;
                        d0f[c] = d0;
                        c2f[c] = -5.0f * D1 + D2 + 16.0f * D3;
                        c3f[c] = 14.0f * D1 - 3.0f * D2 - 32.0f * D3;
                        c4f[c] = -8.0f * D1 + 2.0f * D2 + 16.0f * D3;
                    }
                    ok = emit_quartic_f(sink, wray, nrec, y0f, d0f, c2f, c3f, c4f, nsub, hl / (float)nsub);
                }
                if (!ok) { status = BL_RAY_OVERFLOW; done = true; }
            }
            y = y5;
            K.put(0, K.get(6));
            float fac = (eps == 0.0f) ? 10.0f : 0.9f * powf(eps, -0.2f);
            fac = fminf(10.0f, fmaxf(0.2f, fac));
            if (prev_rej) fac = fminf(fac, 1.0f);
            h = h * df64(fac);
            prev_rej = false;
            r_cur = r5;
            near_grid = r5 < r_grid_up;
            if (!done) {
                if (r5 < r_in_up) { status = BL_RAY_HORIZON; done = true; }
                else if (been_inside && r5 > r_cam_dn) { status = BL_RAY_ESCAPED; done = true; }
                else if (r5 < r_cam_up) been_inside = true;
            }
        } else {
            h = h * df64(fmaxf(0.2f, 0.9f * powf(eps, -0.2f)));
            prev_rej = true;
        }
        if (!done) {
            // |h| < 1e-12 r in FP64; in FP32 it is decided unless the two are close
            const float ha = fabsf(h.hi + h.lo);
            if (ha < 1.001e-12f * r_cur && below_step_limit(ha, r_cur)) {
                status = BL_RAY_UNDERFLOW;
                done = true;
            }
            else if (attempts >= max_steps) { status = BL_RAY_MAX_STEPS; done = true; }
        }
        if (done) {
            const ImageDesc& im = imgs[q];
            const int64_t pix = opix;
            if (im.status) im.status[pix] = status;
            if (im.steps) im.steps[pix] = (int32_t)(attempts < 2147483647 ? attempts : 2147483647);
            if (im.end_state)
#pragma unroll
                for (int c = 0; c < 8; ++c) im.end_state[pix * 8 + c] = df_to_double(c == 4 ? kt : y.get(c));
            if (im.samples) im.samples[pix] = nrec;
            if (want_aux) {
                aux_store(im, 0, pix, -df_to_double(y.t));
                aux_store(im, 1, pix, aux_len);
                aux_store(im, 2, pix, aux_lam);
            }
            RayHdr hd;
            hd.kt = df_to_double(kt);
            hd.nnorm = nnorm;
            hd.nrec = nrec;
            hd.status = status;
            hd.last_in = nrec - 1;   // (not tracked in this form: the transfer starts at the far end)
            hdr[wray] = hd;
            if (status != BL_RAY_HORIZON && status != BL_RAY_ESCAPED)
                atomicAdd(&ctr->bad_rays, 1ull);
            active = false;
            attempts = 0;
            nrec = 0;
            status = 0;
        }
    }
}

}  // namespace bl
