// Native-double Dormand-Prince geodesics (the FP64 and mixed forms). Included by bl_kernels.cuh.
//
// What bounds it: GB300 has two FP64 lanes an SM, so a warp's FP64 instruction occupies its
// scheduler's share of the pipe for 64 cycles whatever its active lanes, its dependences or its
// instruction mix (measured: 64.3 cycles an instruction for one warp a scheduler with 1 to 8
// independent chains and 1 to 32 active lanes; 76 with all four schedulers busy). The time of an
// attempt is its FP64 instruction count, from one resident ray to a full machine. So everything
// here that a double-precision pipe instruction is not needed for is done in integer
// instructions on the bit patterns (scaling by powers of two, maxima and comparisons of
// non-negative values, float <-> double conversions, finiteness), sums whose results are not
// read are left out (the time coordinate's stage sums of stages 1-5, its sub-samples without
// slow light), and the decision into how many samples a step splits is taken in FP32 with an
// error bound, in FP64 only where the bound cannot decide. None of it changes a bit of any
// result.
#pragma once

namespace bl {

// x 2^k for a normal x whose result is normal (one integer add on the exponent field).
__device__ __forceinline__ double scale_exp(double x, int k) {
    return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}
__device__ __forceinline__ long long abs_bits(double x) {
    return __double_as_longlong(x) & 0x7fffffffffffffffll;
}
// a > b, max and min of non-negative doubles on their bit patterns (the order of non-negative
// IEEE values is the order of their bits).
__device__ __forceinline__ bool gt_nonneg(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b);
}
__device__ __forceinline__ double max_abs(double a, double b) {
    const long long x = abs_bits(a), y = abs_bits(b);
    return __longlong_as_double(x > y ? x : y);
}
__device__ __forceinline__ double max_nonneg(double a, double b) {
    return gt_nonneg(a, b) ? a : b;
}
__device__ __forceinline__ double min_nonneg(double a, double b) {
    return gt_nonneg(a, b) ? b : a;
}
// double -> float, round to nearest even, as the conversion instruction does it: the significand
// rounded by an integer add; values outside [2^-126, 2^127) take the instruction.
__device__ __forceinline__ float to_float_rn(double x) {
    const int hi = __double2hiint(x);
    const unsigned ahi = (unsigned)hi & 0x7fffffffu;
    if (ahi - 0x38100000u >= 0x47e00000u - 0x38100000u) {
        float f;   // (volatile: the compiler may not run the instruction ahead of the test)
        asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(x));
        return f;
    }
    const unsigned long long v =
        ((unsigned long long)(ahi - 0x38000000u) << 32) | (unsigned)__double2loint(x);
    const unsigned long long q = v + 0x0fffffffull + ((v >> 29) & 1ull);
    return __uint_as_float((unsigned)(q >> 29) | ((unsigned)hi & 0x80000000u));
}
// double -> float within 2^-23 relative (truncated; below 2^-126 zero), for estimates.
__device__ __forceinline__ float to_float_est(double x) {
    const int hi = __double2hiint(x);
    const unsigned ahi = (unsigned)hi & 0x7fffffffu;
    const unsigned m = ((ahi - 0x38000000u) << 3) | ((unsigned)__double2loint(x) >> 29);
    return __uint_as_float((ahi < 0x38100000u ? 0u : m) | ((unsigned)hi & 0x80000000u));
}
// float -> double, exact (zero and normal values by integer operations).
__device__ __forceinline__ double from_float(float f) {
    const unsigned b = __float_as_uint(f), ab = b & 0x7fffffffu;
    if (ab - 0x00800000u >= 0x7f800000u - 0x00800000u && ab != 0u) {
        double d;
        asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(f));
        return d;
    }
    const unsigned hi = (b & 0x80000000u) | (ab == 0u ? 0u : (ab >> 3) + 0x38000000u);
    return __hiloint2double((int)hi, (int)(ab << 29));
}

// Per-ray constants of the right-hand side.
struct Rhs64 {
    double a, aa, m2;    // spin, its square, 2 M
    bool flat;
};

// a b + c d and a b + c with the roundings written out (the product c d is the rounded one), so
// that every kernel and every launch shape integrates with the same bits.
__device__ __forceinline__ double fma_dot2(double a, double b, double c, double d) {
    return __fma_rn(a, b, __dmul_rn(c, d));
}
__device__ __forceinline__ double mul3(double a, double b, double c) {
    return __dmul_rn(__dmul_rn(a, b), c);
}

// Eq. (geodesic) right-hand side; returns r at the evaluation point.
// With g^ab = eta^ab - f l^a l^b and L = l^a k_a, dx^a/dl = g^ab k_b and
// dk_c/dl = L (1/2 d_c f L + f d_c L), where d_c L is the derivative at fixed k. Instead of the
// nine derivatives d_c l_b, d_c L is formed directly: with A = x k_x + y k_y and B = y k_x - x k_y,
// l_x k_x + l_y k_y = (r A + a B) / (r^2 + a^2) =: L_xy and l_z k_z = z k_z / r, so
//   d_c L = d_c r V + (r k_x - a k_y, r k_y + a k_x, k_z)_c / (r^2 + a^2 or r),
//   V = (A - 2 r L_xy) / (r^2 + a^2) - k_z z / r^2,
// and d_c f = F1 d_c r - [c = z] 2 a^2 z f / (r^4 + a^2 z^2), F1 = f (3 / r - 4 r^3 / (r^4 + a^2 z^2)).
// The same quantities as the nine-derivative form, in about 40 fewer operations.
// Exact scalings are folded away: d_c f is carried halved (F1, the halving in its bracket: f itself
// is zero in flat space and, r^6 overflowing, beyond r = 2e51), so that 1/2 L need not be formed.
// The order of operations and the roundings are part of the method: rays that graze the photon
// orbit amplify them, and every kernel integrates with the same ones (bl_geodf.cuh in
// double-float).
__device__ __forceinline__ double geodesic_rhs64(const double y[8], const Rhs64& C, double dy[8]) {
    const double x = y[1], yy = y[2], z = y[3];
    const double kt = y[4], kx = y[5], ky = y[6], kz = y[7];
    const double a = C.a, aa = C.aa;
    const double q = __dadd_rn(__fma_rn(z, z, fma_dot2(x, x, yy, yy)), -aa);
    const double aaz = __dmul_rn(aa, z);
    const double aaz2 = __dmul_rn(aaz, z);
    const double D2 = __fma_rn(aaz2, 4.0, __dmul_rn(q, q));
    const double iD = rsqrt(D2);
    const double r2 = scale_exp(__fma_rn(D2, iD, q), -1);
    const double ir = rsqrt(r2);
    const double r = __dmul_rn(r2, ir);
    const double s4 = __fma_rn(r2, r2, aaz2);
    const double P = __dadd_rn(r2, aa);
    const double iPs = 1.0 / __dmul_rn(P, s4);
    const double is4 = __dmul_rn(P, iPs);
    const double iP = __dmul_rn(s4, iPs);
    const double f = C.flat ? 0.0 : __dmul_rn(mul3(C.m2, r, r2), is4);
    const double lx = __dmul_rn(fma_dot2(a, yy, r, x), iP);
    const double ly = __dmul_rn(fma_dot2(r, yy, -a, x), iP);
    const double lz = __dmul_rn(z, ir);
    const double A_ = fma_dot2(x, kx, yy, ky);
    const double B_ = fma_dot2(yy, kx, -x, ky);
    const double Lxy = __dmul_rn(fma_dot2(a, B_, r, A_), iP);
    const double L = __fma_rn(lz, kz, __dadd_rn(Lxy, -kt));
    const double fL = __dmul_rn(f, L);
    dy[0] = __dadd_rn(fL, -kt);
    dy[1] = __fma_rn(-lx, fL, kx);
    dy[2] = __fma_rn(-ly, fL, ky);
    dy[3] = __fma_rn(-lz, fL, kz);
    const double riD = __dmul_rn(r, iD);
    const double drx = __dmul_rn(riD, x), dry = __dmul_rn(riD, yy);
    const double drz = __dmul_rn(mul3(z, P, ir), iD);
    const double w = __dmul_rn(kz, ir);
    const double V = fma_dot2(__fma_rn(-scale_exp(r, 1), Lxy, A_), iP, -w, lz);
    const double Sx = fma_dot2(fma_dot2(r, kx, -a, ky), iP, drx, V);
    const double Sy = fma_dot2(fma_dot2(a, kx, r, ky), iP, dry, V);
    const double Sz = __fma_rn(drz, V, w);
    const double F1 = __dmul_rn(f, fma_dot2(1.5, ir, -__dmul_rn(scale_exp(r2, 1), r), is4));
    const double dfx = __dmul_rn(F1, drx), dfy = __dmul_rn(F1, dry);
    const double dfz = __fma_rn(F1, drz, -mul3(aaz, f, is4));
    dy[5] = __dmul_rn(L, fma_dot2(dfx, L, f, Sx));
    dy[6] = __dmul_rn(L, fma_dot2(dfy, L, f, Sy));
    dy[7] = __dmul_rn(L, fma_dot2(dfz, L, f, Sz));
    return r;
}

// Samples of an accepted step (reading: a step longer than ds_max in proper length whose start,
// midpoint or end lies inside the grid splits into ceil(ds / ds_max) parts), decided in FP32:
// the number of parts, or 0 where the FP32 error bound straddles a boundary and FP64 has to
// decide. near1 reports min(r) <= 1.001 r_grid. ym: the midpoint state in FP32.
// Bounds: r^2 from FP32 coordinates is off by at most 4e-7 (R^2 + a^2) / r^2 <= 1.2e-6 relative
// (r > a, else FP64 decides), f by four times that, l by 5e-6, so
// k^t = -k_t + f l^a k_a by at most 2e-5 (|k_t| + f (|k_t| + |k_x| + |k_y| + |k_z|)); the margins
// below are at least twice these.
__device__ __forceinline__ int step_parts_est(const float ym[8], float a, float m, bool flat,
                                              float h, float ds_max, double r0, double r1,
                                              double r_grid, bool& near1) {
    const float x = ym[1], y = ym[2], z = ym[3];
    const float aa = a * a;
    const float q = x * x + y * y + z * z - aa;
    const float r2 = 0.5f * (q + sqrtf(q * q + 4.0f * aa * z * z));
    near1 = true;
    if (!(r2 > aa)) return 0;
    const float ir = rsqrtf(r2), r = r2 * ir;
    const double rs = min_nonneg(r0, r1);
    if (!gt_nonneg(r_grid, rs)) {
        // both ends outside: the midpoint decides
        const float rg = (float)r_grid;
        if (r > rg * 1.00102f && gt_nonneg(rs, r_grid * 1.001)) {
            near1 = false;
            return 1;
        }
        return 0;
    }
    const float s4 = r2 * r2 + aa * z * z, P = r2 + aa;
    const float f = flat ? 0.0f : __fdividef(2.0f * m * r * r2, s4);
    const float iP = __fdividef(1.0f, P);
    const float lx = (r * x + a * y) * iP, ly = (r * y - a * x) * iP, lz = z * ir;
    const float ku = -ym[4] + f * (-ym[4] + lx * ym[5] + ly * ym[6] + lz * ym[7]);
    const float sc = __fdividef(fabsf(h) * rsqrtf(1.0f + f), ds_max);
    const float err = 4e-5f * (fabsf(ym[4]) + f * (fabsf(ym[4]) + fabsf(ym[5]) + fabsf(ym[6]) +
                                                   fabsf(ym[7])));
    const float t = sc * fabsf(ku), dt = sc * err + 4e-5f * t + 1e-20f;
    const float lo = ceilf(t - dt), hi = ceilf(t + dt);
    if (!(lo == hi) || !(hi < 4000.0f)) return 0;
    return hi < 1.0f ? 1 : (int)hi;
}

// Stage derivatives, 7 stages x 7 components: in dynamic shared memory, thread-fastest and
// conflict-free, or a per-thread local array (the 64-warp shape leaves no shared memory for them).
template <bool kSmem> struct KStore64;
template <> struct KStore64<true> {
    double* p;
    __device__ __forceinline__ double& at(int j, int s) { return p[(j * 7 + s) * 128]; }
};
template <> struct KStore64<false> {
    double k[7][7];
    __device__ __forceinline__ double& at(int j, int s) { return k[j][s]; }
};

template <class R, bool kKsmem>
__device__ __forceinline__ void geodesic64_body(const ImageDesc* __restrict__ imgs, int n_images,
                                                int64_t ray_begin, int64_t ray_end,
                                                RayHdr* __restrict__ hdr, RecordSink<R> sink,
                                                int record, BlockSource bs, int lanes = 32) {
    // rays [ray_begin, ray_end) of the batch form this wave; hdr and the chunk tables are
    // indexed by ray - ray_begin
    const int64_t re = wave_end(bs, ray_end);
    const int64_t total_rays = re > ray_begin ? re - ray_begin : 0;
    // FP32 records: the midpoint's increment (h/2) sum_j b_mid,j k_j and the quartic coefficients
    // are formed in FP32 from the state; they move a record by about one FP32 ulp and leave the
    // integration and its step decisions untouched. FP64 records: all in double.
    constexpr bool kFRec = sizeof(R) == sizeof(float);
    Counters* ctr = sink.ctr;
    bool active = false, exhausted = (int)(threadIdx.x & 31) >= lanes;   // lanes that take no rays
    int64_t wray = 0, opix = 0;
    int q = 0, pi = 0, pj = 0;
    double y[8];
    // K(0, c) = f(y); K(1..6, c) stage derivatives of the current attempt. dk_t/dl = 0, so the
    // k_t slot is left out: 7 slots a stage.
    KStore64<kKsmem> Ks;
    if constexpr (kKsmem) {
        extern __shared__ __align__(16) unsigned char geo_smem[];
        Ks.p = reinterpret_cast<double*>(geo_smem) + threadIdx.x;
    }
#define KX(j, c) Ks.at(j, (c) < 4 ? (c) : (c) - 1)
    double h = 0.0, nnorm = 0.0;
    bool been_inside = false, prev_rej = false;
    int64_t attempts = 0, max_steps = 0;
    int32_t nrec = 0, status = 0;
    double r_cam = 0.0, r_in = 0.0, r_grid = 0.0, tol_abs = 0.0, tol_rel = 0.0;
    Rhs64 C{0.0, 0.0, 0.0, false};
    double r_cur = 0.0;             // r at y
    bool want_aux = false;          // auxiliary images: proper length and affine parameter
    bool want_t = false;            // sample times (slow light only)
    double aux_len = 0.0, aux_lam = 0.0;
    int32_t last_in = -1;           // last record of a step reaching within 1.001 r_max

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
            {
                double yd[8];
                pixel_state(im, pi, pj, yd, nnorm);
#pragma unroll
                for (int c = 0; c < 8; ++c) y[c] = yd[c];
            }
            C.a = im.spin;
            C.aa = im.spin * im.spin;
            C.m2 = 2.0 * im.mass;
            C.flat = im.flat != 0;
            r_cam = im.r_cam;
            r_in = im.r_in_over_rhor * im.r_hor;
            r_grid = im.r_max;
            tol_abs = im.tol_abs;
            tol_rel = im.tol_rel;
            max_steps = im.max_steps;
            want_aux = record && im.aux != nullptr;
            want_t = im.n_snap > 1;
            aux_len = aux_lam = 0.0;
            h = -im.h0_frac * (r_cam - im.r_hor);
            prev_rej = false;
        }
        // ---- one Dormand-Prince attempt (Table tab:dp) ----
        // Rolled stage loop: one right-hand-side body run six times keeps the kernel small
        // enough for the instruction cache. K(0) holds f(y) (first same as last), K(s) the
        // stage derivatives; stage 6 is evaluated at the fifth-order solution y5. A ray's first
        // attempt starts at stage 0, which evaluates f(y) at the stage point y, so that the
        // set-up path needs no copy of the right-hand side.
        double ys[8], y5[8];
        double r5 = 0.0;
        y5[4] = y[4];
        ys[4] = y[4];
#pragma unroll 1
        for (int st = need ? 0 : 1; st < 7; ++st) {
            if (st == 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c) ys[c] = y[c];
            } else {
                // earlier stages outer (rolled), components inner: each coefficient is read
                // once per stage term; every component keeps its order of operations. The
                // right-hand side does not read x^t, whose sum only the last row needs.
                double acc[8];
                {
                    const double a0 = DPCoef<double>::a(st, 0);
#pragma unroll
                    for (int c = 1; c < 8; ++c)
                        if (c != 4) acc[c] = a0 * KX(0, c);
                }
                // the last row's second coefficient (b_2 of the fifth-order weights) is zero
#pragma unroll 1
                for (int j = st == 6 ? 2 : 1; j < st; ++j) {
                    const double aj = DPCoef<double>::a(st, j);
#pragma unroll
                    for (int c = 1; c < 8; ++c)
                        if (c != 4) acc[c] = acc[c] + aj * KX(j, c);
                }
#pragma unroll
                for (int c = 1; c < 8; ++c)
                    if (c != 4) ys[c] = y[c] + h * acc[c];
            }
            double fs[8];
            const double rr = geodesic_rhs64(ys, C, fs);
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c != 4) KX(st, c) = fs[c];
            if (st == 0) {
                r_cur = rr;
                been_inside = r_cur < r_cam;
            }
            if (st == 6) {
                r5 = rr;
#pragma unroll
                for (int c = 1; c < 8; ++c) y5[c] = ys[c];
            }
        }
        // x^t at the fifth-order solution (the same sum as the other components')
        {
            double t = DPCoef<double>::a(6, 0) * KX(0, 0);
#pragma unroll 1
            for (int j = 2; j < 6; ++j) t = t + DPCoef<double>::a(6, j) * KX(j, 0);
            y5[0] = y[0] + h * t;
        }
        // Error norm eps = max_c |y5_c - y4_c| / (f_abs + f_rel max(|y_c|, |y5_c|)) with
        // y5 - y4 = h sum (b5 - b4) k; the k_t component's difference is zero.
        double eps;
        bool finite = true;
        {
            double acc[8];
            {
                const double e0 = DPCoef<double>::e(0);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c != 4) acc[c] = e0 * KX(0, c);
            }
#pragma unroll 1
            for (int j = 2; j < 7; ++j) {
                const double ej = DPCoef<double>::e(j);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c != 4) acc[c] = acc[c] + ej * KX(j, c);
            }
            double num = 0.0, den = 1.0;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c == 4) continue;
                const double err = __longlong_as_double(abs_bits(h * acc[c]));
                const double sc = tol_abs + tol_rel * max_abs(y[c], y5[c]);
                finite = finite && finite_bits(err) && finite_bits(y5[c]);
                if (c == 0) {
                    if (__double_as_longlong(err) > 0) { num = err; den = sc; }
                } else if (gt_nonneg(err * den, num * sc)) {
                    num = err;
                    den = sc;
                }
            }
            eps = num / den;
        }
        ++attempts;
        bool done = false;
        if (!finite) {
            status = BL_RAY_NAN;
            done = true;
        } else if (!gt_nonneg(eps, 1.0)) {
            // accepted: samples of this step (camera side first)
            if (record) {
                double ym[8];
                float ymf[8], incm[8];
                if constexpr (kFRec) {
                    const float hh = 0.5f * to_float_rn(h);
                    float acc[8];
                    {
                        const float m0 = c_dpf.m[0].x;
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            if (c != 4) acc[c] = m0 * to_float_rn(KX(0, c));
                    }
#pragma unroll 1
                    for (int j = 2; j < 7; ++j) {
                        const float mj = c_dpf.m[j].x;
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            if (c != 4) acc[c] = fmaf(mj, to_float_rn(KX(j, c)), acc[c]);
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        incm[c] = c == 4 ? 0.0f : __fmul_rn(hh, acc[c]);
                        ym[c] = c == 4 ? y[4] : y[c] + from_float(incm[c]);
                        ymf[c] = to_float_rn(ym[c]);
                    }
                } else {
                    const double hh = scale_exp(h, -1);
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        ym[c] = y[c];
                        if (c == 4 || (c == 0 && !want_t)) continue;
                        double acc = DPCoef<double>::m(0) * KX(0, c);
#pragma unroll 1
                        for (int j = 2; j < 7; ++j) acc = acc + DPCoef<double>::m(j) * KX(j, c);
                        ym[c] = y[c] + hh * acc;
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c) ymf[c] = to_float_est(ym[c]);
                }
                const double hd = h, r0 = r_cur, r1 = r5;
                const ImageDesc& im = imgs[q];
                bool near1 = true;
                int nsub = want_aux ? 0
                                    : step_parts_est(ymf, to_float_est(C.a),
                                                     0.5f * to_float_est(C.m2), C.flat,
                                                     to_float_est(hd), (float)im.ds_max, r0, r1,
                                                     r_grid, near1);
                if (nsub == 0) {
                    KSGeom<double> Gm;
                    ks_geom<double>(ym[1], ym[2], ym[3], im.spin, im.mass, C.flat, Gm);
                    const double L = -ym[4] + Gm.l[1] * ym[5] + Gm.l[2] * ym[6] + Gm.l[3] * ym[7];
                    const double kt_up = -ym[4] + Gm.f * L;
                    // ds/dl = (g_pq k^p k^q)^1/2 = alpha |k^t| for a null ray
                    const double ds = fabs(hd) * fabs(kt_up) / sqrt(1.0 + Gm.f);
                    if (want_aux) {
                        aux_lam += fabs(hd);
                        aux_len += ds;
                    }
                    const double rmin = fmin(Gm.r, fmin(r0, r1));
                    nsub = 1;
                    if (rmin < r_grid && ds > im.ds_max) {
                        const double nd = ceil(ds / im.ds_max);
                        nsub = nd > 4096.0 ? 4097 : (int)nd;
                    }
                    near1 = rmin <= r_grid * 1.001;
                }
                bool ok = true;
                const double hl = fabs(hd);
                if (nsub == 1) {
                    if constexpr (kFRec) {
                        float yf[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) yf[c] = to_float_rn(y[c]);
                        ok = append_record<float, float, double>(sink, wray, nrec, ymf, yf, hl);
                    } else {
                        ok = append_record<double, double, double>(sink, wray, nrec, ym, y, hl);
                    }
                } else if constexpr (kFRec) {
                    // the quartic through y0, y1, h f0, h f1 and y_mid (Shampine 1986), in FP32
                    // about y0 (y_mid - y0 is the midpoint increment), roundings written out
                    const float hf = to_float_rn(h);
                    float y0f[8], d0f[8], c2f[8], c3f[8], c4f[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const float k0 = c == 4 ? 0.0f : to_float_rn(KX(0, c));
                        const float k6 = c == 4 ? 0.0f : to_float_rn(KX(6, c));
                        const float d0 = __fmul_rn(hf, k0);
                        const float D1 = __fadd_rn(c == 4 ? 0.0f : to_float_rn(y5[c] - y[c]), -d0);
                        const float D2 = __fmaf_rn(hf, k6, -d0);
                        const float D3 = __fmaf_rn(-0.5f, d0, incm[c]);
                        y0f[c] = to_float_rn(y[c]);
                        d0f[c] = d0;
                        c2f[c] = __fmaf_rn(16.0f, D3, __fmaf_rn(-5.0f, D1, D2));
                        c3f[c] = __fmaf_rn(-32.0f, D3, __fmaf_rn(14.0f, D1, -__fmul_rn(3.0f, D2)));
                        c4f[c] = __fmaf_rn(16.0f, D3, __fmaf_rn(-8.0f, D1, __fmul_rn(2.0f, D2)));
                    }
                    ok = emit_quartic_f(sink, wray, nrec, y0f, d0f, c2f, c3f, c4f, nsub, hl / nsub);
                } else {
                    double d0[8], c2[8], c3[8], c4[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        if (c == 4) continue;
                        if (c == 0 && !want_t) {
                            d0[0] = c2[0] = c3[0] = c4[0] = 0.0;
                            continue;
                        }
                        d0[c] = hd * KX(0, c);
                        const double D1 = y5[c] - y[c] - d0[c];
                        const double D2 = hd * KX(6, c) - d0[c];
                        const double D3 = ym[c] - y[c] - 0.5 * d0[c];
                        c2[c] = -5.0 * D1 + D2 + 16.0 * D3;
                        c3[c] = 14.0 * D1 - 3.0 * D2 - 32.0 * D3;
                        c4[c] = -8.0 * D1 + 2.0 * D2 + 16.0 * D3;
                    }
                    const double inv = nsub < 15 ? c_inv_int64[nsub] : 1.0 / nsub;
                    const double dls = hl * inv;
                    double s0 = 0.0;   // the part's number
                    for (int s = 0; s < nsub && ok; ++s, s0 += 1.0) {
                        double ysm[8], ynd[8];
                        const double ts = (s0 + 0.5) * inv, tn = s0 * inv;
                        ysm[0] = ysm[4] = ynd[4] = ynd[0] = 0.0;
                        if (want_t) ysm[0] = y[0] + ts * (d0[0] + ts * (c2[0] + ts * (c3[0] + ts * c4[0])));
#pragma unroll
                        for (int c = 1; c < 8; ++c) {
                            if (c == 4) continue;
                            ysm[c] = y[c] + ts * (d0[c] + ts * (c2[c] + ts * (c3[c] + ts * c4[c])));
                            ynd[c] = (s == 0) ? y[c]
                                              : y[c] + tn * (d0[c] + tn * (c2[c] + tn * (c3[c] + tn * c4[c])));
                        }
                        ok = append_record<double, double, double>(sink, wray, nrec, ysm, ynd, dls);
                    }
                }
                if (!ok) { status = BL_RAY_OVERFLOW; done = true; }
                else if (near1) last_in = nrec - 1;
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c == 4) continue;
                y[c] = y5[c];
                KX(0, c) = KX(6, c);
            }
            // (eps = 0 gives the clamp's 10)
            double fac = max_nonneg(0.2, min_nonneg(10.0, 0.9 * inv_fifth_root(eps)));
            if (prev_rej) fac = min_nonneg(fac, 1.0);
            h = h * fac;
            prev_rej = false;
            r_cur = r5;
            if (!done) {
                if (gt_nonneg(r_in, r_cur)) { status = BL_RAY_HORIZON; done = true; }
                else if (been_inside && gt_nonneg(r_cur, r_cam)) { status = BL_RAY_ESCAPED; done = true; }
                else if (gt_nonneg(r_cam, r_cur)) been_inside = true;
            }
        } else {
            h = h * max_nonneg(0.2, 0.9 * inv_fifth_root(eps));
            prev_rej = true;
        }
        if (!done) {
            // |h| < 1e-12 r: 2^-39 of r's power of two decides almost always
            const int eh = (__double2hiint(h) >> 20) & 0x7ff, er = (__double2hiint(r_cur) >> 20) & 0x7ff;
            if (eh - er - 1 < -39 && fabs(h) < 1e-12 * r_cur) {
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
                for (int c = 0; c < 8; ++c) im.end_state[pix * 8 + c] = y[c];
            if (im.samples) im.samples[pix] = nrec;
            if (want_aux) {
                aux_store(im, 0, pix, -y[0]);
                aux_store(im, 1, pix, aux_len);
                aux_store(im, 2, pix, aux_lam);
            }
            RayHdr hd;
            hd.kt = y[4];
            hd.nnorm = nnorm;
            hd.nrec = nrec;
            hd.status = status;
            hd.last_in = last_in;
            hdr[wray] = hd;
            if (status != BL_RAY_HORIZON && status != BL_RAY_ESCAPED)
                atomicAdd(&ctr->bad_rays, 1ull);
            active = false;
            attempts = 0;
            nrec = 0;
            status = 0;
            last_in = -1;
        }
    }
}
#undef KX

// ---------------------------------------------------------------------------------------
// Fixed-rule geodesic integrators (Sec. 2.2): classical RK4 (Table tab:rk4) and Heun's RK2
// (Table tab:rk2) in FP64, step -f_step (r - r_hor) at the start of each step (Eq. rk_step).
// Each step's sample is its cubic Hermite midpoint (y0 + y1)/2 + h (f0 - f1)/8; a step longer
// than ds_max in proper length is subdivided by the same cubic. Persistent like the
// Dormand-Prince kernels, with the same records, outputs and termination rules, and bound like
// them by its FP64 instruction count: one rolled right-hand-side body, the weights' common factor
// taken out of the sums (h/6 (f + 2 k2 + 2 k3 + k4)), conversions, comparisons and the splitting
// decision off the FP64 pipe. RK4 at f_step 0.02, 96^2, mixed form: 72 -> 23.3 ms (540 steps a ray
// on average, 1242 the longest).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ double hermite(double y0, double y1, double f0, double f1, double h,
                                          double h00, double h10, double h01, double h11) {
    return h00 * y0 + h10 * h * f0 + h01 * y1 + h11 * h * f1;
}

// One record in the sink's type from a double state (x^t only where it is read).
template <class R>
__device__ __forceinline__ bool append_state(const RecordSink<R>& sink, int64_t wray, int32_t& nrec,
                                             const double ys[8], const double yn[8], double dl) {
    if constexpr (sizeof(R) == sizeof(float)) {
        float a[8], b[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) { a[c] = to_float_rn(ys[c]); b[c] = to_float_rn(yn[c]); }
        return append_record<float, float, double>(sink, wray, nrec, a, b, dl);
    } else {
        return append_record<double, double, double>(sink, wray, nrec, ys, yn, dl);
    }
}

template <class R>
__global__ void __launch_bounds__(128, 3) geodesic_rk_kernel(const ImageDesc* __restrict__ imgs,
                                                             int n_images, int64_t ray_begin,
                                                             int64_t ray_end,
                                                             RayHdr* __restrict__ hdr,
                                                             RecordSink<R> sink, int record,
                                                             BlockSource bs, int sms) {
    if (sms > 0 && spare_cta(bs, ray_begin, ray_end, sms)) return;
    const int64_t re = wave_end(bs, ray_end);
    const int64_t total_rays = re > ray_begin ? re - ray_begin : 0;
    Counters* ctr = sink.ctr;
    bool active = false, exhausted = false;
    int64_t wray = 0, opix = 0;
    int q = 0, pi = 0, pj = 0;
    double y[8], f[8];
    double nnorm = 0.0, r_cur = 0.0, r_cam = 0.0, r_in = 0.0, r_hor = 0.0;
    double r_grid = 0.0, f_step = 0.0;
    Rhs64 C{0.0, 0.0, 0.0, false};
    int stages = 3;                 // evaluations between f(y) and the step's end
    bool been_inside = false, want_aux = false, want_t = false;
    int64_t nsteps = 0, max_steps = 0;
    int32_t nrec = 0, status = 0;
    double aux_len = 0.0, aux_lam = 0.0;
    while (true) {
        const bool need = !active && !exhausted;
        const unsigned long long got = warp_refill(&ctr->next_ray_geo, need);
        if (need) {
            if ((int64_t)got >= total_rays) exhausted = true;
            else { wray = (int64_t)got; active = true; }
        }
        if (!__any_sync(0xffffffffu, active)) break;
        if (!active) continue;
        if (need) {
            setup_ray(imgs, n_images, bs, ray_begin + wray, q, opix, pi, pj);
            const ImageDesc& im = imgs[q];
            pixel_state(im, pi, pj, y, nnorm);
            C.a = im.spin;
            C.aa = im.spin * im.spin;
            C.m2 = 2.0 * im.mass;
            C.flat = im.flat != 0;
            r_cam = im.r_cam; r_hor = im.r_hor;
            r_in = im.r_in_over_rhor * im.r_hor;
            r_grid = im.r_max;
            f_step = im.f_step;
            stages = im.integrator == BL_INT_RK4 ? 3 : 1;
            max_steps = im.max_steps;
            want_aux = record && im.aux != nullptr;
            want_t = im.n_snap > 1;
            aux_len = aux_lam = 0.0;
            nsteps = 0; nrec = 0; status = BL_RAY_OK;
        }
        // one step; a new ray's first evaluation (st = -1) gives f(y). The stages' points are y +
        // h/2 f, y + h/2 k2, y + h k3 (RK4) or y + h f (RK2), the last evaluation is at the step's
        // end y1.
        double h = 0.0, r1 = 0.0;
        double acc[8], kc[8], ys[8];
        ys[4] = y[4];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = kc[c] = f[c];
        if (!need) h = -f_step * (r_cur - r_hor);
#pragma unroll 1
        for (int st = need ? -1 : 0; st <= stages; ++st) {
            if (st < 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c) ys[c] = y[c];
            } else if (st < stages) {
                const double hs = stages == 3 && st < 2 ? scale_exp(h, -1) : h;
#pragma unroll
                for (int c = 1; c < 8; ++c)
                    if (c != 4) ys[c] = y[c] + hs * kc[c];
            } else {
                const double hw = stages == 3 ? h * (1.0 / 6.0) : scale_exp(h, -1);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c != 4) ys[c] = y[c] + hw * acc[c];
            }
            const double rr = geodesic_rhs64(ys, C, kc);
            if (st < 0) {
                r_cur = rr;
                been_inside = r_cur < r_cam;
                h = -f_step * (r_cur - r_hor);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (c == 4) continue;
                    f[c] = acc[c] = kc[c];
                }
            } else if (st < stages) {
                const double w = stages == 3 && st < 2 ? 2.0 : 1.0;
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (c != 4) acc[c] = acc[c] + w * kc[c];
            } else {
                r1 = rr;
            }
        }
        ++nsteps;
        bool finite = true;
#pragma unroll
        for (int c = 0; c < 8; ++c) finite = finite && finite_bits(ys[c]);
        bool done = false;
        if (!finite) {
            status = BL_RAY_NAN;
            done = true;
        } else {
            // y1 = ys, f1 = kc
            if (record) {
                const ImageDesc& im = imgs[q];
                const double h8 = scale_exp(h, -3);
                double ym[8];
                float ymf[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    ym[c] = y[c];
                    if (c != 4 && (c != 0 || want_t)) ym[c] = 0.5 * (y[c] + ys[c]) + h8 * (f[c] - kc[c]);
                    ymf[c] = to_float_est(ym[c]);
                }
                bool near1 = true;
                int nsub = want_aux ? 0
                                    : step_parts_est(ymf, to_float_est(C.a),
                                                     0.5f * to_float_est(C.m2), C.flat,
                                                     to_float_est(h), (float)im.ds_max, r_cur, r1,
                                                     r_grid, near1);
                const double hl = fabs(h);
                if (nsub == 0) {
                    KSGeom<double> Gm;
                    ks_geom<double>(ym[1], ym[2], ym[3], C.a, im.mass, C.flat, Gm);
                    const double L = -ym[4] + Gm.l[1] * ym[5] + Gm.l[2] * ym[6] + Gm.l[3] * ym[7];
                    const double kt_up = -ym[4] + Gm.f * L;
                    const double ds = hl * fabs(kt_up) / sqrt(1.0 + Gm.f);
                    if (want_aux) { aux_lam += hl; aux_len += ds; }
                    nsub = 1;
                    if (fmin(Gm.r, fmin(r_cur, r1)) < r_grid && ds > im.ds_max) {
                        const double nd = ceil(ds / im.ds_max);
                        nsub = nd > 4096.0 ? 4097 : (int)nd;
                    }
                }
                bool ok = true;
                if (nsub == 1) {
                    ok = append_state(sink, wray, nrec, ym, y, hl);
                } else {
                    const double inv = nsub < 15 ? c_inv_int64[nsub] : 1.0 / nsub;
                    const double dls = hl * inv;
                    double s0 = 0.0;
                    for (int sb = 0; sb < nsub && ok; ++sb, s0 += 1.0) {
                        double ysm[8], ynd[8];
                        ysm[0] = ysm[4] = ynd[0] = ynd[4] = 0.0;
                        {
                            const double t = (s0 + 0.5) * inv, t2 = t * t, t3 = t2 * t;
                            const double h00 = 2 * t3 - 3 * t2 + 1, h10 = t3 - 2 * t2 + t,
                                         h01 = -2 * t3 + 3 * t2, h11 = t3 - t2;
                            if (want_t) ysm[0] = hermite(y[0], ys[0], f[0], kc[0], h, h00, h10, h01, h11);
#pragma unroll
                            for (int c = 1; c < 8; ++c)
                                if (c != 4) ysm[c] = hermite(y[c], ys[c], f[c], kc[c], h, h00, h10, h01, h11);
                        }
                        if (sb == 0) {
#pragma unroll
                            for (int c = 0; c < 8; ++c) ynd[c] = y[c];
                        } else {
                            const double t = s0 * inv, t2 = t * t, t3 = t2 * t;
                            const double h00 = 2 * t3 - 3 * t2 + 1, h10 = t3 - 2 * t2 + t,
                                         h01 = -2 * t3 + 3 * t2, h11 = t3 - t2;
#pragma unroll
                            for (int c = 1; c < 8; ++c)
                                if (c != 4) ynd[c] = hermite(y[c], ys[c], f[c], kc[c], h, h00, h10, h01, h11);
                        }
                        ok = append_state(sink, wray, nrec, ysm, ynd, dls);
                    }
                }
                if (!ok) { status = BL_RAY_OVERFLOW; done = true; }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                if (c == 4) continue;
                y[c] = ys[c];
                f[c] = kc[c];
            }
            r_cur = r1;
            if (!done) {
                if (gt_nonneg(r_in, r_cur)) { status = BL_RAY_HORIZON; done = true; }
                else if (been_inside && gt_nonneg(r_cur, r_cam)) { status = BL_RAY_ESCAPED; done = true; }
                else {
                    if (gt_nonneg(r_cam, r_cur)) been_inside = true;
                    if (fabs(f_step * (r_cur - r_hor)) < 1e-12 * r_cur) { status = BL_RAY_UNDERFLOW; done = true; }
                    else if (nsteps >= max_steps) { status = BL_RAY_MAX_STEPS; done = true; }
                }
            }
        }
        if (done) {
            const ImageDesc& im = imgs[q];
            const int64_t pix = opix;
            if (im.status) im.status[pix] = status;
            if (im.steps) im.steps[pix] = (int32_t)(nsteps < 2147483647 ? nsteps : 2147483647);
            if (im.end_state)
                for (int c = 0; c < 8; ++c) im.end_state[pix * 8 + c] = y[c];
            if (im.samples) im.samples[pix] = nrec;
            if (want_aux) {
                aux_store(im, 0, pix, -y[0]);
                aux_store(im, 1, pix, aux_len);
                aux_store(im, 2, pix, aux_lam);
            }
            RayHdr hd;
            hd.kt = y[4];
            hd.nnorm = nnorm;
            hd.nrec = nrec;
            hd.status = status;
            hd.last_in = nrec - 1;   // (fixed-step integrators: no skip)
            hdr[wray] = hd;
            if (status != BL_RAY_HORIZON && status != BL_RAY_ESCAPED)
                atomicAdd(&ctr->bad_rays, 1ull);
            active = false;
        }
    }
}

}  // namespace bl
