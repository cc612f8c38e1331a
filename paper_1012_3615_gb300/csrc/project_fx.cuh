// The refined projection of project.cuh in fixed point: the FP64 steps (special
// unitary start, residual, first update) as integer multiply-adds on two-limb
// numbers (see dslash_fx.cu), for path sums that are in that form.  About 1,500
// wide multiply-adds of 4 clocks in place of 440 FP64 operations of 64; what
// bounds it now is the instruction count (13,000 a matrix, the FP32 seed among
// them) and their fetch.  16^3x32: 4.50 ms a build, 5.06 with FP64; distance from
// the 64-bit eigenvector projection 0.7e-16 rms, it was 1.6e-16.
// Bounds: rows and columns of A, Y have norms <= 1 (and their rounding), so high
// limbs are below 2^29 and 2^28 and every sum of six products below 2^62; low
// limbs are never INT_MIN, so limbs can be negated.
#pragma once
#include "fx.cuh"
#include "project.cuh"

namespace bri {

constexpr int PY_B = 60;  // fraction bits of Y

// exact sum of products of two-limb numbers of B1 and B2 fraction bits, in units
// of 2^-(B1 + B2 - 64); the cross products are kept 2^63 up (no sign word) and rounded
struct FxSum {
    long long a = -(1ll << 31);
    unsigned long long b = (1ull << 63) + (1ull << 31);
    BRI_D void add(int wh, int wl, int ph, int pl) {
        a += (long long)wh * ph;
        b += (long long)wh * pl;
        b += (long long)wl * ph;
    }
    BRI_D long long get() const { return a + (long long)(b >> 32); }
};
// re, im += w p, or conj(w) p
template <bool CONJ> BRI_D void fx_cmac(const int4 w, const int4 p, FxSum &re, FxSum &im) {
    re.add(w.x, w.y, p.x, p.y);
    im.add(w.x, w.y, p.z, p.w);
    if (CONJ) {
        re.add(w.z, w.w, p.z, p.w);
        im.add(-w.z, -w.w, p.x, p.y);
    } else {
        re.add(-w.z, -w.w, p.z, p.w);
        im.add(w.z, w.w, p.x, p.y);
    }
}
BRI_D int4 fx_pack(long long re, long long im) {
    const int2 a = fx_limbs(re), b = fx_limbs(im);
    return make_int4(a.x, a.y, b.x, b.y);
}
// v / 2^n rounded
BRI_D long long fx_shr(long long v, int n) { return (v + (1ll << (n - 1))) >> n; }
// v 2^sh rounded (|v| 2^sh < 2^62), by shifts
BRI_D long long fx_int(float v, int sh) {
    const unsigned u = __float_as_uint(v), e = u >> 23 & 255u, m = (u & 0x7fffffu) | (e ? 0x800000u : 0u);
    const int s = (int)max(e, 1u) - 150 + sh, r = min(-s, 31);
    const long long f = s >= 0 ? (long long)m << s : (long long)((m + ((1u << r) >> 1)) >> r);
    return (int)u < 0 ? -f : f;
}
BRI_D float fx_float(long long v) {
    const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const float f = fmaf((float)(unsigned)(u >> 32), 4294967296.f, (float)(unsigned)u);
    return v < 0 ? -f : f;
}

// the traceless anti-hermitian part of A^dagger Y (A: 61 fraction bits)
BRI_D M3<float2> ta_residual_fx(const int4 A[9], const int4 Y[9]) {
    constexpr float unit = 0x1p-57f;  // 2^-(61 + PY_B - 64)
    M3<float2> R;
    long long d[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        FxSum im;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const int4 a = A[3 * k + i], y = Y[3 * k + i];
            im.add(a.x, a.y, y.z, y.w);
            im.add(-a.z, -a.w, y.x, y.y);
        }
        d[i] = im.get();
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            FxSum r1, m1, r2, m2;  // B_ij, B_ji
#pragma unroll
            for (int k = 0; k < 3; k++) {
                fx_cmac<true>(A[3 * k + i], Y[3 * k + j], r1, m1);
                fx_cmac<true>(A[3 * k + j], Y[3 * k + i], r2, m2);
            }
            const float2 r = make_float2(0.5f * unit * fx_float(r1.get() - r2.get()),
                                         0.5f * unit * fx_float(m1.get() + m2.get()));
            R.e[3 * i + j] = r;
            R.e[3 * j + i] = make_float2(-r.x, r.y);
        }
    }
    const long long tr = d[0] + d[1] + d[2];
#pragma unroll
    for (int i = 0; i < 3; i++) R.e[4 * i] = make_float2(0.f, unit / 3.f * fx_float(3 * d[i] - tr));
    return R;
}

// y[0..2] *= 1 / |y|, |y|^2 = 1 + n with a small n; false if it is not
BRI_D bool fx_unit_row(int4 y[3]) {
    FxSum s;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        s.add(y[i].x, y[i].y, y[i].x, y[i].y);
        s.add(y[i].z, y[i].w, y[i].z, y[i].w);
    }
    const long long n = s.get() - (1ll << (2 * PY_B - 64));  // units of 2^-56
    const float nf = 0x1p-56f * fx_float(n);
    if (!(fabsf(nf) < 1e-5f)) return false;
    // -n/2 + 3/8 n^2 with 76 fraction bits
    const int2 c = fx_limbs(-(n << 19) + fx_int(0.375f * nf * nf, 76));
#pragma unroll
    for (int i = 0; i < 3; i++) {
        FxSum re, im;
        re.add(c.x, c.y, y[i].x, y[i].y);
        im.add(c.x, c.y, y[i].z, y[i].w);
        y[i] = fx_pack(fx_join(y[i].x, y[i].y) + fx_shr(re.get(), 12), fx_join(y[i].z, y[i].w) + fx_shr(im.get(), 12));
    }
    return true;
}

// the projection of a path sum (two limbs, 61 fraction bits, rows and columns of
// norm <= 1) as FP64 numbers; false: take the general form
BRI_D bool project_fast_fx(const int4 A[9], M3<double2> &out) {
    ProjectionSeed sd;
    int4 Y[9];
    {
        M3<float2> A32, Y32;
#pragma unroll
        for (int i = 0; i < 9; i++) A32.e[i] = make_float2(0x1p-29f * (float)A[i].x, 0x1p-29f * (float)A[i].z);
        if (!project_seed(A32, sd, Y32)) return false;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            if (!(fabsf(Y32.e[i].x) < 1.1f && fabsf(Y32.e[i].y) < 1.1f)) return false;
            Y[i] = fx_pack(fx_int(Y32.e[i].x, PY_B), fx_int(Y32.e[i].y, PY_B));
        }
    }
    // special unitary: row 0 normalised, row 1 orthogonal to it and normalised,
    // row 2 = conj(row 0 x row 1)
    if (!fx_unit_row(Y)) return false;
    {
        FxSum dr, di;
#pragma unroll
        for (int i = 0; i < 3; i++) fx_cmac<true>(Y[i], Y[3 + i], dr, di);
        if (!(fabsf(fx_float(dr.get())) < 0x1p40f && fabsf(fx_float(di.get())) < 0x1p40f)) return false;  // 2^-16
        const int4 d = fx_pack(-(dr.get() << 20), -(di.get() << 20));  // 76 fraction bits
#pragma unroll
        for (int i = 0; i < 3; i++) {
            FxSum re, im;
            fx_cmac<false>(d, Y[i], re, im);
            Y[3 + i] = fx_pack(fx_join(Y[3 + i].x, Y[3 + i].y) + fx_shr(re.get(), 12),
                               fx_join(Y[3 + i].z, Y[3 + i].w) + fx_shr(im.get(), 12));
        }
    }
    if (!fx_unit_row(Y + 3)) return false;
#pragma unroll
    for (int j = 0; j < 3; j++) {
        FxSum r1, i1, r2, i2;
        fx_cmac<false>(Y[(j + 1) % 3], Y[3 + (j + 2) % 3], r1, i1);
        fx_cmac<false>(Y[(j + 2) % 3], Y[3 + (j + 1) % 3], r2, i2);
        Y[6 + j] = fx_pack((r1.get() - r2.get()) << 4, (i2.get() - i1.get()) << 4);
    }
    float last = 0.f;
#pragma unroll 1
    for (int it = 0; it < 5; it++) {
        M3<float2> O = seed_solve(sd, ta_residual_fx(A, Y));
        float w = 0.f;
#pragma unroll
        for (int i = 0; i < 9; i++) {
            O.e[i] = make_float2(-O.e[i].x, -O.e[i].y);
            w = fmaxf(w, fmaxf(fabsf(O.e[i].x), fabsf(O.e[i].y)));
        }
        if (!(w < 2e-5f)) return false;
        if (w > 1e-10f) {
            // Y exp(O): O traceless and its powers (FP32) with 75 fraction bits
            const M3<float2> O2 = m3_mul(O, O), O3 = m3_mul(O, O2);
            int4 E[9];
            const long long t = -(fx_int(O.e[0].y, 75) + fx_int(O.e[4].y, 75));
#pragma unroll
            for (int i = 0; i < 9; i++) {
                const float2 h = cadd(cscale(O2.e[i], 0.5f), cscale(O3.e[i], 1.f / 6.f));
                E[i] = fx_pack(fx_int(O.e[i].x, 75) + fx_int(h.x, 75),
                               (i == 8 ? t : fx_int(O.e[i].y, 75)) + fx_int(h.y, 75));
            }
#pragma unroll
            for (int r = 0; r < 3; r++) {
                int4 n[3];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    FxSum re, im;
#pragma unroll
                    for (int k = 0; k < 3; k++) fx_cmac<false>(Y[3 * r + k], E[3 * k + c], re, im);
                    n[c] = fx_pack(fx_join(Y[3 * r + c].x, Y[3 * r + c].y) + fx_shr(re.get(), 11),
                                   fx_join(Y[3 * r + c].z, Y[3 * r + c].w) + fx_shr(im.get(), 11));
                }
#pragma unroll
                for (int c = 0; c < 3; c++) Y[3 * r + c] = n[c];
            }
        } else {
            M3<float2> Y32;
#pragma unroll
            for (int i = 0; i < 9; i++) Y32.e[i] = make_float2(0x1p-28f * (float)Y[i].x, 0x1p-28f * (float)Y[i].z);
            const M3<float2> D = m3_mul(Y32, O);
#pragma unroll
            for (int i = 0; i < 9; i++)
                Y[i] = fx_pack(fx_join(Y[i].x, Y[i].y) + fx_int(D.e[i].x, PY_B),
                               fx_join(Y[i].z, Y[i].w) + fx_int(D.e[i].y, PY_B));
        }
        // what is left is about w times this step's contraction
        if (w == 0.f || (it > 0 && w * fmaxf(w / last, 1e-7f) < 1e-17f)) {
#pragma unroll
            for (int i = 0; i < 9; i++)
                out.e[i] = make_double2(fx_double(fx_join(Y[i].x, Y[i].y), -PY_B), fx_double(fx_join(Y[i].z, Y[i].w), -PY_B));
            return true;
        }
        last = w;
    }
    return false;
}

}  // namespace bri
