// FP64 back-projection to SU(3) (Sec. 5.2, Eq. proj_SU) on the device.
//
//   P_SU(3){A} = argmax_{Y in SU(3)} Re tr(A^dagger Y)
//
// With A = U S V^dagger, Y = U diag(e^{i theta}) V^dagger and the constraint
// sum theta_i + phi = 0 (mod 2 pi), e^{i phi} = det A / |det A|, the problem is
// to maximise sum_i s_i cos(theta_i).  The paper suggests a grid scan and a local
// maximisation.  Here the stationary points are used directly instead: a
// Lagrange multiplier kappa gives s_i sin(theta_i) = kappa for every i.  At a
// maximum only the smallest singular value may have cos(theta) < 0 (swapping
// phase between two indices would otherwise increase the sum), so the maximum is
//   branch A: theta_i = asin(kappa / s_i) for all i, when sum_i asin(kappa/s_i)
//             can reach the target -phi (mod 2 pi) for kappa in [-s_3, s_3];
//   branch B: theta_3 = pi - asin(kappa / s_3) otherwise.
// Branch A's sum is strictly increasing in kappa, so its root is unique; the
// rarely needed branch B is bracketed by a scan.  A (A^dagger A) eigen-
// decomposition by cyclic complex Jacobi rotations supplies S and V, and
// Y = U diag(e^{i theta_i}) V^dagger with U = A V S^{-1}.
#pragma once
#include "common.cuh"

namespace bri {

// Hermitian 3x3 eigen-decomposition H = V diag(e) V^dagger by Jacobi rotations.
template <typename R, typename T = typename C2<R>::T> BRI_D void herm_eig3(T H[9], T V[9], R e[3]) {
    constexpr R tol = sizeof(R) == 8 ? R(1e-34) : R(1e-13);
    constexpr int sweeps = sizeof(R) == 8 ? 20 : 6;
    auto mk2 = [](R x, R y) { T v; v.x = x; v.y = y; return v; };
    auto n2of = [](T v) { return v.x * v.x + v.y * v.y; };
#pragma unroll
    for (int i = 0; i < 9; i++) V[i] = mk2(i % 4 == 0 ? R(1) : R(0), R(0));
    for (int sweep = 0; sweep < sweeps; sweep++) {
        R off = n2of(H[1]) + n2of(H[2]) + n2of(H[5]);
        R dg = H[0].x * H[0].x + H[4].x * H[4].x + H[8].x * H[8].x;
        if (off <= tol * dg || off == R(0)) break;
#pragma unroll
        for (int pq = 0; pq < 3; pq++) {
            const int p = pq == 2 ? 1 : 0, q = pq == 0 ? 1 : 2;
            T h = H[3 * p + q];
            const R n2 = n2of(h);
            if (n2 == R(0)) continue;
            // FP64 divisions and square roots are long sequences on the FP64
            // pipe: one reciprocal square root serves |h|^-1, one the cosine
            const R ig = rsqrt(n2);
            R a = H[4 * p].x, b = H[4 * q].x;
            R tau = R(0.5) * (b - a) * ig;
            R t = (tau >= 0 ? R(1) : R(-1)) / (fabs(tau) + sqrt(fma(tau, tau, R(1))));
            R c = rsqrt(fma(t, t, R(1))), s = t * c;
            T ep = mk2(h.x * ig, -h.y * ig);  // e^{-i arg h}
            T se = cscale(ep, s), ce = cscale(ep, c);
            // H <- H J, V <- V J   (columns p, q), as FMA chains:
            //   new p = c x_p - x_q se,  new q = s x_p + x_q ce
#pragma unroll
            for (int i = 0; i < 3; i++) {
                T hp = H[3 * i + p], hq = H[3 * i + q];
                H[3 * i + p] = mk2(fma(-hq.x, se.x, fma(hq.y, se.y, c * hp.x)),
                                            fma(-hq.x, se.y, fma(-hq.y, se.x, c * hp.y)));
                H[3 * i + q] = mk2(fma(hq.x, ce.x, fma(-hq.y, ce.y, s * hp.x)),
                                            fma(hq.x, ce.y, fma(hq.y, ce.x, s * hp.y)));
                T vp = V[3 * i + p], vq = V[3 * i + q];
                V[3 * i + p] = mk2(fma(-vq.x, se.x, fma(vq.y, se.y, c * vp.x)),
                                            fma(-vq.x, se.y, fma(-vq.y, se.x, c * vp.y)));
                V[3 * i + q] = mk2(fma(vq.x, ce.x, fma(-vq.y, ce.y, s * vp.x)),
                                            fma(vq.x, ce.y, fma(vq.y, ce.x, s * vp.y)));
            }
            // H <- J^dagger H   (rows p, q):
            //   new p = c y_p - conj(se) y_q,  new q = s y_p + conj(ce) y_q
#pragma unroll
            for (int j = 0; j < 3; j++) {
                T hp = H[3 * p + j], hq = H[3 * q + j];
                H[3 * p + j] = mk2(fma(-se.x, hq.x, fma(-se.y, hq.y, c * hp.x)),
                                            fma(-se.x, hq.y, fma(se.y, hq.x, c * hp.y)));
                H[3 * q + j] = mk2(fma(ce.x, hq.x, fma(ce.y, hq.y, s * hp.x)),
                                            fma(ce.x, hq.y, fma(-ce.y, hq.x, s * hp.y)));
            }
            H[3 * p + q] = mk2(R(0), R(0));
            H[3 * q + p] = mk2(R(0), R(0));
            H[4 * p].y = 0;
            H[4 * q].y = 0;
        }
    }
    e[0] = H[0].x;
    e[1] = H[4].x;
    e[2] = H[8].x;
}

// sum_i asin(kappa/s_i) - t and its derivative (is: the reciprocals 1/s_i)
BRI_D double branch_a(const double s[3], const double is[3], double kappa, double t, double &deriv) {
    double f = -t, d = 0;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double r = kappa * is[i];
        r = fmin(1.0, fmax(-1.0, r));
        f += asin(r);
        d += rsqrt(fmax(fma(s[i], s[i], -kappa * kappa), 1e-300));
    }
    deriv = d;
    return f;
}

// root of branch A for target t, |t| <= M guaranteed by the caller
BRI_D double solve_branch_a(const double s[3], double t) {
    double lo = -s[2], hi = s[2];
    const double is[3] = {1.0 / s[0], 1.0 / s[1], 1.0 / s[2]};
    double kappa = t / (is[0] + is[1] + is[2]);
    kappa = fmin(hi, fmax(lo, kappa));
    for (int it = 0; it < 200; it++) {
        double d;
        double f = branch_a(s, is, kappa, t, d);
        if (f == 0.0) break;
        if (f > 0) hi = kappa; else lo = kappa;
        double kn = kappa - f / d;
        if (!(kn > lo && kn < hi)) kn = 0.5 * (lo + hi);
        if (fabs(kn - kappa) <= 2e-16 * s[2] || hi - lo <= 2e-16 * s[2]) { kappa = kn; break; }
        kappa = kn;
    }
    return kappa;
}

BRI_D double branch_b(const double s[3], double kappa, double t) {
    double r0 = fmin(1.0, fmax(-1.0, kappa / s[0]));
    double r1 = fmin(1.0, fmax(-1.0, kappa / s[1]));
    double r2 = fmin(1.0, fmax(-1.0, kappa / s[2]));
    return asin(r0) + asin(r1) + 3.14159265358979323846 - asin(r2) - t;
}

// maximiser of s1 cos t1 + s2 cos t2 + s3 cos t3 with t1+t2+t3 = -phi (mod 2 pi);
// s must be sorted descending and positive.
BRI_D void phase_solve(const double s[3], double phi, double th[3]) {
    const double PI = 3.14159265358979323846;
    const double c = -phi;
    const double M = asin(fmin(1.0, s[2] / s[0])) + asin(fmin(1.0, s[2] / s[1])) + 0.5 * PI;
    double best = -1e300;
    // Branch A: of the targets t = -phi + 2 pi k only the one of smallest |t|
    // (k = 0, phi in (-pi, pi]) can be the maximum -- the root kappa(t) grows in
    // |kappa| with |t| and the objective sum_i sqrt(s_i^2 - kappa^2) falls with
    // |kappa| -- and if it is out of reach (|t| > M) so are the others.
    if (fabs(c) <= M) {
        const double kappa = solve_branch_a(s, c);
#pragma unroll
        for (int i = 0; i < 3; i++) th[i] = asin(fmin(1.0, fmax(-1.0, kappa / s[i])));
        // place the rounding residue of the constraint on theta_3
        th[2] = c - th[0] - th[1];
        return;
    }
    // branch B: theta_3 = pi - asin(kappa/s_3); the target lies in (M, 2 pi - M)
    double t = c < 0 ? c + 2.0 * PI : c;
    const int NS = 64;
    double prevk = -s[2], prevg = branch_b(s, prevk, t);
    for (int i = 1; i <= NS; i++) {
        double k = -s[2] + 2.0 * s[2] * i / NS;
        double g = branch_b(s, k, t);
        if (prevg == 0.0 || (prevg < 0) != (g < 0)) {
            double lo = prevk, hi = k, glo = prevg;
            for (int it = 0; it < 80; it++) {
                double mid = 0.5 * (lo + hi);
                double gm = branch_b(s, mid, t);
                if ((gm < 0) == (glo < 0)) { lo = mid; glo = gm; } else hi = mid;
            }
            double kappa = 0.5 * (lo + hi);
            double t0 = asin(fmin(1.0, fmax(-1.0, kappa / s[0])));
            double t1 = asin(fmin(1.0, fmax(-1.0, kappa / s[1])));
            double t2 = t - t0 - t1;
            double f = s[0] * cos(t0) + s[1] * cos(t1) + s[2] * cos(t2);
            if (f > best) { best = f; th[0] = t0; th[1] = t1; th[2] = t2; }
        }
        prevk = k;
        prevg = g;
    }
}

BRI_D void swap_cols(double2 U[9], double2 V[9], int a, int b) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double2 t = U[3 * i + a]; U[3 * i + a] = U[3 * i + b]; U[3 * i + b] = t;
        t = V[3 * i + a]; V[3 * i + a] = V[3 * i + b]; V[3 * i + b] = t;
    }
}

BRI_D double2 det3(const double2 A[9]) {
    double2 m0 = csub(cmul(A[4], A[8]), cmul(A[5], A[7]));
    double2 m1 = csub(cmul(A[3], A[8]), cmul(A[5], A[6]));
    double2 m2 = csub(cmul(A[3], A[7]), cmul(A[4], A[6]));
    return cadd(csub(cmul(A[0], m0), cmul(A[1], m1)), cmul(A[2], m2));
}

// singular basis and phases of a projection (for its derivative)
struct ProjectionParts {
    double2 V[9];
    double s[3], th[3];
};

// The projection in FP64 throughout: any matrix, either branch
static __device__ __noinline__ void project_su3_general(const M3<double2> &A, M3<double2> &Y, ProjectionParts *parts) {
    double2 H[9], V[9];
    double e[3];
    // H = A^dagger A
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double2 sum = make_double2(0, 0);
#pragma unroll
            for (int k = 0; k < 3; k++) sum = cadd(sum, cmulc(A.e[3 * k + i], A.e[3 * k + j]));
            H[3 * i + j] = sum;
        }
    herm_eig3<double>(H, V, e);
    // sort eigenpairs descending
    int o[3] = {0, 1, 2};
    if (e[o[0]] < e[o[1]]) { int t = o[0]; o[0] = o[1]; o[1] = t; }
    if (e[o[1]] < e[o[2]]) { int t = o[1]; o[1] = o[2]; o[2] = t; }
    if (e[o[0]] < e[o[1]]) { int t = o[0]; o[0] = o[1]; o[1] = t; }
    double2 Vs[9];
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int i = 0; i < 3; i++) Vs[3 * i + k] = V[3 * i + o[k]];
    // U = A V S^{-1}: the columns of A V are orthogonal with norms s_k.  Taking s_k
    // as those column norms (not as square roots of the eigenvalues of A^dagger A)
    // keeps small singular values accurate; one Gram-Schmidt pass removes the
    // residual non-orthogonality.
    double2 Um[9];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int k = 0; k < 3; k++) {
            double2 sum = make_double2(0, 0);
#pragma unroll
            for (int l = 0; l < 3; l++) sum = cadd(sum, cmul(A.e[3 * i + l], Vs[3 * l + k]));
            Um[3 * i + k] = sum;
        }
    double s[3];
    const double tiny = 1e-300;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        // remove the components along the previous (orthonormal) columns
#pragma unroll
        for (int q = 0; q < k; q++) {
            double2 dot = make_double2(0, 0);
#pragma unroll
            for (int i = 0; i < 3; i++) dot = cadd(dot, cmulc(Um[3 * i + q], Um[3 * i + k]));
#pragma unroll
            for (int i = 0; i < 3; i++) Um[3 * i + k] = csub(Um[3 * i + k], cmul(Um[3 * i + q], dot));
        }
        double nrm = 0;
#pragma unroll
        for (int i = 0; i < 3; i++) nrm += cnorm2(Um[3 * i + k]);
        nrm = sqrt(nrm);
        s[k] = fmax(nrm, tiny);
#pragma unroll
        for (int i = 0; i < 3; i++) Um[3 * i + k] = cscale(Um[3 * i + k], 1.0 / s[k]);
    }
    // the ordering s_0 >= s_1 >= s_2 of the eigenvalues survives up to rounding;
    // restore it exactly for the phase solve
    if (s[0] < s[1]) { double t = s[0]; s[0] = s[1]; s[1] = t; swap_cols(Um, Vs, 0, 1); }
    if (s[1] < s[2]) { double t = s[1]; s[1] = s[2]; s[2] = t; swap_cols(Um, Vs, 1, 2); }
    if (s[0] < s[1]) { double t = s[0]; s[0] = s[1]; s[1] = t; swap_cols(Um, Vs, 0, 1); }
    // e^{i phi} = det(U V^dagger)
    double2 dU = det3(Um), dV = det3(Vs);
    double2 dd = cmulc(dV, dU);
    double phi = atan2(dd.y, dd.x);
    double th[3];
    phase_solve(s, phi, th);
    if (parts) {
#pragma unroll
        for (int i = 0; i < 9; i++) parts->V[i] = Vs[i];
#pragma unroll
        for (int k = 0; k < 3; k++) { parts->s[k] = s[k]; parts->th[k] = th[k]; }
    }
    // Y = U diag(e^{i th}) V^dagger
    double2 ph[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        double sn, cs;
        sincos(th[k], &sn, &cs);
        ph[k] = make_double2(cs, sn);
    }
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double2 sum = make_double2(0, 0);
#pragma unroll
            for (int k = 0; k < 3; k++) sum = cadd(sum, cmul(cmul(Um[3 * i + k], ph[k]), cconj(Vs[3 * j + k])));
            Y.e[3 * i + j] = sum;
        }
}

// ---- FP32 seed and FP64 refinement -------------------------------------------
// At the maximum A^dagger Y = V diag(h_i + i kappa) V^dagger with h_i = s_i
// cos(theta_i): its traceless anti-hermitian part R vanishes.  GB300 runs 64
// FP32 operations for one in FP64, and the general form above takes about
// 3,500 FP64 operations.  So V, h and Y are found in FP32 first; Y is made
// special unitary in FP64 and refined by Y <- Y exp(O), L(O) = -R, with R in
// FP64 and L inverted in the FP32 basis (L as in the derivative, force.cu): an
// error falls by the FP32 accuracy of L per step, 1e-6, 1e-12, 1e-18.  About
// 400 FP64 operations, which still bound it: 262,144 averages of six links
// exp(i 0.5 H) in 209 us instead of 3,080, the hopping fields of 16^3x32
// (path sums in FP64 then, see project_fx.cuh) in 10.1 ms instead of 52.4; the stationarity R comes out at 2e-17 |A| on
// average instead of 1e-16.  What FP32 does not settle (an exponent far from 1,
// branch B or near it, a small h, slow or no convergence, infinities and NaN)
// takes the general form.

// conversions by integer operations: the conversion instructions run at the
// FP64 rate.  Truncated; magnitudes below 2^-126 are taken as zero
BRI_D float to_f32(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v), e = hi & 0x7fffffffu;
    const unsigned m = ((e - 0x38000000u) << 3) | (lo >> 29);
    return __uint_as_float(e < 0x38100000u ? 0u : m | (hi & 0x80000000u));
}
BRI_D double to_f64(float f) {
    const unsigned u = __float_as_uint(f), e = u & 0x7fffffffu;
    const unsigned hi = ((e >> 3) + 0x38000000u) | (u & 0x80000000u);
    return e < 0x00800000u ? 0.0 : __hiloint2double((int)hi, (int)(u << 29));
}
BRI_D float2 to_f32(double2 v) { return make_float2(to_f32(v.x), to_f32(v.y)); }
BRI_D double2 to_f64(float2 v) { return make_double2(to_f64(v.x), to_f64(v.y)); }

struct ProjectionSeed {
    M3<float2> V;  // A^dagger Y = V diag(h + i kappa) V^dagger
    float h[3];
};

// V, h and Y in FP32; false where FP32 is not enough
BRI_D bool project_seed(const M3<float2> &A, ProjectionSeed &sd, M3<float2> &Y) {
    M3<float2> H = m3_mul(m3_dag(A), A);
    float e[3];
    herm_eig3<float>(H.e, sd.V.e, e);
    // U = A V / s: columns by Gram-Schmidt in descending order of s
    M3<float2> Um = m3_mul(A, sd.V);
    auto order = [&](int a, int b) {
        if (e[a] >= e[b]) return;
        const float t = e[a];
        e[a] = e[b];
        e[b] = t;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            float2 z = Um.e[3 * i + a]; Um.e[3 * i + a] = Um.e[3 * i + b]; Um.e[3 * i + b] = z;
            z = sd.V.e[3 * i + a]; sd.V.e[3 * i + a] = sd.V.e[3 * i + b]; sd.V.e[3 * i + b] = z;
        }
    };
    order(0, 1);
    order(1, 2);
    order(0, 1);
    float s[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
#pragma unroll
        for (int q = 0; q < k; q++) {
            float2 d = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 3; i++) d = cadd(d, cmulc(Um.e[3 * i + q], Um.e[3 * i + k]));
#pragma unroll
            for (int i = 0; i < 3; i++) Um.e[3 * i + k] = csub(Um.e[3 * i + k], cmul(Um.e[3 * i + q], d));
        }
        float n2 = 0.f;
#pragma unroll
        for (int i = 0; i < 3; i++) n2 += Um.e[3 * i + k].x * Um.e[3 * i + k].x + Um.e[3 * i + k].y * Um.e[3 * i + k].y;
        const float is = rsqrtf(n2);
        s[k] = n2 * is;
#pragma unroll
        for (int i = 0; i < 3; i++) Um.e[3 * i + k] = cscale(Um.e[3 * i + k], is);
    }
    if (!(s[2] > 0.02f * s[0])) return false;
    auto det = [](const M3<float2> &m) {
        const float2 m0 = csub(cmul(m.e[4], m.e[8]), cmul(m.e[5], m.e[7]));
        const float2 m1 = csub(cmul(m.e[3], m.e[8]), cmul(m.e[5], m.e[6]));
        const float2 m2 = csub(cmul(m.e[3], m.e[7]), cmul(m.e[4], m.e[6]));
        return cadd(csub(cmul(m.e[0], m0), cmul(m.e[1], m1)), cmul(m.e[2], m2));
    };
    const float2 dd = cmulc(det(sd.V), det(Um));
    const float c = -atan2f(dd.y, dd.x);
    // branch A: sum_i asin(kappa / s_i) = c, well inside its reach
    const float is[3] = {1.f / s[0], 1.f / s[1], 1.f / s[2]};
    const float smin = fminf(s[2], fminf(s[0], s[1]));
    float kappa = c / (is[0] + is[1] + is[2]);
    if (!(fabsf(kappa) < 0.9f * smin)) return false;
#pragma unroll 1
    for (int it = 0; it < 5; it++) {
        float f = -c, d = 0.f;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            f += asinf(fminf(1.f, fmaxf(-1.f, kappa * is[i])));
            d += rsqrtf(fmaxf(s[i] * s[i] - kappa * kappa, 1e-20f));
        }
        kappa = fminf(0.99f * smin, fmaxf(-0.99f * smin, kappa - f / d));
    }
    if (!(fabsf(kappa) < 0.95f * smin)) return false;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float sn = kappa * is[k], cs = sqrtf(1.f - sn * sn);
        sd.h[k] = s[k] * cs;
#pragma unroll
        for (int i = 0; i < 3; i++) Um.e[3 * i + k] = cmul(Um.e[3 * i + k], make_float2(cs, sn));
    }
    Y = m3_mul(Um, m3_dag(sd.V));
    return true;
}

// L^{-1} of a traceless anti-hermitian matrix in the FP32 basis; the result is
// anti-hermitian without rounding
BRI_D M3<float2> seed_solve(const ProjectionSeed &sd, const M3<float2> &R) {
    const M3<float2> Vd = m3_dag(sd.V);
    M3<float2> P = m3_mul(Vd, m3_mul(R, sd.V));
    float p[3], tr = 0.f, sp = 0.f, sh = 0.f;
#pragma unroll
    for (int i = 0; i < 3; i++) tr += P.e[4 * i].y;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        p[i] = P.e[4 * i].y - tr * (1.f / 3.f);
        sp += p[i] / sd.h[i];
        sh += 1.f / sd.h[i];
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        P.e[4 * i] = make_float2(0.f, (p[i] - sp / sh) / sd.h[i]);
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            // anti-hermitian part, once for both entries
            const float2 q = cscale(csub(P.e[3 * i + j], cconj(P.e[3 * j + i])), 1.f / (sd.h[i] + sd.h[j]));
            P.e[3 * i + j] = q;
            P.e[3 * j + i] = make_float2(-q.x, q.y);
        }
    }
    P = m3_mul(sd.V, m3_mul(P, Vd));
#pragma unroll
    for (int i = 0; i < 3; i++) {
        P.e[4 * i].x = 0.f;
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            const float2 q = cscale(csub(P.e[3 * i + j], cconj(P.e[3 * j + i])), 0.5f);
            P.e[3 * i + j] = q;
            P.e[3 * j + i] = make_float2(-q.x, q.y);
        }
    }
    return P;
}
// ... in FP64, traceless too
BRI_D M3<double2> su3_algebra_f64(const M3<float2> &O) {
    M3<double2> E;
#pragma unroll
    for (int i = 0; i < 9; i++) E.e[i] = to_f64(O.e[i]);
    E.e[8].y = -(E.e[0].y + E.e[4].y);
    return E;
}

// the traceless anti-hermitian part of A^dagger Y, in FP64, returned in FP32
BRI_D M3<float2> ta_residual(const M3<double2> &A, const M3<double2> &Y) {
    M3<float2> R;
    double d[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double im = 0.0;
#pragma unroll
        for (int k = 0; k < 3; k++)
            im = fma(A.e[3 * k + i].x, Y.e[3 * k + i].y, fma(-A.e[3 * k + i].y, Y.e[3 * k + i].x, im));
        d[i] = im;
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            double re = 0.0, ii = 0.0;  // of B_ij - conj(B_ji)
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const double2 ai = A.e[3 * k + i], aj = A.e[3 * k + j], yi = Y.e[3 * k + i], yj = Y.e[3 * k + j];
                re = fma(ai.x, yj.x, fma(ai.y, yj.y, re));
                re = fma(-aj.x, yi.x, fma(-aj.y, yi.y, re));
                ii = fma(ai.x, yj.y, fma(-ai.y, yj.x, ii));
                ii = fma(aj.x, yi.y, fma(-aj.y, yi.x, ii));
            }
            const float2 r = make_float2(0.5f * to_f32(re), 0.5f * to_f32(ii));
            R.e[3 * i + j] = r;
            R.e[3 * j + i] = make_float2(-r.x, r.y);
        }
    }
    const double tr = (d[0] + d[1] + d[2]) * (1.0 / 3.0);
#pragma unroll
    for (int i = 0; i < 3; i++) R.e[4 * i] = make_float2(0.f, to_f32(d[i] - tr));
    return R;
}

// row 2 = conj(row 0 x row 1) of a special unitary matrix
BRI_D void su3_third_row(M3<double2> &m) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const double2 a = m.e[(j + 1) % 3], b = m.e[3 + (j + 2) % 3], c = m.e[(j + 2) % 3], d = m.e[3 + (j + 1) % 3];
        m.e[6 + j].x = fma(a.x, b.x, fma(-a.y, b.y, fma(-c.x, d.x, c.y * d.y)));
        m.e[6 + j].y = -fma(a.x, b.y, fma(a.y, b.x, fma(-c.x, d.y, -c.y * d.x)));
    }
}

// the refined projection; false: take the general form
BRI_D bool project_fast(const M3<double2> &A, M3<double2> &Y, ProjectionSeed &sd) {
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 9; i++)
        m = max(m, max((unsigned)__double2hiint(A.e[i].x) & 0x7fffffffu, (unsigned)__double2hiint(A.e[i].y) & 0x7fffffffu));
    if (m < 0x3eb00000u || m >= 0x41400000u) return false;  // largest entry in [2^-20, 2^21)
    {
        M3<float2> A32, Y32;
#pragma unroll
        for (int i = 0; i < 9; i++) A32.e[i] = to_f32(A.e[i]);
        if (!project_seed(A32, sd, Y32)) return false;
        // special unitary in FP64: rows 0 and 1 orthonormal (their squared norms are
        // 1 + O(1e-6), the inverse square root a short series), row 2 their product
#pragma unroll
        for (int i = 0; i < 6; i++) Y.e[i] = to_f64(Y32.e[i]);
    }
#pragma unroll
    for (int r = 0; r < 2; r++) {
        if (r == 1) {
            double2 d = make_double2(0.0, 0.0);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                d.x = fma(Y.e[i].x, Y.e[3 + i].x, fma(Y.e[i].y, Y.e[3 + i].y, d.x));
                d.y = fma(Y.e[i].x, Y.e[3 + i].y, fma(-Y.e[i].y, Y.e[3 + i].x, d.y));
            }
#pragma unroll
            for (int i = 0; i < 3; i++) {
                Y.e[3 + i].x = fma(-d.x, Y.e[i].x, fma(d.y, Y.e[i].y, Y.e[3 + i].x));
                Y.e[3 + i].y = fma(-d.x, Y.e[i].y, fma(-d.y, Y.e[i].x, Y.e[3 + i].y));
            }
        }
        double n = -1.0;
#pragma unroll
        for (int i = 0; i < 3; i++) n = fma(Y.e[3 * r + i].x, Y.e[3 * r + i].x, fma(Y.e[3 * r + i].y, Y.e[3 * r + i].y, n));
        if (!(fabs(n) < 1e-5)) return false;  // the series' next term is 5/16 n^3
        const double f = fma(n, fma(n, 0.375, -0.5), 1.0);
#pragma unroll
        for (int i = 0; i < 3; i++) Y.e[3 * r + i] = cscale(Y.e[3 * r + i], f);
    }
    su3_third_row(Y);
    float last = 0.f;
#pragma unroll 1
    for (int it = 0; it < 5; it++) {
        M3<float2> O = seed_solve(sd, ta_residual(A, Y));
        float w = 0.f;
#pragma unroll
        for (int i = 0; i < 9; i++) {
            O.e[i] = make_float2(-O.e[i].x, -O.e[i].y);
            w = fmaxf(w, fmaxf(fabsf(O.e[i].x), fabsf(O.e[i].y)));
        }
        if (!(w < 2e-5f)) return false;
        if (w > 1e-10f) {
            // Y exp(O) in FP64; the terms beyond O are small enough for FP32
            const M3<float2> O2 = m3_mul(O, O), O3 = m3_mul(O, O2);
            M3<double2> E = su3_algebra_f64(O);
#pragma unroll
            for (int i = 0; i < 9; i++)
                E.e[i] = cadd(E.e[i], to_f64(cadd(cscale(O2.e[i], 0.5f), cscale(O3.e[i], 1.f / 6.f))));
            Y = m3_mad(Y, Y, E);
        } else {
            M3<float2> Y32;
#pragma unroll
            for (int i = 0; i < 9; i++) Y32.e[i] = to_f32(Y.e[i]);
            const M3<float2> D = m3_mul(Y32, O);
#pragma unroll
            for (int i = 0; i < 9; i++) Y.e[i] = cadd(Y.e[i], to_f64(D.e[i]));
        }
        // what is left is about w times this step's contraction
        if (it > 0 && w * fmaxf(w / last, 1e-7f) < 1e-17f) return true;
        if (w == 0.f) return true;
        last = w;
    }
    return false;
}

BRI_D M3<double2> project_su3(const M3<double2> &A) {
    M3<double2> Y;
    ProjectionSeed sd;
    if (!project_fast(A, Y, sd)) {
        const M3<double2> a = A;  // in memory for the call only
        M3<double2> y;
        project_su3_general(a, y, nullptr);
        Y = y;
    }
    return Y;
}

}  // namespace bri
