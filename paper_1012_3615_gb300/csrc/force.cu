// Fermion force: dU += d Re(chi^dagger D[U] psi) / dU, with the hops of
// Sec. 5.1 and the projection of Sec. 5.2 differentiated exactly (U treated as
// an unconstrained complex matrix, gradient = df/dRe U + i df/dIm U).
//
// 1. hop gradients: the hop (x, d) contributes Re tr(W_d(x) Z_d(x)) with
//    Z_d(x)[c'][c] = s_d(x) sum_{a,b} chi(x)[a][c]^* M_d[a][b] psi(x+d)[b][c'],
//    M_d = lambda_n + rho_n sum_mu d_mu gamma_mu, so dW_d(x) gets Z_d(x)^dagger.
//    With W_{-d}(x+d) = W_d(x)^dagger the canonical field j collects
//    G_j(x) = Z_d(x)^dagger + Z_{-d}(x+d).
// 2. projection: Y = P(A) maximises Re tr(A^dagger Y) on SU(3), so the traceless
//    anti-hermitian part of A^dagger Y vanishes.  Writing dY = Y dOmega,
//    dOmega in su(3), the derivative of that condition is
//    L(dOmega) = -TA(dA^dagger Y), L(O) = {H, O}/2 - tr(H O)/3, with H the
//    hermitian part of A^dagger Y = V diag(s_i e^{i theta_i}) V^dagger.  In the
//    basis V, L scales the off-diagonal entries by (h_i + h_j)/2
//    (h_i = s_i cos theta_i) and is a rank-one update of diag(h) on the
//    diagonal, so it is inverted in closed form.  L is self-adjoint for
//    <X, Z> = -Re tr(X Z), which gives the vector-Jacobian product
//    G_A = -Y L^{-1}(TA(G^dagger Y)).
// 3. path sums: the averaging recursion A_d(x) = (1/n) sum F(x) A_{d'}(x') is
//    run backwards level by level (gather form, no atomics), and every
//    occurrence of a link collects its share.
#include "ctx.h"
#include "paths.cuh"
#include "project.cuh"

using namespace bri;

namespace {

// Z += conj(chi) (x) m for one colour of m: row cp of the 3x3 matrix
// (Z_cp,c += sum_a conj(chi_a,c) m_a), or its conjugate transpose's column
template <bool DAG> BRI_D void outer_add(M3<double2> &G, int cp, const double2 chi[12], const double2 m[4]) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
        double2 &z = G.e[DAG ? 3 * c + cp : 3 * cp + c];
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const double2 u = chi[3 * a + c], v = m[a];
            z.x = fma(u.x, v.x, fma(u.y, v.y, z.x));
            const double im = DAG ? -1.0 : 1.0;  // the conjugate's imaginary part
            z.y = fma(u.x, im * v.y, fma(-u.y, im * v.x, z.y));
        }
    }
}
// m = (lam + sg rho sum_mu d_mu gamma_mu) p for the four spins of one colour
BRI_D void gamma_mix(const double2 p[4], const int d[4], double lam, double rho, double2 m[4]) {
#pragma unroll
    for (int a = 0; a < 4; a++) m[a] = cscale(p[a], lam);
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        if (d[mu] == 0) continue;  // uniform across the block
        const double r = d[mu] > 0 ? rho : -rho;
#pragma unroll
        for (int a = 0; a < 4; a++) {
            const double2 v = p[gcol(mu, a)];
            const int gr = gre(mu, a), gi = gim(mu, a);
            if (gr != 0) {
                m[a].x = fma(gr > 0 ? r : -r, v.x, m[a].x);
                m[a].y = fma(gr > 0 ? r : -r, v.y, m[a].y);
            } else {
                m[a].x = fma(gi > 0 ? -r : r, v.y, m[a].x);
                m[a].y = fma(gi > 0 ? r : -r, v.x, m[a].y);
            }
        }
    }
}

// step 1 (thread per site, canonical field j = blockIdx.y).  FP64 operations
// bound it: the spin mix of a colour is taken once for its three outer
// products, 470 operations a field where one mix per matrix entry took 1,900:
// 12^4 3.13 -> 0.73 ms
__global__ void k_hop_grad(const double2 *__restrict__ chi, const double2 *__restrict__ psi, double2 *__restrict__ GA,
                           const __grid_constant__ Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (site >= g.V) return;
    const int k = canon_k(j);
    const int n = off_class(k);
    const double lam = g.lamd[n], rho = g.rhod[n];
    int x[4];
    const SiteNb nb = site_nb(g, site, x);
    int d[4];
    float ph = 1.f;
    int y = site;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        d[mu] = off_comp(k, mu);
        if (d[mu] > 0) { y += nb.fw[mu]; ph *= nb.sfw[mu]; }
        if (d[mu] < 0) { y += nb.bw[mu]; ph *= nb.sbw[mu]; }
    }
    // forward hop (x, d):   zf[cp][c] = sum_a chi(x)[a][c]^* (M_d psi(y))[a][cp]
    // reversed hop (y, -d): zb[cp][c] = sum_a chi(y)[a][c]^* (M_{-d} psi(x))[a][cp]
    // (the boundary phase of y -> x equals that of x -> y);  G = ph (zf^dagger + zb)
    M3<double2> G = m3_zero<double2>();
#pragma unroll 1
    for (int dir = 0; dir < 2; dir++) {
        const double2 *cs = chi + (size_t)(dir ? y : site) * 12, *ps = psi + (size_t)(dir ? site : y) * 12;
        double2 c12[12];
#pragma unroll
        for (int i = 0; i < 12; i++) c12[i] = cs[i];
#pragma unroll
        for (int cp = 0; cp < 3; cp++) {
            double2 p[4], m[4];
#pragma unroll
            for (int a = 0; a < 4; a++) p[a] = ps[3 * a + cp];
            gamma_mix(p, d, lam, dir ? -rho : rho, m);
            if (dir) outer_add<false>(G, cp, c12, m);
            else outer_add<true>(G, cp, c12, m);
        }
    }
#pragma unroll
    for (int e = 0; e < 9; e++) GA[((size_t)j * 9 + e) * g.V + site] = cscale(G.e[e], (double)ph);
}

// traceless anti-hermitian part
BRI_D M3<double2> ta_part(const M3<double2> &B) {
    M3<double2> P;
    const double tr = (B.e[0].y + B.e[4].y + B.e[8].y) * (1.0 / 3.0);
#pragma unroll
    for (int i = 0; i < 3; i++) {
        P.e[4 * i] = make_double2(0.0, B.e[4 * i].y - tr);
#pragma unroll
        for (int j = i + 1; j < 3; j++) {
            const double2 q = cscale(csub(B.e[3 * i + j], cconj(B.e[3 * j + i])), 0.5);
            P.e[3 * i + j] = q;
            P.e[3 * j + i] = make_double2(-q.x, q.y);
        }
    }
    return P;
}

// -Y L^{-1}(TA(G^dagger Y)) from the FP32 basis of the projection by
// refinement: L is applied in FP64 (L(X) = TA(H X)) and inverted in FP32, an
// error falls by the FP32 accuracy per step.  Two solves' worth of FP64 matrix
// products where the closed form below takes eight after an FP64
// eigendecomposition.  False: take the closed form.
BRI_D bool project_vjp_fast(const M3<double2> &A, const M3<double2> &G, M3<double2> &out) {
    M3<double2> Y, H;
    ProjectionSeed sd;
    if (!project_fast(A, Y, sd)) return false;
    M3<double2> P = ta_part(m3_mul(m3_dag(G), Y));
    {
        const M3<double2> B = m3_mul(m3_dag(A), Y);
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) H.e[3 * i + j] = cscale(cadd(B.e[3 * i + j], cconj(B.e[3 * j + i])), 0.5);
    }
    // the right-hand side scaled to about 1 for FP32
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < 9; i++)
        m = max(m, max((unsigned)__double2hiint(P.e[i].x) & 0x7fffffffu, (unsigned)__double2hiint(P.e[i].y) & 0x7fffffffu));
    const int e = (int)(m >> 20) - 1023;
    if (e > 900 || (m != 0 && e < -900)) return false;
    const double up = __hiloint2double((1023 + e) << 20, 0), dn = __hiloint2double((1023 - e) << 20, 0);
    M3<double2> Q = m3_zero<double2>();
    if (m != 0) {
#pragma unroll
        for (int i = 0; i < 9; i++) P.e[i] = cscale(P.e[i], dn);
        float last = 0.f, size = 0.f;
        bool done = false;
#pragma unroll 1
        for (int it = 0; it < 6 && !done; it++) {
            M3<float2> R;
#pragma unroll
            for (int i = 0; i < 9; i++) R.e[i] = to_f32(P.e[i]);
            R = seed_solve(sd, R);
            const M3<double2> D = su3_algebra_f64(R);
            float w = 0.f;
#pragma unroll
            for (int i = 0; i < 9; i++) {
                Q.e[i] = cadd(Q.e[i], D.e[i]);
                w = fmaxf(w, fmaxf(fabsf(R.e[i].x), fabsf(R.e[i].y)));
            }
            if (it == 0) size = w;
            // the next step would change Q by about w times this step's contraction
            done = w == 0.f || (it > 0 && w * fmaxf(w / last, 1e-7f) < 1e-17f * size);
            last = w;
            if (done) break;
            const M3<double2> L = ta_part(m3_mul(H, D));
#pragma unroll
            for (int i = 0; i < 9; i++) P.e[i] = csub(P.e[i], L.e[i]);
        }
        if (!done) return false;
    }
    out = m3_mul(Y, Q);
#pragma unroll
    for (int i = 0; i < 9; i++) out.e[i] = cscale(out.e[i], -up);
    return true;
}

// the closed form, in FP64 throughout
static __device__ __noinline__ void project_vjp_general(const M3<double2> &a, const M3<double2> &G, M3<double2> &out) {
    ProjectionParts pp;
    M3<double2> Y;
    project_su3_general(a, Y, &pp);
    // P = TA(G^dagger Y) in the basis V: P' = V^dagger TA(G^dagger Y) V
    M3<double2> B = m3_mul(m3_dag(G), Y);
    M3<double2> Vm, Vd;
    for (int i = 0; i < 9; i++) Vm.e[i] = pp.V[i];
    Vd = m3_dag(Vm);
    M3<double2> Bp = m3_mul(Vd, m3_mul(B, Vm));
    double h[3];
    for (int i = 0; i < 3; i++) h[i] = pp.s[i] * cos(pp.th[i]);
    // anti-hermitian part of Bp (the trace part is removed through the diagonal solve)
    M3<double2> Q;
    for (int i = 0; i < 3; i++)
        for (int jj = 0; jj < 3; jj++) {
            double2 pij = cscale(csub(Bp.e[3 * i + jj], cconj(Bp.e[3 * jj + i])), 0.5);
            if (i != jj) Q.e[3 * i + jj] = cscale(pij, 2.0 / (h[i] + h[jj]));
            else Q.e[3 * i + jj] = pij;
        }
    // diagonal: p_i imaginary, made traceless; q_i = (p_i + m)/h_i, sum q_i = 0
    double p[3], tr = 0;
    for (int i = 0; i < 3; i++) { p[i] = Q.e[4 * i].y; tr += p[i]; }
    for (int i = 0; i < 3; i++) p[i] -= tr / 3.0;
    double sp = 0, sh = 0;
    for (int i = 0; i < 3; i++) { sp += p[i] / h[i]; sh += 1.0 / h[i]; }
    const double m = -sp / sh;
    for (int i = 0; i < 3; i++) Q.e[4 * i] = make_double2(0.0, (p[i] + m) / h[i]);
    M3<double2> Qv = m3_mul(Vm, m3_mul(Q, Vd));
    out = m3_mul(Y, Qv);
    for (int i = 0; i < 9; i++) out.e[i] = cscale(out.e[i], -1.0);
}

// step 2: G_A = VJP of the projection (off-axis canonical fields, in place)
__global__ void k_project_vjp(const double2 *__restrict__ A, double2 *__restrict__ GA, int V) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (site >= V || off_class(canon_k(j)) < 2) return;
    const M3<double2> a = field_load<false>(A, j, V, site), G = field_load<false>(GA, j, V, site);
    M3<double2> out;
    if (!project_vjp_fast(a, G, out)) {
        const M3<double2> ac = a, Gc = G;  // in memory for the call only
        M3<double2> o;
        project_vjp_general(ac, Gc, o);
        out = o;
    }
#pragma unroll
    for (int e = 0; e < 9; e++) GA[((size_t)j * 9 + e) * V + site] = out.e[e];
}

// step 3a, fields e of class n - 1 (list f), from the fields d of class n whose
// path sums read them: for each mu outside e and both signs s, d = e + s mu,
//   A_d(x) has F_{mu,s}(x) A_e(x + s mu) / n:  G_e(y) += F_{mu,s}(x)^dagger G_d(x) / n, x = y - s mu;
// where d is not stored, -d = -e + mu is (s = -1) and has U_mu(x) A_e(y)^dagger / n,
//   x = y + e - mu:                            G_e(y) += G_{-d}(x)^dagger U_mu(x) / n
__global__ void k_path_back(int n, FieldList f, const double2 *__restrict__ A, double2 *__restrict__ GA,
                            const __grid_constant__ Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= g.V) return;
    const int j = f.j[blockIdx.y], k = canon_k(j), V = g.V;
    int x[4];
    const SiteNb nb = site_nb(g, site, x);
    M3<double2> acc = m3_zero<double2>();
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        if (off_at(k, mu) != 0) continue;
#pragma unroll 1
        for (int sg = -1; sg <= 1; sg += 2) {
            const int kd = k + sg * p3_at(mu);
            if (kd > 40) {
                const int z = site + (sg > 0 ? nb.bw[mu] : nb.fw[mu]);
                const M3<double2> Fd = sg > 0 ? field_load<true>(A, link_field(mu), V, z)
                                              : field_load<false>(A, link_field(mu), V, site);
                acc = m3_mad(acc, Fd, field_load<false>(GA, kd - 41, V, z));
            } else {
                const int z = site_at(kd, site, nb);  // y + e - mu
                acc = m3_mad(acc, field_load<true>(GA, 39 - kd, V, z), field_load<false>(A, link_field(mu), V, z));
            }
        }
    }
    const double inv = 1.0 / n;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        double2 &o = GA[((size_t)j * 9 + e) * V + site];
        o = make_double2(fma(acc.e[e].x, inv, o.x), fma(acc.e[e].y, inv, o.y));
    }
}

// step 3b: link gradients (thread per site, mu = blockIdx.y), accumulated into
// dU [V][4][9]: every stored field with d_mu != 0 has the link as the first step
// of one product
__global__ void k_link_grad(const double2 *__restrict__ A, const double2 *__restrict__ GA, double2 *__restrict__ dU,
                            const __grid_constant__ Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int mu = blockIdx.y, V = g.V;
    if (site >= V) return;
    int x[4];
    const SiteNb nb = site_nb(g, site, x);
    int xp = site;
#pragma unroll
    for (int m = 0; m < 4; m++)
        if (m == mu) xp += nb.fw[m];
    M3<double2> sum = field_load<false>(GA, link_field(mu), V, site);
    auto terms = [&](int n, M3<double2> &acc) {
#pragma unroll 1
        for (int j = 0; j < NCANON; j++) {
            const int k = canon_k(j), c = off_at(k, mu);
            if (c == 0 || off_class(k) != n) continue;
            if (c > 0) {
                // A_d(x) has U_mu(x) R: G_d(x) R^dagger
                const PathRest r = path_rest(k, mu, 1, site, nb);
                const M3<double2> Rd = r.dag ? field_load<false>(A, r.j, V, r.site) : field_load<true>(A, r.j, V, r.site);
                acc = m3_mad(acc, field_load<false>(GA, j, V, site), Rd);
            } else {
                // A_d(x + mu) has U_mu(x)^dagger A_{d + mu}(x): A_{d + mu}(x) G_d(x + mu)^dagger
                const int jr = k + p3_at(mu) - 41;  // stored: d's last component stays
                acc = m3_mad(acc, field_load<false>(A, jr, V, site), field_load<true>(GA, j, V, xp));
            }
        }
    };
#pragma unroll 1
    for (int n = 2; n <= 4; n++) {
        M3<double2> acc = m3_zero<double2>();
        terms(n, acc);
        const double inv = 1.0 / n;
#pragma unroll
        for (int e = 0; e < 9; e++) {
            sum.e[e].x = fma(acc.e[e].x, inv, sum.e[e].x);
            sum.e[e].y = fma(acc.e[e].y, inv, sum.e[e].y);
        }
    }
    double2 *o = dU + ((size_t)site * 4 + mu) * 9;
#pragma unroll
    for (int e = 0; e < 9; e++) o[e] = cadd(o[e], sum.e[e]);
}

}  // namespace

// work space: path sums and gradients of the 40 stored fields (11,520 bytes per
// site), stream-ordered from the context's pool.  12^4 (FP64 operations bound
// every step but the first): path sums 0.2 ms (0.93 over all 80 offsets in FP64), hop gradients 0.73
// (3.13), projection 1.51 (8.37), path sums backwards 0.48 (0.98), links 0.56
// (1.16)
bri_status bri_force_impl(bri_ctx *ctx, double2 *dU, const double2 *chi, const double2 *psi, cudaStream_t s) {
    const Geom &g = ctx->g;
    const size_t fields = (size_t)9 * NCANON * g.V;
    double2 *A = nullptr;
    const size_t bytes = sizeof(double2) * 2 * fields;
    cudaError_t e = cudaMallocFromPoolAsync((void **)&A, bytes, ctx->pool, s);
    for (int step = 0; e == cudaErrorMemoryAllocation && step < 2; step++) {
        cudaGetLastError();
        if (bri_give_back(ctx, step, bytes)) e = cudaMallocFromPoolAsync((void **)&A, bytes, ctx->pool, s);
    }
    if (e != cudaSuccess) cudaGetLastError();
    BRI_TRY_CUDA(ctx, e);
    double2 *GA = A + fields;
    auto run = [&]() -> bri_status {
        BRI_RETURN_IF(bri_path_sums(ctx, A, s));
        const int T = 128;
        const unsigned nb = (unsigned)((g.V + T - 1) / T);
        k_hop_grad<<<dim3(nb, NCANON), T, 0, s>>>(chi, psi, GA, g);
        BRI_LAUNCHED(ctx);
        k_project_vjp<<<dim3(nb, NCANON), T, 0, s>>>(A, GA, g.V);
        BRI_LAUNCHED(ctx);
        for (int n = 4; n >= 2; n--) {
            const FieldList f = fields_of_class(n - 1);
            k_path_back<<<dim3(nb, f.n), T, 0, s>>>(n, f, A, GA, g);
            BRI_LAUNCHED(ctx);
        }
        k_link_grad<<<dim3(nb, 4), T, 0, s>>>(A, GA, dU, g);
        BRI_LAUNCHED(ctx);
        return BRI_OK;
    };
    const bri_status st = run();
    BRI_TRY_CUDA(ctx, cudaFreeAsync(A, s));
    return st;
}
