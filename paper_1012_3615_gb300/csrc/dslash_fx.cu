// FP64 stencil apply on the integer and FP32 pipes.
//
// GB300 runs 2 FP64 FMAs per clock and SM, but 32 integer multiply-adds
// 32 x 32 + 64 -> 64 bits and 128 FP32 FMAs, so the colour products, 11,520 of
// the 17,016 FP64 operations of a site, are taken on two-limb fixed-point
// numbers with exact integer sums:
//
//   link entries  w  = fw 2^-62,          fw = (wh + wl) 2^32, |wh| <= 2^30
//   spinors       p  = fp 2^(e(y) - 60),  fp = (ph + pl) 2^32, |ph| <= 2^28,
//                 e(y) the exponent of the largest component of site y
//   products      w p = (wh ph + wh pl + wl ph) 2^(e - 58)
//
// with integers wh, ph and |wl|, |pl| <= 1/2 kept as FP32 numbers; wl pl is
// below 2^-60 of the largest product and dropped.  A 64-bit accumulator holds
// the six high products of a colour row exactly; the twelve cross products, at
// most 2^-30 of the largest product, are summed in packed FP32 FMAs (rounded to
// 2^-24 of themselves) and added as an integer: rows and columns of a link
// have norm <= 1, so |sum wh pl + wl ph| <= 7.9 2^28 < 2^31.  The row is
// rounded to the unit 2^(X_n - 58) of its hop class n, X_n = the largest
// e(y) of the class's neighbours + h_n, and the rows are summed as 64-bit
// integers: once with the class weight lambda and once through gamma_d (entries
// +-1, +-i: additions only).  A class sum holds at most 8, 48, 96, 64 rows
// (hops x directions of gamma_d) of sqrt(6) 2^58: h_n = 0, 2, 3, 3.  Per
// class, the sums are converted and weighted in FP64.  Every row is thus known
// to about 2^-54 of its class's largest neighbour and the sums over hops are exact,
// in any order, where FP64 rounds each of ~480 partial sums: against quad
// precision 1.04e-16 relative (FP64 loop: 1.6e-16) for Gaussian spinors,
// 1.02e-16 (1.6e-16) for a field that falls by e^-2 a step in every direction.
//
// Measured: 16^3x32 0.736 ms (FP64 kernel 4.12; cross products as integers 0.887),
// 8^4 45 us (629; 62), 32^4 5.5 ms (31.2; 6.7).  Per pair and warp 144 wide
// multiply-adds (4 clocks each), 144 packed FMAs (2) and 770 other
// instructions; latency at 12 warps per SM bounds it (issue 42%, long
// scoreboard and fixed-latency waits the top stalls).
//
// A site that meets an infinity, a NaN, a spinor whose components differ by too
// many orders of magnitude (FX_WIDE) or an exponent outside the range of FP64
// scales takes the FP64 loop (fx_slow), as every site does when a link is
// not unitary (one exponent serves all links: one of another size would take
// digits from the rest of the lattice) or a field holds a NaN.
#include <algorithm>
#include <cmath>
#include <string>

#include "dslash_kernel.cuh"
#include "fx.cuh"

using namespace bri;

// canonical field list of the operator in class order (sums are kept per class)
struct FxOrder {
    unsigned char t[NCANON];    // index into Geom::hop
    unsigned char cls[NCANON];  // its class n
};

namespace {

// head room h_n of the class sums
BRI_D int fx_head(int n) { return n == 1 ? 0 : n == 2 ? 2 : 3; }

// A site's components share an exponent, so that one 2^-k of the largest keeps
// 53 - k bits.  A site where a component lies more than this many binary orders
// below the largest of its chirality (zeros included, unless all six are) is
// marked as out of range, and those that see it take the FP64 loop: out of a
// Gaussian field one site in 10^9.  The chiralities may differ by any factor:
// through gamma_d both enter every row.
constexpr unsigned FX_WIDE = 20;

// spinors to limbs [nrhs][Vp/32][12][32] and block exponents [nrhs][V], for n
// sites from s0 on (modulo V)
__global__ void k_fx_spinor(const double2 *__restrict__ in, int4 *__restrict__ p, int *__restrict__ ex, int V, int s0,
                            int n, const int *__restrict__ skip) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, rhs = blockIdx.y;
    if (i >= n || (skip && skip[rhs])) return;
    int site = s0 + i;
    if (site >= V) site -= V;
    double2 v[12];
    load_spinor(in + ((size_t)rhs * V + site) * 12, v);
    unsigned m = 0;
    bool zero = true, wide = false;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        unsigned lo = 0xffffffffu, hi = 0;
#pragma unroll
        for (int k = 6 * h; k < 6 * h + 6; k++) {
            const unsigned a = max(abs_hi(v[k].x), abs_hi(v[k].y));
            lo = min(lo, a);
            hi = max(hi, a);
            zero = zero && v[k].x == 0.0 && v[k].y == 0.0;
        }
        wide = wide || (hi >> 20) > (lo >> 20) + FX_WIDE;
        m = max(m, hi);
    }
    const int f = (int)(m >> 20);
    const bool bad = f == 2047 || wide;
    const int e = bad ? FX_BAD : zero ? FX_ZERO : f - 1022;
    ex[(size_t)rhs * V + site] = e;
    p += (size_t)rhs * 12 * ((V + 31) & ~31) + fx_at(site, 12);
#pragma unroll
    for (int k = 0; k < 12; k++)
        p[32 * k] = (bad || zero) ? make_int4(0, 0, 0, 0) : fx_split_f(v[k].x, v[k].y, FX_PB - e);
}

// one colour row of W p (SGN = 1, w = row c of W) or W^dagger p (SGN = -1,
// w = column c of W) for the two spins in p, rounded to units of
// 2^(e - 58 + sh).  pf: the spinor's high limbs as FP32 numbers
template <int SGN>
BRI_D void fx_row(const int4 w[3], const int4 p[6], const float2 pf[6], int sh, long long half, long long re[2],
                  long long im[2]) {
    // the high products' sums start at half a unit (a zero row stays zero)
    long long ar[2] = {half, half}, ai[2] = {half, half};
    float2 x[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int wr = w[k].x, wi = SGN > 0 ? w[k].z : -w[k].z, ni = SGN > 0 ? -w[k].z : w[k].z;
        const float fr = (float)wr, fi = (float)wi;
        const float lr = __int_as_float(w[k].y), li = SGN > 0 ? __int_as_float(w[k].w) : -__int_as_float(w[k].w);
        const float2 F = make_float2(fr, fi), Fi = make_float2(-fi, fr), G = make_float2(lr, li),
                     Gi = make_float2(-li, lr);
#pragma unroll
        for (int l = 0; l < 2; l++) {
            const int4 q = p[3 * l + k];
            ar[l] += (long long)wr * q.x;
            ai[l] += (long long)wr * q.z;
            ar[l] += (long long)ni * q.z;
            ai[l] += (long long)wi * q.x;
            x[l] = __ffma2_rn(F, f2(__int_as_float(q.y)), x[l]);
            x[l] = __ffma2_rn(Fi, f2(__int_as_float(q.w)), x[l]);
            x[l] = __ffma2_rn(G, f2(pf[3 * l + k].x), x[l]);
            x[l] = __ffma2_rn(Gi, f2(pf[3 * l + k].y), x[l]);
        }
    }
#pragma unroll
    for (int l = 0; l < 2; l++) {
        re[l] = (ar[l] + __float2int_rn(x[l].x)) >> sh;
        im[l] = (ai[l] + __float2int_rn(x[l].y)) >> sh;
    }
}
BRI_D void fx_negate(int4 p[6]) {
#pragma unroll
    for (int k = 0; k < 6; k++)
        p[k] = make_int4(-p[k].x, p[k].y ^ (int)0x80000000, -p[k].z, p[k].w ^ (int)0x80000000);
}

// out = diag p + v, the clover term and the sign of mode 2, for the spins 2h, 2h + 1
template <bool CLOV>
BRI_D void fx_finish(int mode, const double2 *__restrict__ in, double2 *__restrict__ out, int site, int h,
                     const Geom &g, double diag, const double2 v[6]) {
    double2 o[6], p[6];
#pragma unroll
    for (int i = 0; i < 6; i++) p[i] = in[(size_t)site * 12 + 6 * h + i];
#pragma unroll
    for (int i = 0; i < 6; i++) o[i] = make_double2(fma(diag, p[i].x, v[i].x), fma(diag, p[i].y, v[i].y));
    if constexpr (CLOV) {
        double2 c[18];
#pragma unroll
        for (int e = 0; e < 18; e++) c[e] = g.clov64[(size_t)(18 * h + e) * g.V + site];
        clover_block(c, p, o);
    }
    const double s5 = mode == 2 && h == 1 ? -1.0 : 1.0;
#pragma unroll
    for (int i = 0; i < 6; i++) out[(size_t)site * 12 + 6 * h + i] = make_double2(s5 * o[i].x, s5 * o[i].y);
}

// The FP64 loop (the arithmetic of hop_pair with run-time offsets) for one site:
// its threads part = 2 split + h share the list, leave their sums in sum (entry i
// of thread part at [12 part + i][32]) and threads 0 and 1 add them.  Called by whole
// blocks; slow: this thread's site takes part.  Bound by the FP64 pipe; every site
// this way (links of norm 1.5) on 8^4, 12^4, 16^3x32: 0.17, 0.75, 3.99 ms; one
// thread with the whole list 0.61, 1.29, 4.13; the FP64 kernel 0.63, 1.17, 4.12
template <bool CLOV>
__device__ __noinline__ void fx_slow(int mode, const LinkF64 &ll, const double2 *__restrict__ in,
                                     double2 *__restrict__ out, double2 *sum, int site, const Geom &g, double diag,
                                     int part, int parts, bool slow) {
    if (slow) {
        int x[4];
        const SiteNb nb = site_nb(g, site, x);
        AccD acc;
#pragma unroll
        for (int i = 0; i < 12; i++) acc.a[i] = make_double2(0.0, 0.0);
        const double rsign = mode == 1 ? -1.0 : 1.0;
#pragma unroll 1
        for (int t = part * g.nhop / parts; t < (part + 1) * g.nhop / parts; t++) {
            const HopArg &h = g.hop[t];
            int yf, yb;
            float phf, phb;
            hop_nb(h.dm, site, nb, yf, phf, yb, phb);
            const int n = abs(h.dm[0]) + abs(h.dm[1]) + abs(h.dm[2]) + abs(h.dm[3]);
            const double q = (double)(phf * phb), L = g.lamd[n] * (double)phf, R = g.rhod[n] * (double)phf * rsign;
            double2 cf[12];
            {
                const M3<double2> W = ll.load(h.j, site);
                double2 p[12];
                load_spinor(in + (size_t)yf * 12, p);
#pragma unroll
                for (int sp = 0; sp < 4; sp++) mv64<1>(W, p, sp, cf + 3 * sp);
            }
            const M3<double2> W = ll.load(h.j, yb);
            double2 p[12];
            load_spinor(in + (size_t)yb * 12, p);
#pragma unroll
            for (int sp = 0; sp < 4; sp++) {
                double2 cb[3];
                mv64<-1>(W, p, sp, cb);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    double2 &f = cf[3 * sp + c];
                    const double sx = fma(q, cb[c].x, f.x), sy = fma(q, cb[c].y, f.y);
                    f.x = fma(-q, cb[c].x, f.x);
                    f.y = fma(-q, cb[c].y, f.y);
                    acc.a[3 * sp + c].x = fma(L, sx, acc.a[3 * sp + c].x);
                    acc.a[3 * sp + c].y = fma(L, sy, acc.a[3 * sp + c].y);
                }
            }
#pragma unroll
            for (int mu = 0; mu < 4; mu++) {
                if (h.dm[mu] == 0) continue;
                const double rd = R * (double)h.dm[mu];
#pragma unroll
                for (int sp = 0; sp < 4; sp++) {
                    const int s = gcol(mu, sp);
                    const int gr = gre(mu, s), gi = gim(mu, s);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        if (gr != 0) acc_re(acc.a[3 * s + c], rd * (double)gr, cf[3 * sp + c]);
                        else acc_im(acc.a[3 * s + c], rd * (double)gi, cf[3 * sp + c]);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 12; i++) sum[32 * (12 * part + i)] = acc.a[i];
    }
    __syncthreads();
    if (!slow || part > 1) return;
    double2 v[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        v[i] = make_double2(0.0, 0.0);
        for (int k = 0; k < parts; k++) v[i] = cadd(v[i], sum[32 * (12 * k + 6 * part + i)]);
    }
    fx_finish<CLOV>(mode, in, out, site, part, g, diag, v);
}

// One thread per (site, chirality, split): a warp holds 32 sites, its spins
// 2h, 2h + 1, and an S-th of the class-ordered hop list; the two warps
// of a group (h = 0, 1) share the links of a pair, which they copy to shared
// memory one pair ahead (h = 0 those of x, h = 1 those of x - d), and each lane
// copies its neighbours' spinors there as soon as it has taken the last ones.  The splits
// fill the chip on small lattices.  At the end of each class its sums go to
// shared memory in FP64: lambda's to the spins' own rows, gamma_d's to the
// rows of the other chirality (to which gamma_mu maps).
constexpr int FX_REGS = 160;  // 12 warps per SM, as the shared memory allows (168: 3% slower, 128: 10%, spills)
template <int S> constexpr int FX_T = S == 4 ? 256 : 128;  // threads per block
constexpr int FX_STAGE = 2 * 9 * 32;                        // int4 of the links of a pair, 32 sites
template <int S> constexpr int FX_SMEM = FX_T<S> * (12 * 8 + 4 * 4 + 12 * 16) + (FX_T<S> / 64) * 2 * FX_STAGE * 16;

template <int N> BRI_D void fx_copy(uint32_t dst, const int4 *src) {
#pragma unroll
    for (int e = 0; e < N; e++) cp_async16(dst + 512 * e, src + 32 * e);
}
BRI_D int4 lds4i(uint32_t a) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// neighbours x + d and x - d of a pair (d uniform across the warp) and whether
// the fermion phase on the way is -1, from 8 bits of the site's position: bit mu
// is set at the top of direction mu, bit 4 + mu at the bottom (SiteNb holds
// the same in 16 registers)
BRI_D unsigned fx_edges(const Geom &g, int site) {
    unsigned m = 0;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        const int x = site % g.L[mu];
        site /= g.L[mu];
        m |= (x == g.L[mu] - 1 ? 1u << mu : 0u) | (x == 0 ? 16u << mu : 0u);
    }
    return m;
}
BRI_D void fx_nb(const int dm[4], const Geom &g, int site, unsigned edges, int &yf, int &yb, bool &nf, bool &nb) {
    unsigned wf = 0, wb = 0;  // wraps, by direction
    int stride = 1, f = site, b = site;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        const int L = g.L[mu], c = dm[mu];
        if (c != 0) {
            const unsigned up = edges >> mu & 1u, dn = edges >> (4 + mu) & 1u;
            const unsigned ff = c > 0 ? up : dn, bb = c > 0 ? dn : up;
            const int step = c > 0 ? stride : -stride, back = L * step;
            f += step - (ff ? back : 0);
            b -= step - (bb ? back : 0);
            if (g.bc[mu] < 0) {
                wf ^= ff;
                wb ^= bb;
            }
        }
        stride *= L;
    }
    yf = f;
    yb = b;
    nf = wf != 0;
    nb = wb != 0;
}

template <int S, bool CLOV>
__global__ void __maxnreg__(FX_REGS) k_dslash_fx(int mode, const int4 *__restrict__ W, const unsigned *__restrict__ info,
                                                 LinkF64 ll, const int4 *__restrict__ P, const int *__restrict__ ex,
                                                 const double2 *__restrict__ in, double2 *__restrict__ out,
                                                 const __grid_constant__ Geom g, const FxOrder ord, double diag,
                                                 const int *__restrict__ skip) {
    constexpr int T = FX_T<S>, SPB = T / (2 * S);  // threads, sites per block
    extern __shared__ __align__(16) unsigned char fx_sm[];
    double *sm = (double *)fx_sm;  // [12][T]: the result's class sums
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int h = warp & 1, grp = warp >> 1, split = grp % S, sgrp = grp / S;
    const uint32_t stage =
        (uint32_t)__cvta_generic_to_shared(fx_sm + T * 12 * 8) + (uint32_t)(grp * 2 * FX_STAGE + lane) * 16u;
    const int nblk = (g.s1 - g.s0 + SPB - 1) / SPB;
    const int nr = (int)gridDim.x / nblk;
    const int rhs = (int)blockIdx.x % nr;
    if (skip && skip[rhs]) return;
    const int want = g.s0 + ((int)blockIdx.x / nr) * SPB + sgrp * 32 + lane;
    const bool active = want < g.s1;
    const int site = active ? want : g.s1 - 1;
    const int V = g.V, nh = g.nhop;
    const size_t Vp = (size_t)((V + 31) & ~31);
    in += (size_t)rhs * V * 12;
    out += (size_t)rhs * V * 12;
    P += (size_t)rhs * 12 * Vp + 6 * 32 * h;
    ex += (size_t)rhs * V;
    const unsigned edges = fx_edges(g, site);
    // largest block exponent of each class's neighbours: the site's 2 S threads
    // take the pairs in turn
    int X[4] = {FX_ZERO, FX_ZERO, FX_ZERO, FX_ZERO};
#pragma unroll 4
    for (int i = 2 * split + h; i < nh; i += 2 * S) {
        int yf, yb;
        bool nf, nb;
        fx_nb(g.hop[ord.t[i]].dm, g, site, edges, yf, yb, nf, nb);
        const int m = max(ex[yf], ex[yb]), n = ord.cls[i];
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (n == k + 1) X[k] = max(X[k], m);
    }
    int *se = (int *)sm;
#pragma unroll
    for (int k = 0; k < 4; k++) se[k * T + tid] = X[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; k++) {
        for (int q = 0; q < 2 * S; q++) X[k] = max(X[k], se[k * T + (sgrp * 2 * S + q) * 32 + lane]);
        X[k] = X[k] == FX_ZERO ? 0 : X[k] + fx_head(k + 1);
    }
    __syncthreads();
    int *sx = (int *)(fx_sm + T * 12 * 8 + (T / 64) * 2 * FX_STAGE * 16) + tid;  // the four exponents
#pragma unroll
    for (int k = 0; k < 4; k++) sx[k * T] = X[k];
    // this lane's slots of the warp's spinor stage: 6 entries of x + d, 6 of x - d
    const uint32_t pst = (uint32_t)__cvta_generic_to_shared(fx_sm + T * (12 * 8 + 4 * 4) + (T / 64) * 2 * FX_STAGE * 16) +
                         (uint32_t)(warp * 12 * 32 + lane) * 16u;
    const int sg = h ? 1 : -1;  // gamma_1..3 change sign between the chiralities, gamma_4 does not

    long long La[12], Ga[12];  // own rows [spin][colour][re, im]; rows of the other chirality
#pragma unroll
    for (int i = 0; i < 12; i++) {
        La[i] = Ga[i] = 0;
        sm[i * T + tid] = 0.0;
    }
    const int i0 = split * nh / S, i1 = info[1] ? i0 : (split + 1) * nh / S;
    int cls = i0 < i1 ? ord.cls[i0] : 1;
    int Xn = sx[(cls - 1) * T];
    auto flush = [&](int n) {
        const double scale = __hiloint2double((1023 + Xn - FX_AB) << 20, 0);
        const double cl = g.lamd[n] * scale, cg = g.rhod[n] * (mode == 1 ? -scale : scale);
#pragma unroll
        for (int i = 0; i < 12; i++) sm[i * T + tid] = fma(fx_double(La[i], 0), cl, sm[i * T + tid]);
        asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");
#pragma unroll
        for (int i = 0; i < 12; i++) {
            sm[i * T + (tid ^ 32)] = fma(fx_double(Ga[i], 0), cg, sm[i * T + (tid ^ 32)]);
            La[i] = Ga[i] = 0;
        }
    };
    int yf = site, yb = site;
    bool nextf = false, nextb = false;
    int exf = 0, exb = 0;
    const size_t own = fx_at(site, 9);
    auto ahead = [&](int i, int buf) {  // neighbours of pair i and the copies of its links
        const HopArg &hp = g.hop[ord.t[i]];
        fx_nb(hp.dm, g, site, edges, yf, yb, nextf, nextb);
        exf = ex[yf];
        exb = ex[yb];
        fx_copy<9>(stage + (uint32_t)(buf * FX_STAGE + h * 9 * 32) * 16u,
                   W + (size_t)hp.j * 9 * Vp + (h ? fx_at(yb, 9) : own));
    };
    // a spinor's copy into the slots that this lane has read into registers
    auto spinor = [&](int y, int slot) { fx_copy<6>(pst + 512u * slot, P + fx_at(y, 12)); };
    if (i0 < i1) {
        ahead(i0, 0);
        spinor(yf, 0);
        spinor(yb, 6);
    }
    int buf = 0;
#pragma unroll 1
    for (int i = i0; i < i1; i++) {
        // this pair's copies (both warps'), and the other buffer free again
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");
        const int cef = exf, ceb = exb;
        const bool nf = nextf, ng = nextb;
        if (i + 1 < i1) ahead(i + 1, buf ^ 1);
        const HopArg &hp = g.hop[ord.t[i]];
        if (ord.cls[i] != cls) {
            flush(cls);
            cls = ord.cls[i];
            Xn = sx[(cls - 1) * T];
        }
        const uint32_t wf = stage + (uint32_t)(buf * FX_STAGE) * 16u, wb = wf + 9u * 512u;
        buf ^= 1;
        long long f[12];
        {
            int4 p[6];
#pragma unroll
            for (int k = 0; k < 6; k++) p[k] = lds4i(pst + 512u * k);
            const int sh = min(Xn - cef, 63);
            const long long half = (long long)((1ull << sh) >> 1);
            if (nf) fx_negate(p);
            float2 pf[6];
#pragma unroll
            for (int k = 0; k < 6; k++) pf[k] = make_float2((float)p[k].x, (float)p[k].z);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                int4 w[3];
#pragma unroll
                for (int k = 0; k < 3; k++) w[k] = lds4i(wf + 512u * (3 * c + k));
                long long re[2], im[2];
                fx_row<1>(w, p, pf, sh, half, re, im);
#pragma unroll
                for (int l = 0; l < 2; l++) {
                    f[6 * l + 2 * c] = re[l];
                    f[6 * l + 2 * c + 1] = im[l];
                    La[6 * l + 2 * c] += re[l];
                    La[6 * l + 2 * c + 1] += im[l];
                }
            }
        }
        if (i + 1 < i1) spinor(yf, 0);
        {
            int4 p[6];
#pragma unroll
            for (int k = 0; k < 6; k++) p[k] = lds4i(pst + 512u * (6 + k));
            const int sh = min(Xn - ceb, 63);
            const long long half = (long long)((1ull << sh) >> 1);
            if (ng) fx_negate(p);
            float2 pf[6];
#pragma unroll
            for (int k = 0; k < 6; k++) pf[k] = make_float2((float)p[k].x, (float)p[k].z);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                int4 w[3];
#pragma unroll
                for (int k = 0; k < 3; k++) w[k] = lds4i(wb + 512u * (3 * k + c));
                long long re[2], im[2];
                fx_row<-1>(w, p, pf, sh, half, re, im);
#pragma unroll
                for (int l = 0; l < 2; l++) {
                    La[6 * l + 2 * c] += re[l];
                    La[6 * l + 2 * c + 1] += im[l];
                    f[6 * l + 2 * c] -= re[l];
                    f[6 * l + 2 * c + 1] -= im[l];
                }
            }
        }
        if (i + 1 < i1) spinor(yb, 6);
        // gamma_d of the difference: additions to the other chirality's rows (for
        // h = 1 the rows gcol(mu, 2 + l) of gamma_mu; for h = 0 the same places)
        auto gamma_add = [&](int mu, bool pos) {
#pragma unroll
            for (int l = 0; l < 2; l++) {
                const int r = gcol(mu, 2 + l), gr = gre(mu, r), gi = gim(mu, r);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const long long a = f[6 * l + 2 * c], b = f[6 * l + 2 * c + 1];
                    long long &gx = Ga[6 * r + 2 * c], &gy = Ga[6 * r + 2 * c + 1];
                    const bool up = (gr + gi > 0) == pos;
                    if (gr != 0) {
                        gx = up ? gx + a : gx - a;
                        gy = up ? gy + b : gy - b;
                    } else {
                        gx = up ? gx - b : gx + b;
                        gy = up ? gy + a : gy - a;
                    }
                }
            }
        };
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            const int dm = mu < 3 ? sg * hp.dm[mu] : hp.dm[mu];  // uniform across the warp
            if (dm > 0) gamma_add(mu, true);
            else if (dm < 0) gamma_add(mu, false);
        }
    }
    // the partner may still be adding to this warp's rows: with some classes
    // switched off the last pair of a split starts a class of its own
    asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory");
    flush(cls);
    __syncthreads();
    // a site out of the fixed-point range: its sums so far are worth nothing
    bool slow = info[1] != 0;
#pragma unroll
    for (int k = 0; k < 4; k++) slow = slow || abs(sx[k * T]) > 900;
    if (split == 0 && active && !slow) {
        double2 v[6];
#pragma unroll
        for (int i = 0; i < 6; i++) {
            v[i] = make_double2(0.0, 0.0);
            for (int k = 0; k < S; k++) {
                v[i].x += sm[(2 * i) * T + tid + 64 * k];
                v[i].y += sm[(2 * i + 1) * T + tid + 64 * k];
            }
        }
        fx_finish<CLOV>(mode, in, out, site, h, g, diag, v);
    }
    if (!__syncthreads_or(slow && active)) return;
    // the spinor stages of the group's 2 S warps lie behind one another
    double2 *sum = (double2 *)(fx_sm + T * (12 * 8 + 4 * 4) + (T / 64) * 2 * FX_STAGE * 16) + sgrp * 2 * S * 12 * 32 + lane;
    fx_slow<CLOV>(mode, ll, in, out, sum, site, g, diag, 2 * split + h, 2 * S, slow && active);
}

FxOrder fx_order(const Geom &g) {
    FxOrder o{};
    int n = 0;
    for (int c = 1; c <= 4; c++)
        for (int t = 0; t < g.nhop; t++) {
            const int *d = g.hop[t].dm;
            if ((d[0] != 0) + (d[1] != 0) + (d[2] != 0) + (d[3] != 0) != c) continue;
            o.t[n] = (unsigned char)t;
            o.cls[n++] = (unsigned char)c;
        }
    return o;
}

size_t fx_vp(const Geom &g) { return (size_t)((g.V + 31) & ~31); }
size_t fx_bytes(const Geom &g, int nrhs) { return (sizeof(int4) * 12 + sizeof(int)) * fx_vp(g) * nrhs; }

template <int S, bool CLOV>
bri_status fx_launch(int mode, bri_ctx *ctx, const Geom &g, const int4 *P, const int *ex, const void *in, void *out,
                     int nrhs, double diag, const int *skip, cudaStream_t s) {
    constexpr int T = FX_T<S>, SPB = T / (2 * S);
    // the opt-in to more than 48 KB belongs to the device, as a context does
    constexpr unsigned bit = 1u << (S + (CLOV ? 8 : 0));
    if (!(ctx->fx_attr & bit)) {
        BRI_TRY_CUDA(ctx, cudaFuncSetAttribute(k_dslash_fx<S, CLOV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               FX_SMEM<S>));
        ctx->fx_attr |= bit;
    }
    const unsigned nb = (unsigned)((g.s1 - g.s0 + SPB - 1) / SPB) * (unsigned)nrhs;
    k_dslash_fx<S, CLOV><<<nb, T, FX_SMEM<S>, s>>>(mode, ctx->hopsfx, ctx->fxinfo, LinkF64{ctx->hops64, g.V}, P, ex,
                                                   (const double2 *)in, (double2 *)out, g, fx_order(g), diag, skip);
    BRI_LAUNCHED(ctx);
    return BRI_OK;
}

}  // namespace

// for an allocation of `need` bytes, step 0: work space between calls; step 1: the
// fixed-point copy, if that is enough and unless a graph of the program reads it
// (the solver's are captured again).  The next build takes the copy back if there
// is room.  False: nothing was given back
bool bri_give_back(bri_ctx *ctx, int step, size_t need) {
    if (step == 1) {
        size_t room = 0, total = 0;
        if (!ctx->hopsfx || bri_in_program_graph(ctx) || cudaMemGetInfo(&room, &total) != cudaSuccess ||
            room + sizeof(int4) * 9 * NCANON * fx_vp(ctx->g) < need) {
            cudaGetLastError();
            return false;
        }
    }
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (step == 0) {
        if (ctx->pool) cudaMemPoolTrimTo(ctx->pool, 0);
        bri_captured_free(ctx, false);
    } else {
        bri_solver_drop_graphs(ctx);
        cudaFree(ctx->hopsfx);
        ctx->hopsfx = nullptr;
        ctx->have_fx = false;
    }
    return true;
}

cudaError_t bri_malloc_bytes(bri_ctx *ctx, void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    for (int step = 0; e == cudaErrorMemoryAllocation && step < 2; step++) {
        cudaGetLastError();
        if (bri_give_back(ctx, step, bytes)) e = cudaMalloc(p, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();  // not for the next launch to report
        *p = nullptr;
    }
    return e;
}

// memory for the fixed-point copy of the FP64 fields (5,760 bytes a site) and the
// work space pool; without the copy (ctx->hopsfx null) the FP64 kernel is used.
// The copy is taken where three times as much stays free, enough for FP32 fields
// (2,880 bytes), the vectors of an FP64 solve (1,536) and the force (11,520), and
// given back where that was not enough
bri_status bri_fx_reserve(bri_ctx *ctx, cudaStream_t s) {
    const Geom &g = ctx->g;
    ctx->have_fx = false;
    if (!ctx->hopsfx && !bri_capturing(s, nullptr, nullptr)) {
        const size_t bytes = sizeof(int4) * 9 * NCANON * fx_vp(g);
        size_t room = 0, total = 0;
        if (cudaMemGetInfo(&room, &total) != cudaSuccess || room / 4 < bytes ||
            cudaMalloc(&ctx->hopsfx, bytes) != cudaSuccess) {
            cudaGetLastError();
            ctx->hopsfx = nullptr;
        }
    }
    if (!ctx->fxinfo) BRI_TRY_CUDA(ctx, bri_malloc(ctx, &ctx->fxinfo, 2 * sizeof(unsigned)));
    if (!ctx->pool) {
        cudaMemPoolProps pp{};
        pp.allocType = cudaMemAllocationTypePinned;
        pp.location.type = cudaMemLocationTypeDevice;
        pp.location.id = ctx->device;
        BRI_TRY_CUDA(ctx, cudaMemPoolCreate(&ctx->pool, &pp));
        uint64_t keep = 4ull << 30;  // bytes held between calls; released with the context
        BRI_TRY_CUDA(ctx, cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &keep));
    }
    return BRI_OK;
}

// the fixed-point apply can be used: its fields are there, and the class weights
// lie within 2^+-60 or are zero, so that their products with the class scales
// (2^+-958) stay normal numbers with all their digits.  A class whose gamma terms
// are much smaller than its others leaves the chiralities apart, which share an
// exponent (FX_WIDE)
bool bri_fx_ready(const bri_ctx *ctx) {
    if (!ctx->have_fx) return false;
    for (int n = 1; n <= 4; n++) {
        const double lam = std::fabs(ctx->g.lamd[n]), rho = std::fabs(ctx->g.rhod[n]);
        for (double w : {lam, rho})
            if (w != 0.0 && !(w >= 0x1p-60 && w <= 0x1p60)) return false;
        if (rho * (double)(1 << FX_WIDE) < lam) return false;
    }
    return true;
}

// FP64 apply of sites [g.s0, g.s1) in fixed point.  Its work space is stream-ordered
// from the context's pool, during capture held by the graph.  The right-hand
// sides done so far are counted in *ndone; fewer than nrhs with BRI_OK: no
// memory for the limb copies, the caller runs the FP64 kernel on the rest.
bri_status bri_dslash_fx(bri_ctx *ctx, const Geom &g, void *out, const void *in, int nrhs, double m0, int mode,
                         const int *skip, int *ndone, cudaStream_t s) {
    const double diag = m0 + g.lamd[0];
    const size_t field = (size_t)g.V * 12;
    // right-hand sides per launch: up to 2 GB of limb copies
    const int rmax = (int)std::max<size_t>(1, std::min<size_t>(32, ((size_t)2 << 30) / fx_bytes(g, 1)));
    if (nrhs > rmax) {
        for (int r = 0; r < nrhs && *ndone == r; r += rmax)
            BRI_RETURN_IF(bri_dslash_fx(ctx, g, (double2 *)out + r * field, (const double2 *)in + r * field,
                                        nrhs - r < rmax ? nrhs - r : rmax, m0, mode, skip ? skip + r : nullptr, ndone,
                                        s));
        return BRI_OK;
    }
    void *work = nullptr;
    unsigned long long id = 0;
    cudaGraph_t graph = nullptr;
    const bool captured = bri_capturing(s, &id, &graph);
    if (captured) {
        work = bri_captured_work(ctx, s, id, graph, fx_bytes(g, nrhs));
        if (!work) return BRI_OK;
    } else {
        const cudaError_t e = cudaMallocFromPoolAsync(&work, fx_bytes(g, nrhs), ctx->pool, s);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();
            return BRI_OK;
        }
        BRI_TRY_CUDA(ctx, e);
    }
    int4 *P = (int4 *)work;
    int *ex = (int *)(P + 12 * fx_vp(g) * nrhs);
    // a site range reads one time slice beyond each end
    const int S3 = g.L[0] * g.L[1] * g.L[2];
    const bool all = g.s0 == 0 && g.s1 == g.V;
    const long long span = (long long)g.s1 - g.s0 + 2 * S3;
    const int n = all || span >= g.V ? g.V : (int)span, first = n == g.V ? 0 : (g.s0 - S3 + g.V) % g.V;
    auto convert = [&]() -> bri_status {
        k_fx_spinor<<<dim3((unsigned)((n + 127) / 128), (unsigned)nrhs), 128, 0, s>>>((const double2 *)in, P, ex, g.V,
                                                                                      first, n, skip);
        BRI_LAUNCHED(ctx);
        return BRI_OK;
    };
    // splits of the hop list, so that the 608 schedulers have two warps or more;
    // by the lattice alone, so that a right-hand side gives the same bits alone, in
    // a batch and on a range of sites
    const int warps = 2 * ((g.V + 31) / 32);
    const int S = warps >= 2432 ? 1 : warps >= 1216 ? 2 : 4;
    auto launch = g.clov64 ? (S == 1 ? fx_launch<1, true> : S == 2 ? fx_launch<2, true> : fx_launch<4, true>)
                           : (S == 1 ? fx_launch<1, false> : S == 2 ? fx_launch<2, false> : fx_launch<4, false>);
    bri_status st = convert();
    if (st == BRI_OK) st = launch(mode, ctx, g, P, ex, in, out, nrhs, diag, skip, s);
    if (!captured) BRI_TRY_CUDA(ctx, cudaFreeAsync(work, s));
    BRI_RETURN_IF(st);
    *ndone += nrhs;
    return BRI_OK;
}
