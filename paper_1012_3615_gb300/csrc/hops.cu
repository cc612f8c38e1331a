// Link precompute: path-averaged hops (Sec. 5.1), SU(3) back-projection
// (Sec. 5.2) and storage in reduced precision / compressed SU(3) forms.
//
// Path sums by dynamic programming over the first step of every path:
//   A_d(x) = (1/n) sum_{mu in supp d} F_{mu, d_mu}(x) A_{d - d_mu mu}(x + d_mu mu),
//   F_{mu,+}(x) = U_mu(x),  F_{mu,-}(x) = U_mu(x - mu)^dagger,  A_0 = 1,
// which is the average over all n! shortest paths (every path starts with one
// of the n unit steps of d).  The factor 1/n per level only rescales A and the
// projection is invariant under positive rescaling.  Only the 40 stored offsets
// are summed: a rest d' that is not one of them is read as
// A_{d'}(y) = A_{-d'}(y + d')^dagger (path_rest), 104 matrix products per site
// instead of 208.  Level n reads level n-1 at neighbouring sites, so each level
// is one launch over (site, field), in the fields' own array: the projection
// then replaces each path sum by its field in place, so the build holds no
// second copy (5,760 bytes per site instead of 17,424).  16^3x32: 80 offsets in
// FP64 5.6 ms, 40 in FP64 2.7, 40 in fixed point (below) 0.9.
#include <cuda_fp16.h>

#include "ctx.h"
#include "fx.cuh"
#include "links.cuh"
#include "paths.cuh"
#include "project.cuh"
#include "project_fx.cuh"

using namespace bri;

namespace {

// ---- path sums in fixed point ---------------------------------------------------
// The matrix products run on the integer pipe (see dslash_fx.cu: three
// 32 x 32 -> 64-bit multiply-adds for a product, against 64 FP32 instruction
// slots for one FP64 operation): entries as two limbs of v 2^61, rows and
// columns of norm at most 1, so that with hi 2^32 + lo the sums of an entry's
// cross products stay below 2 sqrt(6) 2^60 < 2^63 and those of its high
// products, over the n terms of a level, below n sqrt(6) 2^58.  A level's sum
// is scaled by 2^-1, 2^-2, 2^-2 (n = 2, 3, 4) instead of 1/n.  Known to 2^-57.
// 16^3x32: 0.90 ms (FP64 products: 2.7), the whole build 4.45 ms, of which the
// projection takes 3.1 (project_fx.cuh).
// Links that are not unitary to 2^-16 (only their user knows what they are)
// take the FP64 form; every kernel takes the same branch.  Norms alone would not
// do: products of matrices with rows and columns of norm 1 grow to 1.73^n.
constexpr int PS_B = 61;

// unitary to 2^-16: rows of norm 1 and orthogonal, in FP32 (with the norms in
// FP64 a build of 16^3x32 took 62 us more).  to_f32 wants numbers in its range
BRI_D bool unitary_link(const double2 w[9]) {
    float2 f[9];
    unsigned m = 0;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        m = max(m, max(abs_hi(w[e].x), abs_hi(w[e].y)));
        f[e] = to_f32(w[e]);
    }
    bool ok = m <= FX_ONE;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = i; j < 3; j++) {
            float2 d = make_float2(i == j ? -1.f : 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 3; k++) d = cadd(d, cmulc(f[3 * i + k], f[3 * j + k]));
            ok = ok && d.x * d.x + d.y * d.y <= 0x1p-32f;
        }
    return ok;
}
// info[0] becomes 1 if a link is not unitary, info[1] if the apply has to read
// the FP64 fields
__global__ void k_link_check(const double2 *__restrict__ U, int n, unsigned *info) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 w[9];
#pragma unroll
    for (int e = 0; e < 9; e++) w[e] = U[(size_t)i * 9 + e];
    if (!unitary_link(w)) info[0] = 1;
}

template <bool DAG> BRI_D M3<int4> field_load_fx(const double2 *__restrict__ A, int j, int V, int site) {
    const int4 *p = reinterpret_cast<const int4 *>(A);
    M3<int4> m;
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int4 v = p[((size_t)j * 9 + (DAG ? 3 * c + r : 3 * r + c)) * V + site];
            m.e[3 * r + c] = DAG ? make_int4(v.x, v.y, -v.z, -v.w) : v;
        }
    return m;
}
// sum += F M, entry (i, j) at sum[2 (3 i + j)], in units of 2^-58
BRI_D void fx_mad(const M3<int4> &F, const M3<int4> &M, long long sum[18]) {
    constexpr unsigned long long up = (1ull << 63) + (1ull << 31);  // as in dslash_fx.cu: no sign word, rounded
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            long long re = sum[2 * (3 * i + j)] - (1ll << 31), im = sum[2 * (3 * i + j) + 1] - (1ll << 31);
            unsigned long long br = up, bi = up;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int4 w = F.e[3 * i + k], q = M.e[3 * k + j];
                re += (long long)w.x * q.x;
                im += (long long)w.x * q.z;
                br += (long long)w.x * q.y;
                bi += (long long)w.x * q.w;
                br += (long long)w.y * q.x;
                bi += (long long)w.y * q.z;
                re += (long long)-w.z * q.z;
                im += (long long)w.z * q.x;
                br += (long long)-w.z * q.w;
                bi += (long long)w.z * q.y;
                br += (long long)-w.w * q.z;
                bi += (long long)w.w * q.x;
            }
            sum[2 * (3 * i + j)] = re + (long long)(br >> 32);
            sum[2 * (3 * i + j) + 1] = im + (long long)(bi >> 32);
        }
}
// the path sum of an off-axis field as an FP64 matrix: from limbs, or as it stands
BRI_D M3<double2> path_load(const double2 *__restrict__ A, int j, int V, int site, bool fixed) {
    if (!fixed) return field_load<false>(A, j, V, site);
    const int4 *p = reinterpret_cast<const int4 *>(A);
    M3<double2> m;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        const int4 v = p[((size_t)j * 9 + e) * V + site];
        m.e[e] = make_double2(fx_double(fx_join(v.x, v.y), -PS_B), fx_double(fx_join(v.z, v.w), -PS_B));
    }
    return m;
}

// level n >= 2 of the path sums, field f.j[blockIdx.y]
__global__ void k_path_level(int n, FieldList f, double2 *__restrict__ A, const unsigned *__restrict__ info,
                             const __grid_constant__ Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    if (site >= g.V) return;
    const int j = f.j[blockIdx.y], k = canon_k(j), V = g.V;
    int x[4];
    const SiteNb nb = site_nb(g, site, x);
    if (info[0] == 0) {
        long long sum[18];
#pragma unroll
        for (int i = 0; i < 18; i++) sum[i] = 0;
#pragma unroll 1
        for (int mu = 0; mu < 4; mu++) {
            const int c = off_at(k, mu);
            if (c == 0) continue;
            const PathRest r = path_rest(k, mu, c, site, nb);
            const M3<int4> F = c > 0 ? field_load_fx<false>(A, link_field(mu), V, site)
                                     : field_load_fx<true>(A, link_field(mu), V, site + nb.bw[mu]);
            const M3<int4> M = r.dag ? field_load_fx<true>(A, r.j, V, r.site) : field_load_fx<false>(A, r.j, V, r.site);
            fx_mad(F, M, sum);
        }
        int4 *o = reinterpret_cast<int4 *>(A);
        const int sh = PS_B - 58 - (n == 2 ? 1 : 2);
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const int2 re = fx_limbs(sum[2 * e] << sh), im = fx_limbs(sum[2 * e + 1] << sh);
            o[((size_t)j * 9 + e) * V + site] = make_int4(re.x, re.y, im.x, im.y);
        }
        return;
    }
    M3<double2> acc = m3_zero<double2>();
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int c = off_at(k, mu);
        if (c == 0) continue;
        const PathRest r = path_rest(k, mu, c, site, nb);
        const M3<double2> F = c > 0 ? field_load<false>(A, link_field(mu), V, site)
                                    : field_load<true>(A, link_field(mu), V, site + nb.bw[mu]);
        const M3<double2> M = r.dag ? field_load<true>(A, r.j, V, r.site) : field_load<false>(A, r.j, V, r.site);
        acc = m3_mad(acc, F, M);
    }
    const double inv = 1.0 / n;
#pragma unroll
    for (int e = 0; e < 9; e++) A[((size_t)j * 9 + e) * V + site] = cscale(acc.e[e], inv);
}

// level 1: the links, site-fastest, as limbs or as they are
__global__ void k_path_links(const double2 *__restrict__ U, double2 *__restrict__ A, int V,
                             const unsigned *__restrict__ info) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x, mu = blockIdx.y;
    if (site >= V) return;
    const bool fixed = info[0] == 0;
    int4 *o = reinterpret_cast<int4 *>(A);
#pragma unroll
    for (int e = 0; e < 9; e++) {
        const double2 u = U[((size_t)site * 4 + mu) * 9 + e];
        const size_t i = ((size_t)link_field(mu) * 9 + e) * V + site;
        if (fixed) o[i] = fx_split(u.x, u.y, PS_B);
        else A[i] = u;
    }
}

// limbs to FP64 in place, averages over paths (the force's form of the sums)
__global__ void k_path_f64(const double2 *__restrict__ U, double2 *__restrict__ A, int V,
                           const unsigned *__restrict__ info) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (site >= V || info[0]) return;
    const int n = off_class(canon_k(j));
    if (n == 1) {
        const int mu = j == 0 ? 0 : j == 2 ? 1 : j == 8 ? 2 : 3;
#pragma unroll
        for (int e = 0; e < 9; e++) A[((size_t)j * 9 + e) * V + site] = U[((size_t)site * 4 + mu) * 9 + e];
        return;
    }
    const M3<double2> m = path_load(A, j, V, site, true);
    const double s = n == 2 ? 1.0 : 4.0 / 3.0;  // 2^-1 = 1/2; 2^-2 = (3/4) 1/3; 2^-2 = 1/4 of the level below
#pragma unroll
    for (int e = 0; e < 9; e++) A[((size_t)j * 9 + e) * V + site] = n == 2 ? m.e[e] : cscale(m.e[e], s);
}

// fields from path sums, in place: W_j(x) = U (1-hop) or P_SU(3)(A) (2..4
// hops), and their limbs where there is a fixed-point copy.  Path sums in fixed
// point are projected in it (project_fx.cuh).  168 registers: the code is longer
// than the instruction cache, three blocks an SM hide its fetches better than two
// (16^3x32: 5.56 ms a build at 255 registers, 4.50 at 168 and at 128, 5.06 with
// the FP64 refinement).
__global__ void __launch_bounds__(128, 3) k_project_hops(const double2 *__restrict__ U, double2 *__restrict__ hops64, int4 *__restrict__ fx,
                               unsigned *info, int V) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (site >= V) return;
    const bool fixed = info[0] == 0;
    M3<double2> w;
    bool unitary = false;
    if (off_class(canon_k(j)) == 1) {
        const int mu = j == 0 ? 0 : j == 2 ? 1 : j == 8 ? 2 : 3;
        unitary = fixed;
#pragma unroll
        for (int e = 0; e < 9; e++) w.e[e] = U[((size_t)site * 4 + mu) * 9 + e];
    } else {
        if (fixed) {
            const int4 *p = reinterpret_cast<const int4 *>(hops64);
            int4 A[9];
#pragma unroll
            for (int e = 0; e < 9; e++) A[e] = p[((size_t)j * 9 + e) * V + site];
            unitary = project_fast_fx(A, w);
        }
        if (!unitary) {
            w = project_su3(path_load(hops64, j, V, site, fixed));
            unitary = norm_hi(w.e) <= FX_ONE;  // not of a NaN
        }
    }
#pragma unroll
    for (int e = 0; e < 9; e++) hops64[((size_t)j * 9 + e) * V + site] = w.e[e];
    if (!fx) return;
    if (!fixed || !unitary) info[1] = 1;
    else fx_store(w.e, fx + (size_t)j * 9 * ((V + 31) & ~31), site);
}

__global__ void k_project_batch(const M3<double2> *__restrict__ A, M3<double2> *__restrict__ Y, long n) {
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    M3<double2> a = A[i];
    Y[i] = project_su3(a);
}

// ---- reduced-precision stores -------------------------------------------------
// chunk q (of nq) of field j at site s in the 32-site blocked layout of the
// FP32/FP16 stores (links.cuh): [40][Vp/32][nq][32], Vp = V rounded up to 32
BRI_D size_t blk_idx(int j, int q, int s, int nq, size_t VP) {
    return ((size_t)j * VP + (s & ~31)) * nq + (size_t)q * 32 + (s & 31);
}
BRI_HD size_t pad32(size_t V) { return (V + 31) & ~(size_t)31; }

template <bri_comp C> __global__ void k_store_f32(const double2 *__restrict__ h, LinkStore st, Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (site >= g.V) return;
    double2 w[9];
#pragma unroll
    for (int e = 0; e < 9; e++) w[e] = h[((size_t)j * 9 + e) * g.V + site];
    float4 *a = (float4 *)st.a;
    const size_t VP = pad32(g.V);
    if (C == BRI_LINK_FULL) {
#pragma unroll
        for (int q = 0; q < 4; q++)
            a[blk_idx(j, q, site, 4, VP)] =
                make_float4((float)w[2 * q].x, (float)w[2 * q].y, (float)w[2 * q + 1].x, (float)w[2 * q + 1].y);
        ((float2 *)st.b)[(size_t)j * VP + site] = make_float2((float)w[8].x, (float)w[8].y);
    } else if (C == BRI_LINK_2ROW) {
#pragma unroll
        for (int q = 0; q < 3; q++)
            a[blk_idx(j, q, site, 3, VP)] =
                make_float4((float)w[2 * q].x, (float)w[2 * q].y, (float)w[2 * q + 1].x, (float)w[2 * q + 1].y);
    } else {
        float p[8];
        eight_params(w, p);
        a[blk_idx(j, 0, site, 2, VP)] = make_float4(p[0], p[1], p[2], p[3]);
        a[blk_idx(j, 1, site, 2, VP)] = make_float4(p[4], p[5], p[6], p[7]);
    }
}

BRI_D uint32_t pack_h2(double a, double b) {
    __half2 h = __floats2half2_rn((float)a, (float)b);
    return *reinterpret_cast<uint32_t *>(&h);
}

template <bri_comp C> __global__ void k_store_f16(const double2 *__restrict__ h, LinkStore st, Geom g) {
    const int site = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (site >= g.V) return;
    double2 w[9];
#pragma unroll
    for (int e = 0; e < 9; e++) w[e] = h[((size_t)j * 9 + e) * g.V + site];
    uint4 *a = (uint4 *)st.a;
    const size_t VP = pad32(g.V);
    if (C == BRI_LINK_FULL) {
#pragma unroll
        for (int q = 0; q < 2; q++)
            a[blk_idx(j, q, site, 2, VP)] =
                make_uint4(pack_h2(w[4 * q].x, w[4 * q].y), pack_h2(w[4 * q + 1].x, w[4 * q + 1].y),
                           pack_h2(w[4 * q + 2].x, w[4 * q + 2].y), pack_h2(w[4 * q + 3].x, w[4 * q + 3].y));
        ((uint32_t *)st.b)[(size_t)j * VP + site] = pack_h2(w[8].x, w[8].y);
    } else if (C == BRI_LINK_2ROW) {
        a[blk_idx(j, 0, site, 1, VP)] = make_uint4(pack_h2(w[0].x, w[0].y), pack_h2(w[1].x, w[1].y),
                                                   pack_h2(w[2].x, w[2].y), pack_h2(w[3].x, w[3].y));
        ((uint2 *)st.b)[(size_t)j * VP + site] = make_uint2(pack_h2(w[4].x, w[4].y), pack_h2(w[5].x, w[5].y));
    } else {
        float p[8];
        eight_params(w, p);
        a[blk_idx(j, 0, site, 1, VP)] =
            make_uint4(pack_h2(p[0], p[1]), pack_h2(p[2], p[3]), pack_h2(p[4], p[5]), pack_h2(p[6], p[7]));
    }
}

// site-pair interleaved copies: entry e of field j for sites (i, i + V/2) as
// (Re_i, Re_{i+V/2}, Im_i, Im_{i+V/2}); E = 9 (full) or 6 (2-row)
template <int E> __global__ void k_store_pair_f32(const double2 *__restrict__ h, float4 *__restrict__ out, Geom g) {
    const int H = g.V / 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= H) return;
#pragma unroll
    for (int e = 0; e < E; e++) {
        const double2 wa = h[((size_t)j * 9 + e) * g.V + i], wb = h[((size_t)j * 9 + e) * g.V + i + H];
        out[((size_t)j * E + e) * H + i] = make_float4((float)wa.x, (float)wb.x, (float)wa.y, (float)wb.y);
    }
}
template <int E> __global__ void k_store_pair_f16(const double2 *__restrict__ h, uint2 *__restrict__ out, Geom g) {
    const int H = g.V / 2;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (i >= H) return;
#pragma unroll
    for (int e = 0; e < E; e++) {
        const double2 wa = h[((size_t)j * 9 + e) * g.V + i], wb = h[((size_t)j * 9 + e) * g.V + i + H];
        out[((size_t)j * E + e) * H + i] = make_uint2(pack_h2(wa.x, wb.x), pack_h2(wa.y, wb.y));
    }
}

// [40][9][V] -> [V][40][9], 32 sites x 40 entries at a time through shared
// memory: both sides in runs of 512 and 640 bytes (16^3x32 0.67 ms with one
// 16-byte store per entry and thread)
__global__ void __launch_bounds__(256) k_export_hops(const double2 *__restrict__ h, double2 *__restrict__ out, int V) {
    __shared__ double2 sm[40 * 33];
    const int s0 = blockIdx.x * 32, e0 = blockIdx.y * 40;
    for (int i = threadIdx.x; i < 40 * 32; i += 256) {
        const int e = i >> 5, s = i & 31;
        if (s0 + s < V) sm[e * 33 + s] = h[(size_t)(e0 + e) * V + s0 + s];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 40 * 32; i += 256) {
        const int s = i / 40, e = i - 40 * s;
        if (s0 + s < V) out[(size_t)(s0 + s) * (9 * NCANON) + e0 + e] = sm[e * 33 + s];
    }
}

size_t store_bytes_a(bri_prec p, bri_comp c) {
    if (p == BRI_F32) return c == BRI_LINK_FULL ? 64 : c == BRI_LINK_2ROW ? 48 : 32;
    return c == BRI_LINK_FULL ? 32 : 16;
}
size_t store_bytes_b(bri_prec p, bri_comp c) {
    if (p == BRI_F32) return c == BRI_LINK_FULL ? 8 : 0;
    return c == BRI_LINK_FULL ? 4 : c == BRI_LINK_2ROW ? 8 : 0;
}

}  // namespace

// levels 1 to 4 into A, in the form that ctx->fxinfo calls for
static bri_status path_levels(bri_ctx *ctx, double2 *A, cudaStream_t s) {
    const Geom &g = ctx->g;
    const int T = 128;
    const unsigned nb = (unsigned)((g.V + T - 1) / T);
    k_path_links<<<dim3(nb, 4), T, 0, s>>>(ctx->U, A, g.V, ctx->fxinfo);
    BRI_LAUNCHED(ctx);
    for (int n = 2; n <= 4; n++) {
        const FieldList f = fields_of_class(n);
        k_path_level<<<dim3(nb, f.n), T, 0, s>>>(n, f, A, ctx->fxinfo, g);
        BRI_LAUNCHED(ctx);
    }
    return BRI_OK;
}

bri_status bri_path_sums(bri_ctx *ctx, double2 *A, cudaStream_t s) {
    BRI_RETURN_IF(path_levels(ctx, A, s));
    k_path_f64<<<dim3((unsigned)((ctx->g.V + 127) / 128), NCANON), 128, 0, s>>>(ctx->U, A, ctx->g.V, ctx->fxinfo);
    BRI_LAUNCHED(ctx);
    return BRI_OK;
}

bri_status bri_hops_build_impl(bri_ctx *ctx, cudaStream_t s) {
    const Geom &g = ctx->g;
    if (!ctx->hops64) BRI_TRY_CUDA(ctx, bri_malloc(ctx, &ctx->hops64, sizeof(double2) * 9 * NCANON * (size_t)g.V));
    BRI_RETURN_IF(bri_fx_reserve(ctx, s));
    ctx->have64 = false;
    BRI_TRY_CUDA(ctx, cudaMemsetAsync(ctx->fxinfo, 0, 2 * sizeof(unsigned), s));
    k_link_check<<<(unsigned)(((size_t)g.V * 4 + 127) / 128), 128, 0, s>>>(ctx->U, 4 * g.V, ctx->fxinfo);
    BRI_LAUNCHED(ctx);
    BRI_RETURN_IF(path_levels(ctx, ctx->hops64, s));
    const int T = 128;
    k_project_hops<<<dim3((unsigned)((g.V + T - 1) / T), NCANON), T, 0, s>>>(ctx->U, ctx->hops64, ctx->hopsfx,
                                                                             ctx->fxinfo, g.V);
    BRI_LAUNCHED(ctx);
    ctx->have64 = true;
    ctx->have_fx = ctx->hopsfx != nullptr;
    ctx->f32.valid = false;
    ctx->f16.valid = false;
    ctx->p32.valid = false;
    ctx->p16.valid = false;
    return BRI_OK;
}

bri_status bri_hops_store_impl(bri_ctx *ctx, bri_prec prec, bri_comp comp, cudaStream_t s) {
    if (prec == BRI_F64) return BRI_OK;
    LinkStore &st = prec == BRI_F32 ? ctx->f32 : ctx->f16;
    const size_t V = ctx->g.V;
    // (re)allocate for this compression
    if (st.a && st.comp != comp) {
        cudaFree(st.a);
        if (st.b) cudaFree(st.b);
        st.a = st.b = nullptr;
    }
    st.valid = false;
    st.comp = comp;
    if (!st.a) BRI_TRY_CUDA(ctx, bri_malloc(ctx, &st.a, store_bytes_a(prec, comp) * NCANON * pad32(V)));
    const size_t nb = store_bytes_b(prec, comp);
    if (nb && !st.b) BRI_TRY_CUDA(ctx, bri_malloc(ctx, &st.b, nb * NCANON * pad32(V)));
    const int T = 128;
    dim3 grid((unsigned)((V + T - 1) / T), NCANON);
    if (prec == BRI_F32) {
        if (comp == BRI_LINK_FULL) k_store_f32<BRI_LINK_FULL><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
        else if (comp == BRI_LINK_2ROW) k_store_f32<BRI_LINK_2ROW><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
        else k_store_f32<BRI_LINK_8PARAM><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
    } else {
        if (comp == BRI_LINK_FULL) k_store_f16<BRI_LINK_FULL><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
        else if (comp == BRI_LINK_2ROW) k_store_f16<BRI_LINK_2ROW><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
        else k_store_f16<BRI_LINK_8PARAM><<<grid, T, 0, s>>>(ctx->hops64, st, ctx->g);
    }
    BRI_LAUNCHED(ctx);
    st.valid = true;
    // the site-pair copy follows on first use of its launch variant
    (prec == BRI_F32 ? ctx->p32 : ctx->p16).valid = false;
    return BRI_OK;
}

// site-pair interleaved copy of the stored fields for the pair kernel (full
// and 2-row storage, even t extent), built from the FP64 fields when the pair
// launch variant is first asked for
bri_status bri_pair_store_impl(bri_ctx *ctx, bri_prec prec, cudaStream_t s) {
    const LinkStore &st = prec == BRI_F32 ? ctx->f32 : ctx->f16;
    LinkStore &ps = prec == BRI_F32 ? ctx->p32 : ctx->p16;
    const bri_comp comp = st.comp;
    const size_t V = ctx->g.V;
    const int T = 128;
    ps.valid = false;
    if (!ctx->have64 || comp == BRI_LINK_8PARAM || ctx->g.L[3] % 2 != 0) return BRI_OK;
    const int E = comp == BRI_LINK_FULL ? 9 : 6;
    if (ps.a && ps.comp != comp) {
        cudaFree(ps.a);
        ps.a = nullptr;
    }
    if (!ps.a) BRI_TRY_CUDA(ctx, bri_malloc(ctx, &ps.a, (prec == BRI_F32 ? 16 : 8) * (size_t)E * NCANON * (V / 2)));
    ps.comp = comp;
    dim3 pg((unsigned)((V / 2 + T - 1) / T), NCANON);
    if (prec == BRI_F32) {
        if (E == 9) k_store_pair_f32<9><<<pg, T, 0, s>>>(ctx->hops64, (float4 *)ps.a, ctx->g);
        else k_store_pair_f32<6><<<pg, T, 0, s>>>(ctx->hops64, (float4 *)ps.a, ctx->g);
    } else {
        if (E == 9) k_store_pair_f16<9><<<pg, T, 0, s>>>(ctx->hops64, (uint2 *)ps.a, ctx->g);
        else k_store_pair_f16<6><<<pg, T, 0, s>>>(ctx->hops64, (uint2 *)ps.a, ctx->g);
    }
    BRI_LAUNCHED(ctx);
    ps.valid = true;
    return BRI_OK;
}

bri_status bri_project_impl(bri_ctx *ctx, double2 *Y, const double2 *A, long n, cudaStream_t s) {
    if (n == 0) return BRI_OK;
    const int T = 128;
    k_project_batch<<<(unsigned)((n + T - 1) / T), T, 0, s>>>((const M3<double2> *)A, (M3<double2> *)Y, n);
    BRI_LAUNCHED(ctx);
    return BRI_OK;
}

bri_status bri_export_hops_impl(bri_ctx *ctx, double2 *out, cudaStream_t s) {
    k_export_hops<<<dim3((unsigned)((ctx->g.V + 31) / 32), 9), 256, 0, s>>>(ctx->hops64, out, ctx->g.V);
    BRI_LAUNCHED(ctx);
    return BRI_OK;
}
