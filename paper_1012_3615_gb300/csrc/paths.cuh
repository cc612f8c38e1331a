// Field arrays [40][9][V] of the path sums and their gradients, and the
// recursion over the stored offsets that the precompute runs forwards
// (hops.cu) and the force backwards (force.cu).
#pragma once
#include "common.cuh"

namespace bri {

// stored field of the one-hop offset +mu (k = 40 + 3^mu)
BRI_HD constexpr int link_field(int mu) { return mu == 0 ? 0 : mu == 1 ? 2 : mu == 2 ? 8 : 26; }
// off_comp for a run-time direction
BRI_D int off_at(int k, int mu) {
    const int p3 = mu == 0 ? 1 : mu == 1 ? 3 : mu == 2 ? 9 : 27;
    return (k / p3) % 3 - 1;
}
BRI_D int p3_at(int mu) { return mu == 0 ? 1 : mu == 1 ? 3 : mu == 2 ? 9 : 27; }

// the stored fields of one hop class
struct FieldList {
    unsigned char j[16];
    int n;
};
inline FieldList fields_of_class(int n) {
    FieldList f{};
    for (int j = 0; j < NCANON; j++)
        if (off_class(canon_k(j)) == n) f.j[f.n++] = (unsigned char)j;
    return f;
}

template <bool DAG> BRI_D M3<double2> field_load(const double2 *__restrict__ A, int j, int V, int site) {
    M3<double2> m;
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const double2 v = A[((size_t)j * 9 + (DAG ? 3 * c + r : 3 * r + c)) * V + site];
            m.e[3 * r + c] = DAG ? cconj(v) : v;
        }
    return m;
}

// site reached by offset k
BRI_D int site_at(int k, int site, const SiteNb &nb) {
    int y = site;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        const int c = off_comp(k, mu);
        y += c > 0 ? nb.fw[mu] : c < 0 ? nb.bw[mu] : 0;
    }
    return y;
}

// the rest d' = d - c mu of a path from x that starts with the step c along mu,
// as a stored field: A_{d'}(x + c mu) directly, or A_{-d'}(x + d)^dagger
struct PathRest {
    int j, site;
    bool dag;
};
BRI_D PathRest path_rest(int k, int mu, int c, int site, const SiteNb &nb) {
    const int kr = k - c * p3_at(mu);
    PathRest r;
    r.dag = kr < 40;
    r.j = r.dag ? 39 - kr : kr - 41;
    if (r.dag) r.site = site_at(k, site, nb);
    else {
        int d = 0;
#pragma unroll
        for (int m = 0; m < 4; m++)
            if (m == mu) d = c > 0 ? nb.fw[m] : nb.bw[m];
        r.site = site + d;
    }
    return r;
}

}  // namespace bri
