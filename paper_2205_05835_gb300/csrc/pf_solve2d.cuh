// The phases of the one-launch 2D pressure solve (pf_solve2d.cu): work of one
// CTA of a cluster between two barriers, written over (thread, threads) loops
// and plain pointers, so the same functions run on the host.
//
// A CTA owns a strip of whole rows of every cluster level (levels 0 .. lc - 1);
// rows beyond its strip are read from the neighbouring CTAs' memory. Levels
// lc .. nlev - 1 live in CTA 0.
#pragma once

#include <math.h>

#include "pf_internal.h"

#ifdef __CUDACC__
#define PF_HD __host__ __device__ __forceinline__
#else
#define PF_HD inline
#endif

namespace pf {

constexpr int kS2MaxCTAs = 16;      // largest (non-portable) cluster
constexpr int kS2MaxCluster = 7;    // cluster levels and the view of level lc

// Layout of one level: sizes, coarsening to the next level (see MGLevel) and
// element offsets of its arrays in every CTA's dynamic shared memory; -1: the
// array lives in the workspace (levels 0 and 1 only).
struct S2Lev {
    int nx, ny;
    int cfx, cfy;
    float qx, qy;
    int ox, of, ow0, ow1, od;
};

struct S2Plan {
    int C;             // CTAs of the cluster
    int lc;            // first level held by CTA 0 alone
    int nlev;
    int pre, post, bottom_sweeps;
    int op, oq, oe;    // offsets of p, q, e (-1: workspace)
    int elems;         // dynamic shared memory, elements
    S2Lev lev[kMaxLevels];
};

// First row of CTA c's strip on level l <= lc (c = C: the level's end). Strips
// are multiples of the coarser levels' strips, so a coarse row's children and
// its fine rows' parents belong to the same CTA.
PF_HD int s2_row(const S2Plan& P, int l, int c) {
    if (c >= P.C) return P.lev[l].ny;
    return ((P.lev[P.lc].ny * c) / P.C) << (P.lc - l);
}

// Fits the solve of a hierarchy into a cluster's shared memory: false when it
// does not (too large a grid). single_cells: levels of at most this many cells
// go to CTA 0; cta_cells: cells of level 0 per CTA below which the cluster
// shrinks; beta_global: the face coefficients also exist in the workspace.
template <typename T>
inline bool s2_plan(const MGHier<T>& H, int single_cells, int cta_cells, int max_cluster,
                    size_t smem_bytes, bool beta_global, S2Plan& P) {
    if (H.nlev < 2 || H.lev[0].g.nz != 1) return false;
    P.nlev = H.nlev;
    P.pre = H.pre;
    P.post = H.post;
    P.bottom_sweeps = H.coarse_sweeps;
    for (int l = 0; l < H.nlev; ++l) {
        S2Lev& L = P.lev[l];
        L.nx = H.lev[l].g.nx;
        L.ny = H.lev[l].g.ny;
        L.cfx = H.lev[l].cf[0];
        L.cfy = H.lev[l].cf[1];
        L.qx = H.lev[l].lastw[0];
        L.qy = H.lev[l].lastw[1];
    }
    // the bottom must be small (a hierarchy of even halvings alone may not be)
    if (P.lev[P.nlev - 1].nx > 3 || P.lev[P.nlev - 1].ny > 3) return false;
    P.lc = 1;
    while (P.lc < P.nlev - 1 && P.lc < kS2MaxCluster - 1 &&
           P.lev[P.lc].nx * P.lev[P.lc].ny > single_cells)
        ++P.lc;
    P.C = 1;
    while (2 * P.C <= max_cluster && 2 * P.C <= kS2MaxCTAs && P.lev[P.lc].ny >= 2 * P.C &&
           (long long)P.lev[0].nx * P.lev[0].ny >= (long long)2 * P.C * cta_cells)
        P.C *= 2;
    long long off = 0;
    const long long cap = (long long)(smem_bytes / sizeof(T));
    auto take = [&](long long n) {
        const int o = (int)off;
        off += (n + 3) & ~3LL;
        return o;
    };
    auto fits = [&](int* slot, long long n) {
        *slot = -1;
        if (off + n + 3 <= cap) *slot = take(n);
        return *slot >= 0;
    };
    for (int l = P.nlev - 1; l >= 0; --l) {
        S2Lev& L = P.lev[l];
        long long rows = L.ny;
        if (l < P.lc) {
            rows = 0;
            for (int c = 0; c < P.C; ++c) {
                const int r = s2_row(P, l, c + 1) - s2_row(P, l, c);
                if (r > rows) rows = r;
            }
        }
        const long long n = rows * L.nx;
        if (l >= 1) {
            // coarse levels in shared memory; level 1, if it is a cluster level,
            // may leave what has a place in the workspace there
            const bool must = l >= P.lc || l >= 2;
            int* slots[5] = {&L.od, &L.ox, &L.ow0, &L.ow1, &L.of};
            for (int s = 0; s < 5; ++s)
                if (!fits(slots[s], n) && (must || s == 0)) return false;
        } else {
            // level 0: the arrays that neighbours read and every phase touches first
            int* slots[8] = {&L.ox, &L.ow0, &L.ow1, &L.od, &P.op, &L.of, &P.oq, &P.oe};
            for (int s = 0; s < 8; ++s) fits(slots[s], n);
        }
    }
    if (!beta_global && (P.lev[0].ow0 < 0 || P.lev[0].ow1 < 0)) return false;
    P.elems = (int)off;
    return true;
}

// One level as a CTA sees it: its rows [j0, j0 + rows) (pointers at row j0),
// and the rows around them: xm / xp of x, w1p the y-face coefficients of row
// j0 + rows (wrapped).
template <typename T>
struct S2View {
    int nx, ny, j0, rows;
    int cfx, cfy;
    int seams;          // odd axes: bit 0 x, bit 1 y; bit 2: an axis of one cell
    float qx, qy;
    float inv_nx, inv_nhx;
    T *x, *f, *w0, *w1, *di;
    T *xm, *xp, *w1p;
};

template <typename T>
PF_HD void s2_view_sizes(S2View<T>& v, const S2Lev& L, int j0, int rows) {
    v.nx = L.nx;
    v.ny = L.ny;
    v.j0 = j0;
    v.rows = rows;
    v.cfx = L.cfx;
    v.cfy = L.cfy;
    v.seams = (L.nx > 1 ? (L.nx & 1) : 4) | (L.ny > 1 ? 2 * (L.ny & 1) : 4);
    v.qx = L.qx;
    v.qy = L.qy;
    v.inv_nx = 1.0f / float(L.nx);
    v.inv_nhx = 1.0f / float((L.nx + 1) >> 1);
}
template <typename T>
PF_HD int s2_classes(const S2View<T>& L) { return 2 + 2 * ((L.seams & 1) + ((L.seams >> 1) & 1)); }

// q / n for q < 2^22 with inv = 1 / n rounded to float: q + 1/2 over n lies at
// least 1/(2n) from an integer and the two roundings move it by less.
PF_HD int s2_div(int q, float inv) { return int((float(q) + 0.5f) * inv); }

PF_HD float s2_rcp(float a) {
#ifdef __CUDA_ARCH__
    return __frcp_rn(a);
#else
    return 1.0f / a;
#endif
}
PF_HD double s2_rcp(double a) { return 1.0 / a; }

// sum of the four face coefficients times the neighbours, and of the coefficients
template <typename T>
PF_HD T s2_off(const S2View<T>& L, int r, int i, int idx) {
    const int nx = L.nx;
    const int il = i == 0 ? idx + nx - 1 : idx - 1;
    const int ir = i == nx - 1 ? idx - i : idx + 1;
    const bool last = r == L.rows - 1;
    const T xu = r == 0 ? L.xm[i] : L.x[idx - nx];
    const T xd = last ? L.xp[i] : L.x[idx + nx];
    const T wd = last ? L.w1p[i] : L.w1[idx + nx];
    return L.w0[idx] * L.x[il] + L.w0[ir] * L.x[ir] + L.w1[idx] * xu + wd * xd;
}
template <typename T>
PF_HD T s2_diag(const S2View<T>& L, int r, int i, int idx) {
    const int ir = i == L.nx - 1 ? idx - i : idx + 1;
    const T wd = r == L.rows - 1 ? L.w1p[i] : L.w1[idx + L.nx];
    return (L.w0[idx] + L.w0[ir]) + (L.w1[idx] + wd);
}

// 1 / diagonal of the strip
template <typename T>
PF_HD void s2_invdiag(const S2View<T>& L, int t, int nt) {
    const int n = L.rows * L.nx;
    for (int q = t; q < n; q += nt) {
        const int r = s2_div(q, L.inv_nx);
        L.di[q] = s2_rcp(s2_diag(L, r, q - r * L.nx, q));
    }
}

// Face coefficients of the strip of the next level (see k_coarsen_beta).
template <typename T>
PF_HD void s2_coarsen(const S2View<T>& F, const S2View<T>& C, int t, int nt) {
    const int n = C.rows * C.nx;
    const int vol = F.cfx * F.cfy;
    for (int q = t; q < n; q += nt) {
        const int R = s2_div(q, C.inv_nx);
        const int I = q - R * C.nx, J = C.j0 + R;
        const int ex = F.cfx == 1 ? 1 : (I == C.nx - 1 ? F.nx - 2 * I : 2);
        const int ey = F.cfy == 1 ? 1 : (J == C.ny - 1 ? F.ny - 2 * J : 2);
        const int i0 = F.cfx * I, j0 = F.cfy * J, base = (j0 - F.j0) * F.nx + i0;
        T s0 = T(0), s1 = T(0);
        for (int b = 0; b < ey; ++b) s0 += F.w0[base + b * F.nx];
        for (int a = 0; a < ex; ++a) s1 += F.w1[base + a];
        auto dist = [](int k, int nn, float qq) {   // of the centres of cells k - 1 and k
            return 0.5f * ((k == nn - 1 ? qq : 1.f) +
                           ((k == 0 ? nn - 1 : k - 1) == nn - 1 ? qq : 1.f));
        };
        const float rx = dist(i0, F.nx, F.qx) / (float(F.cfx) * dist(I, C.nx, C.qx));
        const float ry = dist(j0, F.ny, F.qy) / (float(F.cfy) * dist(J, C.ny, C.qy));
        // (the level's equations carry the factor h_0^2 of level 0: a quarter of
        // MGLevel's coefficient, which multiplies ih2 of its own level)
        C.w0[q] = C.nx == 1 ? T(0) : s0 * T(rx / float(vol));
        C.w1[q] = C.ny == 1 ? T(0) : s1 * T(ry / float(vol));
    }
}

PF_HD int s2_seams(int seams, int i, int j, int nx, int ny) {
    return ((seams & 1) && i == nx - 1) + ((seams & 2) && j == ny - 1);
}

// One class of a Gauss-Seidel sweep. zero: first class of a sweep that starts
// from zero (on levels with odd or one-cell axes every other cell is set to
// zero; on the others no cell is read before its class is written).
template <typename T>
PF_HD void s2_gs(const S2View<T>& L, int cls, bool zero, int t, int nt) {
    const int nx = L.nx, nhx = (nx + 1) >> 1, n = L.rows * nhx;
    const int color = cls & 1, want = cls >> 1;
    for (int q = t; q < n; q += nt) {
        const int r = s2_div(q, L.inv_nhx);
        const int m = q - r * nhx, j = L.j0 + r;
        const int par = (j + color) & 1;
        const int i = 2 * m + par, idx = r * nx + i;
        if (!L.seams) {
            L.x[idx] = (zero ? L.f[idx] : L.f[idx] + s2_off(L, r, i, idx)) * L.di[idx];
            continue;
        }
        if (i < nx) {
            if (s2_seams(L.seams, i, j, nx, L.ny) == want)
                L.x[idx] = (zero ? L.f[idx] : L.f[idx] + s2_off(L, r, i, idx)) * L.di[idx];
            else if (zero)
                L.x[idx] = T(0);
        }
        const int o = 2 * m + 1 - par;
        if (zero && o < nx) L.x[r * nx + o] = T(0);
    }
}

// f of the next level: residuals of the children over their nominal number.
// After a sweep the residual of an even level's second colour is zero; with
// one sweep from zero that of the first colour is the neighbours' part alone.
template <typename T>
PF_HD void s2_restrict(const S2View<T>& F, const S2View<T>& C, bool one_sweep, int t, int nt) {
    const int n = C.rows * C.nx;
    const T scale = T(1.0f / float(F.cfx * F.cfy));
    for (int q = t; q < n; q += nt) {
        const int R = s2_div(q, C.inv_nx);
        const int I = q - R * C.nx, J = C.j0 + R;
        T s;
        if (!F.seams && F.cfx == 2 && F.cfy == 2) {
            const int r = 2 * J - F.j0, i = 2 * I, a = r * F.nx + i, b = a + F.nx + 1;
            s = s2_off(F, r, i, a) + s2_off(F, r + 1, i + 1, b);
            if (!one_sweep)
                s += (F.f[a] - s2_diag(F, r, i, a) * F.x[a]) +
                     (F.f[b] - s2_diag(F, r + 1, i + 1, b) * F.x[b]);
        } else {
            const int ex = F.cfx == 1 ? 1 : (I == C.nx - 1 ? F.nx - 2 * I : 2);
            const int ey = F.cfy == 1 ? 1 : (J == C.ny - 1 ? F.ny - 2 * J : 2);
            s = T(0);
            for (int b = 0; b < ey; ++b)
                for (int e = 0; e < ex; ++e) {
                    const int i = F.cfx * I + e, r = F.cfy * J + b - F.j0, a = r * F.nx + i;
                    s += F.f[a] - (s2_diag(F, r, i, a) * F.x[a] - s2_off(F, r, i, a));
                }
        }
        C.f[q] = s * scale;
    }
}

// Coarse neighbour (as an offset -1, 0, +1 from the parent I0) and its weight
// along one axis (see interp_axis of pf_poisson.cu).
template <typename T>
PF_HD void s2_interp(int i, int nf, int nc, int cf, float qf, float qc, int& I0, int& o, T& w) {
    if (cf == 1) {
        I0 = i;
        o = 0;
        w = T(0);
        return;
    }
    I0 = i >> 1;
    if (I0 > nc - 1) I0 = nc - 1;
    if (qc == 1.f) {
        o = (i & 1) ? 1 : -1;
        w = T(0.25);
        return;
    }
    const float wp = 2.f * (I0 == nc - 1 ? qc : 1.f);
    const float d = float(i - 2 * I0) + 0.5f * (i == nf - 1 ? qf : 1.f) - 0.5f * wp;
    o = d >= 0.f ? 1 : -1;
    const int I1 = I0 + o;
    const bool l1 = (I1 < 0 ? nc - 1 : (I1 == nc ? 0 : I1)) == nc - 1;
    w = T((d < 0.f ? -d : d) / (0.5f * wp + (l1 ? qc : 1.f)));
}

// x += interpolation of the next level's x. On even levels only the first
// colour: the post-sweep starts by overwriting the second.
template <typename T>
PF_HD void s2_prolong(const S2View<T>& F, const S2View<T>& C, int t, int nt) {
    const bool half = !F.seams;
    const int nx = F.nx, nh = half ? nx >> 1 : nx, n = F.rows * nh;
    const float inv = half ? F.inv_nhx : F.inv_nx;
    auto row = [&](int R) { return R < 0 ? C.xm : (R >= C.rows ? C.xp : C.x + R * C.nx); };
    for (int q = t; q < n; q += nt) {
        const int r = s2_div(q, inv), m = q - r * nh, j = F.j0 + r;
        const int i = half ? 2 * m + (j & 1) : m;
        int I0, J0, oi, oj;
        T wi, wj;
        s2_interp<T>(i, nx, C.nx, F.cfx, F.qx, C.qx, I0, oi, wi);
        s2_interp<T>(j, F.ny, C.ny, F.cfy, F.qy, C.qy, J0, oj, wj);
        int I1 = I0 + oi;
        I1 = I1 < 0 ? C.nx - 1 : (I1 >= C.nx ? 0 : I1);
        const int R0 = J0 - C.j0;
        const T *c0 = row(R0), *c1 = row(R0 + oj);
        const T a = c0[I0] + wi * (c0[I1] - c0[I0]);
        const T b = c1[I0] + wi * (c1[I1] - c1[I0]);
        F.x[r * nx + i] += a + wj * (b - a);
    }
}

// Sums whose rounding is carried along: float64 sums of the float64 path,
// (hi, lo) float pairs of the mixed one (a float64 accumulation without GB300's
// narrow float64 pipe).
struct S2AccF {
    float s, c;
    PF_HD void add(float v) {
        const float t = s + v, bb = t - s;
        c += (s - (t - bb)) + (v - bb);
        s = t;
    }
    PF_HD void add_prod(float a, float b) {
        const float p = a * b;
        c += fmaf(a, b, -p);
        add(p);
    }
    PF_HD void merge(float s2, float c2) {
        add(s2);
        c += c2;
    }
    PF_HD double value() const { return double(s) + double(c); }
};
struct S2AccD {
    double s;
    PF_HD void add_prod(double a, double b) { s += a * b; }
    PF_HD double value() const { return s; }
};
template <typename T> struct S2AccOf { using type = S2AccD; };
template <> struct S2AccOf<float> { using type = S2AccF; };

// The last class (0) of the last post-sweep of level 0 with the CG products
// rz = f.x and, unless first, zq = x.q over every cell of the strip.
template <typename T, typename A>
PF_HD void s2_gs_dots(const S2View<T>& L, const T* qv, bool first, A& rz, A& zq, int t, int nt) {
    const int nx = L.nx, nhx = (nx + 1) >> 1, n = L.rows * nhx;
    for (int q = t; q < n; q += nt) {
        const int r = s2_div(q, L.inv_nhx);
        const int m = q - r * nhx, j = L.j0 + r;
        const int par = j & 1;
        const int i = 2 * m + par, o = 2 * m + 1 - par;
        if (i < nx) {
            const int idx = r * nx + i;
            const T f = L.f[idx];
            T x;
            if (!L.seams || s2_seams(L.seams, i, j, nx, L.ny) == 0) {
                x = (f + s2_off(L, r, i, idx)) * L.di[idx];
                L.x[idx] = x;
            } else {
                x = L.x[idx];
            }
            rz.add_prod(f, x);
            if (!first) zq.add_prod(x, qv[idx]);
        }
        if (o < nx) {
            const int idx = r * nx + o;
            const T x = L.x[idx];
            rz.add_prod(L.f[idx], x);
            if (!first) zq.add_prod(x, qv[idx]);
        }
    }
}

// p = z + beta p (first: p = z)
template <typename T>
PF_HD void s2_direction(const S2View<T>& L, T* p, T beta, bool first, int t, int nt) {
    const int n = L.rows * L.nx;
    for (int q = t; q < n; q += nt) p[q] = first ? L.x[q] : L.x[q] + beta * p[q];
}

// q = A p and p.q; pm, pp: the rows of p around the strip
template <typename T, typename A>
PF_HD void s2_apply(const S2View<T>& L, const T* p, const T* pm, const T* pp, T* qv, A& pq, int t,
                    int nt) {
    const int nx = L.nx, n = L.rows * nx;
    for (int q = t; q < n; q += nt) {
        const int r = s2_div(q, L.inv_nx), i = q - r * nx;
        const int il = i == 0 ? q + nx - 1 : q - 1;
        const int ir = i == nx - 1 ? q - i : q + 1;
        const bool last = r == L.rows - 1;
        const T pc = p[q];
        T ax = L.w0[q] * (pc - p[il]);
        ax += L.w0[ir] * (pc - p[ir]);
        ax += L.w1[q] * (pc - (r == 0 ? pm[i] : p[q - nx]));
        ax += (last ? L.w1p[i] : L.w1[q + nx]) * (pc - (last ? pp[i] : p[q + nx]));
        qv[q] = ax;
        pq.add_prod(pc, ax);
    }
}

// e += alpha p, r -= alpha q (r: the level's f), per-thread sum of r^2
template <typename T>
PF_HD T s2_update(const S2View<T>& L, const T* p, const T* qv, T* e, T alpha, bool first, int t,
                  int nt) {
    const int n = L.rows * L.nx;
    T rr = T(0);
    for (int q = t; q < n; q += nt) {
        e[q] = first ? alpha * p[q] : e[q] + alpha * p[q];
        const T rv = L.f[q] - alpha * qv[q];
        L.f[q] = rv;
        rr += rv * rv;
    }
    return rr;
}

}  // namespace pf
