// The phases of the one-launch 2D pressure solve (pf_solve2d.cu): work of one
// CTA of a cluster between two barriers, written over (thread, threads) loops
// and plain pointers, so the same functions run on the host.
//
// A CTA owns a strip of whole rows of every cluster level (levels 0 .. lc - 1);
// rows beyond its strip are read from the neighbouring CTAs' memory. Levels
// lc .. nlev - 1 live in CTA 0.
#pragma once

#include <math.h>
#include <string.h>

#include <type_traits>

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
    int ld;            // dense level: solved by its inverse (lc <= ld)
    int pre, post;
    int op, oq, oe, os;   // offsets of p, q, e, s (-1: workspace)
    int om;            // the dense level's inverse, padded rows of s2_pad(cells)
    int elems;         // dynamic shared memory, elements
    unsigned fused;    // bit l: s2_prolong_gs on level l (the same in every CTA)
    S2Lev lev[kMaxLevels];
};

// Row pitch of the dense inverse: 8 segments of a row are read at once, pitch 8
// mod 32 puts four rows of them on different banks (4-byte elements).
PF_HD int s2_pad(int n) { return ((n + 31) & ~31) + 8; }

// First row of CTA c's strip on level l <= lc (c = C: the level's end). Strips
// are multiples of the coarser levels' strips, so a coarse row's children and
// its fine rows' parents belong to the same CTA.
PF_HD int s2_row(const S2Plan& P, int l, int c) {
    if (c >= P.C) return P.lev[l].ny;
    return ((P.lev[P.lc].ny * c) / P.C) << (P.lc - l);
}
inline int s2_max_rows(const S2Plan& P, int l) {
    if (l >= P.lc) return P.lev[l].ny;
    int m = 0;
    for (int c = 0; c < P.C; ++c) {
        const int r = s2_row(P, l, c + 1) - s2_row(P, l, c);
        if (r > m) m = r;
    }
    return m;
}

// What decides the plan: the largest cluster, the dense level's cells, the
// strip's cells up to which the interpolation joins the first post class, the
// largest strip (cells of level 0 per CTA), that of a split that is not the
// cheapest, the dynamic shared memory, and a cost model of an iteration in
// cycles: per cell of the largest strip, per cell of the levels of CTA 0, per
// phase of a cluster and of a CTA.
struct S2Limits {
    int max_cluster, dense_cells, fused_cells, cta_cells, other_cells;
    float cell, single_cell, phase, cta_phase;
    size_t smem_bytes;
};
constexpr int kS2DenseMax = 32;   // cells of a dense level (see s2_gj_publish)
// Largest strip. Beyond it the kernels on the whole chip are faster: a graph step
// of a 512^2 drop takes 2.7 ms in the cluster and 3.0 ms there in mixed precision,
// 7.9 and 8.5 ms in float64 (larger ones do not fit); a mixed step of 576^2 took
// 7.6 and 4.7 ms where one of 512^2 took 3.7 and 4.5.
constexpr int kS2CtaCells = kSolve2dCells / kS2MaxCTAs;
// Shared memory of a CTA, and what the kernel's static arrays leave of it (the
// launch asks the kernel itself; this decides the workspace, without a GPU).
constexpr size_t kS2SmemMax = 227 * 1024;
template <typename T>
constexpr size_t s2_dynamic_smem() {
    return kS2SmemMax - (sizeof(T) == 4 ? 5 : 17) * 1024;
}

template <typename T>
inline S2Limits s2_limits(int max_cluster, size_t smem_bytes) {
    // Cycles measured at 64^2 .. 256^2: a phase of a cluster costs about 900
    // beside its cells, one of a CTA 400. The fused interpolation has 31
    // instructions a cell instead of 4, too many for the float64 pipe.
    const bool f32 = sizeof(T) == 4;
    S2Limits m;
    m.max_cluster = max_cluster;
    m.dense_cells = f32 ? kS2DenseMax : 16;
    m.fused_cells = f32 ? 2048 : 0;
    m.cta_cells = kS2CtaCells;
    m.other_cells = f32 ? 13500 : 9500;
    m.cell = f32 ? 8.f : 28.f;
    m.single_cell = f32 ? 5.f : 13.f;
    m.phase = 900.f;
    m.cta_phase = 400.f;
    m.smem_bytes = smem_bytes;
    return m;
}

// Modelled cycles of an iteration of a split (C and lc chosen).
inline float s2_cost(const S2Plan& P, int nlev, const S2Limits& lim) {
    auto cells = [&](int l) { return P.lev[l].nx * P.lev[l].ny; };
    float c = 5.f * float(P.lc) * (P.C == 1 ? lim.cta_phase : lim.phase);
    for (int l = 0; l < P.lc; ++l)
        c += (l == 0 ? lim.cell : lim.single_cell) * float(s2_max_rows(P, l) * P.lev[l].nx);
    for (int l = P.lc; l < nlev && cells(l) > lim.dense_cells; ++l)
        c += lim.single_cell * float(cells(l)) + 5.f * lim.cta_phase;
    return c;
}

// Places a plan's arrays (C and lc chosen): false when they do not fit.
inline bool s2_place(S2Plan& P, const S2Limits& lim, size_t elem, bool beta_global,
                     bool s_global) {
    auto cells = [&](int l) { return P.lev[l].nx * P.lev[l].ny; };
    if ((long long)s2_max_rows(P, 0) * P.lev[0].nx > lim.cta_cells) return false;
    P.ld = P.lc;
    while (cells(P.ld) > lim.dense_cells) ++P.ld;
    long long off = 0;
    const long long cap = (long long)(lim.smem_bytes / elem);
    auto fits = [&](int* slot, long long n) {
        *slot = -1;
        if (off + n + 3 > cap) return false;
        *slot = (int)off;
        off += (n + 3) & ~3LL;
        return true;
    };
    if (!fits(&P.om, (long long)cells(P.ld) * s2_pad(cells(P.ld)))) return false;
    for (int l = P.ld; l >= 1; --l) {
        // coarse levels in shared memory; level 1, if it is a cluster level,
        // may leave what has a place in the workspace there
        S2Lev& L = P.lev[l];
        const long long n = (long long)s2_max_rows(P, l) * L.nx;
        const bool must = l >= P.lc || l >= 2;
        int* slots[5] = {&L.od, &L.ox, &L.ow0, &L.ow1, &L.of};
        for (int s = 0; s < 5; ++s)
            if (!fits(slots[s], n) && (must || s == 0)) return false;
    }
    // level 0, in the order of use
    S2Lev& L = P.lev[0];
    const long long n0 = (long long)s2_max_rows(P, 0) * L.nx;
    int* slots[9] = {&L.ox, &L.ow0, &L.ow1, &L.of, &L.od, &P.os, &P.oq, &P.op, &P.oe};
    for (int s = 0; s < 9; ++s) fits(slots[s], n0);
    if (P.os < 0 && !s_global && L.ox < 0) return false;   // (x's workspace place is free)
    if (!beta_global && (L.ow0 < 0 || L.ow1 < 0)) return false;
    P.fused = 0;
    for (int l = 0; l < P.ld; ++l) {
        const S2Lev &F = P.lev[l], &N = P.lev[l + 1];
        const bool even = F.nx > 1 && F.ny > 1 && F.nx % 2 == 0 && F.ny % 2 == 0;
        if (even && N.qx == 1.f && N.qy == 1.f && s2_max_rows(P, l) * F.nx <= lim.fused_cells)
            P.fused |= 1u << l;
    }
    P.elems = (int)off;
    return true;
}

// The plan of a hierarchy's solve: of the splits that fit a cluster's shared
// memory the one with the least modelled cost (more cluster levels make the
// strips coarser and unequal, fewer leave more to CTA 0); false when none does.
// beta_global: the face coefficients also exist in the workspace; s_global: so
// does a place for s.
template <typename T>
inline bool s2_plan(const MGHier<T>& H, const S2Limits& lim, bool beta_global, bool s_global,
                    S2Plan& P) {
    if (H.nlev < 2 || H.lev[0].g.nz != 1) return false;
    S2Plan Q;
    Q.pre = H.pre;
    Q.post = H.post;
    for (int l = 0; l < H.nlev; ++l) {
        S2Lev& L = Q.lev[l];
        L.nx = H.lev[l].g.nx;
        L.ny = H.lev[l].g.ny;
        L.cfx = H.lev[l].cf[0];
        L.cfy = H.lev[l].cf[1];
        L.qx = H.lev[l].lastw[0];
        L.qy = H.lev[l].lastw[1];
    }
    // the bottom must be small (a hierarchy of even halvings alone may not be)
    if (H.lev[H.nlev - 1].g.ncell > lim.dense_cells) return false;
    float best = -1.f, least = -1.f;
    for (int lc = 1; lc < H.nlev && lc < kS2MaxCluster; ++lc)
        for (int C = 1; C <= lim.max_cluster && C <= kS2MaxCTAs && C <= Q.lev[lc].ny; C *= 2) {
            Q.lc = lc;
            Q.C = C;
            const float c = s2_cost(Q, H.nlev, lim);
            if (least < 0.f || c < least) least = c;
            if (best >= 0.f && c >= best) continue;
            if (!s2_place(Q, lim, sizeof(T), beta_global, s_global)) continue;
            best = c;
            P = Q;
        }
    if (best < 0.f) return false;
    // A split that is not the cheapest has unequal strips or more in CTA 0, and
    // the kernels overtake it sooner, on odd sizes (three classes a sweep) sooner
    // yet. Graph steps, strip's cells: cluster and kernels. Float64: 268^2 (7504)
    // 5.0 and 6.3 ms, 468 x 156 (9360) 6.3 and 7.6, 692 x 144 (11072) 7.0 and 6.7, 548 x 164
    // (10960) 7.8 and 6.3; odd: 313 x 54 (3130) 5.5 and 8.5, 301 x 299 (8428) 13.1 and
    // 9.5. Mixed: 468 x 276 (13104) 2.7 and 3.0, 704 x 188 (14080) equal, 580 x 276
    // (16240) 4.8 and 3.3.
    const int n0 = s2_max_rows(P, 0) * P.lev[0].nx;
    const bool odd = (P.lev[0].nx | P.lev[0].ny) & 1;
    return best == least || n0 <= (odd ? lim.other_cells / 2 : lim.other_cells);
}

// One level as a CTA sees it: its rows [j0, j0 + rows) (pointers at row j0),
// and the rows around them: xm / xp of x, w1p the y-face coefficients of row
// j0 + rows (wrapped).
template <typename T>
struct S2View {
    int nx, ny, j0, rows;
    int cfx, cfy;
    int seams;          // odd axes: bit 0 x, bit 1 y; bit 2: an axis of one cell
    int lf, lh;         // log2 of the threads along a row: cells, pairs of cells
    float qx, qy;
    T *x, *f, *w0, *w1, *di;
    T *xm, *xp, *w1p;
};

constexpr int kS2Threads = 512;

PF_HD int s2_log2(int n) {   // threads along a row of n items
    int l = 0;
    while ((1 << l) < n && (2 << l) <= kS2Threads) ++l;
    return l;
}
template <typename T>
PF_HD void s2_view_sizes(S2View<T>& v, const S2Lev& L, int j0, int rows) {
    v.nx = L.nx;
    v.ny = L.ny;
    v.j0 = j0;
    v.rows = rows;
    v.cfx = L.cfx;
    v.cfy = L.cfy;
    v.seams = (L.nx > 1 ? (L.nx & 1) : 4) | (L.ny > 1 ? 2 * (L.ny & 1) : 4);
    v.lf = s2_log2(L.nx);
    v.lh = s2_log2((L.nx + 1) >> 1);
    v.qx = L.qx;
    v.qy = L.qy;
}
template <typename T>
PF_HD int s2_classes(const S2View<T>& L) { return L.seams ? 3 : 2; }

// Loops of a CTA's threads over its cells (f(r, i)) or pairs (2m, 2m + 1) of
// cells of a row (f(r, m)): powers of two of threads along a row, so no thread
// divides by the level's size.
template <typename F>
PF_HD void s2_cells(int n, int rows, int lw, int t, F f) {
    const int i0 = t & ((1 << lw) - 1);
    for (int r = t >> lw; r < rows; r += kS2Threads >> lw)
        for (int i = i0; i < n; i += 1 << lw) f(r, i);
}

// The same for val(r, i), which only reads, and put(r, i, value): a thread with
// several rows forms two rows' values before it stores the first, so that their
// loads overlap (a store between them would order them). More rows at once, or
// predicated ones, slowed the many phases with one row a thread by a quarter.
template <typename V, typename F, typename G>
PF_HD void s2_map(int n, int rows, int lw, int t, F val, G put) {
    const int i0 = t & ((1 << lw) - 1), dr = kS2Threads >> lw;
    int r = t >> lw;
    if (!std::is_same<V, double>::value && sizeof(V) <= 8)   // (float64 phases wait for the pipe)
        for (; r + dr < rows; r += 2 * dr)
            for (int i = i0; i < n; i += 1 << lw) {
                const V a = val(r, i), b = val(r + dr, i);
                put(r, i, a);
                put(r + dr, i, b);
            }
    for (; r < rows; r += dr)
        for (int i = i0; i < n; i += 1 << lw) put(r, i, val(r, i));
}

PF_HD float s2_rcp(float a) {
#ifdef __CUDA_ARCH__
    return __frcp_rn(a);
#else
    return 1.0f / a;
#endif
}
PF_HD double s2_rcp(double a) { return 1.0 / a; }

// The four neighbours of a cell of the strip: offsets along the row, and the
// rows above and below (chosen before the load, so the loads of a cell issue
// together).
template <typename T>
struct S2Nb {
    int il, ir;
    const T *xu, *xd, *wd;
};
template <typename T>
PF_HD S2Nb<T> s2_nb(const S2View<T>& L, int r, int i, int idx) {
    const int nx = L.nx;
    S2Nb<T> n;
    n.il = i == 0 ? idx + nx - 1 : idx - 1;
    n.ir = i == nx - 1 ? idx - i : idx + 1;
    const bool last = r == L.rows - 1;
    n.xu = r == 0 ? L.xm + i : L.x + (idx - nx);
    n.xd = last ? L.xp + i : L.x + (idx + nx);
    n.wd = last ? L.w1p + i : L.w1 + (idx + nx);
    return n;
}
// a plus the sum of the four face coefficients times the neighbours; the sum of
// the coefficients
template <typename T>
PF_HD T s2_off(const S2View<T>& L, int r, int i, int idx, T a) {
    const S2Nb<T> n = s2_nb(L, r, i, idx);
    const T wl = L.w0[idx], wr = L.w0[n.ir], wu = L.w1[idx], wd = *n.wd;
    const T xl = L.x[n.il], xr = L.x[n.ir], xu = *n.xu, xd = *n.xd;
    // (one chain of multiply-adds: a float64 one takes a warp 63 cycles alone and
    // 19 cycles of the SM, so their number counts, not their dependence)
    a += wl * xl;
    a += wr * xr;
    a += wu * xu;
    return a + wd * xd;
}
template <typename T>
PF_HD T s2_diag(const S2View<T>& L, int r, int i, int idx) {
    const S2Nb<T> n = s2_nb(L, r, i, idx);
    return (L.w0[idx] + L.w0[n.ir]) + (L.w1[idx] + *n.wd);
}

// 1 / diagonal of the strip
template <typename T>
PF_HD void s2_invdiag(const S2View<T>& L, int t) {
    s2_cells(L.nx, L.rows, L.lf, t, [&](int r, int i) {
        const int q = r * L.nx + i;
        L.di[q] = s2_rcp(s2_diag(L, r, i, q));
    });
}

// Face coefficients of the strip of the next level (see k_coarsen_beta).
template <typename T>
PF_HD void s2_coarsen(const S2View<T>& F, const S2View<T>& C, int t) {
    s2_cells(C.nx, C.rows, C.lf, t, [&](int R, int I) {
        const int J = C.j0 + R, q = R * C.nx + I;
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
        // (the level's equations are those of MGLevel times h_0^2 and the cell's
        // nominal volume over level 0's, so f is a plain sum of residuals)
        C.w0[q] = C.nx == 1 ? T(0) : s0 * T(rx);
        C.w1[q] = C.ny == 1 ? T(0) : s1 * T(ry);
    });
}

// Classes of the cells of a level with an odd or one-cell axis: the sum modulo 3
// of a value per axis that alternates 0, 1 and is 2 on the last cell of an odd
// axis, so two neighbours never share a class (three phases a sweep, where
// colours with the seams' cells apart take four to six).
PF_HD int s2_class(int seams, int i, int j, int nx, int ny) {
    const int a = ((seams & 1) && i == nx - 1 ? 2 : (i & 1)) +
                  ((seams & 2) && j == ny - 1 ? 2 : (j & 1));
    return a >= 3 ? a - 3 : a;
}

// The first class of a sweep from zero, done where the right-hand side f of a
// cell is formed: x = f / diagonal on the cells of class 0; on levels with odd
// or one-cell axes zero on every other cell (on the others no cell is read
// before its class is written).
template <typename T>
PF_HD void s2_start(const S2View<T>& L, int i, int j, int idx, T f) {
    const bool c0 = ((i + j) & 1) == 0;
    if (!L.seams) {
        if (c0) L.x[idx] = f * L.di[idx];
    } else {
        L.x[idx] = s2_class(L.seams, i, j, L.nx, L.ny) == 0 ? f * L.di[idx] : T(0);
    }
}

// One class of a Gauss-Seidel sweep.
template <typename T>
PF_HD void s2_gs(const S2View<T>& L, int cls, int t) {
    const int nx = L.nx;
    if (!L.seams) {
        const int color = cls;
        s2_map<T>(nx >> 1, L.rows, L.lh, t,
                  [&](int r, int m) {
                      const int i = 2 * m + ((L.j0 + r + color) & 1), idx = r * nx + i;
                      return s2_off(L, r, i, idx, L.f[idx]) * L.di[idx];
                  },
                  [&](int r, int m, T v) { L.x[r * nx + 2 * m + ((L.j0 + r + color) & 1)] = v; });
        return;
    }
    s2_cells(nx, L.rows, L.lf, t, [&](int r, int i) {
        const int idx = r * nx + i;
        if (s2_class(L.seams, i, L.j0 + r, nx, L.ny) != cls) return;
        L.x[idx] = s2_off(L, r, i, idx, L.f[idx]) * L.di[idx];
    });
}

// f of the next level (the sum of the children's residuals) and its sweep's
// start. After a sweep the residual of an even level's second
// colour is zero; with one sweep from zero that of the first colour is the
// neighbours' part alone.
template <typename T>
PF_HD void s2_restrict(const S2View<T>& F, const S2View<T>& C, bool one_sweep, int t) {
    auto value = [&](int R, int I) {
        const int J = C.j0 + R;
        T s;
        if (!F.seams && F.cfx == 2 && F.cfy == 2) {
            const int r = 2 * J - F.j0, i = 2 * I, a = r * F.nx + i, b = a + F.nx + 1;
            s = s2_off(F, r + 1, i + 1, b, s2_off(F, r, i, a, T(0)));
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
                    s += s2_off(F, r, i, a, F.f[a]) - s2_diag(F, r, i, a) * F.x[a];
                }
        }
        return s;
    };
    s2_map<T>(C.nx, C.rows, C.lf, t, value, [&](int R, int I, T s) {
        const int q = R * C.nx + I;
        C.f[q] = s;
        s2_start(C, I, C.j0 + R, q, s);
    });
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
    if (qc == 1.f) {
        o = (i & 1) ? 1 : -1;
        w = T(0.25);
        return;
    }
    if (I0 > nc - 1) I0 = nc - 1;
    const float wp = 2.f * (I0 == nc - 1 ? qc : 1.f);
    const float d = float(i - 2 * I0) + 0.5f * (i == nf - 1 ? qf : 1.f) - 0.5f * wp;
    o = d >= 0.f ? 1 : -1;
    const int I1 = I0 + o;
    const bool l1 = (I1 < 0 ? nc - 1 : (I1 == nc ? 0 : I1)) == nc - 1;
    w = T((d < 0.f ? -d : d) / (0.5f * wp + (l1 ? qc : 1.f)));
}
template <typename T>
PF_HD const T* s2_coarse_row(const S2View<T>& C, int R) {
    return R < 0 ? C.xm : (R >= C.rows ? C.xp : C.x + R * C.nx);
}

// x += interpolation of the next level's x. On even levels only the first
// colour: the post-sweep starts by overwriting the second.
template <typename T>
PF_HD void s2_prolong(const S2View<T>& F, const S2View<T>& C, int t) {
    const int nx = F.nx;
    const bool uniform = F.cfx == 2 && F.cfy == 2 && C.qx == 1.f && C.qy == 1.f;
    auto value = [&](int r, int i) {
        const int j = F.j0 + r;
        int I0, J0, oi, oj;
        T wi, wj;
        s2_interp<T>(i, nx, C.nx, F.cfx, F.qx, C.qx, I0, oi, wi);
        s2_interp<T>(j, F.ny, C.ny, F.cfy, F.qy, C.qy, J0, oj, wj);
        int I1 = I0 + oi;
        I1 = I1 < 0 ? C.nx - 1 : (I1 >= C.nx ? 0 : I1);
        const T *c0 = s2_coarse_row(C, J0 - C.j0), *c1 = s2_coarse_row(C, J0 - C.j0 + oj);
        if (uniform) {
            T v = F.x[r * nx + i] + T(0.5625) * c0[I0];
            v += T(0.1875) * (c0[I1] + c1[I0]);
            return v + T(0.0625) * c1[I1];
        }
        const T a = c0[I0] + wi * (c0[I1] - c0[I0]);
        const T b = c1[I0] + wi * (c1[I1] - c1[I0]);
        return F.x[r * nx + i] + (a + wj * (b - a));
    };
    auto col = [&](int r, int m) { return 2 * m + ((F.j0 + r) & 1); };
    if (!F.seams)
        s2_map<T>(nx >> 1, F.rows, F.lh, t, [&](int r, int m) { return value(r, col(r, m)); },
                  [&](int r, int m, T v) { F.x[r * nx + col(r, m)] = v; });
    else
        s2_map<T>(nx, F.rows, F.lf, t, value, [&](int r, int i, T v) { F.x[r * nx + i] = v; });
}

// The interpolation and the second colour of an even level's first post-sweep
// in one phase: the first colour's interpolated values are formed by the cells
// that read them (they are overwritten by the next class).
template <typename T>
PF_HD void s2_prolong_gs(const S2View<T>& F, const S2View<T>& C, int t) {
    const int nx = F.nx;
    s2_map<T>(nx >> 1, F.rows, F.lh, t, [&](int r, int m) {
        const int j = F.j0 + r, par = (j + 1) & 1, i = 2 * m + par, idx = r * nx + i;
        // parents' rows of fine row j (c0, its other neighbour c1); rows j - 1 and
        // j + 1 share the parent of j or have it as their other neighbour
        const int R = (j >> 1) - C.j0, I = m;
        const int oj = (j & 1) ? 1 : -1;
        const T *c0 = s2_coarse_row(C, R), *c1 = s2_coarse_row(C, R + oj);
        const int Im = I == 0 ? C.nx - 1 : I - 1, Ip = I == C.nx - 1 ? 0 : I + 1;
        // column interpolations of rows c0 and c1 at fine columns i - 1, i, i + 1
        T a0[3], a1[3];
        const T qt = T(0.25);
        if (par) {   // i odd: i - 1 and i in parent I, i + 1 in parent Ip
            const T x0 = c0[Im], x1 = c0[I], x2 = c0[Ip], y0 = c1[Im], y1 = c1[I], y2 = c1[Ip];
            a0[0] = x1 + qt * (x0 - x1);
            a0[1] = x1 + qt * (x2 - x1);
            a0[2] = x2 + qt * (x1 - x2);
            a1[0] = y1 + qt * (y0 - y1);
            a1[1] = y1 + qt * (y2 - y1);
            a1[2] = y2 + qt * (y1 - y2);
        } else {     // i even: i - 1 in parent Im, i and i + 1 in parent I
            const T x0 = c0[Im], x1 = c0[I], x2 = c0[Ip], y0 = c1[Im], y1 = c1[I], y2 = c1[Ip];
            a0[0] = x0 + qt * (x1 - x0);
            a0[1] = x1 + qt * (x0 - x1);
            a0[2] = x1 + qt * (x2 - x1);
            a1[0] = y0 + qt * (y1 - y0);
            a1[1] = y1 + qt * (y0 - y1);
            a1[2] = y1 + qt * (y2 - y1);
        }
        const T pl = a0[0] + qt * (a1[0] - a0[0]), pr = a0[2] + qt * (a1[2] - a0[2]);
        // the sibling row (same parent) leans on the other side's coarse row; the
        // row across the parent's edge has parent c1 and leans on c0
        const T *c2 = s2_coarse_row(C, R - oj);
        const int In = par ? Ip : Im;
        const T b2 = c2[I] + qt * (c2[In] - c2[I]);
        const T sib = a0[1] + qt * (b2 - a0[1]);
        const T far = a1[1] + qt * (a0[1] - a1[1]);
        const T pu = oj < 0 ? far : sib, pd = oj < 0 ? sib : far;
        const S2Nb<T> n = s2_nb(F, r, i, idx);
        const T wl = F.w0[idx], wr = F.w0[n.ir], wu = F.w1[idx], wd = *n.wd;
        const T xl = F.x[n.il], xr = F.x[n.ir], xu = *n.xu, xd = *n.xd;
        return (F.f[idx] + ((wl * (xl + pl) + wr * (xr + pr)) +
                            (wu * (xu + pu) + wd * (xd + pd)))) * F.di[idx];
    }, [&](int r, int m, T v) { F.x[r * nx + 2 * m + ((F.j0 + r + 1) & 1)] = v; });
}

// ---- dense level ----
// M = pseudo-inverse of the level's A: the inverse of A + (sigma / n) 1 1^T
// (symmetric positive definite) by Gauss-Jordan elimination without pivoting
// (build, fill, n steps of elimination), with the means of its rows
// and columns, weighted by A's diagonal, removed (means, then project). x is
// defined up to a constant; this choice keeps it small where the coefficients
// are large. A plain zero mean puts the light phase at the offset that the
// heavy drop's large x asks for, and the rounding of A x there costs float32
// solves at density ratio 1000 their convergence. A barrier follows each of
// these functions.
template <typename T>
PF_HD void s2_dense_build(const S2View<T>& L, T* M, int t) {
    const int n = L.nx * L.ny, ld = s2_pad(n);
    T sig = T(0);
    for (int k = 0; k < L.nx; ++k) sig += s2_diag(L, 0, k, k);
    sig /= T(L.nx * n);
    for (int q = t; q < n * ld; q += kS2Threads) M[q] = q % ld < n ? sig : T(0);
}
template <typename T>
PF_HD void s2_dense_fill(const S2View<T>& L, T* M, int t) {
    const int n = L.nx * L.ny, ld = s2_pad(n);
    for (int a = t; a < n; a += kS2Threads) {
        const int j = a / L.nx, i = a - j * L.nx;
        T* row = M + a * ld;
        const int il = j * L.nx + (i == 0 ? L.nx - 1 : i - 1), ir = j * L.nx + (i + 1 == L.nx ? 0 : i + 1);
        const int iu = (j == 0 ? L.ny - 1 : j - 1) * L.nx + i, id = (j + 1 == L.ny ? 0 : j + 1) * L.nx + i;
        const T w[4] = {L.w0[a], L.w0[ir], L.w1[a], L.w1[id]};
        const int c[4] = {il, ir, iu, id};
        for (int k = 0; k < 4; ++k) {
            row[a] += w[k];
            row[c[k]] -= w[k];
        }
    }
}
// Elimination: a thread keeps its two elements (column t % 32, rows t / 32 and
// t / 32 + 16) in registers; publish copies column k, row k and the pivot's
// reciprocal of the current matrix into one of two buffers, step reads them.
// One barrier a step. (64 cells took 45 us a solve, more than the level that
// 16 to 27 cells add costs in ten V-cycles.)
constexpr int kS2Col = kS2DenseMax, kS2ColRow = 2 * kS2DenseMax + 1;   // the row's offset; size
template <typename T>
PF_HD void s2_gj_publish(const T (&m)[2], int n, int k, T* buf, int t) {
    const int c = t & 31, r0 = t >> 5;
    if (c >= n || k >= n) return;
    if (c == k) {
        if (r0 < n) buf[r0] = m[0];
        if (r0 + 16 < n) buf[r0 + 16] = m[1];
    }
    if (r0 == (k & 15)) {
        const T v = k < 16 ? m[0] : m[1];
        buf[kS2Col + c] = v;
        if (c == k) buf[2 * kS2Col] = s2_rcp(v);
    }
}
template <typename T>
PF_HD void s2_gj_step(T (&m)[2], int n, int k, const T* buf, int t) {
    const int c = t & 31, r0 = t >> 5;
    if (c >= n) return;
    const T rk = (c == k ? T(1) : buf[kS2Col + c]) * buf[2 * kS2Col];
    if (r0 < n) m[0] = r0 == k ? rk : (c == k ? T(0) : m[0]) - buf[r0] * rk;
    if (r0 + 16 < n) m[1] = r0 + 16 == k ? rk : (c == k ? T(0) : m[1]) - buf[r0 + 16] * rk;
}
template <typename T>
PF_HD void s2_gj_move(T (&m)[2], T* M, int n, bool store, int t) {
    const int c = t & 31, ld = s2_pad(n);
    for (int i = 0; i < 2; ++i) {
        const int r = (t >> 5) + 16 * i;
        if (c < n && r < n) {
            if (store) M[r * ld + c] = m[i];
            else m[i] = M[r * ld + c];
        }
    }
}
// the weights, in the second buffer
template <typename T>
PF_HD void s2_dense_weights(const S2View<T>& L, T* d, int t) {
    if (t < L.nx * L.ny) {
        const int r = t / L.nx, i = t - r * L.nx;
        d[t] = s2_diag(L, r, i, t);
    }
}
// (k = 1: row and column means; 2: their mean)
template <typename T>
PF_HD void s2_dense_means(const T* M, int n, int k, T* colrow, int t) {
    const int ld = s2_pad(n);
    const T* d = colrow + kS2ColRow;
    T s = T(0), w = T(0);
    if (k == 1 && (t < n || (t >= kS2Col && t < kS2Col + n))) {
        for (int c = 0; c < n; ++c) {
            s += d[c] * (t < kS2Col ? M[t * ld + c] : M[c * ld + t - kS2Col]);
            w += d[c];
        }
        colrow[t] = s / w;
    } else if (k == 2 && t == 2 * kS2Col) {
        for (int c = 0; c < n; ++c) {
            s += d[c] * colrow[c];
            w += d[c];
        }
        colrow[t] = s / w;
    }
}
template <typename T>
PF_HD void s2_dense_project(T* M, int n, const T* colrow, int t) {
    const int ld = s2_pad(n), c = t & 31;
    if (c < n)
        for (int r = t >> 5; r < n; r += kS2Threads >> 5)
            M[r * ld + c] -= (colrow[r] + colrow[kS2Col + c]) - colrow[2 * kS2Col];
}
// x = M f of the part of thread t: row t / 8, every eighth column from t % 8
template <typename T>
PF_HD T s2_dense_part(const T* M, const T* f, int n, int t) {
    const int r = t >> 3;
    T s = T(0);
    if (r < n) {
        const T* row = M + r * s2_pad(n);
        for (int c = t & 7; c < n; c += 8) s += row[c] * f[c];
    }
    return s;
}

// Sums of products as accurate as float64 ones: float64 sums of the float64
// path; on the mixed one three floats (float64 multiply-adds would run on
// GB300's two-lane float64 pipe). A product is split into its value and its
// exact rounding error, the sums' rounding errors go into the second word and
// that one's into the third. Mean error over sum |a b| of 32 random products:
// 8e-18, float64 2e-17; with two words 1.8e-15, for 3 % less time of a 256^2
// mixed step. The operations are spelled out, since a contracted multiply-add
// would count an error twice.
PF_HD float s2_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
PF_HD float s2_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
PF_HD float s2_two_sum(float a, float b, float& lo) {
    const float s = s2_add(a, b), bb = s2_add(s, -a);
    lo = s2_add(s2_add(a, -s2_add(s, -bb)), s2_add(b, -bb));
    return s;
}
struct S2AccF {
    float s, c, d;
    PF_HD void add_prod(float a, float b) {
        const float p = s2_mul(a, b), e = fmaf(a, b, -p);
        float t, v;
        s = s2_two_sum(s, p, t);
        const float w = s2_add(t, e);
        c = s2_two_sum(c, w, v);
        d = s2_add(d, s2_add(v, s2_add(s2_add(t, -w), e)));
    }
    // (commutative bit for bit: every CTA forms the same totals)
    PF_HD void merge(const S2AccF& o) {
        float t, u, v;
        s = s2_two_sum(s, o.s, t);
        c = s2_two_sum(c, o.c, u);
        c = s2_two_sum(c, t, v);
        d = s2_add(s2_add(d, o.d), s2_add(u, v));
    }
    PF_HD double value() const { return double(s) + (double(c) + double(d)); }
};
struct S2AccD {
    double s;
    PF_HD void add_prod(double a, double b) { s += a * b; }
    PF_HD void merge(const S2AccD& o) { s += o.s; }
    PF_HD double value() const { return s; }
};
template <typename T> struct S2AccOf { using type = S2AccD; };
template <> struct S2AccOf<float> { using type = S2AccF; };

// Range of the mixed path. Its system is scaled by h^2 (times 2^m: h^2 2^m lies in
// [1/2, 1)) and its norms are sums of float squares, so residuals are taken times
// 2^-k, which brings their norm near 1, and the right-hand side's norm times
// 2^-kf. Powers of two: the same bits but for what would leave float's range. k is
// 0 in a solve's first residual, whose norm is not known, and comes from the
// inner solve's last norm after each refinement; a norm outside [2^-16, 2^48], or
// one that has over- or underflowed, costs further passes with the k that it asks
// for. Right-hand sides of 1e-25 to 1e30 take the iterations of 1; without this
// a 64^2 solve stalled below 1e-9 and a start far off left float's range.
PF_HD double s2_pow2(int e) {   // 2^e, |e| <= 1000
    const long long b = (long long)(1023 + e) << 52;
    double d;
    memcpy(&d, &b, sizeof(d));
    return d;
}
PF_HD int s2_half_log2(double a) {   // exponent of the square root, a positive and normal
    long long b;
    memcpy(&b, &a, sizeof(b));
    return (int)((b >> 52) - 1023) >> 1;
}
struct S2Scale {
    int k, kf, m;
    float scale, fscale;   // 2^-k, 2^-kf
    float unscale;         // 2^(k - m): takes the inner solve's e back to x
};
PF_HD void s2_scale_set(S2Scale& s, int k, int kf) {
    // (2^-k and 2^(k - m) stay normal floats)
    k = k < s.m - 120 ? s.m - 120 : (k > s.m + 120 ? s.m + 120 : k);
    s.k = k < -120 ? -120 : (k > 120 ? 120 : k);
    s.kf = kf;
    s.scale = float(s2_pow2(-s.k));
    s.fscale = float(s2_pow2(-s.kf));
    s.unscale = float(s2_pow2(s.k - s.m));
}
PF_HD void s2_scale_init(S2Scale& s, int m) {
    s.m = m;
    s2_scale_set(s, 0, 0);
}
PF_HD void s2_scale_next(S2Scale& s, double rr_in) {
    if (rr_in > 1e-300 && rr_in < 1e300) s2_scale_set(s, s.k + s2_half_log2(rr_in), s.kf);
}
// After a residual pass: its squared norms ffs (first: of the right-hand side)
// and rr as summed become ff and rr unscaled; true where the pass is to be done
// again with the scales set here.
PF_HD bool s2_scale_check(S2Scale& s, bool first, int pass, double rtol2, double ffs, double& ff,
                          double& rr) {
    constexpr int far = 64;            // one step towards a norm out of range
    constexpr double tiny = 8e-31;     // smaller sums may have lost squares
    const double rrs = rr;
    int k = s.k, kf = s.kf;
    if (first) {
        ff = ffs * s2_pow2(2 * kf);
        if (kf == 0) kf = !(ffs < 1e300) ? far : (ffs < tiny ? -far : 0);
    }
    rr = rrs * s2_pow2(2 * k);
    const double lost = tiny * s2_pow2(2 * k);   // what rr may have lost, amply
    if (!(rrs < 1e300)) {
        if (pass == 0) k += far;
    } else if (!(rr + lost <= rtol2 * ff)) {   // (else converged)
        if (rrs < tiny) {
            if (pass == 0) k -= far;
        } else {
            const int e = s2_half_log2(rrs);
            if (e < -16 || e > 48) k += e;
        }
    }
    if (pass == 2 || (k == s.k && kf == s.kf)) return false;
    s2_scale_set(s, k, kf);
    return true;
}

// s = A z (z: the level's x) and the products z.r, z.s and, unless first, z.q.
template <typename T, typename A>
PF_HD void s2_apply_dots(const S2View<T>& L, const T* qv, T* sv, bool first, A& rz, A& zq, A& zs,
                         int t) {
    const int nx = L.nx;
    s2_map<T>(nx, L.rows, L.lf, t, [&](int r, int i) {
        const int q = r * nx + i;
        const S2Nb<T> n = s2_nb(L, r, i, q);
        const T z = L.x[q], w0 = L.w0[q], wr = L.w0[n.ir], w1 = L.w1[q], w3 = *n.wd;
        const T xl = L.x[n.il], xr = L.x[n.ir], xu = *n.xu, xd = *n.xd;
        T ax = w0 * (z - xl);
        ax += wr * (z - xr);
        ax += w1 * (z - xu);
        ax += w3 * (z - xd);
        rz.add_prod(z, L.f[q]);
        zs.add_prod(z, ax);
        if (!first) zq.add_prod(z, qv[q]);
        return ax;
    }, [&](int r, int i, T v) { sv[r * nx + i] = v; });
}

// p = z + beta p, q = s + beta q, e += alpha p, r -= alpha q (r: the level's
// f), the next sweep's start; per-thread sum of r^2.
template <typename T>
PF_HD T s2_update(const S2View<T>& L, const T* sv, T* p, T* qv, T* e, T alpha, T beta, bool first,
                  int t) {
    const int nx = L.nx;
    T rr = T(0);
    s2_cells(nx, L.rows, L.lf, t, [&](int r, int i) {
        const int k = r * nx + i;
        const T z = L.x[k], s = sv[k], f = L.f[k];
        T pn = z, qn = s, en = T(0);
        if (!first) {
            pn += beta * p[k];
            qn += beta * qv[k];
            en = e[k];
        }
        const T rv = f - alpha * qn;
        p[k] = pn;
        qv[k] = qn;
        e[k] = en + alpha * pn;
        L.f[k] = rv;
        s2_start(L, i, L.j0 + r, k, rv);
        rr += rv * rv;
    });
    return rr;
}

}  // namespace pf
