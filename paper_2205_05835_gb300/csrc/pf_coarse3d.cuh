// The phases of the 3D coarse V-cycle of one thread-block cluster
// (pf_coarse3d.cu): work of one CTA between two barriers, written over
// (thread, threads) loops and plain pointers, so the same functions run on the
// host. A CTA owns a slab of whole planes of every cluster level (levels
// l0 .. lc - 1); planes beyond it are read from the neighbouring CTAs' memory.
// Levels lc .. ld live in CTA 0; level ld is solved by its inverse. The 2D
// counterpart, with more on the choices, is pf_solve2d.cuh.
#pragma once

#include "pf_solve2d.cuh"

namespace pf {

constexpr int kC3MaxCTAs = 8;     // portable cluster size
constexpr int kC3MaxCluster = 5;  // cluster levels and the view of level lc

struct C3Lev {
    int nx, ny, nz;
    int cf[3];
    float q[3];
    int ox, of, ow[3], od;   // element offsets in every CTA's dynamic shared memory
};

struct C3Plan {
    int C, l0, lc, ld;
    int pre, post;
    int om, elems;
    float kappa[kMaxLevels];   // scale of level l's equations (see c3_plan)
    C3Lev lev[kMaxLevels];
};

PF_HD int c3_plane(const C3Plan& P, int l, int c) {
    if (c >= P.C) return P.lev[l].nz;
    return ((P.lev[P.lc].nz * c) / P.C) << (P.lc - l);
}
inline int c3_max_planes(const C3Plan& P, int l) {
    if (l >= P.lc) return P.lev[l].nz;
    int m = 0;
    for (int c = 0; c < P.C; ++c) {
        const int r = c3_plane(P, l, c + 1) - c3_plane(P, l, c);
        if (r > m) m = r;
    }
    return m;
}

// Fits the levels l0 .. of a 3D hierarchy into a cluster's shared memory; false
// when they do not fit. The arrays' offsets depend on the geometry only.
template <typename T>
inline bool c3_plan(const MGHier<T>& H, int l0, size_t smem_bytes, int dense_cells, C3Plan& P) {
    if (l0 < 1 || l0 >= H.nlev || H.lev[0].g.nz < 2) return false;
    P.l0 = l0;
    P.pre = H.pre;
    P.post = H.post;
    float kap = 1.f;
    for (int l = 0; l < H.nlev; ++l) {
        C3Lev& L = P.lev[l];
        L.nx = H.lev[l].g.nx;
        L.ny = H.lev[l].g.ny;
        L.nz = H.lev[l].g.nz;
        int vol = 1;
        for (int d = 0; d < 3; ++d) {
            L.cf[d] = H.lev[l].cf[d];
            L.q[d] = H.lev[l].lastw[d];
            vol *= L.cf[d];
        }
        // level l's equations times kappa h_l^2: the next level's right-hand
        // side is then the plain sum of the children's residuals
        P.kappa[l] = kap;
        if (l >= l0) kap *= 0.25f * float(vol);
    }
    auto cells = [&](int l) { return P.lev[l].nx * P.lev[l].ny * P.lev[l].nz; };
    if (cells(H.nlev - 1) > dense_cells) return false;
    P.ld = l0;
    while (cells(P.ld) > dense_cells) ++P.ld;
    const long long cap = (long long)(smem_bytes / sizeof(T));
    // cycles of a V-cycle: per cell of the largest slab and of CTA 0's levels,
    // per phase of a cluster and of a CTA
    const float cell = sizeof(T) == 4 ? 7.f : 30.f;
    float best = -1.f;
    C3Plan Q = P;
    for (int lc = l0; lc <= P.ld && lc - l0 < kC3MaxCluster; ++lc)
        for (int C = 1; C <= kC3MaxCTAs && C <= P.lev[lc].nz; C *= 2) {
            if (lc == l0 && C > 1) break;
            Q.lc = lc;
            Q.C = C;
            long long off = (long long)cells(P.ld) * s2_pad(cells(P.ld));
            float c = 0.f;
            for (int l = l0; l <= P.ld; ++l) {
                const long long n = (long long)c3_max_planes(Q, l) * P.lev[l].nx * P.lev[l].ny;
                off += 6 * ((n + 3) & ~3LL);
                if (l < P.ld) c += cell * float(n) + 5.f * (l < lc && C > 1 ? 900.f : 400.f);
            }
            if (off > cap) continue;
            if (best < 0.f || c < best) {
                best = c;
                P.lc = lc;
                P.C = C;
            }
        }
    if (best < 0.f) return false;
    long long off = 0;
    auto take = [&](long long n) {
        const int o = (int)off;
        off += (n + 3) & ~3LL;
        return o;
    };
    P.om = take((long long)cells(P.ld) * s2_pad(cells(P.ld)));
    for (int l = P.ld; l >= l0; --l) {
        C3Lev& L = P.lev[l];
        const long long n = (long long)c3_max_planes(P, l) * L.nx * L.ny;
        L.ox = take(n);
        L.of = take(n);
        for (int d = 0; d < 3; ++d) L.ow[d] = take(n);
        L.od = take(n);
    }
    P.elems = (int)off;
    return true;
}

// One level as a CTA sees it: its planes [k0, k0 + np) (pointers at plane k0)
// and the planes around them.
template <typename T>
struct C3View {
    int nx, ny, nz, k0, np, sxy;
    int cf[3];
    int seams;          // odd axes: bits 0 - 2; bit 3: an axis of one cell
    int lf, lh;         // log2 of the threads along a row: cells, pairs of cells
    float q[3];
    float inv_ny;
    T *x, *f, *w[3], *di;
    T *xm, *xp, *w2p;
};
template <typename T>
PF_HD void c3_view_sizes(C3View<T>& v, const C3Lev& L, int k0, int np) {
    v.nx = L.nx;
    v.ny = L.ny;
    v.nz = L.nz;
    v.k0 = k0;
    v.np = np;
    v.sxy = L.nx * L.ny;
    for (int d = 0; d < 3; ++d) {
        v.cf[d] = L.cf[d];
        v.q[d] = L.q[d];
    }
    v.seams = (L.nx > 1 ? (L.nx & 1) : 8) | (L.ny > 1 ? 2 * (L.ny & 1) : 8) |
              (L.nz > 1 ? 4 * (L.nz & 1) : 8);
    v.lf = s2_log2(L.nx);
    v.lh = s2_log2((L.nx + 1) >> 1);
    v.inv_ny = 1.0f / float(L.ny);
}
template <typename T>
PF_HD int c3_classes(const C3View<T>& L) { return L.seams ? 3 : 2; }
// class of a cell of a level with an odd or one-cell axis (see s2_class)
PF_HD int c3_class(int s, int i, int j, int k, int nx, int ny, int nz) {
    const int a = ((s & 1) && i == nx - 1 ? 2 : (i & 1)) + ((s & 2) && j == ny - 1 ? 2 : (j & 1)) +
                  ((s & 4) && k == nz - 1 ? 2 : (k & 1));
    return a >= 6 ? 0 : (a >= 3 ? a - 3 : a);
}

// Loops over the rows (r: plane, j) of a slab and n items of a row. The plane
// of a row comes from a float reciprocal: (q + 1/2) / ny lies at least
// 1/(2 ny) from an integer, more than the roundings for q < 2^22.
template <typename F>
PF_HD void c3_cells(int n, int ny, int np, float inv_ny, int lw, int t, F f) {
    const int i0 = t & ((1 << lw) - 1), rows = ny * np;
    for (int q = t >> lw; q < rows; q += kS2Threads >> lw) {
        const int r = int((float(q) + 0.5f) * inv_ny), j = q - r * ny;
        for (int i = i0; i < n; i += 1 << lw) f(r, j, i);
    }
}

template <typename T>
struct C3Nb {
    int il, ir, jl, jr;
    const T *zu, *zd, *wz;
};
template <typename T>
PF_HD C3Nb<T> c3_nb(const C3View<T>& L, int r, int j, int i, int idx) {
    const int nx = L.nx, in = idx - r * L.sxy;
    C3Nb<T> n;
    n.il = i == 0 ? idx + nx - 1 : idx - 1;
    n.ir = i == nx - 1 ? idx - i : idx + 1;
    n.jl = j == 0 ? idx + L.sxy - nx : idx - nx;
    n.jr = j == L.ny - 1 ? idx - j * nx : idx + nx;
    const bool last = r == L.np - 1;
    n.zu = r == 0 ? L.xm + in : L.x + (idx - L.sxy);
    n.zd = last ? L.xp + in : L.x + (idx + L.sxy);
    n.wz = last ? L.w2p + in : L.w[2] + (idx + L.sxy);
    return n;
}
// a plus the six coefficients times the neighbours; the sum of the coefficients
template <typename T>
PF_HD T c3_off(const C3View<T>& L, int r, int j, int i, int idx, T a) {
    const C3Nb<T> n = c3_nb(L, r, j, i, idx);
    const T w0 = L.w[0][idx], w1 = L.w[0][n.ir], w2 = L.w[1][idx], w3 = L.w[1][n.jr],
            w4 = L.w[2][idx], w5 = *n.wz;
    const T x0 = L.x[n.il], x1 = L.x[n.ir], x2 = L.x[n.jl], x3 = L.x[n.jr], x4 = *n.zu, x5 = *n.zd;
    a += w0 * x0;
    a += w1 * x1;
    a += w2 * x2;
    a += w3 * x3;
    a += w4 * x4;
    return a + w5 * x5;
}
template <typename T>
PF_HD T c3_diag(const C3View<T>& L, int r, int j, int i, int idx) {
    const C3Nb<T> n = c3_nb(L, r, j, i, idx);
    return ((L.w[0][idx] + L.w[0][n.ir]) + (L.w[1][idx] + L.w[1][n.jr])) + (L.w[2][idx] + *n.wz);
}

// first class of a sweep from zero, with the right-hand side (see s2_start)
template <typename T>
PF_HD void c3_start(const C3View<T>& L, int r, int j, int i, int idx, T f) {
    const int k = L.k0 + r;
    const bool c0 = ((i + j + k) & 1) == 0;
    if (!L.seams) {
        if (c0) L.x[idx] = f * L.di[idx];
    } else {
        L.x[idx] = c3_class(L.seams, i, j, k, L.nx, L.ny, L.nz) == 0 ? f * L.di[idx] : T(0);
    }
}

template <typename T>
PF_HD void c3_gs(const C3View<T>& L, int cls, int t) {
    const int nx = L.nx;
    if (L.seams) {
        c3_cells(nx, L.ny, L.np, L.inv_ny, L.lf, t, [&](int r, int j, int i) {
            const int idx = (r * L.ny + j) * nx + i;
            if (c3_class(L.seams, i, j, L.k0 + r, nx, L.ny, L.nz) == cls)
                L.x[idx] = c3_off(L, r, j, i, idx, L.f[idx]) * L.di[idx];
        });
        return;
    }
    c3_cells(nx >> 1, L.ny, L.np, L.inv_ny, L.lh, t, [&](int r, int j, int m) {
        const int i = 2 * m + ((j + L.k0 + r + cls) & 1);
        const int idx = (r * L.ny + j) * nx + i;
        L.x[idx] = c3_off(L, r, j, i, idx, L.f[idx]) * L.di[idx];
    });
}

template <typename T>
PF_HD void c3_restrict(const C3View<T>& F, const C3View<T>& C, bool one_sweep, int t) {
    const bool even = !F.seams && F.cf[0] == 2 && F.cf[1] == 2 && F.cf[2] == 2;
    c3_cells(C.nx, C.ny, C.np, C.inv_ny, C.lf, t, [&](int R, int J, int I) {
        const int K = C.k0 + R;
        T s = T(0);
        if (even) {
            // the children of the first colour: the second's residual is zero
            const int r = 2 * K - F.k0, j = 2 * J, i = 2 * I;
            for (int q = 0; q < 4; ++q) {
                const int dz = q >> 1, dy = q & 1, dx = (dz + dy) & 1;
                const int idx = ((r + dz) * F.ny + j + dy) * F.nx + i + dx;
                s = c3_off(F, r + dz, j + dy, i + dx, idx, s);
                if (!one_sweep)
                    s += F.f[idx] - c3_diag(F, r + dz, j + dy, i + dx, idx) * F.x[idx];
            }
        } else {
            const int ex = F.cf[0] == 1 ? 1 : (I == C.nx - 1 ? F.nx - 2 * I : 2);
            const int ey = F.cf[1] == 1 ? 1 : (J == C.ny - 1 ? F.ny - 2 * J : 2);
            const int ez = F.cf[2] == 1 ? 1 : (K == C.nz - 1 ? F.nz - 2 * K : 2);
            for (int c = 0; c < ez; ++c)
                for (int b = 0; b < ey; ++b)
                    for (int e = 0; e < ex; ++e) {
                        const int i = F.cf[0] * I + e, j = F.cf[1] * J + b,
                                  r = F.cf[2] * K + c - F.k0;
                        const int idx = (r * F.ny + j) * F.nx + i;
                        s += c3_off(F, r, j, i, idx, F.f[idx]) -
                             c3_diag(F, r, j, i, idx) * F.x[idx];
                    }
        }
        const int idx = (R * C.ny + J) * C.nx + I;
        C.f[idx] = s;
        c3_start(C, R, J, I, idx, s);
    });
}

template <typename T>
PF_HD void c3_prolong(const C3View<T>& F, const C3View<T>& C, int t) {
    const int nx = F.nx;
    const bool uniform = F.cf[0] == 2 && F.cf[1] == 2 && F.cf[2] == 2 && C.q[0] == 1.f &&
                         C.q[1] == 1.f && C.q[2] == 1.f;
    auto plane = [&](int R) -> const T* {
        return R < 0 ? C.xm : (R >= C.np ? C.xp : C.x + R * C.sxy);
    };
    auto cell = [&](int r, int j, int i) {
        const int k = F.k0 + r;
        int I0, J0, K0, oi, oj, ok;
        T wi, wj, wk;
        s2_interp<T>(i, nx, C.nx, F.cf[0], F.q[0], C.q[0], I0, oi, wi);
        s2_interp<T>(j, F.ny, C.ny, F.cf[1], F.q[1], C.q[1], J0, oj, wj);
        s2_interp<T>(k, F.nz, C.nz, F.cf[2], F.q[2], C.q[2], K0, ok, wk);
        int I1 = I0 + oi, J1 = J0 + oj;
        I1 = I1 < 0 ? C.nx - 1 : (I1 >= C.nx ? 0 : I1);
        J1 = J1 < 0 ? C.ny - 1 : (J1 >= C.ny ? 0 : J1);
        const T *p0 = plane(K0 - C.k0), *p1 = plane(K0 - C.k0 + ok);
        const int a00 = J0 * C.nx + I0, a10 = J0 * C.nx + I1, a01 = J1 * C.nx + I0,
                  a11 = J1 * C.nx + I1;
        T& x = F.x[(r * F.ny + j) * nx + i];
        if (uniform) {
            T v = x + T(0.421875) * p0[a00];
            v += T(0.140625) * ((p0[a10] + p0[a01]) + p1[a00]);
            v += T(0.046875) * ((p0[a11] + p1[a10]) + p1[a01]);
            x = v + T(0.015625) * p1[a11];
            return;
        }
        const T c0 = p0[a00] + wi * (p0[a10] - p0[a00]), c1 = p0[a01] + wi * (p0[a11] - p0[a01]);
        const T d0 = p1[a00] + wi * (p1[a10] - p1[a00]), d1 = p1[a01] + wi * (p1[a11] - p1[a01]);
        const T c = c0 + wj * (c1 - c0), d = d0 + wj * (d1 - d0);
        x += c + wk * (d - c);
    };
    if (!F.seams)   // the post-sweep starts by overwriting the second colour
        c3_cells(nx >> 1, F.ny, F.np, F.inv_ny, F.lh, t, [&](int r, int j, int m) {
            cell(r, j, 2 * m + ((j + F.k0 + r) & 1));
        });
    else
        c3_cells(nx, F.ny, F.np, F.inv_ny, F.lf, t, cell);
}

// ---- dense level: the matrix before the elimination (see s2_dense_build) ----
template <typename T>
PF_HD void c3_dense_build(const C3View<T>& L, T* M, int t) {
    const int n = L.sxy * L.nz, ld = s2_pad(n);
    T sig = T(0);
    for (int k = 0; k < L.nx; ++k) sig += c3_diag(L, 0, 0, k, k);
    sig /= T(L.nx * n);
    for (int q = t; q < n * ld; q += kS2Threads) M[q] = q % ld < n ? sig : T(0);
}
template <typename T>
PF_HD void c3_dense_fill(const C3View<T>& L, T* M, int t) {
    const int n = L.sxy * L.nz, ld = s2_pad(n);
    for (int a = t; a < n; a += kS2Threads) {
        const int k = a / L.sxy, j = (a - k * L.sxy) / L.nx, i = a - (k * L.ny + j) * L.nx;
        const int kz = (k + 1 == L.nz ? 0 : k + 1), km = (k == 0 ? L.nz - 1 : k - 1);
        const C3Nb<T> nb = c3_nb(L, k, j, i, a);
        const int d = a + (kz - k) * L.sxy, u = a + (km - k) * L.sxy;
        const T w[6] = {L.w[0][a], L.w[0][nb.ir], L.w[1][a], L.w[1][nb.jr], L.w[2][a], L.w[2][d]};
        const int c[6] = {nb.il, nb.ir, nb.jl, nb.jr, u, d};
        T* row = M + a * ld;
        for (int q = 0; q < 6; ++q) {
            row[a] += w[q];
            row[c[q]] -= w[q];
        }
    }
}
template <typename T>
PF_HD void c3_dense_weights(const C3View<T>& L, T* d, int t) {
    const int n = L.sxy * L.nz;
    if (t < n) {
        const int k = t / L.sxy, j = (t - k * L.sxy) / L.nx, i = t - (k * L.ny + j) * L.nx;
        d[t] = c3_diag(L, k, j, i, t);
    }
}

}  // namespace pf
