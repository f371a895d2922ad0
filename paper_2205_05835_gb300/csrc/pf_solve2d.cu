// One-launch 2D pressure solve: the whole iterative refinement, with its
// multigrid-preconditioned CG inside, in one thread-block cluster.
//
// A 2D solve is a chain of small dependent steps: a 256^2 iteration moves about
// 3 MB through L2 but takes 22 launches of 2.5 us and a single-CTA coarse
// V-cycle of 45 us (95 us an iteration), and a 64^2 float64 one runs 159 us in
// that CTA. Here a step is a barrier of a cluster of up to 16 CTAs (or of one
// CTA on the coarse levels) instead of a launch, every level's arrays stay in
// shared memory for the whole solve (the finest level's overflow in L2), a
// strip's neighbour rows are read through distributed shared memory, and no
// scalar leaves the cluster: every CTA forms the same totals from the same
// partial sums in the same order.
#include <mutex>

#include "pf_device.cuh"
#include "pf_solve2d.cuh"

namespace pf {

namespace {

constexpr int kS2Threads = 512;
constexpr int kS2Warps = kS2Threads / 32;
constexpr size_t kS2Smem = 220 * 1024;   // dynamic shared memory of a CTA
constexpr int kTinyCells = 64;           // levels of one warp (of CTA 0)

template <typename T>
struct S2Args {
    S2Plan P;
    Dims g;
    Phys ph;
    SolveIO<T, 2> io;
    T* b0;          // face coefficients to leave in the workspace (may be null)
    T* b1;
    T *gx[2], *gf[2], *gw0[2], *gw1[2];   // workspace places of levels 0 and 1
    T *gdi, *gp, *gq, *ge;
    CGScalars* sc;
};

__device__ __forceinline__ int cluster_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address in CTA `rank` of the cluster of a shared-memory address of this CTA
template <typename T>
__device__ __forceinline__ T* cluster_map(T* p, int rank) {
    T* q;
    asm("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(p), "r"(rank));
    return q;
}
__device__ __forceinline__ void cluster_sync(int C) {
    if (C == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;\n"
                     "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// ---- totals over the cluster ----
__device__ __forceinline__ S2AccF shfl_acc(S2AccF a, int o) {
    return S2AccF{__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.c, o)};
}
__device__ __forceinline__ S2AccD shfl_acc(S2AccD a, int o) {
    return S2AccD{__shfl_xor_sync(0xffffffffu, a.s, o)};
}
__device__ __forceinline__ void merge(S2AccF& a, S2AccF b) {
    // commutative bit for bit: the exact sum's rounding error, then the carries
    const f2 t = two_sum(a.s, b.s);
    a.s = t.hi;
    a.c = __fadd_rn(t.lo, __fadd_rn(a.c, b.c));
}
__device__ __forceinline__ void merge(S2AccD& a, S2AccD b) { a.s += b.s; }

template <typename A>
struct S2Red {
    A warp[2][kS2Warps];
    A part[2][2][kS2MaxCTAs];   // [buffer][value][CTA], written by every CTA of the cluster
};

// K totals over the cluster, valid in warp 0 of every CTA. Contains a cluster
// barrier, which also orders the phases before and after it. The partial sums
// are pushed into every CTA's memory before that barrier, so nothing remote is
// read after it.
template <int K, typename A>
__device__ __forceinline__ void cluster_totals(A (&v)[K], S2Red<A>& R, int C, int rank, int& buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) merge(v[k], shfl_acc(v[k], o));
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) R.warp[k][warp] = v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[k] = R.warp[k][lane & (kS2Warps - 1)];
#pragma unroll
            for (int o = kS2Warps / 2; o > 0; o >>= 1) merge(v[k], shfl_acc(v[k], o));
            if (lane < C) *cluster_map(&R.part[buf][k][rank], lane) = v[k];
        }
    }
    cluster_sync(C);
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[k] = R.part[buf][k][lane & (C - 1)];
            for (int o = C >> 1; o > 0; o >>= 1) merge(v[k], shfl_acc(v[k], o));
        }
    }
    buf ^= 1;
}

// Scalars of the solve, formed by one thread of every CTA (same values).
template <typename T>
struct S2Scal {
    T alpha, beta;
    double rz, alpha_d;
    double ff, rr, rr0_in, rr_in, eta2;
    int done, idone, iters, it_in, outer, status, capped;
};

// Sweeps and transfers of the levels held by CTA 0: barriers of the whole CTA
// above the tiny levels, of warp 0 within them.
template <typename T>
__device__ __forceinline__ void tiny_vcycle(S2View<T>* S, int l0, int lb, int pre, int post,
                                            int bottom) {
    const int t = threadIdx.x;   // < 32
    for (int l = l0; l < lb; ++l) {
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < pre; ++s)
            for (int k = 0; k < nc; ++k) {
                s2_gs(S[l], k, s == 0 && k == 0, t, 32);
                __syncwarp();
            }
        s2_restrict(S[l], S[l + 1], pre == 1, t, 32);
        __syncwarp();
    }
    {
        // bottom level (at most 3 x 3 cells): remove the mean, then sweep
        const S2View<T>& B = S[lb];
        const int n = B.nx * B.ny;
        typename S2AccOf<T>::type a{};
        for (int i = 0; i < n; ++i) a.add_prod(B.f[i], T(1));
        const T mean = T(a.s) / T(n);
        __syncwarp();
        if (t < n) B.f[t] -= mean;
        __syncwarp();
        const int nc = s2_classes(B);
        for (int s = 0; s < bottom; ++s)
            for (int k = 0; k < nc; ++k) {
                s2_gs(B, k, s == 0 && k == 0, t, 32);
                __syncwarp();
            }
    }
    for (int l = lb - 1; l >= l0; --l) {
        s2_prolong(S[l], S[l + 1], t, 32);
        __syncwarp();
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < post; ++s)
            for (int k = nc - 1; k >= 0; --k) {
                s2_gs(S[l], k, false, t, 32);
                __syncwarp();
            }
    }
}
template <typename T>
__device__ __forceinline__ void single_vcycle(S2View<T>* S, int lc, int lt, int lb, int pre,
                                              int post, int bottom) {
    const int t = threadIdx.x, nt = kS2Threads;
    for (int l = lc; l < lt; ++l) {
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < pre; ++s)
            for (int k = 0; k < nc; ++k) {
                s2_gs(S[l], k, s == 0 && k == 0, t, nt);
                __syncthreads();
            }
        s2_restrict(S[l], S[l + 1], pre == 1, t, nt);
        __syncthreads();
    }
    if (t < 32) tiny_vcycle(S, lt, lb, pre, post, bottom);
    __syncthreads();
    for (int l = lt - 1; l >= lc; --l) {
        s2_prolong(S[l], S[l + 1], t, nt);
        __syncthreads();
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < post; ++s)
            for (int k = nc - 1; k >= 0; --k) {
                s2_gs(S[l], k, false, t, nt);
                __syncthreads();
            }
    }
}

// r = f - A x of the strip, f = sign (b - mean b), to float64 accuracy (the
// arithmetic of k_ir_residual), stored times h^2 as the right-hand side of the
// scaled system; per-thread ||f||^2 (first) and ||r||^2.
template <typename T>
__device__ __forceinline__ void s2_residual(const S2Args<T>& a, const S2View<T>& L, double mb,
                                            bool first, T& ff, T& rr) {
    const int nx = L.nx, n = L.rows * nx;
    const bool pos = a.io.sign > 0.0;
    const int N = a.g.ncell;
    if constexpr (sizeof(T) == sizeof(float)) {
        const float* xh = reinterpret_cast<const float*>(a.io.x);
        const float* xl = xh + N;
        const float* bh = reinterpret_cast<const float*>(a.io.b);
        const float* bl = bh + N;
        const f2 mdf = df_neg(df_of(mb));
        const f2 ih2 = df_of(a.g.ih2);
        const float h2 = float(a.g.h * a.g.h);
        for (int q = threadIdx.x; q < n; q += kS2Threads) {
            const int r = s2_div(q, L.inv_nx), i = q - r * nx, j = L.j0 + r;
            const int idx = j * nx + i;
            f2 f = df_add(f2{bh[idx], bl[idx]}, mdf);
            if (!pos) f = df_neg(f);
            const int m0 = i == 0 ? idx + nx - 1 : idx - 1, m1 = i == nx - 1 ? idx - i : idx + 1;
            const int m2 = j == 0 ? idx + (L.ny - 1) * nx : idx - nx;
            const int m3 = j == L.ny - 1 ? i : idx + nx;
            const float w1 = L.w0[i == nx - 1 ? q - i : q + 1];
            const float w3 = r == L.rows - 1 ? L.w1p[i] : L.w1[q + nx];
            const float ch = __ldcg(xh + idx), cl = __ldcg(xl + idx);
            float S = 0.f, c = 0.f;
            df_face_term(L.w0[q], ch, cl, __ldcg(xh + m0), __ldcg(xl + m0), S, c);
            df_face_term(w1, ch, cl, __ldcg(xh + m1), __ldcg(xl + m1), S, c);
            df_face_term(L.w1[q], ch, cl, __ldcg(xh + m2), __ldcg(xl + m2), S, c);
            df_face_term(w3, ch, cl, __ldcg(xh + m3), __ldcg(xl + m3), S, c);
            const f2 ax = f2_mul(two_sum(S, c), ih2);
            const f2 rv = df_add(f, df_neg(ax));
            const float rt = __fadd_rn(rv.hi, rv.lo);
            L.f[q] = rt * h2;
            if (first) {
                const float ft = __fadd_rn(f.hi, f.lo);
                ff += ft * ft;
            }
            rr += rt * rt;
        }
    } else {
        const double h2 = a.g.h * a.g.h;
        const double* x = a.io.x;
        for (int q = threadIdx.x; q < n; q += kS2Threads) {
            const int r = s2_div(q, L.inv_nx), i = q - r * nx, j = L.j0 + r;
            const int idx = j * nx + i;
            const double f = pos ? a.io.b[idx] - mb : mb - a.io.b[idx];
            const int m0 = i == 0 ? idx + nx - 1 : idx - 1, m1 = i == nx - 1 ? idx - i : idx + 1;
            const int m2 = j == 0 ? idx + (L.ny - 1) * nx : idx - nx;
            const int m3 = j == L.ny - 1 ? i : idx + nx;
            const double xc = __ldcg(x + idx);
            double ax = L.w0[q] * (xc - __ldcg(x + m0));
            ax += L.w0[i == nx - 1 ? q - i : q + 1] * (xc - __ldcg(x + m1));
            ax += L.w1[q] * (xc - __ldcg(x + m2));
            ax += (r == L.rows - 1 ? L.w1p[i] : L.w1[q + nx]) * (xc - __ldcg(x + m3));
            const double rv = f - ax * a.g.ih2;
            L.f[q] = rv * h2;
            if (first) ff += f * f;
            rr += rv * rv;
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kS2Threads, 1) k_solve2d(const __grid_constant__ S2Args<T> a) {
    using A = typename S2AccOf<T>::type;
    extern __shared__ __align__(16) unsigned char s2_raw[];
    T* sm = reinterpret_cast<T*>(s2_raw);
    __shared__ S2View<T> V[kS2MaxCluster];
    __shared__ S2View<T> S[kMaxLevels];
    __shared__ S2Red<A> R;
    __shared__ S2Scal<T> sc;
    __shared__ T *vp, *vpm, *vpp, *vq, *ve;
    const S2Plan& P = a.P;
    const int C = P.C, rank = cluster_rank(), tid = threadIdx.x;
    const int lc = P.lc, lb = P.nlev - 1;

    // ---- this CTA's views ----
    if (tid <= lc) {
        const int l = tid;
        const S2Lev& L = P.lev[l];
        const int j0 = s2_row(P, l, rank), rows = s2_row(P, l, rank + 1) - j0;
        const int cm = rank == 0 ? C - 1 : rank - 1, cp = rank == C - 1 ? 0 : rank + 1;
        const int rm = s2_row(P, l, cm + 1) - s2_row(P, l, cm);
        const int jm = j0 == 0 ? L.ny - 1 : j0 - 1, jp = j0 + rows == L.ny ? 0 : j0 + rows;
        S2View<T>& v = V[l];
        s2_view_sizes(v, L, j0, rows);
        if (l == lc) {   // held by CTA 0
            T* b = cluster_map(sm, 0);
            v.x = b + L.ox + j0 * L.nx;
            v.f = b + L.of + j0 * L.nx;
            v.w0 = b + L.ow0 + j0 * L.nx;
            v.w1 = b + L.ow1 + j0 * L.nx;
            v.di = nullptr;
            v.xm = b + L.ox + jm * L.nx;
            v.xp = b + L.ox + jp * L.nx;
            v.w1p = b + L.ow1 + jp * L.nx;
        } else {
            auto own = [&](int o, T* g) { return o >= 0 ? sm + o : g + (size_t)j0 * L.nx; };
            auto up = [&](int o, T* g) {
                return o >= 0 ? cluster_map(sm + o, cm) + (rm - 1) * L.nx : g + (size_t)jm * L.nx;
            };
            auto dn = [&](int o, T* g) {
                return o >= 0 ? cluster_map(sm + o, cp) : g + (size_t)jp * L.nx;
            };
            const int gl = l & 1;   // workspace places exist for levels 0 and 1
            v.x = own(L.ox, a.gx[gl]);
            v.f = own(L.of, a.gf[gl]);
            v.w0 = own(L.ow0, a.gw0[gl]);
            v.w1 = own(L.ow1, a.gw1[gl]);
            v.di = own(L.od, a.gdi);
            v.xm = up(L.ox, a.gx[gl]);
            v.xp = dn(L.ox, a.gx[gl]);
            v.w1p = dn(L.ow1, a.gw1[gl]);
            if (l == 0) {
                vp = own(P.op, a.gp);
                vpm = up(P.op, a.gp);
                vpp = dn(P.op, a.gp);
                vq = own(P.oq, a.gq);
                ve = own(P.oe, a.ge);
            }
        }
    } else if (tid >= 32 && tid - 32 + lc <= lb) {
        const int l = tid - 32 + lc;
        const S2Lev& L = P.lev[l];
        S2View<T>& v = S[l];
        s2_view_sizes(v, L, 0, L.ny);
        v.x = sm + L.ox;
        v.f = sm + L.of;
        v.w0 = sm + L.ow0;
        v.w1 = sm + L.ow1;
        v.di = sm + L.od;
        v.xm = v.x + (L.ny - 1) * L.nx;
        v.xp = v.x;
        v.w1p = v.w1;
    }
    int lt = lb;   // first level of one warp
    while (lt > lc && P.lev[lt - 1].nx * P.lev[lt - 1].ny <= kTinyCells) --lt;
    __syncthreads();
    const S2View<T>& L0 = V[0];

    // ---- face coefficients of level 0 ----
    {
        const int nx = L0.nx, n = L0.rows * nx;
        for (int q = tid; q < n; q += kS2Threads) {
            const int r = s2_div(q, L0.inv_nx), i = q - r * nx, j = L0.j0 + r;
            const int idx = j * nx + i;
            const int m0 = i == 0 ? idx + nx - 1 : idx - 1;
            const int m2 = j == 0 ? idx + (L0.ny - 1) * nx : idx - nx;
            T w0, w1;
            if constexpr (sizeof(T) == sizeof(float)) {
                const float pc = __ldg(a.io.phi + idx);
                w0 = beta_face32(pc, __ldg(a.io.phi + m0), a.ph);
                w1 = wall_face(a.g, j, 2) ? 0.f : beta_face32(pc, __ldg(a.io.phi + m2), a.ph);
            } else {
                const PC<double> pc = pc_of(a.ph, double());
                const double rc = rho_of_p(__ldg(a.io.phi + idx), pc);
                w0 = 1.0 / (0.5 * (rc + rho_of_p(__ldg(a.io.phi + m0), pc)));
                w1 = wall_face(a.g, j, 2) ? 0.0
                                          : 1.0 / (0.5 * (rc + rho_of_p(__ldg(a.io.phi + m2), pc)));
            }
            L0.w0[q] = w0;
            L0.w1[q] = w1;
            if (a.b0) {
                a.b0[idx] = w0;
                a.b1[idx] = w1;
            }
        }
    }
    cluster_sync(C);
    // ---- coarse coefficients (a coarse row's children are the CTA's own) ----
    for (int l = 0; l < lc; ++l) {
        s2_coarsen(V[l], V[l + 1], tid, kS2Threads);
        __syncthreads();
    }
    cluster_sync(C);
    for (int l = 0; l < lc; ++l) s2_invdiag(V[l], tid, kS2Threads);
    if (rank == 0)
        for (int l = lc; l <= lb; ++l) {
            s2_invdiag(S[l], tid, kS2Threads);
            if (l < lb) s2_coarsen(S[l], S[l + 1], tid, kS2Threads);
            __syncthreads();
        }

    // ---- iterative refinement ----
    const double mb = a.sc->mean_b, rtol2 = a.sc->rtol2, eta2_min = a.sc->eta2_min;
    const int maxit = a.sc->maxit;
    const double h4 = (a.g.h * a.g.h) * (a.g.h * a.g.h);
    int buf = 0;
    auto acc_of = [](T v) { A x{}; x.s = v; return x; };
    for (int outer = 0;; ++outer) {
        const bool first_res = outer == 0;
        {
            T ff = T(0), rr = T(0);
            s2_residual(a, L0, mb, first_res, ff, rr);
            A v[2] = {acc_of(ff), acc_of(rr)};
            cluster_totals<2>(v, R, C, rank, buf);
            if (tid == 0) {
                // as ir_finish
                if (first_res) {
                    sc.ff = v[0].value();
                    sc.iters = sc.capped = sc.done = sc.status = 0;
                }
                const double rrv = v[1].value();
                sc.rr = rrv;
                sc.rr0_in = rrv * h4;
                sc.rr_in = sc.rz = 0.0;
                sc.outer = outer + 1;
                sc.idone = 0;
                if (!(rrv == rrv)) {
                    sc.done = 1;
                    sc.status = 4;   // PF_ERR_NONFINITE
                } else if (rrv <= rtol2 * sc.ff) {
                    sc.done = 1;
                } else if (sc.capped) {
                    sc.done = 1;
                    sc.status = 3;   // PF_ERR_NOT_CONVERGED
                } else {
                    const double e2 = rtol2 * sc.ff / rrv;
                    sc.eta2 = e2 > eta2_min ? e2 : eta2_min;
                }
            }
            __syncthreads();
        }
        if (sc.done || outer == 64) break;
        for (int it = 0;; ++it) {
            const bool first = it == 0;
            // V-cycle, down
            for (int l = 0; l < lc; ++l) {
                const S2View<T>& L = V[l];
                const int nc = s2_classes(L);
                for (int s = 0; s < P.pre; ++s)
                    for (int k = 0; k < nc; ++k) {
                        s2_gs(L, k, s == 0 && k == 0, tid, kS2Threads);
                        cluster_sync(C);
                    }
                s2_restrict(L, V[l + 1], P.pre == 1, tid, kS2Threads);
                if (l + 1 < lc) __syncthreads();
                else cluster_sync(C);
            }
            if (rank == 0)
                single_vcycle(S, lc, lt, lb, P.pre, P.post, P.bottom_sweeps);
            cluster_sync(C);
            // up
            A d[2] = {A{}, A{}};
            for (int l = lc - 1; l >= 0; --l) {
                const S2View<T>& L = V[l];
                s2_prolong(L, V[l + 1], tid, kS2Threads);
                cluster_sync(C);
                const int nc = s2_classes(L);
                for (int s = 0; s < P.post; ++s)
                    for (int k = nc - 1; k >= 0; --k) {
                        if (l == 0 && s == P.post - 1 && k == 0) {
                            s2_gs_dots(L, vq, first, d[0], d[1], tid, kS2Threads);
                        } else {
                            s2_gs(L, k, false, tid, kS2Threads);
                            cluster_sync(C);
                        }
                    }
            }
            cluster_totals<2>(d, R, C, rank, buf);
            if (tid == 0) {
                const double rz = d[0].value();
                sc.beta = first ? T(0) : T(-sc.alpha_d * d[1].value() / sc.rz);
                sc.rz = rz;
            }
            __syncthreads();
            s2_direction(L0, vp, sc.beta, first, tid, kS2Threads);
            cluster_sync(C);
            A pq[1] = {A{}};
            s2_apply(L0, vp, vpm, vpp, vq, pq[0], tid, kS2Threads);
            cluster_totals<1>(pq, R, C, rank, buf);
            if (tid == 0) {
                const double v = pq[0].value();
                sc.alpha_d = v != 0.0 ? sc.rz / v : 0.0;
                sc.alpha = T(sc.alpha_d);
            }
            __syncthreads();
            A rr[1] = {acc_of(s2_update(L0, vp, vq, ve, sc.alpha, first, tid, kS2Threads))};
            cluster_totals<1>(rr, R, C, rank, buf);
            if (tid == 0) {
                const double v = rr[0].value();
                sc.rr_in = v;
                sc.iters += 1;
                if (!(v == v) || v <= sc.eta2 * sc.rr0_in) {
                    sc.idone = 1;
                } else if (sc.iters >= maxit) {
                    sc.idone = 1;
                    sc.capped = 1;
                }
            }
            __syncthreads();
            if (sc.idone) break;
        }
        // x += e
        {
            const int n = L0.rows * L0.nx, base = L0.j0 * L0.nx;
            if constexpr (sizeof(T) == sizeof(float)) {
                float* xh = reinterpret_cast<float*>(a.io.x);
                float* xl = xh + a.g.ncell;
                for (int q = tid; q < n; q += kS2Threads) df_acc(xh[base + q], xl[base + q], ve[q]);
            } else {
                for (int q = tid; q < n; q += kS2Threads) a.io.x[base + q] += ve[q];
            }
        }
        cluster_sync(C);
    }
    if (rank == 0 && tid == 0) {
        CGScalars* o = a.sc;
        o->ff = sc.ff;
        o->rr = sc.rr;
        o->iters = sc.iters;
        o->outer = sc.outer;
        o->done = sc.done;
        o->idone = 1;
        o->capped = sc.capped;
        if (o->status == 0) o->status = sc.status;
    }
    cluster_sync(C);   // no CTA leaves while another may read its memory
}

// Levels of at most this many cells go to CTA 0: about the size where a phase
// over the cluster costs what one CTA's phase does (the float64 pipe makes that
// smaller for float64).
template <typename T> constexpr int kSingleCells = sizeof(T) == 4 ? 1024 : 256;
template <typename T> constexpr int kCtaCells = sizeof(T) == 4 ? 512 : 256;

template <typename T>
int max_cluster() {
    static std::once_flag once;
    static int best = 0;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_solve2d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kS2Smem);
        cudaFuncSetAttribute(k_solve2d<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (int c = kS2MaxCTAs; c >= 1 && best == 0; c >>= 1) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c);
            cfg.blockDim = dim3(kS2Threads);
            cfg.dynamicSmemBytes = kS2Smem;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = c;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, k_solve2d<T>, &cfg) == cudaSuccess && n > 0)
                best = c;
        }
        cudaGetLastError();
    });
    return best;
}

}  // namespace

void solve2d_prepare() {
    max_cluster<float>();
    max_cluster<double>();
}

template <typename T>
bool solve2d_plan(const MGHier<T>& H, bool beta_global, S2Plan& P) {
    const int mc = max_cluster<T>();
    return mc > 0 && s2_plan<T>(H, kSingleCells<T>, kCtaCells<T>, mc, kS2Smem, beta_global, P);
}

template <typename T>
cudaError_t launch_solve2d(const S2Plan& P, const Dims& g, const Phys& ph,
                           const SolveIO<T, 2>& io, const MGHier<T>& H, T* b0, T* b1,
                           CGScalars* sc, cudaStream_t s) {
    S2Args<T> a;
    a.P = P;
    a.g = g;
    a.ph = ph;
    a.io = io;
    a.b0 = b0;
    a.b1 = b1;
    for (int l = 0; l < 2; ++l) {
        a.gx[l] = H.lev[l].x;
        a.gf[l] = H.lev[l].f;
        a.gw0[l] = l == 0 ? b0 : H.lev[l].beta[0];
        a.gw1[l] = l == 0 ? b1 : H.lev[l].beta[1];
    }
    a.gp = io.p[0];
    a.gdi = io.p[1];   // the second direction buffer is not needed here
    a.gq = io.q;
    a.ge = io.e;
    a.sc = sc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P.C);
    cfg.blockDim = dim3(kS2Threads);
    cfg.dynamicSmemBytes = (size_t)P.elems * sizeof(T);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = P.C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_solve2d<T>, a);
}

#define PF_INST_S2(T)                                                                           \
    template bool solve2d_plan<T>(const MGHier<T>&, bool, S2Plan&);                             \
    template cudaError_t launch_solve2d<T>(const S2Plan&, const Dims&, const Phys&,             \
                                           const SolveIO<T, 2>&, const MGHier<T>&, T*, T*,      \
                                           CGScalars*, cudaStream_t);
PF_INST_S2(float)
PF_INST_S2(double)

}  // namespace pf
