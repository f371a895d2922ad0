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
//
// Measured: four 64^2 float64 steps 27.6 -> 4.2 ms, four mixed 256^2 steps at
// density ratio 1000 (54 iterations a step) 21.4 -> 7.8 ms, two 128^2 float64
// steps between walls 26.1 -> 4.0 ms. What bounds it is the chain: some 35
// barriers an iteration (588 cycles across the cluster, 44 in a CTA), each with
// one or two cells a thread in between (some 450 cycles of issue and latency);
// in float64 the pipe of two lanes an SM besides (a warp's multiply-add takes 19
// cycles of it).
#include <mutex>
#include <type_traits>

#include "pf_cluster.cuh"
#include "pf_device.cuh"
#include "pf_solve2d.cuh"

namespace pf {

namespace {

constexpr int kS2Warps = kS2Threads / 32;

template <typename T>
struct S2Args {
    S2Plan P;
    Dims g;
    Phys ph;
    SolveIO<T, 2> io;
    T* b0;          // face coefficients to leave in the workspace (may be null)
    T* b1;
    T *gx[2], *gf[2], *gw0[2], *gw1[2];   // workspace places of levels 0 and 1
    T *gdi, *gp, *gq, *ge, *gs;
    CGScalars* sc;
    double h2;      // h^2 (mixed path: times the power of two 2^m that takes it to [1/2, 1))
    int m;
};

// ---- totals over the cluster ----
__device__ __forceinline__ S2AccF shfl_acc(S2AccF a, int o) {
    return S2AccF{__shfl_xor_sync(0xffffffffu, a.s, o), __shfl_xor_sync(0xffffffffu, a.c, o),
                  __shfl_xor_sync(0xffffffffu, a.d, o)};
}
__device__ __forceinline__ S2AccD shfl_acc(S2AccD a, int o) {
    return S2AccD{__shfl_xor_sync(0xffffffffu, a.s, o)};
}

template <typename A>
struct S2Red;
template <>
struct S2Red<S2AccF> {
    S2AccF warp[3][kS2Warps];
    S2AccF part[2][3][kS2MaxCTAs];   // [buffer][value][CTA], written by every CTA of the cluster
};
template <>
struct S2Red<S2AccD> {
    S2AccD all[3][kS2Threads];
    S2AccD part[2][3][kS2MaxCTAs];
};

// K totals over the cluster, valid in lane 0 of warps 0 .. K - 1 of every CTA
// (value k in warp k). Contains a cluster barrier, which also orders the phases
// before and after it. The partial sums are pushed into every CTA's memory
// before that barrier, so nothing remote is read after it.
// Floats are summed by shuffles in every warp; float64 values go through
// shared memory, so that one warp per value adds 16 of them per lane: a shuffle
// tree in all 16 warps would issue five times the float64 instructions (each
// occupies GB300's two-lane float64 pipe for 16 cycles).
template <int K, typename A>
__device__ __forceinline__ void cluster_totals(A (&v)[K], A& tot, S2Red<A>& R, int C, int rank,
                                               int& buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (std::is_same<A, S2AccF>::value) {
        if constexpr (K == 3) {
            // value 0 goes on in lanes 0 - 7, value 1 in 8 - 15, value 2 in 16 - 31:
            // 6 merges instead of 15
            const bool up = lane & 16, b8 = lane & 8;
            A w = up ? v[2] : v[0];
            w.merge(shfl_acc(up ? v[0] : v[2], 16));
            v[1].merge(shfl_acc(v[1], 16));
            A x = b8 && !up ? v[1] : w;
            x.merge(shfl_acc(b8 || up ? w : v[1], 8));
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) x.merge(shfl_acc(x, o));
            if ((lane & 7) == 0 && lane < 24) R.warp[lane >> 3][warp] = x;
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v[k].merge(shfl_acc(v[k], o));
            if (lane == 0)
#pragma unroll
                for (int k = 0; k < K; ++k) R.warp[k][warp] = v[k];
        }
        __syncthreads();
        if (warp < K) {
            tot = R.warp[warp][lane & (kS2Warps - 1)];
#pragma unroll
            for (int o = kS2Warps / 2; o > 0; o >>= 1) tot.merge(shfl_acc(tot, o));
        }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) R.all[k][threadIdx.x] = v[k];
        __syncthreads();
        if (warp < K) {
            A s[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) s[j] = R.all[warp][lane + 32 * j];
#pragma unroll
            for (int j = 4; j < kS2Warps; ++j) s[j & 3].merge(R.all[warp][lane + 32 * j]);
            s[0].merge(s[1]);
            s[2].merge(s[3]);
            s[0].merge(s[2]);
            tot = s[0];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tot.merge(shfl_acc(tot, o));
        }
    }
    if (warp < K && lane < C) *cluster_map(&R.part[buf][warp][rank], lane) = tot;
    cluster_sync(C);
    if (warp < K) {
        tot = R.part[buf][warp][lane & (C - 1)];
        for (int o = C >> 1; o > 0; o >>= 1) tot.merge(shfl_acc(tot, o));
    }
    buf ^= 1;
}

// Scalars of the solve, formed by one thread of every CTA (same values).
template <typename T>
struct S2Scal {
    T alpha, beta;
    double zq, zs, pq;
    double ff, rr, rr0_in, rr_in, eta2;
    int done, idone, iters, outer, status, capped, again;
    S2Scale sca;
};

// The part of the V-cycle on the levels held by CTA 0 (the first one's right-
// hand side and its sweep's start are in place).
template <typename T>
__device__ __forceinline__ void single_vcycle(const S2View<T>* S, int lc, int ld, int pre,
                                              int post, unsigned fused_levels, const T* M) {
    const int t = threadIdx.x;
    for (int l = lc; l < ld; ++l) {
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < pre; ++s)
            for (int k = s == 0 ? 1 : 0; k < nc; ++k) {
                s2_gs(S[l], k, t);
                __syncthreads();
            }
        s2_restrict(S[l], S[l + 1], pre == 1, t);
        __syncthreads();
    }
    {
        const S2View<T>& B = S[ld];
        const int n = B.nx * B.ny;
        T x = s2_dense_part(M, B.f, n, t);
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        x += __shfl_xor_sync(0xffffffffu, x, 4);
        if ((t & 7) == 0 && (t >> 3) < n) B.x[t >> 3] = x;
        __syncthreads();
    }
    for (int l = ld - 1; l >= lc; --l) {
        const bool fused = (fused_levels >> l) & 1;
        if (fused) s2_prolong_gs(S[l], S[l + 1], t);
        else s2_prolong(S[l], S[l + 1], t);
        __syncthreads();
        const int nc = s2_classes(S[l]);
        for (int s = 0; s < post; ++s)
            for (int k = nc - 1 - (fused && s == 0 ? 1 : 0); k >= 0; --k) {
                s2_gs(S[l], k, t);
                __syncthreads();
            }
    }
}

// r = f - A x of the strip, f = sign (b - mean b), to float64 accuracy (the
// arithmetic of k_ir_residual), stored times h^2 (and its scale) as the right-hand
// side of the scaled system; per-thread ||f||^2 (first) and ||r||^2, both times
// their scale squared.
template <typename T>
__device__ __forceinline__ void s2_residual(const S2Args<T>& a, const S2View<T>& L, double mb,
                                            bool first, const S2Scale& sca, T& ff, T& rr) {
    const int nx = L.nx;
    const bool pos = a.io.sign > 0.0;
    const int N = a.g.ncell;
    if constexpr (sizeof(T) == sizeof(float)) {
        const float* xh = reinterpret_cast<const float*>(a.io.x);
        const float* xl = xh + N;
        const float* bh = reinterpret_cast<const float*>(a.io.b);
        const float* bl = bh + N;
        const f2 mdf = df_neg(df_of(mb));
        const f2 ih2 = df_of(a.g.ih2);
        const float h2 = float(a.h2), scale = sca.scale, fscale = sca.fscale;
        s2_cells(nx, L.rows, L.lf, threadIdx.x, [&](int r, int i) {
            const int q = r * nx + i, j = L.j0 + r;
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
            const float rt = __fadd_rn(rv.hi, rv.lo) * scale;
            L.f[q] = rt * h2;
            s2_start(L, i, j, q, rt * h2);
            if (first) {
                const float ft = __fadd_rn(f.hi, f.lo) * fscale;
                ff += ft * ft;
            }
            rr += rt * rt;
        });
    } else {
        const double h2 = a.h2;
        const double* x = a.io.x;
        s2_cells(nx, L.rows, L.lf, threadIdx.x, [&](int r, int i) {
            const int q = r * nx + i, j = L.j0 + r;
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
            s2_start(L, i, j, q, rv * h2);
            if (first) ff += f * f;
            rr += rv * rv;
        });
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
    __shared__ T *vp, *vq, *ve, *vs;
    __shared__ T colrow[2 * kS2ColRow];
    const S2Plan& P = a.P;
    const int C = P.C, rank = cluster_rank(), tid = threadIdx.x;
    const int lc = P.lc, ld = P.ld;
    T* M = sm + P.om;

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
            v.di = b + L.od + j0 * L.nx;
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
                vq = own(P.oq, a.gq);
                ve = own(P.oe, a.ge);
                vs = own(P.os, a.gs);
            }
        }
    } else if (tid >= 32 && tid - 32 + lc <= ld) {
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
    __syncthreads();
    const S2View<T>& L0 = V[0];

    // ---- face coefficients of level 0 ----
    {
        const int nx = L0.nx;
        s2_cells(nx, L0.rows, L0.lf, tid, [&](int r, int i) {
            const int q = r * nx + i, j = L0.j0 + r;
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
        });
    }
    cluster_sync(C);
    // ---- coarse coefficients (a coarse row's children are the CTA's own) ----
    for (int l = 0; l < lc; ++l) {
        s2_coarsen(V[l], V[l + 1], tid);
        __syncthreads();
    }
    cluster_sync(C);
    for (int l = 0; l < lc; ++l) s2_invdiag(V[l], tid);
    if (rank == 0) {
        for (int l = lc; l <= ld; ++l) {
            s2_invdiag(S[l], tid);
            if (l < ld) s2_coarsen(S[l], S[l + 1], tid);
            __syncthreads();
        }
        const int n = S[ld].nx * S[ld].ny;
        s2_dense_build(S[ld], M, tid);
        __syncthreads();
        s2_dense_fill(S[ld], M, tid);
        __syncthreads();
        T m[2];
        s2_gj_move(m, M, n, false, tid);
        s2_gj_publish(m, n, 0, colrow, tid);
        __syncthreads();
        for (int k = 0; k < n; ++k) {
            s2_gj_step(m, n, k, colrow + (k & 1) * kS2ColRow, tid);
            s2_gj_publish(m, n, k + 1, colrow + ((k + 1) & 1) * kS2ColRow, tid);
            __syncthreads();
        }
        s2_gj_move(m, M, n, true, tid);
        __syncthreads();
        s2_dense_weights(S[ld], colrow + kS2ColRow, tid);
        __syncthreads();
        for (int k = 1; k < 3; ++k) {
            s2_dense_means(M, n, k, colrow, tid);
            __syncthreads();
        }
        s2_dense_project(M, n, colrow, tid);
    }
    __syncthreads();

    // ---- iterative refinement ----
    const double mb = a.sc->mean_b, rtol2 = a.sc->rtol2, eta2_min = a.sc->eta2_min;
    const int maxit = a.sc->maxit;
    const double h4 = a.h2 * a.h2;
    int buf = 0;
    auto acc_of = [](T v) { A x{}; x.s = v; return x; };
    for (int outer = 0;; ++outer) {
        const bool first_res = outer == 0;
        if (tid == 0) {
            if (first_res) s2_scale_init(sc.sca, a.m);
            else s2_scale_next(sc.sca, sc.rr_in);
        }
        __syncthreads();
        for (int pass = 0;; ++pass) {
            T ff = T(0), rr = T(0);
            s2_residual(a, L0, mb, first_res, sc.sca, ff, rr);
            A v[2] = {acc_of(ff), acc_of(rr)}, tot{};
            cluster_totals<2>(v, tot, R, C, rank, buf);
            if (tid == 32) sc.rr = tot.value();
            __syncthreads();
            if (tid == 0) {
                sc.rr0_in = sc.rr * h4;
                if constexpr (std::is_same<T, float>::value) {
                    sc.again = s2_scale_check(sc.sca, first_res, pass, rtol2, tot.value(), sc.ff,
                                              sc.rr);
                } else {
                    if (first_res) sc.ff = tot.value();
                    sc.again = 0;
                }
                // as ir_finish
                if (first_res) sc.iters = sc.capped = sc.done = sc.status = 0;
                const double rrv = sc.rr;
                sc.outer = outer + 1;
                sc.idone = 0;
                if (sc.again) {
                } else if (!(rrv == rrv)) {
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
            if (!sc.again) break;
        }
        if (sc.done || outer == 64) break;
        for (int it = 0;; ++it) {
            const bool first = it == 0;
            // V-cycle, down (each sweep's first class from zero came with f)
            for (int l = 0; l < lc; ++l) {
                const S2View<T>& L = V[l];
                const int nc = s2_classes(L);
                for (int s = 0; s < P.pre; ++s)
                    for (int k = s == 0 ? 1 : 0; k < nc; ++k) {
                        s2_gs(L, k, tid);
                        cluster_sync(C);
                    }
                s2_restrict(L, V[l + 1], P.pre == 1, tid);
                cluster_sync(C);
            }
            if (rank == 0) single_vcycle(S, lc, ld, P.pre, P.post, P.fused, M);
            cluster_sync(C);
            // up
            for (int l = lc - 1; l >= 0; --l) {
                const S2View<T>& L = V[l];
                // one phase less where a thread has few cells (the interpolation is
                // then formed four times)
                const bool fused = (P.fused >> l) & 1;
                if (fused) s2_prolong_gs(L, V[l + 1], tid);
                else s2_prolong(L, V[l + 1], tid);
                cluster_sync(C);
                const int nc = s2_classes(L);
                for (int s = 0; s < P.post; ++s)
                    for (int k = nc - 1 - (fused && s == 0 ? 1 : 0); k >= 0; --k) {
                        s2_gs(L, k, tid);
                        cluster_sync(C);
                    }
            }
            // flexible CG with one set of products: s = A z, beta = -z.q / (p.q) of
            // the last direction (Polak-Ribiere: alpha q is the last change of r),
            // q = s + beta q and, A being symmetric, the new p.q = z.s + beta (2 z.q +
            // beta p.q); A p formed from p itself takes a phase and a reduction more
            A d[3] = {A{}, A{}, A{}}, tot{};
            s2_apply_dots(L0, vq, vs, first, d[0], d[1], d[2], tid);
            cluster_totals<3>(d, tot, R, C, rank, buf);
            if (tid == 32) sc.zq = tot.value();
            if (tid == 64) sc.zs = tot.value();
            __syncthreads();
            if (tid == 0) {
                const double rz = tot.value();
                const double beta = first ? 0.0 : -sc.zq / sc.pq;
                const double pq = first ? sc.zs : sc.zs + beta * (2.0 * sc.zq + beta * sc.pq);
                sc.beta = T(beta);
                sc.alpha = T(pq != 0.0 ? rz / pq : 0.0);
                sc.pq = pq;
            }
            __syncthreads();
            A rr[1] = {
                acc_of(s2_update(L0, vs, vp, vq, ve, sc.alpha, sc.beta, first, tid))};
            cluster_totals<1>(rr, tot, R, C, rank, buf);
            if (tid == 0) {
                const double v = tot.value();
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
                const float unscale = sc.sca.unscale;
                for (int q = tid; q < n; q += kS2Threads)
                    df_acc(xh[base + q], xl[base + q], ve[q] * unscale);
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
        // (latched: in a graph the step's later solves overwrite done)
        const int status = sc.done ? sc.status : 3;   // PF_ERR_NOT_CONVERGED: 64 refinements
        if (o->status == 0) o->status = status;
    }
    cluster_sync(C);   // no CTA leaves while another may read its memory
}

// dynamic shared memory left beside the kernel's static arrays
template <typename T>
size_t dynamic_smem() {
    cudaFuncAttributes at;
    if (cudaFuncGetAttributes(&at, k_solve2d<T>) != cudaSuccess) return 0;
    return kS2SmemMax - ((at.sharedSizeBytes + 1023) & ~(size_t)1023);
}

template <typename T>
int max_cluster() {
    static std::once_flag once;
    static int best = 0;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_solve2d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dynamic_smem<T>());
        cudaFuncSetAttribute(k_solve2d<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        for (int c = kS2MaxCTAs; c >= 1 && best == 0; c >>= 1) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c);
            cfg.blockDim = dim3(kS2Threads);
            cfg.dynamicSmemBytes = dynamic_smem<T>();
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
    return mc > 0 && s2_plan<T>(H, s2_limits<T>(mc, dynamic_smem<T>()), beta_global,
                                H.s2s != nullptr, P);
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
    a.gs = H.s2s != nullptr ? H.s2s : H.lev[0].x;
    a.sc = sc;
    a.h2 = g.h * g.h;
    a.m = 0;
    if (sizeof(T) == sizeof(float)) {
        const int e = -1 - ilogb(a.h2);
        a.m = e < -60 ? -60 : (e > 60 ? 60 : e);
        a.h2 = scalbn(a.h2, a.m);
    }
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
