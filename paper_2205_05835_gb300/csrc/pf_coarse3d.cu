// The coarse part of a 3D V-cycle in one launch of a thread-block cluster: the
// levels from about 32^3 cells down, each level's arrays in shared memory,
// slabs of planes per CTA, the level of at most 32 cells solved
// by its inverse. It replaces, per V-cycle, four launches per level of a few
// thousand cells (4 to 5 us each) and a single-CTA kernel whose ~70 dependent
// phases took 41 us at 16^3 in float32 and 118 us at 12^3 in float64. One launch
// takes 65k cycles from 32^3 (float32), 120k from 24^3 (float64; 69k in float32)
// and 141k from 40 x 30 x 18 (float32). Its phases wait for each other: the
// levels of CTA 0 take a fifth to a half, the interpolation from them (remote
// loads) up to a fifth, staging the coefficients up to a seventh.
// Copying the planes of CTA 0's level before the interpolation, right-hand side
// and coefficients in 16-byte pieces, and a higher cost of odd levels in the
// plan gave 3 to 5 % on a 160 x 120 x 72 step and lost 1 % on a 192 x 160 x 96
// solve: not done.
#include <mutex>

#include "pf_cluster.cuh"
#include "pf_coarse3d.cuh"
#include "pf_device.cuh"

namespace pf {

namespace {

constexpr size_t kC3Smem = 212 * 1024;   // dynamic shared memory of a CTA

template <typename T>
struct C3Args {
    C3Plan P;
    const T* beta[kMaxLevels][3];
    int dioff[kMaxLevels];   // offset of a level's inverse diagonals
    T* di;
    T* minv;                 // the dense level's inverse
    const T* f;              // level l0: right-hand side and correction
    T* x;
    T h2;                    // h^2 of level l0
    const CGScalars* sc;
};

// Once per solve: inverse diagonals of every level (blocks 1 ..) and the dense
// level's inverse (block 0).
template <typename T>
__global__ void __launch_bounds__(kS2Threads) k_c3_setup(const __grid_constant__ C3Args<T> a) {
    const C3Plan& P = a.P;
    const int tid = threadIdx.x;
    if (blockIdx.x > 0) {
        const int t0 = (blockIdx.x - 1) * kS2Threads + tid, nt = (gridDim.x - 1) * kS2Threads;
        for (int l = P.l0; l < P.ld; ++l) {
            const C3Lev& L = P.lev[l];
            const int n = L.nx * L.ny * L.nz, sxy = L.nx * L.ny;
            const T kap = T(P.kappa[l]);
            for (int q = t0; q < n; q += nt) {
                const int k = q / sxy, j = (q - k * sxy) / L.nx, i = q - (k * L.ny + j) * L.nx;
                const int ir = i == L.nx - 1 ? q - i : q + 1;
                const int jr = j == L.ny - 1 ? q - j * L.nx : q + L.nx;
                const int kr = k == L.nz - 1 ? q - k * sxy : q + sxy;
                const T d = ((a.beta[l][0][q] + a.beta[l][0][ir]) +
                             (a.beta[l][1][q] + a.beta[l][1][jr])) +
                            (a.beta[l][2][q] + a.beta[l][2][kr]);
                a.di[a.dioff[l] + q] = s2_rcp(kap * d);
            }
        }
        return;
    }
    extern __shared__ __align__(16) unsigned char c3_raw[];
    T* M = reinterpret_cast<T*>(c3_raw);
    __shared__ C3View<T> v;
    __shared__ T colrow[2 * kS2ColRow];
    __shared__ T w[3][kS2DenseMax];
    const C3Lev& L = P.lev[P.ld];
    const int n = L.nx * L.ny * L.nz;
    const T kap = T(P.kappa[P.ld]);
    if (tid < 3 * kS2DenseMax) {
        const int d = tid / kS2DenseMax, q = tid % kS2DenseMax;
        if (q < n) w[d][q] = kap * a.beta[P.ld][d][q];
    }
    if (tid == 0) {
        c3_view_sizes(v, L, 0, L.nz);
        for (int d = 0; d < 3; ++d) v.w[d] = w[d];
        v.w2p = w[2];
        v.x = v.f = v.di = v.xm = v.xp = w[0];   // (not read)
    }
    __syncthreads();
    c3_dense_build(v, M, tid);
    __syncthreads();
    c3_dense_fill(v, M, tid);
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
    c3_dense_weights(v, colrow + kS2ColRow, tid);
    __syncthreads();
    for (int k = 1; k < 3; ++k) {
        s2_dense_means(M, n, k, colrow, tid);
        __syncthreads();
    }
    s2_dense_project(M, n, colrow, tid);
    __syncthreads();
    for (int q = tid; q < n * s2_pad(n); q += kS2Threads) a.minv[q] = M[q];
}

// coefficients (scaled) and inverse diagonals of a CTA's part of level l
template <typename T>
__device__ __forceinline__ void c3_load(const C3Args<T>& a, const C3View<T>& v, int l, bool dense) {
    const int n = v.np * v.sxy, base = v.k0 * v.sxy;
    const T kap = T(a.P.kappa[l]);
    if (dense) return;   // (the dense level needs its inverse only)
#pragma unroll 4
    for (int q = threadIdx.x; q < n; q += kS2Threads) {
        v.w[0][q] = kap * __ldg(a.beta[l][0] + base + q);
        v.w[1][q] = kap * __ldg(a.beta[l][1] + base + q);
        v.w[2][q] = kap * __ldg(a.beta[l][2] + base + q);
        v.di[q] = __ldg(a.di + a.dioff[l] + base + q);
    }
}

template <typename T>
__global__ void __launch_bounds__(kS2Threads, 1) k_coarse3d(const __grid_constant__ C3Args<T> a) {
    if (a.sc->done || a.sc->idone) return;   // (the same in every CTA)
    extern __shared__ __align__(16) unsigned char c3_raw[];
    T* sm = reinterpret_cast<T*>(c3_raw);
    __shared__ C3View<T> V[kC3MaxCluster];
    __shared__ C3View<T> S[kMaxLevels];
    const C3Plan& P = a.P;
    const int C = P.C, rank = cluster_rank(), tid = threadIdx.x;
    const int l0 = P.l0, lc = P.lc, ld = P.ld;
    if (tid <= lc - l0) {
        const int l = l0 + tid;
        const C3Lev& L = P.lev[l];
        const int k0 = c3_plane(P, l, rank), np = c3_plane(P, l, rank + 1) - k0;
        const int cm = rank == 0 ? C - 1 : rank - 1, cp = rank == C - 1 ? 0 : rank + 1;
        const int nm = c3_plane(P, l, cm + 1) - c3_plane(P, l, cm);
        const int km = k0 == 0 ? L.nz - 1 : k0 - 1, kp = k0 + np == L.nz ? 0 : k0 + np;
        C3View<T>& v = V[tid];
        c3_view_sizes(v, L, k0, np);
        const int s = v.sxy;
        if (l == lc) {   // held by CTA 0
            T* b = cluster_map(sm, 0);
            v.x = b + L.ox + k0 * s;
            v.f = b + L.of + k0 * s;
            v.di = b + L.od + k0 * s;
            for (int d = 0; d < 3; ++d) v.w[d] = b + L.ow[d] + k0 * s;
            v.xm = b + L.ox + km * s;
            v.xp = b + L.ox + kp * s;
            v.w2p = b + L.ow[2] + kp * s;
        } else {
            v.x = sm + L.ox;
            v.f = sm + L.of;
            v.di = sm + L.od;
            for (int d = 0; d < 3; ++d) v.w[d] = sm + L.ow[d];
            v.xm = cluster_map(sm + L.ox, cm) + (nm - 1) * s;
            v.xp = cluster_map(sm + L.ox, cp);
            v.w2p = cluster_map(sm + L.ow[2], cp);
        }
    } else if (tid >= 32 && tid - 32 + lc <= ld) {
        const int l = tid - 32 + lc;
        const C3Lev& L = P.lev[l];
        C3View<T>& v = S[l];
        c3_view_sizes(v, L, 0, L.nz);
        v.x = sm + L.ox;
        v.f = sm + L.of;
        v.di = sm + L.od;
        for (int d = 0; d < 3; ++d) v.w[d] = sm + L.ow[d];
        v.xm = v.x + (L.nz - 1) * v.sxy;
        v.xp = v.x;
        v.w2p = v.w[2];
    }
    __syncthreads();
    // ---- stage in ----
    for (int l = l0; l < lc; ++l) c3_load(a, V[l - l0], l, l == ld);
    if (rank == 0) {
        for (int l = lc; l <= ld; ++l) c3_load(a, S[l], l, l == ld);
        const C3View<T>& B = S[ld];
        const int n = B.sxy * B.nz;
        for (int q = tid; q < n * s2_pad(n); q += kS2Threads) sm[P.om + q] = __ldg(a.minv + q);
    }
    const bool alone = lc == l0;   // level l0 in CTA 0 (then the cluster has one CTA)
    const C3View<T>& top = alone ? S[l0] : V[0];
    __syncthreads();
    c3_cells(top.nx, top.ny, top.np, top.inv_ny, top.lf, tid, [&](int r, int j, int i) {
        const int q = (r * top.ny + j) * top.nx + i;
        const T f = a.h2 * a.f[top.k0 * top.sxy + q];
        top.f[q] = f;
        if (l0 < ld) c3_start(top, r, j, i, q, f);
    });
    cluster_sync(C);
    // ---- down ----
    for (int l = l0; l < lc; ++l) {
        const C3View<T>& L = V[l - l0];
        const int nc = c3_classes(L);
        for (int s = 0; s < P.pre; ++s)
            for (int k = s == 0 ? 1 : 0; k < nc; ++k) {
                c3_gs(L, k, tid);
                cluster_sync(C);
            }
        c3_restrict(L, V[l + 1 - l0], P.pre == 1, tid);
        cluster_sync(C);
    }
    if (rank == 0) {
        for (int l = lc; l < ld; ++l) {
            const int nc = c3_classes(S[l]);
            for (int s = 0; s < P.pre; ++s)
                for (int k = s == 0 ? 1 : 0; k < nc; ++k) {
                    c3_gs(S[l], k, tid);
                    __syncthreads();
                }
            c3_restrict(S[l], S[l + 1], P.pre == 1, tid);
            __syncthreads();
        }
        const C3View<T>& B = S[ld];
        const int n = B.sxy * B.nz;
        T x = s2_dense_part(sm + P.om, B.f, n, tid);
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        x += __shfl_xor_sync(0xffffffffu, x, 4);
        if ((tid & 7) == 0 && (tid >> 3) < n) B.x[tid >> 3] = x;
        __syncthreads();
        for (int l = ld - 1; l >= lc; --l) {
            c3_prolong(S[l], S[l + 1], tid);
            __syncthreads();
            const int nc = c3_classes(S[l]);
            for (int s = 0; s < P.post; ++s)
                for (int k = nc - 1; k >= 0; --k) {
                    c3_gs(S[l], k, tid);
                    __syncthreads();
                }
        }
    }
    cluster_sync(C);
    for (int l = lc - 1; l >= l0; --l) {
        const C3View<T>& L = V[l - l0];
        c3_prolong(L, V[l + 1 - l0], tid);
        cluster_sync(C);
        const int nc = c3_classes(L);
        for (int s = 0; s < P.post; ++s)
            for (int k = nc - 1; k >= 0; --k) {
                c3_gs(L, k, tid);
                cluster_sync(C);
            }
    }
    // (the last barrier above: no CTA leaves while another reads its memory)
    const int n = top.np * top.sxy;
    for (int q = tid; q < n; q += kS2Threads) a.x[top.k0 * top.sxy + q] = top.x[q];
}

template <typename T>
void c3_attributes() {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_coarse3d<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kC3Smem);
    });
}

template <typename T>
C3Args<T> c3_args(const C3Plan& P, const MGHier<T>& H, const CGScalars* sc) {
    C3Args<T> a;
    a.P = P;
    int off = 0;
    for (int l = P.l0; l <= P.ld; ++l) {
        for (int d = 0; d < 3; ++d) a.beta[l][d] = H.lev[l].beta[d];
        a.dioff[l] = off;
        off += H.lev[l].g.ncell;
    }
    a.di = H.c3_di;
    a.minv = H.c3_minv;
    a.f = H.lev[P.l0].f;
    a.x = H.lev[P.l0].x;
    a.h2 = T(H.lev[P.l0].g.h * H.lev[P.l0].g.h);
    a.sc = sc;
    return a;
}

}  // namespace

void coarse3d_prepare() {
    c3_attributes<float>();
    c3_attributes<double>();
}

template <typename T>
bool coarse3d_plan(const MGHier<T>& H, int l0, C3Plan& P) {
    return c3_plan<T>(H, l0, kC3Smem, kS2DenseMax, P);
}
template <typename T>
void coarse3d_sizes(const C3Plan& P, size_t* di, size_t* minv) {
    *di = 0;
    for (int l = P.l0; l <= P.ld; ++l)
        *di += (size_t)P.lev[l].nx * P.lev[l].ny * P.lev[l].nz;
    const C3Lev& L = P.lev[P.ld];
    const int n = L.nx * L.ny * L.nz;
    *minv = (size_t)n * s2_pad(n);
}

template <typename T>
void launch_coarse3d_setup(const C3Plan& P, const MGHier<T>& H, cudaStream_t s) {
    c3_attributes<T>();
    const C3Lev& L = P.lev[P.ld];
    const int n = L.nx * L.ny * L.nz;
    int blocks = (H.lev[P.l0].g.ncell + kS2Threads - 1) / kS2Threads;
    k_c3_setup<T><<<1 + (blocks < 152 ? blocks : 152), kS2Threads, n * s2_pad(n) * sizeof(T), s>>>(
        c3_args<T>(P, H, nullptr));
}

template <typename T>
void launch_coarse3d(const C3Plan& P, const MGHier<T>& H, const CGScalars* sc, cudaStream_t s) {
    c3_attributes<T>();
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
    cudaLaunchKernelEx(&cfg, k_coarse3d<T>, c3_args<T>(P, H, sc));
}

#define PF_INST_C3(T)                                                                         \
    template bool coarse3d_plan<T>(const MGHier<T>&, int, C3Plan&);                           \
    template void coarse3d_sizes<T>(const C3Plan&, size_t*, size_t*);                         \
    template void launch_coarse3d_setup<T>(const C3Plan&, const MGHier<T>&, cudaStream_t);    \
    template void launch_coarse3d<T>(const C3Plan&, const MGHier<T>&, const CGScalars*,       \
                                     cudaStream_t);
PF_INST_C3(float)
PF_INST_C3(double)

}  // namespace pf
