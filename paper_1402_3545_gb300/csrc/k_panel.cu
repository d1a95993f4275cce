// k_panel.cu -- the paper's own operator: Eq. (1) on one gnomonic cubed-sphere panel with
// homogeneous Dirichlet conditions on the panel boundary, in the factorised form of Eq. (14)
// "LocalMatrixStencil" (Sec. 3.1), native FP64 (the paper's precision):
//
//   (A u)_{T,k} = (|T| E_k - alpha_T) u_{T,k} + sum_{T'} alpha_{TT'} u_{T',k}
//                 - |T| (B_k u_{T,k-1} + C_k u_{T,k+1}),
//   E_k = a_k - b_k - c_k,  B_k = -b_k,  C_k = -c_k  (B_0 = 0, C_{nz-1} = 0: Neumann),
//
// alpha_{TT'} < 0 the two-point flux coefficients of the four faces of T (a face on the panel
// boundary couples to a ghost value of 0 but still counts in alpha_T = their sum), |T| the cell's
// area. Only the coefficient arithmetic differs from the flat box: per column four face
// coefficients and the area instead of cx, cy and v; per level three radial vectors.
//
// Every kernel maps one thread to one vertical column and 32 consecutive x columns to a warp
// (coalesced rows, Sec. 3.1); horizontal neighbours come through the read-only cache. The Thomas
// factors of the column blocks are computed once per level (k_panel_factors): 1/m_k, the forward
// multiplier |T| B_k / m_k and the backward one |T| C_k / m_k, per cell. The forward-eliminated
// values go into the output field itself, which the back substitution then overwrites, so the
// sweeps need no scratch. On large levels the FP64 kernels are bound by the FP64 pipe, so their
// arithmetic is arranged for few instructions per cell: 9 for a residual, 9 for a Smooth without a
// norm (in the form (1 - rho) u + rho M^{-1}(f + H u), H the horizontal couplings: the vertical part of
// A u is not formed; 14 with the norm), 4 for the prolongation. Small levels leave most of the chip
// idle with a thread per column and 2 nz dependent FP64 operations (about 80 cycles each) per sweep:
// there a column is cut into chunks of planes (k_panel_chunk), and the pointwise kernels take a few
// planes per thread. FP32 (the mixed solve's inner cycles) keeps one thread per column throughout.
#include <algorithm>

#include "kernels.cuh"
#include "panel.cuh"

namespace tpmg {

namespace {

constexpr int CH = 16;  // chunks of a column in the chunked sweeps

template <class T>
struct PCol {
    int i, j;
    bool act, hw, he, hs, hn;  // in range; which horizontal neighbours lie on the panel
    size_t c;
    T area, aw, ae, as, an, at;
};

template <class T>
__device__ __forceinline__ PCol<T> panel_col(const PanelLvT<T>& L, int i, int j) {
    PCol<T> q;
    q.i = i;
    q.j = j;
    q.act = q.i < L.nx && q.j < L.ny;
    if (!q.act) return q;
    q.c = (size_t)q.j * L.nx + q.i;
    q.hw = q.i > 0;
    q.he = q.i < L.nx - 1;
    q.hs = q.j > 0;
    q.hn = q.j < L.ny - 1;
    q.area = __ldg(L.area + q.c);
    q.aw = __ldg(L.ax + (size_t)q.j * (L.nx + 1) + q.i);
    q.ae = __ldg(L.ax + (size_t)q.j * (L.nx + 1) + q.i + 1);
    q.as = __ldg(L.ay + (size_t)q.j * L.nx + q.i);
    q.an = __ldg(L.ay + (size_t)(q.j + 1) * L.nx + q.i);
    q.at = (q.aw + q.ae) + (q.as + q.an);
    return q;
}

template <class T>
__device__ __forceinline__ PCol<T> panel_col(const PanelLvT<T>& L) {
    return panel_col(L, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y * blockDim.y + threadIdx.y);
}

// (A u)_{T,k} given the centre value, its vertical neighbours (0 beyond the column) and
// |T| B_k, |T| C_k; the horizontal neighbours of plane k are read here (0 beyond the panel)
template <class T>
__device__ __forceinline__ T panel_Au(const PanelLvT<T>& L, const PCol<T>& q, const T* __restrict__ x, size_t b, int k,
                                     T uc, T um, T up, T tb, T tc) {
    const T xw = q.hw ? __ldg(x + b + q.c - 1) : T(0);
    const T xe = q.he ? __ldg(x + b + q.c + 1) : T(0);
    const T xs = q.hs ? __ldg(x + b + q.c - L.nx) : T(0);
    const T xn = q.hn ? __ldg(x + b + q.c + L.nx) : T(0);
    T s = fma(q.area, __ldg(L.E + k), -q.at) * uc;  // the diagonal
    s = fma(q.aw, xw, s);
    s = fma(q.ae, xe, s);
    s = fma(q.as, xs, s);
    s = fma(q.an, xn, s);
    s = fma(-tb, um, s);
    return fma(-tc, up, s);
}

// f - A u (APPLY: A u) at one cell in FP64, nine operations: the vertical and the |T| part of the diagonal share
// one product with |T|
template <bool APPLY = false>
__device__ __forceinline__ double panel_res(const PanelLv& L, const PCol<double>& q, const double* __restrict__ x, size_t b,
                                            int k, double fk, double uc, double um, double up) {
    const double xw = q.hw ? __ldg(x + b + q.c - 1) : 0.0;
    const double xe = q.he ? __ldg(x + b + q.c + 1) : 0.0;
    const double xs = q.hs ? __ldg(x + b + q.c - L.nx) : 0.0;
    const double xn = q.hn ? __ldg(x + b + q.c + L.nx) : 0.0;
    const double v = fma(-__ldg(L.C + k), up, fma(-__ldg(L.B + k), um, __ldg(L.E + k) * uc));
    if (APPLY) return fma(q.area, v, fma(q.an, xn, fma(q.as, xs, fma(q.ae, xe, fma(q.aw, xw, -q.at * uc)))));
    double r = fma(q.at, uc, fk);
    r = fma(-q.aw, xw, r);
    r = fma(-q.ae, xe, r);
    r = fma(-q.as, xs, r);
    r = fma(-q.an, xn, r);
    return fma(-q.area, v, r);
}
// f + H u: the right-hand side of a smoothing step's line solves (four operations)
__device__ __forceinline__ double panel_rhs(const PanelLv& L, const PCol<double>& q, const double* __restrict__ x, size_t b,
                                            double fk) {
    const double xw = q.hw ? __ldg(x + b + q.c - 1) : 0.0;
    const double xe = q.he ? __ldg(x + b + q.c + 1) : 0.0;
    const double xs = q.hs ? __ldg(x + b + q.c - L.nx) : 0.0;
    const double xn = q.hn ? __ldg(x + b + q.c + L.nx) : 0.0;
    return fma(-q.an, xn, fma(-q.as, xs, fma(-q.ae, xe, fma(-q.aw, xw, fk))));
}

}  // namespace

// Thomas factors of every column block of level L: m_0 = D_0, m_k = D_k - (|T| B_k)^2 / m_{k-1}
// with D_k = |T| E_k - alpha_T (the off-diagonals of row k are -|T| B_k below, -|T| C_k above, and
// C_{k-1} = B_k); stored 1/m_k, |T| B_k / m_k and |T| C_k / m_k.
// wf, wb (if not null): the products of the forward and of the backward multipliers over each chunk of
// pp planes, [chunk][column] (k_panel_chunk).
__global__ void __launch_bounds__(128) k_panel_factors(PanelLv L, double* __restrict__ inv, double* __restrict__ fl,
                                                       double* __restrict__ fw, double* __restrict__ wf,
                                                       double* __restrict__ wb, int pp) {
    const PCol<double> q = panel_col(L);
    if (!q.act) return;
    const size_t pl = (size_t)L.nx * L.ny;
    double m_prev = 1.0, pf = 1.0, pb = 1.0;
    for (int k = 0; k < L.nz; ++k) {
        const double d = fma(q.area, L.E[k], -q.at);
        const double tb = q.area * L.B[k];
        const double m = (k == 0) ? d : d - tb * tb / m_prev;
        const double iv = 1.0 / m;
        inv[(size_t)k * pl + q.c] = iv;
        fl[(size_t)k * pl + q.c] = tb * iv;
        const double w = q.area * L.C[k] * iv;
        fw[(size_t)k * pl + q.c] = w;
        m_prev = m;
        if (wf) {
            pf *= tb * iv;
            pb *= w;
            if ((k + 1) % pp == 0 || k + 1 == L.nz) {
                wf[(size_t)(k / pp) * pl + q.c] = pf;
                wb[(size_t)(k / pp) * pl + q.c] = pb;
                pf = pb = 1.0;
            }
        }
    }
}

// MODE 0 Smooth: out = u + coef M^{-1} (f - A u) (Eq. (11)), partial sums of ||f - A u||^2
// MODE 1 Residual (FP32; FP64: k_panel_point): out = f - A u
// MODE 2 line solve: out = coef M^{-1} u (u is the right-hand side)
// T is the arithmetic (double or float); the norm's partial sums are accumulated in T.
// NORM (FP64 Smooth): with the sums; without them the Smooth takes the form that needs no residual.
template <int MODE, class T, bool NORM>
__global__ void __launch_bounds__(128) k_panel_sweep(PanelLvT<T> L, T coef, const T* __restrict__ u,
                                                     const T* __restrict__ f, T* out, double* partials,
                                                     const int* done) {
    if (done && *(volatile const int*)done) return;
    const PCol<T> q = panel_col(L);
    const size_t pl = (size_t)L.nx * L.ny;
    const int nz = L.nz;
    T acc = 0;
    constexpr bool RHS = MODE == 0 && sizeof(T) == 8 && !NORM;
    if (q.act) {
        T um = 0, uc = (MODE != 2) ? __ldg(u + q.c) : T(0), dp = 0;
        T tb = 0;  // |T| B_k (B_0 = 0); |T| C_k = |T| B_{k+1} is carried to the next plane
#pragma unroll 2
        for (int k = 0; k < nz; ++k) {
            const size_t b = (size_t)k * pl;
            if constexpr (RHS) {
                const double r = panel_rhs(L, q, u, b, __ldg(f + b + q.c));
                dp = fma(__ldg(L.fl + b + q.c), dp, r * __ldg(L.inv + b + q.c));
                out[b + q.c] = dp;
                continue;
            }
            const T tc = (k + 1 < nz) ? q.area * __ldg(L.B + k + 1) : T(0);
            T r;
            if (MODE != 2) {
                const T up = (k + 1 < nz) ? __ldg(u + b + pl + q.c) : T(0);
                const T fk = __ldg(f + b + q.c);
                if constexpr (sizeof(T) == 8) r = panel_res(L, q, u, b, k, fk, uc, um, up);
                else r = fk - panel_Au(L, q, u, b, k, uc, um, up, tb, tc);
                um = uc;
                uc = up;
            } else {
                r = __ldg(u + b + q.c);
            }
            if (MODE != 2 && partials) acc = fma(r, r, acc);
            if (MODE != 1) {
                dp = fma(__ldg(L.fl + b + q.c), dp, r * __ldg(L.inv + b + q.c));  // forward elimination
                out[b + q.c] = dp;  // the output field holds d'_k until the back substitution
            } else {
                out[b + q.c] = r;
            }
            tb = tc;
        }
        if (MODE != 1) {
            T x = 0;
            for (int k = nz - 1; k >= 0; --k) {
                const size_t id = (size_t)k * pl + q.c;
                x = fma(__ldg(L.fw + id), x, out[id]);
                if constexpr (RHS) out[id] = fma(coef, x, (1.0 - coef) * __ldg(u + id));
                else out[id] = (MODE == 0) ? fma(coef, x, __ldg(u + id)) : coef * x;
            }
        }
    }
    if (MODE != 2 && partials) {
        const double s = block_sum((double)acc);
        if (threadIdx.x == 0 && threadIdx.y == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------- columns cut into chunks of planes
// FP64 sweeps of the small levels: a block owns 8 columns, each cut into 16 chunks of PP planes with a thread
// per chunk. Both recurrences (y_k = a_k + fl_k y_{k-1}, a_k = b_k / m_k; x_k = y_k + fw_k x_{k+1}) run
// twice per chunk: from zero, for the value the chunk hands on, and, once the carried value is known
// (the earlier chunks' values chained by the chunks' products of multipliers, wf and wb), for the
// chunk's own values. That is one more operation per cell and direction and 2 (2 PP + 16) instead of
// 2 nz dependent ones: on 64^2 x 128 a Smooth took 186 us with a thread per column.
// MODE 0 Smooth, 2 line solve (u the right-hand side), 4 RestrictSmooth (u the fine residual r_f:
// f_c = sum of the children to fc, out = coef M^{-1} f_c).
template <int MODE, int PP, bool NORM, int CB>
__global__ void __launch_bounds__(CB * CH) k_panel_chunk(PanelLv L, double coef, const double* __restrict__ u,
                                                         const double* __restrict__ f, double* out,
                                                         double* __restrict__ fc, double* partials, const int* done) {
    __shared__ double sy[CH][CB], sx[CH][CB];
    if (done && *(volatile const int*)done) return;
    const int tx = threadIdx.x, w = threadIdx.y, nz = L.nz, k0 = w * PP;
    // (a thread beyond the last column works on it and stores nothing)
    const int col = blockIdx.x * CB + tx, ncol = L.nx * L.ny;
    const bool act = col < ncol;
    const int cc = act ? col : ncol - 1;
    const PCol<double> q = panel_col(L, cc % L.nx, cc / L.nx);
    const size_t pl = (size_t)L.nx * L.ny;
    const int np = !act || k0 >= nz ? 0 : (nz - k0 < PP ? nz - k0 : PP);  // planes of this thread
    // Every load is unconditional (planes beyond the column repeat its last one), so that a pass's loads
    // are in flight together; planes beyond np get zeros and leave both chains at zero.
    double a[PP], y = 0.0, acc = 0.0;
    auto plane = [&](int p) { return (size_t)(k0 + p < nz ? k0 + p : nz - 1) * pl; };
    {
        const int kf = k0 < nz ? k0 : nz - 1;
        double um = 0.0, uc = 0.0, fl[PP];
        if (MODE == 0 && NORM) {
            uc = __ldg(u + (size_t)kf * pl + q.c);
            um = __ldg(u + (size_t)(kf > 0 ? kf - 1 : 0) * pl + q.c);
            if (kf == 0) um = 0.0;
        }
#pragma unroll
        for (int p = 0; p < PP; ++p) {
            const bool in = p < np;
            const int k = k0 + p < nz ? k0 + p : nz - 1;
            const size_t b = plane(p), id = b + q.c;
            double r;
            if (MODE == 0 && NORM) {
                double up = __ldg(u + (k + 1 < nz ? id + pl : id));
                if (k + 1 == nz) up = 0.0;
                r = panel_res(L, q, u, b, k, __ldg(f + id), uc, um, up);
                if (in) acc = fma(r, r, acc);
                um = uc;
                uc = up;
            } else if (MODE == 0) {
                r = panel_rhs(L, q, u, b, __ldg(f + id));
            } else if (MODE == 4) {
                const size_t nxf = 2 * (size_t)L.nx;
                const double* rf = u + 4 * b + (size_t)(2 * q.j) * nxf + 2 * q.i;
                r = (__ldg(rf) + __ldg(rf + 1)) + (__ldg(rf + nxf) + __ldg(rf + nxf + 1));
                if (in) fc[id] = r;
            } else {
                r = __ldg(u + id);
            }
            const double iv = __ldg(L.inv + id);
            fl[p] = __ldg(L.fl + id);
            a[p] = in ? r * iv : 0.0;
        }
#pragma unroll
        for (int p = 0; p < PP; ++p) y = fma(p < np ? fl[p] : 0.0, y, a[p]);
    }
    sy[w][tx] = y;
    const int last = (nz - 1) / PP;
    __syncthreads();
    if (w == 0) {  // one thread per column: each chunk's carried value in the place of what it hands on
        y = 0.0;
#pragma unroll 4
        for (int c = 0; c <= last; ++c) {
            const double e = sy[c][tx];
            sy[c][tx] = y;
            y = fma(__ldg(L.wf + (size_t)c * pl + q.c), y, e);
        }
    }
    __syncthreads();
    y = sy[w][tx];
#pragma unroll
    for (int p = 0; p < PP; ++p) {
        const double m = __ldg(L.fl + plane(p) + q.c);
        y = fma(p < np ? m : 0.0, y, a[p]);
        a[p] = p < np ? y : 0.0;
    }
    double x = 0.0;
#pragma unroll
    for (int p = PP - 1; p >= 0; --p) {
        const double m = __ldg(L.fw + plane(p) + q.c);
        x = fma(p < np ? m : 0.0, x, a[p]);
    }
    sx[w][tx] = x;
    __syncthreads();
    if (w == 0) {
        x = 0.0;
#pragma unroll 4
        for (int c = last; c >= 0; --c) {
            const double e = sx[c][tx];
            sx[c][tx] = x;
            x = fma(__ldg(L.wb + (size_t)c * pl + q.c), x, e);
        }
    }
    __syncthreads();
    x = sx[w][tx];
#pragma unroll
    for (int p = PP - 1; p >= 0; --p) {
        const size_t id = plane(p) + q.c;
        const double m = __ldg(L.fw + id), uo = MODE == 0 ? __ldg(u + id) : 0.0;
        x = fma(p < np ? m : 0.0, x, a[p]);
        if (p < np) out[id] = MODE == 0 ? fma(coef, x, NORM ? uo : (1.0 - coef) * uo) : coef * x;
    }
    if (MODE == 0 && NORM) {
        const double s = block_sum(acc);
        if (tx == 0 && w == 0) partials[blockIdx.x] = s;
    }
}

// FP64 Residual (MODE 1, stored in TO) and apply (MODE 3), pointwise: planes blockIdx.z * pz .. of each
// column, partial sums of ||f - A u||^2
template <int MODE, class TO>
__global__ void __launch_bounds__(128) k_panel_point(PanelLv L, const double* __restrict__ u,
                                                     const double* __restrict__ f, TO* __restrict__ out,
                                                     double* partials, const int* done, int pz) {
    if (done && *(volatile const int*)done) return;
    const PCol<double> q = panel_col(L);
    const size_t pl = (size_t)L.nx * L.ny;
    const int nz = L.nz, k0 = blockIdx.z * pz, k1 = k0 + pz < nz ? k0 + pz : nz;
    double acc = 0.0;
    if (q.act && k0 < k1) {
        size_t b = (size_t)k0 * pl;
        double um = k0 > 0 ? __ldg(u + b - pl + q.c) : 0.0, uc = __ldg(u + b + q.c);
#pragma unroll 4
        for (int k = k0; k < k1; ++k, b += pl) {
            const double up = k + 1 < nz ? __ldg(u + b + pl + q.c) : 0.0;
            const double r = panel_res<MODE == 3>(L, q, u, b, k, MODE == 3 ? 0.0 : __ldg(f + b + q.c), uc, um, up);
            out[b + q.c] = (TO)r;
            if (MODE == 1 && partials) acc = fma(r, r, acc);
            um = uc;
            uc = up;
        }
    }
    if (MODE == 1 && partials) {
        const double s = block_sum(acc);
        if (threadIdx.x == 0 && threadIdx.y == 0)
            partials[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    }
}

// RestrictSmooth onto level Lc: f_c = sum of the 2 x 2 children's residuals r_f (the equations are
// integrated over the cells), u_c = rho M_c^{-1} f_c (the first smoothing step from zero).
template <class T>
__global__ void __launch_bounds__(128) k_panel_restrict_smooth(PanelLvT<T> Lc, T rho, const T* __restrict__ rf,
                                                               T* __restrict__ fc, T* uc, const int* done) {
    if (done && *(volatile const int*)done) return;
    const PCol<T> q = panel_col(Lc);
    if (!q.act) return;
    const size_t plc = (size_t)Lc.nx * Lc.ny, nxf = 2 * (size_t)Lc.nx, plf = 4 * plc;
    const size_t f0 = (size_t)(2 * q.j) * nxf + 2 * q.i;
    T dp = 0;
    for (int k = 0; k < Lc.nz; ++k) {
        const T* r = rf + (size_t)k * plf + f0;
        const T s = (__ldg(r) + __ldg(r + 1)) + (__ldg(r + nxf) + __ldg(r + nxf + 1));
        const size_t id = (size_t)k * plc + q.c;
        fc[id] = s;
        dp = fma(__ldg(Lc.fl + id), dp, s * __ldg(Lc.inv + id));
        uc[id] = dp;
    }
    T x = 0;
    for (int k = Lc.nz - 1; k >= 0; --k) {
        const size_t id = (size_t)k * plc + q.c;
        x = fma(__ldg(Lc.fw + id), x, uc[id]);
        uc[id] = rho * x;
    }
}

// u_f += P u_c: bilinear in the logical grid (weights 3/4 and 1/4 per direction), a coarse
// neighbour beyond the panel boundary contributing 0. A thread takes the two fine rows of a coarse one, which
// share their x part: four operations per fine cell. P u_c is formed before it is added, so that only the last
// rounding is relative to u_f, of which the correction is a small part.
template <class T>
__global__ void __launch_bounds__(128) k_panel_prolongate(int nxc, int nyc, int nz, const T* __restrict__ uc,
                                                          T* __restrict__ uf, const int* done, int pz) {
    if (done && *(volatile const int*)done) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
    const int nxf = 2 * nxc;
    if (i >= nxf || J >= nyc) return;
    const int I = i >> 1, I2 = (i & 1) ? I + 1 : I - 1;
    const bool in2 = I2 >= 0 && I2 < nxc, js = J > 0, jn = J + 1 < nyc;
    const size_t plc = (size_t)nxc * nyc, c0 = (size_t)J * nxc + I, cx = (size_t)J * nxc + I2,
                 fo = (size_t)(2 * J) * nxf + i;
    const int k0 = blockIdx.z * pz, k1 = k0 + pz < nz ? k0 + pz : nz;
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const T* p = uc + (size_t)k * plc;
        T* o = uf + (size_t)k * 4 * plc + fo;
        const T o0 = o[0], o1 = o[nxf];
        T h = T(0.5625) * __ldg(p + c0);
        if (in2) h = fma(T(0.1875), __ldg(p + cx), h);
        T v0 = h, v1 = h;
        if (js) v0 = fma(T(0.1875), __ldg(p + c0 - nxc), v0);
        if (js && in2) v0 = fma(T(0.0625), __ldg(p + cx - nxc), v0);
        if (jn) v1 = fma(T(0.1875), __ldg(p + c0 + nxc), v1);
        if (jn && in2) v1 = fma(T(0.0625), __ldg(p + cx + nxc), v1);
        o[0] = o0 + v0;
        o[nxf] = o1 + v1;
    }
}

// ---------------------------------------------------------------- fused CG kernels (Sec. 3.1)
// SpMV: u += alpha p; p = z + beta p; q = A z + beta q; sigma = <p, q> (alpha, beta from the previous
// iteration in the device scalars; the u update lags one iteration, as in the flat-box CG)
__global__ void __launch_bounds__(128) k_panel_cg_spmv(PanelLv L, const Scalars* __restrict__ sc, double* u,
                                                       double* p, const double* __restrict__ z, double* q,
                                                       double* partials) {
    if (*(volatile const int*)&sc->done) return;
    const PCol<double> c = panel_col(L);
    const size_t pl = (size_t)L.nx * L.ny;
    const double alpha = sc->alpha, beta = sc->beta;
    double acc = 0.0;
    if (c.act) {
        double zm = 0.0, zc = __ldg(z + c.c), tb = 0.0;
        for (int k = 0; k < L.nz; ++k) {
            const size_t b = (size_t)k * pl, id = b + c.c;
            const double tc = (k + 1 < L.nz) ? c.area * __ldg(L.B + k + 1) : 0.0;
            const double zp = (k + 1 < L.nz) ? __ldg(z + id + pl) : 0.0;
            const double az = panel_Au(L, c, z, b, k, zc, zm, zp, tb, tc);
            const double po = p[id];
            u[id] = fma(alpha, po, u[id]);
            const double pn = fma(beta, po, zc);
            const double qn = fma(beta, q[id], az);
            p[id] = pn;
            q[id] = qn;
            acc = fma(pn, qn, acc);
            zm = zc;
            zc = zp;
            tb = tc;
        }
    }
    const double s = block_sum(acc);
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// Tridiag: r -= alpha q; z = M^{-1} r; partial sums of <r, r> (first nparts slots) and <r, z> (next)
__global__ void __launch_bounds__(128) k_panel_cg_tridiag(PanelLv L, const Scalars* __restrict__ sc, double* r,
                                                          const double* __restrict__ q, double* z, double* partials,
                                                          int nparts) {
    if (*(volatile const int*)&sc->done) return;
    const PCol<double> c = panel_col(L);
    const size_t pl = (size_t)L.nx * L.ny;
    const double alpha = sc->alpha;
    double rr = 0.0, rz = 0.0;
    if (c.act) {
        double dp = 0.0;
        for (int k = 0; k < L.nz; ++k) {
            const size_t id = (size_t)k * pl + c.c;
            const double rk = fma(-alpha, __ldg(q + id), r[id]);
            r[id] = rk;
            rr = fma(rk, rk, rr);
            dp = fma(__ldg(L.fl + id), dp, rk * __ldg(L.inv + id));
            z[id] = dp;
        }
        double x = 0.0;
        for (int k = L.nz - 1; k >= 0; --k) {
            const size_t id = (size_t)k * pl + c.c;
            x = fma(__ldg(L.fw + id), x, z[id]);
            z[id] = x;
            rz = fma(r[id], x, rz);
        }
    }
    const double s1 = block_sum(rr);
    __syncthreads();
    const double s2 = block_sum(rz);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        partials[blockIdx.y * gridDim.x + blockIdx.x] = s1;
        partials[nparts + blockIdx.y * gridDim.x + blockIdx.x] = s2;
    }
}

static dim3 panel_grid(int nx, int ny) { return dim3((nx + 31) / 32, (ny + 3) / 4); }

int panel_blocks(int nx, int ny) {
    const dim3 g = panel_grid(nx, ny);
    return (int)(g.x * g.y);
}

void launch_panel_cg_spmv(const PanelLv& L, const Scalars* sc, double* u, double* p, const double* z, double* q,
                          double* partials, cudaStream_t s) {
    k_panel_cg_spmv<<<panel_grid(L.nx, L.ny), dim3(32, 4), 0, s>>>(L, sc, u, p, z, q, partials);
    note_launch();
}

void launch_panel_cg_tridiag(const PanelLv& L, const Scalars* sc, double* r, const double* q, double* z,
                             double* partials, cudaStream_t s) {
    k_panel_cg_tridiag<<<panel_grid(L.nx, L.ny), dim3(32, 4), 0, s>>>(L, sc, r, q, z, partials,
                                                                        panel_blocks(L.nx, L.ny));
    note_launch();
}

void launch_panel_factors(const PanelLv& L, double* inv, double* fl, double* fw, double* wf, double* wb, cudaStream_t s) {
    k_panel_factors<<<panel_grid(L.nx, L.ny), dim3(32, 4), 0, s>>>(L, inv, fl, fw, wf, wb, panel_chunk_planes(L.nz));
    note_launch();
}

// planes per block of the pointwise kernels with `blocks` blocks a plane: 16 where the level fills the GPU with them, else
// 4, in equal parts, half as many where a thread takes two rows (the prolongation: 896 x 144 x 14 17.0 us, 18.4 with 16
// planes; 448 x 10 x 77 4.8, 5.4 with four); one or two where that gives at most 1024 blocks (a thread that takes four
// planes waits for memory four times: 64^2 x 3 prolongation 3.2 us, 2.6 with one)
static int point_planes(int nx, int ny, int nz, int blocks, int rows = 1) {
    for (int p = 1; p <= 2; ++p)
        if (blocks * ((nz + p - 1) / p) <= 1024) return p;
    const int p = (size_t)nx * ny > 65536 ? 16 / rows : 4 / rows, slabs = (nz + p - 1) / p;
    return (nz + slabs - 1) / slabs;
}

// The chunked sweep where the level has its chunk products (PanelLvT::wf). Returns the number of blocks, or
// -1 where it does not apply.
template <int MODE, int PP, int CB>
static int run_panel_chunk_cb(const PanelLv& L, double coef, const double* u, const double* f, double* out, double* fc,
                              double* partials, const int* done, cudaStream_t s) {
    const int nb = (L.nx * L.ny + CB - 1) / CB;
    constexpr int WR = 32 / CB;  // the chunks that the column has, in whole warps
    const dim3 b(CB, ((L.nz + PP - 1) / PP + WR - 1) / WR * WR);
    if (MODE == 0 && partials) k_panel_chunk<MODE, PP, MODE == 0, CB><<<nb, b, 0, s>>>(L, coef, u, f, out, fc, partials, done);
    else k_panel_chunk<MODE, PP, false, CB><<<nb, b, 0, s>>>(L, coef, u, f, out, fc, nullptr, done);
    note_launch();
    return nb;
}
// columns per block: 8, fewer where the blocks would not reach every SM
template <int MODE, int PP>
static int run_panel_chunk(const PanelLv& L, double coef, const double* u, const double* f, double* out, double* fc,
                           double* partials, const int* done, cudaStream_t s) {
    if (L.nx * L.ny <= 512) return run_panel_chunk_cb<MODE, PP, 2>(L, coef, u, f, out, fc, partials, done, s);
    if (L.nx * L.ny <= 2048) return run_panel_chunk_cb<MODE, PP, 4>(L, coef, u, f, out, fc, partials, done, s);
    return run_panel_chunk_cb<MODE, PP, 8>(L, coef, u, f, out, fc, partials, done, s);
}
template <int MODE>
static int panel_chunk(const PanelLv& L, double coef, const double* u, const double* f, double* out, double* fc,
                       double* partials, const int* done, cudaStream_t s) {
    if (!L.wf || !L.wb) return -1;
    // with the norm (14 operations a cell) the largest levels are bound by the FP64 pipe but where their planes fill the rows of
    // chunks: 180^2 x 40 62 us in chunks / 53, 128 x 254 x 169 344 / 276, 180^2 x 96 128 / 152
    if (MODE == 0 && partials && (size_t)L.nx * L.ny > 28672 && (L.nz < 64 || L.nz > 128)) return -1;
    switch (panel_chunk_planes(L.nz)) {
        case 4: return run_panel_chunk<MODE, 4>(L, coef, u, f, out, fc, partials, done, s);
        case 8: return run_panel_chunk<MODE, 8>(L, coef, u, f, out, fc, partials, done, s);
        default: return run_panel_chunk<MODE, 16>(L, coef, u, f, out, fc, partials, done, s);
    }
}

template <int MODE, class TO>
static int panel_point(const PanelLv& L, const double* u, const double* f, TO* out, double* partials, const int* done,
                       cudaStream_t s) {
    dim3 g = panel_grid(L.nx, L.ny);
    int pz = point_planes(L.nx, L.ny, L.nz, (int)(g.x * g.y));
    if (partials) {
        // as many slabs of planes as max_partials leaves room for, of four planes or more unless 256 blocks do with fewer (32 x
        // 28 x 3 5.4 us with one, 6.4 with three), and below the size that takes 16 at most MIN_PARTIALS blocks (one block
        // adds the sums up: 138 x 446 x 36 62 us with 5040 of them, 58 with 560; fewer leave the last round of blocks short: 134
        // x 258 x 130 119 us with 975, 109 with 1300)
        const int blocks = (int)(g.x * g.y), least = blocks * ((L.nz + pz - 1) / pz) <= 256 ? pz : std::max(pz, 4);
        int slabs = std::min((L.nz + least - 1) / least, std::max(max_partials(L.nx, L.ny), MIN_PARTIALS) / blocks);
        if ((size_t)L.nx * L.ny <= 65536) slabs = std::min(slabs, MIN_PARTIALS / blocks);
        slabs = std::max(slabs, 1);
        pz = (L.nz + slabs - 1) / slabs;
    }
    g.z = (L.nz + pz - 1) / pz;
    k_panel_point<MODE, TO><<<g, dim3(32, 4), 0, s>>>(L, u, f, out, partials, done, pz);
    note_launch();
    return (int)(g.x * g.y * g.z);
}

template <class T>
int launch_panel_sweep(int mode, const PanelLvT<T>& L, double coef, const T* u, const T* f, T* out, double* partials,
                       const int* done, cudaStream_t s) {
    const dim3 g = panel_grid(L.nx, L.ny), b(32, 4);
    const T c = (T)coef;
    if constexpr (sizeof(T) == 8) {
        if (mode == PANEL_RESIDUAL) return panel_point<1, double>(L, u, f, out, partials, done, s);
        if (mode == PANEL_APPLY) return panel_point<3, double>(L, u, f, out, nullptr, done, s);
        const int nb = mode == PANEL_SMOOTH ? panel_chunk<0>(L, coef, u, f, out, nullptr, partials, done, s)
                                            : panel_chunk<2>(L, coef, u, f, out, nullptr, nullptr, done, s);
        if (nb >= 0) return nb;
    }
    if (mode == PANEL_LINESOLVE) k_panel_sweep<2, T, false><<<g, b, 0, s>>>(L, c, u, f, out, nullptr, done);
    else if (mode == PANEL_SMOOTH && partials) k_panel_sweep<0, T, true><<<g, b, 0, s>>>(L, c, u, f, out, partials, done);
    else if (mode == PANEL_SMOOTH) k_panel_sweep<0, T, false><<<g, b, 0, s>>>(L, c, u, f, out, nullptr, done);
    else if constexpr (sizeof(T) == 4) k_panel_sweep<1, T, true><<<g, b, 0, s>>>(L, c, u, f, out, partials, done);
    note_launch();
    return (int)(g.x * g.y);
}

int launch_panel_residual_to_f32(const PanelLv& L, const double* u, const double* f, float* r, double* partials,
                                 const int* done, cudaStream_t s) {
    return panel_point<1, float>(L, u, f, r, partials, done, s);
}

template <class T>
void launch_panel_restrict_smooth(const PanelLvT<T>& Lc, double rho, const T* rf, T* fc, T* uc, const int* done,
                                  cudaStream_t s) {
    if constexpr (sizeof(T) == 8)
        if (panel_chunk<4>(Lc, rho, rf, nullptr, uc, fc, nullptr, done, s) >= 0) return;
    k_panel_restrict_smooth<T><<<panel_grid(Lc.nx, Lc.ny), dim3(32, 4), 0, s>>>(Lc, (T)rho, rf, fc, uc, done);
    note_launch();
}

template <class T>
void launch_panel_prolongate(int nxc, int nyc, int nz, const T* uc, T* uf, const int* done, cudaStream_t s) {
    dim3 g = panel_grid(2 * nxc, nyc);
    const int pz = point_planes(2 * nxc, 2 * nyc, nz, (int)(g.x * g.y), 2);
    g.z = (nz + pz - 1) / pz;
    k_panel_prolongate<T><<<g, dim3(32, 4), 0, s>>>(nxc, nyc, nz, uc, uf, done, pz);
    note_launch();
}

#define TPMG_PANEL_INST(T)                                                                                       \
    template int launch_panel_sweep<T>(int, const PanelLvT<T>&, double, const T*, const T*, T*, double*, const int*, \
                                       cudaStream_t);                                                            \
    template void launch_panel_restrict_smooth<T>(const PanelLvT<T>&, double, const T*, T*, T*, const int*,        \
                                                  cudaStream_t);                                                  \
    template void launch_panel_prolongate<T>(int, int, int, const T*, T*, const int*, cudaStream_t);
TPMG_PANEL_INST(double)
TPMG_PANEL_INST(float)

}  // namespace tpmg
