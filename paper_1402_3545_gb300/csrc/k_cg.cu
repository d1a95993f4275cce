// k_cg.cu -- the two fused kernels of the line-preconditioned CG iteration (Sec. 3.1, kernel list
// "Conjugate Gradient"), with the BLAS-1 updates and the dot products folded into the sweeps.
//
// Fused SpMV (iteration j, scalars of iteration j-1):
//   u <- u + alpha_{j-1} p ; p <- z + beta_{j-1} p ; q <- A z + beta_{j-1} q ; sigma = <p, q>
// which uses A p_j = A z_j + beta_{j-1} A p_{j-1}, so the stencil is applied to z and the
// solution update lags one iteration behind (finished by k_cg_finish).
// Fused Tridiag:
//   r <- r - alpha_j q ; z <- M^{-1} r ; <r, r> ; <r, z>
// One thread owns one vertical column; the sums are reduced per block and summed in a fixed order
// by the finalize kernels (k_util.cu), which also compute alpha and beta on the device.
#include <algorithm>

#include "kernels.cuh"
#include "sweep_x2.cuh"

namespace tpmg {

static constexpr int TX = 32;
__device__ __forceinline__ int wrapc(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <class P>
__global__ void __launch_bounds__(256) k_cg_spmv(Lv<P> L, const Scalars* __restrict__ sc,
                                                 typename P::S* __restrict__ u,
                                                 typename P::S* __restrict__ p,
                                                 const typename P::S* __restrict__ z,
                                                 typename P::S* __restrict__ q, double* partials) {
    typedef typename P::R R;
    if (*(volatile const int*)&sc->done) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    const bool act = i < L.nx && j < L.ny;
    typename P::Acc acc = 0, cmp = 0;
    if (act) {
        const size_t pl = (size_t)L.nx * L.ny, c = (size_t)j * L.nx + i;
        const size_t cw = (size_t)j * L.nx + wrapc(i - 1, L.nx), ce = (size_t)j * L.nx + wrapc(i + 1, L.nx);
        const size_t cs = (size_t)wrapc(j - 1, L.ny) * L.nx + i, cn = (size_t)wrapc(j + 1, L.ny) * L.nx + i;
        const R alpha = P::cst(sc->alpha), beta = P::cst(sc->beta);
        const R cx = P::cst(L.cx), cy = P::cst(L.cy), vv = P::ld(L.v, c);
        const R dh = P::cst(1.0 + 2.0 * L.cx + 2.0 * L.cy);
        const R dh1 = P::add(dh, vv), dh2 = P::add(dh1, vv);
        R zm = P::zero(), zc = P::ld(z, c);
        for (int k = 0; k < L.nz; ++k) {
            const size_t b = (size_t)k * pl, id = b + c;
            R zp = (k + 1 < L.nz) ? P::ld(z, b + pl + c) : P::zero();
            R hx = P::add(P::ld(z, b + cw), P::ld(z, b + ce));
            R hy = P::add(P::ld(z, b + cs), P::ld(z, b + cn));
            R diag = (L.nz == 1) ? dh : ((k == 0 || k == L.nz - 1) ? dh1 : dh2);
            R az = P::mul(diag, zc);
            az = P::sub(az, P::mul(cx, hx));
            az = P::sub(az, P::mul(cy, hy));
            az = P::sub(az, P::mul(vv, P::add(zm, zp)));
            R pold = P::ld_plain(p, id);
            P::st(u, id, P::add(P::ld_plain(u, id), P::mul(alpha, pold)));
            R pn = P::add(zc, P::mul(beta, pold));
            R qn = P::add(az, P::mul(beta, P::ld_plain(q, id)));
            P::st(p, id, pn);
            P::st(q, id, qn);
            P::acc_dot(acc, cmp, pn, qn);
            zm = zc;
            zc = zp;
        }
    }
    double s = block_sum(P::acc_get(acc, cmp));
    if (threadIdx.x == 0 && threadIdx.y == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// The fused SpMV with two x-adjacent columns per thread and SPMV_PZ planes per block: the vertical neighbours
// stay in registers, the x neighbours come from the adjacent lanes, and a plane's six 16-byte loads (DW; 8 bytes
// in FP32) are in flight together. 512^2 x 128 double-word 372 us (seven fields, 277 at the copy rate): DRAM 0.61 busy with
// a quarter of the warps (114 registers); 390 with a thread per pair of cells, whose 64-bit divisions for the
// cell's indices and five stencil loads it does without. Requires nx even; ALIGNED: pair-aligned fields.
constexpr int SPMV_PZ = 16, SPMV_TY = 8;
template <class P, bool ALIGNED>
struct CgPair {
    typedef typename P::S S;
    typename P::R a, b;
    __device__ __forceinline__ void ldg(const S* p) {
        if constexpr (!ALIGNED) {
            a = P::ld(p, 0);
            b = P::ld(p, 1);
        } else if constexpr (sizeof(S) == 8) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(p));
            get(reinterpret_cast<const S*>(&t));
        } else {
            const float2 t = __ldg(reinterpret_cast<const float2*>(p));
            get(reinterpret_cast<const S*>(&t));
        }
    }
    __device__ __forceinline__ void ld(const S* p) {  // a field that is written too
        if constexpr (!ALIGNED) {
            get(p);
        } else if constexpr (sizeof(S) == 8) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            get(reinterpret_cast<const S*>(&t));
        } else {
            const float2 t = *reinterpret_cast<const float2*>(p);
            get(reinterpret_cast<const S*>(&t));
        }
    }
    __device__ __forceinline__ void get(const S* q) {
        a = P::ld_plain(q, 0);
        b = P::ld_plain(q, 1);
    }
    __device__ __forceinline__ void st(S* p) const {
        if constexpr (!ALIGNED) {
            P::st(p, 0, a);
            P::st(p, 1, b);
        } else if constexpr (sizeof(S) == 8) {
            float4 t;
            P::st(reinterpret_cast<S*>(&t), 0, a);
            P::st(reinterpret_cast<S*>(&t), 1, b);
            *reinterpret_cast<float4*>(p) = t;
        } else {
            float2 t;
            P::st(reinterpret_cast<S*>(&t), 0, a);
            P::st(reinterpret_cast<S*>(&t), 1, b);
            *reinterpret_cast<float2*>(p) = t;
        }
    }
    __device__ __forceinline__ void zero() { a = b = P::zero(); }
};
__device__ __forceinline__ float lane_up(float x) { return __shfl_up_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ float lane_dn(float x) { return __shfl_down_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ dw lane_up(dw x) { return dw{lane_up(x.hi), lane_up(x.lo)}; }
__device__ __forceinline__ dw lane_dn(dw x) { return dw{lane_dn(x.hi), lane_dn(x.lo)}; }

// FOLD: the block's w < 32 pairs of SPMV_TY rows lie behind one another in its threads, a warp holds the end of one
// row and the start of the next; else w = 32, a row per warp
template <class P, bool ALIGNED, bool FOLD>
__global__ void __launch_bounds__(32 * SPMV_TY) k_cg_spmv_march(Lv<P> L, SweepK<P> K, const Scalars* __restrict__ sc,
                                                                typename P::S* __restrict__ u,
                                                                typename P::S* __restrict__ p,
                                                                const typename P::S* __restrict__ z,
                                                                typename P::S* __restrict__ q, double* partials, int pz,
                                                                int w) {
    typedef typename P::R R;
    typedef CgPair<P, ALIGNED> V;
    if (*(volatile const int*)&sc->done) return;
    const int nx = L.nx, ny = L.ny, nz = L.nz, lane = FOLD ? threadIdx.x & 31 : threadIdx.x;
    const int jt = FOLD ? threadIdx.x / w : threadIdx.y, it = FOLD ? threadIdx.x - jt * w : lane;
    const int i = 2 * (blockIdx.x * (FOLD ? w : 32) + it), j = blockIdx.y * SPMV_TY + jt;
    const int k0 = blockIdx.z * pz, k1 = k0 + pz < nz ? k0 + pz : nz;
    const size_t pl = (size_t)nx * ny;
    const R alpha = P::cst(sc->alpha), beta = P::cst(sc->beta);
    typename P::Acc acc = 0, cmp = 0;
    if (FOLD || j < ny) {  // (else a whole warp: one row)
        const bool act = i < nx && (!FOLD || (jt < SPMV_TY && j < ny));
        const int ii = i < nx ? i : nx - 2, jj = !FOLD || j < ny ? j : ny - 1;  // lanes beyond repeat the last pair, store nothing
        const size_t row = (size_t)jj * nx, c = row + ii, b0 = (size_t)k0 * pl;
        const size_t rs = (size_t)wrapc(jj - 1, ny) * nx + ii, rn = (size_t)wrapc(jj + 1, ny) * nx + ii;
        // the columns beyond the ends of the warp, the block's rows and the grid's: every lane loads one on either side,
        // those that need none the warp's first or last lane's (one sector a row)
        const bool lw = lane == 0 || (FOLD && it == 0), le = lane == 31 || i + 2 >= nx || (FOLD && it == w - 1);
        size_t cw, ce;
        if (FOLD) {
            cw = row + wrapc(ii - 1, nx);
            ce = row + (ii + 2 < nx ? ii + 2 : 0);
            const size_t first = __shfl_sync(0xffffffffu, cw, 0), last = __shfl_sync(0xffffffffu, ce, 31);
            if (!lw) cw = first;
            if (!le) ce = last;
        } else {
            const int iw = i - 2 * lane;
            cw = row + wrapc(iw - 1, nx);
            ce = row + (iw + 64 < nx ? iw + 64 : 0);
        }
        const R v0 = P::ld(L.v, c), v1 = P::ld(L.v, c + 1);
        const R d1a = P::add(K.dh, v0), d1b = P::add(K.dh, v1), d2a = P::add(d1a, v0), d2b = P::add(d1b, v1);
        const bool iso = K.iso != 0;
        V zm, zc;
        zm.zero();
        zc.ldg(z + b0 + c);
        if (k0 > 0) zm.ldg(z + b0 - pl + c);
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            const size_t b = (size_t)k * pl, id = b + c;
            V zp, zs, zn, po, qo, uo;
            zp.ldg(z + (k + 1 < nz ? id + pl : id));
            zs.ldg(z + b + rs);
            zn.ldg(z + b + rn);
            po.ld(p + id);
            qo.ld(q + id);
            uo.ld(u + id);
            const R zl = P::ld(z, b + cw), zr = P::ld(z, b + ce);
            R zw = lane_up(zc.b), ze = lane_dn(zc.a);
            if (lw) zw = zl;
            if (le) ze = zr;
            if (k + 1 == nz) zp.zero();
            const bool end = k == 0 || k == nz - 1;
            const R da = nz == 1 ? K.dh : (end ? d1a : d2a), db = nz == 1 ? K.dh : (end ? d1b : d2b);
            // A z = -(f - A z) with f = 0: the sweep residual of a zero right-hand side, negated
            const R az0 = P::neg(sweep_residual<P>(P::zero(), da, zc.a, zw, zc.b, zs.a, zn.a, zm.a, zp.a, K.cx, K.cy, v0, iso));
            const R az1 = P::neg(sweep_residual<P>(P::zero(), db, zc.b, zc.a, ze, zs.b, zn.b, zm.b, zp.b, K.cx, K.cy, v1, iso));
            V un, pn, qn;
            un.a = P::fma(alpha, po.a, uo.a);
            un.b = P::fma(alpha, po.b, uo.b);
            pn.a = P::fma(beta, po.a, zc.a);
            pn.b = P::fma(beta, po.b, zc.b);
            qn.a = P::fma(beta, qo.a, az0);
            qn.b = P::fma(beta, qo.b, az1);
            if (act) {
                un.st(u + id);
                pn.st(p + id);
                qn.st(q + id);
                P::acc_dot(acc, cmp, pn.a, qn.a);
                P::acc_dot(acc, cmp, pn.b, qn.b);
            }
            zm = zc;
            zc = zp;
        }
    }
    const double s = block_sum(P::acc_get(acc, cmp));
    if (threadIdx.x == 0 && threadIdx.y == 0)
        partials[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
}

template <class P>
__global__ void __launch_bounds__(256) k_cg_tridiag(Lv<P> L, const Scalars* __restrict__ sc,
                                                    typename P::S* __restrict__ r,
                                                    const typename P::S* __restrict__ q,
                                                    typename P::S* __restrict__ z, double* partials) {
    typedef typename P::R R;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (*(volatile const int*)&sc->done) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
    const bool act = i < L.nx && j < L.ny;
    typename P::Acc arr = 0, crr = 0, arz = 0, crz = 0;
    if (act) {
        const int nt = blockDim.x * blockDim.y, tid = threadIdx.y * blockDim.x + threadIdx.x;
        R* dp = reinterpret_cast<R*>(smem_raw);
        R* w = dp + (size_t)L.nz * nt;
        const size_t pl = (size_t)L.nx * L.ny, c = (size_t)j * L.nx + i;
        const R alpha = P::cst(sc->alpha);
        const R vv = P::ld(L.v, c), vv2 = P::mul(vv, vv);
        const R dh = P::cst(1.0 + 2.0 * L.cx + 2.0 * L.cy);
        const R dh1 = P::add(dh, vv), dh2 = P::add(dh1, vv);
        R inv_prev = P::zero(), d_prev = P::zero();
        for (int k = 0; k < L.nz; ++k) {
            const size_t id = (size_t)k * pl + c;
            R rn = P::sub(P::ld_plain(r, id), P::mul(alpha, P::ld(q, id)));
            P::st(r, id, rn);
            P::acc_dot(arr, crr, rn, rn);
            R diag = (L.nz == 1) ? dh : ((k == 0 || k == L.nz - 1) ? dh1 : dh2);
            R m = (k == 0) ? diag : P::sub(diag, P::mul(vv2, inv_prev));
            R inv = P::rcp(m);
            R d = P::mul(P::add(rn, P::mul(vv, d_prev)), inv);
            dp[(size_t)k * nt + tid] = d;
            w[(size_t)k * nt + tid] = P::mul(vv, inv);
            inv_prev = inv;
            d_prev = d;
        }
        R xn = P::zero();
        for (int k = L.nz - 1; k >= 0; --k) {
            const size_t id = (size_t)k * pl + c;
            xn = P::add(dp[(size_t)k * nt + tid], P::mul(w[(size_t)k * nt + tid], xn));
            P::st(z, id, xn);
            P::acc_dot(arz, crz, P::ld_plain(r, id), xn);
        }
    }
    double s1 = block_sum(P::acc_get(arr, crr));
    double s2 = block_sum(P::acc_get(arz, crz));
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const int b = blockIdx.y * gridDim.x + blockIdx.x, nb = gridDim.x * gridDim.y;
        partials[b] = s1;
        partials[nb + b] = s2;
    }
}

// The same fused Tridiag with the level's precomputed Thomas factors (1/m_k, v/m_k) and the
// forward-eliminated values on a per-block stack in the global scratch (L.gstack): a persistent
// grid of a few blocks per SM loops over tiles of 32 x 4 columns. No reciprocal per cell and no
// shared-memory stack, so the SM holds as many warps as its registers allow.
template <class P>
__global__ void __launch_bounds__(128) k_cg_tridiag_gs(Lv<P> L, const Scalars* __restrict__ sc,
                                                       typename P::S* __restrict__ r,
                                                       const typename P::S* __restrict__ q,
                                                       typename P::S* __restrict__ z, double* partials) {
    typedef typename P::R R;
    typedef typename P::S S;
    if (*(volatile const int*)&sc->done) return;
    const int nx = L.nx, ny = L.ny, nz = L.nz;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int tiles_x = (nx + 31) / 32, ntiles = tiles_x * ((ny + 3) / 4);
    const size_t pl = (size_t)nx * ny;
    const bool percol = L.fac_percol != 0;
    S* gst = reinterpret_cast<S*>(L.gstack) + (size_t)blockIdx.x * nz * 128;
    const R nalpha = P::neg(P::cst(sc->alpha));
    typename P::Acc arr = 0, crr = 0, arz = 0, crz = 0;
    // q, the factors and z stream through L2 evict-first; the stack is stored evict-last and each
    // of its lines is dropped once read (see the persistent Smooth)
    const unsigned long long pol_first = l2_evict_first(), pol_last = l2_evict_last();
    constexpr int LANES_PER_LINE = 128 / (int)sizeof(S);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int i = (tile % tiles_x) * 32 + threadIdx.x, j = (tile / tiles_x) * 4 + threadIdx.y;
        const bool active = i < nx && j < ny;
        const size_t c = (size_t)j * nx + i;
        const R vv = active ? P::ld(L.v, c) : P::zero();
        R d_prev = P::zero();
        for (int k = 0; k < nz && active; ++k) {
            const size_t id = (size_t)k * pl + c;
            const R rn = P::fma(nalpha, ld_pol(q + id, pol_first), P::ld_plain(r, id));
            P::st(r, id, rn);
            P::acc_dot(arr, crr, rn, rn);
            const R inv = percol ? ld_pol(L.finv + id, pol_first) : P::ld(L.finv, k);
            d_prev = P::mul(P::fma(vv, d_prev, rn), inv);
            st_pol(gst + (size_t)k * 128 + tid, d_prev, pol_last);
        }
        R xn = P::zero();
        for (int k = nz - 1; k >= 0; --k) {
            const size_t id = (size_t)k * pl + c;
            if (active) {
                const R w = percol ? ld_pol(L.fw + id, pol_first) : P::ld(L.fw, k);
                xn = P::fma(w, xn, P::ld_plain(gst, (size_t)k * 128 + tid));
                st_pol(z + id, xn, pol_first);
                P::acc_dot(arz, crz, P::ld_plain(r, id), xn);
            }
            // every lane of the warp has consumed its stack value of plane k: drop the dead lines
            __syncwarp();
            if (tid % LANES_PER_LINE == 0) l2_discard(gst + (size_t)k * 128 + tid);
        }
    }
    double s1 = block_sum(P::acc_get(arr, crr));
    double s2 = block_sum(P::acc_get(arz, crz));
    if (tid == 0) {
        partials[blockIdx.x] = s1;
        partials[gridDim.x + blockIdx.x] = s2;
    }
}

// The fused Tridiag on two columns per thread, plane-pipelined like the two-column Smooth
// (sweep_x2.cuh): each plane's r, q and (where the elimination has not converged) 1/m_k pairs
// arrive by cp.async PD planes ahead; the forward-eliminated values go to the block's scratch slot
// (evict-last, each line dropped from L2 once read back). <r, z> is taken in the forward sweep: with
// the column block M = U^T D U (D = diag(m_k), U unit upper bidiagonal), the elimination gives
// yh = U^{-T} r (yh_k = r_k + v d'_{k-1}) and d'_k = yh_k / m_k, so <r, M^{-1} r> = sum_k yh_k d'_k,
// a sum of non-negative terms, and the back substitution does not read r again.
// Tiles of 64 x TY columns; requires nx % 64 == 0, ny % TY == 0, 16-byte aligned fields.
template <class P, int TY, int PD>
__global__ void __launch_bounds__(32 * TY) k_cg_tridiag_x2(Lv<P> L, const Scalars* __restrict__ sc,
                                                           typename P::S* __restrict__ r,
                                                           const typename P::S* __restrict__ q,
                                                           typename P::S* __restrict__ z, double* partials) {
    typedef typename P::S S;
    typedef typename P::R R;
    constexpr int NT = 32 * TY, SL = 2 * NT;  // values per ring slot and array
    constexpr int PB = 2 * (int)sizeof(S);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (*(volatile const int*)&sc->done) return;
    const int nx = L.nx, ny = L.ny, nz = L.nz, tid = threadIdx.y * 32 + threadIdx.x;
    const size_t pl = (size_t)nx * ny;
    const int tiles_x = nx / 64, ntiles = tiles_x * (ny / TY);
    const bool percol = L.fac_percol != 0;
    const int k0 = L.fac_k0;
    S* ringR = reinterpret_cast<S*>(smem_raw);
    S* ringQ = ringR + PD * SL;
    S* ringI = ringQ + PD * SL;
    S* gst = reinterpret_cast<S*>(L.gstack) + (size_t)blockIdx.x * nz * SL;
    const R nalpha = P::neg(P::cst(sc->alpha));
    const unsigned long long pol_first = l2_evict_first(), pol_last = l2_evict_last();
    typename P::Acc arr = 0, crr = 0, arz = 0, crz = 0;
    const R vzero = P::zero();
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int i0 = (tile % tiles_x) * 64, j0 = (tile / tiles_x) * TY;
        const size_t c = (size_t)(j0 + threadIdx.y) * nx + i0 + 2 * threadIdx.x;
        __syncthreads();  // the previous tile's rings are no longer read
        auto issue_plane = [&](int k, int slot) {
            if (k < nz) {
                const size_t id = (size_t)k * pl + c;
                cp_async<PB>(&ringR[slot * SL + 2 * tid], r + id);
                cp_async_pol<PB>(&ringQ[slot * SL + 2 * tid], q + id, pol_first);
                if (percol && !(k >= k0 && k <= nz - 2))
                    cp_async_pol<PB>(&ringI[slot * SL + 2 * tid], L.finv + id, pol_first);
            }
            cp_commit();
        };
        for (int sl = 0; sl < PD; ++sl) issue_plane(sl, sl);
        const R v0 = P::ld(L.v, c), v1 = P::ld(L.v, c + 1);
        R ci0 = vzero, ci1 = vzero, cw0 = vzero, cw1 = vzero;
        if (percol && k0 <= nz - 2) {
            const size_t rr = (size_t)(nz - 2) * pl + c;
            ci0 = P::ld(L.finv, rr);
            ci1 = P::ld(L.finv, rr + 1);
            cw0 = P::ld(L.fw, rr);
            cw1 = P::ld(L.fw, rr + 1);
        }
        R dp0 = vzero, dp1 = vzero;
        int slot = 0;
        for (int k = 0; k < nz; ++k) {
            cp_wait<PD - 1>();  // this thread's copies of plane k
            const int o = slot * SL + 2 * tid;
            const R rn0 = P::fma(nalpha, P::ld_plain(ringQ, o), P::ld_plain(ringR, o));
            const R rn1 = P::fma(nalpha, P::ld_plain(ringQ, o + 1), P::ld_plain(ringR, o + 1));
            const size_t id = (size_t)k * pl + c;
            st_pair_pol(r + id, rn0, rn1, pol_first);
            P::acc_dot(arr, crr, rn0, rn0);
            P::acc_dot(arr, crr, rn1, rn1);
            R i0v, i1v;
            if (!percol) {
                i0v = i1v = P::ld(L.finv, k);
            } else if (k >= k0 && k <= nz - 2) {
                i0v = ci0;
                i1v = ci1;
            } else {
                i0v = P::ld_plain(ringI, o);
                i1v = P::ld_plain(ringI, o + 1);
            }
            const R yh0 = P::fma(v0, dp0, rn0), yh1 = P::fma(v1, dp1, rn1);
            dp0 = P::mul(yh0, i0v);
            dp1 = P::mul(yh1, i1v);
            P::acc_dot(arz, crz, yh0, dp0);
            P::acc_dot(arz, crz, yh1, dp1);
            st_pair_pol(gst + ((size_t)k * NT + tid) * 2, dp0, dp1, pol_last);
            issue_plane(k + PD, slot);
            slot = (slot + 1 == PD) ? 0 : slot + 1;
        }
        cp_wait<0>();
        __syncthreads();  // the backward ring reuses the forward ring's shared memory
        S* bW = reinterpret_cast<S*>(smem_raw);
        S* bD = bW + PD * SL;
        auto issue_back = [&](int k, int s2) {
            if (k >= 0) {
                if (percol && !(k >= k0 && k <= nz - 2))
                    cp_async_pol<PB>(&bW[s2 * SL + 2 * tid], L.fw + (size_t)k * pl + c, pol_first);
                cp_async<PB>(&bD[s2 * SL + 2 * tid], gst + ((size_t)k * NT + tid) * 2);
            }
            cp_commit();
        };
        for (int sl = 0; sl < PD; ++sl) issue_back(nz - 1 - sl, sl);
        R x0 = vzero, x1 = vzero;
        slot = 0;
        for (int k = nz - 1; k >= 0; --k) {
            cp_wait<PD - 1>();
            {
                // plane k of the stack has landed for every lane of the warp: its lines are dead
                constexpr int LANES_PER_LINE = 128 / PB;
                __syncwarp();
                if (tid % LANES_PER_LINE == 0) l2_discard(gst + ((size_t)k * NT + tid) * 2);
            }
            const int o = slot * SL + 2 * tid;
            R w0, w1;
            if (!percol) {
                w0 = w1 = P::ld(L.fw, k);
            } else if (k >= k0 && k <= nz - 2) {
                w0 = cw0;
                w1 = cw1;
            } else {
                w0 = P::ld_plain(bW, o);
                w1 = P::ld_plain(bW, o + 1);
            }
            x0 = P::fma(w0, x0, P::ld_plain(bD, o));
            x1 = P::fma(w1, x1, P::ld_plain(bD, o + 1));
            st_pair_pol(z + (size_t)k * pl + c, x0, x1, pol_first);
            issue_back(k - PD, slot);
            slot = (slot + 1 == PD) ? 0 : slot + 1;
        }
        cp_wait<0>();
    }
    const double s1 = block_sum(P::acc_get(arr, crr));
    const double s2 = block_sum(P::acc_get(arz, crz));
    if (tid == 0) {
        partials[blockIdx.x] = s1;
        partials[gridDim.x + blockIdx.x] = s2;
    }
}

static constexpr int CGX_TY = 2, CGX_PD = 4;
template <class P>
static bool cg_x2_fits(const Lv<P>& L) {
    return P::id != 0 && L.gstack && L.finv && L.fw && L.nx % 64 == 0 && L.ny % CGX_TY == 0;
}
template <class P>
static size_t cg_x2_smem() {
    return (size_t)CGX_PD * 3 * 2 * 32 * CGX_TY * sizeof(typename P::S);
}
template <class P>
static int cg_x2_blocks(const Lv<P>& L) {
    static int per_sm = 0, nsm = 0;
    if (per_sm == 0) {
        auto kern = k_cg_tridiag_x2<P, CGX_TY, CGX_PD>;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cg_x2_smem<P>());
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * CGX_TY, cg_x2_smem<P>());
        if (per_sm > 10) per_sm = 10;
        if (per_sm < 1) per_sm = 1;
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    }
    int nb = nsm * per_sm;
    // the scratch slots: 64 TY columns per block out of gstack_bytes
    const int slots = nsm * GS_BLOCKS_PER_SM * GS_MAX_NT / (2 * 32 * CGX_TY);
    if (nb > slots) nb = slots;
    const int ntiles = (L.nx / 64) * (L.ny / CGX_TY);
    return nb < ntiles ? nb : ntiles;
}

// u <- u + alpha p : the lagged solution update after the last iteration.
template <class P>
__global__ void k_cg_finish(size_t n, const Scalars* __restrict__ sc, typename P::S* __restrict__ u,
                            const typename P::S* __restrict__ p) {
    const typename P::R alpha = P::cst(sc->alpha);
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        P::st(u, t, P::add(P::ld_plain(u, t), P::mul(alpha, P::ld(p, t))));
}

// the marching SpMV for the FP32-pipe policies (native FP64 keeps the column kernel, bound by its pipe)
template <class P>
static dim3 spmv_march_grid(const Lv<P>& L, int& pz, int& w) {
    // a row's pairs to its warps; folded, in equal parts, where that leaves a quarter of the lanes or more without a pair
    // (FP32 78 x 628 x 203 107 us, 70 folded; 34 x 700 x 16 15.5, 9.7)
    const int pairs = L.nx / 2, parts = (pairs + 31) / 32;
    dim3 g(parts, (L.ny + SPMV_TY - 1) / SPMV_TY);
    // SPMV_PZ planes per block, fewer where that leaves a quarter of the SMs without one (with 16 everywhere FP32 32 x 42 x 66
    // took 11.3 us, with the two scalar kernels of a call; 8.8 with a thread per pair of cells; where the SMs are full, more
    // and shorter slabs cost: double-word 128^2 x 128 80 us with ten, 73 with eight); one partial sum per block: as many
    // slabs of planes as max_partials leaves room for
    const int cols = (int)(g.x * g.y), room = max_partials(L.nx, L.ny) / cols;
    int nzs = (L.nz + SPMV_PZ - 1) / SPMV_PZ;
    bool fold = 4 * pairs <= 3 * 32 * parts;
    int from = 114, upto = 152;
    if (P::id == 1 && fold) {
        // FP32's folded rows wait longer per plane: fewer planes still, three blocks an SM where there would not be two (88 x
        // 180 x 45 16.7 us with one, 11.2 with three, 11.9 a row per warp); a row per warp between (88 x 180 x 128 19.0 us, 16.3)
        from = 2 * 152;
        upto = 3 * 152;
        fold = parts == 1 || cols * nzs < from || cols * nzs >= upto;
    }
    w = fold ? (pairs + parts - 1) / parts : 32;
    if (cols * nzs < from) nzs = std::max(nzs, std::min(L.nz, (upto + cols - 1) / cols));
    nzs = std::min(nzs, std::max(room, 1));
    pz = (L.nz + nzs - 1) / nzs;
    g.z = (L.nz + pz - 1) / pz;
    return g;
}
template <class P>
int cg_spmv_blocks(const Lv<P>& L) {
    if (L.nx % 2 == 0 && P::id != 0) {
        int pz, w;
        const dim3 g = spmv_march_grid(L, pz, w);
        return (int)(g.x * g.y * g.z);
    }
    return sweep_shape(L.nx, L.ny, L.nz, sizeof(typename P::R), false).nblocks();
}
template <class P>
int launch_cg_spmv(const Lv<P>& L, const Scalars* sc, typename P::S* u, typename P::S* p,
                   const typename P::S* z, typename P::S* q, double* partials, cudaStream_t s) {
    if constexpr (P::id != 0)
        if (L.nx % 2 == 0) {
            int pz, w;
            const dim3 g = spmv_march_grid(L, pz, w);
            const SweepK<P> K = sweep_k<P>(L.cx, L.cy, 1.0);
            const bool al = (((uintptr_t)u | (uintptr_t)p | (uintptr_t)z | (uintptr_t)q) & (2 * sizeof(typename P::S) - 1)) == 0;
            auto run = [&](auto kern) {
                const dim3 b = w == 32 ? dim3(32, SPMV_TY) : dim3((w * SPMV_TY + 31) / 32 * 32);
                kern<<<g, b, 0, s>>>(L, K, sc, u, p, z, q, partials, pz, w);
            };
            if (w == 32) al ? run(k_cg_spmv_march<P, true, false>) : run(k_cg_spmv_march<P, false, false>);
            else al ? run(k_cg_spmv_march<P, true, true>) : run(k_cg_spmv_march<P, false, true>);
            note_launch();
            return (int)(g.x * g.y * g.z);
        }
    Shape sh = sweep_shape(L.nx, L.ny, L.nz, sizeof(typename P::R), false);
    k_cg_spmv<P><<<sh.grid, sh.block, 0, s>>>(L, sc, u, p, z, q, partials);
    note_launch();
    return sh.nblocks();
}
// blocks of the fused Tridiag (= partial sums per quantity); the persistent form when the level has
// its factors and the scratch
template <class P>
int cg_tridiag_blocks(const Lv<P>& L) {
    if constexpr (P::id != 0) {
        const int nb = cg_tile_blocks(L);
        if (nb >= 0) return nb;
    }
    if (cg_x2_fits(L)) return cg_x2_blocks(L);
    if (L.gstack && L.finv && L.fw) {
        static int per_sm = 0;
        if (per_sm == 0) {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cg_tridiag_gs<P>, 128, 0);
            if (per_sm > GS_BLOCKS_PER_SM) per_sm = GS_BLOCKS_PER_SM;
            if (per_sm < 1) per_sm = 1;
        }
        int nsm = 0, dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const int ntiles = ((L.nx + 31) / 32) * ((L.ny + 3) / 4);
        const int nb = nsm * per_sm;
        return nb < ntiles ? nb : ntiles;
    }
    return sweep_shape(L.nx, L.ny, L.nz, sizeof(typename P::R), true).nblocks();
}
template <class P>
int launch_cg_tridiag(const Lv<P>& L, const Scalars* sc, typename P::S* r, const typename P::S* q,
                      typename P::S* z, double* partials, cudaStream_t s) {
    if constexpr (P::id != 0)
        if ((((uintptr_t)r | (uintptr_t)q | (uintptr_t)z) & 15) == 0) {
            const int nb = launch_cg_tile(L, sc, r, q, z, partials, s);
            if (nb >= 0) return nb;
        }
    if (cg_x2_fits(L)) {
        const int nb = cg_x2_blocks(L);
        k_cg_tridiag_x2<P, CGX_TY, CGX_PD><<<nb, dim3(32, CGX_TY), cg_x2_smem<P>(), s>>>(L, sc, r, q, z, partials);
        note_launch();
        return nb;
    }
    if (L.gstack && L.finv && L.fw) {
        const int nb = cg_tridiag_blocks(L);
        k_cg_tridiag_gs<P><<<nb, dim3(32, 4), 0, s>>>(L, sc, r, q, z, partials);
        note_launch();
        return nb;
    }
    Shape sh = sweep_shape(L.nx, L.ny, L.nz, sizeof(typename P::R), true);
    if (sh.smem > 32 * 1024)
        cudaFuncSetAttribute(k_cg_tridiag<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh.smem);
    k_cg_tridiag<P><<<sh.grid, sh.block, sh.smem, s>>>(L, sc, r, q, z, partials);
    note_launch();
    return sh.nblocks();
}
template <class P>
void launch_cg_finish(size_t n, const Scalars* sc, typename P::S* u, const typename P::S* p,
                      cudaStream_t s) {
    size_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_cg_finish<P><<<(unsigned)blocks, 256, 0, s>>>(n, sc, u, p);
    note_launch();
}

#define TPMG_CG_INST(P)                                                                             \
    template int cg_spmv_blocks<P>(const Lv<P>&);                                                   \
    template int cg_tridiag_blocks<P>(const Lv<P>&);                                                \
    template int launch_cg_spmv<P>(const Lv<P>&, const Scalars*, P::S*, P::S*, const P::S*, P::S*,  \
                                   double*, cudaStream_t);                                         \
    template int launch_cg_tridiag<P>(const Lv<P>&, const Scalars*, P::S*, const P::S*, P::S*,      \
                                      double*, cudaStream_t);                                      \
    template void launch_cg_finish<P>(size_t, const Scalars*, P::S*, const P::S*, cudaStream_t);

TPMG_CG_INST(PolF64)
TPMG_CG_INST(PolF32)
TPMG_CG_INST(PolDW)

}  // namespace tpmg
