// restrict_tile.cuh -- Residual of a fine level and RestrictSmooth onto the coarse one in one pass
// (f_c = R (f - A u), u_c = rho M_c^{-1} f_c), on tiles of whole columns: the planes in parallel, only the
// coarse recurrences one plane after the other (as in sweep_tile.cuh, FP32 and double-word).
//
// A block owns 512 bytes of x-adjacent fine columns on two rows, that is one coarse row of half as many
// columns, over all planes; its shared memory holds the coarse right-hand sides (256 bytes per plane).
// Eight warps take contiguous ranges of planes; a lane forms the residuals of 16 bytes of columns on both
// rows (x neighbours by shuffles, the rows' vertical neighbours in registers, the rows above and below read
// again), restricts them and writes f_c. One warp then runs the coarse elimination and back substitution
// through shared memory. The plane-marching form (sweep_x2.cuh, MODE_RESTRICT) holds the two rows on two
// threads, one of which alone runs the coarse recurrence, plane by plane between two block barriers.
// The per-cell arithmetic and its order are the same, so the results are the same bits.
// Measured: FP32 1024 x 512 x 64 83 us (4.0 TB/s of algorithmic traffic; 134 plane-marching), 512^2 x 128 83
// (132), 256^2 x 128 17 (62); bound by the latency of the loads (six of 16 bytes per 16 cells; 119 registers leave a
// fifth of the warps, DRAM 0.51 busy). Levels of few planes leave the warps without work (launch_residual_restrict).
#pragma once
#include <type_traits>

#include "kernels.cuh"
#include "sweep_x2.cuh"

namespace tpmg {

namespace {

constexpr int RNT = 256, RNW = RNT / 32;

template <class P>
struct RVec {  // 16 bytes of adjacent fine columns
    typedef typename P::S S;
    typedef typename P::R R;
    static constexpr int N = 16 / (int)sizeof(S);
    R v[N];
    // RO: through the read-only cache, else (fields that this kernel itself writes) by ordinary loads
    template <bool RO>
    __device__ __forceinline__ void ldf(const S* p) {
        const float4 t = RO ? __ldg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
        const S* q = reinterpret_cast<const S*>(&t);
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = P::ld_plain(q, e);
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = P::zero();
    }
};
// H adjacent coarse columns (8 bytes: two FP32 or one double-word value)
template <class P, int H>
struct HVec {
    typedef typename P::S S;
    typename P::R v[H];
    static_assert(H * sizeof(S) == 8, "one 8-byte access");
    __device__ __forceinline__ void get(const S* p) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        const S* q = reinterpret_cast<const S*>(&t);
#pragma unroll
        for (int e = 0; e < H; ++e) v[e] = P::ld_plain(q, e);
    }
    __device__ __forceinline__ void put(S* p) const {
        float2 t;
        S* q = reinterpret_cast<S*>(&t);
#pragma unroll
        for (int e = 0; e < H; ++e) P::sts(q, e, v[e]);
        *reinterpret_cast<float2*>(p) = t;
    }
};
__device__ __forceinline__ float up1(float x) { return __shfl_up_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ float dn1(float x) { return __shfl_down_sync(0xffffffffu, x, 1); }
__device__ __forceinline__ dw up1(dw x) { return dw{up1(x.hi), up1(x.lo)}; }
__device__ __forceinline__ dw dn1(dw x) { return dw{dn1(x.hi), dn1(x.lo)}; }

}  // namespace

// One tile: fine columns bx * W .., rows 2 by and 2 by + 1.
// kw: planes of the coarse level whose factors are kept per column behind the nz planes of f_c (0 when its
// lambda^2 is constant: two tables of nz values)
template <class P, bool ISO, bool RO>
__device__ __forceinline__ void restrict_tile_body(const Lv<P>& L, const SweepK<P>& K, const XRestrict<P>& xr,
                                                   const typename P::S* u, const typename P::S* f, int kw, int bx, int by,
                                                   unsigned char* smem_raw) {
    typedef typename P::S S;
    typedef typename P::R R;
    typedef RVec<P> V;
    constexpr int N = V::N, H = N / 2, W = 32 * N, NC = 32 * H;  // H coarse columns per lane
    S* const Z = reinterpret_cast<S*>(smem_raw);
    const int nx = L.nx, ny = L.ny, nz = L.nz;
    S* const ZW = Z + (size_t)nz * NC;
    const Lv<P>& C = xr.Lc;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int i0 = bx * W, j0 = by * 2;
    const size_t pl = (size_t)nx * ny, plc = pl / 4;
    const size_t c = (size_t)j0 * nx + i0 + lane * N;                              // this lane's first fine column
    const size_t cc = (size_t)by * (nx / 2) + i0 / 2 + lane * H;           // ... and coarse column
    const int ch = (nz + RNW - 1) / RNW, klo = warp * ch, khi = klo + ch < nz ? klo + ch : nz;
    const bool percol = C.fac_percol != 0;

    // coarse factors: 1/m_k of the planes before the converged ones, or the tables
    if (percol) {
        for (int k = klo; k < khi && k < kw; ++k)
            cp_async<(int)sizeof(S) * H>(ZW + (size_t)k * NC + lane * H, C.finv + (size_t)k * plc + cc);
    } else {
        for (int k = tid; k < nz; k += RNT) {
            ZW[k] = C.finv[k];
            ZW[nz + k] = C.fw[k];
        }
    }
    cp_commit();

    // ---- residuals of both rows, restricted
    if (klo < khi) {
        const int js = j0 == 0 ? ny - 1 : j0 - 1, jn = j0 + 2 == ny ? 0 : j0 + 2;
        const bool hcol = lane == 0 || lane == 31;
        const int hi = lane == 0 ? (i0 == 0 ? nx - 1 : i0 - 1) : (i0 + W == nx ? 0 : i0 + W);
        const size_t p0 = (size_t)klo * pl;
        const S* pu = u + p0 + c;
        const S* pf = f + p0 + c;
        const S* ps = u + p0 + (size_t)js * nx + i0 + lane * N;
        const S* pn = u + p0 + (size_t)jn * nx + i0 + lane * N;
        const S* pe = u + p0 + (size_t)j0 * nx + hi;
        S* fc = xr.fc + (size_t)klo * plc + cc;
        S* z = Z + klo * NC + lane * H;
        const R cx = K.cx, cy = K.cy, dh = K.dh;
        V um[2], uc[2], vv[2], dg[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            um[r].zero();
            uc[r].template ldf<RO>(pu + r * nx);
            if (klo > 0) um[r].template ldf<RO>(pu + r * nx - pl);
#pragma unroll
            for (int q = 0; q < N; ++q) {
                vv[r].v[q] = P::ld(L.v, c + r * nx + q);
                dg[r].v[q] = P::add(P::add(dh, vv[r].v[q]), vv[r].v[q]);
            }
        }
        for (int k = klo; k < khi; ++k, z += NC) {
            const bool top = k + 1 == nz;
            V up[2], fk[2], hs, hn;
            R e[2] = {P::zero(), P::zero()};
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                up[r].template ldf<RO>(pu + r * nx + (top ? 0 : pl));
                fk[r].template ldf<RO>(pf + r * nx);
                if (hcol) e[r] = RO ? P::ld(pe + r * nx, 0) : P::ld_plain(pe + r * nx, 0);
            }
            hs.template ldf<RO>(ps);
            hn.template ldf<RO>(pn);
            pu += pl;
            pf += pl;
            ps += pl;
            pn += pl;
            pe += pl;
            if (top) {
                up[0].zero();
                up[1].zero();
            }
            const bool end = k == 0 || top;
            R res[2][N];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                R wl = up1(uc[r].v[N - 1]), el = dn1(uc[r].v[0]);
                if (lane == 0) wl = e[r];
                if (lane == 31) el = e[r];
                V d = dg[r];
                if (end) {
#pragma unroll
                    for (int q = 0; q < N; ++q) d.v[q] = nz == 1 ? dh : P::add(dh, vv[r].v[q]);
                }
#pragma unroll
                for (int q = 0; q < N; ++q) {
                    const R w = q == 0 ? wl : uc[r].v[q > 0 ? q - 1 : 0], ee = q == N - 1 ? el : uc[r].v[q < N - 1 ? q + 1 : q];
                    const R s = r == 0 ? hs.v[q] : uc[0].v[q], n = r == 0 ? uc[1].v[q] : hn.v[q];
                    res[r][q] = sweep_residual<P>(fk[r].v[q], d.v[q], uc[r].v[q], w, ee, s, n, um[r].v[q], up[r].v[q], cx, cy,
                                                  vv[r].v[q], ISO);
                }
            }
            HVec<P, H> fq;
#pragma unroll
            for (int q = 0; q < H; ++q)
                fq.v[q] = P::mul(xr.quarter, P::add(P::add(res[0][2 * q], res[0][2 * q + 1]),
                                                    P::add(res[1][2 * q], res[1][2 * q + 1])));
            fq.put(fc);
            fq.put(z);
            fc += plc;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                um[r] = uc[r];
                uc[r] = up[r];
            }
        }
    }
    cp_wait<0>();
    __syncthreads();

    // ---- the coarse recurrences: one warp, H columns per lane
    if (warp != 0) return;
    constexpr int KB = 8;
    constexpr int TAB = 0, COL = 1, CONV = 2;  // factors: per-plane table, per column and plane, converged
    const int clast = nz >= 2 ? nz - 2 : 0;
    S* const zl = Z + lane * H;
    S* const wl = ZW + lane * H;
    typedef HVec<P, H> HV;
    auto lds = [&](const S* p) {
        HV h;
        h.get(p);
        return h;
    };
    HV v, d, x, cinv, einv, cwv;
#pragma unroll
    for (int q = 0; q < H; ++q) {
        v.v[q] = P::ld(C.v, cc + q);
        d.v[q] = x.v[q] = P::zero();
        cinv.v[q] = einv.v[q] = cwv.v[q] = P::zero();
        if (percol) {
            cinv.v[q] = P::ld(C.finv, (size_t)clast * plc + cc + q);
            einv.v[q] = P::ld(C.finv, (size_t)(nz - 1) * plc + cc + q);
            cwv.v[q] = P::ld(C.fw, (size_t)clast * plc + cc + q);  // (that of plane nz-1 meets x = 0)
        }
    }
    auto forward = [&](auto kind, int k, int ke, const HV& inv) {
        constexpr int F = decltype(kind)::value;
        auto factor = [&](int kk) {
            HV h = inv;
            if (F == COL) h = lds(wl + kk * NC);
            if (F == TAB) {
                const R t = P::ld_plain(ZW, kk);
#pragma unroll
                for (int q = 0; q < H; ++q) h.v[q] = t;
            }
            return h;
        };
        auto step = [&](int kk, const HV& r, const HV& iv) {
            if (F == COL) {
                HV w;
#pragma unroll
                for (int q = 0; q < H; ++q) w.v[q] = P::mul(v.v[q], iv.v[q]);
                w.put(wl + kk * NC);
            }
#pragma unroll
            for (int q = 0; q < H; ++q) d.v[q] = P::mul(P::fma(v.v[q], d.v[q], r.v[q]), iv.v[q]);
            d.put(zl + kk * NC);
        };
        for (; k + KB <= ke; k += KB) {
            HV r[KB], iv[KB];
#pragma unroll
            for (int t = 0; t < KB; ++t) {
                r[t] = lds(zl + (k + t) * NC);
                iv[t] = factor(k + t);
            }
#pragma unroll
            for (int t = 0; t < KB; ++t) step(k + t, r[t], iv[t]);
        }
        for (; k < ke; ++k) step(k, lds(zl + k * NC), factor(k));
    };
    S* uo = xr.uc + (size_t)(nz - 1) * plc + cc;
    auto backward = [&](auto kind, int k, int ke) {  // planes k-1 .. ke
        constexpr int F = decltype(kind)::value;
        auto factor = [&](int kk) {
            HV h = cwv;
            if (F == COL) h = lds(wl + kk * NC);
            if (F == TAB) {
                const R t = P::ld_plain(ZW, nz + kk);
#pragma unroll
                for (int q = 0; q < H; ++q) h.v[q] = t;
            }
            return h;
        };
        auto step = [&](const HV& dk, const HV& w) {
            HV o;
#pragma unroll
            for (int q = 0; q < H; ++q) {
                x.v[q] = P::fma(w.v[q], x.v[q], dk.v[q]);
                o.v[q] = P::mul(xr.rho, x.v[q]);
            }
            o.put(uo);
            uo -= plc;
        };
        for (; k - KB >= ke; k -= KB) {
            HV dk[KB], w[KB];
#pragma unroll
            for (int t = 0; t < KB; ++t) {
                dk[t] = lds(zl + (k - 1 - t) * NC);
                w[t] = factor(k - 1 - t);
            }
#pragma unroll
            for (int t = 0; t < KB; ++t) step(dk[t], w[t]);
        }
        for (; k > ke; --k) step(lds(zl + (k - 1) * NC), factor(k - 1));
    };
    if (percol) {
        forward(std::integral_constant<int, COL>(), 0, kw, cinv);
        forward(std::integral_constant<int, CONV>(), kw, nz - 1, cinv);
        forward(std::integral_constant<int, CONV>(), nz - 1, nz, einv);
        backward(std::integral_constant<int, CONV>(), nz, kw);
        backward(std::integral_constant<int, COL>(), kw, 0);
    } else {
        forward(std::integral_constant<int, TAB>(), 0, nz, cinv);
        backward(std::integral_constant<int, TAB>(), nz, 0);
    }
}

}  // namespace tpmg
