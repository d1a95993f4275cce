// sweep_tile.cuh -- Smooth (Eq. 11) and line solve (Eq. 9) on tiles of whole columns held in shared
// memory: the planes of a tile are worked on in parallel, only the recurrences run one plane after
// the other.
//
// A block owns 512 bytes of columns over all nz planes, in one, two or four rows: nz * 512 bytes of shared
// memory. Its eight warps take contiguous ranges of planes:
//   1. form the right-hand side of the line solves (Smooth: f - A u) of their planes:
//      f arrives by cp.async for all planes at once, u by batches of planes whose loads are issued together;
//      x neighbours and the tile's inner rows come from the other lanes by shuffles;
//   2. one thread per column (FP32: per four) eliminates forward through shared memory (the only serial part, a
//      chain of a multiply-add and a multiply per plane); the other warps load the u of step 3 or 5 meanwhile;
//   3. FP32: all threads form g_k = u_k + rho d'_k - w_k u_{k+1} (see sweep_x2.cuh);
//   4. the same threads substitute back;
//   5. where step 4 does not yield the result, all threads form and write it as 16-byte vectors.
// Up to three blocks per SM overlap one another's phases. The plane-marching sweeps keep one plane's
// loads, elimination and stack store of every column in one chain, and their Thomas stack in a
// global scratch (8 or 16 bytes of L2 traffic per cell); here nothing but the fields moves.
// Measured, FP32: Smooth 1024^2 x 128 397 us (530 marching; 4.1 TB/s of algorithmic traffic), 128^2 x 128 9.0 (48);
// line solve 165 (345; 6.5 TB/s). A Smooth tile of 128 planes takes 48 000 cycles among three: step 1 half, step 2
// 16 %, step 3 14 %, step 4 20 %. No single rate is reached (DRAM 0.46, L2 0.32, shared-memory wavefronts 0.48):
// with all loads but one taken out it still takes 276 us, so the phases' own work bounds it, not the traffic alone.
// The per-cell arithmetic and its order are those of the other sweeps, so the results are the same
// bits in every precision.
//
// Factors: with lambda^2 varying, 1/m_k of the planes before the converged ones (Lv::fac_k0) comes with
// the tile's other reads into shared memory, where the forward sweep replaces it by w_k = v/m_k (the
// stored factor's bits) for the back substitution; with lambda^2 constant, two tables of nz values.
#pragma once
#include <type_traits>

#include "kernels.cuh"
#include "sweep_x2.cuh"

namespace tpmg {

namespace {

constexpr int TNT = 256;  // threads of a block
constexpr int TNW = TNT / 32;
constexpr int TPB = 512;  // bytes of a tile plane: TR rows of TPB / TR bytes

template <class P>
struct TileVec {  // 16 bytes of adjacent columns
    typedef typename P::S S;
    typedef typename P::R R;
    static constexpr int N = 16 / (int)sizeof(S);
    R v[N];
    __device__ __forceinline__ void from(const float4& t) {
        const S* p = reinterpret_cast<const S*>(&t);
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = P::ld_plain(p, e);
    }
    __device__ __forceinline__ void ldg(const S* p) { from(__ldg(reinterpret_cast<const float4*>(p))); }
    __device__ __forceinline__ void lds(const S* p) { from(*reinterpret_cast<const float4*>(p)); }
    // a field: through the read-only cache, or by ordinary loads where this kernel itself writes it
    template <bool RO>
    __device__ __forceinline__ void ldf(const S* p) {
        if (RO) ldg(p);
        else lds(p);
    }
    __device__ __forceinline__ void sts(S* p) const {
        float4 t;
        S* q = reinterpret_cast<S*>(&t);
#pragma unroll
        for (int e = 0; e < N; ++e) P::sts(q, e, v[e]);
        *reinterpret_cast<float4*>(p) = t;
    }
    __device__ __forceinline__ void stg(S* p) const {  // storage rounding (P::st) applied
        float4 t;
        S* q = reinterpret_cast<S*>(&t);
#pragma unroll
        for (int e = 0; e < N; ++e) P::sts(q, e, P::rnd(v[e]));
        *reinterpret_cast<float4*>(p) = t;
    }
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = P::zero();
    }
};

// CV adjacent columns of a plane in the recurrences
template <class P, int CV>
struct TileCol : TileVec<P> {
    typedef typename P::R R;
    static_assert(CV == TileVec<P>::N, "16 bytes, or one column");
    __device__ __forceinline__ void fill(R x) {
#pragma unroll
        for (int q = 0; q < CV; ++q) this->v[q] = x;
    }
};
template <class P>
struct TileCol<P, 1> {
    typedef typename P::S S;
    typedef typename P::R R;
    R v[1];
    __device__ __forceinline__ void ldg(const S* p) { v[0] = P::ld(p, 0); }
    __device__ __forceinline__ void lds(const S* p) { v[0] = P::ld_plain(p, 0); }
    __device__ __forceinline__ void sts(S* p) const { P::sts(p, 0, v[0]); }
    __device__ __forceinline__ void stg(S* p) const { P::st(p, 0, v[0]); }
    __device__ __forceinline__ void zero() { v[0] = P::zero(); }
    __device__ __forceinline__ void fill(R x) { v[0] = x; }
};

__device__ __forceinline__ float shfl_up_v(float x, int d) { return __shfl_up_sync(0xffffffffu, x, d); }
__device__ __forceinline__ float shfl_dn_v(float x, int d) { return __shfl_down_sync(0xffffffffu, x, d); }
__device__ __forceinline__ dw shfl_up_v(dw x, int d) { return dw{shfl_up_v(x.hi, d), shfl_up_v(x.lo, d)}; }
__device__ __forceinline__ dw shfl_dn_v(dw x, int d) { return dw{shfl_dn_v(x.hi, d), shfl_dn_v(x.lo, d)}; }

__device__ __forceinline__ void tile_cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

}  // namespace

// MODE_CGTRI: the fused Tridiag of CG, u the residual r (rewritten: r -= alpha q), f = q, out = z = M^{-1} r,
// partial sums of <r, r> and, behind them, of <r, z>: with M = U^T D U the elimination gives yh = U^{-T} r
// and d' = D^{-1} yh, so <r, M^{-1} r> = sum_k yh_k d'_k, and the back substitution does not read r again.
constexpr int MODE_CGTRI = 16;
// u's element type: only MODE_CGTRI writes it
template <class P, int MODE>
using TileU = std::conditional_t<MODE == MODE_CGTRI, typename P::S, const typename P::S>;

// One tile: columns bx * W .., rows by * TR ...
// kw: planes whose factors are kept per column in shared memory behind the nz planes of the tile (0
// when lambda^2 is constant). ISO: square cells; NORM: partial sums of ||f - A u||^2, this tile's at part of
// nparts (both compile-time: as runtime choices their instructions were issued either way). RO: the fields read
// are not written by the kernel
template <class P, int MODE, int TR, bool ISO, bool NORM, bool RO>
__device__ __forceinline__ void sweep_tile_body(const Lv<P>& L, const SweepK<P>& K, TileU<P, MODE>* u,
                                                const typename P::S* f, typename P::S* out, double* partials, int kw,
                                                const Scalars* sc, int bx, int by, int part, int nparts,
                                                unsigned char* smem_raw) {
    typedef typename P::S S;
    typedef typename P::R R;
    typedef TileVec<P> V;
    // values held ahead of their use: not in the batched kernel (!RO), whose registers they overflow (31.0 ms for its
    // 12 problems against 28.7)
    constexpr bool AHEAD = RO;
    constexpr bool CG = MODE == MODE_CGTRI;
    constexpr bool SM = MODE == MODE_SMOOTH;  // a stencil, and u in the result
    constexpr bool GFORM = MODE == MODE_SMOOTH && P::id == 1;
    constexpr bool DIRECT = GFORM || MODE == MODE_LINESOLVE || CG;  // the back substitution yields the result
    constexpr int G = 32 / TR;                                // lanes of a tile row
    constexpr int N = V::N, W = G * N, NC = TR * W;
    S* const Z = reinterpret_cast<S*>(smem_raw);
    const int nx = L.nx, ny = L.ny, nz = L.nz;
    S* const ZW = Z + (size_t)nz * NC;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, lx = lane % G, ry = lane / G;
    const int i0 = bx * W, j0 = by * TR;
    const size_t pl = (size_t)nx * ny;
    const size_t c = (size_t)(j0 + ry) * nx + i0 + lx * N;  // this thread's first column
    const int zo = lane * N;                                // ... in a tile plane
    const int ch = (nz + TNW - 1) / TNW, klo = warp * ch, khi = klo + ch < nz ? klo + ch : nz;
    const bool percol = L.fac_percol != 0;
    typename P::Acc acc = 0, cmp = 0, az = 0, cz = 0;

    // ---- 1. the right-hand side of the line solves
    {
        const S* src = (SM ? f : u) + (size_t)klo * pl + c;
        const S* inv = L.finv + (size_t)klo * pl + c;
        S* z = Z + klo * NC + zo;
        for (int k = klo; k < khi; ++k, src += pl, z += NC) tile_cp16(z, src);
        if (percol) {  // 1/m_k of the planes before the converged ones; the forward sweep turns them into w_k
            z = ZW + klo * NC + zo;
            for (int k = klo; k < khi && k < kw; ++k, inv += pl, z += NC) tile_cp16(z, inv);
        } else {
            for (int k = tid; k < nz; k += TNT) {
                cp_async<(int)sizeof(S)>(ZW + k, L.finv + k);
                cp_async<(int)sizeof(S)>(ZW + nz + k, L.fw + k);
            }
        }
        cp_commit();
    }
    if constexpr (SM) {
        if (klo < khi) {
            // the rows next to the tile's first and last one (one row: both, two or more: a lane meets at
            // most one of them), and the columns left and right of it (first and last lane of a row)
            const int js = j0 == 0 ? ny - 1 : j0 - 1, jn = j0 + TR == ny ? 0 : j0 + TR;
            const bool hrow = TR <= 2 || ry == 0 || ry == TR - 1;
            // every lane loads the left or the right one: a load under a condition would be waited for on the spot
            const int hi = lx < G / 2 ? (i0 == 0 ? nx - 1 : i0 - 1) : (i0 + W == nx ? 0 : i0 + W);
            const size_t p0 = (size_t)klo * pl;
            const S* pu = u + p0 + c;
            const S* ph = u + p0 + (size_t)(ry == 0 ? js : jn) * nx + i0 + lx * N;
            const S* ph1 = u + p0 + (size_t)jn * nx + i0 + lx * N;  // TR == 1
            const S* pe = u + p0 + (size_t)(j0 + ry) * nx + hi;
            S* z = Z + klo * NC + zo;
            constexpr int D = TR == 1 ? 2 : (P::id == 1 && RO ? 4 : 3);  // planes fetched together
            const R cx = K.cx, cy = K.cy, dh = K.dh;
            V um, uc, vv, dg;
            um.zero();
            dg.zero();
            uc.template ldf<RO>(pu);
            if (klo > 0) um.template ldf<RO>(pu - pl);
            vv.ldg(L.v + c);
            bool first = true;
            // one batch of B planes from plane k: all their loads, then their arithmetic
            auto batch = [&](auto bc, int k) {
                constexpr int B = decltype(bc)::value;
                V ru[B], rh[B], rh1[B];
                R re[B];
                const bool top = k + B == nz;  // the last plane has no upper neighbour
#pragma unroll
                for (int t = 0; t < B; ++t) {  // u of plane k+t+1, the halo of plane k+t
                    ru[t].template ldf<RO>(t + 1 == B && top ? pu : pu + pl);
                    if (!hrow) rh[t].zero();
                    if (hrow) rh[t].template ldf<RO>(ph);
                    if (TR == 1) rh1[t].template ldf<RO>(ph1);
                    re[t] = RO ? P::ld(pe, 0) : P::ld_plain(pe, 0);
                    pu += pl;
                    ph += pl;
                    ph1 += pl;
                    pe += pl;
                }
                if (first) {  // (the first batch's loads are on their way too)
                    cp_wait<0>();  // this thread's pieces of f
#pragma unroll
                    for (int q = 0; q < N; ++q) dg.v[q] = P::add(P::add(dh, vv.v[q]), vv.v[q]);
                    first = false;
                }
                if (top) ru[B - 1].zero();
#pragma unroll
                for (int t = 0; t < B; ++t, z += NC) {
                    V r;
                    r.lds(z);
                    R wl = shfl_up_v(uc.v[N - 1], 1), el = shfl_dn_v(uc.v[0], 1);
                    if (lx == 0) wl = re[t];
                    if (lx == G - 1) el = re[t];
                    V d = dg;
                    if (k + t == 0 || k + t == nz - 1) {
#pragma unroll
                        for (int q = 0; q < N; ++q) d.v[q] = nz == 1 ? dh : P::add(dh, vv.v[q]);
                    }
#pragma unroll
                    for (int q = 0; q < N; ++q) {
                        R s = rh[t].v[q], n = rh[t].v[q];
                        if constexpr (TR == 1) {
                            n = rh1[t].v[q];
                        } else if constexpr (TR == 2 && P::id == 1) {
                            // the other row; which of the two is the south one does not change their sum
                            n = __shfl_xor_sync(0xffffffffu, uc.v[q], G);
                        } else {
                            const R su = shfl_up_v(uc.v[q], G), nd = shfl_dn_v(uc.v[q], G);
                            if (ry != 0) s = su;
                            if (ry != TR - 1) n = nd;
                        }
                        const R w = q == 0 ? wl : uc.v[q > 0 ? q - 1 : 0];
                        const R e = q == N - 1 ? el : uc.v[q < N - 1 ? q + 1 : q];
                        r.v[q] = sweep_residual<P>(r.v[q], d.v[q], uc.v[q], w, e, s, n, um.v[q], ru[t].v[q], cx, cy,
                                                   vv.v[q], ISO);
                        if (NORM) P::acc_dot(acc, cmp, r.v[q], r.v[q]);
                    }
                    r.sts(z);
                    um = uc;
                    uc = ru[t];
                }
            };
            int k = klo;
            for (; k + D <= khi; k += D) batch(std::integral_constant<int, D>(), k);
            for (; k < khi; ++k) batch(std::integral_constant<int, 1>(), k);
        }
    }
    if constexpr (CG) {
        const R nalpha = P::neg(P::cst(sc->alpha));
        const S* pq = f + (size_t)klo * pl + c;
        S* pr = u + (size_t)klo * pl + c;
        S* z = Z + klo * NC + zo;
        bool landed = false;
#pragma unroll 4
        for (int k = klo; k < khi; ++k, pq += pl, pr += pl, z += NC) {
            V q, r;
            q.template ldf<RO>(pq);
            if (!landed) {
                cp_wait<0>();  // this thread's pieces of r
                landed = true;
            }
            r.lds(z);
#pragma unroll
            for (int t = 0; t < N; ++t) {
                r.v[t] = P::fma(nalpha, q.v[t], r.v[t]);
                P::acc_dot(acc, cmp, r.v[t], r.v[t]);
            }
            r.stg(pr);
            r.sts(z);
        }
    }
    cp_wait<0>();
    __syncthreads();

    // ---- 2. forward elimination, CV columns per thread, four planes' values read ahead of four planes'
    // steps (per-column factors: eight planes at a time). FP32: one
    // warp, four columns per thread (as many issue slots as one column each on four warps take for
    // one); the longer chains of the 8-byte policies take one column per thread
    constexpr int KB = 8, KP = 4, CV = P::id == 1 ? N : 1, CT = NC / CV;
    constexpr int TAB = 0, COL = 1, CONV = 2;  // factors: per-plane table, per column and plane, converged
    typedef TileCol<P, CV> C;
    const bool col = tid < CT;
    const int c0 = tid * CV;  // first column in the tile plane
    const size_t gc = col ? (size_t)(j0 + c0 / W) * nx + i0 + c0 % W : 0;
    const int clast = nz >= 2 ? nz - 2 : 0;  // plane of the converged factors
    if (col) {
        C v, d;
        v.ldg(L.v + gc);
        d.zero();
        auto sweep = [&](auto kind, int k, int ke, const C& inv) {
            constexpr int F = decltype(kind)::value;
            S* z = Z + k * NC + c0;
            S* zw = F == TAB ? ZW + k : ZW + k * NC + c0;
            auto step = [&](S* zk, S* zwk, const C& r, const C& iv) {
                if (F == COL) {
                    C w;
#pragma unroll
                    for (int q = 0; q < CV; ++q) w.v[q] = P::mul(v.v[q], iv.v[q]);
                    w.sts(zwk);
                }
#pragma unroll
                for (int q = 0; q < CV; ++q) {
                    if constexpr (CG) {
                        const R yh = P::fma(v.v[q], d.v[q], r.v[q]);
                        d.v[q] = P::mul(yh, iv.v[q]);
                        P::acc_dot(az, cz, yh, d.v[q]);
                    } else {
                        d.v[q] = P::mul_u(P::fma_u(v.v[q], d.v[q], r.v[q]), iv.v[q]);
                    }
                }
                d.sts(zk);
            };
            auto factor = [&](C& iv, const S* zwk) {
                if (F == TAB) iv.fill(P::ld_plain(zwk, 0));
                if (F == COL) iv.lds(zwk);
                if (F == CONV) iv = inv;
            };
            constexpr int WS = F == TAB ? 1 : NC;
            if (F == COL || !AHEAD) {
                for (; k + KB <= ke; k += KB, z += KB * NC, zw += KB * WS) {
                    C r[KB], iv[KB];
#pragma unroll
                    for (int q = 0; q < KB; ++q) {
                        r[q].lds(z + q * NC);
                        factor(iv[q], zw + q * WS);
                    }
#pragma unroll
                    for (int q = 0; q < KB; ++q) step(z + q * NC, zw + q * WS, r[q], iv[q]);
                }
            } else if (k + KP <= ke) {
                C ra[KP], ia[KP], rb[KP], ib[KP];
                auto get = [&](C* r, C* iv, int ahead) {
#pragma unroll
                    for (int q = 0; q < KP; ++q) {
                        r[q].lds(z + (ahead + q) * NC);
                        factor(iv[q], zw + (ahead + q) * WS);
                    }
                };
                auto run = [&](const C* r, const C* iv) {
#pragma unroll
                    for (int q = 0; q < KP; ++q) step(z + q * NC, zw + q * WS, r[q], iv[q]);
                    k += KP;
                    z += KP * NC;
                    zw += KP * WS;
                };
                get(ra, ia, 0);
                while (k + 3 * KP <= ke) {
                    get(rb, ib, KP);
                    run(ra, ia);
                    get(ra, ia, KP);
                    run(rb, ib);
                }
                run(ra, ia);
                if (k + KP <= ke) {
                    get(rb, ib, 0);
                    run(rb, ib);
                }
            }
            for (; k < ke; ++k, z += NC, zw += WS) {
                C r, iv;
                r.lds(z);
                factor(iv, zw);
                step(z, zw, r, iv);
            }
        };
        C cinv;
        cinv.zero();
        if (percol) {
            C einv;
            cinv.ldg(L.finv + (size_t)clast * pl + gc);
            einv.ldg(L.finv + (size_t)(nz - 1) * pl + gc);
            sweep(std::integral_constant<int, COL>(), 0, kw, cinv);
            sweep(std::integral_constant<int, CONV>(), kw, nz - 1, cinv);
            sweep(std::integral_constant<int, CONV>(), nz - 1, nz, einv);
        } else {
            sweep(std::integral_constant<int, TAB>(), 0, nz, cinv);
        }
    }

    // u of the planes klo .. for what follows the recurrences: GB of them (and one more) are loaded ahead of the
    // barrier, behind which the other warps wait for the recurrences
    constexpr int GB = AHEAD ? 8 : 4;
    V ua[GB + 1];
    auto fetch = [&](int k) {  // planes k .. k + GB; past the last one needed, that again
        const int kl = GFORM && khi < nz ? khi : khi - 1;
        const S* p = u + (size_t)k * pl + c;
#pragma unroll
        for (int t = 0; t < (GFORM ? GB + 1 : GB); ++t) {
            ua[t].template ldf<RO>(p);
            if (k + t < kl) p += pl;
        }
    };
    if (AHEAD && GFORM && klo < khi) fetch(klo);
    __syncthreads();
    if (!AHEAD && GFORM && klo < khi) fetch(klo);

    // ---- 3. FP32: g_k = u_k + rho d'_k - w_k u_{k+1}
    if constexpr (GFORM) {
        if (klo < khi) {
            const R cf = K.coef;
            V cw;
            cw.zero();
            if (percol) cw.ldg(L.fw + (size_t)clast * pl + c);  // the converged v/m_k
            S* z = Z + klo * NC + zo;
            for (int k = klo; k < khi; k += GB) {
                if (k > klo) fetch(k);
#pragma unroll
                for (int t = 0; t < GB; ++t, z += NC) {
                    if (k + t >= khi) break;
                    V g, w = cw;
                    g.lds(z);
                    if (k + t < kw) w.lds(ZW + (k + t) * NC + zo);
                    if (!percol) {
                        const R wk = P::ld_plain(ZW, nz + k + t);
#pragma unroll
                        for (int q = 0; q < N; ++q) w.v[q] = wk;
                    }
                    if (k + t + 1 == nz) ua[t + 1].zero();
#pragma unroll
                    for (int q = 0; q < N; ++q)
                        g.v[q] = P::fma(P::neg(w.v[q]), ua[t + 1].v[q], P::fma(cf, g.v[q], ua[t].v[q]));
                    g.sts(z);
                }
            }
        }
        __syncthreads();
    }

    // ---- 4. back substitution
    if (col) {
        C x;
        x.zero();
        S* po = out + (size_t)(nz - 1) * pl + gc;
        auto sweep = [&](auto kind, int k, int ke, const C& cw) {  // planes k-1 .. ke
            constexpr int F = decltype(kind)::value;
            S* z = Z + (k - 1) * NC + c0;
            const S* zw = F == TAB ? ZW + nz + k - 1 : ZW + (k - 1) * NC + c0;
            auto factor = [&](C& w, const S* zwk) {
                if (F == TAB) w.fill(P::ld_plain(zwk, 0));
                if (F == COL) w.lds(zwk);
                if (F == CONV) w = cw;
            };
            auto step = [&](S* zk, const C& d, const C& w) {
#pragma unroll
                for (int q = 0; q < CV; ++q)
                    x.v[q] = CG ? P::fma(w.v[q], x.v[q], d.v[q]) : P::fma_u(w.v[q], x.v[q], d.v[q]);
                if (DIRECT) {
                    C o = x;
                    if (MODE == MODE_LINESOLVE) {
#pragma unroll
                        for (int q = 0; q < CV; ++q) o.v[q] = P::mul(K.coef, x.v[q]);
                    }
                    o.stg(po);
                    po -= pl;
                } else {
                    x.sts(zk);
                }
            };
            constexpr int WS = F == TAB ? 1 : NC;
            if (F == COL || !AHEAD) {
                for (; k - KB >= ke; k -= KB, z -= KB * NC, zw -= KB * WS) {
                    C d[KB], w[KB];
#pragma unroll
                    for (int q = 0; q < KB; ++q) {
                        d[q].lds(z - q * NC);
                        factor(w[q], zw - q * WS);
                    }
#pragma unroll
                    for (int q = 0; q < KB; ++q) step(z - q * NC, d[q], w[q]);
                }
            } else if (k - KP >= ke) {
                C da[KP], wa[KP], db[KP], wb[KP];
                auto get = [&](C* d, C* w, int ahead) {
#pragma unroll
                    for (int q = 0; q < KP; ++q) {
                        d[q].lds(z - (ahead + q) * NC);
                        factor(w[q], zw - (ahead + q) * WS);
                    }
                };
                auto run = [&](const C* d, const C* w) {
#pragma unroll
                    for (int q = 0; q < KP; ++q) step(z - q * NC, d[q], w[q]);
                    k -= KP;
                    z -= KP * NC;
                    zw -= KP * WS;
                };
                get(da, wa, 0);
                while (k - 3 * KP >= ke) {
                    get(db, wb, KP);
                    run(da, wa);
                    get(da, wa, KP);
                    run(db, wb);
                }
                run(da, wa);
                if (k - KP >= ke) {
                    get(db, wb, 0);
                    run(db, wb);
                }
            }
            for (; k > ke; --k, z -= NC, zw -= WS) {
                C d, w;
                d.lds(z);
                factor(w, zw);
                step(z, d, w);
            }
        };
        C cw;
        cw.zero();
        if (percol) {
            cw.ldg(L.fw + (size_t)clast * pl + gc);  // (that of plane nz-1 meets x = 0)
            sweep(std::integral_constant<int, CONV>(), nz, kw, cw);
            sweep(std::integral_constant<int, COL>(), kw, 0, cw);
        } else {
            sweep(std::integral_constant<int, TAB>(), nz, 0, cw);
        }
    }

    // ---- 5. the result of the forms that add u
    if constexpr (!DIRECT) {
        if (klo < khi) fetch(klo);
        __syncthreads();
        const R cf = K.coef;
        S* po = out + (size_t)klo * pl + c;
        const S* z = Z + klo * NC + zo;
        for (int k = klo; k < khi; k += GB) {
            if (k > klo) fetch(k);
#pragma unroll
            for (int t = 0; t < GB; ++t, po += pl, z += NC) {
                if (k + t >= khi) break;
                V x;
                x.lds(z);
#pragma unroll
                for (int q = 0; q < N; ++q) x.v[q] = P::fma(cf, x.v[q], ua[t].v[q]);
                x.stg(po);
            }
        }
    }
    if (NORM) {
        const double sm = block_sum(P::acc_get(acc, cmp));
        if (tid == 0) partials[part] = sm;
        if constexpr (CG) {
            __syncthreads();
            const double sz = block_sum(P::acc_get(az, cz));
            if (tid == 0) partials[nparts + part] = sz;
        }
    }
}

template <class P, int MODE, int TR, bool ISO, bool NORM>
__global__ void __launch_bounds__(TNT, 3)
    k_sweep_tile(Lv<P> L, SweepK<P> K, TileU<P, MODE>* __restrict__ u, const typename P::S* __restrict__ f,
                 typename P::S* __restrict__ out, double* partials, const int* done, int kw, const Scalars* sc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (done && *(volatile const int*)done) return;
    sweep_tile_body<P, MODE, TR, ISO, NORM, true>(L, K, u, f, out, partials, kw, sc, blockIdx.x, blockIdx.y,
                                                  blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, smem_raw);
}

template <class P, int MODE, int TR, bool ISO, bool NORM>
static int run_sweep_tile(const Lv<P>& L, double coef, TileU<P, MODE>* u, const typename P::S* f,
                          typename P::S* out, double* partials, const int* done, cudaStream_t s, const Scalars* sc) {
    typedef typename P::S S;
    int kw = 0;
    if (L.fac_percol) kw = factor_planes(L);
    const size_t smem = (size_t)(L.nz + kw) * TPB + (L.fac_percol ? 0 : 2 * (size_t)L.nz * sizeof(S));
    auto kern = k_sweep_tile<P, MODE, TR, ISO, NORM>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 256 * TPB);
    const dim3 grd(L.nx / (TPB / TR / (int)sizeof(S)), L.ny / TR);
    kern<<<grd, TNT, smem, s>>>(L, sweep_k<P>(L.cx, L.cy, coef), u, f, out, partials, done, kw, sc);
    note_launch();
    return (int)(grd.x * grd.y);
}

// Rows of a level's tiles, 0 where it has none. two: two rows wherever they fit. The launch takes 65535 rows of tiles.
template <class P>
static int tile_rows(int nx, int ny, bool two) {
    constexpr int W = TPB / (int)sizeof(typename P::S), MAXR = 65535;
    if (nx % W == 0 && !(two && ny % 2 == 0) && ny <= MAXR) return 1;
    if (nx % (W / 2) == 0 && ny % 2 == 0 && ny / 2 <= MAXR) return 2;
    return nx % (W / 4) == 0 && ny % 4 == 0 && ny / 4 <= MAXR ? 4 : 0;
}
template <class P, int MODE, bool ISO, bool NORM>
static int run_sweep_tile_rows(const Lv<P>& L, double coef, TileU<P, MODE>* u, const typename P::S* f,
                               typename P::S* out, double* partials, const int* done, cudaStream_t s,
                               const Scalars* sc = nullptr) {
    // FP32 Smooth: two rows of 64 columns share their inner rows and so load two rows of u per row instead of
    // three (1024^2 x 128 396 us, 429 with one row of 128, 436 with four of 32)
    switch (tile_rows<P>(L.nx, L.ny, P::id == 1 && MODE == MODE_SMOOTH)) {
        case 1: return run_sweep_tile<P, MODE, 1, ISO, NORM>(L, coef, u, f, out, partials, done, s, sc);
        case 2: return run_sweep_tile<P, MODE, 2, ISO, NORM>(L, coef, u, f, out, partials, done, s, sc);
        case 4: return run_sweep_tile<P, MODE, 4, ISO, NORM>(L, coef, u, f, out, partials, done, s, sc);
        default: return -1;
    }
}

// Where the fused Tridiag runs on tiles. Double-word: as the Smooth. FP32: everywhere from 16 planes (against one column a
// thread: 352^2 x 70 CG iteration 138 us, 237), but on large levels that take the two-column sweep, the faster one there
// (us, tile / sweep; with the call's scalar kernels): 128 x 64 x 16 12 / 13, 160^2 x 64 17 / 37; 256^2 x 32 23 / 19, x 64
// 30 / 29, x 96 37 / 41; 512^2 x 32 55 / 40, x 96 102 / 104; 1024 x 512 x 16 82 / 37. In between, as long as three blocks an
// SM take the level in one wave, tiles from 24 planes: tile over sweep, 34816 to 58368 columns, 1.07-1.10 at 16 planes,
// 0.91-1.00 at 24, 0.73-0.84 at 48.
template <class P>
static bool cg_tile_pays(const Lv<P>& L) {
    const size_t cols = (size_t)L.nx * L.ny;
    if (P::id != 1) return tile_pays(L);
    const bool pairs = L.gstack && L.nx % 64 == 0 && L.ny % 2 == 0;
    const int from = cols <= 32768 ? 16 : cols <= 3 * 152 * 128 ? 24 : 65;
    return L.nz >= 16 && (!pairs || (cols <= 65536 && L.nz >= from));
}
template <class P>
int cg_tile_blocks(const Lv<P>& L) {
    if (L.nz > 128 || !L.finv || !L.fw || !cg_tile_pays(L)) return -1;
    auto al = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
    if (!al(L.v) || (L.fac_percol && (!al(L.finv) || !al(L.fw)))) return -1;
    const int tr = tile_rows<P>(L.nx, L.ny, false);
    return tr ? L.nx / (TPB / tr / (int)sizeof(typename P::S)) * (L.ny / tr) : -1;
}
template <class P>
int launch_cg_tile(const Lv<P>& L, const Scalars* sc, typename P::S* r, const typename P::S* q, typename P::S* z,
                   double* partials, cudaStream_t s) {
    if (cg_tile_blocks(L) < 0) return -1;
    return run_sweep_tile_rows<P, MODE_CGTRI, true, true>(L, 1.0, r, q, z, partials, &sc->done, s, sc);
}

template <class P, int MODE>
int launch_sweep_tile(const Lv<P>& L, double coef, const typename P::S* u, const typename P::S* f, typename P::S* out,
                      double* partials, const int* done, cudaStream_t s) {
    if (L.nz > 128 || !L.finv || !L.fw) return -1;
    auto al = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
    if (!al(u) || (MODE != MODE_LINESOLVE && !al(f)) || !al(out) || !al(L.v) || (L.fac_percol && (!al(L.finv) || !al(L.fw))))
        return -1;
    // the line solve has no stencil and no norm
    constexpr bool ONE = MODE == MODE_LINESOLVE, NN = MODE != MODE_SMOOTH;
    if (ONE || L.cx == L.cy) {
        if (NN || !partials) return run_sweep_tile_rows<P, MODE, true, false>(L, coef, u, f, out, partials, done, s);
        return run_sweep_tile_rows<P, MODE, true, !NN>(L, coef, u, f, out, partials, done, s);
    }
    if (NN || !partials) return run_sweep_tile_rows<P, MODE, ONE, false>(L, coef, u, f, out, partials, done, s);
    return run_sweep_tile_rows<P, MODE, ONE, !NN>(L, coef, u, f, out, partials, done, s);
}

}  // namespace tpmg
