// k_batched.cu -- the batched persistent solver: many independent problems of different sizes in
// one cooperative launch.
//
// Each problem runs mixed-precision iterative refinement: r = f - A u in double-word arithmetic
// (stored FP32), one FP32 V-cycle of Algorithm 1 on A e = r from e = 0, u += e. The host turns the
// cycle of every problem into a list of phases; phase p holds one task per problem (the problem's
// p-th step: a Smooth, Residual, RestrictSmooth, Prolongate, ... on one of its levels), each task cut
// into tiles. The persistent blocks stride over the tiles of a phase and then
// meet at a grid barrier; problems of fewer levels simply have no task in the late phases. The
// barrier is a counter plus generation word; every wait is bounded by a time limit after which
// the kernel raises an error flag and all blocks return (TPMG_ERR_TIMEOUT on the host).
//
// Forms of a task (batched_form):
//  - BF_TILE1, BF_TILE2: Smooth and first line solve on whole columns in shared memory, 128 x 1 or 64 x 2 FP32
//    columns a tile, as the single-problem solver's (sweep_tile.cuh; here the one-row tile is the faster one); the
//    fused Residual + RestrictSmooth on tiles of 128 x 2 fine columns (restrict_tile.cuh);
//  - BF_COLS: 32 columns of the level in order, planes in parallel over the eight warps, one warp running the
//    recurrences in shared memory, their factors there too: all other shapes;
//  - Residuals (FP32 and the outer double-word one), Prolongate and the correction: pointwise.
// Three blocks of 256 threads per SM, set by the tiles' 65 KB at 128 planes, or two where a tile's per-column factors
// take it to 84 KB (BTILE_SMEM2). Ten cycles of 256^2 x 64, 512 x 256 x 128, 128^2 x 64 and 64 x 128 x 32, ms: lambda^2
// constant 10.4, varying 13.9 (two blocks; 16.9 with those levels on BF_COLS). 256^2 x 200 and 128 x 256 x 200 (BF_COLS)
// 14.7 and 16.7 (20.2 with a limit of 98 KB, which moves some of their levels to tiles); oblong cells the same. With
// BF_COLS' factors read from global memory plane by plane the varying ones took 28 and 31 ms.
// What is left: the FP32 tiles (0.55 of the copy rate), the outer residual and correction (20 bytes per cell each) and,
// once most problems have converged, too few tiles per phase.
#include <type_traits>

#include "kernels.cuh"
#include "restrict_tile.cuh"
#include "sweep_tile.cuh"

namespace tpmg {

constexpr int BNT = 256, BNW = BNT / 32;
static_assert(BNT == TNT && BNT == RNT, "the tiles' block");
constexpr int BPZ = 16;             // planes of a column a pointwise residual tile takes
constexpr int BCH = 4096;           // cells of a correction tile
constexpr int BPU = 1024;           // coarse segments of a Prolongate tile
constexpr size_t BTILE_SMEM = 72 * 1024;  // three blocks of it fit an SM
constexpr size_t BTILE_SMEM2 = 84 * 1024;  // two: tiles with per-column factors

__device__ __forceinline__ int bwrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Grid barrier with a time limit. Returns false (and raises *error) if the wait gave up.
__device__ bool grid_barrier(const BatchDesc& d) {
    __syncthreads();
    __shared__ int ok;
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned* gen = d.bar_gen;
        const unsigned g = *gen;
        __threadfence();
        const unsigned arrived = atomicAdd(d.bar_count, 1u);
        if (arrived == gridDim.x - 1) {
            *d.bar_count = 0;
            __threadfence();
            atomicAdd(d.bar_gen, 1u);
        } else {
            const unsigned long long t0 = global_ns();
            while (*gen == g) {
                if (*(volatile int*)d.error) {
                    ok = 0;
                    break;
                }
                if (global_ns() - t0 > d.timeout_ns) {
                    atomicExch(d.error, 1);
                    ok = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// ---------------------------------------------------------------- tile operations
// Fields are read by ordinary loads: they are written by this kernel, and the read-only path need not see that.

struct BCol {  // a column of a level and its horizontal neighbours
    size_t c, w, e, s, n;
    bool act;
};
__device__ __forceinline__ BCol bcol(int nx, int ny, int col) {
    BCol q;
    q.act = col < nx * ny;
    if (!q.act) col = nx * ny - 1;
    const int j = col / nx, i = col - j * nx;
    q.c = (size_t)col;
    q.w = (size_t)j * nx + bwrap(i - 1, nx);
    q.e = (size_t)j * nx + bwrap(i + 1, nx);
    q.s = (size_t)bwrap(j - 1, ny) * nx + i;
    q.n = (size_t)bwrap(j + 1, ny) * nx + i;
    return q;
}
// FP32 residual of a cell
template <bool SW>
__device__ __forceinline__ float bresidual(const SweepK<PolF32>& K, float diag, float vv, float fk, float uc, float w, float e,
                                           float s, float n, float um, float up) {
    if (SW) return sweep_residual<PolF32>(fk, diag, uc, w, e, s, n, um, up, K.cx, K.cy, vv, K.iso != 0);
    const float cx = K.cx, cy = K.cy, hx = w + e, hy = s + n;
    return fk - (diag * uc - cx * hx - cy * hy - vv * (um + up));
}
template <class P>
__device__ __forceinline__ typename P::R bload(const typename P::S* p, size_t i) { return P::ld_plain(p, i); }

// r = f - A u on planes of BNT columns; the sum of squares of the thread's residuals (SUM)
template <class P, class PO, bool SW, bool SUM>
__device__ double t_residual(int nx, int ny, int nz, const SweepK<P>& K, const typename P::S* vp, const typename P::S* u,
                             const typename P::S* f, typename PO::S* r, int tile) {
    typedef typename P::R R;
    const int tx = (nx * ny + BNT - 1) / BNT;
    const BCol q = bcol(nx, ny, (tile % tx) * BNT + threadIdx.x);
    const size_t pl = (size_t)nx * ny;
    const int k0 = tile / tx * BPZ, k1 = k0 + BPZ < nz ? k0 + BPZ : nz;
    typename P::Acc acc = 0, cmp = 0;
    if (q.act) {
        const R vv = P::ld(vp, q.c), dh1 = P::add(K.dh, vv), dh2 = P::add(dh1, vv);
        const bool iso = K.iso != 0;
        const size_t b0 = (size_t)k0 * pl;
        const typename P::S *pw = u + b0 + q.w, *pe = u + b0 + q.e, *ps = u + b0 + q.s, *pn = u + b0 + q.n,
                            *pu = u + b0 + q.c, *pf = f + b0 + q.c;
        typename PO::S* pr = r + b0 + q.c;
        R um = k0 > 0 ? bload<P>(pu - pl, 0) : P::zero(), uc = bload<P>(pu, 0);
        // two planes' loads are issued together
        constexpr int D = 2;
        for (int k = k0; k < k1; k += D) {
            R up[D], w[D], e[D], s[D], n[D], fk[D];
#pragma unroll
            for (int t = 0; t < D; ++t) {
                const size_t o = (size_t)(k + t < nz ? t : 0) * pl;       // past the end: plane k again, not used
                const size_t o1 = (size_t)(k + t + 1 < nz ? t + 1 : 0) * pl;
                up[t] = bload<P>(pu, o1);
                w[t] = bload<P>(pw, o);
                e[t] = bload<P>(pe, o);
                s[t] = bload<P>(ps, o);
                n[t] = bload<P>(pn, o);
                fk[t] = bload<P>(pf, o);
            }
#pragma unroll
            for (int t = 0; t < D; ++t) {
                if (k + t >= k1) break;
                if (k + t + 1 == nz) up[t] = P::zero();
                const R dg = nz == 1 ? K.dh : (k + t == 0 || k + t == nz - 1 ? dh1 : dh2);
                R rk;
                if constexpr (P::id == 1) rk = bresidual<SW>(K, dg, vv, fk[t], uc, w[t], e[t], s[t], n[t], um, up[t]);
                else rk = sweep_residual<P>(fk[t], dg, uc, w[t], e[t], s[t], n[t], um, up[t], K.cx, K.cy, vv, iso);
                if constexpr (PO::id == P::id) P::st(reinterpret_cast<typename P::S*>(pr), (size_t)t * pl, rk);
                else PO::st(pr, (size_t)t * pl, PO::from_f(P::to_f(rk)));
                if (SUM) P::acc_dot(acc, cmp, rk, rk);
                um = uc;
                uc = up[t];
            }
            pw += D * pl;
            pe += D * pl;
            ps += D * pl;
            pn += D * pl;
            pu += D * pl;
            pf += D * pl;
            pr += D * pl;
        }
    }
    return P::acc_get(acc, cmp);
}

enum { BM_SMOOTH = 0, BM_LINE = 1, BM_RESTRICT = 2 };

// Levels of 64-column multiples (and ny of 4) have the arithmetic of the single-problem sweeps in every form (SW:
// sweep_residual's order, the Smooth's back substitution over g_k = u_k + rho d_k - w_k u_{k+1}), the others the
// plain one; a form that takes a level over gives the same bits.
__host__ __device__ __forceinline__ bool bsweeps(int nx, int ny) { return nx % 64 == 0 && ny % 4 == 0; }

// The right-hand side of a column's line solve at plane k: f - A u (Smooth), f, or the restricted residual
template <int MODE, bool SW>
struct BRhs {
    const float *u, *f;
    BCol q;
    size_t pl;
    float vv, dh1, dh2;
    size_t f00;  // BM_RESTRICT: the first of the column's four fine ones
    int nxf;
    __device__ BRhs(const BLevelDesc& L, const float* u_, const float* f_, int col) : u(u_), f(f_) {
        q = bcol(L.nx, L.ny, col);
        pl = (size_t)L.nx * L.ny;
        vv = __ldg(L.v + q.c);
        dh1 = L.krho.dh + vv;
        dh2 = dh1 + vv;
        nxf = 2 * L.nx;
        const int j = (int)(q.c / L.nx), i = (int)(q.c - (size_t)j * L.nx);
        f00 = (size_t)(2 * j) * nxf + 2 * i;
    }
    __device__ __forceinline__ float at(const BLevelDesc& L, int k) const {
        const size_t b = (size_t)k * pl;
        if (MODE == BM_LINE) return f[b + q.c];
        if (MODE == BM_RESTRICT) {
            const float* p = u + 4 * b + f00;
            return 0.25f * ((p[0] + p[1]) + (p[nxf] + p[nxf + 1]));
        }
        const int nz = L.nz;
        const float um0 = u[b - (k > 0 ? pl : 0) + q.c], up0 = u[b + (k + 1 < nz ? pl : 0) + q.c];
        const float um = k > 0 ? um0 : 0.f, up = k + 1 < nz ? up0 : 0.f;
        const float dg = nz == 1 ? L.krho.dh : (k == 0 || k == nz - 1 ? dh1 : dh2);
        return bresidual<SW>(L.krho, dg, vv, f[b + q.c], u[b + q.c], u[b + q.w], u[b + q.e], u[b + q.s], u[b + q.n], um, up);
    }
};

// BF_COLS: out = u + rho M^{-1}(f - A u), rho M^{-1} f, or (u the fine residual) fc = R u, out = rho M^{-1} fc.
// Factors as in sweep_tile.cuh: two tables of nz values behind the planes, or (percol) 1/m_k of the planes before the
// converged ones, which the elimination turns into w_k.
template <int MODE, bool SW>
__device__ void t_cols(const BLevelDesc& L, float rho, const float* u, const float* f, float* fc, float* out, int tile,
                       unsigned char* smem) {
    float* const Z = reinterpret_cast<float*>(smem);
    const int nz = L.nz, kw = L.kw, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, clast = nz >= 2 ? nz - 2 : 0;
    const bool percol = L.percol != 0;
    float* const T = Z + (size_t)nz * 32;
    const BRhs<MODE, SW> R(L, u, f, tile * 32 + lane);
    constexpr bool GF = MODE == BM_SMOOTH && SW;  // the back substitution yields the result
    constexpr int TAB = 0, COL = 1, CONV = 2;     // factors: per-plane table, per column and plane, converged
    const size_t pl = R.pl, c = R.q.c;
    float cw = 0.f;  // the converged w_k (that of plane nz-1 meets x = 0)
    if (percol) {
        for (int k = warp; k < kw; k += BNW) T[k * 32 + lane] = __ldg(L.finv + (size_t)k * pl + c);
        cw = __ldg(L.fw + (size_t)clast * pl + c);
    } else {
        for (int k = threadIdx.x; k < nz; k += BNT) {
            T[k] = __ldg(L.finv + k);
            T[nz + k] = __ldg(L.fw + k);
        }
    }
    constexpr int D = MODE == BM_SMOOTH ? 2 : 4;
    for (int k = warp; k < nz; k += D * BNW) {
        float r[D];
#pragma unroll
        for (int t = 0; t < D; ++t) r[t] = R.at(L, k + t * BNW < nz ? k + t * BNW : k);
#pragma unroll
        for (int t = 0; t < D; ++t) {
            const int kk = k + t * BNW;
            if (kk >= nz) break;
            Z[kk * 32 + lane] = r[t];
            if (MODE == BM_RESTRICT && R.q.act) fc[(size_t)kk * pl + c] = r[t];
        }
    }
    __syncthreads();
    constexpr int KB = 8;
    if (warp == 0) {
        const float vv = R.vv;
        float d = 0.f;
        auto forward = [&](auto kind, int k, int ke, float inv) {
            constexpr int F = decltype(kind)::value;
            auto factor = [&](int kk) { return F == TAB ? T[kk] : (F == COL ? T[kk * 32 + lane] : inv); };
            auto step = [&](int kk, float r, float iv) {
                if (F == COL) T[kk * 32 + lane] = PolF32::mul(vv, iv);
                d = PolF32::mul(PolF32::fma(vv, d, r), iv);
                Z[kk * 32 + lane] = d;
            };
            for (; k + KB <= ke; k += KB) {
                float r[KB], iv[KB];
#pragma unroll
                for (int t = 0; t < KB; ++t) {
                    r[t] = Z[(k + t) * 32 + lane];
                    iv[t] = factor(k + t);
                }
#pragma unroll
                for (int t = 0; t < KB; ++t) step(k + t, r[t], iv[t]);
            }
            for (; k < ke; ++k) step(k, Z[k * 32 + lane], factor(k));
        };
        if (percol) {
            const float cinv = __ldg(L.finv + (size_t)clast * pl + c), einv = __ldg(L.finv + (size_t)(nz - 1) * pl + c);
            forward(std::integral_constant<int, COL>(), 0, kw, 0.f);
            forward(std::integral_constant<int, CONV>(), kw, nz - 1, cinv);
            forward(std::integral_constant<int, CONV>(), nz - 1, nz, einv);
        } else {
            forward(std::integral_constant<int, TAB>(), 0, nz, 0.f);
        }
    }
    if (GF) {
        __syncthreads();
        for (int k = warp; k < nz; k += BNW) {
            const float u0 = u[(size_t)k * pl + c], u1 = u[(size_t)(k + 1 < nz ? k + 1 : k) * pl + c];
            const float w = !percol ? T[nz + k] : (k < kw ? T[k * 32 + lane] : cw);
            Z[k * 32 + lane] = PolF32::fma(-w, k + 1 < nz ? u1 : 0.f, PolF32::fma(rho, Z[k * 32 + lane], u0));
        }
        __syncthreads();
    }
    if (warp == 0) {
        float x = 0.f;
        auto put = [&](int kk, float xk) {
            if (MODE == BM_SMOOTH && !GF) Z[kk * 32 + lane] = xk;
            else if (R.q.act) out[(size_t)kk * pl + c] = GF ? xk : PolF32::mul(rho, xk);
        };
        auto backward = [&](auto kind, int k, int ke) {  // planes k-1 .. ke
            constexpr int F = decltype(kind)::value;
            auto factor = [&](int kk) { return F == TAB ? T[nz + kk] : (F == COL ? T[kk * 32 + lane] : cw); };
            for (; k - KB >= ke; k -= KB) {
                float dk[KB], w[KB];
#pragma unroll
                for (int t = 0; t < KB; ++t) {
                    dk[t] = Z[(k - 1 - t) * 32 + lane];
                    w[t] = factor(k - 1 - t);
                }
#pragma unroll
                for (int t = 0; t < KB; ++t) {
                    x = PolF32::fma(w[t], x, dk[t]);
                    put(k - 1 - t, x);
                }
            }
            for (; k > ke; --k) {
                x = PolF32::fma(factor(k - 1), x, Z[(k - 1) * 32 + lane]);
                put(k - 1, x);
            }
        };
        if (percol) {
            backward(std::integral_constant<int, CONV>(), nz, kw);
            backward(std::integral_constant<int, COL>(), kw, 0);
        } else {
            backward(std::integral_constant<int, TAB>(), nz, 0);
        }
    }
    if (MODE == BM_SMOOTH && !GF) {
        __syncthreads();
        if (R.q.act)
            for (int kk = warp; kk < nz; kk += BNW)
                out[(size_t)kk * pl + c] = PolF32::fma(rho, Z[kk * 32 + lane], u[(size_t)kk * pl + c]);
    }
}

// u_f += P u_c (bilinear, cell centred, periodic). A segment is the 2 x 2 fine cells of one coarse column in one
// plane; where nxc is even, two adjacent ones (16 bytes of both fine rows).
__device__ void t_prolongate(const BLevelDesc& Lf, const float* uc, float* uf, int tile) {
    const int nxc = Lf.nx / 2, nyc = Lf.ny / 2;
    const size_t plc = (size_t)nxc * nyc;
    const bool two = nxc % 2 == 0;
    const int nu = two ? nxc / 2 : nxc;
    const long long n = (long long)nu * nyc * Lf.nz;
    long long id = (long long)tile * BPU + threadIdx.x;
    for (int t = 0; t < BPU / BNT && id < n; ++t, id += BNT) {
        const int kJ = (int)(id / nu), I = (int)(id - (long long)kJ * nu) * (two ? 2 : 1), J = kJ % nyc, k = kJ / nyc;
        const float* cp = uc + (size_t)k * plc;
        float* p0 = uf + (size_t)k * 4 * plc + (size_t)(2 * J) * (2 * nxc) + 2 * I;
        float* p1 = p0 + 2 * nxc;
        const int Im = bwrap(I - 1, nxc), Ip = bwrap(I + (two ? 2 : 1), nxc);
        const float* rows[3] = {cp + (size_t)bwrap(J - 1, nyc) * nxc, cp + (size_t)J * nxc, cp + (size_t)bwrap(J + 1, nyc) * nxc};
        auto val = [](float c, float x, float y, float d) {
            return __fmaf_rn(0.0625f, d, __fmaf_rn(0.1875f, y, __fmaf_rn(0.5625f, c, __fmul_rn(0.1875f, x))));
        };
        if (two) {
            float4 o0 = *reinterpret_cast<const float4*>(p0), o1 = *reinterpret_cast<const float4*>(p1);
            float a[3][4];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const float2 m = *reinterpret_cast<const float2*>(rows[r] + I);
                a[r][0] = rows[r][Im];
                a[r][1] = m.x;
                a[r][2] = m.y;
                a[r][3] = rows[r][Ip];
            }
            o0.x = __fadd_rn(o0.x, val(a[1][1], a[1][0], a[0][1], a[0][0]));
            o0.y = __fadd_rn(o0.y, val(a[1][1], a[1][2], a[0][1], a[0][2]));
            o0.z = __fadd_rn(o0.z, val(a[1][2], a[1][1], a[0][2], a[0][1]));
            o0.w = __fadd_rn(o0.w, val(a[1][2], a[1][3], a[0][2], a[0][3]));
            o1.x = __fadd_rn(o1.x, val(a[1][1], a[1][0], a[2][1], a[2][0]));
            o1.y = __fadd_rn(o1.y, val(a[1][1], a[1][2], a[2][1], a[2][2]));
            o1.z = __fadd_rn(o1.z, val(a[1][2], a[1][1], a[2][2], a[2][1]));
            o1.w = __fadd_rn(o1.w, val(a[1][2], a[1][3], a[2][2], a[2][3]));
            *reinterpret_cast<float4*>(p0) = o0;
            *reinterpret_cast<float4*>(p1) = o1;
        } else {
            const float c = rows[1][I], xm = rows[1][Im], xp = rows[1][Ip];
            p0[0] = __fadd_rn(p0[0], val(c, xm, rows[0][I], rows[0][Im]));
            p0[1] = __fadd_rn(p0[1], val(c, xp, rows[0][I], rows[0][Ip]));
            p1[0] = __fadd_rn(p1[0], val(c, xm, rows[2][I], rows[2][Im]));
            p1[1] = __fadd_rn(p1[1], val(c, xp, rows[2][I], rows[2][Ip]));
        }
    }
}

// u += e (double-word plus FP32), finest level: four cells a thread, their loads before the stores
__device__ void t_correct(const BProbDesc& pb, const float* e, int tile) {
    const BLevelDesc& L = pb.lev[pb.L];
    const size_t n = (size_t)L.nx * L.ny * L.nz, n4 = n / 4;
    const size_t q0 = (size_t)tile * (BCH / 4);
    for (int t = 0; t < BCH / 4 / BNT; ++t) {
        const size_t q = q0 + t * BNT + threadIdx.x;
        if (q >= n4) break;
        float4* pu = reinterpret_cast<float4*>(pb.uD) + 2 * q;
        const float4 a = pu[0], b = pu[1], ev = reinterpret_cast<const float4*>(e)[q];
        auto add = [](float hi, float lo, float x) { return PolDW::add(dw{hi, lo}, PolDW::from_f(x)); };
        const dw r0 = add(a.x, a.y, ev.x), r1 = add(a.z, a.w, ev.y), r2 = add(b.x, b.y, ev.z), r3 = add(b.z, b.w, ev.w);
        pu[0] = make_float4(r0.hi, r0.lo, r1.hi, r1.lo);
        pu[1] = make_float4(r2.hi, r2.lo, r3.hi, r3.lo);
    }
    if (tile == 0 && threadIdx.x < n - 4 * n4) {  // the last one to three cells
        const size_t id = 4 * n4 + threadIdx.x;
        PolDW::st(pb.uD, id, PolDW::add(PolDW::ld_plain(pb.uD, id), PolDW::from_f(e[id])));
    }
}

// per-problem convergence decision after the outer residual (Eq. 10), fixed-order sum
__device__ void t_final(const BatchDesc& d, int prob, int it) {
    const BProbDesc& pb = d.probs[prob];
    // a problem that has finished keeps its iteration count, residual and place in the count of
    // active problems (only this block writes this problem's state, before the next barrier)
    if (!*(volatile int*)&d.state[prob].active) return;
    __shared__ double buf[BNT];
    const int tid = threadIdx.x, nt = BNT;
    double s = 0.0;
    for (int q = tid; q < pb.fine_tiles; q += nt) s += d.partials[pb.part_base + q];
    buf[tid] = s;
    __syncthreads();
    for (int h = nt / 2; h > 0; h >>= 1) {
        if (tid < h) buf[tid] += buf[tid + h];
        __syncthreads();
    }
    if (tid == 0) {
        BState& st = d.state[prob];
        const double nrm = sqrt(buf[0]);
        if (!isfinite(nrm)) {
            st.nonfinite = 1;
            st.active = 0;
            atomicSub(d.n_active, 1);
        } else if (it == 0) {
            st.r0 = nrm;
            st.rel = 1.0;
            st.iters = 0;
            if (pb.history) pb.history[0] = 1.0;
            if (nrm == 0.0) st.converged = 1;
            if (nrm == 0.0 || d.max_iter <= 0) {
                st.active = 0;
                atomicSub(d.n_active, 1);
            }
        } else {
            st.iters = it;
            st.rel = nrm / st.r0;
            if (pb.history) pb.history[it] = st.rel;
            if (st.rel < d.tol) st.converged = 1;
            if (st.rel < d.tol || it >= d.max_iter) {
                st.active = 0;
                atomicSub(d.n_active, 1);
            }
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------- the persistent kernel
__device__ __forceinline__ Lv<PolF32> lv32(const BLevelDesc& b) {
    Lv<PolF32> L;
    L.nx = b.nx;
    L.ny = b.ny;
    L.nz = b.nz;
    L.cx = b.cx;
    L.cy = b.cy;
    L.v = b.v;
    L.finv = b.finv;
    L.fw = b.fw;
    L.fac_percol = b.percol;
    L.variant = -1;
    return L;
}

// Smooth or first line solve of a task on whole-column tiles
template <int MODE, int TR>
__device__ __forceinline__ void tile_task(const BTask& tk, const BLevelDesc& bl, int loc, unsigned char* smem) {
    constexpr int W = TPB / TR / (int)sizeof(float);
    const int tx = bl.nx / W, by = loc / tx, bx = loc - by * tx;
    const float* u = (const float*)(MODE == MODE_LINESOLVE ? tk.b : tk.a);
    if (MODE == MODE_LINESOLVE || bl.k1.iso)
        sweep_tile_body<PolF32, MODE, TR, true, false, false>(lv32(bl), bl.krho, u, (const float*)tk.b, (float*)tk.out, nullptr,
                                                              bl.kw, nullptr, bx, by, 0, 0, smem);
    else
        sweep_tile_body<PolF32, MODE, TR, false, false, false>(lv32(bl), bl.krho, u, (const float*)tk.b, (float*)tk.out, nullptr,
                                                               bl.kw, nullptr, bx, by, 0, 0, smem);
}

__global__ void __launch_bounds__(BNT, 3) k_batched(BatchDesc d) {
    extern __shared__ __align__(16) unsigned char bsmem[];
    constexpr int TB = 128;  // tasks of a phase whose first tiles are kept in shared memory
    __shared__ int base[TB];
    const float rho = (float)d.rho;
    for (int it = 0; it <= d.max_iter; ++it) {
        for (int ph = 0; ph < d.nphase; ++ph) {
            const int tb = d.phase_begin[ph], te = d.phase_begin[ph + 1];
            const int ntiles = d.phase_tiles[ph];
            for (int t = threadIdx.x; t < te - tb && t < TB; t += BNT) base[t] = d.tasks[tb + t].tile_base;
            __syncthreads();
            for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
                // the task owning tile t (tasks of a phase are sorted by tile_base)
                int lo = 0, hi = te - tb - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if ((mid < TB ? base[mid] : d.tasks[tb + mid].tile_base) <= t) lo = mid;
                    else hi = mid - 1;
                }
                const BTask& tk = d.tasks[tb + lo];
                if (tk.type == BT_FINAL) {
                    t_final(d, tk.prob, it);
                    continue;
                }
                if (!*(volatile int*)&d.state[tk.prob].active) continue;
                const int loc = t - tk.tile_base, form = tk.form;
                const BProbDesc& pb = d.probs[tk.prob];
                const BLevelDesc& bl = pb.lev[tk.level];
                const bool sw = bsweeps(bl.nx, bl.ny);
                const float *a = (const float*)tk.a, *b = (const float*)tk.b;
                float *o = (float*)tk.out, *o2 = (float*)tk.out2;
                switch (tk.type) {
                    case BT_OUTRES: {
                        const double s = block_sum(t_residual<PolDW, PolF32, true, true>(bl.nx, bl.ny, bl.nz, pb.kD, pb.vD, pb.uD,
                                                                                   pb.fD, pb.r32, loc));
                        if (threadIdx.x == 0) d.partials[pb.part_base + loc] = s;
                        break;
                    }
                    case BT_LS0:
                        if (form == BF_TILE1) tile_task<MODE_LINESOLVE, 1>(tk, bl, loc, bsmem);
                        else if (form == BF_TILE2) tile_task<MODE_LINESOLVE, 2>(tk, bl, loc, bsmem);
                        else t_cols<BM_LINE, true>(bl, rho, nullptr, b, nullptr, o, loc, bsmem);
                        break;
                    case BT_SMOOTH:
                        if (form == BF_TILE1) tile_task<MODE_SMOOTH, 1>(tk, bl, loc, bsmem);
                        else if (form == BF_TILE2) tile_task<MODE_SMOOTH, 2>(tk, bl, loc, bsmem);
                        else if (sw) t_cols<BM_SMOOTH, true>(bl, rho, a, b, nullptr, o, loc, bsmem);
                        else t_cols<BM_SMOOTH, false>(bl, rho, a, b, nullptr, o, loc, bsmem);
                        break;
                    case BT_RESID:
                        if (sw) t_residual<PolF32, PolF32, true, false>(bl.nx, bl.ny, bl.nz, bl.k1, bl.v, a, b, o, loc);
                        else t_residual<PolF32, PolF32, false, false>(bl.nx, bl.ny, bl.nz, bl.k1, bl.v, a, b, o, loc);
                        break;
                    case BT_RS:
                        t_cols<BM_RESTRICT, true>(bl, rho, a, nullptr, o, o2, loc, bsmem);
                        break;
                    case BT_RRS: {
                        const BLevelDesc& bc = pb.lev[tk.level - 1];
                        const XRestrict<PolF32> xr{lv32(bc), bc.krho.coef, 0.25f, o, o2};
                        const int tx = bl.nx / 128, by = loc / tx, bx = loc - by * tx;
                        if (bl.k1.iso) restrict_tile_body<PolF32, true, false>(lv32(bl), bl.k1, xr, a, b, bc.kw, bx, by, bsmem);
                        else restrict_tile_body<PolF32, false, false>(lv32(bl), bl.k1, xr, a, b, bc.kw, bx, by, bsmem);
                        break;
                    }
                    case BT_PROL:
                        t_prolongate(bl, a, o, loc);
                        break;
                    case BT_CORR:
                        t_correct(pb, a, loc);
                        break;
                    default:
                        break;
                }
                __syncthreads();  // before the next tile takes the shared memory
            }
            if (!grid_barrier(d)) return;
            // after the convergence phase every block sees the same count of active problems
            if (ph == 1 && *(volatile int*)d.n_active == 0) return;
        }
    }
}

// ---------------------------------------------------------------- tasks and launch
// The vector tiles take the levels with the sweeps' arithmetic, all others the 32-column form.
int batched_form(int type, int nx, int ny, int nz, int percol, int kw) {
    if (type != BT_SMOOTH && type != BT_LS0 && type != BT_RRS) return BF_COLS;
    const int tile = nx % 128 == 0 ? BF_TILE1 : BF_TILE2;
    const bool fits = bsweeps(nx, ny) && batched_smem(type, tile, nz, percol, kw) <= (percol ? BTILE_SMEM2 : BTILE_SMEM);
    // (BT_RRS: nx, ny of the fine level, percol and kw of the coarse one)
    if (type == BT_RRS) return fits && tile == BF_TILE1 ? BF_TILE1 : -1;
    return fits ? tile : BF_COLS;
}
size_t batched_smem(int type, int form, int nz, int percol, int kw) {
    const size_t tables = percol ? 0 : 2 * (size_t)nz * sizeof(float);
    if (type == BT_RRS) return (size_t)(nz + (percol ? kw : 0)) * 256 + tables;
    if (type != BT_SMOOTH && type != BT_LS0 && type != BT_RS) return 0;
    if (form == BF_COLS) return (size_t)(nz + (percol ? kw : 0)) * 128 + tables;
    return (size_t)(nz + (percol ? kw : 0)) * TPB + tables;
}
int batched_tiles(int type, int form, int nx, int ny, int nz) {
    const long long cols = (long long)nx * ny;
    auto up = [](long long a, long long b) { return (int)((a + b - 1) / b); };
    switch (type) {
        case BT_SMOOTH:
        case BT_LS0:
        case BT_RS: return up(cols, form == BF_COLS ? 32 : 128);
        case BT_RRS: return nx / 128 * (ny / 2);
        case BT_RESID:
        case BT_OUTRES: return up(cols, BNT) * up(nz, BPZ);
        case BT_PROL: return up((long long)(nx / 2 % 2 == 0 ? nx / 4 : nx / 2) * (ny / 2) * nz, BPU);
        case BT_CORR: return up(cols * nz, BCH);
        default: return 1;
    }
}
int batched_blocks_per_sm(size_t smem) {
    int nb = 0;
    if (cudaFuncSetAttribute(k_batched, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BTILE_SMEM2) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_batched, BNT, smem) != cudaSuccess)
        return 0;
    return nb;
}
cudaError_t launch_batched(const BatchDesc& d, int grid, size_t smem, cudaStream_t s) {
    BatchDesc arg = d;
    void* args[] = {&arg};
    cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_batched, dim3(grid), dim3(BNT), args, smem, s);
    if (e == cudaSuccess) note_launch();
    return e;
}

}  // namespace tpmg
