// k_chunk.cu -- native FP64 kernels of small levels and of grids that fit no tile (f64_columns): columns cut into
// chunks of planes; and the pointwise Residual of every policy.
//
// With a thread per column these levels leave most of the chip waiting on 2 nz dependent FP64 operations
// (about 80 cycles each); cyclic reduction (k_coarse.cu, the other policies) shortens the chain to log2 nz
// steps but takes 2 log2(nz) + 1 operations per cell for the solve alone on a pipe that issues 1/74 of the
// FP32 rate. Here a block owns 8 columns (2 or 4 on the smallest levels), each cut into up to 16 chunks of PP
// planes with a thread per chunk (only those that nz planes have: idle ones would take the pipe all the same,
// 450 x 330 x 4 200 us with all 16), and
// both recurrences of the Thomas algorithm, y_k = b_k / m_k + w_k y_{k-1} and x_k = y_k + w_k x_{k+1}
// (w_k = v / m_k), run twice per chunk: from zero, for the value the chunk hands on, and, once the carried
// value is known (the earlier chunks' values chained by the chunks' products of w_k), for the chunk's own
// values. One more operation per cell and direction (11 for a Smooth), 2 (2 PP + chunks) dependent ones.
// The forward-error bound is that of the Thomas algorithm: the second pass is its recurrence, and the
// carried value's own rounding enters damped by the products, all below 1.
// Measured per Smooth inside a graph: 64^2 x 128 16 us (cyclic reduction 30), 128^2 x 128 49 us (thread per
// column 72), 64^2 x 64 10 us (17); 300 x 150 x 60 with the norm 116 us, 185 with a thread per column.
#include <algorithm>

#include "kernels.cuh"

namespace tpmg {

namespace {

constexpr int CH = 16;  // chunks of a column

__device__ __forceinline__ int kwrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

struct CCol {
    int i, j;
    bool act;
    size_t c, w, e, s, n;  // in-plane offsets of the column and its neighbours
};
__device__ __forceinline__ CCol chunk_col(int nx, int ny, int col) {
    CCol q;
    q.act = col < nx * ny;
    const int cc = q.act ? col : 0;
    q.i = cc % nx;
    q.j = cc / nx;
    q.c = cc;
    q.w = (size_t)q.j * nx + kwrap(q.i - 1, nx);
    q.e = (size_t)q.j * nx + kwrap(q.i + 1, nx);
    q.s = (size_t)kwrap(q.j - 1, ny) * nx + q.i;
    q.n = (size_t)kwrap(q.j + 1, ny) * nx + q.i;
    return q;
}
// The value carried into chunk w of a column (lane = 2 w + column) from what the chunks before (UP) or behind
// it hand on, e, and their products of multipliers, cw (0 beyond the column)
template <bool UP>
__device__ __forceinline__ double chunk_scan(double e, double cw, int w) {
#pragma unroll
    for (int d = 1; d < CH; d *= 2) {
        const double ee = UP ? __shfl_up_sync(0xffffffffu, e, 2 * d) : __shfl_down_sync(0xffffffffu, e, 2 * d);
        const double cc = UP ? __shfl_up_sync(0xffffffffu, cw, 2 * d) : __shfl_down_sync(0xffffffffu, cw, 2 * d);
        if (UP ? w >= d : w + d < CH) {
            e = fma(cw, ee, e);
            cw *= cc;
        }
    }
    const double c = UP ? __shfl_up_sync(0xffffffffu, e, 2) : __shfl_down_sync(0xffffffffu, e, 2);
    return (UP ? w == 0 : w == CH - 1) ? 0.0 : c;
}
// f + cx (u_w + u_e) + cy (u_s + u_n) (sweep_rhs's form)
__device__ __forceinline__ double chunk_rhs(const double* __restrict__ u, const CCol& q, double fk, double cx, double cy) {
    return fma(cy, __ldg(u + q.s) + __ldg(u + q.n), fma(cx, __ldg(u + q.w) + __ldg(u + q.e), fk));
}

}  // namespace

// product of w_k over each chunk of pp planes, [chunk][column] (lambda^2 varying) or [chunk]
__global__ void __launch_bounds__(128) k_chunk_products(Lv<PolF64> L, double* __restrict__ out, int pp) {
    const int ncol = L.fac_percol ? L.nx * L.ny : 1, col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= ncol) return;
    double p = 1.0;
    for (int k = 0; k < L.nz; ++k) {
        p *= L.fw[(size_t)k * ncol + col];
        if ((k + 1) % pp == 0 || k + 1 == L.nz) {
            out[(size_t)(k / pp) * ncol + col] = p;
            p = 1.0;
        }
    }
}

// MODE 0 Smooth: out = u + coef M^{-1}(f - A u); NORM with the partial sums of ||f - A u||^2, without them in
// the form (1 - coef) u + coef M^{-1}(f + H u). MODE 1 line solve: out = coef M^{-1} u. MODE 2 RestrictSmooth:
// fc = R u (u the fine residual in PF's storage), out = coef M^{-1} fc.
template <class PF, int MODE, int PP, bool NORM, int CB>
__global__ void __launch_bounds__(CB * CH) k_chunk(Lv<PolF64> L, double coef, const typename PF::S* __restrict__ uin,
                                                   const double* __restrict__ f, double* __restrict__ out,
                                                   double* __restrict__ fc, double* partials, const int* done) {
    __shared__ double sy[CH][CB], sx[CH][CB];
    if (done && *(volatile const int*)done) return;
    const double* u = reinterpret_cast<const double*>(uin);  // (MODE 2 reads uin)
    const int tx = threadIdx.x, w = threadIdx.y, nz = L.nz, k0 = w * PP;
    const CCol q = chunk_col(L.nx, L.ny, blockIdx.x * CB + tx);
    const size_t pl = (size_t)L.nx * L.ny;
    const int np = !q.act || k0 >= nz ? 0 : (nz - k0 < PP ? nz - k0 : PP);  // planes of this thread
    // Every load is unconditional (planes beyond the column repeat its last one), so that a pass's loads
    // are in flight together; planes beyond np get a = w = 0 and leave both chains at zero.
    const size_t fs = L.fac_percol ? pl : 1, fo = L.fac_percol ? q.c : 0;  // factors of plane k at k * fs + fo
    double a[PP], wk[PP], y = 0.0, acc = 0.0;
    {
        const int kf = k0 < nz ? k0 : nz - 1;
        double um = 0.0, uc = 0.0, vv = 0.0, dh1 = 0.0, dh2 = 0.0;
        if (MODE == 0 && NORM) {
            uc = __ldg(u + (size_t)kf * pl + q.c);
            um = __ldg(u + (size_t)(kf > 0 ? kf - 1 : 0) * pl + q.c);
            if (kf == 0) um = 0.0;
            vv = __ldg(L.v + q.c);
            dh1 = (1.0 + 2.0 * L.cx + 2.0 * L.cy) + vv;
            dh2 = dh1 + vv;
        }
#pragma unroll
        for (int p = 0; p < PP; ++p) {
            const bool in = p < np;
            const int k = k0 + p < nz ? k0 + p : nz - 1;
            const size_t b = (size_t)k * pl, id = b + q.c;
            double r;
            if (MODE == 0) {
                r = chunk_rhs(u + b, q, __ldg(f + id), L.cx, L.cy);
                if (NORM) {
                    double up = __ldg(u + (k + 1 < nz ? id + pl : id));
                    if (k + 1 == nz) up = 0.0;
                    const double dg = nz == 1 ? dh1 - vv : (k == 0 || k == nz - 1 ? dh1 : dh2);
                    r = fma(vv, um + up, fma(-dg, uc, r));
                    if (in) acc = fma(r, r, acc);
                    um = uc;
                    uc = up;
                }
            } else if (MODE == 2) {
                typedef Conv<PF, PolF64> CV;
                const size_t nxf = 2 * (size_t)L.nx, c0 = (size_t)k * 4 * pl + (size_t)(2 * q.j) * nxf + 2 * q.i;
                r = 0.25 * ((CV::f(PF::ld(uin, c0)) + CV::f(PF::ld(uin, c0 + 1))) +
                            (CV::f(PF::ld(uin, c0 + nxf)) + CV::f(PF::ld(uin, c0 + nxf + 1))));
                if (in) fc[id] = r;
            } else {
                r = __ldg(u + id);
            }
            const double iv = __ldg(L.finv + (size_t)k * fs + fo), wv = __ldg(L.fw + (size_t)k * fs + fo);
            a[p] = in ? r * iv : 0.0;
            wk[p] = in ? wv : 0.0;
        }
    }
#pragma unroll
    for (int p = 0; p < PP; ++p) y = fma(wk[p], y, a[p]);
    const double* cw = L.chunkw + fo;  // the chunks' products
    const int last = (nz - 1) / PP;
    double cwc = 0.0, pw[CB == 2 ? 1 : CH];
    if constexpr (CB == 2) {  // a warp holds all chunks of its two columns: a scan of four steps
        if (w <= last) cwc = __ldg(cw + (size_t)w * fs);
        y = chunk_scan<true>(y, cwc, w);
    } else {
        if (w == 0) {
#pragma unroll
            for (int c = 0; c < CH; ++c) pw[c] = __ldg(cw + (size_t)(c <= last ? c : 0) * fs);
        }
        sy[w][tx] = y;
        __syncthreads();
        if (w == 0) {  // one thread per column: each chunk's carried value in the place of what it hands on
            y = 0.0;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                if (c > last) break;
                const double e = sy[c][tx];
                sy[c][tx] = y;
                y = fma(pw[c], y, e);
            }
        }
        __syncthreads();
        y = sy[w][tx];
    }
#pragma unroll
    for (int p = 0; p < PP; ++p) {
        y = fma(wk[p], y, a[p]);
        a[p] = p < np ? y : 0.0;
    }
    double x = 0.0;
#pragma unroll
    for (int p = PP - 1; p >= 0; --p) x = fma(wk[p], x, a[p]);
    double uo[MODE == 0 ? PP : 1];
    if (MODE == 0) {
#pragma unroll
        for (int p = 0; p < PP; ++p) uo[p] = __ldg(u + (size_t)(k0 + p < nz ? k0 + p : nz - 1) * pl + q.c);
    }
    if constexpr (CB == 2) {
        x = chunk_scan<false>(x, cwc, w);
    } else {
        sx[w][tx] = x;
        __syncthreads();
        if (w == 0) {
            x = 0.0;
#pragma unroll
            for (int c = CH - 1; c >= 0; --c) {
                if (c > last) continue;
                const double e = sx[c][tx];
                sx[c][tx] = x;
                x = fma(pw[c], x, e);
            }
        }
        __syncthreads();
        x = sx[w][tx];
    }
    const double keep = 1.0 - coef;
#pragma unroll
    for (int p = PP - 1; p >= 0; --p) {
        x = fma(wk[p], x, a[p]);
        if (p < np) out[(size_t)(k0 + p) * pl + q.c] = MODE == 0 ? fma(coef, x, NORM ? uo[p] : keep * uo[p]) : coef * x;
    }
    if (MODE == 0 && NORM) {
        const double s = block_sum(acc);
        if (tx == 0 && w == 0) partials[blockIdx.x] = s;
    }
}

// Residual, pointwise: planes blockIdx.y * pz .. of a column per thread, the sweeps' arithmetic in its order
// (sweep_residual), so the same bits as their Residual. On levels of few tiles the marching Residual has one
// chain per column: 128^2 x 128 FP64 110 us, 34 here; FP32 17 / 8.7; double-word 78 / 62
// (both with its conversions).
template <class P, class PO>
__global__ void __launch_bounds__(128) k_residual_point(Lv<P> L, SweepK<P> K, const typename P::S* __restrict__ u,
                                                        const typename P::S* __restrict__ f,
                                                        typename PO::S* __restrict__ r, double* partials,
                                                        const int* done, int pz) {
    typedef typename P::R R;
    if (done && *(volatile const int*)done) return;
    const CCol q = chunk_col(L.nx, L.ny, blockIdx.x * 128 + threadIdx.x);
    const size_t pl = (size_t)L.nx * L.ny;
    const int nz = L.nz, k0 = blockIdx.y * pz, k1 = k0 + pz < nz ? k0 + pz : nz;
    typename P::Acc acc = 0, cmp = 0;
    if (q.act && k0 < k1) {
        const R vv = P::ld(L.v, q.c), dh1 = P::add(K.dh, vv), dh2 = P::add(dh1, vv);
        const bool iso = K.iso != 0;
        R um = k0 > 0 ? P::ld(u, (size_t)(k0 - 1) * pl + q.c) : P::zero(), uc = P::ld(u, (size_t)k0 * pl + q.c);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
            const size_t b = (size_t)k * pl;
            const R up = k + 1 < nz ? P::ld(u, b + pl + q.c) : P::zero();
            const R dg = nz == 1 ? K.dh : (k == 0 || k == nz - 1 ? dh1 : dh2);
            const R rk = sweep_residual<P>(P::ld(f, b + q.c), dg, uc, P::ld(u, b + q.w), P::ld(u, b + q.e),
                                           P::ld(u, b + q.s), P::ld(u, b + q.n), um, up, K.cx, K.cy, vv, iso);
            if constexpr (PO::id == P::id)
                PO::st(reinterpret_cast<typename PO::S*>(r), b + q.c, rk);
            else
                PO::st(r, b + q.c, PO::from_f(P::to_f(rk)));
            if (partials) P::acc_dot(acc, cmp, rk, rk);
            um = uc;
            uc = up;
        }
    }
    if (partials) {
        const double s = block_sum(P::acc_get(acc, cmp));
        if (threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------- launchers
// 16 chunks of 4, 8 or 16 planes
int chunk_planes(int nz) { return nz <= 4 * CH ? 4 : (nz <= 8 * CH ? 8 : 16); }

size_t chunk_count(const Lv<PolF64>& L) {
    return (size_t)((L.nz + chunk_planes(L.nz) - 1) / chunk_planes(L.nz)) * (L.fac_percol ? (size_t)L.nx * L.ny : 1);
}

void launch_chunk_products(const Lv<PolF64>& L, double* out, cudaStream_t s) {
    const int ncol = L.fac_percol ? L.nx * L.ny : 1;
    k_chunk_products<<<(ncol + 127) / 128, 128, 0, s>>>(L, out, chunk_planes(L.nz));
    note_launch();
}

template <class PF, int MODE, int PP, int CB>
static int run_chunk_cb(const Lv<PolF64>& L, double coef, const typename PF::S* u, const double* f, double* out, double* fc,
                        double* partials, const int* done, cudaStream_t s) {
    const int nb = (L.nx * L.ny + CB - 1) / CB;
    // the chunks that the column has, in whole warps (the scan of CB == 2 takes all of its warp)
    constexpr int WR = 32 / CB;
    const int rows = ((L.nz + PP - 1) / PP + WR - 1) / WR * WR;
    const dim3 b(CB, CB == 2 ? CH : rows);
    if (MODE == 0 && partials)
        k_chunk<PF, MODE, PP, MODE == 0, CB><<<nb, b, 0, s>>>(L, coef, u, f, out, fc, partials, done);
    else
        k_chunk<PF, MODE, PP, false, CB><<<nb, b, 0, s>>>(L, coef, u, f, out, fc, nullptr, done);
    note_launch();
    return nb;
}
// columns per block: 8, fewer where the blocks would not reach every SM
template <class PF, int MODE, int PP>
static int run_chunk(const Lv<PolF64>& L, double coef, const typename PF::S* u, const double* f, double* out, double* fc,
                     double* partials, const int* done, cudaStream_t s) {
    if (L.nx * L.ny <= 512) return run_chunk_cb<PF, MODE, PP, 2>(L, coef, u, f, out, fc, partials, done, s);
    if (L.nx * L.ny <= 2048) return run_chunk_cb<PF, MODE, PP, 4>(L, coef, u, f, out, fc, partials, done, s);
    return run_chunk_cb<PF, MODE, PP, 8>(L, coef, u, f, out, fc, partials, done, s);
}
template <class PF, int MODE>
static int chunk_sweep(const Lv<PolF64>& L, double coef, const typename PF::S* u, const double* f, double* out, double* fc,
                       double* partials, const int* done, cudaStream_t s) {
    if (!L.chunkw) return -1;
    switch (chunk_planes(L.nz)) {
        case 4: return run_chunk<PF, MODE, 4>(L, coef, u, f, out, fc, partials, done, s);
        case 8: return run_chunk<PF, MODE, 8>(L, coef, u, f, out, fc, partials, done, s);
        default: return run_chunk<PF, MODE, 16>(L, coef, u, f, out, fc, partials, done, s);
    }
}

int launch_smooth_chunk(const Lv<PolF64>& L, double rho, const double* u, const double* f, double* uo, double* partials,
                        const int* done, cudaStream_t s) {
    return chunk_sweep<PolF64, 0>(L, rho, u, f, uo, nullptr, partials, done, s);
}
int launch_line_solve_chunk(const Lv<PolF64>& L, const double* b, double* x, double scale, const int* done, cudaStream_t s) {
    return chunk_sweep<PolF64, 1>(L, scale, b, nullptr, x, nullptr, nullptr, done, s);
}
template <class PF>
int launch_restrict_smooth_chunk(const Lv<PolF64>& Lc, double rho, const typename PF::S* rf, double* fc, double* uc,
                                 const int* done, cudaStream_t s) {
    // larger coarse levels with tiles: the column sweep, whose values the fused Residual + RestrictSmooth
    // reproduces
    if ((size_t)Lc.nx * Lc.ny > (size_t)PCR_MAX_COLS && Lc.nx % 32 == 0) return -1;
    return chunk_sweep<PF, 2>(Lc, rho, rf, nullptr, uc, fc, nullptr, done, s);
}
template int launch_restrict_smooth_chunk<PolF64>(const Lv<PolF64>&, double, const double*, double*, double*, const int*,
                                                  cudaStream_t);
template int launch_restrict_smooth_chunk<PolDW>(const Lv<PolF64>&, double, const float2*, double*, double*, const int*,
                                                 cudaStream_t);

// Planes per thread of the residual. Small levels: one where that gives at most 1024 blocks (a thread that takes four
// planes waits for memory four times: FP64 32^2 x 32 3.5 us, 2.6 with one), two or four where that does; with the norm at
// most 256 where four planes allow it (the sum over the blocks is one block's work: FP64 64^2 x 29 8.9 us with 928
// blocks, 7.7 with 256). Else as many as leave 16 blocks per 128 columns (room for one partial sum per 8 columns,
// max_partials), and above CHUNK_MAX_COLS columns, where the columns alone fill the GPU, 4.
static int residual_planes(int nx, int ny, int nz, bool norm) {
    if ((size_t)nx * ny > (size_t)CHUNK_MAX_COLS) return (nz + 3) / 4;
    const int cb = (nx * ny + 127) / 128;
    auto slabs = [&](int p) { return (nz + p - 1) / p; };
    int p = 1;
    while (p < 4 && cb * slabs(p) > (norm ? 256 : 1024)) p *= 2;
    if (cb * slabs(p) > 1024) p = std::max(4, (nz + 15) / 16);
    return slabs(slabs(p));  // in equal parts
}

template <class P>
int residual_point_blocks(const Lv<P>& L) {
    const int pz = residual_planes(L.nx, L.ny, L.nz, true);
    return (L.nx * L.ny + 127) / 128 * ((L.nz + pz - 1) / pz);
}
template <class P, class PO>
int launch_residual_point(const Lv<P>& L, const typename P::S* u, const typename P::S* f, typename PO::S* r,
                          double* partials, const int* done, cudaStream_t s) {
    const int pz = residual_planes(L.nx, L.ny, L.nz, partials != nullptr);
    const dim3 g((L.nx * L.ny + 127) / 128, (L.nz + pz - 1) / pz);
    k_residual_point<P, PO><<<g, 128, 0, s>>>(L, sweep_k<P>(L.cx, L.cy, 1.0), u, f, r, partials, done, pz);
    note_launch();
    return (int)(g.x * g.y);
}
#define TPMG_POINT_INST(P, PO)                                                                              \
    template int launch_residual_point<P, PO>(const Lv<P>&, const P::S*, const P::S*, PO::S*, double*, const int*, \
                                              cudaStream_t);
TPMG_POINT_INST(PolF64, PolF64)
TPMG_POINT_INST(PolF32, PolF32)
TPMG_POINT_INST(PolF32B, PolF32B)
TPMG_POINT_INST(PolDW, PolDW)
TPMG_POINT_INST(PolDW, PolF32)
template int residual_point_blocks<PolF64>(const Lv<PolF64>&);
template int residual_point_blocks<PolF32>(const Lv<PolF32>&);
template int residual_point_blocks<PolF32B>(const Lv<PolF32B>&);
template int residual_point_blocks<PolDW>(const Lv<PolDW>&);

}  // namespace tpmg
