// panel.cuh -- the cubed-sphere panel operator's level view and launchers (k_panel.cu), used by the
// C-ABI layer. Native FP64, and FP32 for the inner V-cycles of the mixed-precision solve.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "kernels.cuh"

namespace tpmg {

// One multigrid level of the panel operator (Eq. (14)) as the kernels see it, in value type T
// (double or float): nx x ny columns of nz cells, x fastest. Geometry: area[j*nx + i] = |T|;
// ax[j*(nx+1) + i] the coefficient alpha of the x-face between cells i-1 and i of row j (i = 0 and nx:
// the panel boundary); ay[j*nx + i] that of the y-face between rows j-1 and j (j = 0..ny). Radial
// vectors (nz each, shared by the levels): E = a - b - c, B = -b, C = -c with B[0] = C[nz-1] = 0 and
// C[k] = B[k+1]. Thomas factors per cell: inv = 1/m_k, fl = |T| B_k / m_k, fw = |T| C_k / m_k.
template <class T>
struct PanelLvT {
    int nx, ny, nz;
    const T* area;
    const T* ax;
    const T* ay;
    const T* E;
    const T* B;
    const T* C;
    const T* inv;
    const T* fl;
    const T* fw;
    // FP64, small levels (panel_chunked): products of fl and of fw over each chunk of
    // panel_chunk_planes(nz) planes, [chunk][column]; null elsewhere
    const T* wf = nullptr;
    const T* wb = nullptr;
};
typedef PanelLvT<double> PanelLv;

enum { PANEL_SMOOTH = 0, PANEL_RESIDUAL = 1, PANEL_LINESOLVE = 2, PANEL_APPLY = 3 };

// planes per chunk of a column in the chunked sweeps: up to 16 chunks of 4, 8 or 16 planes
inline int panel_chunk_planes(int nz) { return nz <= 64 ? 4 : (nz <= 128 ? 8 : 16); }
// Levels that sweep their columns in chunks: where a thread per column leaves the GPU waiting on its
// recurrences (128^2 x 128 Smooth 193 us with one thread per column at a floor of 36), and not on few planes, where
// the chunks' barriers and second passes outweigh that. Smooth / with the norm, time in chunks over the other form's:
// 72^2 x 4 0.85 / 1.05, x 6 0.71 / 0.95; 128^2 x 8 0.87 / 1.17, x 10 0.76 / 1.02; 152^2 x 10 0.78 / 1.15, x 12 0.66 / 1.01;
// 180^2 x 12 0.92 / 1.36, x 24 0.87 / 1.33, x 32 0.68 / 1.03, x 64 0.73 / 0.97.
inline bool panel_chunked(int nx, int ny, int nz) {
    const size_t cols = (size_t)nx * ny;
    if (cols > (size_t)CHUNK_MAX_COLS) return false;
    return nz >= (cols <= 10240 ? 6 : (cols <= 16384 ? 10 : (cols <= 24576 ? 12 : 32)));
}
// wf, wb: the chunk products, or null
void launch_panel_factors(const PanelLv& L, double* inv, double* fl, double* fw, double* wf, double* wb, cudaStream_t s);
// mode PANEL_*: Smooth (coef = rho) and Residual write partial sums of ||f - A u||^2 when partials is
// non-null; the line solve takes its right-hand side in u and scales by coef. Returns the number of
// thread blocks (= partial sums written).
template <class T>
int launch_panel_sweep(int mode, const PanelLvT<T>& L, double coef, const T* u, const T* f, T* out, double* partials,
                       const int* done, cudaStream_t s);
// r = f - A u in FP64 stored as FP32 (the mixed solve's outer residual), partial sums of ||r||^2
int launch_panel_residual_to_f32(const PanelLv& L, const double* u, const double* f, float* r, double* partials,
                                 const int* done, cudaStream_t s);
template <class T>
void launch_panel_restrict_smooth(const PanelLvT<T>& Lc, double rho, const T* rf, T* fc, T* uc, const int* done,
                                  cudaStream_t s);
template <class T>
void launch_panel_prolongate(int nxc, int nyc, int nz, const T* uc, T* uf, const int* done, cudaStream_t s);
// fused CG kernels on the finest level (Sec. 3.1): SpMV writes one partial sum of <p, q> per block,
// Tridiag those of <r, r> and then of <r, z> (panel_blocks(nx, ny) each)
struct Scalars;
int panel_blocks(int nx, int ny);
void launch_panel_cg_spmv(const PanelLv& L, const Scalars* sc, double* u, double* p, const double* z, double* q,
                          double* partials, cudaStream_t s);
void launch_panel_cg_tridiag(const PanelLv& L, const Scalars* sc, double* r, const double* q, double* z,
                             double* partials, cudaStream_t s);

}  // namespace tpmg
