// k_restrict_tile.cu -- the launch of the fused Residual + RestrictSmooth on whole-column tiles
#include "restrict_tile.cuh"

namespace tpmg {

template <class P, bool ISO>
__global__ void __launch_bounds__(RNT, 2) k_restrict_tile(Lv<P> L, SweepK<P> K, XRestrict<P> xr,
                                                          const typename P::S* __restrict__ u,
                                                          const typename P::S* __restrict__ f, const int* done, int kw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (done && *(volatile const int*)done) return;
    restrict_tile_body<P, ISO, true>(L, K, xr, u, f, kw, blockIdx.x, blockIdx.y, smem_raw);
}

template <class P>
int launch_restrict_tile(const Lv<P>& L, const Lv<P>& Lc, double rho, const typename P::S* u, const typename P::S* f,
                         typename P::S* fc, typename P::S* uc, const int* done, cudaStream_t s) {
    typedef typename P::S S;
    constexpr int W = 512 / (int)sizeof(S), PLANE = 256;
    if (L.nx % W || L.ny % 2 || L.ny / 2 > 65535) return -1;  // (rows of tiles that a launch takes)
    auto al = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
    if (!al(fc) || !al(uc) || (Lc.fac_percol && !al(Lc.finv))) return -1;
    int kw = 0;
    if (Lc.fac_percol) kw = factor_planes(Lc);
    const size_t smem = (size_t)(L.nz + kw) * PLANE + (Lc.fac_percol ? 0 : 2 * (size_t)L.nz * sizeof(S));
    if (smem > 512 * PLANE) return -1;
    const dim3 grd(L.nx / W, L.ny / 2);
    XRestrict<P> xr{Lc, P::hcst(rho), P::hcst(0.25), fc, uc};
    auto run = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 512 * PLANE);
        kern<<<grd, RNT, smem, s>>>(L, sweep_k<P>(L.cx, L.cy, 1.0), xr, u, f, done, kw);
    };
    if (L.cx == L.cy) run(k_restrict_tile<P, true>);
    else run(k_restrict_tile<P, false>);
    note_launch();
    return (int)(grd.x * grd.y);
}
template int launch_restrict_tile<PolF32>(const Lv<PolF32>&, const Lv<PolF32>&, double, const float*, const float*, float*,
                                          float*, const int*, cudaStream_t);
template int launch_restrict_tile<PolDW>(const Lv<PolDW>&, const Lv<PolDW>&, double, const float2*, const float2*, float2*,
                                         float2*, const int*, cudaStream_t);

}  // namespace tpmg
