// k_nn_grad.cu -- parameter gradients of the learned stage's network and the data gradient of its last
// layer (the 16 -> 16 layers' data gradients are the convolutions of k_nn.cu).
//
// Every weight gradient is a GEMM with the cells as its K dimension, dW[co][n] = sum_p dy[p][co] X[p][n]
// with n running over (tap, ci) and X the input shifted by the tap, on mma.sync m16n8k16 with BF16
// operands and FP32 accumulators (M = 16 is all a layer has, far below the 128 rows of a tcgen05 tile).
// The steps (tile of 64 x 8 columns, plane) of the whole grid are numbered tile by tile and dealt to
// the blocks in equal contiguous ranges: each block marches in z through rings of planes fetched two
// planes ahead, and writes one partial per weight and bias at its end (at most 2 blocks per SM, so the
// final reduction reads a few MB).
// Rounding: the tensor cores cut an accumulator's low bits off instead of rounding them, an error that does not
// average out: same-signed sums lose about half a unit in the last place per MMA (2.6e-5 of the sum in 430 of
// them). So no accumulator lives long: the thin layers add each MMA's 16 cells to FP32 sums by ordinary
// additions, the 16 -> 16 layers pass theirs on every D16_FLUSH planes, and biases are ordinary additions,
// FP32 over 32 planes or a tile's and FP64 from there.
#include <cuda_bf16.h>

#include "kernels.cuh"
#include "nn.cuh"

namespace tpmg {

namespace {

constexpr int GX = 64, GY = 8;         // cells of a tile plane in x and y
constexpr int ROWB = 32;               // bytes of a cell's 16 channels

__device__ __forceinline__ int gwrap(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}
__device__ __forceinline__ unsigned gsa(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// 16-byte copy, or 16 zero bytes when !ok (src must still be a valid address)
__device__ __forceinline__ void gcp16(void* dst, const void* src, bool ok) {
    const int bytes = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(gsa(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void gcommit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void gwait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void gldm_t(unsigned addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void gmma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// byte offset of 16-byte half h of 32-byte cell row r: the halves of rows 4..7 (mod 8) swap places, so
// the 8 rows of an ldmatrix phase fall on distinct banks
__device__ __forceinline__ int gswz(int r, int h) { return r * ROWB + ((h ^ ((r >> 2) & 1)) << 4); }

// sum of the four cells that a lane's registers of one row of an A fragment hold
__device__ __forceinline__ float gsum(uint32_t lo, uint32_t hi) {
    return (__uint_as_float(lo << 16) + __uint_as_float(lo & 0xffff0000u)) +
           (__uint_as_float(hi << 16) + __uint_as_float(hi & 0xffff0000u));
}

// the block's contiguous share [s0, s1) of the steps
__device__ __forceinline__ void share(long nsteps, long& s0, long& s1) {
    s0 = nsteps * blockIdx.x / gridDim.x;
    s1 = nsteps * (blockIdx.x + 1) / gridDim.x;
}

}  // namespace

// ---------------------------------------------------------------- 16 -> 16 layers
// Twelve warps: warp w owns the x-shift dx = w / 4 (its nine (dz, dy) taps: 72 accumulators) on the
// 16-cell column w % 4 of the tile. The x rows (B, shifted by dx) are each read once; the dy rows (A)
// they meet, planes k-1 .. k+1 and rows y-1 .. y+1, stay in a rolling 3 x 3 window of fragments that
// takes three new ones per row: 4 ldmatrix for 18 MMAs, against one per tap. The bias gradient adds up
// the dx = 1 warps' dy fragments. Rings: 5 planes of dy (10 rows), 3 of x (66 cells a row). Every D16_FLUSH
// planes (256 MMAs to an accumulator) and at the end the four 16-cell columns add their sums, in order, to the
// block's in shared memory, [x-shift, dz, dy, half of ci][lane][4], 16 bytes a lane.
// Measured on 256^2 x 64 (4.2 M cells, 58 GFLOP): 165 us, the tensor pipe 0.59 busy with one block of 12 warps per SM.
constexpr int D16_NT = 384, D16_DYP = (GY + 2) * GX * ROWB, D16_XP = GY * (GX + 2) * ROWB;
constexpr int D16_RING = 5 * D16_DYP + 3 * D16_XP;
constexpr int D16_OUT = 27 * 256 + 16;  // weights, then biases
constexpr int D16_SMEM = D16_RING + 27 * 256 * (int)sizeof(float);
constexpr int D16_FLUSH = 32;

__global__ void __launch_bounds__(D16_NT) k_dw16_march(const __nv_bfloat16* __restrict__ x,
                                                       const __nv_bfloat16* __restrict__ dy,
                                                       float* __restrict__ partials, int nx, int ny, int nz) {
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* const DY = smem;
    unsigned char* const X = smem + 5 * D16_DYP;
    float* const red = reinterpret_cast<float*>(smem + D16_RING);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dx = warp >> 2, xc = (warp & 3) * 16;
    const int q8 = lane >> 3, rr = lane & 7;
    float acc[3][3][2][4];
    __shared__ double redb[16];
    float b0 = 0.f, b1 = 0.f;  // biases of output channels lane / 4 and 8 + lane / 4
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int d = 0; d < 4; ++d) acc[a][b][c][d] = 0.f;
    for (int q = tid; q < 27 * 256; q += D16_NT) red[q] = 0.f;
    if (tid < 16) redb[tid] = 0.0;
    // this thread's sums to the block's
    auto flush = [&]() {
        for (int c = 0; c < 4; ++c) {
            __syncthreads();
            if ((warp & 3) != c) continue;
#pragma unroll
            for (int dz = 0; dz < 3; ++dz)
#pragma unroll
                for (int t = 0; t < 3; ++t)
#pragma unroll
                    for (int nt = 0; nt < 2; ++nt) {
                        float4* r = reinterpret_cast<float4*>(red) + (((dx * 3 + dz) * 3 + t) * 2 + nt) * 32 + lane;
                        float* a = acc[dz][t][nt];
                        float4 v = *r;
                        v.x += a[0];
                        v.y += a[1];
                        v.z += a[2];
                        v.w += a[3];
                        *r = v;
                        a[0] = a[1] = a[2] = a[3] = 0.f;
                    }
            if (dx == 1) {
                for (int h = 1; h < 4; h <<= 1) {
                    b0 += __shfl_xor_sync(0xffffffffu, b0, h);
                    b1 += __shfl_xor_sync(0xffffffffu, b1, h);
                }
                if ((lane & 3) == 0) {  // (the block's in FP64)
                    redb[lane >> 2] += b0;
                    redb[8 + (lane >> 2)] += b1;
                }
                b0 = b1 = 0.f;
            }
        }
    };
    int since = 0;
    const int tiles_x = nx / GX, tiles_y = (ny + GY - 1) / GY;
    long s0, s1;
    share((long)tiles_x * tiles_y * nz, s0, s1);

    while (s0 < s1) {
        const long tile = s0 / nz;
        const int zb = (int)(s0 % nz), ze = (int)(s1 - s0 < nz - zb ? zb + (s1 - s0) : nz);
        s0 += ze - zb;
        const int x0 = (int)(tile % tiles_x) * GX, y0 = (int)(tile / tiles_x) * GY;
        // planes outside the grid are zero (their dy contributes nothing)
        auto load_dy = [&](int z) {
            const bool in = z >= 0 && z < nz;
            unsigned char* dst = DY + ((z + 1) % 5) * D16_DYP;
            const __nv_bfloat16* src = dy + (size_t)(in ? z : 0) * ny * nx * 16;
            for (int q = tid; q < (GY + 2) * GX * 2; q += D16_NT) {
                const int c = q >> 1, row = c / GX, col = c % GX;
                gcp16(dst + gswz(c, q & 1), src + ((size_t)gwrap(y0 - 1 + row, ny) * nx + x0 + col) * 16 + (q & 1) * 8, in);
            }
        };
        auto load_x = [&](int z) {
            unsigned char* dst = X + (z % 3) * D16_XP;
            const __nv_bfloat16* src = x + (size_t)z * ny * nx * 16;
            for (int q = tid; q < GY * (GX + 2) * 2; q += D16_NT) {
                const int c = q >> 1, row = c / (GX + 2), col = c % (GX + 2);
                const int gi = x0 - 1 + col, i = gi < 0 ? nx - 1 : (gi >= nx ? 0 : gi);
                const bool in = y0 + row < ny;
                gcp16(dst + gswz(c, q & 1), src + ((size_t)(in ? y0 + row : 0) * nx + i) * 16 + (q & 1) * 8, in);
            }
        };
        __syncthreads();  // the previous segment's planes are no longer read
        load_dy(zb - 1);
        load_dy(zb);
        load_dy(zb + 1);
        load_x(zb);
        gcommit();
        if (zb + 1 < ze) {
            load_dy(zb + 2);
            load_x(zb + 1);
        }
        gcommit();
        for (int z = zb; z < ze; ++z) {
            gwait<1>();       // planes of this step (all but the newest group)
            __syncthreads();  // ... of every thread; and the previous step's reads are done
            if (z + 2 < ze) {
                load_dy(z + 3);
                load_x(z + 2);
            }
            gcommit();
            // dy planes z+1, z, z-1 meet taps dz = 0, 1, 2
            unsigned pd[3];
#pragma unroll
            for (int dz = 0; dz < 3; ++dz) pd[dz] = gsa(DY + ((z + 2 - dz) % 5) * D16_DYP);
            const unsigned px = gsa(X + (z % 3) * D16_XP);
            const int acell = xc + (q8 >> 1) * 8 + rr, ah = q8 & 1;   // A = dy^T: stored [cell][co]
            const int bcell = xc + dx + (q8 & 1) * 8 + rr, bh = q8 >> 1;  // B = x: stored [cell][ci]
            uint32_t A[3][3][4];  // [dz][halo row mod 3]
            float p0 = 0.f, p1 = 0.f;  // the plane's bias sums
#pragma unroll
            for (int dz = 0; dz < 3; ++dz)
#pragma unroll
                for (int h = 0; h < 2; ++h) gldm_t(pd[dz] + gswz(h * GX + acell, ah), A[dz][h]);
#pragma unroll
            for (int y = 0; y < GY; ++y) {
                if (y0 + y < ny) {
                    uint32_t B[4];
                    gldm_t(px + gswz(y * (GX + 2) + bcell, bh), B);
#pragma unroll
                    for (int dz = 0; dz < 3; ++dz) gldm_t(pd[dz] + gswz((y + 2) * GX + acell, ah), A[dz][(y + 2) % 3]);
#pragma unroll
                    for (int dz = 0; dz < 3; ++dz)
#pragma unroll
                        for (int t = 0; t < 3; ++t) {  // x row y meets dy row y + 1 - t (halo row y + 2 - t)
                            gmma(acc[dz][t][0], A[dz][(y + 2 - t) % 3], B[0], B[1]);
                            gmma(acc[dz][t][1], A[dz][(y + 2 - t) % 3], B[2], B[3]);
                        }
                    if (dx == 1) {
                        const uint32_t(&a)[4] = A[1][(y + 1) % 3];
                        p0 += gsum(a[0], a[2]);
                        p1 += gsum(a[1], a[3]);
                    }
                }
            }
            b0 += p0;
            b1 += p1;
            if (++since == D16_FLUSH) {
                flush();
                since = 0;
            }
        }
        gwait<0>();
    }
    flush();
    __syncthreads();
    float* const out = partials + (size_t)blockIdx.x * D16_OUT;
    for (int q = tid; q < 27 * 256; q += D16_NT) {  // weight (co, ci, tap): where the fragments keep it
        const int co = q / 432, ci = q / 27 % 16, tap = q % 27;
        const int part = ((tap % 3 * 3 + tap / 9) * 3 + tap / 3 % 3) * 2 + ci / 8;
        out[q] = red[(part * 32 + co % 8 * 4 + ci % 8 / 2) * 4 + co / 8 * 2 + ci % 2];
    }
    if (tid < 16) out[27 * 256 + tid] = (float)redb[tid];
}

// ---------------------------------------------------------------- first and last layer
// The thin layers as the same GEMM. First layer: M = co, A = d1 (16 channels), N = (tap, ci) of the
// input, read at p + d. Last layer (LAST): M = ci, A = a3, N = the 27 taps of d4, read at p - d; d4
// is FP32 and enters as the exact sum of three BF16 parts (8 + 8 + 8 significant bits), one MMA
// each, the smallest first, so nothing of it is rounded. Eight warps, one row of the tile each; A by ldmatrix from a
// 3-plane ring; the thin operand from a 4-plane ring of channel-separated rows, kept twice, once
// shifted by a cell, so that a lane's pair of cells is one aligned word for every x-shift. Bias
// gradients: the sum of the A fragments (first layer), or of d4 as it is loaded (last layer).
// Measured on 256^2 x 64: 65 us (first, cin = 2) and 83 us (last).
template <int CIN, bool LAST>
struct ThinShape {
    static constexpr int NCH = LAST ? 3 : CIN;            // thin rows stored per plane row
    static constexpr int N = LAST ? 27 : 27 * CIN;        // columns of the GEMM
    static constexpr int NTL = (N + 7) / 8;
    static constexpr int AP = GY * GX * ROWB;             // bytes of an A plane
    static constexpr int RS = 72;                         // row stride of the thin ring (bf16)
    static constexpr int CP = (GY + 2) * RS;              // one copy of one channel of a plane
    static constexpr int TP = NCH * 2 * CP;               // bf16 of a thin plane
    static constexpr int SMEM = 3 * AP + 4 * TP * 2;
    static constexpr int OUT = 16 * N + (LAST ? 1 : 16);  // weights, then biases
};

template <int CIN, bool LAST>
__global__ void __launch_bounds__(256) k_dw_thin(const __nv_bfloat16* __restrict__ x, const float* __restrict__ d4,
                                                 const __nv_bfloat16* __restrict__ wide, float* __restrict__ partials,
                                                 int nx, int ny, int nz) {
    typedef ThinShape<CIN, LAST> SH;
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* const AR = smem;
    __nv_bfloat16* const T = reinterpret_cast<__nv_bfloat16*>(smem + 3 * SH::AP);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q8 = lane >> 3, rr = lane & 7, g = lane >> 2, t = lane & 3;
    __shared__ double redb[8][16];
    float acc[SH::NTL][4];
    // biases: of channels lane / 4 and 8 + lane / 4, or (LAST) of this thread's cells; FP32 sums of a tile's planes
    float f0 = 0.f, f1 = 0.f;
    double b0 = 0.0, b1 = 0.0;
    int off[SH::NTL], ddz[SH::NTL];  // word offset within a thin plane, plane offset 0..2, of the lane's columns
#pragma unroll
    for (int j = 0; j < SH::NTL; ++j) {
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
        const int n = 8 * j + g < SH::N ? 8 * j + g : 0;  // columns beyond N repeat column 0 (not stored)
        const int tap = LAST ? n : n / CIN, ch = LAST ? 0 : n % CIN;
        int dz = tap / 9, dyy = (tap / 3) % 3, o = tap % 3;
        if (LAST) {
            dz = 2 - dz;
            dyy = 2 - dyy;
            o = 2 - o;
        }
        ddz[j] = dz;
        off[j] = (ch * 2 + (o == 1)) * (SH::CP / 2) + (warp + dyy) * (SH::RS / 2) + (o == 2) + t;
    }
    const int tiles_x = nx / GX, tiles_y = (ny + GY - 1) / GY;
    long s0, s1;
    share((long)tiles_x * tiles_y * nz, s0, s1);
    constexpr int TC = (GY + 2) * (GX + 2), TPT = (TC + 255) / 256;  // thin cells of a plane, per thread

    while (s0 < s1) {
        const long tile = s0 / nz;
        const int zb = (int)(s0 % nz), ze = (int)(s1 - s0 < nz - zb ? zb + (s1 - s0) : nz);
        s0 += ze - zb;
        const int x0 = (int)(tile % tiles_x) * GX, y0 = (int)(tile / tiles_x) * GY;
        auto load_a = [&](int z) {
            unsigned char* dst = AR + (z % 3) * SH::AP;
            const __nv_bfloat16* src = wide + (size_t)z * ny * nx * 16;
            for (int q = tid; q < GY * GX * 2; q += 256) {
                const int c = q >> 1, row = c / GX, col = c % GX;
                const bool in = y0 + row < ny;
                gcp16(dst + gswz(c, q & 1), src + ((size_t)(in ? y0 + row : 0) * nx + x0 + col) * 16 + (q & 1) * 8, in);
            }
        };
        uint32_t tv[TPT];  // a thin plane on its way from global to shared memory
        auto fetch = [&](int z) {
#pragma unroll
            for (int q = 0; q < TPT; ++q) {
                const int c = tid + q * 256;
                tv[q] = 0;
                if (c < TC && z >= 0 && z < nz) {
                    const int row = c / (GX + 2), gi = x0 - 1 + c % (GX + 2);
                    const size_t p = ((size_t)z * ny + gwrap(y0 - 1 + row, ny)) * nx + (gi < 0 ? nx - 1 : (gi >= nx ? 0 : gi));
                    if (LAST) tv[q] = __float_as_uint(__ldg(d4 + p));
                    else if (CIN == 2) tv[q] = __ldg(reinterpret_cast<const unsigned*>(x) + p);
                    else tv[q] = __ldg(reinterpret_cast<const unsigned short*>(x) + p);
                }
            }
        };
        auto store = [&](int z) {
            __nv_bfloat16* P = T + ((z + 4) & 3) * SH::TP;
#pragma unroll
            for (int q = 0; q < TPT; ++q) {
                const int c = tid + q * 256;
                if (c >= TC) break;
                const int row = c / (GX + 2), col = c % (GX + 2);
                __nv_bfloat16 part[SH::NCH];
                if (LAST) {
                    const float v = __uint_as_float(tv[q]);
                    const bool own = row >= 1 && row <= GY && y0 + row - 1 < ny && col >= 1 && col <= GX;
                    if (own && z >= zb && z < ze) f0 += v;
                    part[0] = __float2bfloat16_rn(v);
                    const float r1 = v - __bfloat162float(part[0]);
                    part[1 % SH::NCH] = __float2bfloat16_rn(r1);
                    part[2 % SH::NCH] = __float2bfloat16_rn(r1 - __bfloat162float(part[1 % SH::NCH]));
                } else {
                    part[0] = __ushort_as_bfloat16((unsigned short)(tv[q] & 0xffff));
                    if (CIN == 2) part[1 % SH::NCH] = __ushort_as_bfloat16((unsigned short)(tv[q] >> 16));
                }
#pragma unroll
                for (int ch = 0; ch < SH::NCH; ++ch) {
                    __nv_bfloat16* r = P + ch * 2 * SH::CP + row * SH::RS;
                    r[col] = part[ch];
                    if (col > 0) r[SH::CP + col - 1] = part[ch];
                }
            }
        };
        __syncthreads();
        for (int z = zb - 1; z <= zb + 1; ++z) {
            fetch(z);
            store(z);
        }
        load_a(zb);
        gcommit();
        if (zb + 1 < ze) load_a(zb + 1);
        gcommit();
        for (int z = zb; z < ze; ++z) {
            gwait<1>();
            __syncthreads();
            if (z + 2 < ze) load_a(z + 2);
            gcommit();
            if (z + 1 < ze) fetch(z + 2);
            if (y0 + warp < ny) {
                const unsigned pa = gsa(AR + (z % 3) * SH::AP);
                float p0 = 0.f, p1 = 0.f;  // the plane's bias sums
                const uint32_t* base[SH::NTL];
#pragma unroll
                for (int j = 0; j < SH::NTL; ++j)
                    base[j] = reinterpret_cast<const uint32_t*>(T + ((z + 3 + ddz[j]) & 3) * SH::TP) + off[j];
#pragma unroll
                for (int c = 0; c < GX / 16; ++c) {
                    uint32_t A[4];
                    gldm_t(pa + gswz(warp * GX + c * 16 + (q8 >> 1) * 8 + rr, q8 & 1), A);
                    float d[SH::NTL][4];
#pragma unroll
                    for (int pc = LAST ? 2 : 0; pc >= 0; --pc) {
                        if (pc != 1)  // (the two small parts share an accumulator)
#pragma unroll
                            for (int j = 0; j < SH::NTL; ++j) d[j][0] = d[j][1] = d[j][2] = d[j][3] = 0.f;
#pragma unroll
                        for (int j = 0; j < SH::NTL; ++j) {
                            const uint32_t* b = base[j] + pc * SH::CP + c * 8;
                            gmma(d[j], A, b[0], b[4]);
                        }
                        if (pc != 2)
#pragma unroll
                            for (int j = 0; j < SH::NTL; ++j)
#pragma unroll
                                for (int e = 0; e < 4; ++e) acc[j][e] += d[j][e];
                    }
                    if (!LAST) {
                        p0 += gsum(A[0], A[2]);
                        p1 += gsum(A[1], A[3]);
                    }
                }
                f0 += p0;
                f1 += p1;
            }
            if (z + 1 < ze) store(z + 2);
        }
        gwait<0>();
        b0 += f0;  // (not in the loop over the planes, where the compiler adds at every one of them: 23 % of the FP64 pipe)
        b1 += f1;
        f0 = f1 = 0.f;
    }
    for (int h = 1; h < (LAST ? 32 : 4); h <<= 1) {
        b0 += __shfl_xor_sync(0xffffffffu, b0, h);
        if (!LAST) b1 += __shfl_xor_sync(0xffffffffu, b1, h);
    }
    if (t == 0) {
        redb[warp][g] = b0;
        redb[warp][8 + g] = b1;
    }
    // the warps' sums add up in shared memory, in order
    float* red = reinterpret_cast<float*>(smem);
    for (int w = 0; w < 8; ++w) {
        __syncthreads();
        if (warp != w) continue;
#pragma unroll
        for (int j = 0; j < SH::NTL; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int m = g + 8 * (e >> 1), n = 8 * j + 2 * t + (e & 1);
                if (n < SH::N) {
                    float* r = red + (LAST ? m * 27 + n : (m * CIN + n % CIN) * 27 + n / CIN);
                    *r = w == 0 ? acc[j][e] : *r + acc[j][e];
                }
            }
    }
    __syncthreads();
    if (tid < SH::OUT - 16 * SH::N) {
        double b = redb[0][tid];
        for (int w = 1; w < 8; ++w) b += redb[w][tid];
        red[16 * SH::N + tid] = (float)b;
    }
    __syncthreads();
    for (int q = tid; q < SH::OUT; q += 256) partials[(size_t)blockIdx.x * SH::OUT + q] = red[q];
}

// out[e] = sum over blocks b of partials[b * nelem + e]: 8 threads per element over b = y, y + 8, ...,
// their sums added in order (double)
__global__ void __launch_bounds__(256) k_reduce_parts(const float* __restrict__ partials, int nblocks, int nelem,
                                                      float* __restrict__ out) {
    __shared__ double red[8][32];
    const int e = blockIdx.x * 32 + threadIdx.x;
    double s = 0.0;
    if (e < nelem)
        for (int b = threadIdx.y; b < nblocks; b += 8) s += partials[(size_t)b * nelem + e];
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && e < nelem) {
        for (int y = 1; y < 8; ++y) s += red[y][threadIdx.x];
        out[e] = (float)s;
    }
}

// ---------------------------------------------------------------- data gradient of the last layer
// d3[ci](p) = mask(a3) * sum_d W4[ci][d] d4(p - d): the transposed 16 <- 1 convolution, FP32, taps in
// ascending order. 432 multiply-adds per cell: a thread owns 2 x 2 cells (32 apart in x, so a warp's accesses stay
// contiguous; two rows share their d4 loads) and reads each weight as part of a 16-byte vector for all four. 136 us
// on 256^2 x 64: the FP32 pipe 0.40 busy, the issue slots 0.63, with a quarter of the warps (116 registers) that wait
// for d4; one cell per thread with a weight load per multiply-add takes 225 us.
__global__ void __launch_bounds__(128) k_bwd_last(const float* __restrict__ d4, const __nv_bfloat16* __restrict__ W,
                                                  const __nv_bfloat16* __restrict__ a3, __nv_bfloat16* __restrict__ d3,
                                                  int nx, int ny, int nz) {
    __shared__ __align__(16) float w[27 * 16];  // [tap][ci]
    for (int q = threadIdx.x; q < 16 * 27; q += 128) w[(q % 27) * 16 + q / 27] = __bfloat162float(W[q]);
    __syncthreads();
    const int hx = nx / 2;  // threads of a row pair
    const size_t t = (size_t)blockIdx.x * 128 + threadIdx.x;
    if (t >= (size_t)hx * (ny / 2) * nz) return;
    const int ip = (int)(t % hx), j0 = 2 * (int)((t / hx) % (ny / 2)), k = (int)(t / ((size_t)hx * (ny / 2)));
    const int i0 = (ip / 32) * 64 + ip % 32;
    int col[2][3], row[4];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int i = i0 + 32 * c + 1 - d;  // i - dx, dx = d - 1
            col[c][d] = i < 0 ? i + nx : (i >= nx ? i - nx : i);
        }
#pragma unroll
    for (int r = 0; r < 4; ++r) row[r] = gwrap(j0 - 1 + r, ny) * nx;
    float acc[2][2][16];  // [y][x][ci]
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int ci = 0; ci < 16; ++ci) acc[a][c][ci] = 0.f;
#pragma unroll 1
    for (int dz = 0; dz < 3; ++dz) {
        const int kk = k + 1 - dz;
        if (kk < 0 || kk >= nz) continue;
        const float* p = d4 + (size_t)kk * ny * nx;
#pragma unroll 1
        for (int dyy = 0; dyy < 3; ++dyy) {
            const int rA = row[dyy == 0 ? 2 : (dyy == 1 ? 1 : 0)], rB = row[dyy == 0 ? 3 : (dyy == 1 ? 2 : 1)];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float g[2][2] = {{__ldg(p + rA + col[0][d]), __ldg(p + rA + col[1][d])},
                                       {__ldg(p + rB + col[0][d]), __ldg(p + rB + col[1][d])}};
                const float4* wt = reinterpret_cast<const float4*>(w + ((dz * 3 + dyy) * 3 + d) * 16);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 wv = wt[q];
#pragma unroll
                    for (int a = 0; a < 2; ++a)
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            acc[a][c][4 * q] = fmaf(wv.x, g[a][c], acc[a][c][4 * q]);
                            acc[a][c][4 * q + 1] = fmaf(wv.y, g[a][c], acc[a][c][4 * q + 1]);
                            acc[a][c][4 * q + 2] = fmaf(wv.z, g[a][c], acc[a][c][4 * q + 2]);
                            acc[a][c][4 * q + 3] = fmaf(wv.w, g[a][c], acc[a][c][4 * q + 3]);
                        }
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const size_t p = ((size_t)k * ny + j0 + a) * nx + i0 + 32 * c;
            __align__(16) __nv_bfloat16 m[16], o[16];
            reinterpret_cast<uint4*>(m)[0] = __ldg(reinterpret_cast<const uint4*>(a3 + p * 16));
            reinterpret_cast<uint4*>(m)[1] = __ldg(reinterpret_cast<const uint4*>(a3 + p * 16) + 1);
#pragma unroll
            for (int ci = 0; ci < 16; ++ci) o[ci] = __float2bfloat16_rn(__bfloat162float(m[ci]) > 0.f ? acc[a][c][ci] : 0.f);
            reinterpret_cast<uint4*>(d3 + p * 16)[0] = reinterpret_cast<uint4*>(o)[0];
            reinterpret_cast<uint4*>(d3 + p * 16)[1] = reinterpret_cast<uint4*>(o)[1];
        }
}

// ---------------------------------------------------------------- launchers
// blocks: `per_sm` per SM, at most one per step
static int grad_blocks(int nx, int ny, int nz, int per_sm) {
    int nsm = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long steps = (long)(nx / GX) * ((ny + GY - 1) / GY) * nz;
    const long nb = (long)nsm * per_sm < NN_GRAD_MAX_BLOCKS ? (long)nsm * per_sm : NN_GRAD_MAX_BLOCKS;
    return (int)(nb < steps ? nb : steps);
}
static void reduce_parts(const float* part, int nb, int nelem, float* out, cudaStream_t s) {
    k_reduce_parts<<<(nelem + 31) / 32, dim3(32, 8), 0, s>>>(part, nb, nelem, out);
    note_launch();
}

void nn_dw16(const __nv_bfloat16* x, const __nv_bfloat16* dy, float* part, float* grad, int nx, int ny, int nz,
             cudaStream_t s) {
    const int nb = grad_blocks(nx, ny, nz, 1);
    cudaFuncSetAttribute(k_dw16_march, cudaFuncAttributeMaxDynamicSharedMemorySize, D16_SMEM);
    k_dw16_march<<<nb, D16_NT, D16_SMEM, s>>>(x, dy, part, nx, ny, nz);
    note_launch();
    reduce_parts(part, nb, D16_OUT, grad, s);
}

template <int CIN, bool LAST>
static void run_thin(const __nv_bfloat16* x, const float* d4, const __nv_bfloat16* wide, float* part, float* grad, int nx,
                     int ny, int nz, cudaStream_t s) {
    typedef ThinShape<CIN, LAST> SH;
    const int nb = grad_blocks(nx, ny, nz, 2);
    cudaFuncSetAttribute(k_dw_thin<CIN, LAST>, cudaFuncAttributeMaxDynamicSharedMemorySize, SH::SMEM);
    k_dw_thin<CIN, LAST><<<nb, 256, SH::SMEM, s>>>(x, d4, wide, part, nx, ny, nz);
    note_launch();
    reduce_parts(part, nb, SH::OUT, grad, s);
}
void nn_dw_first(int cin, const __nv_bfloat16* x, const __nv_bfloat16* d1, float* part, float* grad, int nx, int ny,
                 int nz, cudaStream_t s) {
    if (cin == 1) run_thin<1, false>(x, nullptr, d1, part, grad, nx, ny, nz, s);
    else run_thin<2, false>(x, nullptr, d1, part, grad, nx, ny, nz, s);
}
void nn_dw_last(const __nv_bfloat16* a3, const float* d4, float* part, float* grad, int nx, int ny, int nz,
                cudaStream_t s) {
    run_thin<1, true>(nullptr, d4, a3, part, grad, nx, ny, nz, s);
}
void nn_bwd_last(const float* d4, const __nv_bfloat16* w4, const __nv_bfloat16* a3, __nv_bfloat16* d3, int nx, int ny,
                 int nz, cudaStream_t s) {
    const size_t nt = (size_t)(nx / 2) * (ny / 2) * nz;
    k_bwd_last<<<(unsigned)((nt + 127) / 128), 128, 0, s>>>(d4, w4, a3, d3, nx, ny, nz);
    note_launch();
}

}  // namespace tpmg
