// FP32 (y, z) convolution of planes whose padded form does not fit one CTA
// (static kernel): one CTA per x-frequency plane.
//
// The route through device memory (k_fft_xf along y, k_fft_zconv, k_fft_xi along
// y) moves 2.2 times the plane three times.  Only the y axis has to be padded to
// hold the plane between the passes: the z rows of a y-transformed plane are
// padded, transformed, multiplied and cropped one at a time, in registers.  So
// M_y x N_z complex values stay in shared memory (512 x 32: 135 KB) and the plane
// is read and written once.  The short transforms, their twiddles and their order
// are those of that route (FourStep<float>), so the results are the same bit for
// bit.
//   Y1, Y2: y pass 1 from global memory, y pass 2, in place on slots k1 N2 + .;
//   Z: a thread takes a row ky = k1 + N1 k2 (slot k1 N2 + k2), its M_z values in
//      registers, kernel values from the kx slice staged in shared memory;
//   V1, V2: inverse y pass A in place, pass B to global memory.
// Slot s starts at s (N_z + 1) + s / N2: the y passes' lanes run along z, the z
// pass's lanes along k1 (slots N2 apart), both on distinct banks.
// 256 threads, one CTA per SM (the z pass holds a padded row in registers): bound
// by the passes' arithmetic and shared-memory latency at 8 warps.  24 grids of
// 256 x 256 x 32: 1.33 ms against 2.11 ms through device memory; 64 of
// 128 x 128 x 32: 1.59 against 2.11 ms; 96 of 64 x 256 x 8: 0.37 against 0.54 ms.
#include <algorithm>

#include "sie_fft.cuh"
#include "sie_plan.h"

namespace sie {
namespace {

constexpr int kThreads = 256;

template <int N1, int N2, int Z1, int Z2> struct LargeGeo {
    static constexpr int My = N1 * N2, Mz = Z1 * Z2, Ny = My / 2, Nz = Mz / 2;
    static constexpr int P = Nz + 1, NS = My * P + N1;                    // float2 in the slots
    static constexpr int HY = My / 2 + 1, HZ = Mz / 2 + 1;                // spectrum slice
    static constexpr size_t smem = size_t(NS) * sizeof(float2) + size_t(2 * Mz) * sizeof(float2) +
                                   size_t(HY * HZ) * sizeof(float);
    static __device__ __forceinline__ int at(int slot) { return slot * P + slot / N2; }
};

// one z row in registers: pad, transform, times h, inverse, crop (rows of P values in shared memory)
template <int Z1, int Z2>
__device__ __forceinline__ void z_row(float2 *row, const float *h, const float2 *tf, const float2 *ti) {
    constexpr int Mz = Z1 * Z2;
    using F = FourStep<float, Z1, Z2>;
    float2 a[Z1][Z2];
#pragma unroll
    for (int j2 = 0; j2 < Z2; ++j2) {
        float2 v[Z1];
#pragma unroll
        for (int j1 = 0; j1 < Z1 / 2; ++j1) v[j1] = row[j2 + Z2 * j1];
        F::fwd1(v, j2, tf);
#pragma unroll
        for (int k1 = 0; k1 < Z1; ++k1) a[k1][j2] = v[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < Z1; ++k1) {
        F::fwd2(a[k1], k1, tf);
#pragma unroll
        for (int k2 = 0; k2 < Z2; ++k2) a[k1][k2] = cscale(a[k1][k2], h[fold_index(k1 + Z1 * k2, Mz)]);
        F::inv1(a[k1], k1, ti);
    }
#pragma unroll
    for (int p2 = 0; p2 < Z2; ++p2) {
        float2 v[Z1];
#pragma unroll
        for (int k1 = 0; k1 < Z1; ++k1) v[k1] = a[k1][p2];
        F::inv2(v, p2, ti);
#pragma unroll
        for (int p1 = 0; p1 < Z1 / 2; ++p1) row[p2 + Z2 * p1] = v[p1];
    }
}

// In place on planes [N_y][N_z] of buf [ngrids][Mx][N_y][N_z]; a CTA takes one kx and
// a run of gpc grids, for which it stages the kx slice of the spectrum Hp
// [fold kx][fold ky][fold kz] and the z twiddles once.
template <int N1, int N2, int Z1, int Z2>
__global__ void __launch_bounds__(kThreads, 1)
    k_plane_large(float2 *__restrict__ buf, int ngrids, int gpc, int lgMx, const float *__restrict__ Hp,
                  const float2 *__restrict__ tfy, const float2 *__restrict__ tiy, const float2 *__restrict__ tfz,
                  const float2 *__restrict__ tiz) {
    using G = LargeGeo<N1, N2, Z1, Z2>;
    using F = FourStep<float, N1, N2>;
    constexpr int Nz = G::Nz;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *S = reinterpret_cast<float2 *>(smem_raw), *s_tf = S + G::NS, *s_ti = s_tf + G::Mz;
    float *Hs = reinterpret_cast<float *>(s_ti + G::Mz);
    const int Mx = 1 << lgMx, kx = blockIdx.x & (Mx - 1);
    const int b0 = (blockIdx.x >> lgMx) * gpc, b1 = min(ngrids, b0 + gpc);
    {
        const float *Hk = Hp + int64_t(fold_index(kx, Mx)) * (G::HY * G::HZ);
        for (int i = threadIdx.x; i < G::HY * G::HZ; i += kThreads) Hs[i] = __ldg(Hk + i);
        for (int i = threadIdx.x; i < G::Mz; i += kThreads) {
            s_tf[i] = __ldg(tfz + i);
            s_ti[i] = __ldg(tiz + i);
        }
    }
    for (int b = b0; b < b1; ++b) {
        float2 *plane = buf + (int64_t(b) * Mx + kx) * (G::Ny * Nz);
        // Y1: columns (z, j2), the loads of a round of items first
        constexpr int NI = Nz * N2, ROUND = NI >= 4 * kThreads ? 4 : NI >= 2 * kThreads ? 2 : 1;
        for (int it0 = threadIdx.x; it0 < NI; it0 += ROUND * kThreads) {
            float2 in[ROUND][N1 / 2];
#pragma unroll
            for (int q = 0; q < ROUND; ++q) {
                const int it = it0 + q * kThreads, z = it % Nz, j2 = it / Nz;
                if (it < NI)
#pragma unroll
                    for (int j1 = 0; j1 < N1 / 2; ++j1) in[q][j1] = plane[(j2 + N2 * j1) * Nz + z];
            }
#pragma unroll
            for (int q = 0; q < ROUND; ++q) {
                const int it = it0 + q * kThreads, z = it % Nz, j2 = it / Nz;
                if (it >= NI) break;
                float2 v[N1];
#pragma unroll
                for (int j1 = 0; j1 < N1 / 2; ++j1) v[j1] = in[q][j1];
                F::fwd1(v, j2, tfy);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1) S[G::at(k1 * N2 + j2) + z] = v[k1];
            }
        }
        __syncthreads();
        for (int it = threadIdx.x; it < Nz * N1; it += kThreads) {   // Y2
            const int z = it % Nz, k1 = it / Nz;
            float2 *c = S + G::at(k1 * N2) + z;
            float2 v[N2];
#pragma unroll
            for (int j2 = 0; j2 < N2; ++j2) v[j2] = c[j2 * G::P];
            F::fwd2(v, k1, tfy);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) c[k2 * G::P] = v[k2];
        }
        __syncthreads();
        for (int ky = threadIdx.x; ky < G::My; ky += kThreads)       // Z
            z_row<Z1, Z2>(S + G::at((ky % N1) * N2 + ky / N1), Hs + fold_index(ky, G::My) * G::HZ, s_tf, s_ti);
        __syncthreads();
        for (int it = threadIdx.x; it < Nz * N1; it += kThreads) {   // V1
            const int z = it % Nz, k1 = it / Nz;
            float2 *c = S + G::at(k1 * N2) + z;
            float2 v[N2];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) v[k2] = c[k2 * G::P];
            F::inv1(v, k1, tiy);
#pragma unroll
            for (int p2 = 0; p2 < N2; ++p2) c[p2 * G::P] = v[p2];
        }
        __syncthreads();
        for (int it = threadIdx.x; it < NI; it += kThreads) {        // V2
            const int z = it % Nz, p2 = it / Nz;
            float2 v[N1];
#pragma unroll
            for (int k1 = 0; k1 < N1; ++k1) v[k1] = S[G::at(k1 * N2 + p2) + z];
            F::inv2(v, p2, tiy);
#pragma unroll
            for (int p1 = 0; p1 < N1 / 2; ++p1) plane[(p2 + N2 * p1) * Nz + z] = v[p1];
        }
        __syncthreads();
    }
}

template <int N1, int N2, int Z1, int Z2>
int launch(pfft_plan *p, float2 *spec, int32_t ngrids, cudaStream_t s) {
    using G = LargeGeo<N1, N2, Z1, Z2>;
    auto kern = k_plane_large<N1, N2, Z1, Z2>;
    if (int rc = set_smem((const void *)kern, G::smem)) return rc;
    int lgMx = 0;
    while ((1 << lgMx) < p->Mx) ++lgMx;
    // grids per CTA: up to 8 share the staged spectrum while eight waves remain
    const int64_t planes = int64_t(ngrids) * p->Mx;
    const int gpc = int(std::max<int64_t>(1, std::min<int64_t>(8, planes / (8 * int64_t(p->sms)))));
    const int64_t ctas = int64_t(p->Mx) * ((ngrids + gpc - 1) / gpc);
    if (ctas > INT32_MAX) return fail(SIE_ERR_ARG, "plane convolution: too many grids");
    kern<<<unsigned(ctas), kThreads, G::smem, s>>>(spec, ngrids, gpc, lgMx, p->d_Hp32, p->d_tf32[1], p->d_ti32[1],
                                                   p->d_tf32[2], p->d_ti32[2]);
    SIE_LAUNCH_CHECK(p);
    return SIE_OK;
}

}  // namespace

// done = false: a size it is not built for (M_y below 256, M_z above 64)
int plane_large_f32(pfft_plan *p, float2 *spec, int32_t ngrids, cudaStream_t s, bool &done) {
    done = true;
    if (p->My == 512 && p->Mz == 16) return launch<16, 32, 4, 4>(p, spec, ngrids, s);
    if (p->My == 512 && p->Mz == 32) return launch<16, 32, 4, 8>(p, spec, ngrids, s);
    if (p->My == 512 && p->Mz == 64) return launch<16, 32, 8, 8>(p, spec, ngrids, s);
    if (p->My == 256 && p->Mz == 64) return launch<16, 16, 8, 8>(p, spec, ngrids, s);
    done = false;
    return SIE_OK;
}

}  // namespace sie
