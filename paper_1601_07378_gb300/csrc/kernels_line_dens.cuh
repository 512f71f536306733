// kernels_line_dens.cuh -- charge density of the line path: rho(r) = sum_n f_n
// |psi_n(r)|^2 over the dense rows (kernels_line.h).
//
// Block (z, group of at most 16 bands): for each band inverse y, then inverse
// x, whose outputs are squared and added in FP32 to the group's partial sums
// [group][z][x][y]; the groups are added in order by the reduction, which also
// turns the grid to [x][y][z].  A pair of warps owns its columns for the whole
// group, so every sum is one thread's, in band order, and stays in L1 / L2
// between the bands (37 KB a z at 96^3).  One transform at a time needs fewer
// registers than the y/x pass: 16 warps an SM at 96^3.  Per 640 bands the pass
// takes 0.77 ms at 96^3 and 1.25 at 100^3, where the inverse y-pass and the
// density x-pass took 1.01 and 2.93.
#pragma once

#include "kernels_impl.cuh"
#include "kernels_line.cuh"

namespace vloc {
namespace line {

constexpr int dens_minb(int n) { return n <= 48 ? 6 : n <= 64 ? 5 : n <= 96 ? 4 : n <= 108 ? 3 : 2; }
template <int CLS, int N1, int N2> struct YXD : YX<CLS, N1, N2> {
    static constexpr int NBB = 1, MINB = dens_minb(N1 > N2 ? N1 : N2);
    static constexpr size_t smem = (size_t)YX<CLS, N1, N2>::SLOT * sizeof(float2);
};

template <int CLS, int N1, int N2>
__global__ void __launch_bounds__(64 * YXD<CLS, N1, N2>::PAIRS, YXD<CLS, N1, N2>::MINB)
    kl_dens(Tables t, const float2* D, int nb, int bpg, const float* occ, long long b_base,
            int pair_mode, long long nreal, float* __restrict__ partial) {
    pdl_begin();
    using C = YXD<CLS, N1, N2>;
    constexpr int M = N1 / 2, Q = N1 / 4, AP = C::AP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, role = (threadIdx.x >> 5) & 1, pair = threadIdx.x >> 6;
    const int z = blockIdx.x, grp = blockIdx.y;
    const int b0 = grp * bpg, b1 = min(nb, b0 + bpg);
    YXStep s;
    s.dband = (long long)t.row * t.n3;
    s.krange = t.krange;
    s.trim = 0;
    s.p0 = 0;
    s.planes = 2 * (N1 / 4) + 1;
    s.nbb = 1;
    float* const pz = partial + ((long long)grp * t.n3 + z) * (N1 * N2);
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        if (b > b0) __syncthreads();  // the last band's columns have been read
        s.d = const_cast<float2*>(D) + b * s.dband + (long long)z * t.row + (N2 / 4) * C::PP;
        yx_body<N2, C, N2, 1>(0, s);
        __syncthreads();
        double wxd, wyd;
        density_weights(occ, b_base + b, pair_mode, nreal, wxd, wyd);
        const float wx = (float)wxd, wy = (float)wyd;
#pragma unroll 1
        for (int l0 = pair * 32; l0 < N2; l0 += C::PAIRS * 32) {
            const bool act = N2 % 32 == 0 || l0 + lane < N2;
            const int c = min(l0 + lane, N2 - 1);
            const float2* ax = reinterpret_cast<const float2*>(smem_raw) + Q * AP + c;
            float2 u[M];
            auto ld = [&](auto k) { return ax[decltype(k)::value * AP]; };
            half_load<N1>(u, ld);
            half_fold<N1>(u, role, ld);
            RDft<M, +1>::run(u);
            if (!act) continue;
            float* q = pz + role * N2 + c;
            if (b == b0) {
                sfor<M>([&](auto j) { q[2 * N2 * decltype(j)::value] = wx * u[j].x * u[j].x + wy * u[j].y * u[j].y; });
            } else {
                sfor<M>([&](auto j) { q[2 * N2 * decltype(j)::value] += wx * u[j].x * u[j].x + wy * u[j].y * u[j].y; });
            }
        }
    }
}

template <int CLS, int N1, int N2>
int launch_dens_n(const Tables& t, const float2* D, long long nb, int bpg, const float* occ, long long b_base, int pair,
                  long long nreal, float* partial, cudaStream_t st) {
    using C = YXD<CLS, N1, N2>;
    if (const cudaError_t e = smem_optin<kl_dens<CLS, N1, N2>>(C::smem)) return (int)e;
    return pdl_launch(kl_dens<CLS, N1, N2>, dim3(t.n3, (unsigned)((nb + bpg - 1) / bpg)), 64 * C::PAIRS, C::smem, st,
        t, D, (int)nb, bpg, occ, b_base, pair, nreal, partial);
}
template <int CLS, int N1>
int LaunchDens<CLS, N1>::run(const Tables& t, const float2* D, long long nb, int bpg, const float* occ, long long b_base,
                             int pair, long long nreal, float* partial, cudaStream_t st) {
    static_assert(yx_partner(CLS, N1, dens_pair), "a length without kernels");
#define VLOC_CASE(N) \
    case N:          \
        if constexpr (dens_pair(CLS, N1, N)) \
            return launch_dens_n<CLS, N1, N>(t, D, nb, bpg, occ, b_base, pair, nreal, partial, st); \
        else break;
    if constexpr (CLS == 0) switch (t.n2) { VLOC_LINE_C48(VLOC_CASE) default: break; }
    if constexpr (CLS == 1) switch (t.n2) { VLOC_LINE_C96(VLOC_CASE) default: break; }
    if constexpr (CLS == 2) switch (t.n2) { VLOC_LINE_C144(VLOC_CASE) default: break; }
#undef VLOC_CASE
    return (int)cudaErrorInvalidValue;
}

}  // namespace line
}  // namespace vloc
