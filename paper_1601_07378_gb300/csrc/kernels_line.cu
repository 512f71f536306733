// kernels_line.cu -- dispatch of the line path (kernels_line.h) and the
// transpose of V that its y/x pass reads.
#include "kernels_line.h"
#include "pdl.cuh"

namespace vloc {
namespace line {

namespace {
bool in_c48(int n) {
    switch (n) {
#define VLOC_CASE(N) case N:
        VLOC_LINE_C48(VLOC_CASE) return true;
        default: return false;
    }
}
bool in_c96(int n) {
    switch (n) {
        VLOC_LINE_C96(VLOC_CASE) return true;
        default: return false;
    }
}
bool in_c144(int n) {
    switch (n) {
        VLOC_LINE_C144(VLOC_CASE) return true;
        default: return false;
    }
}
}  // namespace

int yx_class(int n1, int n2) {
    const int cls = in_c48(n1) && in_c48(n2) ? 0 : in_c96(n1) && in_c96(n2) ? 1 : in_c144(n1) && in_c144(n2) ? 2 : -1;
    return cls >= 0 && yx_pair(cls, n1, n2) ? cls : -1;
}
bool z_length(int n3) {
    switch (n3) {
        VLOC_LINE_Z_A(VLOC_CASE) VLOC_LINE_Z_B(VLOC_CASE) VLOC_LINE_Z_C(VLOC_CASE) VLOC_LINE_Z_D(VLOC_CASE) return true;
        default: return false;
    }
#undef VLOC_CASE
}

// The y/x pass does the same work for a z whatever the sphere; the y- and
// x-passes it replaces do less the fewer planes are occupied, and waste the rest
// of their tiles of 32 z.  Their cost a z is about
//     w (f + 1.1 - 0.2 q),  w = 32 ceil(n3 / 32) / n3,
// in y-passes over all 2 (n1 / 4) + 1 planes, f of which are occupied and q = 1
// where all are (the x-pass then knows them at compile time).  The table has the
// cost, in twentieths, from which the y/x pass is the faster one: 0 where it
// always was.  Gamma pairs cost their z-passes 6 % more.
// Measured with both forms on every cell of these lengths within 1.35 of each
// other, at f = 0.2 to 1, plain and Gamma (1848 pairs of times): always taking
// the line path lost more than 1 % at 460 of them (up to 1.64: 128 x 96 x 96
// with r = 6.5), the rule at 42 (up to 1.06); the density 310 (1.52) and 75 of
// 1752 (1.13); among spheres that fill the smallest axis no more than 1.04.
// Some, us for five launches / line path: 144^3 r = 9.5 568 / 763, r = 36 1068 /
// 1000; 128^3 r = 18.5 617 / 648, r = 32 877 / 800, Gamma 894 / 923; 96^3 r = 8.5
// 529 / 505; 72^3 r = 4.5 644 / 476; density 128^3 r = 18.5 404 / 439, 100^3 r =
// 9.5 758 / 432.
static const struct { unsigned char n1, n2, apply, density; } kPays[] = {
    {24, 24, 41, 0}, {24, 32, 30, 0}, {32, 24, 38, 0}, {32, 32, 31, 0}, {48, 48, 33, 36},
    {48, 60, 0, 30}, {48, 64, 0, 0}, {60, 48, 0, 28}, {60, 60, 0, 0}, {60, 64, 0, 0},
    {60, 72, 0, 0}, {60, 80, 0, 0}, {64, 48, 31, 38}, {64, 60, 30, 35}, {64, 64, 32, 28},
    {64, 72, 29, 39}, {64, 80, 29, 39}, {72, 60, 0, 28}, {72, 64, 0, 0}, {72, 72, 0, 39},
    {72, 80, 0, 31}, {72, 96, 27, 28}, {80, 60, 28, 29}, {80, 64, 25, 0}, {80, 72, 31, 41},
    {80, 80, 27, 33}, {80, 96, 28, 0}, {80, 100, 35, 40}, {96, 72, 35, 38}, {96, 80, 32, 34},
    {96, 96, 28, 26}, {96, 100, 35, 37}, {96, 120, 32, 30}, {96, 128, 32, 28}, {100, 80, 47, 0},
    {100, 96, 39, 0}, {100, 100, 37, 0}, {100, 120, 34, 0}, {100, 128, 37, 0}, {120, 96, 39, 0},
    {120, 100, 37, 0}, {120, 120, 29, 0}, {120, 128, 29, 0}, {120, 144, 34, 0}, {128, 96, 40, 38},
    {128, 100, 37, 59}, {128, 120, 32, 38}, {128, 128, 37, 38}, {128, 144, 37, 56}, {144, 120, 37, 0},
    {144, 128, 40, 0}, {144, 144, 40, 29},
};
bool pays(int n1, int n2, int n3, int planes, bool gamma, bool density) {
    const int all = 2 * (n1 / 4) + 1;
    const double w = 32.0 * ((n3 + 31) / 32) / n3;
    const double cost = w * ((double)planes / all + 1.1 - (planes == all ? 0.2 : 0.0));
    for (const auto& k : kPays)
        if (k.n1 == n1 && k.n2 == n2)
            return 20.0 * cost >= (density ? (double)k.density : k.apply * (gamma ? 1.06 : 1.0));
    return true;
}

// 32 x 32 tiles of (y, z) at one x through shared memory, so that both sides
// are coalesced; 7 MB of traffic at 96^3 (9 us with its launch), once per call.
__global__ void __launch_bounds__(256) k_vt(const float* V, float* __restrict__ VT, int n2, int n3) {
    pdl_begin();
    __shared__ float tile[32][33];
    const int z0 = blockIdx.x * 32, y0 = blockIdx.y * 32, x = blockIdx.z, n1 = gridDim.z;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int j = ty; j < 32; j += 8)
        if (y0 + j < n2 && z0 + tx < n3) tile[j][tx] = V[((long long)x * n2 + y0 + j) * n3 + z0 + tx];
    __syncthreads();
    for (int j = ty; j < 32; j += 8)
        if (z0 + j < n3 && y0 + tx < n2) VT[((long long)(z0 + j) * n1 + x) * n2 + y0 + tx] = tile[tx][j];
}
int launch_vt(const float* V, float* VT, const Tables& t, cudaStream_t st) {
    return pdl_launch(k_vt, dim3((t.n3 + 31) / 32, (t.n2 + 31) / 32, t.n1), 256, 0, st, V, VT, t.n2, t.n3);
}

#define VLOC_CASE_INV(N) case N: return LaunchZ<N>::inv(t, tw3, c, nb, nreal, D, st);
#define VLOC_CASE_FWD(N) case N: return LaunchZ<N>::fwd(t, tw3, D, nb, nreal, out, diag, c, st);
int launch_z_inv(const Tables& t, const float2* tw3, const float2* c, long long nb, long long nreal, float2* D,
                 cudaStream_t st) {
    switch (t.n3) {
        VLOC_LINE_Z_A(VLOC_CASE_INV) VLOC_LINE_Z_B(VLOC_CASE_INV) VLOC_LINE_Z_C(VLOC_CASE_INV) VLOC_LINE_Z_D(VLOC_CASE_INV)
        default: return (int)cudaErrorInvalidValue;
    }
}
int launch_z_fwd(const Tables& t, const float2* tw3, const float2* D, long long nb, long long nreal, float2* out,
                 const float* diag, const float2* c, cudaStream_t st) {
    switch (t.n3) {
        VLOC_LINE_Z_A(VLOC_CASE_FWD) VLOC_LINE_Z_B(VLOC_CASE_FWD) VLOC_LINE_Z_C(VLOC_CASE_FWD) VLOC_LINE_Z_D(VLOC_CASE_FWD)
        default: return (int)cudaErrorInvalidValue;
    }
}
#undef VLOC_CASE_INV
#undef VLOC_CASE_FWD
int launch_dens(const Tables& t, const float2* D, long long nb, int bpg, const float* occ, long long b_base, int pair,
                long long nreal, float* partial, cudaStream_t st) {
#define VLOC_CASE0(N) case N: return LaunchDens<0, N>::run(t, D, nb, bpg, occ, b_base, pair, nreal, partial, st);
#define VLOC_CASE1(N) case N: return LaunchDens<1, N>::run(t, D, nb, bpg, occ, b_base, pair, nreal, partial, st);
#define VLOC_CASE2(N) case N: return LaunchDens<2, N>::run(t, D, nb, bpg, occ, b_base, pair, nreal, partial, st);
    if (t.cls == 0) switch (t.n1) { VLOC_LINE_D48(VLOC_CASE0) default: break; }
    if (t.cls == 1) switch (t.n1) { VLOC_LINE_D96(VLOC_CASE1) default: break; }
    if (t.cls == 2) switch (t.n1) { VLOC_LINE_D144(VLOC_CASE2) default: break; }
#undef VLOC_CASE0
#undef VLOC_CASE1
#undef VLOC_CASE2
    return (int)cudaErrorInvalidValue;
}
// Tiles of 32 (y, z) at one x: the partial sums read along y, the result
// written along z.  Sum over the groups as in k_reduce_partials_f32.
__global__ void __launch_bounds__(256) k_dens_reduce(const float* partial, int ng, int n2, int n3,
                                                     double* __restrict__ acc, int first, float* __restrict__ out) {
    pdl_begin();
    __shared__ float ts[32][33], tc[32][33];
    const int z0 = blockIdx.x * 32, y0 = blockIdx.y * 32, x = blockIdx.z, n1 = gridDim.z;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long N = (long long)n1 * n2 * n3;
    for (int j = ty; j < 32; j += 8) {
        float s = 0.f, c = 0.f;
        if (z0 + j < n3 && y0 + tx < n2) {
            const float* q = partial + ((long long)(z0 + j) * n1 + x) * n2 + y0 + tx;
#pragma unroll 4
            for (int g = 0; g < ng; ++g) {
                const float p = q[g * N];
                const float t = __fadd_rn(s, p);
                const float bp = __fsub_rn(t, s);  // the part of p that t took
                c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(p, bp)));
                s = t;
            }
        }
        ts[j][tx] = s;
        tc[j][tx] = c;
    }
    __syncthreads();
    for (int j = ty; j < 32; j += 8)
        if (y0 + j < n2 && z0 + tx < n3) {
            const long long i = ((long long)x * n2 + y0 + j) * n3 + z0 + tx;
            const double tot = (first ? 0.0 : acc[i]) + ((double)ts[tx][j] + (double)tc[tx][j]);
            if (out) out[i] = (float)tot;
            else acc[i] = tot;
        }
}
int launch_dens_reduce(const Tables& t, const float* partial, int ng, double* acc, int first, float* out,
                       cudaStream_t st) {
    return pdl_launch(k_dens_reduce, dim3((t.n3 + 31) / 32, (t.n2 + 31) / 32, t.n1), 256, 0, st, partial, ng, t.n2,
        t.n3, acc, first, out);
}
int launch_yx(const Tables& t, const float2* tw2, const float* VT, long long nb, float2* D, cudaStream_t st) {
#define VLOC_CASE0(N) case N: return LaunchYX<0, N>::run(t, tw2, VT, nb, D, st);
#define VLOC_CASE1(N) case N: return LaunchYX<1, N>::run(t, tw2, VT, nb, D, st);
#define VLOC_CASE2(N) case N: return LaunchYX<2, N>::run(t, tw2, VT, nb, D, st);
    if (t.cls == 0) switch (t.n1) { VLOC_LINE_C48(VLOC_CASE0) default: break; }
    if (t.cls == 1) switch (t.n1) { VLOC_LINE_C96(VLOC_CASE1) default: break; }
    if (t.cls == 2) switch (t.n1) { VLOC_LINE_C144(VLOC_CASE2) default: break; }
#undef VLOC_CASE0
#undef VLOC_CASE1
#undef VLOC_CASE2
    return (int)cudaErrorInvalidValue;
}

}  // namespace line
}  // namespace vloc
