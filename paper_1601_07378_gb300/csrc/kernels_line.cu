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

// 32 x 32 tiles of (y, z) at one x through shared memory, so that both sides
// are coalesced; 7 MB of traffic at 96^3 (about 3 us), once per call.
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
