// kernels_line.cuh -- the y/x pass of the line path (kernels_line.h).
//
// Every 1-D transform of length N is two half transforms of M = N / 2 points,
// each held in one thread's registers (line_dft.cuh): with inputs only at
// |k| <= N / 4, x[n] and x[n + M] are never both nonzero (but for n = N / 4),
// so the even outputs are the M-point DFT of u[n] = x[n] or x[n - M] and the
// odd outputs that of u[n] w^k, and neither half needs a butterfly with the
// other.  The forward transform runs the same way back: X[k] = E[n] + w^-n
// O[n] for k = n >= 0 and E[n] - w^-n O[n] for k = n - M < 0, one addition per
// kept output.  Role 0 is the even half, role 1 the odd; a pair of warps with
// the same lanes' lines does the two roles.
//
// What bounds the pass at 96^3: 12 warps an SM (168 registers) keep the FMA
// pipe 53 % and the issue slots 54 % busy, the rest goes to barriers, shared
// memory and V's loads; 2.28 ms per 1024 bands, where the inverse y-, x- and
// forward y-pass of the five-launch chain take 3.03 at the copy bandwidth.
// Measured slower: quarter lines on four lanes with shuffles (20 warps an SM,
// but 65 % of the load/store wavefronts: 4.3 ms), 128 registers and 16 warps
// (spills, and 3 column groups over 2 pairs: 2.46), 6 warps a block (two
// schedulers get twice the warps: 2.4-2.7), a queue of line groups over the
// pairs of one persistent block (all phases' code live at once: 5.0).
#pragma once

#include "fft_core.cuh"
#include "kernels_line.h"
#include "line_dft.cuh"
#include "pdl.cuh"
#include "smem_optin.cuh"

namespace vloc {
namespace line {

__device__ __forceinline__ void bar_pair(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

// *p if lim >= k (k a constant), else 0; and the store: one compare and one
// predicated access each (the compiler's own form branches around every load).
// Volatile with a memory clobber: the dense rows are another launch's output
// (pdl.cuh) and the step's own, so their loads keep their place among barriers
// and stores.
template <int k> __device__ __forceinline__ float2 ld_if_ge(const float2* p, int lim) {
    float2 v;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ge.s32 q, %3, %4;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
                 "@q ld.global.v2.f32 {%0, %1}, [%2];\n\t}"
                 : "=&f"(v.x), "=&f"(v.y)
                 : "l"(p), "r"(lim), "n"(k)
                 : "memory");
    return v;
}
template <int k> __device__ __forceinline__ void st_if_ge(float2* p, float2 v, int lim) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ge.s32 q, %3, %4;\n\t@q st.global.v2.f32 [%2], {%0, %1};\n\t}" ::"f"(v.x),
                 "f"(v.y), "l"(p), "r"(lim), "n"(k)
                 : "memory");
}

// signed index of half-transform element n
template <int N> constexpr int kof(int n) { return n <= N / 4 ? n : n - N / 2; }
// u <- half inputs of `role` from ld(k), k a compile-time constant
template <int N, class L> __device__ __forceinline__ void half_load(float2 (&u)[N / 2], const L& ld) {
    sfor<N / 2>([&](auto n) { u[n] = ld(std::integral_constant<int, kof<N>(decltype(n)::value)>{}); });
}
template <int N, class L> __device__ __forceinline__ void half_fold(float2 (&u)[N / 2], int role, const L& ld) {
    constexpr int M = N / 2, Q = N / 4;
    if constexpr (2 * Q == M) {  // k = Q and k = -Q are the same element
        const float2 b = ld(std::integral_constant<int, -Q>{});
        u[Q] = role ? csub(u[Q], b) : cadd(u[Q], b);
    }
    if (role) sfor<M>([&](auto n) { u[n] = Tw<N, +1, kof<N>(decltype(n)::value)>::mul(u[n]); });
}

// ------------------------------------------------------------- y/x pass
// Configuration for n1 = N1, n2 = N2 of size class CLS: pitch PP of the dense
// rows, pitch AP and slot SLOT of the shared (plane, column) array, NBB bands
// per step (two where their slots leave room for MINB blocks: the 3 column
// groups of each 96-point band then divide evenly over the pairs), PAIRS warp
// pairs per block, MINB blocks per SM (by the registers of an M-point line: 2
// M and about 40 more; a cap below that spills and measured slower, 1.87 ->
// 2.20 ms at 128^3, 0.37 -> 0.40 at 80^3 x 256).
constexpr int yx_minb(int n) {
    return n <= 48 ? 6 : n <= 64 ? 5 : n <= 72 ? 4 : n <= 108 ? 3 : 2;
}
template <int CLS, int N1, int N2> struct YX {
    static constexpr int NM = N1 > N2 ? N1 : N2;
    static constexpr int PP = class_pitch(CLS), AP = N2 | 1, SLOT = (2 * (N1 / 4) + 1) * AP;
    static constexpr int NBB = yx_bands(N1, N2), PAIRS = 2, MINB = yx_minb(NM);
    static constexpr size_t smem = (size_t)NBB * SLOT * sizeof(float2);
};

struct YXStep {
    float2* d;           // dense rows of this z, band 0 of the step, at k = 0, h = -n1/4
    long long dband;     // dense elements per band
    const float* v;      // VT of this z
    const int2* krange;
    const float2* tw2;   // exp(2 pi i j / n2)
    int nbb, p0, planes, trim;  // planes [p0, p0 + planes) as lines, `trim` thin ones on either side
};

// One of the three phases of a step (kind 0 inverse y, 1 inverse x, times V,
// forward x, 2 forward y) for lines of length N, its lines (band-major) dealt
// 32 at a time to the warp pairs.  All kinds end in one M-point DFT body, the
// inverse one: the forward transform is the inverse of the conjugate, and the
// conjugation rides on the multiply by V and on the final store.  (Two bodies
// instead of four keep the code of a step small enough for the instruction
// cache; with four the kernel was held up by instruction fetches.)  KINDS: bit
// set of the kinds wanted of this length (all three for n1 = n2).
template <int N, class C, int N2, int KINDS>
__device__ __forceinline__ void yx_body(int kind_, const YXStep& s) {
    constexpr int M = N / 2, Q = N / 4, AP = C::AP, PP = C::PP, SLOT = C::SLOT, PAIRS = C::PAIRS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* const A = reinterpret_cast<float2*>(smem_raw);
    const int lane = threadIdx.x & 31, role = (threadIdx.x >> 5) & 1, pair = threadIdx.x >> 6;
    asm volatile("" : "+r"(kind_));  // one body for the kinds, not a specialised copy of each
    const int kind = KINDS == 7 ? kind_ : KINDS == 5 ? kind_ & 2 : KINDS == 2 ? 1 : 0;
    const int per = kind == 1 ? N2 : s.planes, p0 = kind == 1 ? 0 : s.p0, lines = per * s.nbb;
#pragma unroll 1
    for (int l0 = pair * 32; l0 < lines; l0 += PAIRS * 32) {
        const bool act = l0 + lane < lines;
        const int ln = min(l0 + lane, lines - 1);
        const int bb = ln / per, c = ln - bb * per + p0;
        float2* ay = A + bb * SLOT + c * AP;      // kinds 0, 2: the plane's row
        float2* ax = A + bb * SLOT + Q * AP + c;  // kind 1: the column, at h = 0
        float2* d = s.d + bb * s.dband + c;
        float2 u[M];
        int2 kr = make_int2(1, -1);
        if (kind == 2) {
            kr = act ? s.krange[c] : kr;
            sfor<M>([&](auto j) { u[j] = ay[2 * decltype(j)::value + role]; });
        } else {
            auto ldx = [&](auto k) { return ax[decltype(k)::value * AP]; };
            auto ldy = [&](auto kc) {
                constexpr int k = decltype(kc)::value;
                return k >= 0 ? ld_if_ge<k>(d + k * PP, kr.y) : ld_if_ge<-k>(d + k * PP, -kr.x);
            };
            if (kind == 0) {
                kr = act ? s.krange[c] : kr;
                half_load<N>(u, ldy);
            } else {
                half_load<N>(u, ldx);
            }
            half_fold<N>(u, role, [&](auto k) { return kind == 0 ? ldy(k) : ldx(k); });
        }
        if (kind == 1) {
            RDft<M, +1>::run(u);
            const float* v = s.v + role * N2 + c;
            sfor<M>([&](auto j) {  // conj(psi V)
                const float w = v[2 * N2 * decltype(j)::value];
                u[j] = make_float2(u[j].x * w, -u[j].y * w);
            });
        }
        RDft<M, +1>::run(u);
        if (kind == 0) {
            if (act) sfor<M>([&](auto j) { ay[2 * decltype(j)::value + role] = u[j]; });
            continue;
        }
        if (role) sfor<M>([&](auto n) { u[n] = Tw<N, +1, decltype(n)::value>::mul(u[n]); });
        bar_pair(1 + pair);  // both halves have read the line
        // role 1 leaves its half of every output in the line's slots, role 0
        // adds its own and keeps (x) or writes out (y) the sums
        if (kind == 1) {
            if (role && act) {
                sfor<M>([&](auto n) { ax[kof<N>(decltype(n)::value) * AP] = u[n]; });
                if constexpr (2 * Q == M) ax[-Q * AP] = u[Q];
            }
            bar_pair(1 + pair);
            if (!role && act) {
                sfor<M>([&](auto n) {
                    constexpr int k = kof<N>(decltype(n)::value);
                    ax[k * AP] = k >= 0 ? cadd(u[n], ax[k * AP]) : csub(u[n], ax[k * AP]);
                });
                if constexpr (2 * Q == M) ax[-Q * AP] = csub(u[Q], ax[-Q * AP]);
            }
        } else {
            if (role && act) sfor<M>([&](auto n) { ay[decltype(n)::value] = u[n]; });
            bar_pair(1 + pair);
            if (!role)
                sfor<M>([&](auto nc) {
                    constexpr int n = decltype(nc)::value;
                    const float2 o = ay[n];
                    if constexpr (n <= Q) st_if_ge<n>(d + n * PP, make_float2(u[n].x + o.x, -u[n].y - o.y), kr.y);
                    if constexpr (n - M >= -Q)
                        st_if_ge<M - n>(d + (n - M) * PP, make_float2(u[n].x - o.x, o.y - u[n].y), -kr.x);
                });
        }
        // the pair's next line group touches other rows and columns
    }
}

// The thin planes of a y phase (at most two sticks each: the rim of the
// sphere), one a warp, by direct sums, where taking them off the lines saves
// the pairs a round of groups: 65 planes at 128^3, R = 32, are three groups
// and two rounds, 63 are two and one (1.87 -> 1.63 ms per 256 bands; two bands
// of 33 planes at 64^3 0.196 -> 0.190).  Where they save a group but no round
// (98 lines at 96^3) they cost more than they give, 2.28 -> 2.63 ms.
template <class C, int N2> __device__ __forceinline__ void yx_thin(bool fwd, const YXStep& s) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int tasks = 2 * s.trim * s.nbb;
#pragma unroll 1
    for (int i = threadIdx.x >> 5; i < tasks; i += 2 * C::PAIRS) {
        const int bb = i / (2 * s.trim), q = i - bb * 2 * s.trim;
        const int p = q < s.trim ? s.p0 - 1 - q : s.p0 + s.planes + q - s.trim;
        float2* a = reinterpret_cast<float2*>(smem_raw) + bb * C::SLOT + p * C::AP;
        float2* d = s.d + bb * s.dband + p;
        const int2 kr = s.krange[p];
        if (!fwd) {
#pragma unroll 1
            for (int y = lane; y < N2; y += 32) {
                float2 v = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int k = kr.x; k <= kr.y; ++k) v = cadd(v, cmul(d[k * C::PP], s.tw2[(k * y + N2 * N2) % N2]));
                a[y] = v;
            }
        } else {  // the array holds conjugates
#pragma unroll 1
            for (int k = kr.x; k <= kr.y; ++k) {
                float2 v = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int y = lane; y < N2; y += 32) v = cadd(v, cmul(a[y], s.tw2[(k * y + N2 * N2) % N2]));
#pragma unroll
                for (int m = 16; m; m >>= 1) {
                    v.x += __shfl_xor_sync(0xffffffffu, v.x, m);
                    v.y += __shfl_xor_sync(0xffffffffu, v.y, m);
                }
                if (lane == 0) d[k * C::PP] = make_float2(v.x, -v.y);
            }
        }
    }
}

// Block (z, group of bpc bands), NBB bands at a time.
template <int CLS, int N1, int N2>
__global__ void __launch_bounds__(64 * YX<CLS, N1, N2>::PAIRS, YX<CLS, N1, N2>::MINB)
    kl_yx(Tables t, const float2* __restrict__ tw2, const float* VT, int nb, int bpc, float2* D) {
    pdl_begin();
    using C = YX<CLS, N1, N2>;
    constexpr int NBB = C::NBB;
    const int z = blockIdx.x;
    const int b0 = blockIdx.y * bpc, b1 = min(nb, b0 + bpc);
    YXStep s;
    s.dband = (long long)t.row * t.n3;
    s.v = VT + (size_t)z * N1 * N2;
    s.krange = t.krange;
    s.tw2 = tw2;
    s.trim = yx_thins(N1, N2) ? t.trim : 0;
    s.p0 = s.trim;
    s.planes = 2 * (N1 / 4) + 1 - 2 * s.trim;
#pragma unroll 1
    for (int b = b0; b < b1; b += NBB) {
        s.nbb = min(NBB, b1 - b);
        s.d = D + b * s.dband + (long long)z * t.row + (N2 / 4) * C::PP;
#pragma unroll 1
        for (int kind = 0; kind < 3; ++kind) {
            if (b > b0 || kind > 0) __syncthreads();  // the last phase's rows are written, or have been read
            if constexpr (N1 == N2) {
                yx_body<N1, C, N2, 7>(kind, s);
            } else {
                if (kind == 1) yx_body<N1, C, N2, 2>(kind, s);
                else yx_body<N2, C, N2, 5>(kind, s);
            }
            if constexpr (yx_thins(N1, N2))
                if (kind != 1) yx_thin<C, N2>(kind == 2, s);
        }
    }
}

// ------------------------------------------------------------ launchers
template <int CLS, int N1, int N2>
int launch_yx_n(const Tables& t, const float2* tw2, const float* VT, long long nb, float2* D, cudaStream_t st) {
    using C = YX<CLS, N1, N2>;
    if (const cudaError_t e = smem_optin<kl_yx<CLS, N1, N2>>(C::smem)) return (int)e;
    // bands per block, as measured (8 against 4: 2.28 and 2.30 ms at 96^3 x
    // 1024, 0.342 and 0.334 at 80^3 x 256, 0.956 and 0.931 at 100^3, 1.62 and
    // 1.59 at 128^3), but few enough that the grid is four waves deep
    int bpc = C::NBB == 2 && N2 % 32 == 0 ? 8 : 4;
    while (bpc > C::NBB && (long long)t.n3 * ((nb + bpc - 1) / bpc) < 152ll * C::MINB * 4) bpc /= 2;
    return pdl_launch(kl_yx<CLS, N1, N2>, dim3(t.n3, (unsigned)((nb + bpc - 1) / bpc)), 64 * C::PAIRS, C::smem, st,
        t, tw2, VT, (int)nb, bpc, D);
}
// n1 = N1, every n2 of the class
template <int CLS, int N1>
int LaunchYX<CLS, N1>::run(const Tables& t, const float2* tw2, const float* VT, long long nb, float2* D, cudaStream_t st) {
    static_assert(yx_partner(CLS, N1, yx_pair), "a length without kernels");
#define VLOC_CASE(N) \
    case N:          \
        if constexpr (yx_pair(CLS, N1, N)) return launch_yx_n<CLS, N1, N>(t, tw2, VT, nb, D, st); \
        else break;
    if constexpr (CLS == 0) switch (t.n2) { VLOC_LINE_C48(VLOC_CASE) default: break; }
    if constexpr (CLS == 1) switch (t.n2) { VLOC_LINE_C96(VLOC_CASE) default: break; }
    if constexpr (CLS == 2) switch (t.n2) { VLOC_LINE_C144(VLOC_CASE) default: break; }
#undef VLOC_CASE
    return (int)cudaErrorInvalidValue;
}

}  // namespace line
}  // namespace vloc
