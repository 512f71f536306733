// kernels_line_z.cuh -- the z-passes of the line path (kernels_line.h).
//
// The two-stage quarter-band transforms of kernels_ct.cuh over tiles of 32
// sticks, with the dense rows in the cylinder's place: consecutive sticks of a
// tile are consecutive in every dense row, so the inverse's last stage writes
// them and the forward's first stage reads them straight from registers (no
// pass through the tile buffer to turn sticks into rows, one barrier less).
#pragma once

#include "kernels_ct.cuh"
#include "kernels_line.h"

namespace vloc {
namespace line {

// line pair 2 s, 2 s + 1 of the group in row e of the dense band
template <bool GM> struct DenseRows;
template <> struct DenseRows<false> {  // an aligned pair of positions
    float2* p;
    int row;
    __device__ __forceinline__ P2f operator()(int e, int) const { return *reinterpret_cast<const P2f*>(p + e * row); }
    __device__ __forceinline__ void operator()(int e, int, P2f v) const { *reinterpret_cast<P2f*>(p + e * row) = v; }
};
template <> struct DenseRows<true> {  // two positions, -1 absent
    float2* d;
    int pa, pb, row;
    __device__ __forceinline__ P2f operator()(int e, int) const {
        P2f v = czero<P2f>();
        if (pa >= 0) v.a = d[e * row + pa];
        if (pb >= 0) v.b = d[e * row + pb];
        return v;
    }
    __device__ __forceinline__ void operator()(int e, int, P2f v) const {
        if (pa >= 0) d[e * row + pa] = v.a;
        if (pb >= 0) d[e * row + pb] = v.b;
    }
};
template <bool GM> __device__ __forceinline__ bool dense_rows(const Tables& t, int g, int slot, float2* d, DenseRows<GM>& r) {
    const int pa = t.gpos[g * 32 + 2 * slot], pb = t.gpos[g * 32 + 2 * slot + 1];
    r.row = t.row;
    if constexpr (GM) {
        r.d = d; r.pa = pa; r.pb = pb;
    } else {
        r.p = d + (pa >= 0 ? pa : pb - 1);
    }
    return pa >= 0 || pb >= 0;
}

// Lane -> (line pair, unit) of the stages that meet the caller's arrays (the
// inverse's first, the forward's last).  ED (caller lists in stick order): a warp
// takes 8 line pairs and 4 consecutive units instead of 16 and 2, so that an
// access covers 32 bytes of each stick's run; these accesses are most of a
// block's load/store wavefronts.  Forward 0.430 -> 0.422 ms (96^3 x 1024 bands),
// 0.266 -> 0.259 (128^3 x 256); inverse 0.266 -> 0.259 (120^3 x 256), 0.0875 ->
// 0.0861 (64^3 x 512), 96^3 x 1024 0.452 -> 0.449 on one GPU and 0.470 -> 0.473
// on another.  Lists in another order have no runs to cover and lose rows of the
// table that two units share (shuffled, 96^3: 0.653 -> 0.673, 0.516 -> 0.524),
// so they keep 16 and 2.
template <bool ED> __device__ __forceinline__ int edge_slot() {
    return ED ? (threadIdx.x & 7) + ((threadIdx.x >> 5) & 1) * 8 : slot_of();
}
template <bool ED> __device__ __forceinline__ int edge_unit() {
    return ED ? ((threadIdx.x >> 3) & 3) + (threadIdx.x >> 6) * 4 : 2 * warp_of() + sub_of();
}
static_assert(kWarps % 2 == 0, "edge mapping: warps in pairs");

// MODE 0: first-stage inputs through the group's dense table, 1: addressed
// from the sticks' runs (caller lists in stick order), 2: Gamma-point pairs.
template <int N, int MODE>
__global__ void __launch_bounds__(kThreads, minb_k1(N)) kl_z_inv(Tables t, const float2* __restrict__ tw3,
                                                            const float2* coeffs, long long nreal,
                                                            float2* __restrict__ D) {
    pdl_begin();
    using SC = Sched<N>;
    static_assert(SC::nst == 2, "quarter-band z-pass: two-stage lengths");
    using QR = QRows<N>;
    constexpr int R0 = QR::R0, NA = QR::NA, W = kWarps;
    constexpr int UA = (NA + 2 * W - 1) / (2 * W);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    float2* stw = buf + N * kLdP;
    const int g = blockIdx.x;
    const long long b = blockIdx.y;
    const int slot = slot_of(), sub = sub_of(), warp = warp_of();
    DenseRows<MODE == 2> dr;
    const bool act = dense_rows<MODE == 2>(t, g, slot, D + b * (long long)t.row * N, dr);
    SmemP sb{buf};
    if constexpr (MODE < 2) {
        const float2* c = coeffs + b * t.npw;
        const int slot = edge_slot<MODE == 1>();
#pragma unroll
        for (int u = 0; u < UA; ++u) {
            const int i = edge_unit<MODE == 1>() + 2 * W * u;
            if (NA % (2 * W) == 0 || i < NA) {
                P2f h[R0];
                if constexpr (MODE == 1) {
                    const int4 ra = t.run_tab[g * 32 + 2 * slot], rb = t.run_tab[g * 32 + 2 * slot + 1];
                    auto at = [&](const int4& r, int x) {
                        const int p = (x <= N / 2 ? x : x - N) - r.y;
                        return (p >= 0 && p < r.z) ? c[r.x + p] : make_float2(0.f, 0.f);
                    };
                    sfor<R0>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        if constexpr (QR::kind(r) == 0) h[r] = czero<P2f>();
                        else h[r] = P2f{at(ra, i + r * NA), at(rb, i + r * NA)};
                    });
                } else {
                    const int* zd = t.zd + (size_t)g * (QR::groups() * NA) * 32 + 2 * slot;
                    int2 e[R0];
                    sfor<R0>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        if constexpr (QR::kind(r) != 0)
                            e[r] = *reinterpret_cast<const int2*>(zd + (QR::group(r) * NA + i) * 32);
                    });
                    sfor<R0>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        if constexpr (QR::kind(r) == 0) h[r] = czero<P2f>();
                        else
                            h[r] = P2f{e[r].x >= 0 ? c[e[r].x] : make_float2(0.f, 0.f),
                                       e[r].y >= 0 ? c[e[r].y] : make_float2(0.f, 0.f)};
                    });
                }
                DftZ<R0, +1, QR::mask()>::run(h);
#pragma unroll
                for (int r = 0; r < R0; ++r) sb(i * R0 + r, slot, h[r]);
            }
        }
    } else {
        // scatter of the pairs into the rows the first stage reads, then the
        // stage in place
        constexpr int B = VLOC_SCATTER_BATCH, RW = kLdP / 2;
        int4 en[B];
        float2 va[B], vb[B];
        const float2* a = coeffs + 2 * b * t.npw;
        const float2* bb = 2 * b + 1 < nreal ? a + t.npw : nullptr;
        const int e1 = t.gh_ptr[g + 1], base0 = t.gh_ptr[g] + (int)threadIdx.x;
        gamma_load<B>(t.gh, base0, e1, a, bb, en, va, vb);
        for (int i = threadIdx.x; i < N * RW; i += kThreads)
            if (xq_row_read<N>(i / RW)) reinterpret_cast<float4*>(buf)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        gamma_store<B>(buf, en, va, vb);
        for (int base = base0 + B * kThreads; base < e1; base += B * kThreads) {
            gamma_load<B>(t.gh, base, e1, a, bb, en, va, vb);
            gamma_store<B>(buf, en, va, vb);
        }
        __syncthreads();
        P2f h[UA][R0];
#pragma unroll
        for (int u = 0; u < UA; ++u) {
            const int i = 2 * (warp + u * W) + sub;
            if (NA % (2 * W) == 0 || i < NA) {
                sfor<R0>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    if constexpr (QR::kind(r) == 0) h[u][r] = czero<P2f>();
                    else h[u][r] = sb(i + r * NA, slot);
                });
                DftZ<R0, +1, QR::mask()>::run(h[u]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < UA; ++u) {
            const int i = 2 * (warp + u * W) + sub;
            if (NA % (2 * W) == 0 || i < NA) {
#pragma unroll
                for (int r = 0; r < R0; ++r) sb(i * R0 + r, slot, h[u][r]);
            }
        }
    }
    load_tw<float>(stw, tw3, N);
    __syncthreads();
    NatStage<N, +1, W, 1>::template run<false>(stw, sb, dr, slot, sub, warp, act);
}

// Forward: first stage (reversed schedule) straight from the dense rows; the
// last one stores each result to its caller position through the dense table
// or (Gamma) leaves it in the tile for the gather that separates the
// pairs; times 1/N, plus diag times the band.  ED: see edge_slot.
template <int N, bool GM, bool ED>
__global__ void __launch_bounds__(kThreads, GM ? minb_k4q(N, true) : minb_k4d(N))
    kl_z_fwd(Tables t, const float2* __restrict__ tw3, const float2* D, long long nreal, float2* out,
             float scale, const float* diag, const float2* cin) {
    pdl_begin();
    using SC = Sched<N>;
    static_assert(SC::nst == 2, "quarter-band z-pass: two-stage lengths");
    using QR = QRows<N>;
    constexpr int R0 = QR::R0, NA = QR::NA, W = kWarps;
    using L = RevStage<N, -1, W, 1>;  // radix R0, rows i + r NA
    static_assert(L::NI == NA, "last forward stage rows");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    float2* stw = buf + N * kLdP;
    const int g = blockIdx.x;
    const long long b = blockIdx.y;
    const int slot = slot_of(), sub = sub_of(), warp = warp_of();
    DenseRows<GM> dr;
    const bool act = dense_rows<GM>(t, g, slot, const_cast<float2*>(D) + b * (long long)t.row * N, dr);
    SmemP sb{buf};
    RevStage<N, -1, W, 0>::template run<false>(stw, dr, sb, slot, sub, warp, act);
    load_tw<float>(stw, tw3, N);
    if constexpr (!GM) {
        // The table's entries are requested before the barrier where a thread
        // has one unit (64^3 x 512 bands 0.078 -> 0.071 ms, 96^3 x 1024 0.422 ->
        // 0.422, shuffled list 0.512 -> 0.510); with two they cost registers
        // (120^3 x 256 0.2234 -> 0.2243).
        constexpr bool AHEAD = L::U == 1;
        const int slot = edge_slot<ED>();
        const int* zd = t.zd + (size_t)g * (QR::groups() * NA) * 32 + 2 * slot;
        int2 e[R0];
        auto entries = [&](int i) {
            sfor<R0>([&](auto rc) {
                constexpr int r = decltype(rc)::value;
                if constexpr (QR::kind(r) != 0) e[r] = *reinterpret_cast<const int2*>(zd + (QR::group(r) * NA + i) * 32);
            });
        };
        if (AHEAD && (L::NI % (2 * W) == 0 || edge_unit<ED>() < L::NI)) entries(edge_unit<ED>());
        __syncthreads();
        if (!ED && !act) return;  // ED: `act` is not this lane's line pair; the table's -1 drops absent ones
        float2* o = out + b * t.npw;
        const float2* ci = diag ? cin + b * t.npw : cin;
#pragma unroll
        for (int u = 0; u < L::U; ++u) {
            const int i = edge_unit<ED>() + 2 * W * u;
            if (L::NI % (2 * W) == 0 || i < L::NI) {
                if (!AHEAD) entries(i);
                P2f h[R0];
                L::compute_unit(h, stw, sb, i, slot);
                sfor<R0>([&](auto rc) {
                    constexpr int r = decltype(rc)::value;
                    if constexpr (QR::kind(r) != 0) {
                        auto put = [&](int x, float2 v) {
                            if (x < 0) return;
                            v = cscale(v, scale);
                            if (diag) {  // H = diag + A (c is read before out is written: they may alias)
                                const float d = diag[x];
                                const float2 cv = ci[x];
                                v = make_float2(v.x + d * cv.x, v.y + d * cv.y);
                            }
                            o[x] = v;
                        };
                        put(e[r].x, h[r].a);
                        put(e[r].y, h[r].b);
                    }
                });
            }
        }
    } else {
        __syncthreads();
        P2f h[L::U][R0];
        if (act) L::compute(h, stw, sb, slot, sub, warp);
        __syncthreads();
        if (act) {
#pragma unroll
            for (int u = 0; u < L::U; ++u) {
                const int i = 2 * (warp + u * W) + sub;
                if (L::NI % (2 * W) == 0 || i < L::NI) {
                    sfor<R0>([&](auto rc) {
                        constexpr int r = decltype(rc)::value;
                        if constexpr (QR::kind(r) != 0) sb(i + r * NA, slot, h[u][r]);
                    });
                }
            }
        }
        __syncthreads();
        const bool two = 2 * b + 1 < nreal;
        const float2* ca = diag ? cin + 2 * b * t.npw : cin;
        gather_gamma(t.gh, t.gh_ptr[g], t.gh_ptr[g + 1], buf, out + 2 * b * t.npw,
                     two ? out + (2 * b + 1) * t.npw : nullptr, scale, diag, ca, diag ? ca + t.npw : ca);
    }
}

// ------------------------------------------------------------ launchers
template <int N, int MODE>
int launch_z_inv_n(const Tables& t, const float2* tw3, const float2* c, long long nb, long long nreal, float2* D,
                   cudaStream_t st) {
    if (const cudaError_t e = smem_optin<kl_z_inv<N, MODE>>(CtSmem<N>::sm)) return (int)e;
    return pdl_launch(kl_z_inv<N, MODE>, dim3(t.G, (unsigned)nb), kThreads, CtSmem<N>::sm, st, t, tw3, c, nreal, D);
}
template <int N>
int LaunchZ<N>::inv(const Tables& t, const float2* tw3, const float2* c, long long nb, long long nreal, float2* D,
                    cudaStream_t st) {
    return t.gamma  ? launch_z_inv_n<N, 2>(t, tw3, c, nb, nreal, D, st)
           : t.runs ? launch_z_inv_n<N, 1>(t, tw3, c, nb, nreal, D, st)
                    : launch_z_inv_n<N, 0>(t, tw3, c, nb, nreal, D, st);
}
template <int N, bool GM, bool ED>
int launch_z_fwd_n(const Tables& t, const float2* tw3, const float2* D, long long nb, long long nreal, float2* out,
                   const float* diag, const float2* c, cudaStream_t st) {
    if (const cudaError_t e = smem_optin<kl_z_fwd<N, GM, ED>>(CtSmem<N>::sm)) return (int)e;
    const float scale = (float)(1.0 / ((double)t.n1 * t.n2 * t.n3));
    return pdl_launch(kl_z_fwd<N, GM, ED>, dim3(t.G, (unsigned)nb), kThreads, CtSmem<N>::sm, st, t, tw3, D, nreal, out,
        scale, diag, c);
}
template <int N>
int LaunchZ<N>::fwd(const Tables& t, const float2* tw3, const float2* D, long long nb, long long nreal, float2* out,
                    const float* diag, const float2* c, cudaStream_t st) {
    return t.gamma  ? launch_z_fwd_n<N, true, false>(t, tw3, D, nb, nreal, out, diag, c, st)
           : t.runs ? launch_z_fwd_n<N, false, true>(t, tw3, D, nb, nreal, out, diag, c, st)
                    : launch_z_fwd_n<N, false, false>(t, tw3, D, nb, nreal, out, diag, c, st);
}

}  // namespace line
}  // namespace vloc
