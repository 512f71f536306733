// kernels_line.h -- the line path: the V_loc apply as three launches (plus
// one that transposes V), for FP32 plans whose sphere lies in the quarter
// band of every axis (|h| <= n1/4, |k| <= n2/4, |l| <= n3/4: the workload of
// Sec. 4.3, where the grid is about four cut-off radii wide).
//
// Between the launches a band is stored densely, [z][k + n2/4][h + n1/4],
// rows of PP elements (the widest plane set of the size class), so that
//  * the z-passes, whose lanes are sticks in that order, read and write it
//    coalesced without a transpose, and
//  * one thread block holds everything the y- and x-passes of one z need: it
//    reads the z row's sticks, runs inverse y, inverse x, times V, forward x
//    and forward y with the (plane, y) array in shared memory, and writes the
//    sticks back.  The slab of the five-launch chain never reaches memory:
//    6.4 MB of traffic per band at 96^3 against 20.9 MB.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vloc {
namespace line {

// Size classes of the y/x kernel: both n1 and n2 in the class's list (a kernel
// per pair); the class fixes the pitch of the dense rows.
#define VLOC_LINE_C48(X) X(24) X(30) X(32) X(36) X(40) X(48)
#define VLOC_LINE_C96(X) X(48) X(50) X(54) X(60) X(64) X(72) X(80) X(90) X(96)
#define VLOC_LINE_C144(X) X(80) X(90) X(96) X(100) X(108) X(120) X(128) X(144)
// z lengths
#define VLOC_LINE_Z_A(X) X(24) X(30) X(32) X(36) X(40) X(48)
#define VLOC_LINE_Z_B(X) X(50) X(54) X(60) X(64) X(72) X(80)
#define VLOC_LINE_Z_C(X) X(90) X(96) X(100) X(108)
#define VLOC_LINE_Z_D(X) X(120) X(128) X(144)

// Pairs with a kernel: the smallest class that holds both, and no axis more
// than 1.35 times the other (the axes of one cell's grid follow its sides;
// every pair more costs build time).
constexpr bool yx_pair(int cls, int n1, int n2) {
    const int hi = n1 > n2 ? n1 : n2, lo = n1 > n2 ? n2 : n1;
    return 20 * hi <= 27 * lo && (cls == 0 || hi > (cls == 1 ? 48 : 96));
}
// Whether the thin planes' code is in the kernels of n1 (its presence costs
// about 4 %): where at most two planes off either side of a full quarter
// sphere save the two warp pairs a round of 32-line groups.
constexpr int yx_rounds(int lines) { return (lines + 63) / 64; }
constexpr int yx_bands(int n1, int n2) { return (n1 > n2 ? n1 : n2) <= 96 ? 2 : 1; }  // bands per step
constexpr bool yx_thins(int n1, int n2) {
    const int m = yx_bands(n1, n2), planes = 2 * (n1 / 4) + 1;
    return yx_rounds(m * (planes - 4)) < yx_rounds(m * planes);
}
// Whether n1 has a kernel with any n2 of the class
#define VLOC_OR(N) || ok(cls, n1, N)
template <class F> constexpr bool yx_partner(int cls, int n1, F ok) {
    return (cls == 0 && (false VLOC_LINE_C48(VLOC_OR))) || (cls == 1 && (false VLOC_LINE_C96(VLOC_OR))) ||
           (cls == 2 && (false VLOC_LINE_C144(VLOC_OR)));
}
#undef VLOC_OR
// class index 0, 1, 2 (up to 48, 96, 144), or -1
int yx_class(int n1, int n2);
bool z_length(int n3);
// Whether the form is the faster one for a cell of `planes` occupied x-planes
// (lengths with compile-time five-launch kernels)
bool pays(int n1, int n2, int n3, int planes, bool gamma, bool density);
// elements between the k rows of the dense layout
constexpr int class_pitch(int cls) { return cls == 0 ? 28 : cls == 1 ? 52 : 76; }

// Device tables of a plan.  A group is 32 sticks (one z-pass block) in the
// order of their dense positions, lanes 2 s and 2 s + 1 an aligned pair of
// positions (-1 where one of the two is not a stick); for Gamma-point plans 16
// sticks and their mirrors (-h, -k), so that G and -G share a group.
struct Tables {
    const int* gpos;      // [G][32] dense position (k + n2/4) PP + h + n1/4 of a lane's stick, or -1
    const int* zd;        // plain: [G][rows][32] caller index at each first-stage row (as DevTables::zdense), or -1
    const int4* run_tab;  // runs: [G][32] {first caller index, its l, count, 0}
    const int* gh_ptr;    // Gamma: [G + 1] the groups' ranges of gh
    const int4* gh;       // {half-list index, position of G, of -G, 0}, position = z | lane << 16
    const int2* krange;   // [2 (n1/4) + 1] first and last k of each plane's sticks ({1, -1}: none)
    int G;
    int n1, n2, n3;
    int row;              // dense elements per z, (2 (n2/4) + 1) PP
    int cls, gamma, runs;
    int trim;             // thin planes taken off either side by the y phases
    long long npw;        // plane waves per band in the caller's arrays
};
inline size_t band_elems(const Tables& t) { return (size_t)t.row * t.n3; }

// VT [z][x][y] = V [x][y][z]
int launch_vt(const float* V, float* VT, const Tables& t, cudaStream_t st);
// D [nb][n3][row]: inverse z-pass of nb bands (Gamma: of nb pairs formed from
// nreal real bands); y/x pass with V in place; forward z-pass into out (times
// 1/N, plus diag times c).  Each returns the cudaError_t of its launch.
int launch_z_inv(const Tables& t, const float2* tw3, const float2* c, long long nb, long long nreal, float2* D,
                 cudaStream_t st);
int launch_yx(const Tables& t, const float2* tw2, const float* VT, long long nb, float2* D, cudaStream_t st);
int launch_z_fwd(const Tables& t, const float2* tw3, const float2* D, long long nb, long long nreal, float2* out,
                 const float* diag, const float2* c, cudaStream_t st);

// Density: partial sums [group][z][x][y] of groups of at most bpg bands of D
// (see launch_k3d_density), and their sum over the ng groups, in order and
// compensated as launch_reduce_partials_f32, turned to [x][y][z]
int launch_dens(const Tables& t, const float2* D, long long nb, int bpg, const float* occ, long long b_base, int pair,
                long long nreal, float* partial, cudaStream_t st);
int launch_dens_reduce(const Tables& t, const float* partial, int ng, double* acc, int first, float* out,
                       cudaStream_t st);

// instantiated per length / class in kernels_line_*.cu
template <int N> struct LaunchZ {
    static int inv(const Tables& t, const float2* tw3, const float2* c, long long nb, long long nreal, float2* D,
                   cudaStream_t st);
    static int fwd(const Tables& t, const float2* tw3, const float2* D, long long nb, long long nreal, float2* out,
                   const float* diag, const float2* c, cudaStream_t st);
};
// the density of n1 with compile-time density kernels in the five-launch chain
// (elsewhere the group sums are FP64)
#define VLOC_LINE_D48(X) X(32) X(48)
#define VLOC_LINE_D96(X) X(48) X(60) X(64) X(72) X(80) X(96)
#define VLOC_LINE_D144(X) X(80) X(96) X(100) X(120) X(128) X(144)
// and n2 whose lines fill both warp pairs of a block, which takes a band at a
// time (32^3 x 300 bands 56 against 45 us)
constexpr bool dens_pair(int cls, int n1, int n2) { return yx_pair(cls, n1, n2) && n2 > 32; }
template <int CLS, int N1> struct LaunchDens {
    static int run(const Tables& t, const float2* D, long long nb, int bpg, const float* occ, long long b_base, int pair,
                   long long nreal, float* partial, cudaStream_t st);
};
template <int CLS, int N1> struct LaunchYX {
    static int run(const Tables& t, const float2* tw2, const float* VT, long long nb, float2* D, cudaStream_t st);
};

}  // namespace line
}  // namespace vloc
