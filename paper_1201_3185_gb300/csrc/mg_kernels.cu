// Multigrid kernels of the QUMOND solves (Section 2, steps 2 and 4): red-black
// Gauss-Seidel half-sweeps, residual restriction, prolongation, boundary
// injection, the single-CTA coarse-grid solver, and the FP64 outer steps of
// the defect correction.  T is the smoothing precision (float or double).
//
// Level arrays use the colour-split layout of qumond_internal.h.  Two facts
// of red-black Gauss-Seidel are used to skip dead work (both exact in exact
// arithmetic, so the iterates are those of the textbook V-cycle):
//  * a node's update does not read its own old value, so after a coarse-grid
//    correction only the black nodes need the prolonged correction before the
//    next red half-sweep, and an FMG interpolation only has to fill black
//    nodes;
//  * right after a black half-sweep the black residuals are zero, so the
//    residual to restrict is nonzero only at red nodes.
#include "qumond_internal.h"
#include "fixed_conv.h"

#include <cstdio>

namespace qumond {

namespace {

constexpr int kBX = 32;
constexpr int kBY = 8;

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

// ---------------------------------------------------------------------------
// One half-sweep: every interior node of `colour` is set to
//   (sum of its 6 neighbours - h^2 f) / 6,
// its neighbours all being of the other colour.  ZERO: the neighbours are
// known to be zero (first sweep of a correction that starts from zero).
template <typename T, bool ZERO>
__device__ __forceinline__ void rb_node(T* __restrict__ own, const T* __restrict__ other, const T* __restrict__ f,
                                        const LevelView& v, int colour, T h2, T sixth, int m, int j, int k)
{
    const int p = (colour + j + k) & 1;  // parity of i in this row
    if (p == 0 && m == 0) return;        // i = 0 is a boundary node
    const long long row = ((long long)k * (v.n + 1) + j) * v.M;
    T s = T(0);
    if (!ZERO) {
        const T* o = other + row;
        const long long P = v.M, Q = (long long)v.M * (v.n + 1);
        s = (o[m - 1 + p] + o[m + p]) + (o[m - P] + o[m + P]) + (o[m - Q] + o[m + Q]);
    }
    own[row + m] = (s - h2 * f[row + m]) * sixth;
}

// The set index of a context with several sets, folded into blockIdx.z
// (per planes per set): returns it and the plane index within the set.
__device__ __forceinline__ int set_of(int per, int& within)
{
    if ((int)gridDim.z == per) {  // one set: no division
        within = (int)blockIdx.z;
        return 0;
    }
    const int s = (int)blockIdx.z / per;
    within = (int)blockIdx.z - s * per;
    return s;
}

template <typename T, bool ZERO>
__global__ void __launch_bounds__(kBX * kBY)
rb_half_kernel(T* __restrict__ own, const T* __restrict__ other, const T* __restrict__ f, LevelView v, int colour,
               T h2, T sixth, const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(v.n - 1, kz);
    if (act && !act[set].cont) return;
    const long long so = (long long)set * 2 * v.cs;
    const int half = v.n >> 1;
    const int m = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y + 1;
    const int k = kz + 1;
    if (m >= half || j >= v.n) return;
    rb_node<T, ZERO>(own + so, other + so, f + so, v, colour, h2, sixth, m, j, k);
}

// The same half-sweep on FP32 levels with four consecutive entries of a row
// per thread (the parity of i is the same along a row): 16-byte loads of the
// row, its four neighbour rows and f, two scalars for the x-neighbours past
// the ends, one 16-byte store; the node arithmetic is rb_node's, in the same
// order.  half = n/2 is a multiple of 4, so a group lies wholly inside or
// outside the row's entries; the scalar before entry 0 (read from the padding
// at the end of the previous row) only feeds the boundary node i = 0, which
// is not written.
// Block shapes: VX threads along a row (4 VX entries) x 128/VX rows.  The
// default 8 x 16 suits large levels; the small levels (n/2 = 8 .. 32 entries
// per row) leave most of an 8-wide block idle, so a context can pick 4 x 32 or
// 2 x 64 for levels n <= 64 (params.tile_small).  Every shape gives the same
// bits: each thread's entries are updated by the same arithmetic.
constexpr int kVX = 8;  // default: 32 entries x 16 rows per block
constexpr int kVThreads = 128;
constexpr int kVBlocksPerSM = 16;  // full occupancy (<= 32 registers): the small levels are latency-bound
constexpr int kTileSmallN = 64;  // the alternative shapes apply to levels with n <= this

template <bool ZERO, int VX = kVX>
__global__ void __launch_bounds__(kVThreads, kVBlocksPerSM)
rb_half4_kernel(float* __restrict__ own, const float* __restrict__ other, const float* __restrict__ f, LevelView v,
                int colour, float h2, float sixth, const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(v.n - 1, kz);
    if (act && !act[set].cont) return;
    {
        const long long so = (long long)set * 2 * v.cs;
        own += so, other += so, f += so;
    }
    const int half = v.n >> 1;
    const int mA = 4 * (blockIdx.x * VX + threadIdx.x);
    const int j = blockIdx.y * (kVThreads / VX) + threadIdx.y + 1;
    const int k = kz + 1;
    if (mA >= half || j >= v.n) return;
    const int p = (colour + j + k) & 1;
    const long long row = ((long long)k * (v.n + 1) + j) * v.M;
    float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (!ZERO) {
        const float* o = other + row + mA;
        const long long P = v.M, Q = (long long)v.M * (v.n + 1);
        const float4 V = *reinterpret_cast<const float4*>(o);
        const float x[6] = {o[-1], V.x, V.y, V.z, V.w, o[4]};  // entries mA-1 .. mA+4
        const float4 Y0 = *reinterpret_cast<const float4*>(o - P), Y1 = *reinterpret_cast<const float4*>(o + P);
        const float4 Z0 = *reinterpret_cast<const float4*>(o - Q), Z1 = *reinterpret_cast<const float4*>(o + Q);
        const float y0[4] = {Y0.x, Y0.y, Y0.z, Y0.w}, y1[4] = {Y1.x, Y1.y, Y1.z, Y1.w};
        const float z0[4] = {Z0.x, Z0.y, Z0.z, Z0.w}, z1[4] = {Z1.x, Z1.y, Z1.z, Z1.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float lo = p ? x[e + 1] : x[e];
            const float hi = p ? x[e + 2] : x[e + 1];
            sum[e] = (lo + hi) + (y0[e] + y1[e]) + (z0[e] + z1[e]);
        }
    }
    const float4 F = *reinterpret_cast<const float4*>(f + row + mA);
    const float fv[4] = {F.x, F.y, F.z, F.w};
    float r[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) r[e] = (sum[e] - h2 * fv[e]) * sixth;
    if (p == 0 && mA == 0) {  // i = 0 is a boundary node
        own[row + 1] = r[1], own[row + 2] = r[2], own[row + 3] = r[3];
    } else {
        *reinterpret_cast<float4*>(own + row + mA) = make_float4(r[0], r[1], r[2], r[3]);
    }
}

// The first sweep of a correction that starts from zero, both half-sweeps in
// one pass (FP32 levels, four entries per thread as in rb_half4_kernel).  The
// red half-sweep from zero sets each interior red node to (0 - h^2 f)/6, a
// function of its own f alone, so the black half-sweep after it can form its
// red neighbours from f instead of reading them back: each thread writes the
// four red entries of its row that rb_half4_kernel<true> would write and
// updates the four black entries of the row with rb_half4_kernel<false>'s
// sums in their order, so the results are the same bits as the two launches.
// Red neighbours on the boundary (i, j or k = 0 or n) are not written by the
// red half-sweep; they are read from e, as the black half-sweep reads them.
constexpr int kFirstBlocksPerSM = 10;  // <= 48 registers: the fused sweep holds both colours' values
template <int VX = kVX>
__global__ void __launch_bounds__(kVThreads, kFirstBlocksPerSM)
rb_first4_kernel(float* __restrict__ e, const float* __restrict__ f, LevelView v, float h2, float sixth,
                 const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(v.n - 1, kz);
    if (act && !act[set].cont) return;
    {
        const long long so = (long long)set * 2 * v.cs;
        e += so, f += so;
    }
    float* red = e;
    float* black = e + v.cs;
    const float* fr = f;
    const float* fb = f + v.cs;
    const int n = v.n, half = n >> 1;
    const int mA = 4 * (blockIdx.x * VX + threadIdx.x);
    const int j = blockIdx.y * (kVThreads / VX) + threadIdx.y + 1;
    const int k = kz + 1;
    if (mA >= half || j >= n) return;
    const int pr = (j + k) & 1;  // parity of i along this row: red entries
    const int pb = pr ^ 1;       // black entries
    const long long row = ((long long)k * (n + 1) + j) * v.M;
    const long long P = v.M, Q = (long long)v.M * (n + 1);
    const float zero = 0.0f;
    // red entries mA-1 .. mA+4 of this row after the half-sweep from zero
    const float* fo = fr + row + mA;
    const float4 FV = *reinterpret_cast<const float4*>(fo);
    const float fv[4] = {FV.x, FV.y, FV.z, FV.w};
    float rr[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) rr[q] = (zero - h2 * fv[q]) * sixth;
    float x[6] = {(zero - h2 * fo[-1]) * sixth, rr[0], rr[1], rr[2], rr[3], (zero - h2 * fo[4]) * sixth};
    if (pr == 0) {  // red boundary nodes of the row: i = 0 (entry 0) and i = n (entry half)
        if (mA == 0) x[1] = red[row];
        if (mA + 4 == half) x[5] = red[row + half];
    }
    // red entries mA .. mA+3 of the neighbouring rows (boundary rows as stored)
    float y0[4], y1[4], z0[4], z1[4];
    auto nbr = [&](long long off, bool bnd, float* out) {
        if (bnd) {
            const float4 E = *reinterpret_cast<const float4*>(red + row + mA + off);
            out[0] = E.x, out[1] = E.y, out[2] = E.z, out[3] = E.w;
        } else {
            const float4 F = *reinterpret_cast<const float4*>(fr + row + mA + off);
            out[0] = (zero - h2 * F.x) * sixth, out[1] = (zero - h2 * F.y) * sixth;
            out[2] = (zero - h2 * F.z) * sixth, out[3] = (zero - h2 * F.w) * sixth;
        }
    };
    nbr(-P, j == 1, y0);
    nbr(P, j + 1 == n, y1);
    nbr(-Q, k == 1, z0);
    nbr(Q, k + 1 == n, z1);
    const float4 FB = *reinterpret_cast<const float4*>(fb + row + mA);
    const float fbv[4] = {FB.x, FB.y, FB.z, FB.w};
    float rb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float lo = pb ? x[q + 1] : x[q];
        const float hi = pb ? x[q + 2] : x[q + 1];
        const float sum = (lo + hi) + (y0[q] + y1[q]) + (z0[q] + z1[q]);
        rb[q] = (sum - h2 * fbv[q]) * sixth;
    }
    if (pr == 0 && mA == 0) {  // i = 0 is a boundary node
        red[row + 1] = rr[1], red[row + 2] = rr[2], red[row + 3] = rr[3];
    } else {
        *reinterpret_cast<float4*>(red + row + mA) = make_float4(rr[0], rr[1], rr[2], rr[3]);
    }
    if (pb == 0 && mA == 0) {
        black[row + 1] = rb[1], black[row + 2] = rb[2], black[row + 3] = rb[3];
    } else {
        *reinterpret_cast<float4*>(black + row + mA) = make_float4(rb[0], rb[1], rb[2], rb[3]);
    }
}

// Residual f - L u at the red node (i, j, k) of a level.
template <typename T>
__device__ __forceinline__ T red_residual(const T* __restrict__ e, const T* __restrict__ f, const LevelView& v, int i,
                                          int j, int k, T ih2)
{
    const int p = (j + k) & 1;
    const int m = i >> 1;
    const long long row = ((long long)k * (v.n + 1) + j) * v.M;
    const T* eb = e + v.cs + row;
    const long long P = v.M, Q = (long long)v.M * (v.n + 1);
    const T s = (eb[m - 1 + p] + eb[m + p]) + (eb[m - P] + eb[m + P]) + (eb[m - Q] + eb[m + Q]);
    return f[row + m] - (s - T(6) * e[row + m]) * ih2;
}

// Full weighting of the residual onto the coarse interior node (I, J, K):
// weight 1/8 at the coinciding fine node and 1/32 at its 12 edge neighbours
// (the other 14 fine nodes of the stencil are black, residual zero).
template <typename T>
__device__ __forceinline__ void restrict_node(const T* __restrict__ ef, const T* __restrict__ ff, const LevelView& vf,
                                              T* __restrict__ fc, const LevelView& vc, T ih2, int I, int J, int K)
{
    const int i = 2 * I, j = 2 * J, k = 2 * K;
    T edge = (red_residual(ef, ff, vf, i + 1, j + 1, k, ih2) + red_residual(ef, ff, vf, i - 1, j + 1, k, ih2))
           + (red_residual(ef, ff, vf, i + 1, j - 1, k, ih2) + red_residual(ef, ff, vf, i - 1, j - 1, k, ih2));
    edge += (red_residual(ef, ff, vf, i + 1, j, k + 1, ih2) + red_residual(ef, ff, vf, i - 1, j, k + 1, ih2))
          + (red_residual(ef, ff, vf, i + 1, j, k - 1, ih2) + red_residual(ef, ff, vf, i - 1, j, k - 1, ih2));
    edge += (red_residual(ef, ff, vf, i, j + 1, k + 1, ih2) + red_residual(ef, ff, vf, i, j - 1, k + 1, ih2))
          + (red_residual(ef, ff, vf, i, j + 1, k - 1, ih2) + red_residual(ef, ff, vf, i, j - 1, k - 1, ih2));
    const T centre = red_residual(ef, ff, vf, i, j, k, ih2);
    fc[node_off(vc, I, J, K)] = T(0.125) * centre + T(0.03125) * edge;
}

// A coarse node a thread, on small FP32 levels.
__global__ void __launch_bounds__(kBX * kBY)
restrict_nodes_kernel(const float* __restrict__ ef, const float* __restrict__ ff, LevelView vf, float* __restrict__ fc,
                          LevelView vc, float ih2, const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(vc.n - 1, kz);
    if (act && !act[set].cont) return;
    const long long sf = (long long)set * 2 * vf.cs, sc = (long long)set * 2 * vc.cs;
    const int I = blockIdx.x * kBX + threadIdx.x + 1;
    const int J = blockIdx.y * kBY + threadIdx.y + 1;
    const int K = kz + 1;
    if (I >= vc.n || J >= vc.n) return;
    restrict_node<float>(ef + sf, ff + sf, vf, fc + sc, vc, ih2, I, J, K);
}

// FP64: a CTA takes 16 x 4 x 2 coarse nodes and evaluates each red residual under
// them once into shared memory, 765 for 128 nodes (the first of the even ones of
// a row, 23 of them, belong to the tile beside).  With the 13 residuals of every
// node evaluated anew it is bound by the two FP64 lanes a clock (a 129^3 solve of 36
// restrictions: 785 us, 510 so, launches included); in FP32 at n = 32 and 64 it is
// bound by latency, and the second phase costs more (33^3 solve: 398 us, 405 so).
// The arithmetic is restrict_node's.
constexpr int kTI = 16, kTJ = 4, kTK = 2;             // coarse nodes of a CTA
constexpr int kTRow = kTI + 1;                        // red nodes of a fine row
constexpr int kTRows = 2 * kTJ + 1, kTPlanes = 2 * kTK + 1;

template <typename T>
__global__ void __launch_bounds__(kTI * kTJ * kTK)
restrict_tile_kernel(const T* __restrict__ ef, const T* __restrict__ ff, LevelView vf, T* __restrict__ fc,
                          LevelView vc, T ih2, int zper, const SolveState* __restrict__ act)
{
    __shared__ T res[kTPlanes][kTRows][kTRow];
    int zt;
    const int set = set_of(zper, zt);
    if (act && !act[set].cont) return;
    ef += (long long)set * 2 * vf.cs;
    ff += (long long)set * 2 * vf.cs;
    fc += (long long)set * 2 * vc.cs;
    const int I0 = blockIdx.x * kTI + 1, J0 = blockIdx.y * kTJ + 1, K0 = zt * kTK + 1;
    const int t = (int)threadIdx.x;
    for (int w = t; w < kTPlanes * kTRows * kTRow; w += kTI * kTJ * kTK) {
        const int q = w % kTRow, b = w / kTRow % kTRows, c = w / (kTRow * kTRows);
        const int j = 2 * J0 - 1 + b, k = 2 * K0 - 1 + c;
        const int i = 2 * (I0 - 1 + q) + ((j + k) & 1);
        if (i > 0 && i < vf.n && j < vf.n && k < vf.n) res[c][b][q] = red_residual(ef, ff, vf, i, j, k, ih2);
    }
    __syncthreads();
    const int a = t % kTI, b = t / kTI % kTJ, c = t / (kTI * kTJ);
    const int I = I0 + a, J = J0 + b, K = K0 + c;
    if (I >= vc.n || J >= vc.n || K >= vc.n) return;
    // the coarse node's fine row and plane; odd i = 2I -+ 1 at a and a + 1, even i = 2I at a + 1
    const T(*p0)[kTRow] = &res[2 * c + 1][2 * b + 1];
    const T(*pm)[kTRow] = &res[2 * c][2 * b + 1];
    const T(*pp)[kTRow] = &res[2 * c + 2][2 * b + 1];
    T edge = (p0[1][a + 1] + p0[1][a]) + (p0[-1][a + 1] + p0[-1][a]);
    edge += (pp[0][a + 1] + pp[0][a]) + (pm[0][a + 1] + pm[0][a]);
    edge += (pp[1][a + 1] + pp[-1][a + 1]) + (pm[1][a + 1] + pm[-1][a + 1]);
    fc[node_off(vc, I, J, K)] = T(0.125) * p0[0][a + 1] + T(0.03125) * edge;
}

// The same restriction on FP32 levels without recomputation: a CTA owns a
// tile of 32 x 8 coarse (I, J) columns and rk coarse planes (up to 8, fewer
// when the level has too few tiles to fill the GPU), and marches over
// the fine planes 2K0-1 .. 2K1-1.  For each fine plane it computes the red
// residuals of the rows 2J0-1 .. 2J0+15 and entries I0-1 .. I0+34 once (four
// consecutive entries per thread, 16-byte loads, red_residual's arithmetic in
// its order) into a three-plane shared ring; after each odd plane 2K+1 it
// full-weights coarse plane K from the ring with restrict_node's sums in their
// order.  A red residual is evaluated once per CTA instead of by each of the
// up to four coarse nodes that weight it, and the loads of fine plane k+1 are
// issued before the barriers of plane k.
constexpr int kRI = 32, kRJ = 8, kRK = 8;  // coarse tile and the most planes per CTA
constexpr int kRG = 9;                     // groups of four red entries per fine row (36 entries)
constexpr int kRR = 2 * kRJ + 1;           // fine rows per tile
static_assert(kRR * kRG <= kRI * kRJ, "one thread per residual group");

__global__ void __launch_bounds__(kRI * kRJ)
restrict_resid4_kernel(const float* __restrict__ ef, const float* __restrict__ ff, LevelView vf,
                       float* __restrict__ fc, LevelView vc, float ih2, int rk, int zper,
                       const SolveState* __restrict__ act)
{
    __shared__ __align__(16) float ring[3][kRR][kRG * 4];
    int kz;
    const int set = set_of(zper, kz);
    if (act && !act[set].cont) return;
    {
        const long long sf = (long long)set * 2 * vf.cs;
        ef += sf, ff += sf, fc += (long long)set * 2 * vc.cs;
    }
    const int n = vf.n, nc = vc.n;
    const int I0 = 1 + blockIdx.x * kRI, J0 = 1 + blockIdx.y * kRJ, K0 = 1 + kz * rk;
    const int K1 = min(K0 + rk, nc);  // coarse planes K0 .. K1-1
    const int t = threadIdx.x;
    const int mbase = I0 - 1;          // a multiple of 32: the groups start on 16-byte boundaries
    // residual phase: row rr, group rg of the fine tile
    const int rr = t / kRG, rg = t % kRG;
    const int jf = 2 * J0 - 1 + rr;
    const int m0 = mbase + 4 * rg;
    const bool ract = t < kRR * kRG && jf >= 1 && jf <= n - 1 && m0 < vf.M;
    // coarse phase: node (I, J)
    const int cI = t % kRI, cJ = t / kRI;
    const int I = I0 + cI, J = J0 + cJ;
    const bool cact = I <= nc - 1 && J <= nc - 1;
    const long long P = vf.M, Q = (long long)vf.M * (n + 1);
    // the inputs of one fine plane: the black row with its two outer neighbours, the black rows j-1, j+1
    // and planes k-1, k+1, the red values and f
    struct In {
        float4 V, Y0, Y1, Z0, Z1, E, F;
        float xl, xr;
    };
    auto load = [&](int k, In& d) {
        const long long row = ((long long)k * (n + 1) + jf) * vf.M + m0;
        const float* eb = ef + vf.cs + row;
        d.V = *reinterpret_cast<const float4*>(eb);
        d.xl = eb[-1], d.xr = eb[4];
        d.Y0 = *reinterpret_cast<const float4*>(eb - P), d.Y1 = *reinterpret_cast<const float4*>(eb + P);
        d.Z0 = *reinterpret_cast<const float4*>(eb - Q), d.Z1 = *reinterpret_cast<const float4*>(eb + Q);
        d.E = *reinterpret_cast<const float4*>(ef + row);
        d.F = *reinterpret_cast<const float4*>(ff + row);
    };
    In cur;
    if (ract) load(2 * K0 - 1, cur);
    for (int k = 2 * K0 - 1; k <= 2 * K1 - 1; ++k) {
        if (ract) {
            const int p = (jf + k) & 1;
            const float x[6] = {cur.xl, cur.V.x, cur.V.y, cur.V.z, cur.V.w, cur.xr};
            const float y0[4] = {cur.Y0.x, cur.Y0.y, cur.Y0.z, cur.Y0.w}, y1[4] = {cur.Y1.x, cur.Y1.y, cur.Y1.z, cur.Y1.w};
            const float z0[4] = {cur.Z0.x, cur.Z0.y, cur.Z0.z, cur.Z0.w}, z1[4] = {cur.Z1.x, cur.Z1.y, cur.Z1.z, cur.Z1.w};
            const float ev[4] = {cur.E.x, cur.E.y, cur.E.z, cur.E.w}, fv[4] = {cur.F.x, cur.F.y, cur.F.z, cur.F.w};
            float r[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float lo = p ? x[e + 1] : x[e];
                const float hi = p ? x[e + 2] : x[e + 1];
                const float sum = (lo + hi) + (y0[e] + y1[e]) + (z0[e] + z1[e]);
                r[e] = fv[e] - (sum - 6.0f * ev[e]) * ih2;
            }
            *reinterpret_cast<float4*>(&ring[k % 3][rr][4 * rg]) = make_float4(r[0], r[1], r[2], r[3]);
            // the next plane's loads are in flight across the barriers and the coarse plane below
            if (k < 2 * K1 - 1) load(k + 1, cur);
        }
        __syncthreads();
        if ((k & 1) && k >= 2 * K0 + 1 && cact) {
            const int K = (k - 1) >> 1;
            const float(*pm)[kRG * 4] = ring[(k + 1) % 3];  // fine plane 2K-1
            const float(*p0)[kRG * 4] = ring[(k + 2) % 3];  // 2K
            const float(*pp)[kRG * 4] = ring[k % 3];        // 2K+1
            // fine node (i, j) = (2I, 2J): row 2cJ+1 of the tile; entries I-1 (i-1) and I (i, i+1)
            const int a = 2 * cJ + 1, lo = cI, hi = cI + 1;
            float edge = (p0[a + 1][hi] + p0[a + 1][lo]) + (p0[a - 1][hi] + p0[a - 1][lo]);
            edge += (pp[a][hi] + pp[a][lo]) + (pm[a][hi] + pm[a][lo]);
            edge += (pp[a + 1][hi] + pp[a - 1][hi]) + (pm[a + 1][hi] + pm[a - 1][hi]);
            const float centre = p0[a][hi];
            fc[node_off(vc, I, J, K)] = 0.125f * centre + 0.03125f * edge;
        }
        __syncthreads();
    }
}

// The coarse-grid correction / FMG interpolation on FP32 levels with four
// consecutive black entries of a fine row per thread.  For a coarse row
// (J', K') the nodes I = mA .. mA+4 alternate between the two colour arrays
// (entries mA/2 .. mA/2+2 and mA/2 .. mA/2+1), read with 8-byte loads; the
// sums are prolong_node's, in its order, and the fine row is read and
// written with 16-byte accesses.
template <bool ADD, int VX = kVX>
__global__ void __launch_bounds__(kVThreads, kVBlocksPerSM)
prolong_black4_kernel(const float* __restrict__ ec, LevelView vc, float* __restrict__ ef, LevelView vf,
                      const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(vf.n - 1, kz);
    if (act && !act[set].cont) return;
    ec += (long long)set * 2 * vc.cs;
    ef += (long long)set * 2 * vf.cs;
    const int half = vf.n >> 1;
    const int mA = 4 * (blockIdx.x * VX + threadIdx.x);
    const int j = blockIdx.y * (kVThreads / VX) + threadIdx.y + 1;
    const int k = kz + 1;
    if (mA >= half || j >= vf.n) return;
    const int p = (1 + j + k) & 1;  // parity of i of the black nodes in this row
    const int J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
    // coarse nodes I = mA + d (d = 0..4) of row (Jr, Kr)
    auto row5 = [&](int Jr, int Kr, float* c) {
        const int ca = (mA + Jr + Kr) & 1;  // colour of the even d
        const long long base = ((long long)Kr * (vc.n + 1) + Jr) * vc.M + (mA >> 1);
        const float* A = ec + (long long)ca * vc.cs + base;
        const float* B = ec + (long long)(ca ^ 1) * vc.cs + base;
        const float2 a2 = *reinterpret_cast<const float2*>(A);
        const float2 b2 = *reinterpret_cast<const float2*>(B);
        c[0] = a2.x, c[1] = b2.x, c[2] = a2.y, c[3] = b2.y, c[4] = A[2];
    };
    float c00[5], c10[5], c01[5], c11[5];  // (J0, K0), (J1, K0), (J0, K1), (J1, K1)
    row5(J0, K0, c00);
    row5(J1, K0, c10);
    row5(J0, K1, c01);
    row5(J1, K1, c11);
    const long long o = vf.cs + ((long long)k * (vf.n + 1) + j) * vf.M + mA;
    float4 cur = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (ADD) cur = *reinterpret_cast<const float4*>(ef + o);
    const float cv[4] = {cur.x, cur.y, cur.z, cur.w};
    float r[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        // I0 = mA + e, I1 = mA + e + p
        const float a0 = c00[e], a1 = p ? c00[e + 1] : c00[e];
        const float b0 = c10[e], b1 = p ? c10[e + 1] : c10[e];
        const float d0 = c01[e], d1 = p ? c01[e + 1] : c01[e];
        const float g0 = c11[e], g1 = p ? c11[e + 1] : c11[e];
        float sv = (a0 + a1) + (b0 + b1);
        sv += (d0 + d1) + (g0 + g1);
        sv *= 0.125f;
        r[e] = ADD ? cv[e] + sv : sv;
    }
    if (p == 0 && mA == 0) {  // i = 0 is a boundary node
        ef[o + 1] = r[1], ef[o + 2] = r[2], ef[o + 3] = r[3];
    } else {
        *reinterpret_cast<float4*>(ef + o) = make_float4(r[0], r[1], r[2], r[3]);
    }
}

// Full weighting of a right-hand side (both colours) onto coarse interior nodes.
template <typename T>
__global__ void __launch_bounds__(kBX * kBY)
restrict_full_kernel(const T* __restrict__ ff, LevelView vf, T* __restrict__ fc, LevelView vc)
{
    int kz;
    const int set = set_of(vc.n - 1, kz);
    ff += (long long)set * 2 * vf.cs;
    fc += (long long)set * 2 * vc.cs;
    const int I = blockIdx.x * kBX + threadIdx.x + 1;
    const int J = blockIdx.y * kBY + threadIdx.y + 1;
    const int K = kz + 1;
    if (I >= vc.n || J >= vc.n) return;
    // node i = 2I of a row lies at entry I of one colour, i = 2I -+ 1 at I - 1 and I of the other
    const int P = vf.M;
    const long long Q = (long long)P * (vf.n + 1);
    const T* at = ff + ((2 * K) * Q + (long long)(2 * J) * P + I);
    T acc = T(0);
#pragma unroll
    for (int c = -1; c <= 1; ++c)
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
            const bool odd = ((b + c) & 1) != 0;  // j + k odd: the even nodes are black
            const T* even = at + (c * Q + b * P) + (odd ? vf.cs : 0);
            const T* other = at + (c * Q + b * P) + (odd ? 0 : vf.cs);
            const T w = T(b == 0 ? 0.5 : 0.25) * T(c == 0 ? 0.5 : 0.25);
            acc += (T(0.25) * w) * other[-1];
            acc += (T(0.5) * w) * even[0];
            acc += (T(0.25) * w) * other[0];
        }
    fc[node_off(vc, I, J, K)] = acc;
}

// Trilinear prolongation of a coarse array to the black interior nodes of the
// next finer level: assign (FMG interpolation) or add (coarse-grid correction).
template <typename T, bool ADD>
__device__ __forceinline__ void prolong_node(const T* __restrict__ ec, const LevelView& vc, T* __restrict__ ef,
                                             const LevelView& vf, int m, int j, int k)
{
    const int p = (1 + j + k) & 1;
    const int i = 2 * m + p;
    if (i < 1) return;
    const int I0 = i >> 1, I1 = (i + 1) >> 1, J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
    T s = (ec[node_off(vc, I0, J0, K0)] + ec[node_off(vc, I1, J0, K0)])
        + (ec[node_off(vc, I0, J1, K0)] + ec[node_off(vc, I1, J1, K0)]);
    s += (ec[node_off(vc, I0, J0, K1)] + ec[node_off(vc, I1, J0, K1)])
       + (ec[node_off(vc, I0, J1, K1)] + ec[node_off(vc, I1, J1, K1)]);
    s *= T(0.125);
    const long long o = vf.cs + ((long long)k * (vf.n + 1) + j) * vf.M + m;
    ef[o] = ADD ? ef[o] + s : s;
}

template <typename T, bool ADD>
__global__ void __launch_bounds__(kBX * kBY)
prolong_black_kernel(const T* __restrict__ ec, LevelView vc, T* __restrict__ ef, LevelView vf,
                     const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(vf.n - 1, kz);
    if (act && !act[set].cont) return;
    const int half = vf.n >> 1;
    const int m = blockIdx.x * kBX + threadIdx.x;
    const int j = blockIdx.y * kBY + threadIdx.y + 1;
    const int k = kz + 1;
    if (m >= half || j >= vf.n) return;
    prolong_node<T, ADD>(ec + (long long)set * 2 * vc.cs, vc, ef + (long long)set * 2 * vf.cs, vf, m, j, k);
}

// Boundary nodes of a level <- the finest boundary values at the same
// positions (u64: finest natural-layout array with nfine intervals), or 0.
__device__ __forceinline__ void face_node(int face, int a, int b, int n, int& i, int& j, int& k)
{
    switch (face) {
    case 0: i = 0; j = a; k = b; break;
    case 1: i = n; j = a; k = b; break;
    case 2: i = a; j = 0; k = b; break;
    case 3: i = a; j = n; k = b; break;
    case 4: i = a; j = b; k = 0; break;
    default: i = a; j = b; k = n; break;
    }
}

template <typename T>
__global__ void set_boundary_kernel(T* __restrict__ e, LevelView v, const double* __restrict__ u64, int nfine)
{
    int face;
    const int set = set_of(6, face);
    e += (long long)set * 2 * v.cs;
    if (u64) u64 += set * nat_elems(nfine);
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = blockIdx.y;
    if (a > v.n) return;
    int i, j, k;
    face_node(face, a, b, v.n, i, j, k);
    T val = T(0);
    if (u64) {
        const int s = nfine / v.n;
        const long long P = nfine + 1;
        val = (T)u64[(long long)i * s + P * ((long long)j * s + P * (long long)k * s)];
    }
    e[node_off(v, i, j, k)] = val;
}

// ---------------------------------------------------------------------------
// Coarse-grid solver: one CTA runs every level with n <= kCoarseN in shared
// memory (natural layout), so the small levels cost one launch instead of
// dozens.  Level l has n_l = 2 << l intervals; `top` is the level it is
// given (its right-hand side f comes from global memory).
//  fmg = 1: full multigrid from 3^3 up to `top` (boundary values injected
//           from u64, or zero), ncycle V-cycles per level;
//  fmg = 0: one V-cycle from a zero initial guess with zero boundary values.
// With fmg = 1 all nodes of e are written, boundary values included; with
// fmg = 0 the boundary entries of e must be zero on entry and stay so (the
// prolongation that reads e next reads them too), the interior is written.
// The shared-memory routines below stride over their nodes by the block's
// size: the coarse-grid kernel runs them with kCoarseThreads, the cooperative
// and cluster V-cycle kernels with kVsubThreads.  (1024 threads for the
// coarse-grid kernel measured no faster than 512.)
constexpr int kCoarseThreads = 512;
constexpr int kVsubThreads = 512;
constexpr int kMaxCoarseLevels = 4;  // n = 2, 4, 8, 16

__host__ __device__ inline int cube(int n) { return (n + 1) * (n + 1) * (n + 1); }

template <typename T>
struct CoarseSmem {
    T* u[kMaxCoarseLevels];
    T* f[kMaxCoarseLevels];
    T* r[kMaxCoarseLevels];
    T* x[kMaxCoarseLevels];  // row exchange of the levels run by rows
};

// Levels whose V-cycle keeps rows in registers (Row below).  In FP64 the pipe (2 operations
// a clock) bounds these levels, and more threads with a node each keep it
// busier (17^3 V-cycle 71 us either way, 9^3 17 us against 21).
template <typename T>
__host__ __device__ constexpr bool rows_at(int n) { return n >= 8 && sizeof(T) == 4; }
template <typename T, int L>
constexpr bool by_rows() { return rows_at<T>(2 << L); }

// Elements of level n in the coarse solver's shared memory: u, f, r and the row exchange.
template <typename T>
__host__ __device__ inline int row_exchange(int n) { return rows_at<T>(n) ? (n + 1) * (n + 2) * n : 0; }
__host__ __device__ inline int cube4(int n) { return (cube(n) + 3) & ~3; }
template <typename T>
__host__ __device__ inline int coarse_elems(int n) { return 3 * cube4(n) + row_exchange<T>(n); }

template <typename T>
__device__ __forceinline__ void coarse_layout(CoarseSmem<T>& S, T* base, int top)
{
#pragma unroll
    for (int l = 0; l < kMaxCoarseLevels; ++l) {
        if (l > top) break;
        const int c = cube4(2 << l);
        S.x[l] = base;
        S.u[l] = base + row_exchange<T>(2 << l);
        S.f[l] = S.u[l] + c;
        S.r[l] = S.f[l] + c;
        base += coarse_elems<T>(2 << l);
    }
}

// Every level size is a compile-time constant (N = 2 << L), so the index
// arithmetic below is shifts and multiplications.  Each routine is run by the
// whole block (stride blockDim.x, a multiple of 8) and ends with its barrier;
// the level n = 4 has its own form in one warp (warp_vcycle4), which spares it a
// block-wide barrier per phase.

// a b + c rounded once (written out: where a product is the same in every
// sweep, the compiler would round it on its own and keep it).
__device__ __forceinline__ float fused(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fused(double a, double b, double c) { return __fma_rn(a, b, c); }

// One colour of the interior of an N-level: row (j, k) holds that colour's
// nodes at i = first, first + 2, ... (first = 1 or 2), N/2 slots per row.
// The stride is a multiple of N/2, so a thread keeps its slot and steps its
// row (j, k) without divisions (the residual and the prolongation below do
// the same with N lanes per row, the last one idle).
// ZERO: every neighbour is known to be zero.
template <typename T, int N, bool ZERO = false>
__device__ void sm_relax(T* u, const T* f, T h2, int colour)
{
    constexpr int M = N - 1, P = N + 1, H = N / 2, ROWS = M * M;
    const int dr = (int)blockDim.x / H;  // rows advanced per pass
    const int dj = dr % M, dk = dr / M;
    const int sl = (int)threadIdx.x % H;
    int row = (int)threadIdx.x / H;
    int j = row % M + 1, k = row / M + 1;
    for (; row < ROWS; row += dr) {
        const int i = 1 + (((1 + j + k) & 1) != colour ? 1 : 0) + 2 * sl;
        if (i <= M) {
            const int o = i + P * (j + P * k);
            T sum = T(0);
            if (!ZERO) sum = (u[o + 1] + u[o - 1]) + (u[o + P] + u[o - P]) + (u[o + P * P] + u[o - P * P]);
            u[o] = fused(-h2, f[o], sum) * (T(1) / T(6));
        }
        j += dj;
        k += dk;
        if (j > M) {
            j -= M;
            ++k;
        }
    }
    __syncthreads();
}

template <typename T, int N>
__device__ void sm_residual(const T* u, const T* f, T* r, T ih2)
{
    constexpr int M = N - 1, P = N + 1, ROWS = M * M;
    const int dr = (int)blockDim.x / N;  // rows advanced per pass: a row is N lanes, the last one idle
    const int dj = dr % M, dk = dr / M;
    const int i = (int)threadIdx.x % N + 1;
    int row = (int)threadIdx.x / N;
    int j = row % M + 1, k = row / M + 1;
    for (; row < ROWS; row += dr) {
        if (i <= M) {
            const int o = i + P * (j + P * k);
            const T sum = (u[o + 1] + u[o - 1]) + (u[o + P] + u[o - P]) + (u[o + P * P] + u[o - P * P]);
            r[o] = f[o] - (sum - T(6) * u[o]) * ih2;
        }
        j += dj;
        k += dk;
        if (j > M) {
            j -= M;
            ++k;
        }
    }
    __syncthreads();
}

template <typename T, int NF>
__device__ void sm_restrict(const T* fine, T* coarse)
{
    constexpr int NC = NF / 2, MC = NC - 1, PF = NF + 1, PC = NC + 1, TOT = MC * MC * MC;
    for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) {
        const int I = t % MC + 1, J = (t / MC) % MC + 1, K = t / (MC * MC) + 1;
        T acc = T(0);
#pragma unroll
        for (int c = -1; c <= 1; ++c)
#pragma unroll
            for (int b = -1; b <= 1; ++b)
#pragma unroll
                for (int a = -1; a <= 1; ++a) {
                    const T w = T(0.125) * T(a == 0 ? 2 : 1) * T(b == 0 ? 2 : 1) * T(c == 0 ? 2 : 1) * T(0.125);
                    acc += w * fine[(2 * I + a) + PF * ((2 * J + b) + PF * (2 * K + c))];
                }
        coarse[I + PC * (J + PC * K)] = acc;
    }
    __syncthreads();
}

template <typename T, int NC>
__device__ void sm_prolong(const T* coarse, T* fine)
{
    constexpr int NF = 2 * NC, M = NF - 1, PF = NF + 1, PC = NC + 1, ROWS = M * M;
    const int dr = (int)blockDim.x / NF;  // rows advanced per pass: a row is NF lanes, the last one idle
    const int dj = dr % M, dk = dr / M;
    const int i = (int)threadIdx.x % NF + 1;
    int row = (int)threadIdx.x / NF;
    int j = row % M + 1, k = row / M + 1;
    for (; row < ROWS; row += dr) {
        if (i <= M) {
            const int I0 = i >> 1, I1 = (i + 1) >> 1, J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
            T sum = (coarse[I0 + PC * (J0 + PC * K0)] + coarse[I1 + PC * (J0 + PC * K0)])
                  + (coarse[I0 + PC * (J1 + PC * K0)] + coarse[I1 + PC * (J1 + PC * K0)]);
            sum += (coarse[I0 + PC * (J0 + PC * K1)] + coarse[I1 + PC * (J0 + PC * K1)])
                 + (coarse[I0 + PC * (J1 + PC * K1)] + coarse[I1 + PC * (J1 + PC * K1)]);
            sum *= T(0.125);
            const int o = i + PF * (j + PF * k);
            fine[o] = sum;
        }
        j += dj;
        k += dk;
        if (j > M) {
            j -= M;
            ++k;
        }
    }
    __syncthreads();
}

// The correction of the black nodes alone (the red half-sweep after it does not
// read the red ones): as sm_prolong, with the slots of sm_relax.
template <typename T, int NC>
__device__ void sm_correct(const T* coarse, T* fine)
{
    constexpr int NF = 2 * NC, M = NF - 1, PF = NF + 1, PC = NC + 1, H = NF / 2, ROWS = M * M;
    const int dr = (int)blockDim.x / H, sl = (int)threadIdx.x % H;
    for (int row = (int)threadIdx.x / H; row < ROWS; row += dr) {
        const int j = row % M + 1, k = row / M + 1;
        const int i = 1 + ((j + k) & 1) + 2 * sl;
        if (i <= M) {
            const int I0 = i >> 1, I1 = (i + 1) >> 1, J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
            T sum = (coarse[I0 + PC * (J0 + PC * K0)] + coarse[I1 + PC * (J0 + PC * K0)])
                  + (coarse[I0 + PC * (J1 + PC * K0)] + coarse[I1 + PC * (J1 + PC * K0)]);
            sum += (coarse[I0 + PC * (J0 + PC * K1)] + coarse[I1 + PC * (J0 + PC * K1)])
                 + (coarse[I0 + PC * (J1 + PC * K1)] + coarse[I1 + PC * (J1 + PC * K1)]);
            sum *= T(0.125);
            const int o = i + PF * (j + PF * k);
            fine[o] = fine[o] + sum;
        }
    }
    __syncthreads();
}

template <typename T, int N>
__device__ void sm_fill(T* a, T val)
{
    constexpr int TOT = (N + 1) * (N + 1) * (N + 1);
    for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) a[t] = val;
    __syncthreads();
}

// The single unknown of the 3^3 grid (Section 2): u = (sum of 6 nbrs - h^2 f)/6.
template <typename T>
__device__ void sm_coarsest(T* u, const T* f, T h)
{
    if (threadIdx.x == 0) {
        const T sum = (u[14] + u[12]) + (u[16] + u[10]) + (u[22] + u[4]);
        u[13] = (sum - h * h * f[13]) * (T(1) / T(6));
    }
    __syncthreads();
}

// --- the levels n = 8 and 16 with a row of nodes per thread ---------------------------------------------------------
// A phase of these levels is bound by latencies (a few shared-memory reads, a
// short chain of sums, a block barrier), so a thread keeps a whole interior row
// (j, k) and its right-hand side in registers for the whole V-cycle: nodes of
// odd i in O, of even i in E (its last entry the boundary node i = n), the
// x-neighbours are its own, and the rows j +- 1, k +- 1 come from an exchange
// array in vectors of four nodes.  Rows with j + k even (s = 0) take the first
// half of the threads and the others the second, so that a warp updates O or
// E as a whole.  Measured, one V-cycle from the level 17^3 (FP32, its launch
// included): 10.1 us, 17.3 with a node at a time from the natural layout (a
// half-sweep 0.8 us).  The nodes' arithmetic is sm_relax's, sm_residual's and
// sm_prolong's; the correction goes to the black nodes only (the red half-sweep
// after it does not read the red ones).
template <typename T>
struct alignas(16) RowVec {
    T v[4];
};

template <typename T, int N>
struct Row {
    static constexpr int M = N - 1, P = N + 1, H = N / 2, NV = N / 8;
    static constexpr int ROWS = 2 * (N + 1) * (H + 1);         // rows (s, k, j >> 1) of the exchange
    static constexpr int HALF = (M * M / 2 + 1 + 31) / 32 * 32;  // threads of the rows of one s
    int s, j, k;
    bool on;
    T O[H], E[H], eL;  // i = 1, 3, ..; 2, 4, .., N; i = 0
    T fO[H], fE[H];

    __device__ __forceinline__ Row()
    {
        const int t = (int)threadIdx.x;
        s = t >= HALF ? 1 : 0;
        const int r = t - s * HALF;
        // planes in pairs: for s = 0 plane 2q+1 has H rows (odd j) and plane 2q+2 H-1 (even j); for s = 1 the reverse
        const int q = r / M, m = r - q * M, first = s ? H - 1 : H;
        k = 2 * q + 1 + (m >= first ? 1 : 0);
        j = m < first ? 2 * m + (s ? 2 : 1) : 2 * (m - first) + (s ? 1 : 2);
        on = t < 2 * HALF && k <= M;
    }
    static __device__ __forceinline__ int row(int sv, int kv, int jv) { return (sv * P + kv) * (H + 1) + (jv >> 1); }
    static __device__ __forceinline__ RowVec<T>* vec(T* x, int v, int even, int r)
    {
        return reinterpret_cast<RowVec<T>*>(x) + (v * 2 + even) * ROWS + r;
    }
    template <bool EVEN>
    __device__ __forceinline__ void put(T* x) const
    {
        const T* a = EVEN ? E : O;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            RowVec<T> w;
#pragma unroll
            for (int e = 0; e < 4; ++e) w.v[e] = a[4 * v + e];
            *vec(x, v, EVEN, row(s, k, j)) = w;
        }
    }
    // the sums of the six neighbours of the row's nodes of one parity of i; ZERO: known to be zero
    template <bool EVEN>
    __device__ __forceinline__ void sums(T* x, T (&sum)[H]) const
    {
        const int o = s ^ 1;
        const int ym = row(o, k, j - 1), yp = row(o, k, j + 1), zm = row(o, k - 1, j), zp = row(o, k + 1, j);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const RowVec<T> a = *vec(x, v, EVEN, ym), b = *vec(x, v, EVEN, yp);
            const RowVec<T> c = *vec(x, v, EVEN, zm), d = *vec(x, v, EVEN, zp);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int q = 4 * v + e;
                const T right = EVEN ? (q + 1 < H ? O[q + 1 < H ? q + 1 : 0] : T(0)) : E[q];
                const T left = EVEN ? O[q] : (q == 0 ? eL : E[q == 0 ? 0 : q - 1]);
                sum[q] = (right + left) + (b.v[e] + a.v[e]) + (d.v[e] + c.v[e]);
            }
        }
    }
    template <bool EVEN, bool ZERO>
    __device__ __forceinline__ void relax_own(T* x, T h2)
    {
        T sum[H];
        if (ZERO) {
#pragma unroll
            for (int q = 0; q < H; ++q) sum[q] = T(0);
        } else {
            sums<EVEN>(x, sum);
        }
#pragma unroll
        for (int q = 0; q < (EVEN ? H - 1 : H); ++q) {
            T& u = EVEN ? E[q] : O[q];
            u = fused(-h2, EVEN ? fE[q] : fO[q], sum[q]) * (T(1) / T(6));
        }
        put<EVEN>(x);
    }
    template <bool ZERO>
    __device__ __forceinline__ void relax(T* x, T h2, int colour)
    {
        if (on) {
            if ((s ^ colour) == 0) relax_own<true, ZERO>(x, h2);  // this colour's nodes of the row have even i
            else relax_own<false, ZERO>(x, h2);
        }
        __syncthreads();
    }
    // Residual of every interior node of the row into r: rows of N + 4, odd i first and even i from H on, so that the
    // threads of restrict_rows read neighbouring words.
    static constexpr int RS = N + 4;
    __device__ __forceinline__ void residual(T* x, T* r, T ih2) const
    {
        if (on) {
            T* at = r + RS * (j - 1 + M * (k - 1));
            auto half = [&](const T* f, const T* u, const T (&sum)[H], T* to) {
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    RowVec<T> w;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = 4 * v + e;
                        w.v[e] = fused(-fused(T(-6), u[q], sum[q]), ih2, f[q]);
                    }
                    reinterpret_cast<RowVec<T>*>(to)[v] = w;
                }
            };
            T sum[H];
            sums<false>(x, sum);
            half(fO, O, sum, at);
            sums<true>(x, sum);
            half(fE, E, sum, at + H);
        }
        __syncthreads();
    }
    // sm_restrict from that layout
    static __device__ __forceinline__ void restrict_rows(const T* r, T* coarse)
    {
        constexpr int MC = H - 1, PC = H + 1;
        for (int t = (int)threadIdx.x; t < MC * MC * MC; t += (int)blockDim.x) {
            const int I = t % MC + 1, J = (t / MC) % MC + 1, K = t / (MC * MC) + 1;
            T acc = T(0);
#pragma unroll
            for (int c = -1; c <= 1; ++c)
#pragma unroll
                for (int b = -1; b <= 1; ++b) {
                    const T* at = r + RS * (2 * J + b - 1 + M * (2 * K + c - 1)) + I - 1;
                    const T w = T(0.125) * T(b == 0 ? 2 : 1) * T(c == 0 ? 2 : 1) * T(0.125);
                    acc += w * at[0];
                    acc += T(2) * w * at[H];
                    acc += w * at[1];
                }
            coarse[I + PC * (J + PC * K)] = acc;
        }
        __syncthreads();
    }
    // the correction of the row's black nodes from the natural coarse array c
    __device__ __forceinline__ void correct(T* x, const T* c)
    {
        if (on) {
            constexpr int PC = H + 1;
            const T* c00 = c + PC * ((j >> 1) + PC * (k >> 1));
            const T* c10 = c + PC * (((j + 1) >> 1) + PC * (k >> 1));
            const T* c01 = c + PC * ((j >> 1) + PC * ((k + 1) >> 1));
            const T* c11 = c + PC * (((j + 1) >> 1) + PC * ((k + 1) >> 1));
            if (s == 0) {  // black: odd i = 2q + 1, between I = q and q + 1
#pragma unroll
                for (int q = 0; q < H; ++q) {
                    T sum = (c00[q] + c00[q + 1]) + (c10[q] + c10[q + 1]);
                    sum += (c01[q] + c01[q + 1]) + (c11[q] + c11[q + 1]);
                    sum *= T(0.125);
                    O[q] = O[q] + sum;
                }
                put<false>(x);
            } else {  // even i = 2q + 2, on I = q + 1
#pragma unroll
                for (int q = 0; q < H - 1; ++q) {
                    T sum = (c00[q + 1] + c00[q + 1]) + (c10[q + 1] + c10[q + 1]);
                    sum += (c01[q + 1] + c01[q + 1]) + (c11[q + 1] + c11[q + 1]);
                    sum *= T(0.125);
                    E[q] = E[q] + sum;
                }
                put<true>(x);
            }
        }
        __syncthreads();
    }
    __device__ __forceinline__ void load_f(const T* f)
    {
        const T* at = f + P * (j + P * k);
#pragma unroll
        for (int q = 0; q < H; ++q) {
            fO[q] = on ? at[2 * q + 1] : T(0);
            fE[q] = on && q < H - 1 ? at[2 * q + 2] : T(0);
        }
    }
    __device__ __forceinline__ void load_u(const T* u)
    {
        const T* at = u + P * (j + P * k);
        eL = on ? at[0] : T(0);
#pragma unroll
        for (int q = 0; q < H; ++q) {
            O[q] = on ? at[2 * q + 1] : T(0);
            E[q] = on ? at[2 * q + 2] : T(0);
        }
    }
    // The same row of a level in global memory (colour-split rows of lv.M entries): the colour with even i holds
    // i = 2m at m, the other i = 2m + 1.
    __device__ __forceinline__ void load_f(const T* __restrict__ f, const LevelView& lv)
    {
        clear_f();
        if (!on) return;
        const long long at = ((long long)k * P + j) * lv.M;
        const T* ev = f + (s ? lv.cs : 0) + at;  // s = 0: red has even i
        const T* od = f + (s ? 0 : lv.cs) + at;
#pragma unroll
        for (int q = 0; q < H; ++q) {
            fO[q] = od[q];
            if (q < H - 1) fE[q] = ev[q + 1];
        }
    }
    __device__ __forceinline__ void store_u(T* __restrict__ e, const LevelView& lv) const
    {
        if (!on) return;
        const long long at = ((long long)k * P + j) * lv.M;
        T* ev = e + (s ? lv.cs : 0) + at;
        T* od = e + (s ? 0 : lv.cs) + at;
#pragma unroll
        for (int q = 0; q < H; ++q) {
            od[q] = O[q];
            if (q < H - 1) ev[q + 1] = E[q];
        }
    }
    __device__ __forceinline__ void clear_f()
    {
#pragma unroll
        for (int q = 0; q < H; ++q) fO[q] = T(0), fE[q] = T(0);
    }
    // zero boundary rows in the exchange
    static __device__ __forceinline__ void clear_boundary(T* x)
    {
        for (int t = (int)threadIdx.x; t < 4 * N; t += (int)blockDim.x) {
            const int side = t / N, a = t - side * N;
            const int jv = side == 0 ? 0 : side == 1 ? N : a + (side == 3 ? 1 : 0);
            const int kv = side == 0 ? a + 1 : side == 1 ? a : side == 2 ? 0 : N;
            const RowVec<T> z = {{T(0), T(0), T(0), T(0)}};
#pragma unroll
            for (int v = 0; v < 2 * NV; ++v) *vec(x, v >> 1, v & 1, row((jv + kv) & 1, kv, jv)) = z;
        }
    }
    __device__ __forceinline__ void clear_u()
    {
        eL = T(0);
#pragma unroll
        for (int q = 0; q < H; ++q) O[q] = T(0), E[q] = T(0);
    }
    __device__ __forceinline__ void store_u(T* u) const
    {
        if (on) {
            T* at = u + P * (j + P * k);
#pragma unroll
            for (int q = 0; q < H; ++q) {
                at[2 * q + 1] = O[q];
                if (q < H - 1) at[2 * q + 2] = E[q];
            }
        }
        __syncthreads();
    }
    // the whole natural array u, boundary rows included, into the exchange
    static __device__ __forceinline__ void fill_exchange(T* x, const T* u)
    {
        for (int t = (int)threadIdx.x; t < P * P; t += (int)blockDim.x) {
            const int jv = t % P, kv = t / P, sv = (jv + kv) & 1;
            const T* at = u + P * (jv + P * kv);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                RowVec<T> o, e;
#pragma unroll
                for (int q = 0; q < 4; ++q) o.v[q] = at[8 * v + 2 * q + 1], e.v[q] = at[8 * v + 2 * q + 2];
                *vec(x, v, 0, row(sv, kv, jv)) = o;
                *vec(x, v, 1, row(sv, kv, jv)) = e;
            }
        }
        __syncthreads();
    }
};

// The V-cycle of the levels n = 4 and 2 in the registers of one warp: a lane per
// node, neighbours by shuffles; u and f are the natural arrays of the level
// n = 4.  The arithmetic of sm_relax, sm_residual, sm_restrict (the terms in the
// order of the lanes), sm_coarsest and sm_prolong.
template <typename T>
__device__ void warp_vcycle4(T* u, const T* f, T h, int npre, int npost)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int P = 5;
    const int l = (int)threadIdx.x & 31, n = l < 27 ? l : 26;
    const int i = n % 3 + 1, j = (n / 3) % 3 + 1, k = n / 9 + 1;
    const int o = i + P * (j + P * k);
    T v = u[o];
    const T fv = f[o];
    const T bx = i == 2 ? T(0) : u[i == 1 ? o - 1 : o + 1];  // the boundary neighbour along each axis, if there is one
    const T by = j == 2 ? T(0) : u[j == 1 ? o - P : o + P];
    const T bz = k == 2 ? T(0) : u[k == 1 ? o - P * P : o + P * P];
    auto sum6 = [&]() {
        const T xp = __shfl_down_sync(kAll, v, 1), xm = __shfl_up_sync(kAll, v, 1);
        const T yp = __shfl_down_sync(kAll, v, 3), ym = __shfl_up_sync(kAll, v, 3);
        const T zp = __shfl_down_sync(kAll, v, 9), zm = __shfl_up_sync(kAll, v, 9);
        return ((i == 3 ? bx : xp) + (i == 1 ? bx : xm)) + ((j == 3 ? by : yp) + (j == 1 ? by : ym)) +
               ((k == 3 ? bz : zp) + (k == 1 ? bz : zm));
    };
    const int colour = (i + j + k) & 1;
    const T h2 = h * h;
    auto relax = [&](int c) {
        const T w = fused(-h2, fv, sum6()) * (T(1) / T(6));
        if (colour == c) v = w;
    };
    for (int q = 0; q < npre; ++q) {
        relax(0);
        relax(1);
    }
    {
        const T r = fused(-fused(T(-6), v, sum6()), T(1) / h2, fv);
        const T w = T(0.125) * T(i == 2 ? 2 : 1) * T(j == 2 ? 2 : 1) * T(k == 2 ? 2 : 1) * T(0.125);
        const T p = w * r;  // exact: w is a power of two
        T acc = T(0);
#pragma unroll
        for (int q = 0; q < 27; ++q) acc += __shfl_sync(kAll, p, q);
        const T hc = h * T(2);
        const T c = fused(-(hc * hc), acc, T(0)) * (T(1) / T(6));
        // the coarse node (1, 1, 1) is the only one that is not zero
        const T x0 = (i >> 1) == 1 ? c : T(0), x1 = ((i + 1) >> 1) == 1 ? c : T(0);
        auto at = [&](int J, int K) { return J == 1 && K == 1 ? x0 + x1 : T(0); };
        const int J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
        T s = at(J0, K0) + at(J1, K0);
        s += at(J0, K1) + at(J1, K1);
        s *= T(0.125);
        v = v + s;
    }
    for (int q = 0; q < npost; ++q) {
        relax(0);
        relax(1);
    }
    if (l < 27) u[o] = v;
}

template <typename T, int L, bool ZERO>
__device__ void sm_vcycle(CoarseSmem<T>& S, T h, int npre, int npost);

// The V-cycle from level L down on a row of nodes per thread: right-hand side
// (and, unless ZERO, the start) in `row`, which holds the result at the end.
template <typename T, int L, bool ZERO>
__device__ __forceinline__ void row_vcycle(CoarseSmem<T>& S, Row<T, (2 << L)>& row, T h, int npre, int npost)
{
    constexpr int N = 2 << L;
    for (int q = 0; q < npre; ++q) {
        if (ZERO && q == 0) row.template relax<true>(S.x[L], h * h, 0);
        else row.template relax<false>(S.x[L], h * h, 0);
        row.template relax<false>(S.x[L], h * h, 1);
    }
    row.residual(S.x[L], S.r[L], T(1) / (h * h));
    Row<T, N>::restrict_rows(S.r[L], S.f[L - 1]);
    if constexpr (!(ZERO && L - 1 >= 2)) sm_fill<T, N / 2>(S.u[L - 1], T(0));
    sm_vcycle<T, L - 1, ZERO && L - 1 >= 2>(S, h * T(2), npre, npost);
    row.correct(S.x[L], S.u[L - 1]);
    for (int q = 0; q < npost; ++q) {
        row.template relax<false>(S.x[L], h * h, 0);
        row.template relax<false>(S.x[L], h * h, 1);
    }
}

// V(npre, npost) cycle from level L down to the 3^3 grid; the coarser levels
// start from zero (zero boundary values), level L from what u[L] holds, or, with
// ZERO, from zero with zero boundary values (only these are read of u[L], and
// the boundary rows of its exchange array are zero).  The levels n <= 4 are run
// by warp 0 while the rest of the block waits.
template <typename T, int L, bool ZERO = false>
__device__ void sm_vcycle(CoarseSmem<T>& S, T h, int npre, int npost)
{
    constexpr int N = 2 << L;
    if constexpr (L == 0) {
        sm_coarsest<T>(S.u[0], S.f[0], h);
    } else if constexpr (L == 1) {
        if (threadIdx.x < 32) warp_vcycle4(S.u[1], S.f[1], h, npre, npost);
        __syncthreads();
    } else if constexpr (by_rows<T, L>()) {
        Row<T, N> row;
        row.load_f(S.f[L]);
        if (ZERO) {
            row.clear_u();
        } else {
            Row<T, N>::fill_exchange(S.x[L], S.u[L]);
            row.load_u(S.u[L]);
        }
        row_vcycle<T, L, ZERO>(S, row, h, npre, npost);
        row.store_u(S.u[L]);
    } else {
        for (int q = 0; q < npre; ++q) {
            if (ZERO && q == 0) sm_relax<T, N, true>(S.u[L], S.f[L], h * h, 0);
            else sm_relax<T, N>(S.u[L], S.f[L], h * h, 0);
            sm_relax<T, N>(S.u[L], S.f[L], h * h, 1);
        }
        sm_residual<T, N>(S.u[L], S.f[L], S.r[L], T(1) / (h * h));
        sm_restrict<T, N>(S.r[L], S.f[L - 1]);
        sm_fill<T, N / 2>(S.u[L - 1], T(0));
        sm_vcycle<T, L - 1, (L - 1 >= 2)>(S, h * T(2), npre, npost);
        sm_correct<T, N / 2>(S.u[L - 1], S.u[L]);
        for (int q = 0; q < npost; ++q) {
            sm_relax<T, N>(S.u[L], S.f[L], h * h, 0);
            sm_relax<T, N>(S.u[L], S.f[L], h * h, 1);
        }
    }
}

// Before a V-cycle by rows that starts from zero on level L: zero boundary rows
// in the exchange arrays, and zero boundary values in u of the levels under it
// (their interior is written before it is read).
template <typename T, int L>
__device__ void clear_rows(CoarseSmem<T>& S)
{
    if constexpr (by_rows<T, L>()) {
        Row<T, (2 << L)>::clear_boundary(S.x[L]);
        if constexpr (L - 1 >= 2)
            for (int t = (int)threadIdx.x; t < cube(1 << L); t += (int)blockDim.x) S.u[L - 1][t] = T(0);
        clear_rows<T, L - 1>(S);
    }
}

// f restricted from level L down to level 0
template <typename T, int L>
__device__ void sm_restrict_down(CoarseSmem<T>& S)
{
    if constexpr (L > 0) {
        sm_restrict<T, (2 << L)>(S.f[L], S.f[L - 1]);
        sm_restrict_down<T, L - 1>(S);
    }
}

// boundary values of level L (and below): injected from the finest grid (nfine intervals), or zero
template <typename T, int L>
__device__ void sm_inject(CoarseSmem<T>& S, const double* __restrict__ u64, int nfine)
{
    constexpr int N = 2 << L, P = N + 1, TOT = P * P * P;
    const int st = u64 ? nfine / N : 0;
    const long long PF = nfine + 1;
    for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) {
        const int i = t % P, j = (t / P) % P, k = t / (P * P);
        const bool inner = i > 0 && i < N && j > 0 && j < N && k > 0 && k < N;
        T val = T(0);
        if (!inner && u64) val = (T)u64[(long long)i * st + PF * ((long long)j * st + PF * (long long)k * st)];
        S.u[L][t] = val;
    }
    if constexpr (L > 0) sm_inject<T, L - 1>(S, u64, nfine);
}

// FMG from the 3^3 grid up to level L: prolong, then ncycle V-cycles per level
template <typename T, int L>
__device__ void sm_fmg_up(CoarseSmem<T>& S, T h0, int ncycle, int npre, int npost)
{
    if constexpr (L == 0) {
        sm_coarsest(S.u[0], S.f[0], h0);
    } else {
        sm_fmg_up<T, L - 1>(S, h0, ncycle, npre, npost);
        const T h = h0 / T(1 << L);
        sm_prolong<T, (2 << (L - 1))>(S.u[L - 1], S.u[L]);
        for (int c = 0; c < ncycle; ++c) sm_vcycle<T, L>(S, h, npre, npost);
    }
}

template <typename T, int TOP>
__device__ void coarse_run(unsigned char* smem_raw, int fmg, T* __restrict__ e, const T* __restrict__ f, LevelView v,
                           T htop, const double* __restrict__ u64, int nfine, int ncycle, int npre, int npost)
{
    CoarseSmem<T> S;
    coarse_layout(S, reinterpret_cast<T*>(smem_raw), TOP);
    constexpr int N = 2 << TOP, P = N + 1, TOT = P * P * P;
    if constexpr (by_rows<T, TOP>()) {
        if (!fmg) {  // the top level goes from global memory to the threads' rows and back (its boundary nodes hold zeros)
            Row<T, N> row;
            row.load_f(f, v);
            row.clear_u();
            clear_rows<T, TOP>(S);
            __syncthreads();
            row_vcycle<T, TOP, true>(S, row, htop, npre, npost);
            row.store_u(e, v);
            return;
        }
    }
    // right-hand side of the top level (interior), zero elsewhere
#pragma unroll 5
    for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) {
        const int i = t % P, j = (t / P) % P, k = t / (P * P);
        const bool inner = i > 0 && i < N && j > 0 && j < N && k > 0 && k < N;
        S.f[TOP][t] = inner ? f[node_off(v, i, j, k)] : T(0);
    }
    if (fmg) {
        __syncthreads();
        sm_restrict_down<T, TOP>(S);
        sm_inject<T, TOP>(S, u64, nfine);
        __syncthreads();
        sm_fmg_up<T, TOP>(S, htop * T(1 << TOP), ncycle, npre, npost);
    } else {
        for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) S.u[TOP][t] = T(0);
        __syncthreads();
        sm_vcycle<T, TOP, (TOP >= 2)>(S, htop, npre, npost);
    }
#pragma unroll 5
    for (int t = threadIdx.x; t < TOT; t += (int)blockDim.x) {
        const int i = t % P, j = (t / P) % P, k = t / (P * P);
        e[node_off(v, i, j, k)] = S.u[TOP][t];
    }
}

template <typename T, int TOP>
__global__ void __launch_bounds__(kCoarseThreads)
coarse_kernel(int fmg, T* __restrict__ e, const T* __restrict__ f, LevelView v, T htop, const double* __restrict__ u64,
              int nfine, int ncycle, int npre, int npost, const SolveState* __restrict__ act)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int set = blockIdx.x;  // one CTA per set
    if (act && !act[set].cont) return;
    const long long so = (long long)set * 2 * v.cs;
    coarse_run<T, TOP>(smem_raw, fmg, e + so, f + so, v, htop, u64 ? u64 + set * nat_elems(nfine) : nullptr, nfine,
                       ncycle, npre, npost);
}

// ---------------------------------------------------------------------------
// The V-cycle below a level, as one cooperative kernel: the levels top .. 1 of
// a.lev (level 0 = the coarse-grid level) are smoothed, restricted and
// corrected phase by phase, every CTA taking a grid-stride share of each
// phase, with a grid barrier between phases; CTA 0 runs the coarse-grid solver
// in shared memory.  Each node's arithmetic is that of the one-launch-per-step
// kernels (rb_node, restrict_node, prolong_node, coarse_run), and nodes within
// a phase are independent, so the result is the same bits.  The barrier
// counter is zeroed before each launch; a barrier that waits too long records
// a fault (reported by the solve as a timeout) and the kernel gives up.
template <typename T>
struct VsubLevel {
    T* e;
    T* f;
    LevelView v;
    T h;
};

constexpr int kVsubMaxLevels = 6;

template <typename T>
struct VsubArgs {
    VsubLevel<T> lev[kVsubMaxLevels];
    int top;        // index of the top level in lev
    int zero_top;   // the top level's correction starts from zero
    int npre, npost;
    unsigned* bar;  // barrier counter (zeroed before the launch)
    int* fault;
    long long polls;  // a barrier gives up after this many polls of the counter
    const SolveState* act;  // cluster form with several sets: skip the sets that have stopped
};

__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned& gen, int* fault, long long polls)
{
    __syncthreads();
    __shared__ int give_up;
    if (threadIdx.x == 0) {
        give_up = 0;
        gen += gridDim.x;
        __threadfence();
        atomicAdd(bar, 1u);
        long long spins = 0;
        while (*(volatile unsigned*)bar < gen) {
            if (++spins > polls) {
                atomicExch(fault, 4);
                give_up = 1;
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
    return give_up == 0;
}

// Phase work is dealt to `nblk` CTAs, this one being `rank`.
template <typename T>
__device__ void vsub_rb(const VsubLevel<T>& L, int colour, bool zero, int rank, int nblk)
{
    const LevelView& v = L.v;
    const int half = v.n >> 1, rows = v.n - 1;
    const long long W = (long long)half * rows * rows;
    const T h2 = L.h * L.h, sixth = T(1) / T(6);
    T* own = L.e + (long long)colour * v.cs;
    const T* other = L.e + (long long)(colour ^ 1) * v.cs;
    const T* f = L.f + (long long)colour * v.cs;
    for (long long w = rank * (long long)blockDim.x + threadIdx.x; w < W; w += (long long)nblk * blockDim.x) {
        const int m = (int)(w % half);
        const long long r = w / half;
        const int j = (int)(r % rows) + 1, k = (int)(r / rows) + 1;
        if (zero)
            rb_node<T, true>(own, other, f, v, colour, h2, sixth, m, j, k);
        else
            rb_node<T, false>(own, other, f, v, colour, h2, sixth, m, j, k);
    }
}

// The V-cycle on lev[top] .. lev[0] with `nblk` CTAs sharing each phase and
// `sync()` between phases (false: a barrier gave up, stop); CTA rank 0 runs
// the coarse-grid level in its shared memory.
template <typename T, class Sync>
__device__ void vsub_body(const VsubArgs<T>& a, const VsubLevel<T>* lev, int rank, int nblk, unsigned char* smem_raw,
                          Sync&& sync)
{
    bool ok = true;
    // down: smooth, restrict
    for (int l = a.top; l >= 1 && ok; --l) {
        const VsubLevel<T>& L = lev[l];
        for (int q = 0; q < a.npre && ok; ++q) {
            vsub_rb(L, 0, q == 0 && (l < a.top || a.zero_top), rank, nblk);
            ok = sync();
            if (!ok) break;
            vsub_rb(L, 1, false, rank, nblk);
            ok = sync();
        }
        if (!ok) break;
        const VsubLevel<T>& C = lev[l - 1];
        const int mc = C.v.n - 1;
        const long long W = (long long)mc * mc * mc;
        const T ih2 = T(1) / (L.h * L.h);
        for (long long w = rank * (long long)blockDim.x + threadIdx.x; w < W; w += (long long)nblk * blockDim.x) {
            const int I = (int)(w % mc) + 1, J = (int)((w / mc) % mc) + 1, K = (int)(w / ((long long)mc * mc)) + 1;
            restrict_node<T>(L.e, L.f, L.v, C.f, C.v, ih2, I, J, K);
        }
        ok = sync();
    }
    if (!ok) return;
    // the coarse-grid level: one V-cycle from zero in CTA 0's shared memory
    if (rank == 0) {
        const VsubLevel<T>& C = lev[0];
        switch (C.v.n) {
        case 2: coarse_run<T, 0>(smem_raw, 0, C.e, C.f, C.v, C.h, nullptr, 0, 0, a.npre, a.npost); break;
        case 4: coarse_run<T, 1>(smem_raw, 0, C.e, C.f, C.v, C.h, nullptr, 0, 0, a.npre, a.npost); break;
        case 8: coarse_run<T, 2>(smem_raw, 0, C.e, C.f, C.v, C.h, nullptr, 0, 0, a.npre, a.npost); break;
        default: coarse_run<T, 3>(smem_raw, 0, C.e, C.f, C.v, C.h, nullptr, 0, 0, a.npre, a.npost); break;
        }
    }
    ok = sync();
    // up: correct, smooth
    for (int l = 1; l <= a.top && ok; ++l) {
        const VsubLevel<T>& L = lev[l];
        const VsubLevel<T>& C = lev[l - 1];
        const int half = L.v.n >> 1, rows = L.v.n - 1;
        const long long W = (long long)half * rows * rows;
        for (long long w = rank * (long long)blockDim.x + threadIdx.x; w < W; w += (long long)nblk * blockDim.x) {
            const int m = (int)(w % half);
            const long long r = w / half;
            prolong_node<T, true>(C.e, C.v, L.e, L.v, m, (int)(r % rows) + 1, (int)(r / rows) + 1);
        }
        ok = sync();
        for (int q = 0; q < a.npost && ok; ++q) {
            vsub_rb(L, 0, false, rank, nblk);
            ok = sync();
            if (!ok) break;
            vsub_rb(L, 1, false, rank, nblk);
            if (l < a.top || q + 1 < a.npost) ok = sync();
        }
    }
}

template <typename T>
__global__ void __launch_bounds__(kVsubThreads) vsub_kernel(VsubArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned gen = 0;
    vsub_body(a, a.lev, (int)blockIdx.x, (int)gridDim.x, smem_raw,
              [&]() { return grid_barrier(a.bar, gen, a.fault, a.polls); });
}

// The same V-cycle as one thread-block cluster per set (csize CTAs; cluster
// s takes set s).  The phases meet at the cluster's hardware barrier with
// release / acquire semantics, so every global write of a phase is visible to
// the whole cluster in the next.  The hardware schedules a cluster's CTAs
// together and every CTA of it passes the same barriers (a set whose
// correction has stopped returns in all of them before the first), so no
// wait is left open.  No grid-wide synchronisation: concurrent solves and
// the sets of a context run side by side.
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename T>
__global__ void __launch_bounds__(kVsubThreads) vcluster_kernel(VsubArgs<T> a, int csize)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int set = (int)blockIdx.x / csize, rank = (int)blockIdx.x - set * csize;
    if (a.act && !a.act[set].cont) return;
    VsubLevel<T> lev[kVsubMaxLevels];
#pragma unroll
    for (int l = 0; l < kVsubMaxLevels; ++l) {
        lev[l] = a.lev[l];
        if (l <= a.top) {
            lev[l].e += (long long)set * 2 * lev[l].v.cs;
            lev[l].f += (long long)set * 2 * lev[l].v.cs;
        }
    }
    vsub_body(a, lev, rank, csize, smem_raw, []() {
        cluster_sync_all();
        return true;
    });
}

// ---------------------------------------------------------------------------
// The V-cycle from the 32-interval level down on one thread-block cluster of C
// CTAs per set.  CTA r owns the planes k0 .. k1-1 of that level; two threads
// hold a row (j, k), 16 nodes each, and its right-hand side in registers for the
// whole V-cycle, as Row does on the levels under it: odd i in O, even i in E,
// the neighbour across the middle of the row by a shuffle, rows with j + k even
// (s = 0) in the first half of the threads and the others in the second.
// Neighbouring rows come from an exchange array in shared memory, which holds the
// slab's planes and one more on each side; a thread whose plane borders another
// CTA's slab also stores its new values into that CTA's copy (distributed shared
// memory), so that every read is local.  Phases, separated by the cluster's
// hardware barrier (release / acquire):
//   npre (red, black) half-sweeps;
//   the red residuals, the first plane's also into the CTA below; then their full
//   weighting, written straight into CTA 0's arrays of the 16-interval level;
//   one V-cycle of the levels 16 .. 2 in CTA 0 (sm_vcycle, as coarse_run);
//   the trilinear correction of the black nodes, from a copy of CTA 0's planes;
//   npost (red, black) half-sweeps;
// then the rows go back to global memory.  The arithmetic of every node is that
// of the per-step kernels (rb_half4_kernel, restrict_node, coarse_run,
// prolong_node) in the same order, with the same constants, so the result is the
// same bits.  Bound by latencies: each phase is a few shared-memory reads, a
// short chain of sums and the cluster's barrier.  Measured with C = 8:
// 19.5 us a launch, 24.3 with a node at a time read from shared memory (and from
// the neighbouring CTA's).
constexpr int kSlabN = 32;
constexpr int kSlabP = kSlabN + 1;
constexpr int kSlabM = ((kSlabN / 2 + 1) + 3) & ~3;  // row length of the colour-split layout (make_view)
constexpr int kSlabCoarseP = kSlabN / 2 + 1;         // 17: natural layout of CTA 0's 16-interval arrays
constexpr int kSlabRow = kSlabP + 1;                 // rows of a plane in the exchange (one of padding)
constexpr int kSlabRes = 20;                         // floats of a row of red residuals (16 and padding)

__host__ __device__ inline int slab_depth(int csize) { return (kSlabN - 1 + csize - 1) / csize; }  // 8, 4, 2: even
// threads of the rows of one s (31 rows in two planes, two threads a row), and of the block (CTA 0 runs Row<16>)
__host__ __device__ inline int slab_half(int csize) { return (slab_depth(csize) * (kSlabN - 1) + 31) / 32 * 32; }
__host__ __device__ inline int slab_threads(int csize)
{
    const int t = 2 * slab_half(csize), c = 2 * Row<float, 16>::HALF;
    return t > c ? t : c;
}
// vectors of four nodes of one half of the rows in the exchange: [vector][parity of i][plane][row]; the other half
// lies four vectors past a multiple of 128 bytes from it, so that the two threads of a row meet different banks
__host__ __device__ inline int slab_half_vecs(int csize) { return 4 * (slab_depth(csize) + 2) * kSlabRow + 4; }

struct SlabArgs {
    float* e;  // the 32-interval level (set 0; set s at + 2 s cs)
    const float* f;
    long long cs;
    float h2, sixth, ih2;  // that level's h^2, 1/6 and 1/h^2 as the per-step kernels take them
    float hc;              // h of the 16-interval level
    int zero_top, npre, npost, csize;
    const SolveState* act;
};

template <class T>
__device__ __forceinline__ T* cluster_map(T* p, int rank)
{
    unsigned long long out;
    asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<T*>(out);
}

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// ---------------------------------------------------------------------------
// The coarse solver from the 16-interval level in FP64, on one cluster of eight
// CTAs per set: coarse_run<double, 3>, a V-cycle from zero or the full multigrid
// with its ncycle V-cycles.  On one multiprocessor a V-cycle is bound by the two
// FP64 lanes a clock: the 3375 nodes take eight operations in each of four sweeps
// and twelve in the residual, 71 of 90 us.  (A 129^3 solve with six V-cycles a level,
// 18 V-cycles and the full multigrid here: 1704 -> 834 us, launches included; the
// levels 2 .. 8, in CTA 0, are half of the rest.)  CTA r owns the planes 2r + 1 and 2r + 2, a
// thread one node of each colour; a node's new value also goes to the CTA whose
// slab its plane borders (distributed shared memory), so that every read is
// local.  The arithmetic is that of sm_relax, sm_residual, sm_restrict,
// sm_prolong and sm_correct.
constexpr int kDeep = 8;             // CTAs: two of the 15 interior planes each
constexpr int kDeepThreads = 256;    // 2 planes x 15 rows x 8 nodes of a colour
constexpr int kDeepPlane = 17 * 17;

size_t deep_smem_bytes()
{
    int elems = 7 * kDeepPlane + 1;  // u: four planes, residuals: three; kept even
    for (int l = 0; l < 3; ++l) elems += coarse_elems<double>(2 << l);
    return sizeof(double) * elems;
}

__global__ void __cluster_dims__(kDeep, 1, 1) __launch_bounds__(kDeepThreads)
coarse_deep_kernel(int fmg, double* __restrict__ e, const double* __restrict__ f, LevelView v, double h,
                   const double* __restrict__ u64, int nfine, int ncycle, int npre, int npost,
                   const SolveState* __restrict__ act)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int P = 17, PP = kDeepPlane;
    const int set = (int)blockIdx.x / kDeep, rank = (int)cluster_rank(), t = (int)threadIdx.x;
    if (act && !act[set].cont) return;  // the whole cluster reads the same flag
    e += (long long)set * 2 * v.cs;
    f += (long long)set * 2 * v.cs;
    if (u64) u64 += set * nat_elems(nfine);
    double* const u = reinterpret_cast<double*>(smem_raw);  // slot p: plane k0 - 1 + p
    double* const res = u + 4 * PP;                         // planes k0, k0 + 1, k0 + 2
    CoarseSmem<double> S;
    coarse_layout(S, res + 3 * PP + 1, 2);
    const int k0 = 2 * rank + 1;
    const double h2 = h * h, ih2 = 1.0 / (h * h);

    // this thread's node of each colour (sm_relax's slots), at o in u
    const int kk = t / 120, j = t % 120 / 8 + 1, m = t % 8, k = k0 + kk;
    const bool row_on = kk < 2 && k < 16;
    int o[2];
    bool on[2];
    double fv[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int i = 1 + (((1 + j + k) & 1) != c ? 1 : 0) + 2 * m;
        on[c] = row_on && i < 16;
        o[c] = on[c] ? i + P * j + PP * (kk + 1) : P + 1 + PP;
        fv[c] = on[c] ? f[node_off(v, i, j, k)] : 0.0;
    }
    // plane k0 is slot 3 of the CTA below, plane k0 + 1 slot 0 of the one above
    double* push = nullptr;
    if (row_on && kk == 0 && rank > 0) push = cluster_map(u, rank - 1) + 2 * PP;
    if (row_on && kk == 1 && rank < kDeep - 1) push = cluster_map(u, rank + 1) - 2 * PP;
    double* const below = row_on && kk == 0 && rank > 0 ? cluster_map(res, rank - 1) + 2 * PP : nullptr;

    // zeros, or the boundary values injected from the finest grid
    for (int p = t; p < 4 * PP; p += kDeepThreads) {
        const int i = p % P, jj = p / P % P, kp = k0 - 1 + p / PP;
        const bool inner = i > 0 && i < 16 && jj > 0 && jj < 16 && kp > 0 && kp < 16;
        double val = 0.0;
        if (fmg && u64 && !inner && kp <= 16) {
            const long long st = nfine / 16, PF = nfine + 1;
            val = u64[i * st + PF * (jj * st + PF * (kp * st))];
        }
        u[p] = val;
    }
    for (int p = t; p < 3 * PP; p += kDeepThreads) res[p] = 0.0;
    if (rank == 0)
        for (int p = t; p < cube(8); p += kDeepThreads) S.u[2][p] = S.f[2][p] = 0.0;
    cluster_sync_all();

    auto sum6 = [&](int at) {
        return (u[at + 1] + u[at - 1]) + (u[at + P] + u[at - P]) + (u[at + PP] + u[at - PP]);
    };
    auto set_node = [&](int c, double x, bool remote) {
        u[o[c]] = x;
        if (push && remote) push[o[c]] = x;
    };
    auto relax = [&](int c, bool zero, bool remote) {
        if (on[c]) set_node(c, fused(-h2, fv[c], zero ? 0.0 : sum6(o[c])) * (1.0 / 6.0), remote);
    };
    // res on this slab, the first plane's values also as the third plane of the CTA below
    auto set_res = [&](int c, double r) {
        res[o[c] - PP] = r;
        if (below) below[o[c] - PP] = r;
    };
    // the full weighting of res on the coarse plane rank + 1, whose fine plane is k0 + 1, into CTA 0
    auto restrict_res = [&]() {
        if (rank < kDeep - 1 && t < 49) {
            const int I = t % 7 + 1, J = t / 7 + 1;
            double acc = 0.0;
#pragma unroll
            for (int c = -1; c <= 1; ++c)
#pragma unroll
                for (int b = -1; b <= 1; ++b)
#pragma unroll
                    for (int a = -1; a <= 1; ++a) {
                        const double w = 0.125 * (a == 0 ? 2 : 1) * (b == 0 ? 2 : 1) * (c == 0 ? 2 : 1) * 0.125;
                        acc += w * res[(2 * I + a) + P * (2 * J + b) + PP * (1 + c)];
                    }
            cluster_map(S.f[2], 0)[I + 9 * (J + 9 * (rank + 1))] = acc;
        }
    };
    // the coarse planes rank and rank + 1, copied once from CTA 0; their interpolation
    auto fetch_coarse = [&]() {
        if (rank != 0) {
            if (t < 162) S.u[2][81 * rank + t] = cluster_map(S.u[2], 0)[81 * rank + t];
            __syncthreads();
        }
    };
    auto interpolated = [&](int c) {
        const int i = o[c] % P;
        const int I0 = i >> 1, I1 = (i + 1) >> 1, J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1;
        const double* const w = S.u[2];
        double sum = (w[I0 + 9 * (J0 + 9 * K0)] + w[I1 + 9 * (J0 + 9 * K0)])
                   + (w[I0 + 9 * (J1 + 9 * K0)] + w[I1 + 9 * (J1 + 9 * K0)]);
        sum += (w[I0 + 9 * (J0 + 9 * K1)] + w[I1 + 9 * (J0 + 9 * K1)])
             + (w[I0 + 9 * (J1 + 9 * K1)] + w[I1 + 9 * (J1 + 9 * K1)]);
        return sum * 0.125;
    };

    if (fmg) {  // the levels 2 .. 8 in CTA 0, then the first values of this one
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (on[c]) set_res(c, fv[c]);
        cluster_sync_all();
        restrict_res();
        cluster_sync_all();
        if (rank == 0) {
            sm_restrict_down<double, 2>(S);
            sm_inject<double, 2>(S, u64, nfine);
            __syncthreads();
            sm_fmg_up<double, 2>(S, h * 8.0, ncycle, npre, npost);
        }
        cluster_sync_all();
        fetch_coarse();
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (on[c]) set_node(c, interpolated(c), true);
        cluster_sync_all();
    } else {
        ncycle = 1;
    }
    for (int cycle = 0; cycle < ncycle; ++cycle) {
        for (int q = 0; q < npre; ++q) {
            relax(0, !fmg && q == 0, true);
            cluster_sync_all();
            relax(1, false, true);
            cluster_sync_all();
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (on[c]) set_res(c, fv[c] - (sum6(o[c]) - 6.0 * u[o[c]]) * ih2);
        cluster_sync_all();
        restrict_res();
        cluster_sync_all();
        if (rank == 0) {
            sm_fill<double, 8>(S.u[2], 0.0);
            sm_vcycle<double, 2, true>(S, h * 2.0, npre, npost);
        }
        cluster_sync_all();
        fetch_coarse();
        if (on[1]) set_node(1, u[o[1]] + interpolated(1), true);
        cluster_sync_all();
        // no CTA touches another's shared memory after its last barrier
        for (int q = 0; q < npost; ++q) {
            relax(0, false, true);
            cluster_sync_all();
            const bool last = cycle == ncycle - 1 && q == npost - 1;
            relax(1, false, !last);
            if (!last) cluster_sync_all();
        }
    }
    __syncthreads();
    // the slab with its boundary nodes, and the planes 0 and 16
    for (int p = t + (rank == 0 ? 0 : PP); p < 3 * PP; p += kDeepThreads) {
        const int i = p % P, jj = p / P % P, kp = k0 - 1 + p / PP;
        e[node_off(v, i, jj, kp)] = u[p];
    }
}

using Vec4 = RowVec<float>;

// Half a row of the 32-interval level: nodes i = 16 half + 1 .. 16 half + 16.
struct SlabRow {
    int s, j, k, half;
    bool on;
    float O[8], E[8], eL;  // odd i; even i (the last one of the second half is the boundary node 32); i = 0
    float fO[8], fE[8];
    Vec4* x;               // the row's first vector in the exchange, and its neighbours' (other rows of the same half)
    int stride;            // vectors between [vector][parity] parts
    int yp, ym, zp, zm;
    Vec4* push;            // the row in the exchange of the CTA that its plane borders, or null

    template <bool EVEN>
    __device__ __forceinline__ void put(bool remote)
    {
        const float* a = EVEN ? E : O;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            Vec4 w;
#pragma unroll
            for (int e = 0; e < 4; ++e) w.v[e] = a[4 * v + e];
            x[(v * 2 + EVEN) * stride] = w;
            if (remote && push) push[(v * 2 + EVEN) * stride] = w;
        }
    }
    // sums of the six neighbours of the nodes of one parity of i (the whole warp takes part)
    template <bool EVEN>
    __device__ __forceinline__ void sums(float (&sum)[8]) const
    {
        const float across = EVEN ? __shfl_down_sync(0xffffffffu, O[0], 1) : __shfl_up_sync(0xffffffffu, E[7], 1);
        const float left0 = half ? across : eL;  // of O[0]
        if (!on) return;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const Vec4* p = x + (v * 2 + EVEN) * stride;
            const Vec4 a = p[ym], b = p[yp], c = p[zm], d = p[zp];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int q = 4 * v + e;
                const float lo = EVEN ? O[q] : (q == 0 ? left0 : E[q == 0 ? 0 : q - 1]);
                const float hi = EVEN ? (q == 7 ? across : O[q == 7 ? 0 : q + 1]) : E[q];
                sum[q] = (lo + hi) + (a.v[e] + b.v[e]) + (c.v[e] + d.v[e]);
            }
        }
    }
    template <bool EVEN, bool ZERO>
    __device__ __forceinline__ void relax_own(float h2, float sixth, bool remote)
    {
        float sum[8];
        if (ZERO) {
#pragma unroll
            for (int q = 0; q < 8; ++q) sum[q] = 0.0f;
        } else {
            sums<EVEN>(sum);
        }
        if (!on) return;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float w = fused(-h2, EVEN ? fE[q] : fO[q], sum[q]) * sixth;
            if (!EVEN) O[q] = w;
            else if (q < 7 || half == 0) E[q] = w;  // not the boundary node
        }
        put<EVEN>(remote);
    }
    template <bool ZERO>
    __device__ __forceinline__ void relax(int colour, float h2, float sixth, bool remote)
    {
        if ((s ^ colour) == 0) relax_own<true, ZERO>(h2, sixth, remote);
        else relax_own<false, ZERO>(h2, sixth, remote);
    }
    // red residuals of the half row (s = 0: even i, s = 1: odd i)
    template <bool EVEN>
    __device__ __forceinline__ void residual(float ih2, float* to, float* remote) const
    {
        float sum[8];
        sums<EVEN>(sum);
        if (!on) return;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            Vec4 w;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int q = 4 * v + e;
                w.v[e] = fused(-fused(-6.0f, EVEN ? E[q] : O[q], sum[q]), ih2, EVEN ? fE[q] : fO[q]);
            }
            reinterpret_cast<Vec4*>(to)[v] = w;
            if (remote) reinterpret_cast<Vec4*>(remote)[v] = w;
        }
    }
    // the correction of the black nodes (prolong_node's sums) from the natural coarse array c
    __device__ __forceinline__ void correct(const float* c)
    {
        if (!on) return;
        constexpr int PC = kSlabCoarseP;
        const int J0 = j >> 1, J1 = (j + 1) >> 1, K0 = k >> 1, K1 = (k + 1) >> 1, I = 8 * half;
        const float* c00 = c + I + PC * (J0 + PC * K0);
        const float* c10 = c + I + PC * (J1 + PC * K0);
        const float* c01 = c + I + PC * (J0 + PC * K1);
        const float* c11 = c + I + PC * (J1 + PC * K1);
        if (s == 0) {  // odd i, between I + q and I + q + 1
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float t = (c00[q] + c00[q + 1]) + (c10[q] + c10[q + 1]);
                t += (c01[q] + c01[q + 1]) + (c11[q] + c11[q + 1]);
                t *= 0.125f;
                O[q] = O[q] + t;
            }
            put<false>(true);
        } else {  // even i, on I + q + 1
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (q == 7 && half) break;
                float t = (c00[q + 1] + c00[q + 1]) + (c10[q + 1] + c10[q + 1]);
                t += (c01[q + 1] + c01[q + 1]) + (c11[q + 1] + c11[q + 1]);
                t *= 0.125f;
                E[q] = E[q] + t;
            }
            put<true>(true);
        }
    }
};

// THREADS: 512 (clusters of 4) or 256
template <int THREADS>
__global__ void __launch_bounds__(THREADS) vslab_kernel(SlabArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int C = a.csize;
    const int set = (int)blockIdx.x / C;
    const int rank = (int)cluster_rank();
    if (a.act && !a.act[set].cont) return;  // the whole cluster reads the same flag
    const int q = slab_depth(C), slots = q + 2;  // slot p of the exchange holds plane k0 - 1 + p
    const int k0 = 1 + rank * q, k1 = min(kSlabN, k0 + q);
    const int t = (int)threadIdx.x, T = (int)blockDim.x;
    Vec4* const ex = reinterpret_cast<Vec4*>(smem_raw);
    const int half_vecs = slab_half_vecs(C);
    float* const rr = reinterpret_cast<float*>(ex + 2 * half_vecs);  // red residuals of planes k0 .. k1
    CoarseSmem<float> S;
    coarse_layout(S, rr + (q + 1) * kSlabP * kSlabRes, 3);
    float* const e = a.e + (long long)set * 2 * a.cs;
    const float* const f = a.f + (long long)set * 2 * a.cs;
    constexpr int kC3 = kSlabCoarseP * kSlabCoarseP * kSlabCoarseP;

    // where a row lies in the exchange, from the first vector of its half: even j first, then odd j, so that the rows
    // of a warp (every other j) lie next to each other
    auto place = [&](int k, int j) { return (k - (k0 - 1)) * kSlabRow + (j >> 1) + (j & 1) * (kSlabN / 2 + 1); };
    const int stride = slots * kSlabRow;

    SlabRow row;
    {
        const int halft = slab_half(C);
        row.s = t >= halft ? 1 : 0;
        const int g = t - row.s * halft, r = g >> 1;
        row.half = g & 1;
        // planes in pairs (k0 is odd): for s = 0 the first has the 16 odd j and the second the 15 even ones; for s = 1
        // the reverse
        const int pr = r / (kSlabN - 1), m = r - pr * (kSlabN - 1), first = row.s ? kSlabN / 2 - 1 : kSlabN / 2;
        row.k = k0 + 2 * pr + (m >= first ? 1 : 0);
        row.j = m < first ? 2 * m + (row.s ? 2 : 1) : 2 * (m - first) + (row.s ? 1 : 2);
        row.on = t < 2 * halft && row.k < k1;
        if (!row.on) row.k = k0, row.j = 1;  // any row: nothing of it is used
        Vec4* const base = ex + row.half * half_vecs;
        row.x = base + place(row.k, row.j);
        row.stride = stride;
        row.yp = place(row.k, row.j + 1) - place(row.k, row.j);
        row.ym = place(row.k, row.j - 1) - place(row.k, row.j);
        row.zp = kSlabRow;
        row.zm = -kSlabRow;
        // the plane's place in the neighbouring CTA: slot q + 1 of the one below, slot 0 of the one above
        row.push = nullptr;
        const int in_plane = place(k0 - 1, row.j);
        if (row.on && row.k == k0 && rank > 0) row.push = cluster_map(base + (q + 1) * kSlabRow + in_plane, rank - 1);
        else if (row.on && row.k == k1 - 1 && rank < C - 1) row.push = cluster_map(base + in_plane, rank + 1);
        // with one plane a slab (the last of 16) both sides would border: it is the last, and has none above
    }
    // the row from global memory: even i = 2m at m of one colour, odd i = 2m + 1 of the other
    const long long at = ((long long)row.k * kSlabP + row.j) * kSlabM + 8 * row.half;
    const long long ev = (row.s ? a.cs : 0) + at, od = (row.s ? 0 : a.cs) + at;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        row.fO[v] = f[od + v];
        row.fE[v] = f[ev + v + 1];
        row.O[v] = a.zero_top ? 0.0f : e[od + v];
        row.E[v] = a.zero_top ? 0.0f : e[ev + v + 1];
    }
    row.eL = a.zero_top ? 0.0f : e[ev];
    // the exchange: zeros, or the planes k0 - 1 .. k1 with their boundary rows
    if (a.zero_top) {
        const Vec4 z = {{0.0f, 0.0f, 0.0f, 0.0f}};
        for (int p = t; p < 2 * half_vecs; p += T) ex[p] = z;
    } else {
        for (int p = t; p < (k1 - k0 + 2) * kSlabP * 2; p += T) {
            const int half = p & 1, jr = (p >> 1) % kSlabP, kr = k0 - 1 + (p >> 1) / kSlabP, sr = (jr + kr) & 1;
            const long long src = ((long long)kr * kSlabP + jr) * kSlabM + 8 * half;
            const float* od_r = e + (sr ? 0 : a.cs) + src;
            const float* ev_r = e + (sr ? a.cs : 0) + src;
            Vec4* to = ex + half * half_vecs + place(kr, jr);
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                Vec4 o, w;
#pragma unroll
                for (int c = 0; c < 4; ++c) o.v[c] = od_r[4 * v + c], w.v[c] = ev_r[4 * v + c + 1];
                to[(v * 2) * stride] = o;
                to[(v * 2 + 1) * stride] = w;
            }
        }
    }
    if (rank == 0) {  // as coarse_run with a zero start: zeros off the interior
        for (int p = t; p < kC3; p += T) S.u[3][p] = 0.0f;
        clear_rows<float, 3>(S);
    }
    cluster_sync_all();

    // pre-smoothing
    for (int v = 0; v < a.npre; ++v) {
        if (v == 0 && a.zero_top) row.relax<true>(0, a.h2, a.sixth, true);
        else row.relax<false>(0, a.h2, a.sixth, true);
        cluster_sync_all();
        row.relax<false>(1, a.h2, a.sixth, true);
        cluster_sync_all();
    }
    // the red residuals; plane k0's are needed by the CTA below too, as its plane k1
    {
        float* to = rr + ((row.k - k0) * kSlabP + row.j) * kSlabRes + 8 * row.half;
        float* remote = row.on && row.k == k0 && rank > 0
                            ? cluster_map(rr + (q * kSlabP + row.j) * kSlabRes + 8 * row.half, rank - 1)
                            : nullptr;
        if (row.s == 0) row.residual<true>(a.ih2, to, remote);
        else row.residual<false>(a.ih2, to, remote);
    }
    cluster_sync_all();
    // their full weighting onto the coarse planes K with 2K in this slab (restrict_node's sums)
    {
        float* fc = rank == 0 ? S.f[3] : cluster_map(S.f[3], 0);
        const int K0 = (k0 + 1) >> 1, K1 = (k1 + 1) >> 1;  // 2K in [k0, k1)
        constexpr int MC = kSlabN / 2 - 1;
        for (int p = t; p < (K1 - K0) * MC * MC; p += T) {
            const int I = p % MC + 1, J = (p / MC) % MC + 1, K = K0 + p / (MC * MC);
            // rows j - 1, j, j + 1 of planes k - 1, k, k + 1 at node i = 2I: odd i = 2I -+ 1 at I - 1 and I, even at I - 1
            const float* r0 = rr + ((2 * K - k0) * kSlabP + 2 * J) * kSlabRes + I - 1;
            const float* rm = r0 - kSlabP * kSlabRes;
            const float* rp = r0 + kSlabP * kSlabRes;
            float edge = (r0[kSlabRes + 1] + r0[kSlabRes]) + (r0[-kSlabRes + 1] + r0[-kSlabRes]);
            edge += (rp[1] + rp[0]) + (rm[1] + rm[0]);
            edge += (rp[kSlabRes] + rp[-kSlabRes]) + (rm[kSlabRes] + rm[-kSlabRes]);
            const float centre = r0[0];
            fc[I + kSlabCoarseP * (J + kSlabCoarseP * K)] = 0.125f * centre + 0.03125f * edge;
        }
    }
    cluster_sync_all();
    if (rank == 0) sm_vcycle<float, 3, true>(S, a.hc, a.npre, a.npost);
    cluster_sync_all();
    // coarse-grid correction; the coarse planes k0/2 .. k1/2 that this slab interpolates from are first copied from
    // CTA 0 into the same place of this CTA's (otherwise unused) coarse arrays, so that CTA 0's shared memory is read
    // once per value
    if (rank != 0) {
        const float* src = cluster_map(S.u[3], 0);
        const int lo = (k0 >> 1) * kSlabCoarseP * kSlabCoarseP;
        const int hi = ((k1 >> 1) + 1) * kSlabCoarseP * kSlabCoarseP;
        for (int p = lo + t; p < hi; p += 4 * T) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (p + u * T < hi) v[u] = src[p + u * T];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (p + u * T < hi) S.u[3][p + u * T] = v[u];
        }
        __syncthreads();
    }
    row.correct(S.u[3]);
    cluster_sync_all();
    // post-smoothing; no CTA reads the last black values from the exchange, nor another CTA's after the last barrier
    for (int v = 0; v < a.npost; ++v) {
        row.relax<false>(0, a.h2, a.sixth, true);
        cluster_sync_all();
        const bool last = v == a.npost - 1;
        row.relax<false>(1, a.h2, a.sixth, !last);
        if (!last) cluster_sync_all();
    }
    if (row.on) {
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            e[od + v] = row.O[v];
            if (v < 7 || row.half == 0) e[ev + v + 1] = row.E[v];
        }
    }
}

// ---------------------------------------------------------------------------
// FP64 outer steps on the caller's natural-layout arrays (n intervals).
__device__ __forceinline__ long long nat(int n, int i, int j, int k)
{
    const long long P = n + 1;
    return (long long)i + P * ((long long)j + P * (long long)k);
}

// FP64 to the smoothing precision, on the integer pipe where it is FP32 (the
// conversion instruction runs on the FP64 pipe, at 2 a clock on each SM).
template <typename T> __device__ __forceinline__ T narrow(double x);
template <> __device__ __forceinline__ double narrow<double>(double x) { return x; }
template <> __device__ __forceinline__ float narrow<float>(double x) { return f64_to_f32_rn(x); }

constexpr int kConvertThreads = 256;

// f = coef rhs on interior nodes, a pair of consecutive nodes (2m, 2m+1) per
// thread of a flat grid: one red and one black entry with the same index m, so the stores of
// a warp are contiguous in each colour array.
template <typename T>
__global__ void convert_rhs_kernel(const double* __restrict__ rhs, double coef, int n, T* __restrict__ f, LevelView v)
{
    const int set = blockIdx.y;
    const unsigned half = (unsigned)n / 2, lh = 31u - (unsigned)__clz((int)half);  // a power of two
    const unsigned idx = blockIdx.x * (unsigned)kConvertThreads + threadIdx.x;     // (plane, row, pair), below 2^30
    const unsigned row2 = idx >> lh, plane = row2 / (unsigned)(n - 1);
    const int m = (int)(idx & (half - 1));
    const int j = (int)(row2 - plane * (unsigned)(n - 1)) + 1, k = (int)plane + 1;
    if (k >= n) return;
    const double* src = rhs + set * nat_elems(n) + nat(n, 2 * m, j, k);
    T* row = f + set * 2 * v.cs + ((long long)k * (v.n + 1) + j) * v.M + m;
    const int c = (2 * m + j + k) & 1;  // colour of node 2m; node 2m+1 has the other one
    double a = src[0], b = src[1];
    if (coef != 1.0) a *= coef, b *= coef;
    if (m > 0) row[(long long)c * v.cs] = narrow<T>(a);  // node 0 is a boundary node
    row[(long long)(c ^ 1) * v.cs] = narrow<T>(b);
}

template <typename T, bool ADD>
__global__ void assign_outer_kernel(double* __restrict__ u, int n, const T* __restrict__ e, LevelView v,
                                    const SolveState* __restrict__ act)
{
    int kz;
    const int set = set_of(n - 1, kz);
    if (act && !act[set].cont) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
    const int j = blockIdx.y + 1, k = kz + 1;
    if (i >= n) return;
    const long long o = set * nat_elems(n) + nat(n, i, j, k);
    const double d = (double)e[set * 2 * v.cs + node_off(v, i, j, k)];
    u[o] = ADD ? u[o] + d : d;
}

constexpr int kOuterThreads = 128;

// r = coef*rhs - L u in FP64 on interior nodes, stored in precision T; each
// block writes its partial sums of r^2 and (coef*rhs)^2 (fixed-order
// reductions, so the norms are reproducible run to run).
template <typename T>
__global__ void __launch_bounds__(kOuterThreads)
residual_outer_kernel(const double* __restrict__ u, const double* __restrict__ rhs, double coef, int n, double ih2,
                      T* __restrict__ r, LevelView v, double* __restrict__ partials)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x + 1;
    const int j = blockIdx.y + 1, k = blockIdx.z + 1;
    double rr = 0.0, ff = 0.0;
    if (i < n) {
        const long long P = n + 1, Q = P * P;
        const long long o = nat(n, i, j, k);
        const double s = (u[o + 1] + u[o - 1]) + (u[o + P] + u[o - P]) + (u[o + Q] + u[o - Q]);
        const double fv = coef * rhs[o];
        const double res = fv - (s - 6.0 * u[o]) * ih2;
        r[node_off(v, i, j, k)] = (T)res;
        rr = res * res;
        ff = fv * fv;
    }
    for (int off = 16; off > 0; off >>= 1) {
        rr += __shfl_down_sync(0xffffffffu, rr, off);
        ff += __shfl_down_sync(0xffffffffu, ff, off);
    }
    __shared__ double sr[kOuterThreads / 32], sf[kOuterThreads / 32];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        sr[w] = rr;
        sf[w] = ff;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int q = 0; q < kOuterThreads / 32; ++q) {
            a += sr[q];
            b += sf[q];
        }
        const long long bid = blockIdx.x + (long long)gridDim.x * (blockIdx.y + (long long)gridDim.y * blockIdx.z);
        partials[2 * bid] = a;
        partials[2 * bid + 1] = b;
    }
}

// The same residual, with rows of the grid dealt to a fixed number of blocks
// (so only a few thousand partial sums need reducing).
constexpr int kResidBlocksPerSM = 16;
constexpr int kResidMaxBlocks = 152 * kResidBlocksPerSM;
constexpr int kRowThreads = 128;

// WANT_F: the norm of coef*rhs too (the first residual of a solve; otherwise
// its partial sums are zero).  The FP64 pipe bounds it, so what is not a sum of
// the result is left out or done on the integer pipe.
template <typename T, bool WANT_F>
__global__ void __launch_bounds__(kRowThreads)
residual_rows_kernel(const double* __restrict__ u, const double* __restrict__ rhs, double coef, int n, double ih2,
                     T* __restrict__ r, LevelView v, double* __restrict__ partials, long long pstride,
                     const SolveState* __restrict__ act)
{
    const int set = blockIdx.y;  // one row of blocks per set
    if (act && !act[set].cont) return;
    u += set * nat_elems(n);
    rhs += set * nat_elems(n);
    r += set * 2 * v.cs;
    partials += set * pstride;
    const long long P = n + 1, Q = P * P;
    const int rows = (n - 1) * (n - 1);
    double rr = 0.0, ff = 0.0;
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const int j = row % (n - 1) + 1, k = row / (n - 1) + 1;
        for (int i = threadIdx.x + 1; i < n; i += kRowThreads) {
            const long long o = nat(n, i, j, k);
            const double s = (u[o + 1] + u[o - 1]) + (u[o + P] + u[o - P]) + (u[o + Q] + u[o - Q]);
            double fv = rhs[o];
            if (coef != 1.0) fv *= coef;
            const double res = fv - (s - 6.0 * u[o]) * ih2;
            r[node_off(v, i, j, k)] = narrow<T>(res);
            rr = fma(res, res, rr);
            if (WANT_F) ff = fma(fv, fv, ff);
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        rr += __shfl_down_sync(0xffffffffu, rr, off);
        ff += __shfl_down_sync(0xffffffffu, ff, off);
    }
    __shared__ double sr[kRowThreads / 32], sf[kRowThreads / 32];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        sr[w] = rr;
        sf[w] = ff;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int q = 0; q < kRowThreads / 32; ++q) {
            a += sr[q];
            b += sf[q];
        }
        partials[2 * blockIdx.x] = a;
        partials[2 * blockIdx.x + 1] = b;
    }
}

constexpr int kReduceThreads = 1024;

__global__ void __launch_bounds__(kReduceThreads) reduce_norms_kernel(const double* __restrict__ partials, int nblocks,
                                                                      double* __restrict__ out)
{
    double a = 0.0, b = 0.0;
    for (int t = threadIdx.x; t < nblocks; t += kReduceThreads) {
        a += partials[2 * t];
        b += partials[2 * t + 1];
    }
    __shared__ double sa[kReduceThreads], sb[kReduceThreads];
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int s = kReduceThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sa[threadIdx.x] += sa[threadIdx.x + s];
            sb[threadIdx.x] += sb[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sa[0];
        out[1] = sb[0];
    }
}

// Sums the partial norms in a fixed order and decides whether the defect
// correction goes on: continue = refine && rel > tol && it < max_it && rel
// finite.  first: this is the residual after FMG (sets the denominator
// ||coef*rhs||, or 1 when it is 0, and it = 0).  Inside a graph the decision
// drives the WHILE node through `handle`.
//
// Several sets (fault == NULL): block s decides for set s; a set whose
// correction has already stopped keeps its state; decide_any_kernel then
// takes over the fault flag and drives the WHILE node.
template <bool GRAPH>
__global__ void __launch_bounds__(kReduceThreads)
decide_kernel(const double* __restrict__ partials, int nblocks, SolveState* __restrict__ st, double tol, int max_it,
              int first, int refine, cudaGraphConditionalHandle handle, int* __restrict__ fault, long long pstride)
{
    const int set = blockIdx.x;
    partials += set * pstride;
    st += set;
    if (!fault && !first && st->cont == 0) return;
    double a = 0.0, b = 0.0;
    for (int t = threadIdx.x; t < nblocks; t += kReduceThreads) {
        a += partials[2 * t];
        b += partials[2 * t + 1];
    }
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
    }
    __shared__ double sa[kReduceThreads / 32], sb[kReduceThreads / 32];
    if ((threadIdx.x & 31) == 0) {
        sa[threadIdx.x >> 5] = a;
        sb[threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        a = sa[threadIdx.x];
        b = sb[threadIdx.x];
        for (int off = 16; off > 0; off >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, off);
            b += __shfl_down_sync(0xffffffffu, b, off);
        }
        if (threadIdx.x == 0) {
            sa[0] = a;
            sb[0] = b;
        }
    }
    if (threadIdx.x == 0) {
        if (first) {
            st->denom = sb[0] > 0.0 ? sqrt(sb[0]) : 1.0;
            st->it = 0;
        } else {
            st->it += 1;
        }
        const double rel = sqrt(sa[0]) / st->denom;
        if (first) st->rel0 = rel;
        st->rel = rel;
        const bool finite = isfinite(rel) && !st->nonfinite;
        const int faulted = (fault && *fault) ? 1 : 0;
        if (first) st->fault = 0;
        if (faulted) {
            st->fault = 1;
            *fault = 0;
        }
        st->converged = (finite && !st->fault && (!refine || rel <= tol)) ? 1 : 0;
        const int cont = (refine && finite && !st->fault && rel > tol && st->it < max_it) ? 1 : 0;
        st->cont = cont;
        if (GRAPH && fault) cudaGraphSetConditional(handle, (unsigned)cont);
    }
}

// After the per-set decisions: a fault recorded since the last check stops
// every set; the loop goes on while any set goes on.
template <bool GRAPH>
__global__ void decide_any_kernel(SolveState* __restrict__ st, int nsets, int first, cudaGraphConditionalHandle handle,
                                  int* __restrict__ fault)
{
    if (threadIdx.x != 0) return;
    const int faulted = *fault;
    if (faulted) *fault = 0;
    unsigned any = 0;
    for (int q = 0; q < nsets; ++q) {
        if (faulted) {
            st[q].fault = 1;
            st[q].converged = 0;
            st[q].cont = 0;
        }
        any |= (unsigned)st[q].cont;
    }
    if (GRAPH) cudaGraphSetConditional(handle, any);
}

inline dim3 half_grid(int n) { return dim3(cdiv(n / 2, kBX), cdiv(n - 1, kBY), (unsigned)(n - 1)); }
inline dim3 inner_grid(int n) { return dim3(cdiv(n - 1, kBX), cdiv(n - 1, kBY), (unsigned)(n - 1)); }
inline dim3 outer_grid(int n) { return dim3(cdiv(n - 1, kOuterThreads), (unsigned)(n - 1), (unsigned)(n - 1)); }

template <typename T>
size_t coarse_smem_bytes(int n)
{
    size_t tot = 0;
    for (int m = 2; m <= n; m *= 2) tot += (size_t)coarse_elems<T>(m);
    return tot * sizeof(T);
}

// shared memory of the slab V-cycle kernel: the exchange, the red residuals, and CTA 0's arrays of the levels 16 .. 2
inline size_t slab_smem_bytes(int csize)
{
    return sizeof(Vec4) * 2 * (size_t)slab_half_vecs(csize) +
           sizeof(float) * (size_t)((slab_depth(csize) + 1) * kSlabP * kSlabRes) + coarse_smem_bytes<float>(kSlabN / 2);
}

}  // namespace

// --- launchers ------------------------------------------------------------
// With several sets every grid's z extent (or, for the per-set kernels, its x
// or y extent) is multiplied by the number of sets; the qumond_create checks
// keep the products within the launch limits.
inline dim3 per_sets(dim3 g, const Sets& sets) { return dim3(g.x, g.y, g.z * (unsigned)sets.n); }

// threads along a row of the row-vector kernels on a level of n intervals
inline int vx_of(int n, const Sets& sets)
{
    if (n > kTileSmallN) return kVX;
    return sets.tile_small == 1 ? 4 : (sets.tile_small == 2 ? 2 : kVX);
}

template <typename T>
void launch_rb_half(T* e, const T* f, const LevelView& v, int colour, bool zero_guess, double h, cudaStream_t s,
                    const Sets& sets)
{
    T* own = e + (long long)colour * v.cs;
    const T* other = e + (long long)(colour ^ 1) * v.cs;
    const T* fc = f + (long long)colour * v.cs;
    const dim3 blk(kBX, kBY);
    if (sizeof(T) == sizeof(float) && v.n >= 8) {
        float* o4 = reinterpret_cast<float*>(own);
        const float* x4 = reinterpret_cast<const float*>(other);
        const float* f4 = reinterpret_cast<const float*>(fc);
        const int vx = vx_of(v.n, sets);
        const dim3 grid(cdiv(v.n / 2, 4 * vx), cdiv(v.n - 1, kVThreads / vx), (unsigned)(v.n - 1) * (unsigned)sets.n);
        const dim3 blk(vx, kVThreads / vx);
        const float h2 = (float)(h * h), sixth = 1.0f / 6.0f;
        switch ((zero_guess ? 8 : 0) + vx) {
        case 8 + 8: rb_half4_kernel<true, 8><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        case 8 + 4: rb_half4_kernel<true, 4><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        case 8 + 2: rb_half4_kernel<true, 2><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        case 8: rb_half4_kernel<false, 8><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        case 4: rb_half4_kernel<false, 4><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        default: rb_half4_kernel<false, 2><<<grid, blk, 0, s>>>(o4, x4, f4, v, colour, h2, sixth, sets.act); break;
        }
        return;
    }
    if (zero_guess)
        rb_half_kernel<T, true><<<per_sets(half_grid(v.n), sets), blk, 0, s>>>(own, other, fc, v, colour, (T)(h * h),
                                                                                T(1) / T(6), sets.act);
    else
        rb_half_kernel<T, false><<<per_sets(half_grid(v.n), sets), blk, 0, s>>>(own, other, fc, v, colour, (T)(h * h),
                                                                                 T(1) / T(6), sets.act);
}

void launch_rb_first(float* e, const float* f, const LevelView& v, double h, cudaStream_t s, const Sets& sets)
{
    const int vx = vx_of(v.n, sets);
    const dim3 grid(cdiv(v.n / 2, 4 * vx), cdiv(v.n - 1, kVThreads / vx), (unsigned)(v.n - 1) * (unsigned)sets.n);
    const dim3 blk(vx, kVThreads / vx);
    const float h2 = (float)(h * h), sixth = 1.0f / 6.0f;
    switch (vx) {
    case 8: rb_first4_kernel<8><<<grid, blk, 0, s>>>(e, f, v, h2, sixth, sets.act); break;
    case 4: rb_first4_kernel<4><<<grid, blk, 0, s>>>(e, f, v, h2, sixth, sets.act); break;
    default: rb_first4_kernel<2><<<grid, blk, 0, s>>>(e, f, v, h2, sixth, sets.act); break;
    }
}

template <typename T>
void launch_restrict_resid_red(const T* ef, const T* ff, const LevelView& vf, T* fc, const LevelView& vc, double hf,
                               cudaStream_t s, const Sets& sets)
{
    if (sizeof(T) == sizeof(float) && vf.n >= 128) {
        // planes per CTA: as many as keep about two CTAs per multiprocessor busy
        static int sms = 0;
        if (sms <= 0) {
            int dev = 0;
            cudaGetDevice(&dev);
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
        }
        const int tiles = (int)(cdiv(vc.n - 1, kRI) * cdiv(vc.n - 1, kRJ)) * sets.n;
        int rk = kRK;
        while (rk > 1 && tiles * (int)cdiv(vc.n - 1, rk) < 2 * sms) --rk;
        const int zper = (int)cdiv(vc.n - 1, rk);
        const dim3 grid(cdiv(vc.n - 1, kRI), cdiv(vc.n - 1, kRJ), (unsigned)(zper * sets.n));
        restrict_resid4_kernel<<<grid, kRI * kRJ, 0, s>>>(reinterpret_cast<const float*>(ef),
                                                           reinterpret_cast<const float*>(ff), vf,
                                                           reinterpret_cast<float*>(fc), vc, (float)(1.0 / (hf * hf)),
                                                           rk, zper, sets.act);
        return;
    }
    const T ih2 = (T)(1.0 / (hf * hf));
    if constexpr (sizeof(T) == sizeof(float)) {
        restrict_nodes_kernel<<<per_sets(inner_grid(vc.n), sets), dim3(kBX, kBY), 0, s>>>(ef, ff, vf, fc, vc, ih2, sets.act);
    } else {
        const int zper = (int)cdiv(vc.n - 1, kTK);
        const dim3 grid(cdiv(vc.n - 1, kTI), cdiv(vc.n - 1, kTJ), (unsigned)(zper * sets.n));
        restrict_tile_kernel<T><<<grid, kTI * kTJ * kTK, 0, s>>>(ef, ff, vf, fc, vc, ih2, zper, sets.act);
    }
}

template <typename T>
void launch_restrict_full(const T* ff, const LevelView& vf, T* fc, const LevelView& vc, cudaStream_t s,
                          const Sets& sets)
{
    restrict_full_kernel<T><<<per_sets(inner_grid(vc.n), sets), dim3(kBX, kBY), 0, s>>>(ff, vf, fc, vc);
}

template <typename T>
void launch_prolong_black(const T* ec, const LevelView& vc, T* ef, const LevelView& vf, bool add, cudaStream_t s,
                          const Sets& sets)
{
    if (sizeof(T) == sizeof(float) && vf.n >= 8) {
        const float* c4 = reinterpret_cast<const float*>(ec);
        float* f4 = reinterpret_cast<float*>(ef);
        const int vx = vx_of(vf.n, sets);
        const dim3 grid(cdiv(vf.n / 2, 4 * vx), cdiv(vf.n - 1, kVThreads / vx), (unsigned)(vf.n - 1) * (unsigned)sets.n);
        const dim3 blk(vx, kVThreads / vx);
        switch ((add ? 8 : 0) + vx) {
        case 8 + 8: prolong_black4_kernel<true, 8><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        case 8 + 4: prolong_black4_kernel<true, 4><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        case 8 + 2: prolong_black4_kernel<true, 2><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        case 8: prolong_black4_kernel<false, 8><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        case 4: prolong_black4_kernel<false, 4><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        default: prolong_black4_kernel<false, 2><<<grid, blk, 0, s>>>(c4, vc, f4, vf, sets.act); break;
        }
        return;
    }
    if (add)
        prolong_black_kernel<T, true><<<per_sets(half_grid(vf.n), sets), dim3(kBX, kBY), 0, s>>>(ec, vc, ef, vf,
                                                                                                  sets.act);
    else
        prolong_black_kernel<T, false><<<per_sets(half_grid(vf.n), sets), dim3(kBX, kBY), 0, s>>>(ec, vc, ef, vf,
                                                                                                   sets.act);
}

template <typename T>
void launch_set_boundary(T* e, const LevelView& v, const double* u64, int nfine, cudaStream_t s, const Sets& sets)
{
    set_boundary_kernel<T><<<dim3(cdiv(v.n + 1, 128), (unsigned)(v.n + 1), 6 * (unsigned)sets.n), 128, 0, s>>>(
        e, v, u64, nfine);
}

template <typename T>
cudaError_t launch_coarse(int fmg, T* e, const T* f, const LevelView& v, double h, const double* u64, int nfine,
                          int ncycle, int npre, int npost, cudaStream_t s, const Sets& sets)
{
    const size_t bytes = coarse_smem_bytes<T>(v.n);
    const unsigned g = (unsigned)sets.n;  // one CTA per set
    const SolveState* act = sets.act;
    switch (v.n) {
    case 2: coarse_kernel<T, 0><<<g, kCoarseThreads, bytes, s>>>(fmg, e, f, v, (T)h, u64, nfine, ncycle, npre, npost, act); break;
    case 4: coarse_kernel<T, 1><<<g, kCoarseThreads, bytes, s>>>(fmg, e, f, v, (T)h, u64, nfine, ncycle, npre, npost, act); break;
    case 8: coarse_kernel<T, 2><<<g, kCoarseThreads, bytes, s>>>(fmg, e, f, v, (T)h, u64, nfine, ncycle, npre, npost, act); break;
    case 16:
        if constexpr (sizeof(T) == sizeof(double)) {
            coarse_deep_kernel<<<kDeep * g, kDeepThreads, deep_smem_bytes(), s>>>(fmg, e, f, v, h, u64, nfine, ncycle, npre,
                                                                                  npost, act);
        } else {
            coarse_kernel<T, 3><<<g, kCoarseThreads, bytes, s>>>(fmg, e, f, v, (T)h, u64, nfine, ncycle, npre, npost, act);
        }
        break;
    default: return cudaErrorInvalidValue;  // the coarse solver covers the levels n = 2 .. 16
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_vsub(T* const* e, T* const* f, const LevelView* v, const double* h, int nlev, int zero_top, int npre,
                        int npost, unsigned* bar, int* fault, long long polls, int grid, cudaStream_t s)
{
    if (nlev < 2 || nlev > kVsubMaxLevels || v[0].n > kCoarseN) return cudaErrorInvalidValue;
    VsubArgs<T> a{};
    for (int l = 0; l < nlev; ++l) a.lev[l] = VsubLevel<T>{e[l], f[l], v[l], (T)h[l]};
    a.top = nlev - 1;
    a.zero_top = zero_top;
    a.npre = npre;
    a.npost = npost;
    a.bar = bar;
    a.fault = fault;
    a.polls = polls;
    cudaError_t err = cudaMemsetAsync(bar, 0, sizeof(unsigned), s);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kVsubThreads);
    cfg.dynamicSmemBytes = coarse_smem_bytes<T>(v[0].n);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, vsub_kernel<T>, a);
}

template <typename T>
cudaError_t launch_vcluster(T* const* e, T* const* f, const LevelView* v, const double* h, int nlev, int zero_top,
                            int npre, int npost, int csize, cudaStream_t s, const Sets& sets)
{
    if (nlev < 2 || nlev > kVsubMaxLevels || v[0].n > kCoarseN || csize < 1) return cudaErrorInvalidValue;
    VsubArgs<T> a{};
    for (int l = 0; l < nlev; ++l) a.lev[l] = VsubLevel<T>{e[l], f[l], v[l], (T)h[l]};
    a.top = nlev - 1;
    a.zero_top = zero_top;
    a.npre = npre;
    a.npost = npost;
    a.act = sets.act;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(csize * sets.n));
    cfg.blockDim = dim3(kVsubThreads);
    cfg.dynamicSmemBytes = coarse_smem_bytes<T>(v[0].n);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)csize;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, vcluster_kernel<T>, a, csize);
}

int vcluster_size(bool fp64)
{
    // the largest cluster (16 needs the non-portable size) of which at least one fits on the device
    for (int cs = 16; cs >= 2; cs /= 2) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)cs);
        cfg.blockDim = dim3(kVsubThreads);
        cfg.dynamicSmemBytes = fp64 ? coarse_smem_bytes<double>(kCoarseN) : coarse_smem_bytes<float>(kCoarseN);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)cs;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        const cudaError_t e = fp64 ? cudaOccupancyMaxActiveClusters(&n, vcluster_kernel<double>, &cfg)
                                   : cudaOccupancyMaxActiveClusters(&n, vcluster_kernel<float>, &cfg);
        if (e == cudaSuccess && n >= 1) return cs;
        (void)cudaGetLastError();
    }
    return 0;
}

cudaError_t launch_vslab(float* e, const float* f, const LevelView& v, double h, double hc, int zero_top, int npre,
                         int npost, int csize, cudaStream_t s, const Sets& sets)
{
    if (v.n != kSlabN || v.M != kSlabM || (v.cs & 3) != 0 || (reinterpret_cast<uintptr_t>(e) & 15) != 0 ||
        (reinterpret_cast<uintptr_t>(f) & 15) != 0 || !(csize == 4 || csize == 8 || csize == 16))
        return cudaErrorInvalidValue;
    SlabArgs a{};
    a.e = e;
    a.f = f;
    a.cs = v.cs;
    a.h2 = (float)(h * h);
    a.sixth = 1.0f / 6.0f;
    a.ih2 = (float)(1.0 / (h * h));
    a.hc = (float)hc;
    a.zero_top = zero_top;
    a.npre = npre;
    a.npost = npost;
    a.csize = csize;
    a.act = sets.act;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(csize * sets.n));
    cfg.blockDim = dim3((unsigned)slab_threads(csize));
    cfg.dynamicSmemBytes = slab_smem_bytes(csize);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)csize;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return slab_threads(csize) > 256 ? cudaLaunchKernelEx(&cfg, vslab_kernel<512>, a)
                                     : cudaLaunchKernelEx(&cfg, vslab_kernel<256>, a);
}

int vslab_size(int want)
{
    // `want` CTAs per cluster (4, 8 or 16) if at least one such cluster fits on the device, else 0
    if (!(want == 4 || want == 8 || want == 16)) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)want);
    cfg.blockDim = dim3((unsigned)slab_threads(want));
    cfg.dynamicSmemBytes = slab_smem_bytes(want);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)want;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    const cudaError_t err = slab_threads(want) > 256 ? cudaOccupancyMaxActiveClusters(&n, vslab_kernel<512>, &cfg)
                                                     : cudaOccupancyMaxActiveClusters(&n, vslab_kernel<256>, &cfg);
    if (err == cudaSuccess && n >= 1) return want;
    (void)cudaGetLastError();
    return 0;
}

int vsub_grid(int sms)
{
    // one CTA per SM: the kernel's shared memory (the coarse solver's) allows one or more per SM
    return sms;
}

template <typename T>
void launch_convert_rhs(const double* rhs, double coef, int n, T* f, const LevelView& v, cudaStream_t s,
                        const Sets& sets)
{
    const dim3 g(cdiv((long long)(n - 1) * (n - 1) * (n / 2), kConvertThreads), (unsigned)sets.n);
    convert_rhs_kernel<T><<<g, kConvertThreads, 0, s>>>(rhs, coef, n, f, v);
}

template <typename T>
void launch_assign_outer(double* u, int n, const T* e, const LevelView& v, bool add, cudaStream_t s, const Sets& sets)
{
    if (add)
        assign_outer_kernel<T, true><<<per_sets(outer_grid(n), sets), kOuterThreads, 0, s>>>(u, n, e, v, sets.act);
    else
        assign_outer_kernel<T, false><<<per_sets(outer_grid(n), sets), kOuterThreads, 0, s>>>(u, n, e, v, sets.act);
}

int residual_outer_blocks(int n)
{
    const dim3 g = outer_grid(n);
    return (int)(g.x * g.y * g.z);
}

template <typename T>
int launch_residual_outer(const double* u, const double* rhs, double coef, int n, double h, T* r, const LevelView& v,
                          double* partials, cudaStream_t s)
{
    residual_outer_kernel<T><<<outer_grid(n), kOuterThreads, 0, s>>>(u, rhs, coef, n, 1.0 / (h * h), r, v, partials);
    return residual_outer_blocks(n);
}

int residual_rows_blocks(int n)
{
    const int rows = (n - 1) * (n - 1);
    return rows < kResidMaxBlocks ? rows : kResidMaxBlocks;
}

template <typename T>
int launch_residual_rows(const double* u, const double* rhs, double coef, int n, double h, bool want_f, T* r,
                         const LevelView& v, double* partials, cudaStream_t s, const Sets& sets)
{
    const int nb = residual_rows_blocks(n);
    const dim3 g(nb, sets.n);
    const double ih2 = 1.0 / (h * h);
    if (want_f)
        residual_rows_kernel<T, true><<<g, kRowThreads, 0, s>>>(u, rhs, coef, n, ih2, r, v, partials, sets.pstride,
                                                                sets.act);
    else
        residual_rows_kernel<T, false><<<g, kRowThreads, 0, s>>>(u, rhs, coef, n, ih2, r, v, partials, sets.pstride,
                                                                 sets.act);
    return nb;
}

void launch_decide(const double* partials, int nblocks, SolveState* st, double tol, int max_it, bool first,
                   bool refine, const cudaGraphConditionalHandle* handle, int* fault, cudaStream_t s, const Sets& sets)
{
    if (sets.n == 1) {
        if (handle)
            decide_kernel<true><<<1, kReduceThreads, 0, s>>>(partials, nblocks, st, tol, max_it, first, refine,
                                                             *handle, fault, 0);
        else
            decide_kernel<false><<<1, kReduceThreads, 0, s>>>(partials, nblocks, st, tol, max_it, first, refine, 0,
                                                              fault, 0);
        return;
    }
    decide_kernel<false><<<sets.n, kReduceThreads, 0, s>>>(partials, nblocks, st, tol, max_it, first, refine, 0,
                                                           nullptr, sets.pstride);
    if (handle)
        decide_any_kernel<true><<<1, 32, 0, s>>>(st, sets.n, first, *handle, fault);
    else
        decide_any_kernel<false><<<1, 32, 0, s>>>(st, sets.n, first, 0, fault);
}

cudaError_t prepare_kernels()
{
    if (cudaFuncSetAttribute(vsub_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)coarse_smem_bytes<float>(kCoarseN)) != cudaSuccess ||
        cudaFuncSetAttribute(vsub_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)coarse_smem_bytes<double>(kCoarseN)) != cudaSuccess ||
        cudaFuncSetAttribute(vcluster_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)coarse_smem_bytes<float>(kCoarseN)) != cudaSuccess ||
        cudaFuncSetAttribute(vcluster_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)coarse_smem_bytes<double>(kCoarseN)) != cudaSuccess ||
        cudaFuncSetAttribute(vcluster_kernel<float>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess ||
        cudaFuncSetAttribute(vcluster_kernel<double>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess)
        return cudaGetLastError();
    if (cudaFuncSetAttribute(vslab_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)slab_smem_bytes(4)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(vslab_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)slab_smem_bytes(8)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(vslab_kernel<256>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return cudaGetLastError();
    return cudaFuncSetAttribute(coarse_kernel<float, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)coarse_smem_bytes<float>(kCoarseN));
}

void launch_reduce_norms(const double* partials, int nblocks, double* out, cudaStream_t s)
{
    reduce_norms_kernel<<<1, kReduceThreads, 0, s>>>(partials, nblocks, out);
}

#define QUMOND_INSTANTIATE(T)                                                                                          \
    template void launch_rb_half<T>(T*, const T*, const LevelView&, int, bool, double, cudaStream_t, const Sets&);    \
    template void launch_restrict_resid_red<T>(const T*, const T*, const LevelView&, T*, const LevelView&, double,    \
                                               cudaStream_t, const Sets&);                                             \
    template void launch_restrict_full<T>(const T*, const LevelView&, T*, const LevelView&, cudaStream_t,             \
                                          const Sets&);                                                                \
    template void launch_prolong_black<T>(const T*, const LevelView&, T*, const LevelView&, bool, cudaStream_t,       \
                                          const Sets&);                                                                \
    template void launch_set_boundary<T>(T*, const LevelView&, const double*, int, cudaStream_t, const Sets&);        \
    template cudaError_t launch_vsub<T>(T* const*, T* const*, const LevelView*, const double*, int, int, int, int,     \
                                        unsigned*, int*, long long, int, cudaStream_t);                               \
    template cudaError_t launch_vcluster<T>(T* const*, T* const*, const LevelView*, const double*, int, int, int, int, \
                                            int, cudaStream_t, const Sets&);                                           \
    template cudaError_t launch_coarse<T>(int, T*, const T*, const LevelView&, double, const double*, int, int, int,  \
                                          int, cudaStream_t, const Sets&);                                             \
    template void launch_convert_rhs<T>(const double*, double, int, T*, const LevelView&, cudaStream_t, const Sets&); \
    template void launch_assign_outer<T>(double*, int, const T*, const LevelView&, bool, cudaStream_t, const Sets&);  \
    template int launch_residual_outer<T>(const double*, const double*, double, int, double, T*, const LevelView&,    \
                                          double*, cudaStream_t);                                                      \
    template int launch_residual_rows<T>(const double*, const double*, double, int, double, bool, T*,                  \
                                         const LevelView&, double*, cudaStream_t, const Sets&);

QUMOND_INSTANTIATE(float)
QUMOND_INSTANTIATE(double)

}  // namespace qumond
