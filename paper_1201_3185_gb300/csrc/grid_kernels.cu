// Grid kernels of the QUMOND path on natural-layout FP64 arrays: the
// fixed-point CIC deposit (Section 2 step 1), nested-box boundary values
// (Section 2), the QUMOND source (Section 2 step 3, Eq. 2), forces and the
// rotation curve (Section 2, Eq. 4; box rule of Section 3.1).
#include "qumond_internal.h"
#include "fixed_conv.h"

#include <cstring>

namespace qumond {

namespace {

inline unsigned cdiv(long long a, long long b) { return (unsigned)((a + b - 1) / b); }

__device__ __forceinline__ long long nat(int n, int i, int j, int k)
{
    const long long P = n + 1;
    return (long long)i + P * ((long long)j + P * (long long)k);
}

// ---------------------------------------------------------------------------
// Cloud-in-cell deposit in 64-bit fixed point.  Every product is an
// individually rounded FP64 operation (no fused multiply-add), and the
// conversion rounds half to even, so each corner's integer share is the same
// on any machine and the grid does not depend on the order of the atomics.
//
// The FP64 pipe (2 operations a clock on each SM, conversions and comparisons
// among them) bounds the kernel before the atomics do, so it runs the 27
// roundings of the definition only: the range test, the cells and the
// conversions of the shares work on the bits, on the integer pipe beside it.
// Measured with the clearing of the grid and the density (below) at 2e6
// particles in a 257^3 box: 178 us, 271 us with FP64 comparisons, floors and
// conversions (47 FP64 instructions a particle, two a node in the density).

// Index coordinate t in [0, n)?  `top`: the bits of (double)n.  Positive
// doubles order as their bits; -0 is in, negative values and NaNs are out.
__device__ __forceinline__ bool in_axis(double t, long long top)
{
    const long long b = __double_as_longlong(t);
    return (b >= 0 && b < top) || b == (long long)0x8000000000000000ULL;
}

// Integer part of 0 <= t < 2^20 and the offset t - floor(t): for t >= 1 the
// integer part is the top of the significand, and t without the bits below it
// is floor(t).
__device__ __forceinline__ int cell_of(double t, double& d)
{
    const int hi = __double2hiint(t);
    const int sh = 1043 - (hi >> 20);  // 20 - exponent: fraction bits in the high word
    const bool low = hi < 0x3ff00000;  // t < 1 (or -0)
    d = t - __hiloint2double(low ? 0 : hi & (int)(0xffffffffu << (sh & 31)), 0);
    return low ? 0 : ((hi & 0xfffff) | 0x100000) >> (sh & 31);
}

// round(w) to the nearest integer, ties to even, for |w| < 2^52.
__device__ __forceinline__ long long round_share(double w)
{
    const long long b = __double_as_longlong(w);
    const int ex = (int)(b >> 52) & 0x7ff;
    const int sh = min(1075 - ex, 54);  // 1 .. 54; at 54 the value is below 1/2 and rounds to 0
    const long long m = (b & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
    const long long q = (m + ((m >> sh) & 1) + ((1LL << (sh - 1)) - 1)) >> sh;
    return b < 0 ? -q : q;
}

constexpr int kCicThreads = 256;

__global__ void __launch_bounds__(kCicThreads)
cic_deposit_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                   const double* __restrict__ m, long long np, int n, long long top, double xlo, double ylo, double zlo,
                   double inv_h, double two_shift, unsigned long long* __restrict__ q)
{
    {
        const int set = blockIdx.y;  // one row of blocks per set: np particles each
        const long long po = set * np;
        x += po, y += po, z += po, m += po;
        q += set * nat_elems(n);
    }
    const long long p = blockIdx.x * (long long)kCicThreads + threadIdx.x;
    if (p >= np) return;
    const double px = x[p], py = y[p], pz = z[p], pm = m[p];
    const double tx = __dmul_rn(__dsub_rn(px, xlo), inv_h);
    const double ty = __dmul_rn(__dsub_rn(py, ylo), inv_h);
    const double tz = __dmul_rn(__dsub_rn(pz, zlo), inv_h);
    if (!(in_axis(tx, top) && in_axis(ty, top) && in_axis(tz, top))) return;
    double dx, dy, dz;
    const int i = cell_of(tx, dx), j = cell_of(ty, dy), k = cell_of(tz, dz);
    const double wx[2] = {__dsub_rn(1.0, dx), dx};
    const double wy[2] = {__dsub_rn(1.0, dy), dy};
    const double wz[2] = {__dsub_rn(1.0, dz), dz};
    const double ms = __dmul_rn(pm, two_shift);
    const int P = n + 1;
    unsigned long long* cell = q + (i + (long long)P * (j + (long long)P * k));
    auto corners = [&](auto&& round) {
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const double mx = __dmul_rn(ms, wx[a]);  // ((ms * wx) * wy) * wz, left to right
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const double mxy = __dmul_rn(mx, wy[b]);
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    atomicAdd(cell + (a + P * (b + P * c)), (unsigned long long)round(__dmul_rn(mxy, wz[c])));
            }
        }
    };
    // the shares are at most |ms|: below 2^52 they are rounded on the integer pipe, beyond it (or for an
    // infinite or undefined mass) by the conversion instruction; two branches, so that the instruction is
    // not issued for both
    if (((__double2hiint(ms) >> 20) & 0x7ff) < 1075)
        corners([](double w) { return round_share(w); });
    else
        corners([](double w) { return __double2ll_rn(w); });
}

// rho = q * scale.  The conversion runs on the integer pipe (fixed_conv.h, the
// same rounding), and a warp whose nodes hold no mass, as most nodes of a box,
// skips it and the product: +0 * scale is +0.  Four nodes a thread keep enough
// loads in flight.
constexpr int kRhoThreads = 256, kRhoPer = 4;

__global__ void __launch_bounds__(kRhoThreads)
fixed_to_rho_kernel(const long long* __restrict__ q, double* __restrict__ rho, long long count, double scale)
{
    const long long t = blockIdx.x * (long long)(kRhoThreads * kRhoPer) + threadIdx.x;
    long long v[kRhoPer];
#pragma unroll
    for (int u = 0; u < kRhoPer; ++u) v[u] = t + u * kRhoThreads < count ? q[t + u * kRhoThreads] : 0;
#pragma unroll
    for (int u = 0; u < kRhoPer; ++u) {
        double r = 0.0;
        if (__any_sync(0xffffffffu, v[u] != 0)) r = i64_to_f64_rn_scaled(v[u], 0) * scale;
        if (t + u * kRhoThreads < count) rho[t + u * kRhoThreads] = r;
    }
}

// ---------------------------------------------------------------------------
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

// blockIdx.z = 6 * set + face
__global__ void boundary_zero_kernel(double* __restrict__ u, int n)
{
    const int set = blockIdx.z / 6, face = blockIdx.z - 6 * set;
    const int a = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (a > n) return;
    int i, j, k;
    face_node(face, a, b, n, i, j, k);
    u[set * nat_elems(n) + nat(n, i, j, k)] = 0.0;
}

// Exact FP32 -> FP64 with integer ops (subnormals flushed to zero).
__device__ __forceinline__ double f32_to_f64(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned sign = u & 0x80000000u, e = u & 0x7f800000u;
    unsigned hi = ((u & 0x7fffffffu) >> 3) + (896u << 20), lo = u << 29;
    if (e == 0u) hi = 0u, lo = 0u;
    if (e == 0x7f800000u) hi += 896u << 20;  // exponent 255 to 2047
    return __hiloint2double((int)(sign | hi), (int)lo);
}

// Boundary of a box from its parent (box_ratio times the side, same centre,
// same n): child node i sits at parent index n (r-1)/(2r) + i/r along each
// axis (Section 2: the parent solution is interpolated onto the child's
// boundary).
//
// The ratio is a power of two, so the cell and the offsets 0, 1/r, .. (r-1)/r are
// exact integers, and so are the weights, products of three of them over r^3:
// they are formed on the integer and FP32 pipes, and the FP64 pipe, which bounds
// the kernel, does the eight fused products.  6 faces of 257^2: about 13 us, 60
// with the weights in FP64.
__global__ void boundary_from_parent_kernel(const double* __restrict__ parent, double* __restrict__ u, int n, int ratio)
{
    const int set = blockIdx.z / 6, face = blockIdx.z - 6 * set;  // blockIdx.z = 6 * set + face
    parent += set * nat_elems(n);
    u += set * nat_elems(n);
    const int a = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (a > n) return;
    int i, j, k;
    face_node(face, a, b, n, i, j, k);
    const int lr = 31 - __clz(ratio), q = (n >> 1) * (ratio - 1);  // child node 0 lies at q / r
    const int t[3] = {q + i, q + j, q + k};
    int i0[3], d[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) i0[x] = t[x] >> lr, d[x] = t[x] & (ratio - 1);
    const float unit = __int_as_float((127 - 3 * lr) << 23);  // r^-3
    double v = 0.0;
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
        for (int y = 0; y < 2; ++y)
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const int w = (x ? d[0] : ratio - d[0]) * (y ? d[1] : ratio - d[1]) * (z ? d[2] : ratio - d[2]);
                v = fma(f32_to_f64((float)w * unit), parent[nat(n, i0[0] + x, i0[1] + y, i0[2] + z)], v);
            }
    u[nat(n, i, j, k)] = v;
}

// ---------------------------------------------------------------------------
// QUMOND source by the face-flux difference (Section 2 step 3, Eq. 2).
//
// Precision: the differences of the potential carry the information and are
// taken to ~48 bits; the gradient magnitude, nu and the fluxes are FP32
// (which perturbs the solved potential by ~1e-8 relative).  FP64 arithmetic
// and 64-bit conversions are ~60x slower than FP32 on this GPU, so each FP64
// value is split once, with integer instructions, into an exact pair of FP32
// numbers hi + lo (hi: the top 24 significant bits, lo: the next 24), and a
// difference is (hi_a - hi_b) + (lo_a - lo_b).
//
// Layout: a warp owns 30 x 2 columns of (i, j) and walks k through a chunk of
// planes on its own, without shared memory or block barriers.  Lane l holds
// the column i = i0 - 1 + l of the two rows and of one halo row on each side
// in registers, as hi/lo pairs of the planes k-1, k, k+1; neighbours in x come
// by shuffles (the outer two lanes are halo), neighbours in y and z lie in the
// thread's own registers.  The kernel is bound by instruction issue, so each
// central difference is formed once per node and used by the four faces that
// average it, and the arithmetic is packed in pairs (one instruction rounds
// two sums or products).  Measured at 257^3: 150 us; forming the 15
// differences of a node's three faces from shared-memory planes took 512
// instructions a node and 277 us.  Four rows a warp (fewer halo rows, 119
// registers) took 206 us: too few warps to cover the latencies.

// x = hi + lo exactly up to the 48th significant bit, both FP32, integer ops
// only.  |x| < 2^-126 gives (0, 0); lo is dropped below |x| < 2^-74; beyond
// FP32's range (and for infinities and NaNs) there is no split.
__device__ __noinline__ float2 split_hi_lo_ends(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sign = (unsigned)(b >> 63) << 31;
    const int E = (int)((b >> 52) & 0x7ffu);
    if (E < 897) return make_float2(0.0f, 0.0f);
    if (E > 1150) return make_float2(__double2float_rn(x), 0.0f);
    const unsigned long long M = b & 0xFFFFFFFFFFFFFull;  // 897 <= E < 949
    return make_float2(__uint_as_float(sign | ((unsigned)(E - 896) << 23) | (unsigned)(M >> 29)), 0.0f);
}

// for 949 <= exponent field <= 1150 (the caller's check)
__device__ __forceinline__ unsigned split_field(double x) { return (unsigned)__double2hiint(x) & 0x7ff00000u; }
__device__ __forceinline__ float2 split_hi_lo(double x)
{
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned ex = h & 0x7ff00000u, sign = h & 0x80000000u;
    // exponent E and the fraction's top 23 bits, rebiased by E - 896 (modulo 2^9, the bits that a shift by three
    // leaves); then the fraction's other 29 bits times 2^(E - 948 - 127)
    const float hi = __uint_as_float(sign | ((__funnelshift_l(l, h, 3) - (896u << 23)) & 0x7fffffffu));
    const float r = __uint2float_rn(l & 0x1FFFFFFFu);
    return make_float2(hi, r * __uint_as_float(sign | (((ex << 3) - (948u << 23)) & 0x7fffffffu)));
}

constexpr int kSrcX = 30;         // output columns of a warp: lanes 1 .. 30
constexpr int kSrcY = 2;          // output rows of a warp
constexpr int kSrcR = kSrcY + 2;  // rows held, with the halo
constexpr int kSrcWarps = 4;      // warps of a CTA, along y
constexpr int kSrcKC = 24;        // planes of a chunk

// Differences of hi/lo pairs, both parts in one packed operation.
__device__ __forceinline__ float pair_diff(float2 a, float2 b)
{
    const float2 d = __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
    return d.x + d.y;
}

// Fluxes (times h) through two faces, each from its node P to P + e_axis:
// nu(|g|/a0) * (Phi(Q) - Phi(P)); |g| from the normal difference dn and the
// means of the two nodes' transverse central differences (ta, tb their sums);
// a face with g = 0 carries no flux.
__device__ __forceinline__ float2 face_flux(float2 dn, float2 ta, float2 tb, float inv_h, float four_a0)
{
    const float q = 0.25f * inv_h;
    const float2 gn = __fmul2_rn(dn, make_float2(inv_h, inv_h));
    const float2 ga = __fmul2_rn(ta, make_float2(q, q)), gb = __fmul2_rn(tb, make_float2(q, q));
    const float2 g2 = __ffma2_rn(gb, gb, __ffma2_rn(gn, gn, __fmul2_rn(ga, ga)));
    const float2 y = __ffma2_rn(make_float2(four_a0, four_a0), make_float2(rsqrtf(g2.x), rsqrtf(g2.y)),
                                make_float2(1.0f, 1.0f));
    const float2 w = __fadd2_rn(make_float2(sqrtf(y.x), sqrtf(y.y)), make_float2(1.0f, 1.0f));
    const float2 f = __fmul2_rn(__fmul2_rn(w, make_float2(0.5f, 0.5f)), dn);
    return make_float2(g2.x > 0.0f ? f.x : 0.0f, g2.y > 0.0f ? f.y : 0.0f);
}

// One plane's part of the warp's columns: the values and the differences that
// need no other plane.
struct SrcPlane {
    float2 v[kSrcR];
    float cx[kSrcR];      // Phi(i+1) - Phi(i-1)
    float2 cy;            // Phi(j+1) - Phi(j-1), rows 1, 2
    float2 dx;            // Phi(i+1) - Phi(i), rows 1, 2
    float dy[kSrcY + 1];  // Phi(j+1) - Phi(j), rows 0 .. 2
};

__device__ __forceinline__ void src_plane(const double (&v)[kSrcR], SrcPlane& p)
{
    constexpr unsigned kAll = 0xffffffffu;
    bool fast = true;
#pragma unroll
    for (int r = 0; r < kSrcR; ++r) {
        fast = fast && split_field(v[r]) - (949u << 20) <= (1150u - 949u) << 20;
        p.v[r] = split_hi_lo(v[r]);
    }
    if (!fast) {
#pragma unroll
        for (int r = 0; r < kSrcR; ++r)
            if (split_field(v[r]) - (949u << 20) > (1150u - 949u) << 20) p.v[r] = split_hi_lo_ends(v[r]);
    }
    float dx[kSrcR];
#pragma unroll
    for (int r = 0; r < kSrcR; ++r) {
        const float2 right = make_float2(__shfl_down_sync(kAll, p.v[r].x, 1), __shfl_down_sync(kAll, p.v[r].y, 1));
        const float2 left = make_float2(__shfl_up_sync(kAll, p.v[r].x, 1), __shfl_up_sync(kAll, p.v[r].y, 1));
        p.cx[r] = pair_diff(right, left);
        dx[r] = pair_diff(right, p.v[r]);
    }
    p.dx = make_float2(dx[1], dx[2]);
    p.cy = make_float2(pair_diff(p.v[2], p.v[0]), pair_diff(p.v[3], p.v[1]));
#pragma unroll
    for (int r = 0; r <= kSrcY; ++r) p.dy[r] = pair_diff(p.v[r + 1], p.v[r]);
}

// fluxes through the faces between planes p and q = p + e_z of rows 1, 2
__device__ __forceinline__ float2 src_flux_z(const SrcPlane& p, const SrcPlane& q, float ih, float fa)
{
    const float2 dz = make_float2(pair_diff(q.v[1], p.v[1]), pair_diff(q.v[2], p.v[2]));
    const float2 tx = __fadd2_rn(make_float2(p.cx[1], p.cx[2]), make_float2(q.cx[1], q.cx[2]));
    return face_flux(dz, tx, __fadd2_rn(p.cy, q.cy), ih, fa);
}

__global__ void __launch_bounds__(32 * kSrcWarps)
source_kernel(const double* __restrict__ phi, double* __restrict__ src, int n, float inv_h, float four_a0,
              float inv_h2, int zper)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int set = (int)gridDim.z == zper ? 0 : blockIdx.z / zper;  // blockIdx.z = zper * set + chunk
    const int kc = blockIdx.z - set * zper;
    phi += set * nat_elems(n);
    src += set * nat_elems(n);
    const int lane = threadIdx.x & 31;
    const int i = blockIdx.x * kSrcX - 1 + lane;
    const int j0 = (blockIdx.y * kSrcWarps + (threadIdx.x >> 5)) * kSrcY;  // output rows j0, j0 + 1
    if (j0 > n) return;  // the whole warp
    const int k0 = kc * kSrcKC, k1 = min(k0 + kSrcKC, n + 1);
    const int P = n + 1;
    const long long Q = (long long)P * P;
    // rows j0 - 1 .. j0 + 2 of this lane's column; outside the grid the nearest node (it only feeds boundary
    // nodes, whose source is 0)
    int off[kSrcR];
#pragma unroll
    for (int r = 0; r < kSrcR; ++r) off[r] = min(max(i, 0), n) + P * min(max(j0 - 1 + r, 0), n);
    double v[kSrcR];
    auto fetch = [&](int k) {
        const double* at = phi + Q * min(max(k, 0), n);
#pragma unroll
        for (int r = 0; r < kSrcR; ++r) v[r] = at[off[r]];
    };
    const bool store = lane >= 1 && lane <= kSrcX && i <= n;
    const bool inner0 = i > 0 && i < n && j0 > 0 && j0 < n, inner1 = i > 0 && i < n && j0 + 1 < n;
    const bool store0 = store, store1 = store && j0 + 1 <= n;
    float2 fzm;  // fluxes through the -z faces of plane k
    // sources of plane k from planes m = k-1 and p = k; leaves plane k+1 in q and fetches plane k+2
    auto step = [&](int k, const SrcPlane& m, const SrcPlane& p, SrcPlane& q) {
        src_plane(v, q);
        if (k + 1 < k1) fetch(k + 2);  // in flight while this plane's fluxes are computed
        const float2 fz = src_flux_z(p, q, inv_h, four_a0);
        float cz[kSrcR];
#pragma unroll
        for (int r = 0; r < kSrcR; ++r) cz[r] = pair_diff(q.v[r], m.v[r]);
        const float2 cz12 = make_float2(cz[1], cz[2]);
        const float2 fy01 = face_flux(make_float2(p.dy[0], p.dy[1]),
                                      __fadd2_rn(make_float2(p.cx[0], p.cx[1]), make_float2(p.cx[1], p.cx[2])),
                                      __fadd2_rn(make_float2(cz[0], cz[1]), cz12), inv_h, four_a0);
        const float2 fx = face_flux(
            p.dx, __fadd2_rn(p.cy, make_float2(__shfl_down_sync(kAll, p.cy.x, 1), __shfl_down_sync(kAll, p.cy.y, 1))),
            __fadd2_rn(cz12, make_float2(__shfl_down_sync(kAll, cz[1], 1), __shfl_down_sync(kAll, cz[2], 1))), inv_h,
            four_a0);
        const float2 fxm = make_float2(__shfl_up_sync(kAll, fx.x, 1), __shfl_up_sync(kAll, fx.y, 1));
        const float fy2 = face_flux(make_float2(p.dy[2], 0.0f), make_float2(p.cx[2] + p.cx[3], 0.0f),
                                    make_float2(cz[2] + cz[3], 0.0f), inv_h, four_a0).x;
        const bool inner_k = k > 0 && k < n;
        double* out = src + (Q * k + off[1]);
        const float s0 = ((fx.x - fxm.x) + (fy01.y - fy01.x) + (fz.x - fzm.x)) * inv_h2;
        const float s1 = ((fx.y - fxm.y) + (fy2 - fy01.y) + (fz.y - fzm.y)) * inv_h2;
        if (store0) out[0] = inner0 && inner_k ? f32_to_f64(s0) : 0.0;
        if (store1) out[P] = inner1 && inner_k ? f32_to_f64(s1) : 0.0;
        fzm = fz;
    };
    SrcPlane a, b, c;
    fetch(k0 - 1);
    src_plane(v, a);
    fetch(k0);
    src_plane(v, b);
    fzm = src_flux_z(a, b, inv_h, four_a0);
    fetch(k0 + 1);
    for (int k = k0; k < k1; ++k) {
        step(k, a, b, c);
        a = b;
        b = c;
    }
}

// ---------------------------------------------------------------------------
// Forces at points: finest box whose containing cell has 8 interior corners.
//
// These kernels are bound by the FP64 pipe (2 operations a clock on each SM,
// against 64 integer ones), so what is not arithmetic of the result runs on
// the integer pipe, and a warp looks for every point's box first and
// interpolates once: with the interpolation inside the search, the points of
// a warp that lie in different boxes ran it one box after another.
// Measured at 2e6 points in 3 boxes of 257^3: 336 us, 824 us with the search
// around the interpolation and the 8 corners weighted one by one (222 FP64
// instructions a point, that pipe 86% busy).  The rounding error against
// extended precision at the same index coordinates is a little smaller: 1.04e-16
// of the rms force on 257^3 nodes (1.10e-16), 0.87e-16 on 33^3 (1.01e-16).

// Index coordinates of (x, y, z) in box g, and whether the containing cell has
// interior corners only: 1 <= t < n-1 on each axis.  `top` holds the bits of
// (double)(n-1); positive doubles order as their bits do, negative ones and
// NaNs with the sign bit are negative integers, other NaNs lie above.
__device__ __forceinline__ bool in_cells(const BoxGeom& g, long long top, double x, double y, double z, double* t)
{
    t[0] = (x - g.xlo) * g.inv_h;
    t[1] = (y - g.ylo) * g.inv_h;
    t[2] = (z - g.zlo) * g.inv_h;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const long long b = __double_as_longlong(t[a]);
        ok = ok && b >= 0x3ff0000000000000LL && b < top;
    }
    return ok;
}

// -grad Phi at index coordinates t of box g (in_cells): central differences at
// the cell's corners with CIC weights.  Along each axis the differences of a
// row are weighted first and the four rows after, 22 FP64 operations per
// component where weighting the 8 corners one by one takes 24 and the weights.
// set: which of the context's sets (its potentials sit at set (n+1)^3 in every box)
__device__ __forceinline__ void grad_at(const double* __restrict__ phi, double s, int n, const double* t, double* out)
{
    double d[3], w[3];
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        c[a] = cell_of(t[a], d[a]);
        w[a] = 1.0 - d[a];
    }
    const int P = n + 1;
    const long long Q = (long long)P * P;
    const double* p = phi + (c[0] + (long long)P * c[1] + Q * c[2]);
    // rows along axis U (stride u) at the corners (0, v), (0, z): the weighted difference of the row
    auto part = [&](long long u, long long v, long long z, int U, int V, int Z) {
        auto row = [&](const double* r) {
            return fma(r[2 * u] - r[0], d[U], (r[u] - r[-u]) * w[U]);
        };
        const double lo = fma(row(p + v), d[V], row(p) * w[V]);
        const double hi = fma(row(p + v + z), d[V], row(p + z) * w[V]);
        return fma(hi, d[Z], lo * w[Z]) * s;
    };
    out[0] = part(1, P, Q, 0, 1, 2);
    out[1] = part(P, 1, Q, 1, 0, 2);
    out[2] = part(Q, 1, P, 2, 0, 1);
}

// g = -grad Phi at (x, y, z) from the finest box b <= b0 whose cell is interior; 0 where there is none.
__device__ __forceinline__ void force_at(const BoxSet& boxes, int b0, double x, double y, double z, int set, double* g)
{
    double t[3];
    const double* phi = nullptr;
    double s = 0.0;
    for (int b = b0; b >= 0; --b)
        if (in_cells(boxes.b[b], boxes.top, x, y, z, t)) {
            phi = boxes.b[b].phi;
            s = boxes.b[b].s;
            break;
        }
    g[0] = g[1] = g[2] = 0.0;
    if (phi) grad_at(phi + set * nat_elems(boxes.n), s, boxes.n, t, g);
}

__global__ void forces_kernel(BoxSet boxes, const double* __restrict__ qx, const double* __restrict__ qy,
                              const double* __restrict__ qz, long long nq, double* __restrict__ gx,
                              double* __restrict__ gy, double* __restrict__ gz)
{
    const int set = blockIdx.y;  // one row of blocks per set: nq points each
    {
        const long long po = set * nq;
        qx += po, qy += po, qz += po, gx += po, gy += po, gz += po;
    }
    const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (p >= nq) return;
    double g[3];
    force_at(boxes, boxes.nboxes - 1, qx[p], qy[p], qz[p], set, g);
    gx[p] = g[0];
    gy[p] = g[1];
    gz[p] = g[2];
}

// One CTA per radius bin, one thread per azimuth; the azimuthal mean is
// summed in index order by thread 0, so the result is reproducible.
constexpr int kMaxPhi = 1024;

// With several sets: blockIdx.y = set, its outermost radius rmax_sets[set]
// when given, its bins at set * nbins of the outputs.
__global__ void rotation_curve_kernel(BoxSet boxes, double cx, double cy, double cz, int nbins, double rmax,
                                      const double* __restrict__ rmax_sets, int nphi, double frac,
                                      double* __restrict__ r_out, double* __restrict__ vc_out)
{
    __shared__ double dphidr[kMaxPhi];
    const int set = blockIdx.y;
    if (rmax_sets) rmax = rmax_sets[set];
    r_out += set * (long long)nbins;
    vc_out += set * (long long)nbins;
    const int kb = blockIdx.x;
    const double R = ((double)kb + 0.5) * rmax / (double)nbins;
    int b0 = 0;
    for (int b = boxes.nboxes - 1; b >= 0; --b)
        if (R < frac * boxes.b[b].L) {
            b0 = b;
            break;
        }
    for (int m = threadIdx.x; m < nphi; m += blockDim.x) {
        const double ph = 6.283185307179586476925286766559 * (double)m / (double)nphi;
        double s, c;
        sincos(ph, &s, &c);
        double g[3];
        force_at(boxes, b0, cx + R * c, cy + R * s, cz, set, g);
        dphidr[m] = -(g[0] * c + g[1] * s);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int m = 0; m < nphi; ++m) sum += dphidr[m];
        const double v2 = R * (sum / (double)nphi);
        r_out[kb] = R;
        vc_out[kb] = v2 >= 0.0 ? sqrt(v2) : -sqrt(-v2);
    }
}

// Science extras on the same tracers and box rule as the rotation curve.
// mode 0 (Eq. 3, algebraic MOND): the field at a tracer is nu(|g_N|/a0) g_N
//   from the Newtonian potentials (a tracer with g_N = 0 adds 0), out = sign(s) sqrt(|s|),
//   s = R * mean of -(g . R^);
// mode 1 (Section 5.6, isothermal sech^2(z/h) stellar layer): tracers at height z_eval,
//   s = mean of dPhi/dz * h / (2 tanh(z_eval / h)), out = sign(s) sqrt(|s|) = sigma_z.
__global__ void profile_kernel(BoxSet boxes, double cx, double cy, double cz, int nbins, double rmax, int nphi,
                               double frac, int mode, double a0, double z_eval, double h, double* __restrict__ r_out,
                               double* __restrict__ out)
{
    __shared__ double val[kMaxPhi];
    const int set = blockIdx.y;  // one row of blocks per set
    r_out += set * (long long)nbins;
    out += set * (long long)nbins;
    const int kb = blockIdx.x;
    const double R = ((double)kb + 0.5) * rmax / (double)nbins;
    int b0 = 0;
    for (int b = boxes.nboxes - 1; b >= 0; --b)
        if (R < frac * boxes.b[b].L) {
            b0 = b;
            break;
        }
    const double zt = mode == 1 ? cz + z_eval : cz;
    for (int m = threadIdx.x; m < nphi; m += blockDim.x) {
        const double ph = 6.283185307179586476925286766559 * (double)m / (double)nphi;
        double s, c;
        sincos(ph, &s, &c);
        double g[3];
        force_at(boxes, b0, cx + R * c, cy + R * s, zt, set, g);
        if (mode == 0) {
            const double gm = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
            const double nu = gm > 0.0 ? 0.5 + 0.5 * sqrt(1.0 + 4.0 * a0 / gm) : 0.0;
            val[m] = -nu * (g[0] * c + g[1] * s);
        } else {
            val[m] = -g[2];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int m = 0; m < nphi; ++m) sum += val[m];
        const double mean = sum / (double)nphi;
        const double v2 = mode == 0 ? R * mean : mean * h / (2.0 * tanh(z_eval / h));
        r_out[kb] = R;
        out[kb] = v2 >= 0.0 ? sqrt(v2) : -sqrt(-v2);
    }
}

}  // namespace

// --- launchers ----------------------------------------------------------------
void launch_cic_deposit(const double* x, const double* y, const double* z, const double* m, long long np, int n,
                        double xlo, double ylo, double zlo, double inv_h, double two_shift, int64_t* q,
                        cudaStream_t s, int nsets)
{
    if (np <= 0) return;
    const double dn = (double)n;
    long long top;
    memcpy(&top, &dn, sizeof(top));
    cic_deposit_kernel<<<dim3(cdiv(np, kCicThreads), (unsigned)nsets), kCicThreads, 0, s>>>(
        x, y, z, m, np, n, top, xlo, ylo, zlo, inv_h, two_shift, reinterpret_cast<unsigned long long*>(q));
}

void launch_fixed_to_rho(const int64_t* q, double* rho, long long count, double scale, cudaStream_t s)
{
    fixed_to_rho_kernel<<<cdiv(count, kRhoThreads * kRhoPer), kRhoThreads, 0, s>>>(
        reinterpret_cast<const long long*>(q), rho, count, scale);
}

void launch_boundary_zero(double* u, int n, cudaStream_t s, int nsets)
{
    boundary_zero_kernel<<<dim3(cdiv(n + 1, 128), (unsigned)(n + 1), 6 * (unsigned)nsets), 128, 0, s>>>(u, n);
}

void launch_boundary_from_parent(const double* parent, double* u, int n, int ratio, cudaStream_t s, int nsets)
{
    boundary_from_parent_kernel<<<dim3(cdiv(n + 1, 128), (unsigned)(n + 1), 6 * (unsigned)nsets), 128, 0, s>>>(
        parent, u, n, ratio);
}

void launch_source(const double* phi, double* src, int n, double h, double a0, cudaStream_t s, int nsets)
{
    const unsigned zper = cdiv(n + 1, kSrcKC);
    const dim3 grid(cdiv(n + 1, kSrcX), cdiv(n + 1, kSrcY * kSrcWarps), zper * (unsigned)nsets);
    source_kernel<<<grid, 32 * kSrcWarps, 0, s>>>(phi, src, n, (float)(1.0 / h), (float)(4.0 * a0),
                                                        (float)(1.0 / (h * h)), (int)zper);
}

void launch_forces(const BoxSet& boxes, const double* qx, const double* qy, const double* qz, long long nq,
                   double* gx, double* gy, double* gz, cudaStream_t s, int nsets)
{
    if (nq <= 0) return;
    forces_kernel<<<dim3(cdiv(nq, 128), (unsigned)nsets), 128, 0, s>>>(boxes, qx, qy, qz, nq, gx, gy, gz);
}

void launch_rotation_curve(const BoxSet& boxes, double cx, double cy, double cz, int nbins, double rmax,
                           const double* rmax_sets, int nphi, double frac, double* r_out, double* vc_out,
                           cudaStream_t s, int nsets)
{
    rotation_curve_kernel<<<dim3(nbins, nsets), 128, 0, s>>>(boxes, cx, cy, cz, nbins, rmax, rmax_sets, nphi, frac,
                                                             r_out, vc_out);
}

void launch_profile(const BoxSet& boxes, double cx, double cy, double cz, int nbins, double rmax, int nphi, double frac,
                    int mode, double a0, double z_eval, double h, double* r_out, double* out, cudaStream_t s,
                    int nsets)
{
    profile_kernel<<<dim3(nbins, nsets), 128, 0, s>>>(boxes, cx, cy, cz, nbins, rmax, nphi, frac, mode, a0, z_eval, h,
                                                      r_out, out);
}

// Quality of fit (Section 3.5): chi2[s] = (1/nbins) sum_i ((vc[s][i] - v_obs[i]) / sigma[i])^2.
// One warp per parameter set; lane l sums bins l, l+32, ... and the warp adds
// the 32 partial sums by a fixed shuffle tree, so the result does not depend
// on scheduling.
__global__ void chi2_kernel(const double* __restrict__ vc, const double* __restrict__ v_obs,
                            const double* __restrict__ sigma, int nbins, int nsets, double* __restrict__ chi2)
{
    const int set = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (set >= nsets) return;
    const double* row = vc + (long long)set * nbins;
    double acc = 0.0;
    for (int i = lane; i < nbins; i += 32) {
        const double d = (row[i] - v_obs[i]) / sigma[i];
        acc += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) chi2[set] = acc / (double)nbins;
}

void launch_chi2(const double* vc, const double* v_obs, const double* sigma, int nbins, int nsets, double* chi2,
                 cudaStream_t s)
{
    const int warps = 4;
    chi2_kernel<<<(nsets + warps - 1) / warps, 32 * warps, 0, s>>>(vc, v_obs, sigma, nbins, nsets, chi2);
}

}  // namespace qumond
