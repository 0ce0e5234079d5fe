// Whole red-black sweeps in one pass over an FP32 level (zero boundary
// values: the V-cycles on the correction equation).
//
// A red half-sweep overwrites every interior red node from its black
// neighbours alone, and the black half-sweep after it needs the red values of
// one neighbour in each direction.  So a sweep takes the black values b and
// the right-hand side f to the next black values b': the red values in between
// need not exist in memory.  Two launches of the half-sweeps move 12 bytes a
// node (each reads the other colour and f and writes its own); this pass moves
// 8 (b 2, f 4, b' 2), 6 from a zero start, and costs one launch.  b' goes to
// another array, since neighbouring blocks still read b around their tiles;
// the two change roles from sweep to sweep.  With kProlong the sweep starts from
// b + P e_c, the coarse-grid correction applied as the planes arrive; with
// kRestrict the residual of the red nodes (the black ones' vanishes) is formed
// from b' and the red values a plane later and weighted into the coarser
// level's right-hand side (0.5 bytes more, where the restriction on its own
// reads 6 bytes again and needs the red values in memory); with kRed, the last
// sweep, the red values are written (2 more).
//
// Every node's arithmetic is that of rb_half4_kernel, prolong_black4_kernel and
// restrict_resid4_kernel, in the same order (in pairs: one instruction rounds
// two sums as two would), so the values are the same bits.
//
// Layout: a thread owns four consecutive entries of two rows (j, j+1) of the
// colour-split level and walks k.  Up to n = 256 the LPR = n/8 threads of a row
// hold all of it (the neighbour past its ends is a boundary node, zero); above,
// a tile holds 32 groups of four and one more on each side.  x-neighbours come
// by a shuffle.  A CTA holds 2W rows, of which 2W - 2 get red values and 2W - 4
// are its output; the planes k-1, k, k+1 of b and k-2, k-1, k of the red values
// lie in the threads' registers, and rows that belong to another pair are read
// from the plane's copy in shared memory, one barrier a plane.  j0 and the
// first plane are odd, so the parity of i in every row is known at compile time
// from the parity of k: no selects.  b and f are fetched kAhead planes ahead
// by asynchronous copies into rings in shared memory (each thread copies what
// it will read itself; b's ring is also the copy that the neighbouring rows
// read): with one plane ahead in registers, half the bytes were in flight and
// a sweep of 257^3 took 36 us.
//
// The residual and its restriction follow two and three planes behind, so such
// a tile loses four rows on each side and holds 24 of them (registers, shared
// memory).
//
// Measured at 257^3 (in brackets the launches replaced): from zero 16.7 us
// (29.4), plain 25.1 (36.3), with the restriction 39.2 (66.5), corrected 28.6
// (52.6), with the red values 30.4 (36.3): a V(2,2) leg pair 110 us (185).
// 513^3: 157 (213), 205 (248), 342 (466), 235 (354), 268 (248).  Eight sets of
// 129^3: 19 (32), 27 (41), 38 (71), 31 (56), 34 (41).  The plain sweep moves its
// 8 bytes a node at 5.4 TB/s; the one with the restriction is bound by its
// instructions, 12 warps an SM.
#include "qumond_internal.h"

#include <type_traits>

namespace qumond {

namespace {

constexpr int kPlain = (int)SweepStart::kBlack, kZero = (int)SweepStart::kZero, kProlong = (int)SweepStart::kCorrected;

struct SweepArgs {
    const float* b;    // black values before (kPlain, kProlong); set s at + s * bset
    long long bset;
    float* out;        // black values after; set s at + s * oset
    long long oset;
    float* red;        // red values after (or null); set s at + s * 2 cs
    const float* f;    // both colours
    const float* ec;   // coarser level, both colours (kProlong)
    float* fc;         // right-hand side of the coarser level, both colours (kRestrict)
    LevelView v, vc;
    float h2, sixth, ih2;
    int tiles;         // tiles along j
    int chunk;         // planes of a chunk (even)
    const SolveState* act;
};

__device__ __forceinline__ float4 zero4() { return make_float4(0.0f, 0.0f, 0.0f, 0.0f); }

__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 lo(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 join(float2 l, float2 h) { return make_float4(l.x, l.y, h.x, h.y); }
// four sums, or four a b + c, in two instructions that round each as the scalar ones do
__device__ __forceinline__ float4 add4(const float4& a, const float4& b)
{
    return join(__fadd2_rn(lo(a), lo(b)), __fadd2_rn(hi(a), hi(b)));
}
__device__ __forceinline__ float4 fma4(const float4& a, float b, const float4& c)
{
    return join(__ffma2_rn(lo(a), two(b), lo(c)), __ffma2_rn(hi(a), two(b), hi(c)));
}
__device__ __forceinline__ float4 mul4(const float4& a, float b)
{
    return join(__fmul2_rn(lo(a), two(b)), __fmul2_rn(hi(a), two(b)));
}

// The sum of the six neighbours of four entries of a row with parity P of i: v the row itself in the other colour, nb
// its entry past the end on the side that P needs, y and z pairs of neighbours.
template <int P>
__device__ __forceinline__ float4 sum6(const float4& v, float nb, const float4& y0, const float4& y1, const float4& z0,
                                       const float4& z1)
{
    const float4 x = make_float4(v.x + (P ? v.y : nb), v.y + (P ? v.z : v.x), v.z + (P ? v.w : v.y),
                                 v.w + (P ? nb : v.z));
    return add4(add4(x, add4(y0, y1)), add4(z0, z1));
}

// (sum - h2 f) / 6, and the residual f - (sum - 6 e) / h2
__device__ __forceinline__ float4 relax4(const float4& sum, const float4& f, float h2, float sixth)
{
    return mul4(fma4(f, -h2, sum), sixth);
}
__device__ __forceinline__ float4 resid4(const float4& sum, const float4& e, const float4& f, float ih2)
{
    return fma4(fma4(e, -6.0f, sum), -ih2, f);
}

constexpr int kThreads = 512, kThreadsRed = 384, kThreadsRestrict = 384, kThreadsSmall = 128;
constexpr int kAhead = 2;               // planes in flight
constexpr int kRingB = kAhead + 2;      // planes of b in shared memory
// What a sweep leaves beside the black values: nothing, the red values, or the residual's restriction.
constexpr int kNothing = (int)SweepAfter::kNothing, kRed = (int)SweepAfter::kRed,
              kRestrict = (int)SweepAfter::kRestrict;
static_assert((kRingB & (kRingB - 1)) == 0, "a plane's place in the ring of b is a mask of its index");
constexpr int kWide = 34;               // threads of a row of a tile above n = 256: 32 groups and one on each side

// Planes of red f in shared memory (the residual of plane k-2 needs f again), of black f, and of all that a tile
// holds there: the rings of b and f, two planes of red values, and for the residual two of the new black values and
// two of residuals (of the odd rows; of both where rows straddle warps).
template <int AFTER>
constexpr int ring_fr() { return kAhead + 1 + (AFTER == kRestrict ? 2 : 0); }
constexpr int kRingFb = kAhead + 1;
template <int LPR, int MODE, int AFTER>
constexpr int smem_planes()
{
    return (MODE == kZero ? 0 : kRingB) + ring_fr<AFTER>() + kRingFb + 2 +
           (AFTER == kRestrict ? 2 + (LPR == kWide ? 2 : 1) : 0);
}
// The most threads of a CTA.  The residual takes about 150 registers (12 warps: with 13 an SM's quarter holds four
// warps of at most 128); sweeps that write both colours, and the tiles along rows,
// measured faster with fewer warps (257^3 with the red values: 30.4 us, 32.1 with 512 threads; 513^3 plain: 206, 225).
template <int LPR, int MODE, int AFTER>
constexpr int most_threads()
{
    return AFTER == kRestrict ? kThreadsRestrict
           : AFTER == kRed || (LPR == kWide && MODE != kProlong) ? kThreadsRed : kThreads;
}
constexpr int kSmem = 227 * 1024;  // shared memory of an SM
// Row pairs of the largest tile.
template <int LPR, int MODE, int AFTER>
constexpr int most_pairs()
{
    constexpr int fit = kSmem / (smem_planes<LPR, MODE, AFTER>() * 2 * LPR * 16);
    constexpr int w = most_threads<LPR, MODE, AFTER>() / LPR;
    return fit < w ? fit : w;
}
template <int AFTER>
constexpr int halo_pairs() { return AFTER == kRestrict ? 2 : 1; }  // row pairs on each side that are no output

// bytes: 16, or 0: the 16 bytes are filled with zeros, nothing is read
__device__ __forceinline__ void copy16(float4* dst, const float* src, int bytes)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

template <int LPR, int MODE, int AFTER>
__global__ void __launch_bounds__(most_threads<LPR, MODE, AFTER>())
sweep_kernel(const SweepArgs a)
{
    extern __shared__ __align__(16) float4 sm[];
    constexpr bool kTiledX = LPR == kWide, RED = AFTER == kRed, RES = AFTER == kRestrict;
    constexpr int kRingFr = ring_fr<AFTER>(), HP = halo_pairs<AFTER>();
    const int set = blockIdx.y;
    if (a.act && !a.act[set].cont) return;  // this set's correction has stopped (the whole CTA)
    const int n = kTiledX ? a.v.n : 8 * LPR;
    const int W = (int)blockDim.x / LPR;          // row pairs of the tile
    const int x = (int)threadIdx.x % LPR;
    const int w = (int)threadIdx.x / LPR;
    const int lane = threadIdx.x & 31;
    const int ty = (int)blockIdx.x % a.tiles, tz = (int)blockIdx.x / a.tiles;
    const int gx = kTiledX ? 32 * (int)blockIdx.z + x - 1 : x;  // entries 4 gx .. 4 gx + 3
    const bool gin = !kTiledX || (gx >= 0 && gx < (n >> 3));
    const bool gout = !kTiledX || (x >= 1 && x <= 32);
    const int j0 = 1 + ty * (2 * W - 4 * HP);     // first output row (odd)
    const int kb = 1 + tz * a.chunk;              // first output plane (odd)
    const int ke = min(kb + a.chunk, n);
    const int klast = RES ? ke + 3 : ke;          // the last step
    const int ja = j0 - 2 * HP + 2 * w;           // this thread's rows ja (odd) and ja + 1
    const bool in0 = gin && ja >= 1 && ja < n, in1 = gin && ja + 1 >= 1 && ja + 1 < n;  // interior rows
    const bool all_in = !kTiledX && j0 - 2 * HP >= 1 && j0 - 2 * HP + 2 * W <= n;  // every row of the tile
    const bool pair_out = w >= HP && w < W - HP;
    const bool out0 = gout && pair_out && in0, out1 = gout && pair_out && in1;
    const int M = kTiledX ? a.v.M : 4 * LPR + 4;
    const long long Q = (long long)M * (n + 1);
    const long long row0 = (long long)ja * M + 4 * gx;  // first entry in row ja of plane 0 of a colour
    const float* const b = MODE == kZero ? nullptr : a.b + set * a.bset + row0;
    const float* const fr = a.f + (long long)set * 2 * a.v.cs + row0;
    const float* const fb = fr + a.v.cs;
    float* const out = a.out + set * a.oset + row0;
    float* const red = RED ? a.red + (long long)set * 2 * a.v.cs + row0 : nullptr;
    const int plane4 = 2 * W * LPR;
    const int at0 = 2 * w * LPR + x;  // row ja of a plane in shared memory; row ja + 1 is LPR further
    float4* const sB = sm + at0;
    float4* const sFr = sm + (MODE == kZero ? 0 : kRingB) * plane4 + at0;
    float4* const sFb = sFr + kRingFr * plane4;
    float4* const sR = sFb + kRingFb * plane4;
    float4* const sN = sR + 2 * plane4;  // the new black values, two planes (RES)
    // residuals, two planes: of row ja (RES), and row ja + 1 beside it where the shuffles need it
    constexpr int kResRow = kTiledX ? 2 * LPR : LPR;
    float4* const sE = sN + 2 * plane4 - at0 + w * kResRow + x;
    const int res4 = W * kResRow;
    const bool up = w > 0, dn = w < W - 1;

    // The asynchronous copies of step k: b(k+1), red f(k), black f(k-1), of the rows that use them; rslot, bslot: the
    // places of f's planes in their rings.  A row outside the level reads nothing (zeros), through a pointer that stays
    // inside f.  The addresses run along with k where registers are free, and are formed from k where they are not
    // (kProlong of 257^3: 28.6 us, 33.0 with running ones; kZero 16.6 and 18.3).
    constexpr bool kRun = MODE == kZero || RES;
    const int ks = kb - (RES ? 3 : 1);  // the first step (even)
    const float* pb0 = in0 && MODE != kZero ? b : a.f;
    const float* pb1 = in1 && MODE != kZero ? b + M : a.f;
    const float* pr = fr;
    const float* pk = fb;
    if (kRun) pb0 += Q * (ks + 1), pb1 += Q * (ks + 1), pr += Q * ks, pk += Q * (ks - 1);
    const int bytes0 = in0 ? 16 : 0, bytes1 = in1 ? 16 : 0;
    const bool fr0 = in0 && up, fr1 = in1 && dn;
    const bool fb0 = RES ? in0 && up && dn : out0, fb1 = RES ? in1 && up && dn : out1;
    auto fetch = [&](int k, int rslot, int bslot) {
        if (MODE != kZero) {
            float4* d = sB + ((k + 1) & (kRingB - 1)) * plane4;
            const bool kin = k + 1 >= 0 && k + 1 <= n && k <= klast;
            const long long o = kRun ? 0 : Q * (k + 1);
            copy16(d, kin ? pb0 + o : a.f, kin ? bytes0 : 0);
            copy16(d + LPR, kin ? pb1 + o : a.f, kin ? bytes1 : 0);
        }
        if (k >= 0 && k <= n && k <= klast) {
            const float* at = pr + (kRun ? 0 : Q * k);
            if (fr0) copy16(sFr + rslot * plane4, at, 16);
            if (fr1) copy16(sFr + rslot * plane4 + LPR, at + M, 16);
        }
        if (k > kb - (RES ? 1 : 0) && k <= n + 1 && k <= klast) {
            const float* at = pk + (kRun ? 0 : Q * (k - 1));
            if (fb0) copy16(sFb + bslot * plane4, at, 16);
            if (fb1) copy16(sFb + bslot * plane4 + LPR, at + M, 16);
        }
        if (kRun) pb0 += Q, pb1 += Q, pr += Q, pk += Q;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the entry past the end of a row: to the right (P = 1) or to the left (P = 0); past the tile's row it is a
    // boundary node, or only reaches entries that are not output
    auto beyond = [&](auto Pc, const float4& v, const float4* srow) {
        constexpr int P = decltype(Pc)::value;
        float nb = P ? __shfl_down_sync(0xffffffffu, v.x, 1) : __shfl_up_sync(0xffffffffu, v.w, 1);
        if (kTiledX) {  // rows straddle warps: from the shared copy
            if (P && lane == 31 && x != LPR - 1) nb = srow[1].x;
            if (!P && lane == 0 && x != 0) nb = srow[-1].w;
        }
        if (P ? x == LPR - 1 : x == 0) nb = 0.0f;
        return nb;
    };

    // --- the coarse-grid correction of b's planes (kProlong) --------------------------------------------------
    // Rows Ja = (ja - 1)/2 and Ja + 1 of two coarse planes, fine plane 2K lying on plane K and fine plane 2K + 1
    // between K and K + 1.  c[0..3]: nodes I = 4 gx .. 4 gx + 3, c[4] the next thread's first.
    float ca[2][5], cb[2][5];
    const int Ja = (ja - 1) >> 1, nc = MODE == kProlong ? a.vc.n : 1;
    const float* const ec = MODE == kProlong ? a.ec + (long long)set * 2 * a.vc.cs : nullptr;
    auto load_coarse = [&](int K, float (&c)[2][5]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int J = Ja + r;
            float2 e = make_float2(0.0f, 0.0f), o = e;
            float last = 0.0f;
            if (MODE == kProlong && gin && J >= 1 && J < nc && K >= 1 && K < nc) {
                const int col = (J + K) & 1;  // colour of the nodes with even I
                const long long at = ((long long)K * (nc + 1) + J) * a.vc.M + 2 * gx;
                const float* A = ec + (long long)col * a.vc.cs + at;
                e = *reinterpret_cast<const float2*>(A);
                o = *reinterpret_cast<const float2*>(ec + (long long)(col ^ 1) * a.vc.cs + at);
                if (kTiledX) last = A[2];
            }
            c[r][0] = e.x, c[r][1] = o.x, c[r][2] = e.y, c[r][3] = o.y, c[r][4] = last;
        }
    };
    auto finish_coarse = [&](float (&c)[2][5]) {  // the next thread's first node; past the row a boundary node
        if (!kTiledX) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float nx = __shfl_down_sync(0xffffffffu, c[r][0], 1);
                c[r][4] = x == LPR - 1 ? 0.0f : nx;
            }
        }
    };
    // adds the correction to the rows of fine plane kk (parity KK), whose coarse planes are c0 and c1
    auto correct = [&](auto KKc, int kk, const float (&c0)[2][5], const float (&c1)[2][5], float4& q0, float4& q1) {
        if (MODE != kProlong || kk < 1 || kk >= n) return;
        constexpr int KK = decltype(KKc)::value;
        constexpr int P0 = KK & 1, P1 = P0 ^ 1;  // parity of i of the black nodes in rows ja (odd), ja + 1
        float r0[4], r1[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float s = (c0[0][e] + c0[0][e + P0]) + (c0[1][e] + c0[1][e + P0]);
            s += (c1[0][e] + c1[0][e + P0]) + (c1[1][e] + c1[1][e + P0]);
            r0[e] = s * 0.125f;
            float t = (c0[1][e] + c0[1][e + P1]) + (c0[1][e] + c0[1][e + P1]);
            t += (c1[1][e] + c1[1][e + P1]) + (c1[1][e] + c1[1][e + P1]);
            r1[e] = t * 0.125f;
        }
        if (in0) q0 = make_float4(P0 == 0 && gx == 0 ? q0.x : q0.x + r0[0], q0.y + r0[1], q0.z + r0[2], q0.w + r0[3]);
        if (in1) q1 = make_float4(P1 == 0 && gx == 0 ? q1.x : q1.x + r1[0], q1.y + r1[1], q1.z + r1[2], q1.w + r1[3]);
    };

    float4 bm0 = zero4(), bm1 = zero4(), bc0 = zero4(), bc1 = zero4(), bp0, bp1;  // b: planes k-1, k, k+1
    float4 rm0 = zero4(), rm1 = zero4(), rc0 = zero4(), rc1 = zero4(), rp0, rp1;  // red: planes k-2, k-1, k
    int fs = 0, gs = 0;  // places of red f(k) and black f(k-1) in their rings
    // RES: the new black values of planes k-2, k-3, the residuals of plane k-3 (rows ja, ja + 1), and of the coarse
    // plane in the making its centre and edge terms (restrict_node's, in its order)
    float4 n20 = zero4(), n21 = zero4(), n30 = zero4(), n31 = zero4(), e0 = zero4(), e1 = zero4();
    float4 um = zero4(), tm = zero4(), edge = zero4(), centre = zero4();
    const int Jc = (ja + 1) >> 1;  // the coarse row on row ja + 1
    const int nh = n >> 1;
    float* const fc = RES ? a.fc + (long long)set * 2 * a.vc.cs : nullptr;
    auto left = [&](const float4& v, const float4* srow) {  // the entry before a group of four
        float l = __shfl_up_sync(0xffffffffu, v.w, 1);
        if (kTiledX && lane == 0 && x != 0) l = srow[-1].w;
        return l;
    };
    auto shifted = [](const float4& v, float l) { return make_float4(l, v.x, v.y, v.z); };

    using Even = std::integral_constant<int, 0>;
    using Odd = std::integral_constant<int, 1>;

    // red values of plane k, black values of plane k-1 (KP: parity of k)
    auto step = [&](auto KPc, int k) {
        constexpr int KP = decltype(KPc)::value;
        // the copies of step k + kAhead go where nothing is read any more: b's place held plane k-1, which the
        // neighbouring rows read before the last barrier, f's held what this thread read in step k-1
        fetch(k + kAhead, (fs + kAhead) % kRingFr, gs == 0 ? kRingFb - 1 : gs - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(kAhead) : "memory");
        if (MODE != kZero) {  // plane k+1 has arrived
            float4* s = sB + ((k + 1) & (kRingB - 1)) * plane4;
            bp0 = s[0], bp1 = s[LPR];
            if (MODE == kProlong) {
                if (KP == 0) correct(Odd{}, k + 1, ca, cb, bp0, bp1);  // k+1 odd: between the two coarse planes
                else correct(Even{}, k + 1, cb, cb, bp0, bp1);         // k+1 even: on the upper one
                s[0] = bp0, s[LPR] = bp1;
                if (KP == 1) {
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int e = 0; e < 5; ++e) ca[r][e] = cb[r][e];
                    load_coarse((k + 1) / 2 + 1, cb);  // used from the next step on
                }
            }
        }
        constexpr int P0 = (1 + KP) & 1, P1 = P0 ^ 1;  // parity of i of the red nodes in rows ja (odd), ja + 1
        using Pa = std::integral_constant<int, P0>;
        using Pb = std::integral_constant<int, P1>;
        const float4 f0 = sFr[fs * plane4], f1 = sFr[fs * plane4 + LPR];
        if (MODE == kZero) {
            rp0 = relax4(zero4(), f0, a.h2, a.sixth);
            rp1 = relax4(zero4(), f1, a.h2, a.sixth);
        } else {
            const float4* s = sB + (k & (kRingB - 1)) * plane4;
            const float4 ym = up ? s[-LPR] : zero4(), yp = dn ? s[2 * LPR] : zero4();
            rp0 = relax4(sum6<P0>(bc0, beyond(Pa{}, bc0, s), ym, bc1, bm0, bp0), f0, a.h2, a.sixth);
            rp1 = relax4(sum6<P1>(bc1, beyond(Pb{}, bc1, s + LPR), bc0, yp, bm1, bp1), f1, a.h2, a.sixth);
        }
        if (!all_in || k < 1 || k >= n) {
            if (!in0 || k < 1 || k >= n) rp0 = zero4();
            if (!in1 || k < 1 || k >= n) rp1 = zero4();
        }
        if (gx == 0) {  // i = 0 is a boundary node
            if (P0 == 0) rp0.x = 0.0f;
            if (P1 == 0) rp1.x = 0.0f;
        }
        {
            float4* s = sR + (k & 1) * plane4;
            s[0] = rp0, s[LPR] = rp1;
        }
        if (RES && k >= kb + 3) {  // the residuals of plane q into the coarse plane
            const int q = k - 3;
            const float4* se = sE + ((k - 1) & 1) * res4;
            const float4 e2 = w + 1 < W ? se[kResRow] : zero4();  // row ja + 2
            if (KP == 1) {  // q even: the plane of the coarse nodes
                centre = e1;
                edge = add4(add4(e2, shifted(e2, left(e2, se + kResRow))), add4(e0, shifted(e0, left(e0, se))));
            } else {
                const float4 u = add4(e1, shifted(e1, left(e1, se + LPR))), t = add4(e2, e0);
                const int K = (q - 1) >> 1;
                if (q >= kb + 2 && gout && pair_out && Jc >= 1 && Jc < nh && K < nh && gin) {
                    const float4 s = add4(add4(edge, add4(u, um)), add4(t, tm));
                    const float c0 = 0.125f * centre.x + 0.03125f * s.x, c1 = 0.125f * centre.y + 0.03125f * s.y;
                    const float c2 = 0.125f * centre.z + 0.03125f * s.z, c3 = 0.125f * centre.w + 0.03125f * s.w;
                    const int col = (Jc + K) & 1;  // colour of the nodes with even I
                    const long long at = ((long long)K * (nh + 1) + Jc) * a.vc.M + 2 * gx;
                    float* A = fc + (long long)col * a.vc.cs + at;
                    if (gx == 0) A[1] = c2;  // I = 0 is a boundary node
                    else *reinterpret_cast<float2*>(A) = make_float2(c0, c2);
                    *reinterpret_cast<float2*>(fc + (long long)(col ^ 1) * a.vc.cs + at) = make_float2(c1, c3);
                }
                um = u, tm = t;
            }
        }
        float4 b0 = zero4(), b1 = zero4();
        if (k > kb - (RES ? 1 : 0)) {  // black values of plane k-1, whose rows have the parities of the red ones of plane k
            const float4* s = sR + ((k - 1) & 1) * plane4;
            const float4 ym = up ? s[-LPR] : zero4(), yp = dn ? s[2 * LPR] : zero4();
            const float4 g0 = sFb[gs * plane4], g1 = sFb[gs * plane4 + LPR];
            b0 = relax4(sum6<P0>(rc0, beyond(Pa{}, rc0, s), ym, rc1, rm0, rp0), g0, a.h2, a.sixth);
            b1 = relax4(sum6<P1>(rc1, beyond(Pb{}, rc1, s + LPR), rc0, yp, rm1, rp1), g1, a.h2, a.sixth);
            if (gx == 0) {
                if (P0 == 0) b0.x = 0.0f;
                if (P1 == 0) b1.x = 0.0f;
            }
            const long long o = Q * (k - 1);
            const bool own = !RES || (k - 1 >= kb && k - 1 < ke);
            if (own && out0) *reinterpret_cast<float4*>(out + o) = b0;
            if (own && out1) *reinterpret_cast<float4*>(out + o + M) = b1;
            if (RES) {
                if (!all_in || k - 1 < 1 || k - 1 >= n) {
                    if (!in0 || k - 1 < 1 || k - 1 >= n) b0 = zero4();
                    if (!in1 || k - 1 < 1 || k - 1 >= n) b1 = zero4();
                }
                float4* d = sN + ((k - 1) & 1) * plane4;
                d[0] = b0, d[LPR] = b1;
            }
            if (RED) {
                if (out0) *reinterpret_cast<float4*>(red + o) = rc0;
                if (out1) *reinterpret_cast<float4*>(red + o + M) = rc1;
            }
        }
        if (RES && k >= kb + 2 && k <= ke + 2) {  // red residuals of plane k-2, rows as those of plane k
            const float4* s = sN + (k & 1) * plane4;
            const float4 ym = up ? s[-LPR] : zero4(), yp = dn ? s[2 * LPR] : zero4();
            const int f2 = (fs + kRingFr - 2) % kRingFr;
            const float4 g0 = sFr[f2 * plane4], g1 = sFr[f2 * plane4 + LPR];
            e0 = resid4(sum6<P0>(n20, beyond(Pa{}, n20, s), ym, n21, n30, b0), rm0, g0, a.ih2);
            e1 = resid4(sum6<P1>(n21, beyond(Pb{}, n21, s + LPR), n20, yp, n31, b1), rm1, g1, a.ih2);
            float4* d = sE + (k & 1) * res4;
            d[0] = e0;
            if (kTiledX) d[LPR] = e1;
        }
        if (RES) n30 = n20, n31 = n21, n20 = b0, n21 = b1;
        bm0 = bc0, bm1 = bc1, bc0 = bp0, bc1 = bp1;
        rm0 = rc0, rm1 = rc1, rc0 = rp0, rc1 = rp1;
        fs = fs == kRingFr - 1 ? 0 : fs + 1;
        gs = gs == kRingFb - 1 ? 0 : gs + 1;
        __syncthreads();
    };

#pragma unroll
    for (int q = 0; q < kAhead; ++q) fetch(ks + q, q, q);
    if (MODE != kZero) {  // planes ks - 1 and ks of b
        auto load = [&](int k, float4& q0, float4& q1) {
            if (k >= 1 && k < n) {
                const float* at = b + Q * k;
                if (in0) q0 = *reinterpret_cast<const float4*>(at);
                if (in1) q1 = *reinterpret_cast<const float4*>(at + M);
            }
        };
        load(ks - 1, bm0, bm1);
        load(ks, bc0, bc1);
        if (MODE == kProlong) {
            load_coarse(ks / 2 - 1, ca);
            load_coarse(ks / 2, cb);
            finish_coarse(ca);
            finish_coarse(cb);
            correct(Odd{}, ks - 1, ca, cb, bm0, bm1);
            correct(Even{}, ks, cb, cb, bc0, bc1);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 5; ++e) ca[r][e] = cb[r][e];
            load_coarse(ks / 2 + 1, cb);
        }
        float4* s = sB + (ks & (kRingB - 1)) * plane4;
        s[0] = bc0, s[LPR] = bc1;
        __syncthreads();
    }
    for (int k = ks;; k += 2) {
        if (MODE == kProlong) finish_coarse(cb);
        step(Even{}, k);
        if (k + 1 > klast) break;
        step(Odd{}, k + 1);
        if (k + 2 > klast) break;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Threads of a CTA, rows of a tile and planes of a chunk.  A tile of 2W rows yields 2W - 4 and a chunk of c planes
// reads c + 4 of b, so large CTAs (512 threads, one on an SM) load and recompute least; they are taken where the
// level fills the GPU with them.  Levels that do not are latency-bound and take CTAs of 128 threads: a plain sweep of
// 129^3 7.2 us instead of 7.5, of 65^3 3.9 instead of 4.9; 257^3 25.7 us with 512 threads, 31.5 with 256.
constexpr long long kLarge = 1 << 20;   // threads that a plane-by-plane pass of the level has work for

// The chunk whose waves of CTAs take the fewest plane steps, each CTA taking its planes and `extra` more (the halo and
// the first loads).
int best_chunk(int rows, long long columns, int slots, int extra)
{
    int best = 2;
    long long cost = -1;
    for (int c = 2; c <= 64; c += 2) {
        const long long ctas = columns * ((rows + c - 1) / c);
        const long long t = (ctas + slots - 1) / slots * (c + extra);
        if (cost < 0 || t < cost) cost = t, best = c;
    }
    return best;
}

template <int LPR, int MODE, int AFTER>
void launch(const SweepArgs& in, cudaStream_t s, const Sets& sets)
{
    static int sms = 0;
    if (sms <= 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
    }
    SweepArgs a = in;
    const int rows = a.v.n - 1;
    constexpr int kWarpPairs = LPR >= 32 ? 1 : 32 / LPR;  // row pairs of a warp: W is a multiple
    constexpr int kHalo = 4 * halo_pairs<AFTER>();        // rows of a tile that are no output
    constexpr int kSmall = AFTER == kRestrict && LPR > 8 ? 2 * kThreadsSmall : kThreadsSmall;
    const int maxw = (long long)rows * rows * (a.v.n / 8) * sets.n >= kLarge ? most_pairs<LPR, MODE, AFTER>()
                                                                             : kSmall / LPR;
    const int xt = LPR == kWide ? a.v.n / 256 : 1;         // tiles along a row
    a.tiles = (rows + 2 * maxw - kHalo - 1) / (2 * maxw - kHalo);
    int W = ((rows + a.tiles - 1) / a.tiles + kHalo + 1) / 2;  // 2W - kHalo >= rows / tiles
    W = (W + kWarpPairs - 1) / kWarpPairs * kWarpPairs;
    const int threads = W * LPR;
    const size_t smem = sizeof(float4) * (size_t)smem_planes<LPR, MODE, AFTER>() * 2 * W * LPR;
    const int per_sm = max(1, min(most_threads<LPR, MODE, AFTER>() / threads, (int)(kSmem / smem)));
    a.chunk = best_chunk(rows, (long long)a.tiles * xt * sets.n, sms * per_sm, AFTER == kRestrict ? 11 : 6);
    const dim3 grid((unsigned)(a.tiles * ((rows + a.chunk - 1) / a.chunk)), (unsigned)sets.n, (unsigned)xt);
    sweep_kernel<LPR, MODE, AFTER><<<grid, threads, smem, s>>>(a);
}

// The forms that a V-cycle uses: each leg has an even number of sweeps, the last of which, a plain one, is followed
// by the restriction or leaves the red values.
template <int LPR>
void launch_mode(const SweepArgs& a, int mode, int after, cudaStream_t s, const Sets& sets)
{
    if (mode == kZero) launch<LPR, kZero, kNothing>(a, s, sets);
    else if (mode == kProlong) launch<LPR, kProlong, kNothing>(a, s, sets);
    else if (after == kRestrict) launch<LPR, kPlain, kRestrict>(a, s, sets);
    else if (after == kRed) launch<LPR, kPlain, kRed>(a, s, sets);
    else launch<LPR, kPlain, kNothing>(a, s, sets);
}

template <int LPR, int MODE, int AFTER>
cudaError_t prepare()
{
    return cudaFuncSetAttribute(sweep_kernel<LPR, MODE, AFTER>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(float4) * smem_planes<LPR, MODE, AFTER>() * 2 * LPR * most_pairs<LPR, MODE, AFTER>()));
}

template <int LPR>
cudaError_t prepare_lpr()
{
    cudaError_t e = prepare<LPR, kPlain, kNothing>();
    if (e == cudaSuccess) e = prepare<LPR, kPlain, kRed>();
    if (e == cudaSuccess) e = prepare<LPR, kPlain, kRestrict>();
    if (e == cudaSuccess) e = prepare<LPR, kZero, kNothing>();
    if (e == cudaSuccess) e = prepare<LPR, kProlong, kNothing>();
    return e;
}

}  // namespace

// From n = 32: four launches of about 4 us a V-cycle where there were ten of 2.5 (33^3 solve: 398 us, 366 so; 24 sets of
// it: about a third less).  Under it a block solves all levels in one launch.
bool sweep_level(int n) { return n >= 32; }

cudaError_t prepare_sweep_level(int n)
{
    if (!sweep_level(n)) return cudaSuccess;
    switch (n) {
    case 32: return prepare_lpr<4>();
    case 64: return prepare_lpr<8>();
    case 128: return prepare_lpr<16>();
    case 256: return prepare_lpr<32>();
    default: return prepare_lpr<kWide>();
    }
}

void launch_sweep(float* e, float* t, const float* f, const LevelView& v, SweepStart start, bool to_t, SweepAfter after,
                  const float* ec, float* fc, const LevelView& vc, double h, cudaStream_t s, const Sets& sets)
{
    SweepArgs a{};
    float* eb = e + v.cs;
    a.b = to_t ? eb : t;
    a.bset = to_t ? 2 * v.cs : v.cs;
    a.out = to_t ? t : eb;
    a.oset = to_t ? v.cs : 2 * v.cs;
    a.red = e;
    a.f = f;
    a.ec = ec;
    a.fc = fc;
    a.v = v;
    a.vc = vc;
    a.h2 = (float)(h * h);
    a.sixth = 1.0f / 6.0f;
    a.ih2 = (float)(1.0 / (h * h));
    a.act = sets.act;
    const int mode = (int)start;
    switch (v.n) {
    case 32: launch_mode<4>(a, mode, (int)after, s, sets); break;
    case 64: launch_mode<8>(a, mode, (int)after, s, sets); break;
    case 128: launch_mode<16>(a, mode, (int)after, s, sets); break;
    case 256: launch_mode<32>(a, mode, (int)after, s, sets); break;
    default: launch_mode<kWide>(a, mode, (int)after, s, sets); break;
    }
}

}  // namespace qumond
