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
// the two change roles from sweep to sweep.  The red values are written (2
// more) only where something reads them: before the restriction of the
// residual and after the last sweep.  With PROLONG the sweep starts from
// b + P e_c, the coarse-grid correction applied as the planes are loaded.
//
// Every node's arithmetic is rb_half4_kernel's (and prolong_black4_kernel's),
// in the same order, so the values are the same bits.
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
// Measured at 257^3 (two launches of the half-sweeps, with the prolongation
// where there is one, before): plain 25.7 us (36.2), with the red values written
// 31.7, from zero 16.8 (29.3), corrected 29.2 (52.9).  513^3: 211 (248), 145
// (213), 247 (354).  Eight sets of 129^3: 27 (41), 18 (32), 31 (56).  The
// memory system bounds them (8 bytes a node in 25.7 us: 5.3 TB/s).
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
    LevelView v, vc;
    float h2, sixth;
    int tiles;         // tiles along j
    int chunk;         // planes of a chunk (even)
    const SolveState* act;
};

__device__ __forceinline__ float4 zero4() { return make_float4(0.0f, 0.0f, 0.0f, 0.0f); }

// (sum of the six neighbours - h2 f) / 6 for four entries of a row with parity P of i: v the row itself in the
// other colour, nb its entry past the end on the side that P needs, y and z pairs of neighbours.
template <int P>
__device__ __forceinline__ float4 relax4(const float4& v, float nb, const float4& y0, const float4& y1,
                                         const float4& z0, const float4& z1, const float4& f, float h2, float sixth)
{
    const float o0 = P ? v.y : nb, o1 = P ? v.z : v.x, o2 = P ? v.w : v.y, o3 = P ? nb : v.z;
    const float s0 = (v.x + o0) + (y0.x + y1.x) + (z0.x + z1.x);
    const float s1 = (v.y + o1) + (y0.y + y1.y) + (z0.y + z1.y);
    const float s2 = (v.z + o2) + (y0.z + y1.z) + (z0.z + z1.z);
    const float s3 = (v.w + o3) + (y0.w + y1.w) + (z0.w + z1.w);
    return make_float4((s0 - h2 * f.x) * sixth, (s1 - h2 * f.y) * sixth, (s2 - h2 * f.z) * sixth,
                       (s3 - h2 * f.w) * sixth);
}

constexpr int kAhead = 2;               // planes in flight
constexpr int kRingB = kAhead + 2, kRingF = kAhead + 1;
static_assert((kRingB & (kRingB - 1)) == 0, "a plane's place in the ring of b is a mask of its index");
constexpr int kWide = 34;               // threads of a row of a tile above n = 256: 32 groups and one on each side

// planes of a tile in shared memory: rings of b and of both colours of f, two planes of red values
template <int MODE>
constexpr int smem_planes() { return (MODE == kZero ? 0 : kRingB) + 2 * kRingF + 2; }

__device__ __forceinline__ void copy16(float4* dst, const float* src, bool valid)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = valid ? 16 : 0;  // 0: the 16 bytes are filled with zeros, nothing is read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

template <int LPR, int MODE, bool RED>
__global__ void __launch_bounds__(512)
sweep_kernel(const SweepArgs a)
{
    extern __shared__ __align__(16) float4 sm[];
    constexpr bool kTiledX = LPR == kWide;
    const int set = blockIdx.y;
    if (a.act && !a.act[set].cont) return;  // this set's correction has stopped (the whole CTA)
    const int n = a.v.n;
    const int W = (int)blockDim.x / LPR;          // row pairs of the tile
    const int x = (int)threadIdx.x % LPR;
    const int w = (int)threadIdx.x / LPR;
    const int lane = threadIdx.x & 31;
    const int ty = (int)blockIdx.x % a.tiles, tz = (int)blockIdx.x / a.tiles;
    const int gx = kTiledX ? 32 * (int)blockIdx.z + x - 1 : x;  // entries 4 gx .. 4 gx + 3
    const bool gin = !kTiledX || (gx >= 0 && gx < (n >> 3));
    const bool gout = !kTiledX || (x >= 1 && x <= 32);
    const int j0 = 1 + ty * (2 * W - 4);          // first output row (odd)
    const int kb = 1 + tz * a.chunk;              // first output plane (odd)
    const int ke = min(kb + a.chunk, n);
    const int ja = j0 - 2 + 2 * w;                // this thread's rows ja (odd) and ja + 1
    const bool in0 = gin && ja >= 1 && ja < n, in1 = gin && ja + 1 >= 1 && ja + 1 < n;  // interior rows
    const bool pair_out = w >= 1 && w < W - 1;
    const bool out0 = gout && pair_out && in0, out1 = gout && pair_out && in1;
    const int M = a.v.M;
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
    float4* const sFb = sFr + kRingF * plane4;
    float4* const sR = sFb + kRingF * plane4;
    const bool up = w > 0, dn = w < W - 1;

    // the asynchronous copies of step k: b(k+1), red f(k), black f(k-1), of the rows that use them; `fslot`: k's place
    // in the rings of f
    auto fetch = [&](int k, int fslot) {
        if (MODE != kZero) {
            const bool kin = k + 1 >= 1 && k + 1 < n && k + 1 <= ke + 1;
            float4* d = sB + ((k + 1) & (kRingB - 1)) * plane4;
            const float* at = b + Q * (k + 1);
            copy16(d, kin && in0 ? at : a.f, kin && in0);
            copy16(d + LPR, kin && in1 ? at + M : a.f, kin && in1);
        }
        if (k >= 1 && k < n && k <= ke) {
            const float* at = fr + Q * k;
            if (in0 && up) copy16(sFr + fslot * plane4, at, true);
            if (in1 && dn) copy16(sFr + fslot * plane4 + LPR, at + M, true);
        }
        if (k - 1 >= kb && k - 1 < ke) {
            const float* at = fb + Q * (k - 1);
            if (out0) copy16(sFb + fslot * plane4, at, true);
            if (out1) copy16(sFb + fslot * plane4 + LPR, at + M, true);
        }
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
    int fs = 0;  // place of k in the rings of f

    using Even = std::integral_constant<int, 0>;
    using Odd = std::integral_constant<int, 1>;

    // red values of plane k, black values of plane k-1 (KP: parity of k)
    auto step = [&](auto KPc, int k) {
        constexpr int KP = decltype(KPc)::value;
        // the copies of step k + kAhead go where nothing is read any more: b's place held plane k-1, which the
        // neighbouring rows read before the last barrier, f's held what this thread read in step k-1
        fetch(k + kAhead, fs == 0 ? kRingF - 1 : fs - 1);
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
            const float z = 0.0f;
            rp0 = make_float4((z - a.h2 * f0.x) * a.sixth, (z - a.h2 * f0.y) * a.sixth, (z - a.h2 * f0.z) * a.sixth,
                              (z - a.h2 * f0.w) * a.sixth);
            rp1 = make_float4((z - a.h2 * f1.x) * a.sixth, (z - a.h2 * f1.y) * a.sixth, (z - a.h2 * f1.z) * a.sixth,
                              (z - a.h2 * f1.w) * a.sixth);
        } else {
            const float4* s = sB + (k & (kRingB - 1)) * plane4;
            const float4 ym = up ? s[-LPR] : zero4(), yp = dn ? s[2 * LPR] : zero4();
            rp0 = relax4<P0>(bc0, beyond(Pa{}, bc0, s), ym, bc1, bm0, bp0, f0, a.h2, a.sixth);
            rp1 = relax4<P1>(bc1, beyond(Pb{}, bc1, s + LPR), bc0, yp, bm1, bp1, f1, a.h2, a.sixth);
        }
        const bool kin = k >= 1 && k < n;
        if (!(kin && in0)) rp0 = zero4();
        if (!(kin && in1)) rp1 = zero4();
        if (gx == 0) {  // i = 0 is a boundary node
            if (P0 == 0) rp0.x = 0.0f;
            if (P1 == 0) rp1.x = 0.0f;
        }
        {
            float4* s = sR + (k & 1) * plane4;
            s[0] = rp0, s[LPR] = rp1;
        }
        if (k > kb) {  // black values of plane k-1, whose rows have the parities of the red ones of plane k
            const float4* s = sR + ((k - 1) & 1) * plane4;
            const float4 ym = up ? s[-LPR] : zero4(), yp = dn ? s[2 * LPR] : zero4();
            const float4 g0 = sFb[fs * plane4], g1 = sFb[fs * plane4 + LPR];
            float4 b0 = relax4<P0>(rc0, beyond(Pa{}, rc0, s), ym, rc1, rm0, rp0, g0, a.h2, a.sixth);
            float4 b1 = relax4<P1>(rc1, beyond(Pb{}, rc1, s + LPR), rc0, yp, rm1, rp1, g1, a.h2, a.sixth);
            if (gx == 0) {
                if (P0 == 0) b0.x = 0.0f;
                if (P1 == 0) b1.x = 0.0f;
            }
            const long long o = Q * (k - 1);
            if (out0) *reinterpret_cast<float4*>(out + o) = b0;
            if (out1) *reinterpret_cast<float4*>(out + o + M) = b1;
            if (RED) {
                if (out0) *reinterpret_cast<float4*>(red + o) = rc0;
                if (out1) *reinterpret_cast<float4*>(red + o + M) = rc1;
            }
        }
        bm0 = bc0, bm1 = bc1, bc0 = bp0, bc1 = bp1;
        rm0 = rc0, rm1 = rc1, rc0 = rp0, rc1 = rp1;
        fs = fs == kRingF - 1 ? 0 : fs + 1;
        __syncthreads();
    };

    const int ks = kb - 1;  // the first step (even)
#pragma unroll
    for (int q = 0; q < kAhead; ++q) fetch(ks + q, q);
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
        if (k + 1 > ke) break;
        step(Odd{}, k + 1);
        if (k + 2 > ke) break;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// Threads of a CTA, rows of a tile and planes of a chunk.  A tile of 2W rows yields 2W - 4 and a chunk of c planes
// reads c + 4 of b, so large CTAs (512 threads, one on an SM) load and recompute least; they are taken where the
// level fills the GPU with them.  Levels that do not are latency-bound and take CTAs of 128 threads: a plain sweep of
// 129^3 7.2 us instead of 7.5, of 65^3 3.9 instead of 4.9; 257^3 25.7 us with 512 threads, 31.5 with 256.
constexpr int kThreads = 512, kThreadsSmall = 128;
constexpr long long kLarge = 1 << 20;   // threads that a plane-by-plane pass of the level has work for
constexpr size_t kSmem = 227 * 1024;    // shared memory of an SM

// The chunk whose waves of CTAs take the fewest plane steps, each CTA taking its planes and about six more (the halo
// and the first loads).
int best_chunk(int rows, long long columns, int slots)
{
    int best = 2;
    long long cost = -1;
    for (int c = 2; c <= 64; c += 2) {
        const long long ctas = columns * ((rows + c - 1) / c);
        const long long t = (ctas + slots - 1) / slots * (c + 6);
        if (cost < 0 || t < cost) cost = t, best = c;
    }
    return best;
}

template <int LPR, int MODE, bool RED>
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
    const int maxw = ((long long)rows * rows * (a.v.n / 8) * sets.n >= kLarge ? kThreads : kThreadsSmall) / LPR;
    const int xt = LPR == kWide ? a.v.n / 256 : 1;         // tiles along a row
    a.tiles = (rows + 2 * maxw - 5) / (2 * maxw - 4);
    int W = ((rows + a.tiles - 1) / a.tiles + 5) / 2;      // 2W - 4 >= rows / tiles
    W = (W + kWarpPairs - 1) / kWarpPairs * kWarpPairs;
    const int threads = W * LPR;
    const size_t smem = sizeof(float4) * (size_t)smem_planes<MODE>() * 2 * W * LPR;
    const int per_sm = max(1, min(512 / threads, (int)(kSmem / smem)));
    a.chunk = best_chunk(rows, (long long)a.tiles * xt * sets.n, sms * per_sm);
    const dim3 grid((unsigned)(a.tiles * ((rows + a.chunk - 1) / a.chunk)), (unsigned)sets.n, (unsigned)xt);
    sweep_kernel<LPR, MODE, RED><<<grid, threads, smem, s>>>(a);
}

// The forms that a V-cycle uses: a leg of an even number of sweeps writes the red values in its last one, which is
// a plain one.
template <int LPR>
void launch_mode(const SweepArgs& a, int mode, bool red, cudaStream_t s, const Sets& sets)
{
    if (mode == kZero) launch<LPR, kZero, false>(a, s, sets);
    else if (mode == kProlong) launch<LPR, kProlong, false>(a, s, sets);
    else if (red) launch<LPR, kPlain, true>(a, s, sets);
    else launch<LPR, kPlain, false>(a, s, sets);
}

template <int LPR, int MODE, bool RED>
cudaError_t prepare()
{
    return cudaFuncSetAttribute(sweep_kernel<LPR, MODE, RED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(sizeof(float4) * smem_planes<MODE>() * 2 * kThreads));
}

template <int LPR>
cudaError_t prepare_lpr()
{
    cudaError_t e = prepare<LPR, kPlain, false>();
    if (e == cudaSuccess) e = prepare<LPR, kPlain, true>();
    if (e == cudaSuccess) e = prepare<LPR, kZero, false>();
    if (e == cudaSuccess) e = prepare<LPR, kProlong, false>();
    return e;
}

}  // namespace

bool sweep_level(int n) { return n >= 64; }

cudaError_t prepare_sweep_level(int n)
{
    if (!sweep_level(n)) return cudaSuccess;
    switch (n) {
    case 64: return prepare_lpr<8>();
    case 128: return prepare_lpr<16>();
    case 256: return prepare_lpr<32>();
    default: return prepare_lpr<kWide>();
    }
}

void launch_sweep(float* e, float* t, const float* f, const LevelView& v, SweepStart start, bool to_t, bool red,
                  const float* ec, const LevelView& vc, double h, cudaStream_t s, const Sets& sets)
{
    SweepArgs a{};
    float* eb = e + v.cs;
    a.b = to_t ? eb : t;
    a.bset = to_t ? 2 * v.cs : v.cs;
    a.out = to_t ? t : eb;
    a.oset = to_t ? v.cs : 2 * v.cs;
    a.red = red ? e : nullptr;
    a.f = f;
    a.ec = ec;
    a.v = v;
    a.vc = vc;
    a.h2 = (float)(h * h);
    a.sixth = 1.0f / 6.0f;
    a.act = sets.act;
    const int mode = (int)start;
    switch (v.n) {
    case 64: launch_mode<8>(a, mode, red, s, sets); break;
    case 128: launch_mode<16>(a, mode, red, s, sets); break;
    case 256: launch_mode<32>(a, mode, red, s, sets); break;
    default: launch_mode<kWide>(a, mode, red, s, sets); break;
    }
}

}  // namespace qumond
