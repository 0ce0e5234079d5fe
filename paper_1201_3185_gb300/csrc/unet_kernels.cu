// Kernels of the learned initial guess: a 3-D U-Net (3^3 convolutions, BF16
// activations and weights, FP32 accumulation) that maps (rho, Phi_N) of a box
// to Phi - Phi_N, the starting point of the QUMOND solve (Eq. 2) in place of
// FMG.  Activations are channels-last: voxel v = (z*S + y)*S + x of an S^3
// level holds its channels contiguously, with a row stride `ld` (>= the
// channel count) so that a layer can write into a slice of a concatenation.
//
// The 3^3 convolutions are implicit GEMMs on the tensor cores: M = output
// voxels (a CTA owns a brick of up to 128 voxels), N = output channels, K =
// 27 taps x input channels, in chunks of 16 channels.  A chunk's input brick
// with its one-voxel halo and the chunk's weights are staged in shared memory;
// each warp owns 16 voxels and issues m16n8k16 BF16 MMAs with FP32
// accumulators.  The weight gradient is the same contraction with K = voxels
// (both operands staged transposed), reduced over CTAs in a fixed order.
#include "unet_internal.h"

#include <cstring>

#include <cuda_bf16.h>

namespace qumond {
namespace unet {

namespace {

constexpr int kHaloMax = 432;     // (2+2) x (4+2) x (16+2) voxels: the largest brick halo
constexpr int kHaloStride = 24;   // bf16 per halo voxel: 16 channels + 8 padding (conflict-free A fragments)
constexpr int kWRow = 440;        // bf16 per output channel of a weight chunk: 27 x 16 + 8 padding

__device__ __forceinline__ unsigned lds32(const __nv_bfloat16* p) { return *reinterpret_cast<const unsigned*>(p); }

__device__ __forceinline__ void mma16816(float* d, const unsigned* a, unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<unsigned*>(&v);
}

__device__ __forceinline__ void brick_coords(const Brick& b, int l, int& lz, int& ly, int& lx)
{
    lx = l % b.bx;
    ly = (l / b.bx) % b.by;
    lz = l / (b.bx * b.by);
}

}  // namespace

// ---------------------------------------------------------------------------
// y[v, co] = act( bias[co] + sum_{tap, ci} x[v + off(tap), ci] W[co][tap][ci] ) * (mask[v, co] > 0)
// with zero padding outside the S^3 level; tap = (dz+1)*9 + (dy+1)*3 + (dx+1).
// NTILES = output channels per CTA / 8.  grid = (bricks, Cout / (8 NTILES)).
// The chunks of 16 input channels come by cp.async into a ring of a.stages
// buffers (a load at a time by each thread, a chunk's staging was a chain of
// nine global latencies, 6 us; 128 -> 128 channels at 8^3: 43 -> 23 us).
template <int NTILES>
__global__ void __launch_bounds__(256) conv3_kernel(ConvArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NT = NTILES * 8;
    constexpr int kStage = kHaloMax * kHaloStride + NT * kWRow;  // bf16 of a buffer: halo, weights

    const Brick b = a.brick;
    const int S = a.S;
    const int nbx = S / b.bx, nby = S / b.by;
    const int brick = blockIdx.x;
    const int x0 = (brick % nbx) * b.bx, y0 = ((brick / nbx) % nby) * b.by, z0 = (brick / (nbx * nby)) * b.bz;
    const int co0 = blockIdx.y * NT;
    const int hx = b.bx + 2, hy = b.by + 2, hz = b.bz + 2;
    const int hv_count = hx * hy * hz;
    const int nvox = b.bx * b.by * b.bz;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    const bool warp_on = warp * 16 < nvox;
    // the two rows (voxels) of this thread in the warp's m16 tile
    const int l0 = warp * 16 + g, l1 = l0 + 8;
    const bool v0ok = l0 < nvox, v1ok = l1 < nvox;
    int hc0 = 0, hc1 = 0;  // halo index of the voxel itself (tap 13)
    {
        int lz, ly, lx;
        brick_coords(b, v0ok ? l0 : 0, lz, ly, lx);
        hc0 = ((lz + 1) * hy + (ly + 1)) * hx + (lx + 1);
        brick_coords(b, v1ok ? l1 : 0, lz, ly, lx);
        hc1 = ((lz + 1) * hy + (ly + 1)) * hx + (lx + 1);
    }

    float acc[NTILES][4];
#pragma unroll
    for (int j = 0; j < NTILES; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;

    const int nchunks = a.cin / 16;
    auto stage = [&](int chunk) {
        if (chunk < nchunks) {
            const int ci0 = chunk * 16;
            __nv_bfloat16* halo = reinterpret_cast<__nv_bfloat16*>(smem_raw) + (chunk % a.stages) * kStage;
            __nv_bfloat16* wsm = halo + kHaloMax * kHaloStride;
            // the input brick + halo, 16 channels (two 16-byte pieces per voxel)
            for (int q = threadIdx.x; q < hv_count * 2; q += blockDim.x) {
                const int hv = q >> 1, part = q & 1;
                const int ix = hv % hx, iy = (hv / hx) % hy, iz = hv / (hx * hy);
                const int gx = x0 + ix - 1, gy = y0 + iy - 1, gz = z0 + iz - 1;
                const bool in = gx >= 0 && gx < S && gy >= 0 && gy < S && gz >= 0 && gz < S;
                const long long v = in ? ((long long)gz * S + gy) * S + gx : 0;
                cp_async16(halo + hv * kHaloStride + part * 8, a.in + v * a.ld_in + a.in_off + ci0 + part * 8, in);
            }
            // the weight chunk: W[co0 + n][tap][ci0 .. ci0+15]
            for (int q = threadIdx.x; q < NT * 27 * 2; q += blockDim.x) {
                const int part = q & 1, t = (q >> 1) % 27, n = (q >> 1) / 27;
                cp_async16(wsm + n * kWRow + t * 16 + part * 8,
                           a.w + ((long long)(co0 + n) * 27 + t) * a.cin + ci0 + part * 8, true);
            }
        }
        cp_async_commit();  // a group a chunk, empty past the last
    };
    const int ahead = a.stages - 1;
    for (int c = 0; c < ahead; ++c) stage(c);
    for (int c = 0; c < nchunks; ++c) {
        if (ahead == 0) stage(c);
        cp_async_wait(ahead > 1 ? ahead - 1 : 0);  // chunk c has landed
        __syncthreads();
        if (ahead > 0) stage(c + ahead);  // over chunk c - 1, which every warp has left
        const __nv_bfloat16* halo = reinterpret_cast<const __nv_bfloat16*>(smem_raw) + (c % a.stages) * kStage;
        const __nv_bfloat16* wsm = halo + kHaloMax * kHaloStride;
        if (warp_on) {
#pragma unroll 1
            for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
            for (int r = 0; r < 9; ++r) {
                const int t = (dz + 1) * 9 + r;
                const int off = (dz * hy + r / 3 - 1) * hx + r % 3 - 1;
                const __nv_bfloat16* r0 = halo + (hc0 + off) * kHaloStride + tig * 2;
                const __nv_bfloat16* r1 = halo + (hc1 + off) * kHaloStride + tig * 2;
                unsigned af[4];
                af[0] = lds32(r0);
                af[1] = lds32(r1);
                af[2] = lds32(r0 + 8);
                af[3] = lds32(r1 + 8);
#pragma unroll
                for (int j = 0; j < NTILES; ++j) {
                    const __nv_bfloat16* wp = wsm + (j * 8 + g) * kWRow + t * 16 + tig * 2;
                    mma16816(acc[j], af, lds32(wp), lds32(wp + 8));
                }
            }
        }
        if (ahead == 0) __syncthreads();
    }
    if (!warp_on) return;
    // epilogue: bias, ReLU, mask, BF16 store
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int l = half ? l1 : l0;
        if (l >= nvox) continue;
        int lz, ly, lx;
        brick_coords(b, l, lz, ly, lx);
        const long long v = ((long long)(z0 + lz) * S + (y0 + ly)) * S + (x0 + lx);
#pragma unroll
        for (int j = 0; j < NTILES; ++j) {
            const int co = co0 + j * 8 + tig * 2;
            float r0 = acc[j][half * 2], r1 = acc[j][half * 2 + 1];
            if (a.bias) {
                r0 += a.bias[co];
                r1 += a.bias[co + 1];
            }
            if (a.relu) {
                r0 = fmaxf(r0, 0.0f);
                r1 = fmaxf(r1, 0.0f);
            }
            if (a.mask) {
                const __nv_bfloat16* mp = a.mask + v * a.ld_mask + a.mask_off + co;
                if (!(__bfloat162float(mp[0]) > 0.0f)) r0 = 0.0f;
                if (!(__bfloat162float(mp[1]) > 0.0f)) r1 = 0.0f;
            }
            *reinterpret_cast<unsigned*>(a.out + v * a.ld_out + a.out_off + co) = pack_bf16(r0, r1);
        }
    }
}

Brick brick_for(int S)
{
    // 128 voxels where the level allows (two planes of 4 rows of 16), else the whole level
    Brick b;
    if (S % 16 == 0) {
        b.bz = 2, b.by = 4, b.bx = 16;
    } else if (S == 8) {
        b.bz = 2, b.by = 8, b.bx = 8;
    } else if (S <= 4) {
        b.bz = S, b.by = S, b.bx = S;  // S = 4: 64 voxels; S = 2: 8
    } else {
        // the coarse levels of a size that is no power of two (24, 12 and 6 of 48): the most voxels, up to 128, of a
        // brick that divides the level and whose halo fits its buffer
        b.bz = b.by = b.bx = 1;
        for (int z = 1; z <= S; ++z)
            for (int y = 1; y <= S && z * y <= 128; ++y)
                for (int x = 1; x <= S && z * y * x <= 128; ++x)
                    if (S % z == 0 && S % y == 0 && S % x == 0 && (z + 2) * (y + 2) * (x + 2) <= kHaloMax &&
                        z * y * x > b.bz * b.by * b.bx)
                        b.bz = z, b.by = y, b.bx = x;
    }
    return b;
}

size_t conv3_smem_bytes(int cout_tile)
{
    return (size_t)kHaloMax * kHaloStride * 2 + (size_t)cout_tile * kWRow * 2;
}

// The widest tile of output channels that still gives every multiprocessor a
// block, down to 16: the levels of 16^3 and 8^3 voxels have 32 and 4 bricks, and
// at 64 channels a tile 32 and 8 blocks ran on 152 multiprocessors (192 -> 64
// channels at 16^3: 101 us, 82 us with 16; 128 -> 128 at 8^3: 73 us, 43 us; before
// the ring of chunks).  An
// output channel's sums do not depend on the tile.
int conv3_tile(int cout, int bricks, int sms)
{
    const int tiles[3] = {64, 48, 32};
    for (int t : tiles)
        if (cout % t == 0 && (long long)bricks * (cout / t) >= sms) return t;
    return 16;
}

// Buffers of a chunk ring: the shared memory of a multiprocessor divided among
// the blocks it gets, at least one buffer each (many blocks hide one another's
// loads; a single block needs its next chunks in flight), at most four.
int conv3_stages(size_t stage_bytes, int blocks, int chunks, int sms)
{
    const int per_sm = (blocks + sms - 1) / sms;
    int stages = (int)(kConvSmem / (per_sm * (stage_bytes + 2048)));  // 1 KB a block is the system's; static arrays
    if (stages > chunks) stages = chunks;
    if (stages > kConvStages) stages = kConvStages;
    return stages < 1 ? 1 : stages;
}

template <int NTILES>
static void launch_conv3_t(ConvArgs a, int bricks, cudaStream_t s)
{
    const int nt = NTILES * 8;
    const int blocks = bricks * (a.cout / nt);
    a.stages = conv3_stages(conv3_smem_bytes(nt), blocks, a.cin / 16, a.sms);
    conv3_kernel<NTILES><<<dim3(bricks, a.cout / nt), 256, a.stages * conv3_smem_bytes(nt), s>>>(a);
}

void prepare_conv3()
{
    const int tiles[4] = {16, 32, 48, 64};
    for (int t : tiles) {
        const int smem = (int)conv3_smem_max(conv3_smem_bytes(t));
        if (t == 16) cudaFuncSetAttribute(conv3_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (t == 32) cudaFuncSetAttribute(conv3_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (t == 48) cudaFuncSetAttribute(conv3_kernel<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (t == 64) cudaFuncSetAttribute(conv3_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    }
}

void launch_conv3(ConvArgs a, cudaStream_t s)
{
    if (conv3_tc_applies(a)) {
        launch_conv3_tc(a, s);
        return;
    }
    a.brick = brick_for(a.S);
    const int bricks = (a.S / a.brick.bx) * (a.S / a.brick.by) * (a.S / a.brick.bz);
    switch (conv3_tile(a.cout, bricks, a.sms)) {
    case 64: launch_conv3_t<8>(a, bricks, s); break;
    case 48: launch_conv3_t<6>(a, bricks, s); break;
    case 32: launch_conv3_t<4>(a, bricks, s); break;
    default: launch_conv3_t<2>(a, bricks, s); break;
    }
}

// ---------------------------------------------------------------------------
// Weight gradient: part[blk][co][tap][ci] = sum over the CTA's voxels of
// g[v, co0+co] x[v + off(tap), ci0+ci], for a tile of 16 MT output channels
// and 16 input channels; grid = (vblocks, cout/(16 MT), cin/16).  Warp w takes
// taps w, w+8, w+16, w+24.  The k-dimension is the voxels, while memory holds
// channels contiguous: both operands are staged as they lie in memory, one row
// of 16 MT (or 16) channels per voxel, and ldmatrix transposes 8 x 8 tiles on
// the way to the registers; it takes an address per row, so a tap is an offset
// of the rows in the halo.  (Staged transposed, with three shifted copies of
// the halo in two-byte stores, a brick took 10 us: 273 us for 48 -> 16 channels
// at 64^3, 53 us now, 155 without bricks in flight and with
// the voxels' offsets worked out anew in every brick.)
constexpr int kWgradStages = 3;  // 2 blocks of 3 x 31 KB on a multiprocessor
constexpr int kXRow = 24;  // bf16 of a halo voxel: 16 channels and 8 of padding (8 rows meet all 32 banks)

__device__ __forceinline__ void ldmatrix4_trans(unsigned (&r)[4], const __nv_bfloat16* row)
{
    const unsigned at = (unsigned)__cvta_generic_to_shared(row);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(at)
                 : "memory");
}

template <int MT>
__global__ void __launch_bounds__(256) wgrad_kernel(WgradArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Brick b = a.brick;
    const int S = a.S;
    const int nvox = b.bx * b.by * b.bz;
    constexpr int kGRow = 16 * MT + 8;                     // bf16 of a voxel's gradients, with padding
    const int hx = b.bx + 2, hy = b.by + 2, hz = b.bz + 2;
    const int ring = 128 * kGRow + hx * hy * hz * kXRow;   // bf16 of a buffer: the gradients, the brick's halo
    __nv_bfloat16* const smem = reinterpret_cast<__nv_bfloat16*>(smem_raw);

    const int nbx = S / b.bx, nby = S / b.by;
    const int nbricks = nbx * nby * (S / b.bz);
    const int co0 = blockIdx.y * 16 * MT, ci0 = blockIdx.z * 16;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    const int ntap = warp < 3 ? 4 : 3;  // taps warp, warp+8, warp+16 (, warp+24)
    // the row that this lane addresses in each 16-voxel step: of the gradients, tiles (voxels 0-7, 8-15) x (channels
    // 0-7, 8-15) in the order of the A fragment; of the halo in that of two B fragments
    const int rv = lane & 7, mat = lane >> 3;
    const int grow0 = (rv + (mat >> 1) * 8) * kGRow + (mat & 1) * 8;
    const int xv = rv + (mat & 1) * 8, xc = (mat >> 1) * 8;
    int toff[4];  // the taps' offsets in the halo
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int t = warp + 8 * q;
        toff[q] = (((t / 9 - 1) * hy + ((t / 3) % 3 - 1)) * hx + (t % 3 - 1)) * kXRow;
    }

    float acc[4][MT][2][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 2; ++j) acc[q][m][j][0] = acc[q][m][j][1] = acc[q][m][j][2] = acc[q][m][j][3] = 0.0f;

    // this thread's pieces (8 channels of a voxel) of the gradients and of the halo, and its voxel of each 16-voxel
    // step, by their offsets in a brick: the divisions once, not in every brick
    constexpr int kPieces = (2 * kHaloMax + 255) / 256;
    int gvox[MT], hvox[kPieces], xstep[8];  // gvox: offset in the level; hvox: x | y << 8 | z << 16 (-1: no piece)
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        const int l = (threadIdx.x + 256 * i) / (2 * MT);
        int lz, ly, lx;
        brick_coords(b, l < nvox ? l : 0, lz, ly, lx);
        gvox[i] = l < nvox ? (lz * S + ly) * S + lx : -1;
    }
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
        const int hv = (threadIdx.x + 256 * i) >> 1;
        hvox[i] = hv < hx * hy * hz ? (hv % hx) | ((hv / hx) % hy) << 8 | hv / (hx * hy) << 16 : -1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int l = i * 16 + xv;
        int lz, ly, lx;
        brick_coords(b, l < nvox ? l : 0, lz, ly, lx);  // past nvox any voxel: its gradients are zero
        xstep[i] = (((lz + 1) * hy + (ly + 1)) * hx + (lx + 1)) * kXRow + xc;
    }
    // a brick's operands by cp.async, two bricks ahead
    auto stage = [&](int brick, int slot) {
        if (brick < nbricks) {
            __nv_bfloat16* const gs = smem + slot * ring;
            __nv_bfloat16* const xs = gs + 128 * kGRow;
            const int x0 = (brick % nbx) * b.bx, y0 = ((brick / nbx) % nby) * b.by, z0 = (brick / (nbx * nby)) * b.bz;
            const long long v0 = ((long long)z0 * S + y0) * S + x0;
            // 16 MT channels of nvox voxels (voxels past nvox are zero)
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                const int piece = threadIdx.x + 256 * i, l = piece / (2 * MT), part = piece % (2 * MT);
                const bool in = gvox[i] >= 0;
                cp_async16(gs + l * kGRow + part * 8, a.g + (v0 + (in ? gvox[i] : 0)) * a.ld_g + a.g_off + co0 + part * 8,
                           in);
            }
#pragma unroll
            for (int i = 0; i < kPieces; ++i) {
                if (hvox[i] < 0) continue;
                const int piece = threadIdx.x + 256 * i, part = piece & 1;
                const int gx = x0 + (hvox[i] & 255) - 1, gy = y0 + (hvox[i] >> 8 & 255) - 1, gz = z0 + (hvox[i] >> 16) - 1;
                const bool in = gx >= 0 && gx < S && gy >= 0 && gy < S && gz >= 0 && gz < S;
                const long long v = in ? (gz * S + gy) * S + gx : 0;  // S <= 512: below 2^27
                cp_async16(xs + (piece >> 1) * kXRow + part * 8, a.x + v * a.ld_x + a.x_off + ci0 + part * 8, in);
            }
        }
        cp_async_commit();
    };
    constexpr int kRows = 256 / (16 * MT);
    float bias = 0.0f;
    for (int k = 0; k < kWgradStages - 1; ++k) stage(blockIdx.x + k * gridDim.x, k);
    int slot = 0;
    for (int brick = blockIdx.x; brick < nbricks; brick += gridDim.x) {
        cp_async_wait(kWgradStages - 2);
        __syncthreads();
        // over the brick before, which every warp has left
        stage(brick + (kWgradStages - 1) * gridDim.x, slot > 0 ? slot - 1 : kWgradStages - 1);
        if (blockIdx.z == 0) {  // bias gradient: channel threadIdx.x % (16 MT), every kRows-th voxel
            const __nv_bfloat16* const col = smem + slot * ring + (threadIdx.x / (16 * MT)) * kGRow + threadIdx.x % (16 * MT);
#pragma unroll
            for (int l = 0; l < 128; l += kRows) bias += __bfloat162float(col[l * kGRow]);
        }
        const __nv_bfloat16* const grow = smem + slot * ring + grow0;
        const __nv_bfloat16* const xs = smem + slot * ring + 128 * kGRow;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            if (s * 16 >= nvox) break;
            unsigned af[MT][4];  // co x voxel, shared by the warp's taps
#pragma unroll
            for (int m = 0; m < MT; ++m) ldmatrix4_trans(af[m], grow + s * 16 * kGRow + m * 16);
            const __nv_bfloat16* const xrow = xs + xstep[s];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (q < ntap) {
                    unsigned bf[4];  // voxel x ci: input channels 0-7 and 8-15
                    ldmatrix4_trans(bf, xrow + toff[q]);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int m = 0; m < MT; ++m) mma16816(acc[q][m][j], af[m], bf[2 * j], bf[2 * j + 1]);
                }
            }
        }
        slot = slot + 1 < kWgradStages ? slot + 1 : 0;
    }
    if (blockIdx.z == 0) {
        __shared__ float red[256];
        red[threadIdx.x] = bias;
        __syncthreads();
        if (threadIdx.x < 16 * MT) {
            for (int r = 1; r < kRows; ++r) bias += red[r * 16 * MT + threadIdx.x];
            a.bias_part[(long long)blockIdx.x * a.cout + co0 + threadIdx.x] = bias;
        }
    }
    // partials: part[blk][co (16 MT)][27][16]
    const long long blk = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    float* out = a.part + blk * (16 * MT * 27 * 16);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (q >= ntap) continue;
        const int t = warp + 8 * q;
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int co = m * 16 + g, ci = j * 8 + tig * 2;
                out[((long long)co * 27 + t) * 16 + ci] = acc[q][m][j][0];
                out[((long long)co * 27 + t) * 16 + ci + 1] = acc[q][m][j][1];
                out[((long long)(co + 8) * 27 + t) * 16 + ci] = acc[q][m][j][2];
                out[((long long)(co + 8) * 27 + t) * 16 + ci + 1] = acc[q][m][j][3];
            }
    }
}

// dW[co][tap][ci] (+)= sum over the vblocks of the partials: SLICES threads an
// element take every SLICES-th block each, and their sums are added in order
// (one thread an element, with up to 304 dependent reads on 27 blocks, took
// 24 us, 32 threads 7; with 4 blocks one thread an element reads them at once).
// Four input channels a thread.  The blocks past the weights' add the bias
// gradient's partials, a warp a channel (lane l takes the vblocks l, l + 32, ..).
template <int SLICES>
__global__ void __launch_bounds__(256)
wgrad_reduce_kernel(const float* __restrict__ part, const float* __restrict__ bias_part, int vblocks, int mt, int cout,
                    int cin, float* __restrict__ dw, float* __restrict__ db, int accumulate)
{
    constexpr int kElems = 256 / SLICES;
    __shared__ float4 sum[SLICES][kElems];
    const int total = cout * 27 * cin;
    const int wblocks = (total / 4 + kElems - 1) / kElems;
    if (blockIdx.x >= wblocks) {
        const int c = (blockIdx.x - wblocks) * 8 + (threadIdx.x >> 5);  // cout is a multiple of 8
        float s = 0.0f;
        for (int vb = threadIdx.x & 31; vb < vblocks; vb += 32) s += bias_part[(long long)vb * cout + c];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) db[c] = accumulate ? db[c] + s : s;
        return;
    }
    const int tile_co = 16 * mt;
    const int lane = threadIdx.x % kElems, slice = threadIdx.x / kElems;
    const int e = 4 * (blockIdx.x * kElems + lane);
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (e < total) {
        const int ci = e % cin, t = (e / cin) % 27, co = e / (27 * cin);
        const long long blk0 = ((long long)(ci / 16) * (cout / tile_co) + co / tile_co) * vblocks;
        const float* at = part + blk0 * (tile_co * 27 * 16) + ((long long)(co % tile_co) * 27 + t) * 16 + (ci % 16);
#pragma unroll 5
        for (int vb = slice; vb < vblocks; vb += SLICES) {
            const float4 w = *reinterpret_cast<const float4*>(at + (long long)vb * (tile_co * 27 * 16));
            s.x += w.x, s.y += w.y, s.z += w.z, s.w += w.w;
        }
    }
    if (SLICES > 1) {
        sum[slice][lane] = s;
        __syncthreads();
        if (slice == 0)
            for (int q = 1; q < SLICES; ++q) {
                const float4 w = sum[q][lane];
                s.x += w.x, s.y += w.y, s.z += w.z, s.w += w.w;
            }
    }
    if (slice == 0 && e < total) {  // (a layer's offset in the gradients need not be a multiple of 16 bytes)
        const float v[4] = {s.x, s.y, s.z, s.w};
        for (int k = 0; k < 4; ++k) dw[e + k] = accumulate ? dw[e + k] + v[k] : v[k];
    }
}

int wgrad_mt(int cout) { return cout % 32 == 0 ? 2 : 1; }

size_t wgrad_smem_bytes(int mt, const Brick& b)
{
    return kWgradStages * sizeof(__nv_bfloat16) * (size_t)(128 * (16 * mt + 8) + (b.bx + 2) * (b.by + 2) * (b.bz + 2) * kXRow);
}

int wgrad_vblocks(int S, int cout, int cin, int sms)
{
    const Brick b = brick_for(S);
    const int nbricks = (S / b.bx) * (S / b.by) * (S / b.bz);
    const int tiles = (cout / (16 * wgrad_mt(cout))) * (cin / 16);
    int vb = 2 * sms / tiles;  // one wave: two blocks a multiprocessor
    if (vb > nbricks) vb = nbricks;
    return vb < 1 ? 1 : vb;
}

void prepare_wgrad()
{
    const Brick b = brick_for(128);
    cudaFuncSetAttribute(wgrad_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem_bytes(1, b));
    cudaFuncSetAttribute(wgrad_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem_bytes(2, b));
}

void launch_wgrad(WgradArgs a, int vblocks, float* dw, float* db, int accumulate, cudaStream_t s)
{
    a.brick = brick_for(a.S);
    const int mt = wgrad_mt(a.cout);
    const dim3 grid(vblocks, a.cout / (16 * mt), a.cin / 16);
    const size_t smem = wgrad_smem_bytes(mt, a.brick);
    if (mt == 2)
        wgrad_kernel<2><<<grid, 256, smem, s>>>(a);
    else
        wgrad_kernel<1><<<grid, 256, smem, s>>>(a);
    const int total4 = a.cout * 27 * a.cin / 4, bb = a.cout / 8;
    const float *wp = a.part, *bp = a.bias_part;
    if (vblocks <= 4)
        wgrad_reduce_kernel<1><<<(total4 + 255) / 256 + bb, 256, 0, s>>>(wp, bp, vblocks, mt, a.cout, a.cin, dw, db,
                                                                         accumulate);
    else if (vblocks <= 64)
        wgrad_reduce_kernel<8><<<(total4 + 31) / 32 + bb, 256, 0, s>>>(wp, bp, vblocks, mt, a.cout, a.cin, dw, db,
                                                                       accumulate);
    else
        wgrad_reduce_kernel<32><<<(total4 + 7) / 8 + bb, 256, 0, s>>>(wp, bp, vblocks, mt, a.cout, a.cin, dw, db,
                                                                      accumulate);
}

// ---------------------------------------------------------------------------
// Eight consecutive channels of a voxel as one 16-byte value.
struct Bf8 {
    __nv_bfloat16 v[8];
};
__device__ __forceinline__ Bf8 load8(const __nv_bfloat16* p)
{
    const uint4 w = *reinterpret_cast<const uint4*>(p);
    Bf8 r;
    memcpy(&r, &w, sizeof r);
    return r;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const Bf8& r)
{
    uint4 w;
    memcpy(&w, &r, sizeof w);
    *reinterpret_cast<uint4*>(p) = w;
}

// ---------------------------------------------------------------------------
// 2x2x2 average pooling (S -> S/2) and its adjoint with the skip gradient and the ReLU mask
// (eight channels a thread: the channel counts, row strides and offsets are
// multiples of 8)
__global__ void pool_kernel(const __nv_bfloat16* __restrict__ x, int ld_x, int off_x, int C, int S,
                            __nv_bfloat16* __restrict__ y)
{
    const int Sh = S / 2, groups = C / 8;
    const int total = Sh * Sh * Sh * groups;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = 8 * (e % groups), p = e / groups;
        const int px = p % Sh, py = (p / Sh) % Sh, pz = p / (Sh * Sh);
        float s[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const long long v = ((long long)(2 * pz + (q >> 2)) * S + (2 * py + ((q >> 1) & 1))) * S + 2 * px + (q & 1);
            const Bf8 w = load8(x + v * ld_x + off_x + c);
#pragma unroll
            for (int k = 0; k < 8; ++k) s[k] += __bfloat162float(w.v[k]);
        }
        Bf8 r;
#pragma unroll
        for (int k = 0; k < 8; ++k) r.v[k] = __float2bfloat16_rn(0.125f * s[k]);
        store8(y + (long long)p * C + c, r);
    }
}

// gx[v, c] = (gp[parent(v), c] / 8 + gskip[v, off_s + c]) * (mask[v, off_m + c] > 0)
__global__ void pool_back_kernel(const __nv_bfloat16* __restrict__ gp, const __nv_bfloat16* __restrict__ gskip,
                                 int ld_s, int off_s, const __nv_bfloat16* __restrict__ mask, int ld_m, int off_m,
                                 int C, int S, __nv_bfloat16* __restrict__ gx)
{
    const int Sh = S / 2, groups = C / 8;
    const long long total = (long long)S * S * S * groups;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const unsigned u = (unsigned)e;  // below 2^31 for S <= 512, C <= 128
        const int c = 8 * (int)(u % (unsigned)groups);
        const unsigned v = u / (unsigned)groups;
        const int x = (int)(v % (unsigned)S), y = (int)((v / (unsigned)S) % (unsigned)S), z = (int)(v / ((unsigned)S * S));
        const long long p = ((long long)(z / 2) * Sh + y / 2) * Sh + x / 2;
        const Bf8 a = load8(gp + p * C + c), m = load8(mask + (long long)v * ld_m + off_m + c);
        Bf8 k = a, r;
        if (gskip) k = load8(gskip + (long long)v * ld_s + off_s + c);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float w = 0.125f * __bfloat162float(a.v[q]);
            if (gskip) w += __bfloat162float(k.v[q]);
            if (!(__bfloat162float(m.v[q]) > 0.0f)) w = 0.0f;
            r.v[q] = __float2bfloat16_rn(w);
        }
        store8(gx + (long long)v * C + c, r);
    }
}

// nearest-neighbour upsampling S/2 -> S into channels [0, C) of a concatenation (row stride ld_y)
__global__ void up_kernel(const __nv_bfloat16* __restrict__ x, int C, int S, __nv_bfloat16* __restrict__ y, int ld_y)
{
    const int Sh = S / 2, groups = C / 8;
    const long long total = (long long)S * S * S * groups;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const unsigned u = (unsigned)e;
        const int c = 8 * (int)(u % (unsigned)groups);
        const unsigned v = u / (unsigned)groups;
        const int px = (int)(v % (unsigned)S) / 2, py = (int)((v / (unsigned)S) % (unsigned)S) / 2;
        const int pz = (int)(v / ((unsigned)S * S)) / 2;
        store8(y + (long long)v * ld_y + c, load8(x + (((long long)pz * Sh + py) * Sh + px) * C + c));
    }
}

// gx[p, c] = (sum of gy over the 8 children, channels [0, C) of row stride ld_y) * (mask[p, c] > 0)
__global__ void up_back_kernel(const __nv_bfloat16* __restrict__ gy, int ld_y, const __nv_bfloat16* __restrict__ mask,
                               int C, int S, __nv_bfloat16* __restrict__ gx)
{
    const int Sh = S / 2, groups = C / 8;
    const int total = Sh * Sh * Sh * groups;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        const int c = 8 * (e % groups), p = e / groups;
        const int px = p % Sh, py = (p / Sh) % Sh, pz = p / (Sh * Sh);
        float s[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const long long v = ((long long)(2 * pz + (q >> 2)) * S + (2 * py + ((q >> 1) & 1))) * S + 2 * px + (q & 1);
            const Bf8 w = load8(gy + v * ld_y + c);
#pragma unroll
            for (int k = 0; k < 8; ++k) s[k] += __bfloat162float(w.v[k]);
        }
        const Bf8 m = load8(mask + (long long)p * C + c);
        Bf8 r;
#pragma unroll
        for (int k = 0; k < 8; ++k) r.v[k] = __float2bfloat16_rn(__bfloat162float(m.v[k]) > 0.0f ? s[k] : 0.0f);
        store8(gx + (long long)p * C + c, r);
    }
}

static int ew_blocks(long long total)
{
    long long b = (total + 255) / 256;
    return (int)(b < 152 * 16 ? b : 152 * 16);
}

void launch_pool(const __nv_bfloat16* x, int ld_x, int off_x, int C, int S, __nv_bfloat16* y, cudaStream_t s)
{
    pool_kernel<<<ew_blocks((long long)(S / 2) * (S / 2) * (S / 2) * C / 8), 256, 0, s>>>(x, ld_x, off_x, C, S, y);
}

void launch_pool_back(const __nv_bfloat16* gp, const __nv_bfloat16* gskip, int ld_s, int off_s,
                      const __nv_bfloat16* mask, int ld_m, int off_m, int C, int S, __nv_bfloat16* gx, cudaStream_t s)
{
    pool_back_kernel<<<ew_blocks((long long)S * S * S * C / 8), 256, 0, s>>>(gp, gskip, ld_s, off_s, mask, ld_m, off_m, C,
                                                                         S, gx);
}

void launch_up(const __nv_bfloat16* x, int C, int S, __nv_bfloat16* y, int ld_y, cudaStream_t s)
{
    up_kernel<<<ew_blocks((long long)S * S * S * C / 8), 256, 0, s>>>(x, C, S, y, ld_y);
}

void launch_up_back(const __nv_bfloat16* gy, int ld_y, const __nv_bfloat16* mask, int C, int S, __nv_bfloat16* gx,
                    cudaStream_t s)
{
    up_back_kernel<<<ew_blocks((long long)(S / 2) * (S / 2) * (S / 2) * C / 8), 256, 0, s>>>(gy, ld_y, mask, C, S, gx);
}

// ---------------------------------------------------------------------------
// Network input.  Voxel (x, y, z) of the S^3 input is node (x, y, z) of the
// box's (S+1)^3 grid: channel 0 = rho_scale * rho, channel 1 = Phi_N / phi_scale,
// channel 2 = the box flag, channels 3..15 = 0.
__global__ void input_from_grids_kernel(const double* __restrict__ rho, const double* __restrict__ phiN, int S,
                                        double rho_scale, double inv_phi, float flag, __nv_bfloat16* __restrict__ x0)
{
    const long long total = (long long)S * S * S;
    const int n1 = S + 1;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < total;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % S), y = (int)((v / S) % S), z = (int)(v / ((long long)S * S));
        const long long node = ((long long)z * n1 + y) * n1 + x;
        __nv_bfloat16 row[16];
        row[0] = __float2bfloat16_rn((float)(rho[node] * rho_scale));
        row[1] = __float2bfloat16_rn((float)(phiN[node] * inv_phi));
        row[2] = __float2bfloat16_rn(flag);
#pragma unroll
        for (int c = 3; c < 16; ++c) row[c] = __float2bfloat16_rn(0.0f);
        uint4* dst = reinterpret_cast<uint4*>(x0 + v * 16);
        dst[0] = *reinterpret_cast<uint4*>(&row[0]);
        dst[1] = *reinterpret_cast<uint4*>(&row[8]);
    }
}

// training sample: [0] rho channel, [1] Phi_N channel, [2] target (Phi - Phi_N) / phi_scale, each S^3 BF16
__global__ void make_sample_kernel(const double* __restrict__ rho, const double* __restrict__ phiN,
                                   const double* __restrict__ phi, int S, double rho_scale, double inv_phi,
                                   __nv_bfloat16* __restrict__ sample)
{
    const long long total = (long long)S * S * S;
    const int n1 = S + 1;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < total;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % S), y = (int)((v / S) % S), z = (int)(v / ((long long)S * S));
        const long long node = ((long long)z * n1 + y) * n1 + x;
        sample[v] = __float2bfloat16_rn((float)(rho[node] * rho_scale));
        sample[total + v] = __float2bfloat16_rn((float)(phiN[node] * inv_phi));
        sample[2 * total + v] = __float2bfloat16_rn((float)((phi[node] - phiN[node]) * inv_phi));
    }
}

__global__ void input_from_sample_kernel(const __nv_bfloat16* __restrict__ sample, int S, float flag,
                                         __nv_bfloat16* __restrict__ x0)
{
    const long long total = (long long)S * S * S;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < total;
         v += (long long)gridDim.x * blockDim.x) {
        __nv_bfloat16 row[16];
        row[0] = sample[v];
        row[1] = sample[total + v];
        row[2] = __float2bfloat16_rn(flag);
#pragma unroll
        for (int c = 3; c < 16; ++c) row[c] = __float2bfloat16_rn(0.0f);
        uint4* dst = reinterpret_cast<uint4*>(x0 + v * 16);
        dst[0] = *reinterpret_cast<uint4*>(&row[0]);
        dst[1] = *reinterpret_cast<uint4*>(&row[8]);
    }
}

void launch_input_from_grids(const double* rho, const double* phiN, int S, double rho_scale, double inv_phi,
                             float flag, __nv_bfloat16* x0, cudaStream_t s)
{
    input_from_grids_kernel<<<ew_blocks((long long)S * S * S), 256, 0, s>>>(rho, phiN, S, rho_scale, inv_phi, flag, x0);
}

void launch_make_sample(const double* rho, const double* phiN, const double* phi, int S, double rho_scale,
                        double inv_phi, __nv_bfloat16* sample, cudaStream_t s)
{
    make_sample_kernel<<<ew_blocks((long long)S * S * S), 256, 0, s>>>(rho, phiN, phi, S, rho_scale, inv_phi, sample);
}

void launch_input_from_sample(const __nv_bfloat16* sample, int S, float flag, __nv_bfloat16* x0, cudaStream_t s)
{
    input_from_sample_kernel<<<ew_blocks((long long)S * S * S), 256, 0, s>>>(sample, S, flag, x0);
}

// ---------------------------------------------------------------------------
// Head: yhat[v] = b + sum_c w[c] a[v, c]  (1x1x1 convolution, FP32 output).
// Training form: with target t and scale k = 2 / (S^3 nbatch):
//   loss partial += (yhat - t)^2, dy = k (yhat - t),
//   ga[v, c] = dy w[c] (a[v, c] > 0), head-gradient partials sum dy a[v, c] and sum dy.
__global__ void head_kernel(const __nv_bfloat16* __restrict__ a, const float* __restrict__ wb, long long nvox,
                            float* __restrict__ yhat)
{
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < nvox;
         v += (long long)gridDim.x * blockDim.x) {
        float s = wb[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) s += wb[c] * __bfloat162float(a[v * 16 + c]);
        yhat[v] = s;
    }
}

__global__ void head_train_kernel(const __nv_bfloat16* __restrict__ a, const float* __restrict__ wb,
                                  const __nv_bfloat16* __restrict__ target, long long nvox, float k,
                                  __nv_bfloat16* __restrict__ ga, float* __restrict__ part)
{
    // part[block][0..15] = sum dy a[:, c], [16] = sum dy, [17] = sum (yhat - t)^2
    float pw[18];
#pragma unroll
    for (int c = 0; c < 18; ++c) pw[c] = 0.0f;
    float w[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) w[c] = wb[c];
    const long long chunk = (nvox + gridDim.x - 1) / gridDim.x;
    const long long v0 = blockIdx.x * chunk, v1 = v0 + chunk < nvox ? v0 + chunk : nvox;
    for (long long v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
        float av[16];
        float s = wb[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            av[c] = __bfloat162float(a[v * 16 + c]);
            s += w[c] * av[c];
        }
        const float d = s - __bfloat162float(target[v]);
        const float dy = k * d;
        __nv_bfloat16 row[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            pw[c] += dy * av[c];
            row[c] = __float2bfloat16_rn(av[c] > 0.0f ? dy * w[c] : 0.0f);
        }
        pw[16] += dy;
        pw[17] += d * d;
        uint4* dst = reinterpret_cast<uint4*>(ga + v * 16);
        dst[0] = *reinterpret_cast<uint4*>(&row[0]);
        dst[1] = *reinterpret_cast<uint4*>(&row[8]);
    }
    __shared__ float red[18][256];
#pragma unroll
    for (int c = 0; c < 18; ++c) red[c][threadIdx.x] = pw[c];
    __syncthreads();
    if (threadIdx.x < 18) {
        float t = 0.0f;
        for (int r = 0; r < (int)blockDim.x; ++r) t += red[threadIdx.x][r];
        part[(long long)blockIdx.x * 18 + threadIdx.x] = t;
    }
}

// out[0..16] (+)= head gradients, loss_out (+)= sum of squares * loss_scale
__global__ void head_reduce_kernel(const float* __restrict__ part, int nb, float* __restrict__ dwb, int accumulate,
                                   float* __restrict__ loss, float loss_scale)
{
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;  // a warp a column
    float s = 0.0f;
    for (int b = lane; b < nb; b += 32) s += part[(long long)b * 18 + c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane != 0) return;
    if (c < 17)
        dwb[c] = accumulate ? dwb[c] + s : s;
    else if (loss)
        *loss = (accumulate ? *loss : 0.0f) + s * loss_scale;
}

void launch_head(const __nv_bfloat16* a, const float* wb, long long nvox, float* yhat, cudaStream_t s)
{
    head_kernel<<<ew_blocks(nvox), 256, 0, s>>>(a, wb, nvox, yhat);
}

void launch_head_train(const __nv_bfloat16* a, const float* wb, const __nv_bfloat16* target, long long nvox, float k,
                       __nv_bfloat16* ga, float* part, int nb, float* dwb, int accumulate, float* loss,
                       float loss_scale, cudaStream_t s)
{
    head_train_kernel<<<nb, 256, 0, s>>>(a, wb, target, nvox, k, ga, part);
    head_reduce_kernel<<<1, 18 * 32, 0, s>>>(part, nb, dwb, accumulate, loss, loss_scale);
}

// phi[node] = phiN[node] + phi_scale * yhat[v] on the interior nodes 1..S-1 of each axis
__global__ void apply_guess_kernel(const double* __restrict__ phiN, const float* __restrict__ yhat, int S,
                                   double phi_scale, double* __restrict__ phi)
{
    const long long total = (long long)(S - 1) * (S - 1) * (S - 1);
    const int n1 = S + 1;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int x = 1 + (int)(e % (S - 1)), y = 1 + (int)((e / (S - 1)) % (S - 1)),
                  z = 1 + (int)(e / ((long long)(S - 1) * (S - 1)));
        const long long node = ((long long)z * n1 + y) * n1 + x;
        const long long v = ((long long)z * S + y) * S + x;
        phi[node] = phiN[node] + phi_scale * (double)yhat[v];
    }
}

void launch_apply_guess(const double* phiN, const float* yhat, int S, double phi_scale, double* phi, cudaStream_t s)
{
    apply_guess_kernel<<<ew_blocks((long long)(S - 1) * (S - 1) * (S - 1)), 256, 0, s>>>(phiN, yhat, S, phi_scale, phi);
}

// ---------------------------------------------------------------------------
// Adam on the FP32 master parameters (gradients already averaged over the
// batch), then the BF16 copies in the two layouts the convolutions read:
// forward W[co][tap][ci] and data-gradient Wd[ci][26 - tap][co].
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    }
}

__global__ void weights_bf16_kernel(const float* __restrict__ w, int cout, int cin, __nv_bfloat16* __restrict__ wf,
                                    __nv_bfloat16* __restrict__ wd)
{
    const long long total = (long long)cout * 27 * cin;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int ci = (int)(e % cin), t = (int)((e / cin) % 27), co = (int)(e / (27LL * cin));
        const __nv_bfloat16 h = __float2bfloat16_rn(w[e]);
        wf[e] = h;
        if (wd) wd[((long long)ci * 27 + (26 - t)) * cout + co] = h;
    }
}

void launch_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2, float eps,
                 float c1, float c2, cudaStream_t s)
{
    adam_kernel<<<ew_blocks(n), 256, 0, s>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
}

void launch_weights_bf16(const float* w, int cout, int cin, __nv_bfloat16* wf, __nv_bfloat16* wd, cudaStream_t s)
{
    weights_bf16_kernel<<<ew_blocks((long long)cout * 27 * cin), 256, 0, s>>>(w, cout, cin, wf, wd);
}

__global__ void scale_kernel(float* __restrict__ x, long long n, float k)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        x[i] *= k;
}

void launch_scale(float* x, long long n, float k, cudaStream_t s) { scale_kernel<<<ew_blocks(n), 256, 0, s>>>(x, n, k); }

}  // namespace unet
}  // namespace qumond
