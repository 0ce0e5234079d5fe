// The U-Net's 3^3 convolution on the fifth-generation tensor cores
// (tcgen05): an implicit GEMM with M = 128 output voxels, N = up to 64 output
// channels, K = 27 taps x 16 input channels per chunk, accumulated in tensor
// memory (TMEM) and read back by the four warps for the epilogue.
//
// Layout trick: the input brick of a CTA is 1 or 2 x 16 x 8 voxels (z, y, x) and
// its halo 3 or 4 x 18 x 10; the halo of a 16-channel chunk is kept in shared
// memory as two planes (channels 0-7 and 8-15), 16 bytes per voxel.  Eight
// consecutive voxels of an x-row are then one 8 x 16-byte core matrix of the
// canonical K-major layout, the sixteen y-rows are core matrices a constant
// 160 bytes apart, and the two channel halves a plane apart, so the A operand
// of every tap is a shared-memory descriptor into the same halo (no im2col
// copy).  The weights of the chunk are stored per tap as [channel half]
// [output channel][8 channels].  One thread issues the 27 MMAs of a chunk and
// commits them to an mbarrier; the CTA waits (bounded) before it overwrites
// the chunk's shared memory.
//
// The shared-memory descriptors follow the PTX ISA's canonical K-major layout
// without swizzling: core matrices of 8 rows x 16 bytes, the leading-dimension
// byte offset (bits 16-29) the distance between core matrices adjacent along
// K, the stride-dimension byte offset (bits 32-45) the distance between
// 8-row groups along M (or N).  tc_selftest checks one MMA with that encoding
// against a CPU product (a unit test; the product path does not call it).
#include "unet_internal.h"

#include <cstdio>
#include <cstring>
#include <vector>

namespace qumond {
namespace unet {

namespace {

constexpr int kHX = 10, kHY = 18;  // halo of a ZP x 16 x 8 brick along x and y
__host__ __device__ constexpr int halo_voxels(int zp) { return kHX * kHY * (zp + 2); }
__host__ __device__ constexpr unsigned plane_bytes(int zp) { return (unsigned)halo_voxels(zp) * 16; }  // one channel half
constexpr long long kSpinLimit = 1LL << 24;

// shared memory of one chunk of 16 input channels for NT output channels and ZP planes: halo and weights
__host__ __device__ constexpr unsigned conv3_tc_stage_bytes(int nt, int zp) { return 2 * plane_bytes(zp) + 27u * 2 * nt * 16; }

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, K-major, no swizzle: start address >> 4 in
// bits 0-13; leading-dimension byte offset >> 4 (between core matrices along
// K) in bits 16-29; stride-dimension byte offset >> 4 (between 8-row groups
// along M or N) in bits 32-45; the descriptor version (1) at bit 46; base
// offset 0, swizzle mode 0 (bits 61-63).
__device__ __forceinline__ unsigned long long sdesc(unsigned addr, unsigned kstride, unsigned mnstride)
{
    return (unsigned long long)((addr >> 4) & 0x3FFFu) | ((unsigned long long)((kstride >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)((mnstride >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B, both K-major, N and M
__host__ __device__ constexpr unsigned idesc_bf16(int N, int M)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// bounded wait on an mbarrier phase: gives up after kSpinLimit polls or about a second, whichever comes first;
// false (and *fault = 3) when it gave up
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, int* fault)
{
    long long spins = 0;
    unsigned long long t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        ++spins;
        if ((spins & 1023) == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 1000000000ull) spins = kSpinLimit + 1;
        }
        if (spins > kSpinLimit) {
            if (fault) atomicExch(fault, 3);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tmem_alloc(unsigned* slot, unsigned ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(unsigned taddr, unsigned ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc, int acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ void commit(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float* v)
{
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

// ---------------------------------------------------------------------------
// Self-test: D (128 x 16) = A (128 x 16) B^T (16 x 16) for small integer
// operands, A and B in a compact canonical layout (core matrix (g, h) of rows
// 8g.. and K-columns 8h.. at g*256 + h*128 bytes), read back from TMEM.  Every
// address the descriptors form lies inside A or B.
__global__ void __launch_bounds__(128) tc_selftest_kernel(float* out, int* fault)
{
    __shared__ __align__(128) __nv_bfloat16 A[128 * 16];
    __shared__ __align__(128) __nv_bfloat16 B[16 * 16];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ unsigned slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < 128 * 16; e += 128) {
        const int m = e / 16, k = e % 16;
        A[(m / 8) * 128 + (k / 8) * 64 + (m % 8) * 8 + (k % 8)] = __float2bfloat16_rn((float)((m + 3 * k) % 7 - 3));
    }
    for (int e = tid; e < 16 * 16; e += 128) {
        const int n = e / 16, k = e % 16;
        B[(n / 8) * 128 + (k / 8) * 64 + (n % 8) * 8 + (k % 8)] = __float2bfloat16_rn((float)((2 * n + k) % 5 - 2));
    }
    if (warp == 0) tmem_alloc(&slot, 32);
    if (tid == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_proxy();
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned taddr = slot;
    if (tid == 0) {
        mma(taddr, sdesc(smem_u32(A), 128, 256), sdesc(smem_u32(B), 128, 256), idesc_bf16(16, 128), 0);
        commit(&bar);
    }
    const bool ok = mbar_wait(&bar, 0, fault);
    fence_after();
    float v[16];
    tmem_ld16(taddr + ((unsigned)(warp * 32) << 16), v);
    for (int q = 0; q < 16; ++q) out[(warp * 32 + lane) * 16 + q] = ok ? v[q] : __int_as_float(0x7fc00000);
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, 32);
}

}  // namespace

// ---------------------------------------------------------------------------
// y = act(conv(x)) on the tensor cores, a brick of ZP planes of 16 x 8 voxels
// (M = 128 each) and NT output channels a block.  The chunks of 16 input channels come by cp.async
// into a ring of a.stages buffers; the loads of the chunks ahead and the issue
// of the next 27 MMAs (unrolled: the descriptors are constants beside the base)
// run while a chunk's MMAs do.  Loaded and issued in turn, a chunk took 7.5 us
// on an otherwise idle multiprocessor (16^3, 192 -> 64 channels: 82 us), now
// 2.4 (29 us); 16 -> 16 channels at 64^3: 28 -> 20 us.
template <int NT, int ZP>
__global__ void __launch_bounds__(128) conv3_tc_kernel(ConvArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr unsigned kStage = conv3_tc_stage_bytes(NT, ZP);  // a chunk: halo (2 x kHV x 8), weights (27 x 2 x NT x 8)
    constexpr int kHV = halo_voxels(ZP);
    constexpr unsigned kPlaneBytes = plane_bytes(ZP);
    __shared__ __align__(8) unsigned long long bar[2];  // chunk c: bar[c & 1], phase c / 2
    __shared__ unsigned slot;
    constexpr unsigned kCols = NT * ZP <= 32 ? 32 : NT * ZP <= 64 ? 64 : 128;
    constexpr unsigned kIdesc = idesc_bf16(NT, 128);

    const int S = a.S;
    const int nbx = S / 8, nby = S / 16;
    const int brick = blockIdx.x;
    const int x0 = (brick % nbx) * 8, y0 = ((brick / nbx) % nby) * 16, z0 = brick / (nbx * nby) * ZP;
    const int co0 = blockIdx.y * NT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) tmem_alloc(&slot, kCols);
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned taddr = slot;
    bool ok = true;
    const int nchunks = a.cin / 16;
    auto stage = [&](int chunk) {
        if (chunk < nchunks) {
            const int ci0 = chunk * 16;
            unsigned char* const halo = smem_raw + (chunk % a.stages) * kStage;
            unsigned char* const wts = halo + 2 * kPlaneBytes;
            // the chunk's halo: voxel hv -> planes 0 and 1 (channels ci0..ci0+7, ci0+8..ci0+15)
            for (int q = tid; q < kHV * 2; q += 128) {
                const int hv = q >> 1, part = q & 1;
                const int ix = hv % kHX, iy = (hv / kHX) % kHY, iz = hv / (kHX * kHY);
                const int gx = x0 + ix - 1, gy = y0 + iy - 1, gz = z0 + iz - 1;
                const bool in = gx >= 0 && gx < S && gy >= 0 && gy < S && gz >= 0 && gz < S;
                const long long v = in ? ((long long)gz * S + gy) * S + gx : 0;
                cp_async16(halo + (part * kHV + hv) * 16, a.in + v * a.ld_in + a.in_off + ci0 + part * 8, in);
            }
            // the chunk's weights: W[co0 + n][t][ci0 + 8 part ..] -> wts[(t * 2 + part) * NT + n]
            for (int q = tid; q < 27 * 2 * NT; q += 128) {
                const int part = q & 1, n = (q >> 1) % NT, t = q / (2 * NT);
                cp_async16(wts + ((t * 2 + part) * NT + n) * 16,
                           a.w + ((long long)(co0 + n) * 27 + t) * a.cin + ci0 + part * 8, true);
            }
        }
        cp_async_commit();  // a group a chunk, empty past the last
    };
    // the MMAs that read chunk c's shared memory have completed
    auto done = [&](int c) {
        if (ok) ok = mbar_wait(&bar[c & 1], (unsigned)(c >> 1 & 1), a.fault);
    };
    const int ahead = a.stages - 1;
    for (int c = 0; c < ahead; ++c) stage(c);
    for (int c = 0; c < nchunks; ++c) {
        if (ahead == 0) stage(c);
        cp_async_wait(ahead > 1 ? ahead - 1 : 0);  // chunk c has landed
        const unsigned hbase = smem_u32(smem_raw) + (unsigned)(c % a.stages) * kStage;
        const unsigned wbase = hbase + 2 * kPlaneBytes;
        fence_proxy();
        fence_before();
        __syncthreads();
        fence_after();
        if (tid == 0 && ok) {
#pragma unroll
            for (int t = 0; t < 27; ++t) {
                const int dz = t / 9, dy = (t / 3) % 3, dx = t % 3;  // halo offsets 0..2 of the tap
                const unsigned aoff = (unsigned)(((dz * kHY + dy) * kHX + dx) * 16);
                const unsigned long long bd = sdesc(wbase + (unsigned)(t * 2 * NT * 16), NT * 16, 128);
#pragma unroll
                for (int zp = 0; zp < ZP; ++zp) {
                    const unsigned long long ad = sdesc(hbase + aoff + zp * (kHX * kHY * 16), kPlaneBytes, kHX * 16);
                    mma(taddr + zp * NT, ad, bd, kIdesc, (c > 0 || t > 0) ? 1 : 0);
                }
            }
            commit(&bar[c & 1]);
        }
        // the next load goes over chunk c - 1 (with a single buffer: over this one)
        if (ahead == 0)
            done(c);
        else if (c > 0)
            done(c - 1);
        if (ahead > 0) stage(c + ahead);
    }
    if (ahead > 0) done(nchunks - 1);
    fence_after();
    // epilogue: warp w holds TMEM lanes 32w..32w+31 = brick voxels 32w + lane
    const int m = warp * 32 + lane;
    const int ly = m / 8, lx = m % 8;
#pragma unroll
    for (int cz = 0; cz < NT * ZP; cz += 16) {  // 16 columns: plane cz / NT, channels cz % NT ..
        float r[16];
        tmem_ld16(taddr + ((unsigned)(warp * 32) << 16) + (unsigned)cz, r);
        if (!ok) continue;
        const long long v = ((long long)(z0 + cz / NT) * S + (y0 + ly)) * S + (x0 + lx);
        const int co = co0 + cz % NT;
        __nv_bfloat16 h[16];
        __nv_bfloat16 mk[16];
        if (a.mask) {
            const uint4* mp = reinterpret_cast<const uint4*>(a.mask + v * a.ld_mask + a.mask_off + co);
            *reinterpret_cast<uint4*>(&mk[0]) = mp[0];
            *reinterpret_cast<uint4*>(&mk[8]) = mp[1];
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            float x = r[q];
            if (a.bias) x += a.bias[co + q];
            if (a.relu) x = fmaxf(x, 0.0f);
            if (a.mask && !(__bfloat162float(mk[q]) > 0.0f)) x = 0.0f;
            h[q] = __float2bfloat16_rn(x);
        }
        uint4* dst = reinterpret_cast<uint4*>(a.out + v * a.ld_out + a.out_off + co);
        dst[0] = *reinterpret_cast<uint4*>(&h[0]);
        dst[1] = *reinterpret_cast<uint4*>(&h[8]);
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(taddr, kCols);
}

// Planes of a brick: two share the chunk's weights and two of their halo planes,
// where the level leaves at least four blocks for every multiprocessor (64^3,
// 16 -> 16 channels: 20 us with one plane, 18 with two; 48 -> 16: 54 and 47;
// 16 -> 48: 35 and 27).  Whole networks, one plane everywhere and this rule in
// turn (each side within 0.4 %, the same bits): gradients of a batch of two at
// 64^3 2029 and 1983 us; of one at 48^3 814 and 812, at 80^3 1600 and 1543, at
// 96^3 2155 and 2018, at 128^3 4038 and 3618; an inference at 128^3 1454 and
// 1213.  With the line at eight blocks 64^3 and 96^3 lose (1017, 2036); at two
// 48^3 and 96^3 take 803 and 1950 and nothing is slower, so it may lie lower.
static int conv3_tc_planes(int blocks, int sms) { return blocks >= 2 * 4 * sms ? 2 : 1; }

bool conv3_tc_applies(const ConvArgs& a)
{
    // 16 <= S (the 1 x 16 x 8 brick), channel counts in 16-channel chunks, row strides and offsets in
    // 16-byte units (8 channels) for the vector loads and stores
    return a.use_tc && a.S >= 16 && a.S % 16 == 0 && a.cin % 16 == 0 && a.cout % 16 == 0 &&
           a.ld_in % 8 == 0 && a.in_off % 8 == 0 && a.ld_out % 8 == 0 && a.out_off % 8 == 0 &&
           (!a.mask || (a.ld_mask % 8 == 0 && a.mask_off % 8 == 0));
}

template <int NT, int ZP>
static void prepare_tc()
{
    cudaFuncSetAttribute(conv3_tc_kernel<NT, ZP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)conv3_smem_max(conv3_tc_stage_bytes(NT, ZP)));
}

void prepare_conv3_tc()
{
    prepare_tc<16, 1>(), prepare_tc<32, 1>(), prepare_tc<48, 1>(), prepare_tc<64, 1>();
    prepare_tc<16, 2>(), prepare_tc<32, 2>(), prepare_tc<48, 2>(), prepare_tc<64, 2>();
}

template <int NT>
static void launch_tc(ConvArgs a, int bricks, cudaStream_t s)
{
    const int tiles = a.cout / NT, zp = conv3_tc_planes(bricks * tiles, a.sms);
    const size_t stage = conv3_tc_stage_bytes(NT, zp);
    const dim3 grid((unsigned)(bricks / zp), (unsigned)tiles);
    a.stages = conv3_stages(stage, (int)(grid.x * grid.y), a.cin / 16, a.sms);
    if (zp == 2)
        conv3_tc_kernel<NT, 2><<<grid, 128, a.stages * stage, s>>>(a);
    else
        conv3_tc_kernel<NT, 1><<<grid, 128, a.stages * stage, s>>>(a);
}

void launch_conv3_tc(ConvArgs a, cudaStream_t s)
{
    const int bricks = (a.S / 8) * (a.S / 16) * a.S;
    switch (conv3_tile(a.cout, bricks, a.sms)) {
    case 64: launch_tc<64>(a, bricks, s); break;
    case 48: launch_tc<48>(a, bricks, s); break;
    case 32: launch_tc<32>(a, bricks, s); break;
    default: launch_tc<16>(a, bricks, s); break;
    }
}

// One MMA with the library's descriptor encoding against the CPU product of
// the same small integer operands: 1 if every element matches, 0 if not, -1
// on a CUDA error.  A unit test of the encoding; the product path does not run it.
int tc_selftest()
{
    float* d_out = nullptr;
    int* d_fault = nullptr;
    if (cudaMalloc(&d_out, 128 * 16 * sizeof(float)) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    if (cudaMalloc(&d_fault, sizeof(int)) != cudaSuccess || cudaMemset(d_fault, 0, sizeof(int)) != cudaSuccess) {
        (void)cudaGetLastError();
        cudaFree(d_out);
        return -1;
    }
    std::vector<float> want(128 * 16), got(128 * 16);
    for (int m = 0; m < 128; ++m)
        for (int n = 0; n < 16; ++n) {
            float s = 0.0f;
            for (int k = 0; k < 16; ++k) s += (float)((m + 3 * k) % 7 - 3) * (float)((2 * n + k) % 5 - 2);
            want[m * 16 + n] = s;
        }
    int result = -1;
    tc_selftest_kernel<<<1, 128>>>(d_out, d_fault);
    int fault = 0;
    if (cudaDeviceSynchronize() == cudaSuccess &&
        cudaMemcpy(got.data(), d_out, got.size() * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess &&
        cudaMemcpy(&fault, d_fault, sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess)
        result = (fault == 0 && std::memcmp(got.data(), want.data(), got.size() * sizeof(float)) == 0) ? 1 : 0;
    else
        (void)cudaGetLastError();
    cudaFree(d_out);
    cudaFree(d_fault);
    return result;
}

}  // namespace unet
}  // namespace qumond
