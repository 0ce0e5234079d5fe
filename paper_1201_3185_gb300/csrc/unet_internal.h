// Internal interface of the learned-initial-guess kernels (unet_kernels.cu)
// and the network built from them (unet_api.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>

namespace qumond {
namespace unet {

struct Brick {
    int bz, by, bx;  // voxels of a CTA's output brick along z, y, x (product <= 128)
};

// A 3^3 convolution (zero padding, stride 1) on an S^3 level, channels last.
struct ConvArgs {
    const __nv_bfloat16* in;  // input, row stride ld_in, channels [in_off, in_off + cin)
    int ld_in, in_off, cin;
    const __nv_bfloat16* w;   // weights [cout][27][cin]
    const float* bias;        // cout, or null
    __nv_bfloat16* out;       // output, row stride ld_out, channels [out_off, out_off + cout)
    int ld_out, out_off, cout;
    const __nv_bfloat16* mask;  // multiply output channel co by (mask[v, mask_off + co] > 0), or null
    int ld_mask, mask_off;
    int relu;
    int S;
    int sms;      // multiprocessors of the device
    Brick brick;  // set by the launcher
    int stages;   // set by the launcher: chunks of input channels in flight
    int use_tc;   // 1: the convolution may run on the tcgen05 path (where conv3_tc_applies); 0: mma.sync
    int* fault;   // set to 3 when a bounded wait of the tcgen05 path gave up
};

// Weight gradient of a 3^3 convolution: dW[co][tap][ci] = sum_v g[v, co] x[v + off(tap), ci], and the bias gradient
// sum_v g[v, co].
struct WgradArgs {
    const __nv_bfloat16* x;  // layer input, row stride ld_x, channels [x_off, x_off + cin)
    int ld_x, x_off, cin;
    const __nv_bfloat16* g;  // gradient at the layer output (after the ReLU mask), row stride ld_g
    int ld_g, g_off, cout;
    float* part;             // partial sums, (cout/16MT) x (cin/16) x vblocks x (16MT x 27 x 16) floats
    float* bias_part;        // partial sums, vblocks x cout floats
    int S;
    Brick brick;
};

// 16 bytes of global memory to shared memory, or 16 zero bytes where !in (the address is not read then); through
// the L1, since the blocks of a multiprocessor read the same weights and overlapping halos
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in)
{
    const unsigned at = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(at), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest `pending` (0 to 2) of this thread's groups are complete
__device__ __forceinline__ void cp_async_wait(int pending)
{
    if (pending == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (pending == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 2;" ::: "memory");
}

Brick brick_for(int S);
size_t conv3_smem_bytes(int cout_tile);
int conv3_tile(int cout, int bricks, int sms);  // output channels of a block
constexpr size_t kConvSmem = 226 * 1024;  // of a multiprocessor, for the chunk rings of its blocks
constexpr int kConvStages = 4;
int conv3_stages(size_t stage_bytes, int blocks, int chunks, int sms);
// the most that conv3_stages gives a block
inline size_t conv3_smem_max(size_t stage_bytes)
{
    const size_t n = kConvSmem / (stage_bytes + 2048);
    return stage_bytes * (n < kConvStages ? n : kConvStages);
}
void prepare_conv3();
void launch_conv3(ConvArgs a, cudaStream_t s);

// tcgen05 path (unet_tc.cu)
int tc_selftest();
bool conv3_tc_applies(const ConvArgs& a);
void prepare_conv3_tc();
void launch_conv3_tc(ConvArgs a, cudaStream_t s);

int wgrad_mt(int cout);
size_t wgrad_smem_bytes(int mt, const Brick& b);
int wgrad_vblocks(int S, int cout, int cin, int sms);
void prepare_wgrad();
void launch_wgrad(WgradArgs a, int vblocks, float* dw, float* db, int accumulate, cudaStream_t s);

void launch_pool(const __nv_bfloat16* x, int ld_x, int off_x, int C, int S, __nv_bfloat16* y, cudaStream_t s);
void launch_pool_back(const __nv_bfloat16* gp, const __nv_bfloat16* gskip, int ld_s, int off_s,
                      const __nv_bfloat16* mask, int ld_m, int off_m, int C, int S, __nv_bfloat16* gx, cudaStream_t s);
void launch_up(const __nv_bfloat16* x, int C, int S, __nv_bfloat16* y, int ld_y, cudaStream_t s);
void launch_up_back(const __nv_bfloat16* gy, int ld_y, const __nv_bfloat16* mask, int C, int S, __nv_bfloat16* gx,
                    cudaStream_t s);
void launch_input_from_grids(const double* rho, const double* phiN, int S, double rho_scale, double inv_phi,
                             float flag, __nv_bfloat16* x0, cudaStream_t s);
void launch_make_sample(const double* rho, const double* phiN, const double* phi, int S, double rho_scale,
                        double inv_phi, __nv_bfloat16* sample, cudaStream_t s);
void launch_input_from_sample(const __nv_bfloat16* sample, int S, float flag, __nv_bfloat16* x0, cudaStream_t s);
void launch_head(const __nv_bfloat16* a, const float* wb, long long nvox, float* yhat, cudaStream_t s);
void launch_head_train(const __nv_bfloat16* a, const float* wb, const __nv_bfloat16* target, long long nvox, float k,
                       __nv_bfloat16* ga, float* part, int nb, float* dwb, int accumulate, float* loss,
                       float loss_scale, cudaStream_t s);
void launch_apply_guess(const double* phiN, const float* yhat, int S, double phi_scale, double* phi, cudaStream_t s);
void launch_adam(float* p, const float* g, float* m, float* v, long long n, float lr, float b1, float b2, float eps,
                 float c1, float c2, cudaStream_t s);
void launch_weights_bf16(const float* w, int cout, int cin, __nv_bfloat16* wf, __nv_bfloat16* wd, cudaStream_t s);
void launch_scale(float* x, long long n, float k, cudaStream_t s);

}  // namespace unet
}  // namespace qumond
