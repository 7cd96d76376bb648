// qmcrt_flow.cu -- the learned proposal: a piecewise-linear autoregressive warp of the
// first-scattering coordinates with two 4-layer MLP conditionals.  The entry points of its
// forward pass (qmcrt_warp_fused.cu), of its cross-entropy gradient (qmcrt_train.cu) and
// Adam with the refresh of the bf16 weights.
#include <cmath>
#include <cstring>

#include "qmcrt.h"
#include "qmcrt_flow.cuh"
#include "qmcrt_internal.h"

namespace qmcrt {
namespace {

using namespace flow;
// Workspace bytes per row and pass that qmcrt_warp_workspace_bytes states (the gradient keeps
// its tiles on chip and needs the head of it only: the weight sums).
constexpr int ROW_BYTES = 3328;

uint64_t round128(uint64_t r) { return (r + 127) & ~127ull; }

uint64_t bytes_for(uint64_t rows) { return (uint64_t)ROW_BYTES * rows + 8192; }

int rows_for(uint64_t ws_bytes)
{
    if (ws_bytes < bytes_for(128)) return 0;
    uint64_t r = (ws_bytes - 8192) / ROW_BYTES;
    r &= ~127ull;
    return (int)std::min<uint64_t>(r, 1u << 22);
}


// Weight r of layer l of MLP m into the bf16 copies, row-major and transposed.
__device__ __forceinline__ void put_weight(int m, int l, int r, float v, __nv_bfloat16 *__restrict__ wb,
                                           __nv_bfloat16 *__restrict__ wt)
{
    const int o = r / WD, i = r % WD;
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    wb[bf_w(m, l) + r] = b;
    wt[bf_w(m, l) + i * out_dim(l) + o] = b;
}

// Adam, each updated weight put into the bf16 copies at once.
__global__ void __launch_bounds__(256) k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                                              float *__restrict__ v, int n, float lr, float b1, float b2, float eps,
                                              float bc1, float bc2, __nv_bfloat16 *__restrict__ wb,
                                              __nv_bfloat16 *__restrict__ wt)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        p[i] = pi;
        if (i < KB) continue;
        int r = i - KB, mlp = r / mlp_params(), l = 0;
        r -= mlp * mlp_params();
        while (r >= out_dim(l) * WD + out_dim(l)) {
            r -= out_dim(l) * WD + out_dim(l);
            ++l;
        }
        if (r < out_dim(l) * WD) put_weight(mlp, l, r, pi, wb, wt);
    }
}

__global__ void k_sync(const float *__restrict__ p, __nv_bfloat16 *__restrict__ wb, __nv_bfloat16 *__restrict__ wt)
{
    const int total = QMCRT_WARP_BF16_WEIGHTS;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
        int m = e / (3 * WD * WD + KB * WD), r = e % (3 * WD * WD + KB * WD), l = 0;
        while (r >= out_dim(l) * WD) {
            r -= out_dim(l) * WD;
            ++l;
        }
        put_weight(m, l, r, p[param_w(m, l) + r], wb, wt);
    }
}

unsigned blocks(long long n, int t = 256)
{
    long long b = (n + t - 1) / t;
    return (unsigned)std::max(1ll, std::min(b, 152ll * 32));
}

int check_warp(const qmcrt_warp *w)
{
    if (!w || w->struct_size != sizeof(qmcrt_warp)) return set_error(QMCRT_ERR_INVALID_ARG, "warp descriptor");
    if (!w->d_params || !w->d_weights || !w->d_weights_t) return set_error(QMCRT_ERR_INVALID_ARG, "NULL warp buffers");
    if (((uintptr_t)w->d_weights | (uintptr_t)w->d_weights_t) & 15)
        return set_error(QMCRT_ERR_INVALID_ARG, "warp weights must be 16-byte aligned");
    if (!(w->uniform_mix >= 0.0f && w->uniform_mix < 1.0f))
        return set_error(QMCRT_ERR_INVALID_ARG, "uniform_mix must lie in [0, 1)");
    return QMCRT_OK;
}

int launch_status(const char *what)
{
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QMCRT_OK : set_error(QMCRT_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

}  // namespace
}  // namespace qmcrt

using namespace qmcrt;

extern "C" {

uint64_t qmcrt_warp_workspace_bytes(uint64_t rows) { return bytes_for(round128(rows ? rows : 1)); }

int qmcrt_warp_sync(const qmcrt_warp *warp, void *stream)
{
    int rc = check_warp(warp);
    if (rc) return rc;
    k_sync<<<blocks(QMCRT_WARP_BF16_WEIGHTS), 256, 0, (cudaStream_t)stream>>>(
        warp->d_params, (__nv_bfloat16 *)warp->d_weights, (__nv_bfloat16 *)warp->d_weights_t);
    return launch_status("warp sync");
}

int qmcrt_warp_forward(const qmcrt_warp *warp, const float *d_u, float *d_x, float *d_logj, uint64_t n,
                       void *d_workspace, uint64_t workspace_bytes, void *stream)
{
    (void)d_workspace;
    (void)workspace_bytes;
    int rc = check_warp(warp);
    if (rc) return rc;
    if (!d_u || !d_x || !d_logj) return set_error(QMCRT_ERR_INVALID_ARG, "NULL buffer");
    cudaError_t e = launch_warp_forward_fused(warp->d_params, (const __nv_bfloat16 *)warp->d_weights, d_u, d_x,
                                              d_logj, (long long)n, warp->uniform_mix, warp->d_error,
                                              (cudaStream_t)stream);
    if (e != cudaSuccess) return set_error(QMCRT_ERR_CUDA, "warp forward: %s", cudaGetErrorString(e));
    return QMCRT_OK;
}

int qmcrt_warp_grad(const qmcrt_warp *warp, const float *d_x, const float *d_w, uint64_t n, float *d_grad,
                    float *d_loss, void *d_workspace, uint64_t workspace_bytes, void *stream)
{
    int rc = check_warp(warp);
    if (rc) return rc;
    if (!d_x || !d_w || !d_grad || !d_loss || !d_workspace) return set_error(QMCRT_ERR_INVALID_ARG, "NULL buffer");
    const int R = rows_for(workspace_bytes);
    if (R < 128) return set_error(QMCRT_ERR_INVALID_ARG, "workspace below one pass of 128 rows");
    const cudaError_t e =
        launch_warp_train(warp->d_params, (const __nv_bfloat16 *)warp->d_weights, d_x, d_w, (long long)n, R,
                          warp->uniform_mix, d_grad, d_loss, (double *)d_workspace, warp->d_error, (cudaStream_t)stream);
    return e == cudaSuccess ? QMCRT_OK : set_error(QMCRT_ERR_CUDA, "warp grad: %s", cudaGetErrorString(e));
}

int qmcrt_warp_adam(const qmcrt_warp *warp, const float *d_grad, float *d_m, float *d_v, const qmcrt_adam *opt,
                    void *stream)
{
    int rc = check_warp(warp);
    if (rc) return rc;
    if (!d_grad || !d_m || !d_v || !opt || opt->struct_size != sizeof(qmcrt_adam) || opt->step < 1)
        return set_error(QMCRT_ERR_INVALID_ARG, "adam arguments");
    const float bc1 = (float)(1.0 - std::pow(opt->beta1, opt->step));
    const float bc2 = (float)(1.0 - std::pow(opt->beta2, opt->step));
    k_adam<<<blocks(QMCRT_WARP_PARAMS), 256, 0, (cudaStream_t)stream>>>(
        warp->d_params, d_grad, d_m, d_v, QMCRT_WARP_PARAMS, (float)opt->lr, (float)opt->beta1, (float)opt->beta2,
        (float)opt->eps, bc1, bc2, (__nv_bfloat16 *)warp->d_weights, (__nv_bfloat16 *)warp->d_weights_t);
    return launch_status("warp adam");
}

}  // extern "C"
