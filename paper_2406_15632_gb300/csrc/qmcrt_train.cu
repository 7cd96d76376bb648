// qmcrt_train.cu -- loss and gradient of the learned warp (cross-entropy of logged packets),
// forward and backward of both conditionals fused in one tensor-core kernel.
//
// A CTA keeps the four weight matrices of one MLP in shared memory (104 KB) and takes 128-row
// tiles of the minibatch: features, the four layers forward, the loss gradient of the logits,
// the three layers backward, with every activation and backward signal of the tile in shared
// memory (F 16 KB, H1-H3 32 KB each, the logits' gradient 8 KB) and the products' accumulator
// in TMEM.  The weight gradients dW[l] = dP[l]^T H[l] are summed over the tiles of a slice of about
// 512 rows in TMEM (352 columns beside the 128 of the accumulator) and leave at its end as vector
// reductions into the caller's gradient; bias gradients are summed in registers over all of them.
//
// No operand is ever stored twice: a tile [rows][columns] lies in the canonical no-swizzle
// layout (8 x 16-byte core matrices), which the tensor core reads with its rows as M or N and
// its columns as K, or the other way about, by the descriptor alone ("MN-major": the strides
// between core matrices trade places).  So H is the A operand of the next layer and the B
// operand of the weight gradient, dP the A operand of both, W the B operand forward and
// backward.  A backward signal replaces the activation it was masked with.
//
// What bounds it: the chain of a tile, eight products of some hundred cycles each behind an
// epilogue of 16 warps (TMEM read, bias or mask, bf16 packing).  A layer-by-layer form (14 GEMMs
// through HBM, 8 split-K GEMMs, feature, loss and row-sum kernels) moved 0.5 GB and took 560 us
// for 2^16 rows; this 110 us (10 us a tile, two slices a CTA).
//
// The arithmetic is the oracle's bf16 form: bf16 weights, features, hidden activations and
// backward signals, FP32 accumulation, FP32 biases, loss and gradients.
#include <algorithm>

#include "qmcrt.h"
#include "qmcrt_flow.cuh"
#include "qmcrt_gemm.cuh"
#include "qmcrt_internal.h"

namespace qmcrt {
namespace {

using namespace flow;

constexpr int TT = 512;                               // threads: four quarters of the columns x 128 rows
constexpr int ROWS = 128;                             // rows of a tile (TMEM lanes)
constexpr int LAYER_BYTES = WD * WD * 2;
constexpr int WEIGHT_BYTES = 3 * LAYER_BYTES + KB * WD * 2;
constexpr int F_BYTES = ROWS * 2 * BLOB * 2;          // features of MLP 1; MLP 0 uses half
constexpr int H_BYTES = ROWS * WD * 2;
constexpr int DL_BYTES = ROWS * KB * 2;
constexpr int N_BIAS = 3 * WD + KB;
constexpr int SMEM_BYTES = WEIGHT_BYTES + F_BYTES + 3 * H_BYTES + DL_BYTES + N_BIAS * 4 + 32 + 128;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of a CTA");

// TMEM columns: the products' accumulator, then the weight gradients
constexpr uint32_t C_ACC = 0, C_DW2 = 128, C_DW1 = 256, C_DW0 = 384, C_DW3 = 448, TMEM_COLS = 512;

constexpr uint32_t A_MN = 1u << 15, B_MN = 1u << 16;  // instruction descriptor: operand is MN-major

// Byte offset of element (r, c) of a tile with `cols` columns.
__device__ __forceinline__ uint32_t at(int r, int c, int cols)
{
    return (uint32_t)(((r >> 3) * (cols >> 3) + (c >> 3)) * 128 + (r & 7) * 16 + (c & 7) * 2);
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&p);
}

__device__ __forceinline__ void load32(uint32_t addr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// One operand: its address and how far it moves a K step of 16, the leading and stride byte
// offsets of its descriptor.
struct Operand {
    uint32_t addr, step, lbo, sbo;
};
// rows as M or N, columns as K
__device__ __forceinline__ Operand by_rows(uint32_t tile, int cols) { return {tile, 256u, 128u, (uint32_t)(cols >> 3) * 128u}; }
// columns as M or N, rows as K (MN-major)
__device__ __forceinline__ Operand by_cols(uint32_t tile, int cols)
{
    const uint32_t group = (uint32_t)(cols >> 3) * 128u;
    return {tile, 2u * group, group, 128u};
}

// D[tmem] (+)= A . B over K = 16 steps; `add`: whether the first step adds to D.
__device__ __forceinline__ void mma(uint32_t tmem, Operand a, Operand b, uint32_t idesc, int steps, bool add)
{
    for (int s = 0; s < steps; ++s) {
        const uint64_t ad = umma_desc(a.addr + s * a.step, a.lbo, a.sbo);
        const uint64_t bd = umma_desc(b.addr + s * b.step, b.lbo, b.sbo);
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(add || s > 0 ? 1u : 0u)
            : "memory");
    }
}

// Column sums of a bf16 tile, 4 rows x 8 columns a thread, into the thread's running sums; rows
// in an order that spreads a quarter warp's reads over the banks.
__device__ __forceinline__ void add_columns(const uint8_t *tile, int cols, float (&sum)[8])
{
    const int t = threadIdx.x & 255, top = threadIdx.x >> 8, chunks = cols >> 3, c = t % chunks, g = t / chunks;
    if (g >= ROWS / 8) return;
    const uint8_t *core = tile + (g * chunks + c) * 128;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint4 v = *reinterpret_cast<const uint4 *>(core + ((4 * top + i + c) & 7) * 16);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sum[2 * k] += __uint_as_float(w[k] << 16);
            sum[2 * k + 1] += __uint_as_float(w[k] & 0xffff0000u);
        }
    }
}

// The CTA's sums of a bias gradient into dst[cols] in shared memory.
__device__ __forceinline__ void collect_columns(const float (&sum)[8], int cols, float *dst)
{
    const int t = threadIdx.x & 255, chunks = cols >> 3, c = t % chunks;
    if (t - (t & 31) >= chunks * (ROWS / 8)) return;  // a warp without a share
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float s = sum[k];
        for (int o = chunks; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) < chunks) atomicAdd(dst + 8 * c + k, s);
    }
}

// Sum of the weights and of those in each of the 32 bins of x0 (the first density's only data):
// sums[0], sums[1 .. 32].
__global__ void __launch_bounds__(256) k_weight_sums(const float *__restrict__ x, const float *__restrict__ w,
                                                     long long n, double *__restrict__ sums)
{
    __shared__ double s[KB];
    if (threadIdx.x < KB) s[threadIdx.x] = 0.0;
    __syncthreads();
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x) {
        const int b = max(0, min((int)(x[3 * j] * KB), KB - 1));
        atomicAdd(&s[b], (double)w[j]);
    }
    __syncthreads();
    if (threadIdx.x < KB) {
        double t = s[threadIdx.x];
        if (t != 0.0) atomicAdd(sums + 1 + threadIdx.x, t);
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) atomicAdd(sums, t);
    }
}

// The rows in slices, each summed on chip and then added to the caller's gradient: passes of
// `pass` rows, each cut into slices of `rows` rows (the last pass: `rows_last`).  A slice of about
// 512 rows keeps the tensor core's running sums short.
struct Slices {
    long long n, pass;
    int per_pass, rows, rows_last;  // slices of a whole pass; rows of a slice
    long long whole, count;         // slices of all whole passes; of all passes

    __device__ __forceinline__ void range(long long s, long long &r0, long long &r1) const
    {
        const long long p = s < whole ? s / per_pass : n / pass, k = s < whole ? rows : rows_last;
        r0 = p * pass + (s < whole ? s - p * per_pass : s - whole) * k;
        r1 = min(min(r0 + k, (p + 1) * pass), n);
    }
};

// Loss and gradient of the n samples.  CTAs [0, per) train MLP 0, [per, 2 per) MLP 1.
__global__ void __launch_bounds__(TT, 1) k_train(const float *__restrict__ params, const __nv_bfloat16 *__restrict__ wb,
                                                const float *__restrict__ x, const float *__restrict__ w,
                                                const __grid_constant__ Slices slices, int per,
                                                const double *__restrict__ sums, float mix, float *__restrict__ grad,
                                                float *__restrict__ loss, int *__restrict__ error)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint8_t *sW = sm, *sF = sW + WEIGHT_BYTES, *sH = sF + F_BYTES, *sDL = sH + 3 * H_BYTES;
    float *sBias = reinterpret_cast<float *>(sDL + DL_BYTES);
    unsigned long long *sBar = reinterpret_cast<unsigned long long *>(sBias + N_BIAS);
    uint32_t *sTmem = reinterpret_cast<uint32_t *>(sBar + 2);
    int *sFail = reinterpret_cast<int *>(sTmem + 1);
    float *sLoss = reinterpret_cast<float *>(sFail + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m = blockIdx.x >= per ? 1 : 0, cta = blockIdx.x - m * per;
    const int kin = m ? 2 * BLOB : BLOB;  // feature columns that can be nonzero
    const int quarter = warp >> 2, row = (warp & 3) * 32 + lane;

    for (int l = 0; l < 4; ++l) {
        const __nv_bfloat16 *src = wb + bf_w(m, l);
#pragma unroll 4
        for (int v = tid; v < out_dim(l) * (WD / 8); v += TT) {
            const int r = v / (WD / 8), kb = v % (WD / 8);
            *reinterpret_cast<uint4 *>(sW + l * LAYER_BYTES + at(r, kb * 8, WD)) =
                *reinterpret_cast<const uint4 *>(src + (long long)r * WD + kb * 8);
        }
    }
    for (int i = tid; i < N_BIAS; i += TT) {
        const int l = i < 3 * WD ? i / WD : 3;
        sBias[i] = params[param_b(m, l) + i - l * WD];
    }
    if (tid == 0) {
        *sFail = 0;
        *sLoss = 0.0f;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(sBar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(sBar + 1)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(sTmem)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (blockIdx.x == 0 && warp == 1) {
        // the first density: every row of a bin has the same gradient, so the bins' weights do
        float z[KB], q[KB];
        for (int k = 0; k < KB; ++k) z[k] = params[k];
        softmax32(z, q);
        float qb = q[0];
#pragma unroll
        for (int k = 1; k < KB; ++k)
            if (k == lane) qb = q[k];
        const float Qb = mixed(qb, mix), s = (float)(sums[1 + lane] / sums[0]);
        const float sr = s * (mix != 0.0f ? (1.0f - mix) * qb / Qb : 1.0f);
        float all = sr, lo = s != 0.0f ? -s * logf(KB * Qb) : 0.0f;
        for (int o = 16; o; o >>= 1) {
            all += __shfl_xor_sync(0xffffffffu, all, o);
            lo += __shfl_xor_sync(0xffffffffu, lo, o);
        }
        atomicAdd(grad + lane, qb * all - sr);
        if (lane == 0) atomicAdd(loss, lo);
    }

    // everything written to shared memory is visible to the tensor core, and the accumulator's
    // readers are done; one thread then issues the next products
    auto hand_over = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    // barrier 0: the accumulator; barrier 1: the weight gradients
    uint32_t phase[2] = {0, 0};
    bool ok = true;
    auto commit = [&](int b) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(sBar + b))
                     : "memory");
    };
    auto wait = [&](int b) {
        if (!mbar_wait(smem_u32(sBar + b), phase[b])) {
            *reinterpret_cast<volatile int *>(sFail) = 1;
            ok = false;
        }
        phase[b] ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    };
    hand_over();

    const uint32_t tmem = *sTmem, mine = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const uint32_t uF = smem_u32(sF), uDL = smem_u32(sDL);
    const uint32_t uW = smem_u32(sW), uH = smem_u32(sH);
    const uint32_t i128 = umma_idesc_bf16(ROWS, WD), i32 = umma_idesc_bf16(ROWS, KB);
    float db0[8], db1[8], db2[8], db3[8], my_loss = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) db0[k] = db1[k] = db2[k] = db3[k] = 0.0f;
    const double inv_wsum = 1.0 / *sums;
    const bool vec = (reinterpret_cast<uintptr_t>(grad) & 15) == 0;

    for (long long slice = cta; slice < slices.count && ok; slice += per) {
        long long r0, r1;
        slices.range(slice, r0, r1);
        float nx[3], nw;  // the sample of this thread's row (dead rows: weight zero)
        auto fetch = [&](long long j, long long end) {
            const bool in = j < end;
            nx[0] = in ? x[3 * j] : 0.5f;
            nx[1] = in ? x[3 * j + 1] : 0.5f;
            nx[2] = in ? x[3 * j + 2] : 0.5f;
            nw = in ? w[j] : 0.0f;
        };
        fetch(r0 + row, r1);
        for (long long t0 = r0; t0 < r1; t0 += ROWS) {
            const long long j = t0 + row;
            const bool live = j < r1, more = t0 > r0;  // later tiles of a slice add to its weight gradients
            const float px[3] = {nx[0], nx[1], nx[2]}, pw = nw;
            fetch(t0 + ROWS + row, r1);  // the next tile's sample, while this one is computed
            {
                // one-blob features, a quarter of the columns a thread
                const float x0 = px[0], x1 = px[1];
                const int c0 = quarter * (kin >> 2);
                for (int c = c0; c < c0 + (kin >> 2); c += 8) {
                    const float v = c < BLOB ? x0 : x1;
                    const int f = c < BLOB ? c : c - BLOB;
                    *reinterpret_cast<uint4 *>(sF + at(row, c, kin)) =
                        make_uint4(pack2(blob(v, f), blob(v, f + 1)), pack2(blob(v, f + 2), blob(v, f + 3)),
                                   pack2(blob(v, f + 4), blob(v, f + 5)), pack2(blob(v, f + 6), blob(v, f + 7)));
                }
            }
            // forward
#pragma unroll 1
            for (int l = 0; l < 3; ++l) {
                hand_over();
                if (tid == 0) {
                    mma(tmem + C_ACC, l ? by_rows(uH + (l - 1) * H_BYTES, WD) : by_rows(uF, kin),
                        by_rows(uW + l * LAYER_BYTES, WD), i128, l ? WD / 16 : kin / 16, false);
                    commit(0);
                }
                const float4 *bias = reinterpret_cast<const float4 *>(sBias + l * WD + quarter * 32);
                uint8_t *out = sH + l * H_BYTES;
                wait(0);
                float v[32];
                load32(mine + C_ACC + quarter * 32, v);
#pragma unroll
                for (int k = 0; k < 32; k += 8) {
                    const float4 a = bias[k / 4], b = bias[k / 4 + 1];
                    *reinterpret_cast<uint4 *>(out + at(row, quarter * 32 + k, WD)) =
                        make_uint4(pack2(fmaxf(v[k] + a.x, 0.0f), fmaxf(v[k + 1] + a.y, 0.0f)),
                                   pack2(fmaxf(v[k + 2] + a.z, 0.0f), fmaxf(v[k + 3] + a.w, 0.0f)),
                                   pack2(fmaxf(v[k + 4] + b.x, 0.0f), fmaxf(v[k + 5] + b.y, 0.0f)),
                                   pack2(fmaxf(v[k + 6] + b.z, 0.0f), fmaxf(v[k + 7] + b.w, 0.0f)));
                }
            }
            hand_over();
            if (tid == 0) {
                mma(tmem + C_ACC, by_rows(uH + 2 * H_BYTES, WD), by_rows(uW + 3 * LAYER_BYTES, WD), i32, WD / 16, false);
                commit(0);
            }
            const float ww = quarter == 0 && live ? (float)(pw * inv_wsum) : 0.0f;
            const float xv = quarter == 0 && live ? px[1 + m] : 0.5f;
            wait(0);
            if (quarter == 0) {  // loss and d loss / d logits of the row
                float z[KB], q[KB];
                load32(mine + C_ACC, z);
#pragma unroll
                for (int k = 0; k < KB; ++k) z[k] += sBias[3 * WD + k];
                softmax32(z, q);
                const int b = min((int)(xv * KB), KB - 1);
                // d log Q_b / d z_k = r (delta_bk - s_k), r = (1 - mix) s_b / Q_b (1 without mixing)
                float qb = q[0];
#pragma unroll
                for (int k = 1; k < KB; ++k)
                    if (k == b) qb = q[k];
                const float Qb = mixed(qb, mix);
                const float r = mix != 0.0f ? (1.0f - mix) * qb / Qb : 1.0f;
                if (ww != 0.0f) my_loss += -ww * logf(KB * Qb);
                float g[KB];
#pragma unroll
                for (int k = 0; k < KB; ++k) g[k] = -ww * r * ((k == b ? 1.0f : 0.0f) - q[k]);
#pragma unroll
                for (int k = 0; k < KB; k += 8)
                    *reinterpret_cast<uint4 *>(sDL + at(row, k, KB)) =
                        make_uint4(pack2(g[k], g[k + 1]), pack2(g[k + 2], g[k + 3]), pack2(g[k + 4], g[k + 5]),
                                   pack2(g[k + 6], g[k + 7]));
            }
            // backward: the signal of layer l gives, through W[l] and the activation's mask, the
            // signal of layer l - 1, and its weight gradient; the new signal takes the
            // activation's place once that product has read it
#pragma unroll
            for (int l = 3; l >= 1; --l) {
                hand_over();
                const uint32_t hl = uH + l * H_BYTES, hp = hl - H_BYTES;  // layer l's signal, its input
                if (tid == 0) {
                    if (l == 3) {  // dW3^T = H3^T dL, so that M = 128
                        mma(tmem + C_ACC, by_rows(uDL, KB), by_cols(uW + 3 * LAYER_BYTES, WD), i128 | B_MN, KB / 16, false);
                        commit(0);
                        mma(tmem + C_DW3, by_cols(hp, WD), by_cols(uDL, KB), i32 | A_MN | B_MN, ROWS / 16, more);
                    } else {
                        mma(tmem + C_ACC, by_rows(hl, WD), by_cols(uW + l * LAYER_BYTES, WD), i128 | B_MN, WD / 16, false);
                        commit(0);
                        mma(tmem + (l == 2 ? C_DW2 : C_DW1), by_cols(hl, WD), by_cols(hp, WD), i128 | A_MN | B_MN,
                            ROWS / 16, more);
                    }
                    commit(1);
                }
                if (l == 3) add_columns(sDL, KB, db3);  // while the products run
                else if (l == 2) add_columns(sH + 2 * H_BYTES, WD, db2);
                else add_columns(sH + H_BYTES, WD, db1);
                uint8_t *act = sH + (l - 1) * H_BYTES;
                wait(0);
                float v[32];
                load32(mine + C_ACC + quarter * 32, v);
                uint32_t o[16];
#pragma unroll
                for (int k = 0; k < 32; k += 8) {
                    // activations are >= 0: a nonzero half word passes the signal
                    const uint4 h = *reinterpret_cast<const uint4 *>(act + at(row, quarter * 32 + k, WD));
                    const uint32_t hw[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                    for (int p = 0; p < 4; ++p)
                        o[k / 2 + p] = pack2(hw[p] & 0x7fffu ? v[k + 2 * p] : 0.0f,
                                             hw[p] & 0x7fff0000u ? v[k + 2 * p + 1] : 0.0f);
                }
                wait(1);
#pragma unroll
                for (int k = 0; k < 32; k += 8)
                    *reinterpret_cast<uint4 *>(act + at(row, quarter * 32 + k, WD)) =
                        make_uint4(o[k / 2], o[k / 2 + 1], o[k / 2 + 2], o[k / 2 + 3]);
            }
            hand_over();
            if (tid == 0) {
                mma(tmem + C_DW0, by_cols(uH, WD), by_cols(uF, kin), umma_idesc_bf16(ROWS, kin) | A_MN | B_MN, ROWS / 16,
                    more);
                commit(1);
            }
            add_columns(sH, WD, db0);
            wait(1);
            // a wait that gave up ends the CTA together
            if (__syncthreads_or(!ok)) {
                ok = false;
                break;
            }
        }
        if (!ok) break;
        // the slice's weight gradients: TMEM lane = output (dW3: input) index
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
            const uint32_t col = l == 2 ? C_DW2 : l == 1 ? C_DW1 : C_DW0;
            const int cols = l ? WD : kin, use = cols >> 2, c0 = quarter * use;
            float *dst = grad + param_w(m, l) + row * WD + c0;
            float v[32];
            load32(mine + col + c0, v);  // of dW0 a quarter is narrower: the rest belongs to others
#pragma unroll
            for (int k = 0; k < 32; k += 4) {
                if (k >= use) break;
                if (vec)
                    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + k), "f"(v[k]), "f"(v[k + 1]),
                                 "f"(v[k + 2]), "f"(v[k + 3])
                                 : "memory");
                else
                    for (int e = 0; e < 4; ++e) atomicAdd(dst + k + e, v[k + e]);
            }
        }
        float v[32];
        load32(mine + C_DW3, v);
#pragma unroll
        for (int k = 0; k < KB; ++k)
            if ((k >> 3) == quarter) atomicAdd(grad + param_w(m, 3) + k * WD + row, v[k]);
        // (the next slice's products start behind a hand_over)
    }
    // bias gradients and the loss: summed in shared memory first (the CTAs' 16 warps adding to a few
    // hundred addresses each took 90 us of 164)
    float *sDb = reinterpret_cast<float *>(sF);  // the features are done with
    if (ok) {  // uniform
        if (tid < N_BIAS) sDb[tid] = 0.0f;
        __syncthreads();
        collect_columns(db0, WD, sDb);
        collect_columns(db1, WD, sDb + WD);
        collect_columns(db2, WD, sDb + 2 * WD);
        collect_columns(db3, KB, sDb + 3 * WD);
        for (int o = 16; o; o >>= 1) my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
        if (lane == 0) atomicAdd(sLoss, my_loss);
        __syncthreads();
        if (tid < N_BIAS) atomicAdd(grad + param_b(m, tid < 3 * WD ? tid / WD : 3) + (tid < 3 * WD ? tid % WD : tid - 3 * WD), sDb[tid]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
        if (ok) atomicAdd(loss, *sLoss);
        if (*reinterpret_cast<volatile int *>(sFail) && error) atomicExch(error, 1);
    }
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

}  // namespace

cudaError_t launch_warp_train(const float *params, const __nv_bfloat16 *wb, const float *x, const float *w, long long n,
                              long long pass_rows, float mix, float *grad, float *loss, double *sums, int *error,
                              cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaMemsetAsync(sums, 0, (1 + KB) * sizeof(double), s);
    if (e != cudaSuccess) return e;
    k_weight_sums<<<(unsigned)std::min<long long>((n + 255) / 256, 152 * 2), 256, 0, s>>>(x, w, n, sums);
    // a pass of r rows (a multiple of 128) in floor(r / 512) slices, of whole 64-row steps
    auto slice_rows = [](long long r) {
        const long long splits = std::max(1ll, r / 512);
        return (int)(((r + splits - 1) / splits + 63) / 64 * 64);
    };
    Slices sl;
    sl.n = n;
    sl.pass = pass_rows;
    const long long last = n % pass_rows;
    sl.rows = slice_rows(pass_rows);
    sl.per_pass = (int)((pass_rows + sl.rows - 1) / sl.rows);
    sl.rows_last = slice_rows((last + 127) / 128 * 128);
    sl.whole = n / pass_rows * sl.per_pass;
    sl.count = sl.whole + (last ? (last + sl.rows_last - 1) / sl.rows_last : 0);
    // one CTA per SM, half of them for each MLP
    const int per = (int)std::max(1ll, std::min<long long>(sl.count, sms / 2));
    k_train<<<2 * per, TT, SMEM_BYTES, s>>>(params, wb, x, w, sl, per, sums, mix, grad, loss, error);
    return cudaGetLastError();
}

}  // namespace qmcrt
