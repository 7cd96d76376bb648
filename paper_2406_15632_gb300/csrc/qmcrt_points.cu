// qmcrt_points.cu -- point-set generation (Sec. 3.1), the final image reduction
// (Sec. 3.6: sums of all replicas, in units of the source luminosity) and the padded
// copy of a density grid.
#include <algorithm>

#include "qmcrt_device.cuh"

namespace qmcrt {

// The [count][dims] block is written a tile of PTS_TILE consecutive, aligned indices at a
// time, consecutive threads at consecutive addresses: the bound is the write stream, as long
// as an element costs few instructions.  One thread per element with the whole index took
// 35 ms for 2^20 x 80 Sobol coordinates in FP32 (0.01 TB/s): a 64-bit division per element,
// and 32 direction numbers from constant memory at as many addresses as the warp holds
// dimensions.
//
// Digital points (Sobol, Niederreiter) are linear over GF(2) in the bits of the index, also
// through the Gray code, so point base + j of an aligned tile is x(base) ^ x(j): the part of
// the base once per tile and dimension, the part of j from two 16-entry tables (its low and
// high four bits) that hold for every tile.
constexpr int PTS_BITS = 8, PTS_TILE = 1 << PTS_BITS, PTS_HALF = 1 << (PTS_BITS / 2);
constexpr uint64_t PTS_CTAS = 152 * 8;  // blocks of 256 threads resident at once
constexpr uint64_t PTS_FEW = 38;        // up to so many tiles, eight blocks take one: two blocks an SM
constexpr unsigned PTS_PARTS = 8;

// Sobol direction numbers in global memory: lanes of a warp read them for different
// dimensions, which constant memory would serve one address at a time.
static __device__ const uint32_t d_sobol_v[QMCRT_GEN_DIMS][32] = QMCRT_GEN_SOBOL_V_INIT;

// x * 2^-32 in FP64, exact, by its bits: the FP64 pipe (1/64 of the float rate) takes one conversion and
// one product a value otherwise, which bounds points of few dimensions.
__device__ __forceinline__ double unit_f64(uint32_t x)
{
    const int n = __clz((int)x);
    const uint32_t f = x << (n & 31);  // the leading bit at 31: 1.xxx times 2^(-1 - n)
    return __hiloint2double(x ? (int)((f >> 11) + ((uint32_t)(1021 - n) << 20)) : 0, (int)(f << 21));
}

template <int FMT>
__device__ __forceinline__ void put_u32(void *out, uint64_t e, uint32_t x)
{
    if (FMT == QMCRT_FMT_U32) ((uint32_t *)out)[e] = x;
    else if (FMT == QMCRT_FMT_F32) ((float *)out)[e] = Mth<float>::from_u32(x);
    else ((double *)out)[e] = unit_f64(x);
}

// Four consecutive values, at an element index that is a multiple of four.
template <int FMT>
__device__ __forceinline__ void put4_u32(void *out, uint64_t e, uint4 w)
{
    if (FMT == QMCRT_FMT_U32) {
        *reinterpret_cast<uint4 *>((uint32_t *)out + e) = w;
    } else if (FMT == QMCRT_FMT_F32) {
        *reinterpret_cast<float4 *>((float *)out + e) =
            make_float4(Mth<float>::from_u32(w.x), Mth<float>::from_u32(w.y), Mth<float>::from_u32(w.z),
                        Mth<float>::from_u32(w.w));
    } else {
        double2 *o = reinterpret_cast<double2 *>((double *)out + e);
        o[0] = make_double2(unit_f64(w.x), unit_f64(w.y));
        o[1] = make_double2(unit_f64(w.z), unit_f64(w.w));
    }
}

// The elements [e0, e1) of a tile's [rows][dims] block, thread by thread: f(e, j, d) for
// element e = j dims + d; j and d advance by the block's stride without a division.  The first of
// them from a float quotient, exact here: e < 2^17 and a half is added, so the quotient is 0.5 / dims
// off a whole number at least, and its rounding 2^-6 / dims at most.
template <class F>
__device__ __forceinline__ void tile_elements(uint32_t e0, uint32_t e1, uint32_t dims, F f)
{
    const float per = 1.0f / (float)dims;
    auto quotient = [&](uint32_t v) { return (uint32_t)(((float)v + 0.5f) * per); };
    const uint32_t sj = quotient(blockDim.x), sd = blockDim.x - sj * dims;
    uint32_t e = e0 + threadIdx.x, j = quotient(e), d = e - j * dims;
    for (; e < e1; e += blockDim.x) {
        f(e, j, d);
        j += sj;
        d += sd;
        if (d >= dims) {
            d -= dims;
            ++j;
        }
    }
}

// Sobol, Owen-scrambled Sobol and Niederreiter points.  VEC: a thread takes four consecutive
// dimensions, with 16-byte reads of the tables and stores; for dimension counts that are a
// multiple of four (every row, and so every table row, then starts on 16 bytes) and an output
// on a 16-byte boundary.  `parts` blocks share a tile of a small output (PTS_PARTS).  2^20 x 80 Sobol
// coordinates in FP32 (49 us at the copy rate): 35 ms one element a thread, 105 us by tiles an element at
// a time, 77 four at a time, 57 (5.9 TB/s) with the base's bits over the lanes of a warp instead of one
// after the other in a thread, which also held up few dimensions (2^24 x 1: 78 -> 60 us) and, in the tables,
// short outputs of many (100 x 256 in FP64: 35 us, 12 so).
template <int KIND, int FMT, bool VEC>
__global__ void __launch_bounds__(256) k_points_net(const __grid_constant__ PointsP P, uint64_t first, uint64_t count,
                                                    void *out, uint32_t parts)
{
    extern __shared__ uint4 s_tab4[];  // [PTS_HALF][dims] low bits, the same for the high bits, [dims] base, seeds
    uint32_t *const s_tab = reinterpret_cast<uint32_t *>(s_tab4);
    const uint32_t (*V)[32] = KIND == QMCRT_NIEDERREITER ? d_nied_v : d_sobol_v;
    const uint32_t dims = (uint32_t)P.dims;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t *lo = s_tab, *hi = lo + PTS_HALF * dims, *bs = hi + PTS_HALF * dims, *sd = bs + dims;
    // a thread a dimension and half: the columns of four bits, their 16 sums by one XOR each
    for (uint32_t q = threadIdx.x; q < 2 * dims; q += blockDim.x) {
        const uint32_t half = q >= dims, d = q - half * dims;
        uint32_t *tab = half ? hi : lo, col[PTS_BITS / 2], x[PTS_HALF];
#pragma unroll
        for (int k = 0; k < PTS_BITS / 2; ++k) {
            const uint32_t bit = half * (PTS_BITS / 2) + k;
            col[k] = __ldg(&V[d][bit]);  // through the Gray code a bit is its own column and the one below
            if (KIND != QMCRT_NIEDERREITER && bit) col[k] ^= __ldg(&V[d][bit - 1]);
        }
        x[0] = 0;
        tab[d] = 0;
#pragma unroll
        for (int a = 1; a < PTS_HALF; ++a) {
            const int low = a & -a;
            x[a] = x[a ^ low] ^ col[low == 1 ? 0 : low == 2 ? 1 : low == 4 ? 2 : 3];
            tab[a * dims + d] = x[a];
        }
    }
    if (KIND == QMCRT_SOBOL_OWEN)
        for (uint32_t d = threadIdx.x; d < dims; d += blockDim.x) sd[d] = owen_seed(P.seed, (int)d);
    const uint64_t t0 = first >> PTS_BITS, t1 = (first + count - 1) >> PTS_BITS;
    const uint32_t part = blockIdx.x % parts, per_part = PTS_TILE / parts;
    for (uint64_t t = t0 + blockIdx.x / parts; t <= t1; t += gridDim.x / parts) {
        const uint64_t base = t << PTS_BITS;
        const uint32_t b32 = (uint32_t)base, g = KIND == QMCRT_NIEDERREITER ? b32 : b32 ^ (b32 >> 1);
        __syncthreads();  // the last tile's elements are done with bs
        // a warp a dimension, a lane a bit
        for (uint32_t d = threadIdx.x / 32; d < dims; d += blockDim.x / 32) {
            const uint32_t x = __reduce_xor_sync(FULL_MASK, (g >> lane) & 1u ? __ldg(&V[d][lane]) : 0u);
            if (lane == 0) bs[d] = x;
        }
        __syncthreads();
        const uint32_t j0 = max(base < first ? (uint32_t)(first - base) : 0u, part * per_part);
        const uint32_t j1 = min((uint32_t)min((uint64_t)PTS_TILE, first + count - base), (part + 1) * per_part);
        if (j0 >= j1) continue;  // uniform
        const uint64_t off = (base - first) * dims;  // modulo 2^64: element e of the tile is off + e
        if (VEC) {
            const uint32_t quads = dims / 4;
            tile_elements(j0 * quads, j1 * quads, quads, [&](uint32_t e, uint32_t j, uint32_t q) {
                const uint4 a = reinterpret_cast<const uint4 *>(bs)[q],
                            b = reinterpret_cast<const uint4 *>(lo)[(j & (PTS_HALF - 1)) * quads + q],
                            c = reinterpret_cast<const uint4 *>(hi)[(j >> (PTS_BITS / 2)) * quads + q];
                uint4 x = make_uint4(a.x ^ b.x ^ c.x, a.y ^ b.y ^ c.y, a.z ^ b.z ^ c.z, a.w ^ b.w ^ c.w);
                if (KIND == QMCRT_SOBOL_OWEN) {
                    const uint4 r = reinterpret_cast<const uint4 *>(sd)[q];
                    x = make_uint4(owen_scramble(x.x, r.x), owen_scramble(x.y, r.y), owen_scramble(x.z, r.z),
                                   owen_scramble(x.w, r.w));
                }
                put4_u32<FMT>(out, off + 4 * e, x);
            });
            continue;
        }
        tile_elements(j0 * dims, j1 * dims, dims, [&](uint32_t e, uint32_t j, uint32_t d) {
            uint32_t x = bs[d] ^ lo[(j & (PTS_HALF - 1)) * dims + d] ^ hi[(j >> (PTS_BITS / 2)) * dims + d];
            if (KIND == QMCRT_SOBOL_OWEN) x = owen_scramble(x, sd[d]);
            put_u32<FMT>(out, off + e, x);
        });
    }
}

// Philox: one block of the generator holds four consecutive dimensions of an index, so a
// thread takes four, and stores them as one vector where every row starts on its boundary
// (2^18 x 80 in FP32: 104 -> 33 us).
template <int FMT>
__global__ void __launch_bounds__(256) k_points_philox(const __grid_constant__ PointsP P, uint64_t first,
                                                       uint64_t count, void *out, uint32_t tile, int vec)
{
    const uint32_t dims = (uint32_t)P.dims, quads = (dims + 3) / 4;
    const uint2 key = make_uint2((uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    for (uint64_t r0 = (uint64_t)blockIdx.x * tile; r0 < count; r0 += (uint64_t)gridDim.x * tile) {
        const uint32_t rows = (uint32_t)min((uint64_t)tile, count - r0);
        tile_elements(0, rows * quads, quads, [&](uint32_t, uint32_t j, uint32_t q) {
            const uint64_t i = first + r0 + j;
            const uint4 w = philox4x32_10(make_uint4((uint32_t)i, (uint32_t)(i >> 32), q, 0u), key);
            const uint64_t e = (r0 + j) * dims + 4 * q;
            if (vec) {
                put4_u32<FMT>(out, e, w);
            } else {
                const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (uint32_t k = 0; k < 4; ++k)
                    if (4 * q + k < dims) put_u32<FMT>(out, e + k, x[k]);
            }
        });
    }
}

// Halton, Hammersley and Faure points (values, no integer form), one element a thread: bound by
// the digit expansions and the FP64 division that rounds each fraction (digits by multiplication
// instead of division, and longer-lived blocks, were 0 to 15 % slower).
template <int KIND, int FMT>
__global__ void __launch_bounds__(256) k_points_digits(const __grid_constant__ PointsP base, uint64_t first,
                                                       uint64_t count, void *out)
{
    PointsP P = base;
    P.kind = KIND;
    const uint64_t total = count * (uint64_t)P.dims;
    for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t j = e / (uint64_t)P.dims;
        const int d = (int)(e - j * (uint64_t)P.dims);
        if (FMT == QMCRT_FMT_F32) ((float *)out)[e] = point<float>(P, first + j, d);
        else ((double *)out)[e] = point_f64(P, first + j, d);
    }
}

__global__ void __launch_bounds__(256) k_image_reduce(const void *acc, int mode, double frac_scale, size_t elems,
                                                     int replicas, double scale, double *out)
{
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < elems; e += (size_t)gridDim.x * blockDim.x) {
        if (mode == QMCRT_ACCUM_I64) {
            const long long *a = (const long long *)acc;
            long long s = 0;
            for (int r = 0; r < replicas; ++r) s += a[(size_t)r * elems + e];
            out[e] = (double)s * frac_scale * scale;
        } else {
            const double *a = (const double *)acc;
            double s = 0.0;
            for (int r = 0; r < replicas; ++r) s += a[(size_t)r * elems + e];
            out[e] = s * scale;
        }
    }
}

// Copy of a grid with `pad` layers of sentinel cells on every side.  Interior: the density, with
// empty, negative and NaN cells as +0 (no sign bit); padding: the sentinel -0.0, whose sign bit
// ends a padded walk.  V: float4 for rows and padding of whole vectors, else float.  Bound by the
// copy: a thread walks the padded array at the grid's stride and carries its place along, rows of any
// length alike, four loads ahead.  A call at 256^3, and on the 17-cell rows of 1 x 1 x 10^6: 79 and 933 us
// with a division an element and 4-byte accesses, 31 and 2150 with a warp a row, 25 and 165 so.
constexpr int PAD_BATCH = 4;  // loads in flight a thread
template <class V>
__device__ __forceinline__ V edge_cells();
template <>
__device__ __forceinline__ float edge_cells<float>() { return -0.0f; }
template <>
__device__ __forceinline__ float4 edge_cells<float4>() { return make_float4(-0.0f, -0.0f, -0.0f, -0.0f); }
__device__ __forceinline__ float clean_cells(float v) { return v > 0.0f ? v : 0.0f; }
__device__ __forceinline__ float4 clean_cells(float4 v)
{
    return make_float4(clean_cells(v.x), clean_cells(v.y), clean_cells(v.z), clean_cells(v.w));
}

template <class V>
__global__ void __launch_bounds__(256) k_pad_grid(const float *__restrict__ k, int nx, int ny, int nz, int pad,
                                                 float *__restrict__ out)
{
    constexpr unsigned W = sizeof(V) / sizeof(float);  // cells of an element
    const unsigned ux = (unsigned)(nx + 2 * pad) / W, py = ny + 2 * pad, pz = nz + 2 * pad;
    const unsigned stride = gridDim.x * blockDim.x, total = ux * py * pz;  // a padded grid holds at most 2^31 cells
    const unsigned sr = stride / ux, sx = stride - sr * ux, sz = sr / py, sy = sr - sz * py;
    unsigned e = blockIdx.x * blockDim.x + threadIdx.x, r = e / ux, x = e - r * ux, z = r / py, y = r - z * py;
    while (e < total) {
        V v[PAD_BATCH];
        unsigned at[PAD_BATCH];
#pragma unroll
        for (int b = 0; b < PAD_BATCH; ++b) {
            const unsigned cx = x * W - pad, cy = y - pad, cz = z - pad;  // beyond the grid: large
            const bool in = cx < (unsigned)nx && cy < (unsigned)ny && cz < (unsigned)nz;  // beyond the array: not
            v[b] = edge_cells<V>();
            if (in) v[b] = clean_cells(__ldg(reinterpret_cast<const V *>(k + ((long long)cz * ny + cy) * nx + cx)));
            at[b] = e;
            e += stride;
            x += sx;
            const unsigned c = x >= ux;
            x -= c * ux;
            y += sy + c;
            const unsigned d = y >= py;
            y -= d * py;
            z += sz + d;
        }
#pragma unroll
        for (int b = 0; b < PAD_BATCH; ++b)
            if (at[b] < total) reinterpret_cast<V *>(out)[at[b]] = v[b];
    }
}

static unsigned grid_for(uint64_t n)
{
    uint64_t g = (n + 255) / 256;
    if (g > 152ull * 64) g = 152ull * 64;  // grid-stride beyond 64 blocks per SM
    return (unsigned)(g ? g : 1);
}

template <int KIND, int FMT>
static void launch_points_net(const PointsP &p, uint64_t first, uint64_t count, void *out, cudaStream_t s)
{
    const uint64_t tiles = ((first + count - 1) >> PTS_BITS) - (first >> PTS_BITS) + 1;
    const unsigned parts = tiles <= PTS_FEW && p.dims >= 16 ? PTS_PARTS : 1;
    const unsigned grid = (unsigned)(tiles < PTS_CTAS ? tiles : PTS_CTAS) * parts;
    const size_t smem = (2 * PTS_HALF + 2) * (size_t)p.dims * sizeof(uint32_t);  // 34 KB at 256 dimensions
    if (p.dims % 4 == 0 && ((uintptr_t)out & 15) == 0)
        k_points_net<KIND, FMT, true><<<grid, 256, smem, s>>>(p, first, count, out, parts);
    else
        k_points_net<KIND, FMT, false><<<grid, 256, smem, s>>>(p, first, count, out, parts);
}

template <int FMT>
static cudaError_t launch_points(const PointsP &p, uint64_t first, uint64_t count, void *out, cudaStream_t s)
{
    switch (p.kind) {
    case QMCRT_SOBOL: launch_points_net<QMCRT_SOBOL, FMT>(p, first, count, out, s); break;
    case QMCRT_SOBOL_OWEN: launch_points_net<QMCRT_SOBOL_OWEN, FMT>(p, first, count, out, s); break;
    case QMCRT_NIEDERREITER: launch_points_net<QMCRT_NIEDERREITER, FMT>(p, first, count, out, s); break;
    case QMCRT_PHILOX: {
        // some hundred instructions a block of the generator: tiles of as many rows as give every
        // thread at most one spread a small output over the chip
        const uint64_t quads = ((uint64_t)p.dims + 3) / 4, tile = 256 / quads, tiles = (count + tile - 1) / tile;
        k_points_philox<FMT><<<(unsigned)(tiles < 152 * 64 ? tiles : 152 * 64), 256, 0, s>>>(
            p, first, count, out, (uint32_t)tile, p.dims % 4 == 0 && ((uintptr_t)out & 15) == 0);
        break;
    }
    case QMCRT_HALTON:
        k_points_digits<QMCRT_HALTON, FMT><<<grid_for(count * (uint64_t)p.dims), 256, 0, s>>>(p, first, count, out);
        break;
    case QMCRT_HAMMERSLEY:
        k_points_digits<QMCRT_HAMMERSLEY, FMT><<<grid_for(count * (uint64_t)p.dims), 256, 0, s>>>(p, first, count, out);
        break;
    default: k_points_digits<QMCRT_FAURE, FMT><<<grid_for(count * (uint64_t)p.dims), 256, 0, s>>>(p, first, count, out);
    }
    return cudaGetLastError();
}

cudaError_t launch_generate_points(const PointsP &p, uint64_t first, uint64_t count, int format, void *out,
                                   cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    if (format == QMCRT_FMT_U32) return launch_points<QMCRT_FMT_U32>(p, first, count, out, s);
    if (format == QMCRT_FMT_F32) return launch_points<QMCRT_FMT_F32>(p, first, count, out, s);
    return launch_points<QMCRT_FMT_F64>(p, first, count, out, s);
}

// Blocks of 256 threads with PAD_BATCH elements each, at most per_sm a multiprocessor: single cells at 32
// (four rounds of resident ones; the set-up's divisions weigh on more: 255^3 33 us, 41 at 128), whole
// vectors at 512 (padding is written faster so: 1 x 4096^2 166 us, 191 at 32).
static unsigned pad_blocks(uint64_t elements, unsigned per_sm)
{
    const uint64_t b = (elements + 256 * PAD_BATCH - 1) / (256 * PAD_BATCH);
    return (unsigned)std::min<uint64_t>(b, 152ull * per_sm);
}

cudaError_t launch_pad_grid(const float *k, int nx, int ny, int nz, int pad, float *out, cudaStream_t s)
{
    const uint64_t cells = (uint64_t)(nx + 2 * pad) * (ny + 2 * pad) * (nz + 2 * pad);
    if (nx % 4 == 0 && pad % 4 == 0 && (((uintptr_t)k | (uintptr_t)out) & 15) == 0)
        k_pad_grid<float4><<<pad_blocks(cells / 4, 512), 256, 0, s>>>(k, nx, ny, nz, pad, out);
    else
        k_pad_grid<float><<<pad_blocks(cells, 32), 256, 0, s>>>(k, nx, ny, nz, pad, out);
    return cudaGetLastError();
}

cudaError_t launch_image_reduce(const void *acc, int mode, double frac_scale, size_t elems, int replicas,
                                double scale, double *out, cudaStream_t s)
{
    if (elems == 0) return cudaSuccess;
    k_image_reduce<<<grid_for(elems), 256, 0, s>>>(acc, mode, frac_scale, elems, replicas, scale, out);
    return cudaGetLastError();
}

}  // namespace qmcrt
