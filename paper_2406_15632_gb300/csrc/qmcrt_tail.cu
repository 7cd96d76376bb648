// qmcrt_tail.cu -- qmcrt_tail_map: for one observer direction k, an upper bound per grid
// cell on the optical depth still ahead of a peel-off walk (Sec. 3.6: every peel-off of a
// trace runs along k to the edge of the grid).  Beyond the dense parts of a medium most of
// such a walk crosses cells whose depth cannot matter (the tenuous atmosphere of a disk,
// empty corners of the box); the map lets the walk stop there, leaving out at most the
// caller's tolerance.
//
// Blocks of TAIL_BLOCK^3 cells hold the largest value of their cells (K_b).  Slabs of
// blocks are taken across the axis a of largest |k_a| / h_a.  Within one slab the walk
// crosses at most TAIL_BLOCK cells along a, so along another axis b it moves by at most
// TAIL_BLOCK (h_a |k_b|) / (h_b |k_a|) <= TAIL_BLOCK cells, one more where its starting
// point lies just below a face and one more for the rounding of near-simultaneous
// crossings: from any cell of a block it stays within nlat_b blocks along b (3 for a moving
// axis, fewer for a slow one, 1 where k_b = 0), and it enters the next slab within them.
// A ray from block C therefore gathers at most
//   B(C) = (TAIL_BLOCK h_a / |k_a|) max K_b(lateral blocks of C's slab)
//          + max B(the same lateral blocks of the next slab),
// summed from the slab k leaves through, with every operation rounded up.
#include <algorithm>
#include <cmath>

#include "qmcrt.h"
#include "qmcrt_internal.h"

namespace qmcrt {

namespace {

struct TailGeom {
    int nb[3];       // blocks per axis
    int a, b, c;     // slab axis and the two lateral axes
    int sa, sb, sc;  // the direction's signs along them (0: no component)
    int lb, lc;      // lateral blocks a ray from one block can reach along b, c (offsets 0 .. l-1)
    long long ta, tb, tc;  // block-index steps along a, b, c
    int na, nbb, nbc;      // blocks along a, b, c
    float path;      // longest path through one slab, rounded up
};

__device__ __forceinline__ long long block_index(const int nb[3], int x, int y, int z)
{
    return ((long long)z * nb[1] + y) * nb[0] + x;
}

// K_b: the largest value of each block's cells (the padded grid holds +0 for empty cells
// and -0 in the padding; neither raises the maximum, so a block that reaches past the grid may
// read its whole cube: pad >= TAIL_BLOCK).  VEC: rows of a block as one 16-byte vector.
template <bool VEC>
__global__ void __launch_bounds__(256) k_tail_block_max(const float *__restrict__ K, int nx, int ny, int pad,
                                                        TailGeom g, float *__restrict__ Kb)
{
    const unsigned px = nx + 2 * pad, py = ny + 2 * pad;  // a padded grid holds at most 2^31 cells
    const unsigned blocks = (unsigned)g.nb[0] * g.nb[1] * g.nb[2];
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < blocks; q += gridDim.x * blockDim.x) {
        const unsigned w = q / g.nb[0], bx = q - w * g.nb[0], bz = w / g.nb[1], by = w - bz * g.nb[1];
        const float *base = K + ((bz * TAIL_BLOCK + pad) * py + (by * TAIL_BLOCK + pad)) * px + (bx * TAIL_BLOCK + pad);
        float m = 0.0f;
#pragma unroll
        for (unsigned z = 0; z < TAIL_BLOCK; ++z)
#pragma unroll
            for (unsigned y = 0; y < TAIL_BLOCK; ++y) {
                const float *row = base + (z * py + y) * px;
                if (VEC) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(row));
                    m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                } else {
#pragma unroll
                    for (int x = 0; x < TAIL_BLOCK; ++x) m = fmaxf(m, __ldg(row + x));
                }
            }
        Kb[q] = m;
    }
}

// The lateral maxima of every slab, into the place of the slab's bounds: the part of the
// recurrence that does not depend on the slab before.
__global__ void __launch_bounds__(256) k_tail_lateral(const float *__restrict__ Kb, TailGeom g, float *__restrict__ Bb)
{
    const unsigned blocks = (unsigned)g.nb[0] * g.nb[1] * g.nb[2];
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < blocks; q += gridDim.x * blockDim.x) {
        const unsigned w = q / g.nb[0];
        const int at[3] = {(int)(q - w * g.nb[0]), (int)(w % g.nb[1]), (int)(w / g.nb[1])};
        const int ib = g.b == 0 ? at[0] : at[1], ic = g.c == 2 ? at[2] : at[1];
        float m = 0.0f;
        for (int ob = 0; ob < g.lb; ++ob) {
            if ((unsigned)(ib + g.sb * ob) >= (unsigned)g.nbb) break;
            for (int oc = 0; oc < g.lc; ++oc) {
                if ((unsigned)(ic + g.sc * oc) >= (unsigned)g.nbc) break;
                m = fmaxf(m, __ldg(Kb + (long long)q + g.sb * ob * g.tb + g.sc * oc * g.tc));
            }
        }
        Bb[q] = m;
    }
}

// The slab recurrence, one block of threads: slab after slab against the direction, every
// block of a slab in parallel.  The bounds of the slab before are kept in shared memory and
// maximised along one lateral axis, then along the other, inside a margin of zeros that takes
// the place of bounds checks; a thread's lateral maxima of the next slab are loaded before it
// waits.  Serial over the slabs on one SM: at 64 slabs of 64 x 64 blocks 57 us (380 with nine
// reads a block through L2, 105 with checked offsets).  With 16 blocks a thread (slabs of up to 128 x 128;
// 64 registers do not hold their state) it is still twice as fast as the form through global memory:
// a whole map of 512^3 cells takes 1.18 against 2.73 ms, of 300^3 0.34 against 0.62.
constexpr int SLAB_MARGIN = 2;  // lateral offsets reach 2 blocks either way
__host__ __device__ constexpr int slab_words(int nbb, int nbc)
{
    return (nbb + 2 * SLAB_MARGIN) * (nbc + 2 * SLAB_MARGIN);
}

template <int PER>
__global__ void __launch_bounds__(1024) k_tail_slabs(TailGeom g, float *__restrict__ Bb)
{
    extern __shared__ float s_slab[];  // bounds of the slab before, then their maxima along b
    const int na = g.na, nbb = g.nbb, per_slab = g.nbb * g.nbc, pitch = nbb + 2 * SLAB_MARGIN;
    float *B = s_slab, *M = s_slab + slab_words(nbb, g.nbc);
    for (int t = threadIdx.x; t < 2 * slab_words(nbb, g.nbc); t += 1024) s_slab[t] = 0.0f;
    // an axis the ray moves along by fewer blocks repeats an offset: the maximum is the same
    const int b1 = g.lb > 1 ? g.sb : 0, b2 = g.lb > 2 ? 2 * g.sb : b1;
    const int c1 = g.lc > 1 ? g.sc * pitch : 0, c2 = g.lc > 2 ? 2 * g.sc * pitch : c1;
    int at[PER];      // index in the slab's array, 0 for no block
    long long to[PER];  // index in Bb
    float k[PER];
    const long long down = g.sa > 0 ? -g.ta : g.ta;  // to the slab after this one
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int t = threadIdx.x + p * 1024, ic = t / nbb, ib = t - ic * nbb;
        at[p] = t < per_slab ? (ic + SLAB_MARGIN) * pitch + ib + SLAB_MARGIN : 0;
        to[p] = (g.sa > 0 ? na - 1 : 0) * g.ta + ib * g.tb + ic * g.tc;  // the exit side first
        k[p] = at[p] ? Bb[to[p]] : 0.0f;
    }
    __syncthreads();
    for (int step = 0; step < na; ++step) {
        float ahead[PER];
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            ahead[p] = at[p] && step + 1 < na ? Bb[to[p] + down] : 0.0f;
            if (at[p]) M[at[p]] = fmaxf(B[at[p]], fmaxf(B[at[p] + b1], B[at[p] + b2]));
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            if (at[p]) {
                const float m = fmaxf(M[at[p]], fmaxf(M[at[p] + c1], M[at[p] + c2]));
                const float b = __fadd_ru(__fmul_ru(k[p], g.path), m);
                B[at[p]] = b;
                Bb[to[p]] = b;
            }
            to[p] += down;
            k[p] = ahead[p];
        }
        __syncthreads();
    }
}

// The same recurrence through global memory, for slabs too large for shared memory.
__global__ void __launch_bounds__(1024) k_tail_slabs_wide(TailGeom g, float *__restrict__ Bb)
{
    const int na = g.na, nbb = g.nbb, nbc = g.nbc;
    const int per_slab = nbb * nbc;
    for (int step = 0; step < na; ++step) {
        const int j = g.sa > 0 ? na - 1 - step : step;  // the exit side first
        const int jn = j + g.sa;                          // the slab a ray from slab j enters next
        for (int t = threadIdx.x; t < per_slab; t += blockDim.x) {
            const int ib = t % nbb, ic = t / nbb;
            float nmax = 0.0f;
            for (int ob = 0; step && ob < g.lb; ++ob) {
                const int qb = ib + g.sb * ob;
                if (qb < 0 || qb >= nbb) continue;
                for (int oc = 0; oc < g.lc; ++oc) {
                    const int qc = ic + g.sc * oc;
                    if (qc < 0 || qc >= nbc) continue;
                    nmax = fmaxf(nmax, Bb[jn * g.ta + qb * g.tb + qc * g.tc]);
                }
            }
            float *b = Bb + j * g.ta + ib * g.tb + ic * g.tc;
            *b = __fadd_ru(__fmul_ru(*b, g.path), nmax);
        }
        __syncthreads();
    }
}

// Code of a bound: c = (biased exponent of B, at least 1) + 24, so that B < 2^(c - 150); 0 for
// B = 0; 255 above 2^104 or not finite.
__device__ __forceinline__ uint32_t tail_code(float B)
{
    if (!(B <= 3.0e38f)) return 255u;
    if (!(B > 0.0f)) return 0u;
    const int E = (int)((__float_as_uint(B) >> 23) & 0xffu);
    const int c = max(E, 1) + 24;
    return c > 254 ? 255u : (uint32_t)c;
}

// Codes of the padded grid's cells (0 in the padding), a warp per row: the row's blocks are
// found once, and VEC writes the four cells of a block, which share its code, as one word
// (rows and padding of whole blocks).  16 us at 256^3 (79 with divisions and a
// byte store a cell).
template <bool VEC>
__global__ void __launch_bounds__(256) k_tail_expand(const float *__restrict__ Bb, int nx, int ny, int nz, int pad,
                                                     TailGeom g, uint8_t *__restrict__ map)
{
    const int px = nx + 2 * pad, py = ny + 2 * pad, pz = nz + 2 * pad;
    const long long rows = (long long)py * pz;
    const int lane = threadIdx.x & 31;
    for (long long r = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += (long long)gridDim.x * 8) {
        const int z = (int)(r / py) - pad, y = (int)(r % py) - pad;
        const bool in = z >= 0 && z < nz && y >= 0 && y < ny;
        const float *src = Bb + block_index(g.nb, 0, in ? y / TAIL_BLOCK : 0, in ? z / TAIL_BLOCK : 0);
        uint8_t *dst = map + r * px;
        if (VEC) {
            for (int v = lane; v < px / 4; v += 32) {
                const int x = 4 * v - pad;
                const uint32_t code = in && x >= 0 && x < nx ? tail_code(__ldg(src + x / TAIL_BLOCK)) : 0u;
                reinterpret_cast<uint32_t *>(dst)[v] = code * 0x01010101u;
            }
        } else {
            for (int c = lane; c < px; c += 32) {
                const int x = c - pad;
                dst[c] = (uint8_t)(in && x >= 0 && x < nx ? tail_code(__ldg(src + x / TAIL_BLOCK)) : 0u);
            }
        }
    }
}

template <int PER>
cudaError_t launch_slabs(const TailGeom &g, float *Bb, cudaStream_t s)
{
    const size_t smem = 2 * sizeof(float) * (size_t)slab_words(g.nbb, g.nbc);
    if (smem > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_tail_slabs<PER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_tail_slabs<PER><<<1, 1024, smem, s>>>(g, Bb);
    return cudaGetLastError();
}

int blocks_of(int n) { return (n + TAIL_BLOCK - 1) / TAIL_BLOCK; }

uint64_t aligned(uint64_t bytes) { return (bytes + 255) & ~255ull; }

}  // namespace

uint64_t tail_workspace_bytes(int nx, int ny, int nz)
{
    const uint64_t blocks = (uint64_t)blocks_of(nx) * blocks_of(ny) * blocks_of(nz);
    return 2 * aligned(blocks * sizeof(float));
}

cudaError_t launch_tail_map(const float *k_padded, int nx, int ny, int nz, int pad, const double lo[3],
                            const double hi[3], const double dir[3], uint8_t *map, void *ws, cudaStream_t s)
{
    TailGeom g;
    const int n[3] = {nx, ny, nz};
    double h[3], speed[3];
    for (int q = 0; q < 3; ++q) {
        g.nb[q] = blocks_of(n[q]);
        h[q] = (hi[q] - lo[q]) / n[q];
        speed[q] = std::fabs(dir[q]) / h[q];  // cells crossed per unit path
    }
    g.a = 0;
    for (int q = 1; q < 3; ++q)
        if (speed[q] > speed[g.a]) g.a = q;
    g.b = g.a == 0 ? 1 : 0;
    g.c = g.a == 2 ? 1 : 2;
    auto sgn = [](double v) { return v > 0 ? 1 : (v < 0 ? -1 : 0); };
    const long long step[3] = {1, g.nb[0], (long long)g.nb[0] * g.nb[1]};
    g.na = g.nb[g.a];
    g.nbb = g.nb[g.b];
    g.nbc = g.nb[g.c];
    g.ta = step[g.a];
    g.tb = step[g.b];
    g.tc = step[g.c];
    g.sa = sgn(dir[g.a]);
    g.sb = sgn(dir[g.b]);
    g.sc = sgn(dir[g.c]);
    auto lateral = [&](int q) {
        if (dir[q] == 0.0) return 1;
        const double r = speed[q] / speed[g.a] * (1.0 + 1e-9);  // <= 1 by the choice of a
        const int reach = (TAIL_BLOCK - 1) + (int)std::floor(TAIL_BLOCK * r) + 2;  // farthest cell offset
        return 1 + reach / TAIL_BLOCK;
    };
    g.lb = lateral(g.b);
    g.lc = lateral(g.c);
    const double path = TAIL_BLOCK * h[g.a] / std::fabs(dir[g.a]) * (1.0 + 1e-6);
    g.path = std::nextafter((float)path, 3.0e38f);
    float *Kb = (float *)ws;
    const uint64_t blocks = (uint64_t)g.nb[0] * g.nb[1] * g.nb[2];
    float *Bb = (float *)((char *)ws + aligned(blocks * sizeof(float)));
    const unsigned bgrid = (unsigned)std::min<uint64_t>((blocks + 255) / 256, 152ull * 16);
    // whole vectors: a row of the padded grid, its padding and every block start on one
    const bool whole = nx % TAIL_BLOCK == 0 && pad % TAIL_BLOCK == 0;
    if (whole && ((uintptr_t)k_padded & 15) == 0) k_tail_block_max<true><<<bgrid, 256, 0, s>>>(k_padded, nx, ny, pad, g, Kb);
    else k_tail_block_max<false><<<bgrid, 256, 0, s>>>(k_padded, nx, ny, pad, g, Kb);
    k_tail_lateral<<<bgrid, 256, 0, s>>>(Kb, g, Bb);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const long long per_slab = (long long)g.nbb * g.nbc;
    // a slab of up to 16 blocks a thread whose margins fit shared memory (128 x 128 blocks, a
    // 512^3 grid, take 136 KB)
    if (per_slab > 16 * 1024 || 8ull * (g.nbb + 2 * SLAB_MARGIN) * (g.nbc + 2 * SLAB_MARGIN) > 200 * 1024)
        k_tail_slabs_wide<<<1, 1024, 0, s>>>(g, Bb);
    else if (per_slab <= 1024) e = launch_slabs<1>(g, Bb, s);
    else if (per_slab <= 4 * 1024) e = launch_slabs<4>(g, Bb, s);
    else e = launch_slabs<16>(g, Bb, s);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const uint64_t rows = (uint64_t)(ny + 2 * pad) * (nz + 2 * pad);
    const unsigned egrid = (unsigned)std::min<uint64_t>((rows + 7) / 8, 152ull * 16);
    if (whole && ((uintptr_t)map & 3) == 0) k_tail_expand<true><<<egrid, 256, 0, s>>>(Bb, nx, ny, nz, pad, g, map);
    else k_tail_expand<false><<<egrid, 256, 0, s>>>(Bb, nx, ny, nz, pad, g, map);
    return cudaGetLastError();
}

}  // namespace qmcrt
