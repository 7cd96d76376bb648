// qmcrt_sky.cu -- qmcrt_sky_bound: for rays that start within a radius R of the origin (a
// point source, R = 0, or the surface of a star of radius R), an upper bound on the
// optical depth of every ray whose direction falls in each texel of a cube map.  A packet
// whose direction's bound is below the forcing threshold tau_min cannot scatter (Sec. 3.2:
// rays with tau_1 < tau_min are skipped), so the tracer decides that from one lookup
// instead of walking its ray through the grid; the decision, and hence the image, is the
// walk's.
//
// Cube map: face f = 2 a + (d_a < 0) for the major axis a of the direction (ties to the
// lower axis); on it u, v are the other two components (in increasing axis order) divided
// by |d_a|, in [-1, 1]; texel (iu, iv) = floor((u + 1) / 2 m), floor((v + 1) / 2 m).
//
// Construction.  A ray p + t v with |p| <= R and v in a texel stays within R + t alpha of
// the texel's centre ray t u (alpha: the largest angle between u and the texel's corners),
// so as long as R + t alpha <= D h_min inside the grid, the cell it is in at any t is within
// D cells, in every axis, of the cell the centre ray is in at the same t.  With K_D the grid
// maximised over (2 D + 1)^3 neighbourhoods (on the grid grown by D layers), the ray's
// optical depth is at most the integral of K_D along the centre ray through the grown box:
// one walk per texel.  A texel whose cone outgrows the neighbourhoods gets an infinite bound
// (its rays are always walked).
#include <algorithm>
#include <cmath>

#include "qmcrt.h"
#include "qmcrt_internal.h"

namespace qmcrt {

namespace {

// The maximum over 3^3 neighbourhoods (D = 1, every point source) in one pass: a warp takes
// 32 cells of a row (30 outputs), a thread MAX3_ROWS rows, marching along z with the 3 x 3 maxima
// of the last two planes: its own rows by loads, the neighbours' columns by shuffles.  Only
// values kappa rho > 0 raise the maximum (zero, negative and NaN cells count as empty, as in
// the padded grid the walk reads).  One read of the grid and one write of the grown grid; issue
// and HBM are close (256^3: 345 us for three separable passes, 67 with one row a thread,
// 31 now; 20 at the copy rate).
constexpr int MAX3_ROWS = 4, MAX3_WARPS = 4, MAX3_PLANES = 16;
__global__ void __launch_bounds__(32 * MAX3_WARPS) k_max_filter3(const float *__restrict__ in, float *__restrict__ out,
                                                                 int nx, int ny, int nz)
{
    const int gx = nx + 2, gy = ny + 2, gz = nz + 2;
    const int x = (int)blockIdx.x * 30 + (int)threadIdx.x - 1;  // in the grown grid; its cell is x - 1
    const int y0 = ((int)blockIdx.y * MAX3_WARPS + (int)threadIdx.y) * MAX3_ROWS;
    const int z0 = (int)blockIdx.z * MAX3_PLANES;
    const bool inx = x >= 1 && x <= nx;
    const int put = threadIdx.x >= 1 && threadIdx.x <= 30 && x < gx ? min(MAX3_ROWS, gy - y0) : 0;
    float a[MAX3_ROWS], b[MAX3_ROWS];  // 3 x 3 maxima of the last two planes
#pragma unroll
    for (int r = 0; r < MAX3_ROWS; ++r) a[r] = b[r] = 0.0f;
    const float *src = in + ((long long)(z0 - 2) * ny + (y0 - 2)) * nx + (x - 1);  // read inside the grid only
    float *dst = out + ((long long)z0 * gy + y0) * gx + x;
#pragma unroll 2
    for (int o = 0; o < MAX3_PLANES + 2; ++o, src += (long long)nx * ny) {
        const int z = z0 - 2 + o;  // plane z of the grid, the last of three around plane z of the grown grid
        const bool inz = inx && z >= 0 && z < nz;
        float v[MAX3_ROWS + 2];
#pragma unroll
        for (int r = 0; r < MAX3_ROWS + 2; ++r) {  // rows y0 - 2 + r of the grid
            const float w = inz && (unsigned)(y0 - 2 + r) < (unsigned)ny ? __ldg(src + (long long)r * nx) : 0.0f;
            v[r] = w > 0.0f ? w : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < MAX3_ROWS; ++r) {
            const float m = fmaxf(v[r], fmaxf(v[r + 1], v[r + 2]));
            const float c = fmaxf(m, fmaxf(__shfl_up_sync(0xffffffffu, m, 1), __shfl_down_sync(0xffffffffu, m, 1)));
            if (o >= 2 && z < gz && r < put) dst[(long long)r * gx] = fmaxf(c, fmaxf(a[r], b[r]));
            a[r] = b[r];
            b[r] = c;
        }
        if (o >= 2) dst += (long long)gx * gy;
    }
}

// One pass of the separable maximum filter for wider neighbourhoods (a finite star): out = max
// over the 2D + 1 values of `in` along axis `ax` around each cell of the grown grid
// [nz + 2D][ny + 2D][nx + 2D].  In the first pass `in` is the grid itself (read at the offset
// -D, zero outside it).
__global__ void __launch_bounds__(256) k_max_filter(const float *__restrict__ in, float *__restrict__ out, int nx,
                                                    int ny, int nz, int D, int ax, int first)
{
    const int gx = nx + 2 * D, gy = ny + 2 * D, gz = nz + 2 * D;
    const long long total = (long long)gx * gy * gz;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < total;
         c += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(c % gx), y = (int)((c / gx) % gy), z = (int)(c / ((long long)gx * gy));
        float m = 0.0f;
        for (int o = -D; o <= D; ++o) {
            int q[3] = {x, y, z};
            q[ax] += o;
            float v;
            if (first) {
                const int i = q[0] - D, j = q[1] - D, k = q[2] - D;
                v = (i >= 0 && i < nx && j >= 0 && j < ny && k >= 0 && k < nz) ? in[((long long)k * ny + j) * nx + i]
                                                                                 : 0.0f;
            } else {
                v = (q[0] >= 0 && q[0] < gx && q[1] >= 0 && q[1] < gy && q[2] >= 0 && q[2] < gz)
                        ? in[((long long)q[2] * gy + q[1]) * gx + q[0]]
                        : 0.0f;
            }
            if (v > m) m = v;
        }
        out[c] = m;
    }
}

struct SkyGeom {
    float lo[3], h[3];  // the grown box's lower corner, the cell edges
    int n[3];           // cells of the grown box
    float R, tmax, room;  // start radius, longest path inside the grid, R + t alpha stays below room
    int m;
};

// One walk per texel, in float: the set-up in double took most of the 0.79 ms of 6 x 320^2
// texels on the 256^3 disk (FP64 runs at 1/64 of the float rate), and a walk that indexes its
// axis state by the axis keeps it in local memory.  In float with the axes unrolled 381 us, in
// patches of 8 x 4 texels a warp 297, with face parameters by one fused multiply-add and no cell
// counters 200: issue-bound (76 % of the slots).  The geometry runs four cells ahead of the sum, so
// four loads are in flight.  I: a cell's index, 64 bits for grown grids beyond 2^32 cells (a fine grid
// around a large star grows by D layers a side, whatever the grid itself may hold).  The float counts
// of faces are exact up to 2^24 cells an axis; with more no texel passes the test of its cone below
// (a cell is then 1.2e-7 of the longest path, the angle's own margin 1e-6).
constexpr int SKY_BATCH = 4;
template <class I>
__global__ void __launch_bounds__(256) k_sky_walk(const float *__restrict__ K, const __grid_constant__ SkyGeom g,
                                                  double *__restrict__ map)
{
    const int m = g.m;
    const float inf = __int_as_float(0x7f800000);
    // a warp takes patches of 8 x 4 texels: its rays stay closer together than along a row, where
    // on two of the faces every ray reads its own row of the grid
    const unsigned pu = (m + 7) / 8, pv = (m + 3) / 4, patches = 6 * pu * pv, lane = threadIdx.x & 31;
    const unsigned warps = gridDim.x * (blockDim.x / 32);
    for (unsigned p = (blockIdx.x * blockDim.x + threadIdx.x) / 32; p < patches; p += warps) {
        const int f = (int)(p / (pu * pv)), q = (int)(p - f * (pu * pv));
        const int iv = q / (int)pu * 4 + (int)(lane >> 3), iu = q % (int)pu * 8 + (int)(lane & 7);
        if (iu >= m || iv >= m) continue;
        const unsigned t = ((unsigned)f * m + iv) * m + iu;
        const float du = 1.0f / m;  // half a texel
        const float u = (2 * iu + 1) * du - 1.0f, v = (2 * iv + 1) * du - 1.0f;
        // the texel is a convex patch of the face, so its directions lie within the largest
        // angle between its centre (1, u, v) and its corners: sin = |centre x corner| / (|centre| |corner|)
        const float c2 = 1.0f + u * u + v * v;
        float s2 = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float eu = (k & 1) ? du : -du, ev = (k & 2) ? du : -du;
            const float cu = u + eu, cv = v + ev, w = u * ev - v * eu;
            s2 = fmaxf(s2, (w * w + eu * eu + ev * ev) / (c2 * (1.0f + cu * cu + cv * cv)));
        }
        // (each angle is below 60 degrees; the margins cover the float rounding of the sine and
        // of the centre's direction)
        const float alpha = asinf(fminf(sqrtf(s2), 1.0f)) * (1.0f + 1e-5f) + 1e-6f;
        if (!(g.R + g.tmax * alpha <= g.room)) {
            map[t] = (double)inf;
            continue;
        }
        // the centre ray from the origin through the grown box
        const float un = rsqrtf(c2), w = (f & 1) ? -un : un;
        const int ax = f >> 1;
        const float d[3] = {ax == 0 ? w : u * un, ax == 1 ? w : (ax == 0 ? u : v) * un, ax == 2 ? w : v * un};
        float t0 = 0.0f, t1 = inf;
        bool miss = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float lo = g.lo[a], hi = lo + g.n[a] * g.h[a];
            if (d[a] != 0.0f) {
                const float ta = lo / d[a], tb = hi / d[a];
                t0 = fmaxf(t0, fminf(ta, tb));
                t1 = fminf(t1, fmaxf(ta, tb));
            } else if (0.0f < lo || 0.0f >= hi) {
                miss = true;
            }
        }
        t0 *= 1.0f - 1e-6f;  // a little early
        float sum = 0.0f;
        if (!miss && t1 > t0) {
            // per axis: the first face's parameter and the spacing of the faces, faces crossed so
            // far, the next face's parameter, the index step
            float n0[3], dt[3], cnt[3] = {0.0f, 0.0f, 0.0f}, next[3], tend = inf;
            I st[3], off = 0, stride = 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                // a start on a face may pick the cell on either side: the neighbourhood maximum of
                // either bounds the other's cell, and a wrong side is left after a zero length
                const int c = min(max((int)floorf((t0 * d[a] - g.lo[a]) / g.h[a]), 0), g.n[a] - 1);
                const int left = d[a] > 0.0f ? g.n[a] - 1 - c : c;
                n0[a] = next[a] = inf;
                dt[a] = 0.0f;
                if (d[a] != 0.0f) {
                    n0[a] = next[a] = (g.lo[a] + (float)(d[a] > 0.0f ? c + 1 : c) * g.h[a]) / d[a];
                    dt[a] = g.h[a] / fabsf(d[a]);
                    // the face through which the axis leaves the box, as the walk will compute it:
                    // no step is taken from tend on, so none leaves the box
                    tend = fminf(tend, fmaf((float)left, dt[a], n0[a]));
                }
                st[a] = d[a] > 0.0f ? stride : I(0) - stride;
                off += (I)c * stride;
                stride *= (I)g.n[a];
            }
            float tc = t0;
            while (tc < tend) {
                float len[SKY_BATCH];
                I at[SKY_BATCH];
#pragma unroll
                for (int b = 0; b < SKY_BATCH; ++b) {
                    const float tn = fminf(next[0], fminf(next[1], next[2])), te = fminf(tn, tend);
                    at[b] = off;
                    len[b] = fmaxf(te - tc, 0.0f);
                    tc = fmaxf(tc, te);
                    const bool go = tn < tend, x = go && next[0] == tn, y = go && !x && next[1] == tn, z = go && !x && !y;
                    if (x) {  // face parameters from the crossing count, never accumulated
                        off += st[0];
                        cnt[0] += 1.0f;
                        next[0] = fmaf(cnt[0], dt[0], n0[0]);
                    }
                    if (y) {
                        off += st[1];
                        cnt[1] += 1.0f;
                        next[1] = fmaf(cnt[1], dt[1], n0[1]);
                    }
                    if (z) {
                        off += st[2];
                        cnt[2] += 1.0f;
                        next[2] = fmaf(cnt[2], dt[2], n0[2]);
                    }
                }
#pragma unroll
                for (int b = 0; b < SKY_BATCH; ++b) sum += __ldg(K + at[b]) * len[b];
            }
        }
        // the cone ray and the centre ray cover equal lengths per t: the margin covers the
        // float rounding of the segments and of the sum (a few hundred terms); the tracer's
        // test keeps a further factor of two
        map[t] = (double)sum * (1.0 + 1e-4);
    }
}

}  // namespace

int sky_dilation(const double lo[3], const double hi[3], int nx, int ny, int nz, double radius)
{
    const double hmin = std::min((hi[0] - lo[0]) / nx, std::min((hi[1] - lo[1]) / ny, (hi[2] - lo[2]) / nz));
    return 1 + (int)std::ceil(radius / hmin);
}

uint64_t sky_workspace_bytes(int nx, int ny, int nz, int D)
{
    const uint64_t cells = (uint64_t)(nx + 2 * D) * (ny + 2 * D) * (nz + 2 * D);
    return 2 * ((cells * 4 + 255) & ~255ull);
}

cudaError_t launch_sky_bound(const float *k, int nx, int ny, int nz, const double lo[3], const double hi[3],
                             double radius, int m, double *map, void *ws, cudaStream_t s)
{
    const int D = sky_dilation(lo, hi, nx, ny, nz, radius);
    const uint64_t cells = (uint64_t)(nx + 2 * D) * (ny + 2 * D) * (nz + 2 * D);
    float *A = (float *)ws;
    float *B = (float *)((char *)ws + ((cells * 4 + 255) & ~255ull));
    const unsigned grid = (unsigned)std::min<uint64_t>((cells + 255) / 256, 152ull * 32);
    if (D == 1) {
        const dim3 blocks((nx + 2 + 29) / 30, (ny + 2 + MAX3_ROWS * MAX3_WARPS - 1) / (MAX3_ROWS * MAX3_WARPS),
                          (nz + 2 + MAX3_PLANES - 1) / MAX3_PLANES);
        if (blocks.y <= 65535 && blocks.z <= 65535) {
            k_max_filter3<<<blocks, dim3(32, MAX3_WARPS), 0, s>>>(k, A, nx, ny, nz);
        } else {  // an axis of over half a million cells
            k_max_filter<<<grid, 256, 0, s>>>(k, A, nx, ny, nz, D, 0, 1);
            k_max_filter<<<grid, 256, 0, s>>>(A, B, nx, ny, nz, D, 1, 0);
            k_max_filter<<<grid, 256, 0, s>>>(B, A, nx, ny, nz, D, 2, 0);
        }
    } else {
        k_max_filter<<<grid, 256, 0, s>>>(k, A, nx, ny, nz, D, 0, 1);
        k_max_filter<<<grid, 256, 0, s>>>(A, B, nx, ny, nz, D, 1, 0);
        k_max_filter<<<grid, 256, 0, s>>>(B, A, nx, ny, nz, D, 2, 0);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    SkyGeom g;
    g.m = m;
    g.R = (float)(radius * (1.0 + 1e-6));
    const int n[3] = {nx, ny, nz};
    double hmin = 1e300, far2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double h = (hi[a] - lo[a]) / n[a];
        g.lo[a] = (float)(lo[a] - D * h);
        g.n[a] = n[a] + 2 * D;
        g.h[a] = (float)h;
        hmin = std::min(hmin, h);
        const double ext = std::max(std::fabs(lo[a]), std::fabs(hi[a])) + radius;
        far2 += ext * ext;
    }
    const double tmax = std::sqrt(far2);  // from within R of the origin to the farthest point of the grid
    g.tmax = (float)(tmax * (1.0 + 1e-6));
    // the walk's cell boundaries (face parameters recomputed from the cell index, never
    // accumulated: about ten float roundings of coordinates up to tmax, 6e-7 of it) sit within
    // 3e-6 tmax of the exact ones, taken off the room the neighbourhoods leave; in proportion to
    // the box, so that a bound exists or not whatever the unit of length
    g.room = (float)((D * hmin - 3e-6 * tmax) * (1.0 - 1e-6));
    const long long patches = 6LL * ((m + 7) / 8) * ((m + 3) / 4);
    const unsigned tgrid = (unsigned)std::min<long long>((patches + 7) / 8, 152LL * 32);
    if (cells <= 1ull << 32) k_sky_walk<unsigned><<<tgrid, 256, 0, s>>>(A, g, map);
    else k_sky_walk<unsigned long long><<<tgrid, 256, 0, s>>>(A, g, map);
    return cudaGetLastError();
}

}  // namespace qmcrt
