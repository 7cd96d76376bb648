// qmcrt_wavefront.cu -- multiple scattering as a wavefront of orders (Sec. 3.5, 3.7).
//
// The one-kernel tracer keeps a packet on one thread for all its orders.  Its first
// order is coherent (net-ordered warps start 32 packets in nearly the same direction),
// but from the second order on each lane scatters into its own direction and the warp
// waits for its longest walk.  Here every order is a launch over the packets still
// alive, and between orders the live packets are regrouped by a key built from their
// position (up to 16^3 cells of the box) and their new direction (up to 32 bins in cos theta
// x 64 in phi), so a warp again traces 32 similar rays:
//
//   order 1:   emission, forced step, peel-off, roulette, scattering for order 2 ->
//              queue (with each packet's key, counted in the bucket histogram)
//   order k:   bucket cursors -> record indices into
//              buckets -> forced step (or march), peel-off, roulette, scattering for
//              k+1 -> the other queue
//
// A queued packet is one 64-byte record (128 in FP64) that stays where it was appended:
// the sort moves 4-byte indices, and order k gathers its records through them (two
// whole sectors per record), appending the survivors to the other queue.
//
// Per packet the arithmetic is the one-kernel tracer's, step for step (the scattering
// that opens order k runs at the end of order k-1), so fixed-point images are identical.
// Launch sizes do not depend on the live counts, which stay on the device: the order
// kernels are persistent and read their count when they start.
#include <algorithm>

#include "qmcrt_device.cuh"
#include "qmcrt_support.cuh"

namespace qmcrt {

namespace {

// The regrouping key: position cells of the box, 2^pos per axis, then direction bins, 2^cos in
// cos theta and 2^phi in phi; position-major, so that packets that start close together in
// nearly one direction, which cross nearly the same cells, are traced by one warp and share
// cache lines.  The finest split suits the largest queues; the buckets are cleared and
// scanned once an order whatever the queue holds, so a smaller one takes fewer (wave_bits).
struct WaveKey {
    int pos, cos, phi;  // bits
    int shift;          // low bits of the key dropped (queues too small to hold the cursors)
};
constexpr int WV_MAX_BITS = 23, WV_MAX_BUCKETS = 1 << WV_MAX_BITS;
constexpr int WV_TAIL_BYTES = WV_MAX_BUCKETS / 256;  // counters, behind the histogram

__host__ __device__ constexpr int key_bits(const WaveKey &K) { return 3 * K.pos + K.cos + K.phi - K.shift; }

template <class T>
struct Packet {
    T pos[3], n[3], a[3], S[3], tot, tot2;
};

// One queued packet: its state and its index, one contiguous record (64 bytes in FP32,
// 128 in FP64) moved with 16-byte vector accesses.
template <class T>
struct alignas(16) Rec {
    Packet<T> p;
    uint32_t j;  // point index - first
    uint32_t pad[sizeof(T) == 4 ? 1 : 3];
};
static_assert(sizeof(Rec<float>) == 64 && sizeof(Rec<double>) == 128, "record size");

// Counters of one order: packets appended for it, its chunk counter, its bucket space taken.
struct WaveCount {
    uint32_t live, chunk, space, pad;
};
static_assert(67 * sizeof(WaveCount) <= WV_TAIL_BYTES, "counters of every order (at most 64) and one more, the support");

template <class T>
struct WaveWork {
    Rec<T> *q[2];       // [cap] each: order k reads q[(k + 1) & 1] and appends to q[k & 1]
    WaveCount *count;   // [order]
    uint32_t *keys;     // [cap] bucket of each appended record
    uint32_t *perm;     // [cap] record indices of the queue being read, in bucket order
    uint32_t *hist;     // [buckets] histogram of the appended records
    WaveKey key;
};

template <class T>
__device__ __forceinline__ void copy_rec(Rec<T> *dst, const Rec<T> *src)
{
    const uint4 *s = reinterpret_cast<const uint4 *>(src);
    uint4 *d = reinterpret_cast<uint4 *>(dst);
#pragma unroll
    for (int v = 0; v < (int)(sizeof(Rec<T>) / 16); ++v) d[v] = s[v];
}

// The low six bits of v at the even bit positions.
__device__ __forceinline__ uint32_t spread2(uint32_t v)
{
    v = (v | (v << 4)) & 0x30fu;
    v = (v | (v << 2)) & 0x333u;
    return (v | (v << 1)) & 0x555u;
}

template <class T>
__device__ __forceinline__ uint32_t wave_key(const MediumP<T> &G, const WaveKey &K, const T pos[3], const T n[3])
{
    const int NP = 1 << K.pos, NC = 1 << K.cos, NF = 1 << K.phi;
    uint32_t key = 0;
    for (int c = 0; c < 3; ++c) {
        const T f = (pos[c] - G.lo[c]) / (G.hi[c] - G.lo[c]) * T(NP);
        key = (key << K.pos) | (uint32_t)min(NP - 1, max(0, (int)f));
    }
    const int ct = min(NC - 1, max(0, (int)((n[2] + T(1)) * T(NC) * T(0.5))));
    const float ph = atan2f((float)n[1], (float)n[0]);  // the key only orders packets
    const int pb = min(NF - 1, max(0, (int)((ph + 3.14159265f) * ((float)NF * 0.159154943f))));
    // cos theta and phi bits interleaved: a run of records is a patch of directions rather than a
    // thin ring (1.2 % of the 2^22-packet clumpy run)
    return ((key << (K.cos + K.phi)) | spread2((uint32_t)pb) | (spread2((uint32_t)ct) << 1)) >> K.shift;
}

// Append the lanes with `keep` to queue dst, the queue of order k + 1, with their bucket keys
// and count them in the histogram of the next sort (one queue atomic per warp).  All 32 lanes
// call.
template <class T>
__device__ __forceinline__ void append(const TraceP<T> &P, const WaveWork<T> &W, int k, Rec<T> *dst, bool keep,
                                       const Packet<T> &p, uint32_t j)
{
    const unsigned m = __ballot_sync(FULL_MASK, keep);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int first = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == first) base = atomicAdd(&W.count[k + 1].live, (uint32_t)__popc(m));
    base = __shfl_sync(FULL_MASK, base, first);
    const uint32_t key = keep ? wave_key(P.med, W.key, p.pos, p.n) : 0xffffffffu;
    // lanes with equal keys count into the histogram with one atomic (a warp's
    // packets come from one bucket of the last sort and mostly share their key)
    const unsigned peers = __match_any_sync(FULL_MASK, key);
    if (keep) {
        const uint32_t q = base + __popc(m & ((1u << lane) - 1u));
        Rec<T> r;
        r.p = p;
        r.j = j;
        for (int c = 0; c < (int)(sizeof(r.pad) / 4); ++c) r.pad[c] = 0u;
        copy_rec(dst + q, &r);
        W.keys[q] = key;
        if (lane == __ffs(peers) - 1) atomicAdd(W.hist + key, (uint32_t)__popc(peers));
    }
}

template <class T>
__device__ __forceinline__ void write_log(const TraceP<T> &P, uint64_t i, uint64_t j, const Packet<T> &p)
{
    float *r = P.train_log + 5 * j;
    if (P.warp_x) {
        r[0] = P.warp_x[3 * j];
        r[1] = P.warp_x[3 * j + 1];
        r[2] = P.warp_x[3 * j + 2];
    } else {
        r[0] = (float)point<T>(P.pts, i, 0);
        r[1] = (float)point<T>(P.pts, i, 1);
        r[2] = (float)point<T>(P.pts, i, 2);
    }
    r[3] = (float)p.tot;
    r[4] = (float)Mth<T>::sqrt_(p.tot2);
}

// Order k of a packet that is alive at its start (scattered already if k > 1), with
// depth coordinate wd; then roulette and the scattering that opens order k + 1.  All 32
// lanes call (the peel-off bins into the image).  Returns whether it lives on.
template <class T>
__device__ __forceinline__ bool run_order(const TraceP<T> &P, int k, uint64_t i, bool alive, T wd, Packet<T> &p)
{
    const int base = 4 * (k - 1);
    if (alive) {
        if (k == 1 || P.force_all) {
            T W1;
            if (forced_step<T, true>(P, p.pos, p.n, wd, W1)) {
                p.S[0] *= W1;
                p.S[1] *= W1;
                p.S[2] *= W1;
            } else {
                alive = false;
            }
        } else if (!march(P.med, p.pos, p.n, -Mth<T>::log_(wd))) {
            alive = false;
        }
        if (alive) {
            p.S[0] *= P.dust.albedo;
            p.S[1] *= P.dust.albedo;
            p.S[2] *= P.dust.albedo;
        }
    }
    T out[3] = {T(0), T(0), T(0)};
    T x = T(0), y = T(0);
    const bool contrib = alive && peel_polarized<T, true>(P, p.pos, p.n, p.a, p.S, out, x, y);
    if (contrib && x >= -P.obs.hw && x < P.obs.hw && y >= -P.obs.hw && y < P.obs.hw) {
        p.tot += out[0];
        p.tot2 += out[0] * out[0];
    }
    splat(P, contrib, P.per_order ? k - 1 : 0, x, y, out);
    if (alive) {
        if (k == P.max_orders) {
            alive = false;
        } else if (p.S[0] < P.rr_threshold) {
            if (point<T>(P.pts, i, base + 3) < P.rr_survival) {
                p.S[0] /= P.rr_survival;
                p.S[1] /= P.rr_survival;
                p.S[2] /= P.rr_survival;
            } else {
                alive = false;
            }
        }
    }
    if (alive) scatter(P.dust, point<T>(P.pts, i, base + 4), point<T>(P.pts, i, base + 5), p.n, p.a, p.S);
    return alive;
}

template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_wave_first(const __grid_constant__ TraceP<T> P, WaveWork<T> W)
{
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if ((tid & ~31ull) >= P.ord.threads) return;  // uniform per warp
    uint64_t i = P.first;
    const bool live = packet_index(P.ord, P.first, P.count, tid, i);
    if (!__any_sync(FULL_MASK, live)) return;
    const uint64_t j = i - P.first;
    Packet<T> p;
    for (int c = 0; c < 3; ++c) p.pos[c] = p.a[c] = p.S[c] = T(0);
    p.n[0] = p.n[1] = T(0);
    p.n[2] = T(1);
    p.a[0] = T(1);
    p.tot = p.tot2 = T(0);
    T wd = T(0);
    if (live) {
        T wgt;
        if (P.warp_x) {  // learned proposal: first-order coordinates and their Jacobian
            T sp, cp;
            direction_from((T)P.warp_x[3 * j], (T)P.warp_x[3 * j + 1], p.n, p.a, sp, cp);
            wd = (T)P.warp_x[3 * j + 2];
            wgt = Mth<T>::exp_((T)P.warp_logj[j]);
        } else {
            const int e = 4 * P.max_orders;  // a finite star's two extra emission coordinates
            wd = emit(P, i, p.pos, p.n, p.a, wgt, e, e + 1, 2);
        }
        p.S[0] = wgt;
    }
    const bool on = run_order(P, 1, i, live, wd, p);
    append(P, W, 1, W.q[1], on, p, (uint32_t)j);
    if (live && !on && P.train_log) write_log(P, i, j, p);
}

// Bucket cursors of the queue for order k: every block scans a tile of buckets in order and
// takes the tile's space from one counter (tiles may end up in any order: only packets of
// one tile need to be close), clearing the histogram behind it for the next sort.  The cursors
// lie in the queue that order k will append to.  Bound by the L2 pass over the buckets, of
// which it writes only those that hold records.
constexpr int WV_TILE = 4096, WV_PER = WV_TILE / 256;
__global__ void __launch_bounds__(256) k_wave_cursors(uint32_t *__restrict__ hist, uint32_t *__restrict__ cursor,
                                                      int buckets, WaveCount *cnt)
{
    __shared__ uint32_t s_warp[8], s_base;
    const int t = threadIdx.x, lane = t & 31;
    const int b0 = blockIdx.x * WV_TILE + t * WV_PER;
    uint4 v[WV_PER / 4];
    uint32_t sum = 0;
#pragma unroll
    for (int q = 0; q < WV_PER / 4; ++q) {
        v[q] = b0 + 4 * q < buckets ? *reinterpret_cast<const uint4 *>(hist + b0 + 4 * q) : make_uint4(0, 0, 0, 0);
        sum += v[q].x + v[q].y + v[q].z + v[q].w;
    }
    uint32_t run = sum;  // inclusive over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(FULL_MASK, run, o);
        if (lane >= o) run += x;
    }
    if (lane == 31) s_warp[t >> 5] = run;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        if (w < (t >> 5)) before += s_warp[w];
        all += s_warp[w];
    }
    if (t == 0) s_base = all ? atomicAdd(&cnt->space, all) : 0u;
    __syncthreads();
    if (!sum) return;  // empty buckets have no record to place
    run += s_base + before - sum;
#pragma unroll
    for (int q = 0; q < WV_PER / 4; ++q) {
        const uint4 x = v[q];
        if (!(x.x | x.y | x.z | x.w)) continue;
        uint4 c;
        c.x = run;
        c.y = c.x + x.x;
        c.z = c.y + x.y;
        c.w = c.z + x.z;
        run = c.w + x.w;
        *reinterpret_cast<uint4 *>(cursor + b0 + 4 * q) = c;
        *reinterpret_cast<uint4 *>(hist + b0 + 4 * q) = make_uint4(0, 0, 0, 0);
    }
}

// Bucket order of the appended records: perm[cursor of its key] = record index, one
// cursor atomic per run of equal keys in a warp.
__global__ void __launch_bounds__(256) k_wave_scatter(const uint32_t *__restrict__ keys, uint32_t *__restrict__ cursor,
                                                      uint32_t *__restrict__ perm, const WaveCount *__restrict__ cnt)
{
    const uint32_t n = cnt->live;
    const int lane = threadIdx.x & 31;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t q0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); q0 < n; q0 += stride) {  // uniform per warp
        const uint32_t q = q0 + lane;
        const bool v = q < n;
        const uint32_t key = v ? keys[q] : 0xffffffffu;
        const unsigned peers = __match_any_sync(FULL_MASK, key);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if (v && lane == leader) base = atomicAdd(cursor + key, (uint32_t)__popc(peers));
        base = __shfl_sync(FULL_MASK, base, leader);
        if (v) perm[base + __popc(peers & ((1u << lane) - 1u))] = q;
    }
}

// Order k >= 2 over queue q[(k + 1) & 1] in bucket order; survivors are appended to
// q[k & 1].  FP32 is held to 64 registers (4 blocks, 32 warps per SM; 7 % faster than
// at 80 registers).
template <class T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_wave_order(const __grid_constant__ TraceP<T> P, int k, WaveWork<T> W)
{
    const uint32_t n = W.count[k].live;
    const int lane = threadIdx.x & 31;
    Rec<T> *const src = (k & 1) ? W.q[0] : W.q[1];  // selects, not an indexed parameter array
    Rec<T> *const dst = (k & 1) ? W.q[1] : W.q[0];
    // warps claim 32-packet chunks from a counter: walk lengths differ from chunk to chunk, and a
    // warp that finishes early takes the next one (n <= 2^31, so the counter, which passes n by
    // at most a chunk per warp, cannot wrap).  The first chunks are dealt out, across the CTAs
    // first, so that a short queue is spread evenly over the SMs.  A chunk is claimed only when
    // the warp is free: claimed one ahead (its records prefetched meanwhile) it waits for a long
    // one while other warps have nothing left to do (20 orders of the clumpy envelope, 2^18
    // packets: 2.69 -> 2.15 ms, 2^20: 6.40 -> 6.03, 2^22: 20.9 -> 20.4).  Pools of 4 to 32 adjacent
    // chunks a CTA, for L1, lost more at each order's end than they gained.
    const uint32_t dealt = gridDim.x * (blockDim.x / 32) * 32u;
    uint32_t q0 = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u;
    while (q0 < n) {  // uniform per warp
        const uint32_t q = q0 + lane;
        const bool live = q < n;
        Rec<T> r;
        if (live) {
            copy_rec(&r, src + W.perm[q]);
        } else {
            for (int c = 0; c < 3; ++c) r.p.pos[c] = r.p.n[c] = r.p.a[c] = r.p.S[c] = T(0);
            r.p.tot = r.p.tot2 = T(0);
            r.j = 0;
        }
        const uint64_t i = P.first + r.j;
        const T wd = live ? point<T>(P.pts, i, 4 * (k - 1) + 2) : T(0);
        const bool on = run_order(P, k, i, live, wd, r.p);
        append(P, W, k, dst, on, r.p, r.j);
        if (live && !on && P.train_log) write_log(P, i, r.j, r.p);
        if (lane == 0) q0 = dealt + atomicAdd(&W.count[k].chunk, 32u);
        q0 = __shfl_sync(FULL_MASK, q0, 0);
    }
}

template <class T>
WaveWork<T> carve(void *ws, uint64_t cap)
{
    WaveWork<T> W;
    char *c = (char *)ws;
    auto take = [&](size_t bytes) {
        char *r = c;
        c += (bytes + 255) & ~(size_t)255;
        return r;
    };
    W.q[0] = (Rec<T> *)take(cap * sizeof(Rec<T>));
    W.q[1] = (Rec<T> *)take(cap * sizeof(Rec<T>));
    take(12);
    W.keys = (uint32_t *)take(cap * 4);
    W.perm = (uint32_t *)take(cap * 4);
    W.hist = (uint32_t *)take(WV_MAX_BUCKETS * 4 + WV_TAIL_BYTES);
    W.count = (WaveCount *)(W.hist + WV_MAX_BUCKETS);
    return W;
}

// Bits of the key for n packets.  20-order clumpy envelope, 16^3 position cells x 32 x 64 direction
// bins against 8^3 cells with the same bins: 20.9 / 21.3 ms at 2^22 packets, 6.51 / 6.40 at
// 2^20, 2.75 / 2.69 at 2^18, 1.79 / 1.73 at 2^16, and on a 32^3 grid 5.49 / 5.18 at 2^20.  Now, on 128^3:
// 15.28 / 15.58 at 2^22, 8.29 / 8.36 at 2^21, 6.36 / 6.38 at 2^20.5, 4.73 / 4.70 at 2^20; on 48^3 the coarse
// key is 4 to 6 % faster at any size up to 2^22.  Fewer direction bins lose at every size but the smallest, where no split matters (2^12: 1.15 ms).
// With a three-launch scan, clears and copies an order took up to 150 us on the buckets alone,
// and the same runs 22.3, 8.1, 4.4 and 3.3 ms.
WaveKey wave_bits(uint64_t n, uint64_t queue_bytes)
{
    WaveKey K = {n >= (1ull << 21) ? 4 : 3, 5, 6, 0};
    while (((uint64_t)4 << key_bits(K)) > queue_bytes) ++K.shift;  // the cursors lie in a queue
    return K;
}

template <class T>
cudaError_t launch_wave(TraceP<T> P, void *ws, uint64_t cap, int sms, cudaStream_t s)
{
    if (P.count == 0) return cudaSuccess;
    WaveWork<T> W = carve<T>(ws, cap);
    W.key = wave_bits(P.count, cap * sizeof(Rec<T>));
    const int buckets = 1 << key_bits(W.key);
    cudaError_t e = cudaMemsetAsync(W.count, 0, WV_TAIL_BYTES, s);
    if (e == cudaSuccess && P.max_orders > 1) e = cudaMemsetAsync(W.hist, 0, (size_t)buckets * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    // The support costs a read of the grid, 200 us and the caches at 512^3 (6 us at 256^3), which few
    // packets do not pay for.  512^3 clumpy envelope, us without and with it: 2 orders of 2^10 packets
    // 452 / 524, of 2^12 591 / 561; 5 of 2^8 935 / 1175, of 2^10 1512 / 1314; 1 of 2^16 294 / 327; 256^3: 2
    // of 2^8 138 / 135, 1 of 2^14 72 / 77, of 2^16 90 / 82.  FP64 walks are dearer: a 64th of the packets.
    const uint64_t cells = ((uint64_t)P.med.n[0] * P.med.n[1] * P.med.n[2]) >> (sizeof(T) == 8 ? 6 : 0);
    const bool few = P.max_orders > 1 ? P.count * (P.max_orders - 1) < cells >> 16 : P.count < cells >> 9;
    if (P.med.kind == QMCRT_MEDIUM_GRID && P.med.pad && P.med.inv_half[0] > 0.0f && !few) {
        uint32_t *support = (uint32_t *)(W.count + 66);
        k_support<T><<<(unsigned)std::max(1, sms * 8), 256, 0, s>>>(P.med, support_scale2(P.med), support);
        P.med.support = (const float *)support;
    }
    const uint64_t threads = (P.ord.threads + 31) & ~31ull;
    k_wave_first<T><<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(P, W);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::max(1, sms * (sizeof(T) == 4 ? 4 : 2));  // resident CTAs (launch bounds)
    for (int k = 2; k <= P.max_orders; ++k) {
        // the queue appended by order k - 1 holds order k's packets with their keys and
        // histogram: their indices in bucket order into perm
        uint32_t *cursor = (uint32_t *)W.q[k & 1];
        k_wave_cursors<<<(buckets + WV_TILE - 1) / WV_TILE, 256, 0, s>>>(W.hist, cursor, buckets, W.count + k);
        k_wave_scatter<<<(unsigned)std::max(1, sms * 8), 256, 0, s>>>(W.keys, cursor, W.perm, W.count + k);
        k_wave_order<T><<<grid, 256, 0, s>>>(P, k, W);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

uint64_t wavefront_workspace_bytes(uint64_t cap, int precision)
{
    const uint64_t rec = precision == QMCRT_PREC_F64 ? sizeof(Rec<double>) : sizeof(Rec<float>);
    auto pad = [](uint64_t b) { return (b + 255) & ~255ull; };
    return 2 * pad(cap * rec) + pad(12) + 2 * pad(cap * 4) + pad(WV_MAX_BUCKETS * 4 + WV_TAIL_BYTES);
}

cudaError_t launch_trace_wavefront_f32(const TraceP<float> &p, void *ws, uint64_t cap, int sms, cudaStream_t s)
{
    return launch_wave(p, ws, cap, sms, s);
}

cudaError_t launch_trace_wavefront_f64(const TraceP<double> &p, void *ws, uint64_t cap, int sms, cudaStream_t s)
{
    return launch_wave(p, ws, cap, sms, s);
}

}  // namespace qmcrt
