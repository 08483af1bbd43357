// Immersed-boundary coupling (Sec. 2.3): vertex binning by lattice block,
// spreading of vertex forces onto the lattice and interpolation of the
// lattice velocity to the vertices with Peskin's 4-point kernel, and the
// Euler move of the vertices (Sec. 2.6).
//
// Binning: each vertex gets its stencil anchor (floor(X) per axis, wrapped on
// periodic axes, and the fraction X - floor(X)) and the key of the 8^3 block
// that holds floor(X).  Counting sort: per-block counts (warp-aggregated
// atomics), exclusive scan, scatter with per-block cursors, then each block's
// segment is ordered by vertex id, which makes the permutation the stable
// sort by (key, id) (for read-out; the step itself does not depend on the
// order of the vertices within a bin and skips that sort).
//
// Spreading in two phases without global atomics: each non-empty bin adds
// its vertices' 4x4x4 stencils into an 11^3 tile in shared memory and writes
// the tile out; then each 8^3 block (owner computes) sums the tile positions
// of its neighbouring bins that map onto its nodes and writes F = g + sum for
// every node once (no separate clearing pass).  Interpolation: one CTA per
// non-empty bin stages the velocity of its 11^3 neighbourhood in shared
// memory (FP32: one 4-D tensor copy where the neighbourhood does not wrap)
// and evaluates the 64-node stencils of its own vertices from there (FP32:
// one thread per vertex over 16-byte node records; FP64: half-warps per
// vertex, partial sums reduced with warp shuffles, several CTAs per bin).
// With the Lees-Edwards boundary the vertices whose stencil reaches across
// the plane are kept in one extra bin, handled in k_lees.cu.
#include <cstring>
#include <type_traits>

#include <cooperative_groups.h>
#include <cuda.h>

#include "hemo_internal.cuh"

namespace hemo {

namespace {

inline int nblocks(long long n, int b) { return (int)((n + b - 1) / b); }

__device__ __forceinline__ float sqrt_r(float a) { return sqrtf(a); }
__device__ __forceinline__ double sqrt_r(double a) { return sqrt(a); }

constexpr int TILE = BLK + 3;           // stencil reach: one node below, two above
constexpr int TILE3 = TILE * TILE * TILE;
// strides of a bin's spreading tile, in memory as in the FP32 kernel's shared
// memory
constexpr int TP_Y = SPREAD_PITCH, TP_Z = SPREAD_PLANE, TP_N = SPREAD_NODES;
__device__ __forceinline__ int tile_index(int x, int y, int z) { return x + TP_Y * y + TP_Z * z; }
// Padded shared-memory strides of an 11^3 tile: the 16 lanes (b, c) of a
// half-warp address rows TS_Y*b + TS_Z*c, which fall in 16 distinct banks
// (TS_Y = 12, TS_Z = 161 = 1 mod 32).
constexpr int TS_Y = 12, TS_Z = 161;
constexpr int TILE_SMEM = TS_Z * TILE;

// A thread's walk over the positions q = l0 + TILE (l1 + TILE l2) of an
// 11^3 tile with a stride of blockDim.x: the coordinates advance by the
// stride's digits with carries, without integer division per position.
struct TileWalk {
    int l0, l1, l2, s0, s1, s2;
    __device__ __forceinline__ TileWalk(int q, int stride)
        : l0(q % TILE), l1((q / TILE) % TILE), l2(q / (TILE * TILE)), s0(stride % TILE), s1((stride / TILE) % TILE),
          s2(stride / (TILE * TILE)) {}
    __device__ __forceinline__ void next() {
        l0 += s0;
        if (l0 >= TILE) {
            l0 -= TILE;
            ++l1;
        }
        l1 += s1;
        if (l1 >= TILE) {
            l1 -= TILE;
            ++l2;
        }
        l2 += s2;
    }
};

// origin of bin k
template <typename R>
__device__ __forceinline__ void bin_origin(const View<R> &v, int k, int org[3]) {
    org[0] = (k % v.nb[0]) * BLK;
    org[1] = ((k / v.nb[0]) % v.nb[1]) * BLK;
    org[2] = (k / (v.nb[0] * v.nb[1])) * BLK;
}

template <typename R>
__global__ void anchor_count_kernel(View<R> v) {
    wait_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.nv) return;
    const int c = v.vcell[i];
    if (!index_ok(c >= 0 && c < v.ncell, v.status)) return;
    const int dims[3] = {v.nx, v.ny, v.nz};
    int b[3];
    for (int d = 0; d < 3; ++d) {
        const double X = v.ctr[3 * c + d] + (double)v.off[3 * (size_t)i + d];
        const double fl = floor(X);
        int j = (int)fl;
        const R t = R(X - fl);
        if (v.per[d]) {
            j = wrap(j, dims[d]);
        } else if (!(X >= 0.0 && X < (double)dims[d])) {
            atomicOr(v.status, ST_DOMAIN);
        }
        v.anc_i[3 * (size_t)i + d] = j;
        v.anc_t[3 * (size_t)i + d] = t;
        const int jc = j < 0 ? 0 : (j >= dims[d] ? dims[d] - 1 : j);
        b[d] = jc / BLK;
    }
    const int key = b[0] + v.nb[0] * (b[1] + v.nb[1] * b[2]);
    v.key[i] = key;
    // neighbouring vertex ids mostly share a block: one atomic per group
    const unsigned act = __activemask();
    const unsigned grp = __match_any_sync(act, key);
    if ((threadIdx.x & 31) == __ffs(grp) - 1) atomicAdd(v.counts + key, __popc(grp));
}

// exclusive scan of the block counts by one CTA of 1024 threads, over tiles
// of 4096 consecutive counts, four per thread (16-byte loads and stores
// where the arrays are 16-byte aligned; a thread's own sums, warp shuffles
// over the thread totals, the 32 warp totals by warp 0, a running carry
// between tiles; the next tile's counts are loaded before the current one
// is scanned); the counts are reset to zero for the next binning
__device__ __forceinline__ int4 load_quad(const int *p, int k, int n, bool vec) {
    if (vec && k + 3 < n) return *reinterpret_cast<const int4 *>(p + k);
    return make_int4(k < n ? p[k] : 0, k + 1 < n ? p[k + 1] : 0, k + 2 < n ? p[k + 2] : 0, k + 3 < n ? p[k + 3] : 0);
}
__device__ __forceinline__ void store_quad(int *p, int k, int n, bool vec, int4 q) {
    if (vec && k + 3 < n) {
        *reinterpret_cast<int4 *>(p + k) = q;
        return;
    }
    if (k < n) p[k] = q.x;
    if (k + 1 < n) p[k + 1] = q.y;
    if (k + 2 < n) p[k + 2] = q.z;
    if (k + 3 < n) p[k + 3] = q.w;
}
// With `order` (norder <= nbins <= 4096) also the bins by size: those of more than
// 2 `mean` vertices, then those of more than mean / 2, then the rest, each in
// natural order.
__global__ void __launch_bounds__(1024) scan_kernel(int *counts, int *start, int *cursor, int nbins, int *order,
                                                    int norder, int mean) {
    wait_previous();
    __shared__ int wsum[32], wclass[32];
    __shared__ int carry_s;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const bool vec = (((uintptr_t)counts | (uintptr_t)start | (uintptr_t)cursor) & 15) == 0;
    int carry = 0;
    int4 next = load_quad(counts, 4 * t, nbins, vec);
    for (int base = 0; base < nbins; base += 4096) {
        const int k0 = base + 4 * t;
        const int4 c = next;
        if (base + 4096 < nbins) next = load_quad(counts, k0 + 4096, nbins, vec);
        const int own = c.x + c.y + c.z + c.w;
        int x = own;  // inclusive scan of the thread totals within the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[w] = x;
        __syncthreads();
        if (w == 0) {  // the warp totals' inclusive scan
            int y = wsum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int z = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += z;
            }
            wsum[lane] = y;
            if (lane == 31) carry_s = y;
        }
        __syncthreads();
        const int e0 = carry + (w ? wsum[w - 1] : 0) + x - own;
        const int4 ex = make_int4(e0, e0 + c.x, e0 + c.x + c.y, e0 + c.x + c.y + c.z);
        store_quad(start, k0, nbins, vec, ex);
        store_quad(cursor, k0, nbins, vec, ex);
        store_quad(counts, k0, nbins, vec, make_int4(0, 0, 0, 0));
        if (order) {  // ranks within the first two classes, 16 bits each
            const int n[4] = {c.x, c.y, c.z, c.w};
            int mine = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (k0 + j < norder) mine += n[j] > 2 * mean ? 1 : (2 * n[j] > mean ? 0x10000 : 0);
            int y = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int z = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += z;
            }
            if (lane == 31) wclass[w] = y;
            __syncthreads();
            const int tot = wclass[lane], all = __reduce_add_sync(0xffffffffu, tot);
            const int at = __reduce_add_sync(0xffffffffu, lane < w ? tot : 0) + y - mine;
            int r0 = at & 0xffff, r1 = at >> 16;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = k0 + j, n0 = all & 0xffff, n1 = all >> 16;
                if (k >= norder) break;
                if (n[j] > 2 * mean) order[r0++] = k;
                else if (2 * n[j] > mean) order[n0 + r1++] = k;
                else order[n0 + n1 + k - r0 - r1] = k;
            }
        }
        carry += carry_s;
        __syncthreads();  // (wsum and carry_s are rewritten by the next tile)
    }
    if (t == 0) start[nbins] = carry;
}

// scatter with per-block cursors; lanes of a warp with the same key reserve
// their slots with one atomic
__global__ void scatter_kernel(const int *key, int *cursor, int *perm_raw, int nv, unsigned *status) {
    wait_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nv) return;
    const int k = key[i];
    const int lane = threadIdx.x & 31;
    const unsigned act = __activemask();
    const unsigned grp = __match_any_sync(act, k);
    const int leader = __ffs(grp) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cursor + k, __popc(grp));
    base = __shfl_sync(act, base, leader);
    const int slot = base + __popc(grp & ((1u << lane) - 1u));
    if (index_ok(slot >= 0 && slot < nv, status)) perm_raw[slot] = i;
}

// Few blocks and vertices: scan and scatter by one CTA, the cursors in shared
// memory (48^3 box, 2568 vertices: 4.1 us against 2.6 + 2.5 and the gap between
// two launches).  Above these sizes one SM is the slower.
__global__ void __launch_bounds__(1024) scan_scatter_kernel(int *counts, int *start, int nbins, const int *key, int *perm,
                                                            int nv, unsigned *status) {
    wait_previous();
    __shared__ __align__(16) int cur[SMALL_BINS];
    __shared__ int wsum[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const bool vec = ((uintptr_t)counts & 15) == 0;
    const int k0 = 4 * t;
    const int4 c = load_quad(counts, k0, nbins, vec);
    const int own = c.x + c.y + c.z + c.w;
    int x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    const int total = wsum[lane];
    const int before = __reduce_add_sync(0xffffffffu, lane < w ? total : 0);
    const int e0 = before + x - own;
    const int4 ex = make_int4(e0, e0 + c.x, e0 + c.x + c.y, e0 + c.x + c.y + c.z);
    store_quad(start, k0, nbins, vec && ((uintptr_t)start & 15) == 0, ex);
    store_quad(counts, k0, nbins, vec, make_int4(0, 0, 0, 0));
    store_quad(cur, k0, nbins, true, ex);
    if (t == 1023) start[nbins] = e0 + own;
    __syncthreads();
    for (int i = t; i < nv; i += 1024) {
        const int k = key[i];
        const unsigned act = __activemask();
        const unsigned grp = __match_any_sync(act, k);
        const int leader = __ffs(grp) - 1;
        int base = 0;
        const bool ok = index_ok(k >= 0 && k < nbins, status);
        if (lane == leader && ok) base = atomicAdd(cur + k, __popc(grp));
        base = __shfl_sync(act, base, leader);
        const int slot = base + __popc(grp & ((1u << lane) - 1u));
        if (ok && index_ok(slot >= 0 && slot < nv, status)) perm[slot] = i;
    }
}

// One warp per block: each id's rank among the block's ids (ids are unique)
// is its position.  Segments of up to SORT_SMEM ids are ranked from shared
// memory, SORT_K ids per lane at a time held in registers (one pass over the
// segment per group); longer segments one id at a time from global memory.
constexpr int SORT_SMEM = 1024;
constexpr int SORT_K = 8;
__global__ void __launch_bounds__(128) sort_bins_kernel(const int *start, const int *perm_raw, int *perm, int nbins) {
    wait_previous();
    __shared__ int buf[4][SORT_SMEM];
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    if (w >= nbins) return;
    const int s = start[w], n = start[w + 1] - s;
    const int *seg = perm_raw + s;
    if (n <= SORT_SMEM) {
        for (int a = lane; a < n; a += 32) buf[wl][a] = seg[a];
        __syncwarp();
        const int *sh = buf[wl];
        for (int g0 = 0; g0 < n; g0 += 32 * SORT_K) {
            int va[SORT_K], r[SORT_K];
#pragma unroll
            for (int j = 0; j < SORT_K; ++j) {
                const int a = g0 + lane + 32 * j;
                va[j] = a < n ? sh[a] : 0x7fffffff;
                r[j] = 0;
            }
            for (int b = 0; b < n; ++b) {
                const int x = sh[b];
#pragma unroll
                for (int j = 0; j < SORT_K; ++j) r[j] += x < va[j];
            }
#pragma unroll
            for (int j = 0; j < SORT_K; ++j)
                if (g0 + lane + 32 * j < n) perm[s + r[j]] = va[j];
        }
        return;
    }
    for (int a = lane; a < n; a += 32) {
        const int va = seg[a];
        int r = 0;
        for (int b = 0; b < n; ++b) r += seg[b] < va;
        perm[s + r] = va;
    }
}

// 4-byte asynchronous copy global -> shared (completes at cp_async_wait_all)
__device__ __forceinline__ void cp_async4(float *smem_dst, const float *gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async(double *smem_dst, const double *gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// four consecutive values (FP32: one 16-byte load)
__device__ __forceinline__ void ld4_any(const float *p, float *o) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    o[0] = q.x;
    o[1] = q.y;
    o[2] = q.z;
    o[3] = q.w;
}
__device__ __forceinline__ void ld4_any(const double *p, double *o) {
    for (int k = 0; k < 4; ++k) o[k] = p[k];
}
// Peskin 4-point weights of nodes floor(X) - 1 .. floor(X) + 2 for the
// fraction t = X - floor(X) in [0, 1); one square root serves all four.
template <typename R>
__device__ __forceinline__ void peskin4(R t, R *w) {
    const R q = sqrt_r(R(1) + R(4) * t - R(4) * t * t);
    w[0] = (R(3) - R(2) * t - q) * R(0.125);
    w[1] = (R(3) - R(2) * t + q) * R(0.125);
    w[2] = (R(1) + R(2) * t + q) * R(0.125);
    w[3] = (R(1) + R(2) * t - q) * R(0.125);
}

// Sums of K <= 8 values over each half-warp's 16 lanes, with about K + 3 additions
// per lane instead of 4 K (additions are what the FP64 pipe is short of): at
// every level a lane passes on half of its values and adds the other half.
// Returns value k in out[k] of every lane.
template <typename R, int K>
__device__ __forceinline__ void sum16(const R (&x)[K], R (&out)[K]) {
    constexpr int P = K <= 4 ? 4 : 8;
    const int lane = threadIdx.x & 31;
    R a[P];
#pragma unroll
    for (int k = 0; k < P; ++k) a[k] = k < K ? x[k] : R(0);
    int o = 8;
#pragma unroll
    for (int n = P / 2; n >= 1; n /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const R keep = up ? a[k + n] : a[k], give = up ? a[k] : a[k + n];
            a[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    for (; o >= 1; o /= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    // value k sits in the lanes whose leading bits (from 8 down) spell k
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int src = 0;
#pragma unroll
        for (int n = P / 2, bit = 8; n >= 1; n /= 2, bit /= 2)
            if (k & n) src |= bit;
        out[k] = __shfl_sync(0xffffffffu, a[0], (lane & 16) | src);
    }
}

// FP64 vertex kernels: CTAs per bin, each taking every FP64_BIN_PARTS-th
// chunk of the bin's vertices (FP64 arithmetic is slow per SM, and a bin
// crowded with vertices would otherwise keep one SM busy long after the
// others are done)
constexpr int FP64_BIN_PARTS = 8;

// distinct coordinates of the blocks whose vertices reach block b along an axis
// of n nodes: the neighbours, and for the first block of a periodic axis whose
// last block has a single node the block before that one too (a stencil reaches
// two nodes beyond its block)
__device__ __forceinline__ int neighbour_blocks(int b, int nb, int n, int periodic, int out[4]) {
    int cnt = 0;
    for (int d = periodic && b == 0 && n % BLK == 1 ? -2 : -1; d <= 1; ++d) {
        int q = b + d;
        if (periodic) q = wrap(q, nb);
        else if (q < 0 || q >= nb) continue;
        bool dup = false;
        for (int k = 0; k < cnt; ++k) dup |= out[k] == q;
        if (!dup) out[cnt++] = q;
    }
    return cnt;
}

// The b-th bin of a vertex kernel's grid: by size where the list is kept (-1 in
// the bounds-checked build for an entry that fails its check).
// Bins hold from none to several times the mean, and a grid of a few CTAs per
// SM ends when its largest does: with the largest first, 48 x 39 x 64 channel,
// FP64 interpolation 33 -> 30 us; 64 x 64 x 256 channel, FP32 spreading 27.4 ->
// 25.9, interpolation 29.6 -> 28.3, for 0.7 us more in the scan.  Not for more
// than 4096 bins, where neighbours' tiles share the cache and the end matters
// less.
template <typename R>
__device__ __forceinline__ int bin_of(const View<R> &v, int b) {
    const int k = v.order ? v.order[b] : b;
    return index_ok(k >= 0 && k < v.nbins, v.status) ? k : -1;
}

// FP64 vertex kernels: anchors and weights of one chunk of a bin, staged in
// shared memory, a thread per vertex and axis (the square roots run on the FP64
// pipe and are a long chain): the row in the bin's padded tile (-1 if the
// anchor is outside the bin, i.e. the vertex left the lattice), the vertex id
// and whatever weights(j, i, axis, t) stores for fraction t.
template <typename R, typename Weights>
__device__ __forceinline__ void stage_chunk(const View<R> &v, int p0, int n, const int org[3], int *srow, int *sperm,
                                            Weights weights) {
    for (int q = threadIdx.x; q < 3 * n; q += blockDim.x) {
        const int j = q / 3, ax = q - 3 * j;
        const int i = v.perm[p0 + j];
        if (!index_ok(i >= 0 && i < v.nv, v.status)) {
            if (ax == 0) srow[j] = -1;
            continue;
        }
        weights(j, i, ax, v.anc_t[3 * (size_t)i + ax]);
        if (ax == 0) {
            int row = 0;
            bool ok = true;
            for (int d = 0; d < 3; ++d) {
                const int b = v.anc_i[3 * (size_t)i + d] - org[d];
                ok &= b >= 0 && b < BLK;
                row += b * (d == 0 ? 1 : (d == 1 ? TS_Y : TS_Z));
            }
            srow[j] = ok ? row : -1;
            if (sperm) sperm[j] = i;
        }
    }
}

// the 11^3 neighbourhood of a 3-component field A ([3][N]) requested into a padded
// shared tile by asynchronous copies (zero beyond a non-periodic edge); jtab:
// the wrapped lattice coordinates per axis
template <typename R>
__device__ __forceinline__ void stage_tile(const View<R> &v, const R *A, const int (*jtab)[TILE], R (*tile)[TILE_SMEM]) {
    const size_t N = (size_t)v.N;
    TileWalk tw(threadIdx.x, blockDim.x);
    for (int q = threadIdx.x; q < TILE3; q += blockDim.x, tw.next()) {
        const int jx = jtab[0][tw.l0], jy = jtab[1][tw.l1], jz = jtab[2][tw.l2];
        const int sidx = tw.l0 + TS_Y * tw.l1 + TS_Z * tw.l2;
        if ((jx | jy | jz) < 0) {  // beyond a non-periodic edge: resting wall
            tile[0][sidx] = tile[1][sidx] = tile[2][sidx] = R(0);
        } else {
            const size_t n = (size_t)jx + (size_t)v.nx * ((size_t)jy + (size_t)v.ny * jz);
            for (int d = 0; d < 3; ++d) cp_async(&tile[d][sidx], A + d * N + n);
        }
    }
}

// Phase 1 of spreading: one CTA per non-empty bin adds the 4x4x4 stencils of
// the bin's vertices into an 11^3 shared tile, which is written out whole for
// the owners to gather.
//
// The tile accumulates in fixed point with integer shared atomics (native and
// exact: the sums do not depend on the order of the vertices, so every run
// gives the same bits).  FP32: 32-bit integers; per bin and component the
// scale is the power of two 2^e with e = 30 - ceil(log2(max|F| * n / 8)): a
// node's sum is at most max|F| times the sum of its n weights, each at most
// 1/8, so |sum| * 2^e <= 2^30, and the quantum, max|F| * n * 2^-33 per
// contribution, is below the FP32 rounding of sums of that size.  FP64:
// 64-bit integers with 2^62 in place of 2^30 (quantum max|F| n 2^-65, below
// FP64 rounding).
constexpr int ACC_F32 = 29, ACC_F64 = 61;  // log2 of the bound on a sum, minus one
constexpr int SPREAD_CAP = 352, SP64_THREADS = 512;  // vertices staged at a time, threads (FP64)

// FP64: the scale of a component from its largest force; 0 (and the numeric
// status) for forces that are not finite
__device__ __forceinline__ double tile_scale(double fmax_abs, int n, unsigned *status) {
    const double bound = fmax_abs * n * 0.125;
    if (!(bound <= 3.0e38)) {
        atomicOr(status, ST_NUMERIC);
        return 0.0;
    }
    return bound > 0.0 ? ldexp(1.0, min(ACC_F64 - ilogb(bound), 120)) : 0.0;
}

// FP32.  Two lanes per vertex, lane h adding the stencil's x nodes 2h and
// 2h + 1 (96 contributions each).  The shared atomics run at one warp
// instruction per cycle when the 32 lanes fall in 32 distinct banks, and cost
// a cycle more per collision.  The tile's z stride is 8 (mod 32) banks, so a
// lane that walks its four z layers starting from layer s instead of 0 sits 8 s
// banks further in every instruction (8 * 4 = 32: the walk wraps around with
// the banks).  An item (vertex, h) whose first position is in bank class c =
// (row + 2h) mod 8 can therefore take any of the four lanes of its class (bank c +
// 8m in lane 4c + m).  The bin's
// vertices are sorted by row mod 8 in shared memory, and each row of 32 lanes
// takes four items of each class: conflict-free, with as many rows as the
// fullest class needs (22 % more than a perfect balance on the pipe: 7.3
// atomic cycles per vertex instead of 6; the FP64 kernel's half-warp per
// vertex has two vertices collide, 11.8).  Integer sums do not depend on
// the order, so the walk and the sort leave the bits alone.
//
// Rounding to the fixed-point grid: half of the contributions by a conversion
// (F2I runs at 16 lanes per cycle, and all of them would take twice as long as
// the atomics), half without one: a magnitude c <= 2^24 quanta times 2^-149,
// the smallest denormal, is rounded to the nearest quantum by that
// multiplication, and the bits of the product are the integer (the bits of
// denormals and of the first normal binade count in quanta), the same integer
// as the conversion's.  A contribution is at most 2^30 / n quanta, so bins of at
// least 64 vertices qualify; smaller bins convert, and so does a row of lanes
// with a weight below zero (one that vanishes, rounded), whose contributions
// do not have the forces' signs.
//
// Bound by the shared-memory pipe (75 % busy) and by issue (78 %).  128 x 128 x
// 512 vessel (2.9 M vertices in 14.7 k bins): 242 -> 193 us; the spreading
// phase of the 1000 x 208 x 208 pipe (12.6 M vertices in 54 k bins) 1429 -> 1236
// us (all converted: 1347 with the gather's six CTAs per SM, where half takes
// 1287 and none 1303).  Six CTAs per SM: seven spill.
constexpr int SP_Y = TP_Y, SP_Z = TP_Z, SP_N = TP_N;  // the shared tile
static_assert(SP_Z % 32 == 8 && SP_Y % 8 == 4, "bank classes of the spreading tile");
constexpr int NO_SCALE = -1000;
constexpr int SP_CHUNK = 256;      // vertices sorted at a time, one per thread
constexpr int SP_GRID_MIN = 64;    // fewest vertices of a bin on the denormal grid
constexpr int SP_CONVERT = 12;     // of 24 contributions per layer, those converted there
struct SpreadStage {
    float4 a[SP_CHUNK];  // tx, qx, ty, qy: fraction and sqrt(1 + 4t - 4t^2) per axis
    float4 b[SP_CHUNK];  // tz, qz, F_x, F_y (forces scaled)
    float2 c[SP_CHUNK];  // F_z, tile row (as int)
};

// i = -i for four values if c != 0, as predicated instructions
__device__ __forceinline__ void negate_if(int c, int &i, int &j, int &k, int &l) {
    asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %4, 0;\n\t"
        "@p neg.s32 %0, %0;\n\t@p neg.s32 %1, %1;\n\t@p neg.s32 %2, %2;\n\t@p neg.s32 %3, %3;\n\t}"
        : "+r"(i), "+r"(j), "+r"(k), "+r"(l)
        : "r"(c));
}

// the contributions of an item: forces F, weights (2 w per axis), its first
// position in the tile and its walk's first z layer s; GRID: SP_CONVERT of the
// 24 contributions per layer are converted, the others land on the denormal
// grid; otherwise all are converted
template <bool GRID>
__device__ __forceinline__ void spread_item(int *first, int s, const float (&F)[3], const float (&wx)[2],
                                            const float (&wy)[4], const float (&wz)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        int *const pj = first + SP_Z * ((j + s) & 3);
        float wyz[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) wyz[b] = wy[b] * wz[j];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
#pragma unroll
            for (int b = 0; b < 4; b += 2) {
                const bool conv = !GRID || 8 * d + 2 * b < SP_CONVERT;
                const float Fd = conv ? F[d] : fabsf(F[d]), f0 = Fd * wyz[b], f1 = Fd * wyz[b + 1];
                const float c[4] = {f0 * wx[0], f0 * wx[1], f1 * wx[0], f1 * wx[1]};
                int i[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) i[q] = conv ? __float2int_rn(c[q]) : __float_as_int(c[q] * 0x1p-149f);
                if (!conv) negate_if(F[d] < 0.f, i[0], i[1], i[2], i[3]);
                int *const p = pj + d * SP_N + SP_Y * b;
                atomicAdd(p, i[0]);
                atomicAdd(p + 1, i[1]);
                atomicAdd(p + SP_Y, i[2]);
                atomicAdd(p + SP_Y + 1, i[3]);
            }
        }
    }
}

__global__ void __launch_bounds__(SP_CHUNK, 6) spread_tile_f32_kernel(View<float> v) {
    wait_previous();
    const int k = bin_of(v, blockIdx.x);
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1], n = e - s;
    if (n == 0) return;
    __shared__ __align__(16) int tile[3 * SP_N];
    __shared__ SpreadStage st;
    __shared__ float smax[24];  // [component][warp]
    __shared__ __align__(16) int count[8];  // vertices of the chunk per row mod 8
    constexpr int NW = SP_CHUNK / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < 3 * SP_N / 4; q += SP_CHUNK) reinterpret_cast<int4 *>(tile)[q] = make_int4(0, 0, 0, 0);
    if (tid < 8) count[tid] = 0;
    int org[3];
    bin_origin(v, k, org);
    // chunks of equal size
    const int nch = (n + SP_CHUNK - 1) / SP_CHUNK, csz = (n + nch - 1) / nch;
    // a vertex's record; row -1 outside the bin (domain status already raised) and
    // for a position that is not a number, whose contributions convert to zero
    // but would be the largest integer on the denormal grid
    auto load = [&](int j, float t[3], float F[3]) -> int {
        const int i = v.perm[j];
        if (!index_ok(i >= 0 && i < v.nv, v.status)) return -1;
        int row = 0;
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int b = v.anc_i[3 * (size_t)i + d] - org[d];
            ok &= b >= 0 && b < BLK;
            row += b * (d == 0 ? 1 : (d == 1 ? SP_Y : SP_Z));
            t[d] = v.anc_t[3 * (size_t)i + d];
            ok &= t[d] == t[d];
            F[d] = v.Fv[3 * (size_t)i + d];
        }
        return ok ? row : -1;
    };
    // the first chunk's records, and one scale per component for the whole bin
    float t[3] = {0.f, 0.f, 0.f}, F[3] = {0.f, 0.f, 0.f};
    int row = tid < csz ? load(s + tid, t, F) : -1;
    unsigned m[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) m[d] = __float_as_uint(fabsf(F[d]));  // (order as the floats, NaN above all)
    for (int j = s + csz + tid; j < e; j += SP_CHUNK) {
        const int i = v.perm[j];
        if (!index_ok(i >= 0 && i < v.nv, v.status)) continue;
#pragma unroll
        for (int d = 0; d < 3; ++d) m[d] = max(m[d], __float_as_uint(fabsf(v.Fv[3 * (size_t)i + d])));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        m[d] = __reduce_max_sync(0xffffffffu, m[d]);
        if (lane == 0) smax[d * NW + warp] = __uint_as_float(m[d]);
    }
    __syncthreads();
    int ex[3];  // the scales' exponents; NO_SCALE: no force, or one that is not finite
    {
        unsigned mm = lane < 3 * NW ? __float_as_uint(smax[lane]) : 0u;
#pragma unroll
        for (int o = 1; o < NW; o <<= 1) mm = max(mm, __shfl_xor_sync(0xffffffffu, mm, o));
        const float bound = __uint_as_float(mm) * (float)n * 0.125f;
        int x = min(ACC_F32 + 127 - (int)(__float_as_uint(bound) >> 23), 120);
        if (!(bound <= 3.0e38f)) {
            if (tid < 3 * NW) atomicOr(v.status, ST_NUMERIC);
            x = NO_SCALE;
        }
        if (bound == 0.f) x = NO_SCALE;
#pragma unroll
        for (int d = 0; d < 3; ++d) ex[d] = __shfl_sync(0xffffffffu, x, NW * d);
    }
    auto pow2 = [](int x) { return x == NO_SCALE ? 0.f : __int_as_float((x + 127) << 23); };
    const bool grid = n >= SP_GRID_MIN;
    const float scale[3] = {pow2(ex[0]) * 0.125f, pow2(ex[1]) * 0.125f, pow2(ex[2]) * 0.125f};  // (2 w per axis)
    for (int p = s; p < e; p += csz) {
        if (p != s) {
            __syncthreads();  // the previous chunk is done with the stage
            if (tid < 8) count[tid] = 0;
            row = tid < csz && p + tid < e ? load(p + tid, t, F) : -1;
            __syncthreads();
        }
        // sort by row mod 8: the lanes of a class count together
        unsigned peers = __ballot_sync(0xffffffffu, row >= 0);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const unsigned bal = __ballot_sync(0xffffffffu, row & o);
            peers &= row & o ? bal : ~bal;
        }
        const int leader = __ffs(peers) - 1;
        int rank = 0;
        if (row >= 0 && lane == leader) rank = atomicAdd(count + (row & 7), __popc(peers));
        rank = __shfl_sync(0xffffffffu, rank, leader & 31) + __popc(peers & ((1u << lane) - 1u));
        __syncthreads();
        // lanes 4c .. 4c + 3 serve class c: its count and first position
        const int n0 = count[lane >> 2];
        int f0 = n0;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, f0, o);
            if (lane >= o) f0 += x;
        }
        f0 -= n0;
        const int n1 = __shfl_sync(0xffffffffu, n0, lane + 24), f1 = __shfl_sync(0xffffffffu, f0, lane + 24);  // class c - 2
        const int rows = (__reduce_max_sync(0xffffffffu, n0 + n1) + 3) >> 2;
        const int at = __shfl_sync(0xffffffffu, f0, 4 * (row & 7)) + rank;
        if (row >= 0) {
            float r[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) r[d] = sqrtf(1.f + 4.f * t[d] - 4.f * t[d] * t[d]);
            st.a[at] = make_float4(t[0], r[0], t[1], r[1]);
            st.b[at] = make_float4(t[2], r[2], F[0] * scale[0], F[1] * scale[1]);
            st.c[at] = make_float2(F[2] * scale[2], __int_as_float(row));
        }
        __syncthreads();
        // the items of this lane's class c: half 0 of the vertices of class c,
        // then half 1 of those of class c - 2
        for (int i = warp; i < rows; i += NW) {
            const int it = 4 * i + (lane & 3);
            const bool on = it < n0 + n1;
            const int h = on && it >= n0, q = on ? (h ? f1 + it - n0 : f0 + it) : 0;
            const float4 A = st.a[q], B = st.b[q];
            const float2 C = st.c[q];
            const int pos = __float_as_int(C.y) + 2 * h;  // position of the item's first node
            const int z0 = (lane - (pos >> 3)) & 3;
            // 2 w = (3 - 2t - q, 3 - 2t + q, 1 + 2t + q, 1 + 2t - q) / 4 per axis
            const float ux = h ? fmaf(.5f, A.x, .25f) : fmaf(-.5f, A.x, .75f), gx = h ? -.25f : .25f;
            const float wx[2] = {fmaf(-gx, A.y, ux), fmaf(gx, A.y, ux)};
            const float y0 = fmaf(-.5f, A.z, .75f), y1 = fmaf(.5f, A.z, .25f);
            const float wy[4] = {fmaf(-.25f, A.w, y0), fmaf(.25f, A.w, y0), fmaf(.25f, A.w, y1), fmaf(-.25f, A.w, y1)};
            const float u0 = fmaf(-.5f, B.x, .75f), u1 = fmaf(.5f, B.x, .25f);
            const float v0 = fmaf(-.25f, B.y, u0), v1 = fmaf(.25f, B.y, u0), v2 = fmaf(.25f, B.y, u1), v3 = fmaf(-.25f, B.y, u1);
            // the z weights in the walk's order
            const float r0 = z0 & 1 ? v1 : v0, r1 = z0 & 1 ? v2 : v1, r2 = z0 & 1 ? v3 : v2, r3 = z0 & 1 ? v0 : v3;
            const float wz[4] = {z0 & 2 ? r2 : r0, z0 & 2 ? r3 : r1, z0 & 2 ? r0 : r2, z0 & 2 ? r1 : r3};
            const float F[3] = {B.z, B.w, C.x};
            const bool below = fminf(fminf(fminf(wx[0], wx[1]), fminf(wy[0], wy[3])), fminf(v0, v3)) < 0.f;  // (the others are above 1/4)
            const bool by_grid = grid && !__any_sync(0xffffffffu, on && below);
            if (!on) continue;
            if (by_grid) spread_item<true>(tile + pos, z0, F, wx, wy, wz);
            else spread_item<false>(tile + pos, z0, F, wx, wy, wz);
        }
    }
    __syncthreads();
    // write-out, four nodes per thread
    float4 *out = reinterpret_cast<float4 *>(v.tiles + (size_t)k * 3 * SP_N);
    const float inv[3] = {pow2(ex[0] == NO_SCALE ? NO_SCALE : -ex[0]), pow2(ex[1] == NO_SCALE ? NO_SCALE : -ex[1]),
                          pow2(ex[2] == NO_SCALE ? NO_SCALE : -ex[2])};
    for (int q = tid; q < 3 * SP_N / 4; q += SP_CHUNK) {
        const int4 f = reinterpret_cast<const int4 *>(tile)[q];
        const float iv = q < SP_N / 4 ? inv[0] : (q < 2 * SP_N / 4 ? inv[1] : inv[2]);
        out[q] = make_float4((float)f.x * iv, (float)f.y * iv, (float)f.z * iv, (float)f.w * iv);
    }
}

// FP64: a cluster of three CTAs per bin, one for each force component (three
// times the CTAs on the FP64 pipes, which a bin's vertices keep busy for long);
// each computes the weights of one axis for all three.  A warp takes two
// vertices, each half-warp's 16 lanes own one (y, z) row of the stencil.
// Bound by the FP64 pipe (19 cycles per warp instruction), then by the shared
// atomics: the four weights along x are w0, 1/2 - w3, 1/2 - w0, w3, so a row
// takes three conversions and two products, the other two nodes a subtraction
// of integers (one quantum of rounding instead of a half); the 64-bit sums are kept as two words with the carry taken from
// the first atomic (4 cycles per warp instruction; a 64-bit shared atomic takes
// 12).  48 x 39 x 64 channel with 30 cells: 65 ->
// 50 us; 32^3 box with one cell: 16.7 -> 11.7 us.  Threads for a whole SM's
// registers, so that three CTAs fit and the others follow as these end, the
// largest bins first: the channel 50 -> 35 us.
__device__ __forceinline__ void fixed_add(unsigned *lo, unsigned *hi, long long x) {
    const unsigned xl = (unsigned)x, old = atomicAdd(lo, xl);
    atomicAdd(hi, (unsigned)((unsigned long long)x >> 32) + (old + xl < xl));
}
__global__ void __cluster_dims__(3, 1, 1) __launch_bounds__(SP64_THREADS) spread_tile_kernel(View<double> v) {
    wait_previous();
    constexpr int CAP = SPREAD_CAP, W = 10;  // 2 w0 and 2 w3 along x, four weights along y and z
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int k = bin_of(v, blockIdx.x / 3), d = (int)cluster.block_rank();
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1];
    if (s == e) return;  // (the whole cluster)
    __shared__ unsigned lo[TILE_SMEM], hi[TILE_SMEM];
    __shared__ int srow[CAP];
    __shared__ __align__(16) double sw[W * CAP];
    __shared__ double sF[CAP];
    __shared__ unsigned long long smax[SP64_THREADS / 32];
    __shared__ double scale_s;
    for (int q = threadIdx.x; q < TILE_SMEM; q += blockDim.x) lo[q] = hi[q] = 0u;
    int org[3];
    bin_origin(v, k, org);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int h = lane >> 4, b = lane & 3, c = (lane >> 2) & 3;
    {  // the component's scale for the whole bin: largest |F|, compared as integers (NaN above all)
        unsigned long long m = 0;
        for (int j = s + threadIdx.x; j < e; j += blockDim.x) {
            const int i = v.perm[j];
            if (!index_ok(i >= 0 && i < v.nv, v.status)) continue;
            m = max(m, (unsigned long long)__double_as_longlong(fabs(v.Fv[3 * (size_t)i + d])));
        }
        const unsigned mh = (unsigned)(m >> 32), wh = __reduce_max_sync(0xffffffffu, mh);
        const unsigned wl = __reduce_max_sync(0xffffffffu, mh == wh ? (unsigned)m : 0u);
        if (lane == 0) smax[warp] = (unsigned long long)wh << 32 | wl;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 0; w < nw; ++w) m = max(m, smax[w]);
            scale_s = tile_scale(__longlong_as_double((long long)m), e - s, v.status);
        }
        cluster.sync();  // (and the cluster's shared memory is in place)
    }
    const double scale = scale_s;
    double *peer[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) peer[r] = cluster.map_shared_rank(sw, r) + (d == 0 ? 0 : 4 * d - 2);
    const int nch = (e - s + CAP - 1) / CAP, csz = (e - s + nch - 1) / nch;
    for (int p0 = s; p0 < e; p0 += csz) {
        const int n = min(csz, e - p0);
        if (p0 != s) cluster.sync();
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const int i = v.perm[p0 + j];
            int row = 0;
            bool ok = index_ok(i >= 0 && i < v.nv, v.status);
            if (ok) {
                double w[4];
                peskin4(v.anc_t[3 * (size_t)i + d], w);
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    double *o = peer[r] + W * j;
                    if (d == 0) {
                        o[0] = 2.0 * w[0];
                        o[1] = 2.0 * w[3];
                    } else {
                        for (int a = 0; a < 4; ++a) o[a] = w[a];
                    }
                }
                sF[j] = scale > 0.0 ? v.Fv[3 * (size_t)i + d] * (0.5 * scale) : 0.0;
                for (int a = 0; a < 3; ++a) {
                    const int q = v.anc_i[3 * (size_t)i + a] - org[a];
                    // (exponent bits all set: a position that is not a number adds nothing)
                    const int th = __double2hiint(v.anc_t[3 * (size_t)i + a]);
                    ok &= q >= 0 && q < BLK && (th & 0x7ff00000) != 0x7ff00000;
                    row += q * (a == 0 ? 1 : (a == 1 ? TS_Y : TS_Z));
                }
            }
            srow[j] = ok ? row : -1;
        }
        cluster.sync();
        for (int q = 2 * warp + h; q < n; q += 2 * nw) {
            const int row0 = srow[q];
            if (row0 < 0) continue;  // vertex outside the lattice (domain status already raised)
            const double *w = sw + W * q;
            const double g = sF[q] * (w[2 + b] * w[6 + c]);  // half the row's force
            const double2 x = *reinterpret_cast<const double2 *>(w);
            const long long qh = __double2ll_rn(g), q0 = __double2ll_rn(g * x.x), q3 = __double2ll_rn(g * x.y);
            const long long f[4] = {q0, qh - q3, qh - q0, q3};
            const int row = row0 + TS_Y * b + TS_Z * c;
#pragma unroll
            for (int a = 0; a < 4; ++a) fixed_add(lo + row + a, hi + row + a, f[a]);
        }
    }
    __syncthreads();
    // write-out, divided by the scale (a power of two) through the exponent
    double *out = v.tiles + ((size_t)k * 3 + d) * TP_N;
    const long long ex = scale > 0.0 ? (long long)ilogb(scale) << 52 : 0;
    TileWalk tw(threadIdx.x, blockDim.x);
    for (int q = threadIdx.x; q < TILE3; q += blockDim.x, tw.next()) {
        const int p = tw.l0 + TS_Y * tw.l1 + TS_Z * tw.l2;
        const long long x = scale > 0.0 ? (long long)((unsigned long long)hi[p] << 32 | lo[p]) : 0;
        const long long f = __double_as_longlong((double)x);
        out[tile_index(tw.l0, tw.l1, tw.l2)] = __longlong_as_double(x ? f - ex : 0);
    }
}

// Phase 2 of spreading (owner computes): one CTA per 8^3 block sums, for
// each of its nodes, every tile position of the non-empty neighbouring bins
// that maps onto the node (several positions when a periodic axis is shorter
// than a tile), in a fixed order, and writes F = g + sum once.  Per axis a
// table built once per block lists, for each local coordinate, the pairs
// (neighbour slot, tile position) that land on it.
constexpr int GATHER_MAXE = 2 * TILE;  // entries per (axis, local coordinate)
template <typename R>
__global__ void __launch_bounds__(256) spread_gather_kernel(View<R> v) {
    wait_previous();
    __shared__ int nbin[64];  // bin of neighbour slot (sz*16 + sy*4 + sx), -1 if empty
    __shared__ int lb[3][4], nsl[3];
    __shared__ unsigned char cnt[3][BLK];
    __shared__ unsigned char ent_slot[3][BLK][GATHER_MAXE], ent_pos[3][BLK][GATHER_MAXE];
    const int k = blockIdx.x;
    const int bc[3] = {k % v.nb[0], (k / v.nb[0]) % v.nb[1], k / (v.nb[0] * v.nb[1])};
    const int dims[3] = {v.nx, v.ny, v.nz};
    const int t = threadIdx.x;
    if (t < 3) nsl[t] = neighbour_blocks(bc[t], v.nb[t], dims[t], v.per[t], lb[t]);
    __syncthreads();
    if (t < 3 * BLK) {  // table of axis d, local coordinate l
        const int d = t / BLK, l = t % BLK;
        const int x = bc[d] * BLK + l;
        int n = 0;
        for (int sl = 0; sl < nsl[d]; ++sl) {
            const int o = lb[d][sl] * BLK - 1;  // tile origin along d
            if (v.per[d]) {
                for (int p = wrap(x - o, dims[d]); p < TILE && n < GATHER_MAXE; p += dims[d]) {
                    ent_slot[d][l][n] = (unsigned char)sl;
                    ent_pos[d][l][n++] = (unsigned char)p;
                }
            } else if (x - o >= 0 && x - o < TILE) {
                ent_slot[d][l][n] = (unsigned char)sl;
                ent_pos[d][l][n++] = (unsigned char)(x - o);
            }
        }
        cnt[d][l] = (unsigned char)n;
    } else if (t >= 32 && t < 32 + 64) {  // neighbour slot -> bin
        const int sl = t - 32, a = sl / 16, b = (sl / 4) % 4, c = sl % 4;
        int kk = -1;
        if (a < nsl[2] && b < nsl[1] && c < nsl[0]) {
            kk = lb[0][c] + v.nb[0] * (lb[1][b] + v.nb[1] * lb[2][a]);
            if (v.start[kk + 1] == v.start[kk]) kk = -1;
        }
        nbin[sl] = kk;
    }
    __syncthreads();
    const size_t N = (size_t)v.N;
    for (int q = t; q < BLK * BLK * BLK; q += blockDim.x) {
        const int l0 = q % BLK, l1 = (q / BLK) % BLK, l2 = q / (BLK * BLK);
        const int x = bc[0] * BLK + l0, y = bc[1] * BLK + l1, z = bc[2] * BLK + l2;
        if (x >= v.nx || y >= v.ny || z >= v.nz) continue;
        R f0 = R(0), f1 = R(0), f2 = R(0);
        for (int iz = 0; iz < cnt[2][l2]; ++iz)
            for (int iy = 0; iy < cnt[1][l1]; ++iy)
                for (int ix = 0; ix < cnt[0][l0]; ++ix) {
                    const int kk = nbin[16 * ent_slot[2][l2][iz] + 4 * ent_slot[1][l1][iy] + ent_slot[0][l0][ix]];
                    if (kk < 0) continue;
                    const R *tt = v.tiles + (size_t)kk * 3 * TP_N;
                    const int ti = tile_index(ent_pos[0][l0][ix], ent_pos[1][l1][iy], ent_pos[2][l2][iz]);
                    f0 += tt[ti];
                    f1 += tt[TP_N + ti];
                    f2 += tt[2 * TP_N + ti];
                }
        const size_t n = (size_t)x + (size_t)v.nx * ((size_t)y + (size_t)v.ny * z);
        const bool wall = !v.spread_all_nodes && (v.ntype[n] & 0x7f);
        v.F[n] = wall ? R(0) : v.g[0] + f0;
        v.F[N + n] = wall ? R(0) : v.g[1] + f1;
        v.F[2 * N + n] = wall ? R(0) : v.g[2] + f2;
    }
}

// Phase 2 with at least three blocks along every axis (neighbour blocks
// distinct) and whole blocks along the periodic ones: along an axis the lower neighbour's tile covers this block's
// local coordinates 0, 1 (tile positions 9, 10), the block's own tile all
// eight (positions 1..8) and the upper neighbour's coordinate 7 (position
// 0).  Each thread owns two nodes and adds, slot by slot in a fixed order,
// the tile values that land on them.
//
// Latency-bound, so many small threads: eight CTAs per SM (32 registers; six:
// the spreading phase of the pipe 1251 instead of 1236 us).  A thread per
// component and z column (a third fewer instructions, all loads at constant
// offsets, 56 registers) took 1384, one per component and node 1814.
template <typename R>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 8 : 1) spread_gather3_kernel(View<R> v) {
    wait_previous();
    __shared__ int nbin[27];  // bin of slot (sz + 1) * 9 + (sy + 1) * 3 + (sx + 1), -1 if empty or absent
    const int k = blockIdx.x;
    const int bc[3] = {k % v.nb[0], (k / v.nb[0]) % v.nb[1], k / (v.nb[0] * v.nb[1])};
    const int t = threadIdx.x;
    if (t < 27) {
        const int sz = t / 9 - 1, sy = (t / 3) % 3 - 1, sx = t % 3 - 1;
        const int sl[3] = {sx, sy, sz};
        int c[3];
        bool ok = true;
        for (int d = 0; d < 3; ++d) {
            c[d] = bc[d] + sl[d];
            if (v.per[d]) c[d] = wrap(c[d], v.nb[d]);
            else ok &= c[d] >= 0 && c[d] < v.nb[d];
        }
        int kk = -1;
        if (ok) {
            kk = c[0] + v.nb[0] * (c[1] + v.nb[1] * c[2]);
            if (v.start[kk + 1] == v.start[kk]) kk = -1;
        }
        nbin[t] = kk;
    }
    __syncthreads();
    const size_t N = (size_t)v.N;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int q = t + 256 * h;
        const int l[3] = {q % BLK, (q / BLK) % BLK, q / (BLK * BLK)};
        const int x = bc[0] * BLK + l[0], y = bc[1] * BLK + l[1], z = bc[2] * BLK + l[2];
        if (x >= v.nx || y >= v.ny || z >= v.nz) continue;
        R f0 = R(0), f1 = R(0), f2 = R(0);
        // per axis: the slots reaching this coordinate and the tile position there
        int ns[3], sl[3][2] = {{0, 0}, {0, 0}, {0, 0}}, ps[3][2] = {{0, 0}, {0, 0}, {0, 0}};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            // entry 0: lower neighbour (l < 2) or own block; entry 1: own block
            // (l < 2) or upper neighbour (l = 7)
            const bool lo = l[d] < 2, hi = l[d] == BLK - 1;
            sl[d][0] = lo ? 0 : 1;
            ps[d][0] = lo ? l[d] + 9 : l[d] + 1;
            sl[d][1] = lo ? 1 : 2;
            ps[d][1] = lo ? l[d] + 1 : 0;
            ns[d] = (lo || hi) ? 2 : 1;
        }
        // at most two slots per axis: fixed trip counts keep the tables in
        // registers; the tile addresses of all eight (slot x, y, z) choices
        // are formed first and the loads issued predicated, so that they are
        // all in flight together (summed in the same order, iz, iy, ix)
        const R *src[8];
        bool on[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const int ix = m & 1, iy = (m >> 1) & 1, iz = m >> 2;
            const bool in = iz < ns[2] && iy < ns[1] && ix < ns[0];
            const int kk = in ? nbin[9 * sl[2][iz] + 3 * sl[1][iy] + sl[0][ix]] : -1;
            on[m] = kk >= 0;
            src[m] = v.tiles + (size_t)(kk < 0 ? 0 : kk) * 3 * TP_N + tile_index(ps[0][ix], ps[1][iy], ps[2][iz]);
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            if (on[m]) {
                f0 += src[m][0];
                f1 += src[m][TP_N];
                f2 += src[m][2 * TP_N];
            }
        }
        const size_t n = (size_t)x + (size_t)v.nx * ((size_t)y + (size_t)v.ny * z);
        const bool wall = !v.spread_all_nodes && (v.ntype[n] & 0x7f);
        v.F[n] = wall ? R(0) : v.g[0] + f0;
        v.F[N + n] = wall ? R(0) : v.g[1] + f1;
        v.F[2 * N + n] = wall ? R(0) : v.g[2] + f2;
    }
}

// The move of vertex i by its interpolated velocity U (dt = 1), Sec. 2.6:
// INTEG 0 Euler; 1 Euler, keeping U; 2 the two-step Adams-Bashforth form
// with the kept velocity of the previous step, keeping U.  All loads are
// issued before the stores (off and Uprev are distinct buffers).
//
// With the adaptive separation on (v.off_eval set) it returns the vertex's
// displacement since the last force evaluation, |off - off_eval| of the new
// offsets (held steps do not re-base, so that is X - X_eval); else 0.
template <int INTEG, typename R>
__device__ __forceinline__ R move_vertex(const View<R> &v, int i, R U0, R U1, R U2) {
    R *o = v.off + 3 * (size_t)i;
    const R x0 = o[0], x1 = o[1], x2 = o[2];
    R n0, n1, n2;
    if constexpr (INTEG == 0) {
        n0 = x0 + U0;
        n1 = x1 + U1;
        n2 = x2 + U2;
    } else {
        R *p = v.Uprev + 3 * (size_t)i;
        if constexpr (INTEG == 2) {
            const R p0 = p[0], p1 = p[1], p2 = p[2];
            n0 = x0 + (R(1.5) * U0 - R(0.5) * p0);
            n1 = x1 + (R(1.5) * U1 - R(0.5) * p1);
            n2 = x2 + (R(1.5) * U2 - R(0.5) * p2);
        } else {
            n0 = x0 + U0;
            n1 = x1 + U1;
            n2 = x2 + U2;
        }
        p[0] = U0;
        p[1] = U1;
        p[2] = U2;
    }
    o[0] = n0;
    o[1] = n1;
    o[2] = n2;
    if (!v.off_eval) return R(0);
    const R *e = v.off_eval + 3 * (size_t)i;
    const R d0 = n0 - e[0], d1 = n1 - e[1], d2 = n2 - e[2];
    return sqrt_r(d0 * d0 + d1 * d1 + d2 * d2);
}

// the largest displacement of a warp's vertices into the adaptive word (as
// double bits: non-negative doubles order as their bit patterns); every
// lane calls it
__device__ __forceinline__ void adapt_max(unsigned long long *adapt, double d) {
    unsigned long long m = (unsigned long long)__double_as_longlong(d);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long q = __shfl_xor_sync(0xffffffffu, m, o);
        m = q > m ? q : m;
    }
    if ((threadIdx.x & 31) == 0 && m) atomicMax(adapt, m);
}

// Adaptive separation, once per step before the membrane kernels: evaluate
// the forces on the first step, when `every` steps have passed since the last
// evaluation, or when a vertex has moved more than tol since it; the
// displacement word is cleared for the coming step's interpolation.
__global__ void adapt_decide_kernel(unsigned long long *a, double tol, int every) {
    wait_previous();
    const bool eval = a[3] || a[1] >= (unsigned long long)every || __longlong_as_double((long long)a[0]) > tol;
    a[2] = eval ? 1ull : 0ull;
    a[4] += eval ? 1ull : 0ull;  // evaluations so far
    a[1] = eval ? 1ull : a[1] + 1ull;
    a[3] = 0ull;
    a[0] = 0ull;
}

// Anchors, keys and bin counts on a step between two membrane-force
// evaluations (Sec. 2.6), vertex-parallel: no re-base, so each vertex is at
// X = (hi + lo of the centroid of the last re-base) + offset.
template <typename R>
__global__ void __launch_bounds__(256) hold_bins_kernel(View<R> v) {
    wait_previous();
    if (v.adapt && v.adapt[2]) return;  // adaptive separation: this step evaluates the forces
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.nv) return;
    const int c = v.vcell[i];
    if (!index_ok(c >= 0 && c < v.ncell, v.status)) return;
    const R *cs = v.csp + 6 * (size_t)c;
    const R *o = v.off + 3 * (size_t)i;
    const R ch[3] = {cs[0], cs[1], cs[2]}, cl[3] = {cs[3], cs[4], cs[5]}, oi[3] = {o[0], o[1], o[2]};
    bin_vertex(v, (size_t)i, ch, cl, oi);
}

// Interpolation and vertex move: one CTA per non-empty bin stages u of the
// 11^3 neighbourhood in shared memory (padded strides; lattice coordinates
// of the tile's rows from per-axis tables built once); a warp takes two
// vertices, each half-warp's lanes own one (y, z) stencil row, and the 16
// partial sums are reduced with warp shuffles (sum16).  FP64 only; bound by the
// staging's latency for few vertices (the tile by asynchronous copies while
// the weights are computed, a thread per vertex and axis) and by the FP64 pipe:
// 32^3 box with one cell 20.5 -> 16.4 us, 48 x 39 x 64 channel with 30 cells
// 45 -> 35 us.
constexpr int INTERP_CAP = 32;  // vertices per chunk
template <typename R, int INTEG>
__global__ void __launch_bounds__(256) interpolate_kernel(View<R> v, int parts) {
    wait_previous();
    drop_dead_lines(v);
    constexpr int CAP = INTERP_CAP;
    const int k = bin_of(v, blockIdx.x % v.nbins), part = blockIdx.x / v.nbins;  // CTA part takes chunks part, part + parts, ...
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1];
    if (s + part * CAP >= e) return;
    __shared__ R tile[3][TILE_SMEM];
    __shared__ int srow[CAP], sperm[CAP];
    __shared__ R sw[12 * CAP];
    __shared__ int jtab[3][TILE];  // wrapped lattice coordinate, -1 beyond a non-periodic edge
    int org[3];
    bin_origin(v, k, org);
    if (threadIdx.x < 3 * TILE) {
        const int d = threadIdx.x / TILE, l = threadIdx.x % TILE;
        const int dims = d == 0 ? v.nx : (d == 1 ? v.ny : v.nz);
        int j = org[d] - 1 + l;
        if (v.per[d]) j = wrap(j, dims);
        else if (j < 0 || j >= dims) j = -1;
        jtab[d][l] = j;
    }
    __syncthreads();
    stage_tile(v, (const R *)v.u, jtab, tile);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int h = lane >> 4, b = lane & 3, c = (lane >> 2) & 3;
    for (int c0 = s + part * CAP; c0 < e; c0 += parts * CAP) {
        const int n = min(CAP, e - c0);
        if (c0 != s + part * CAP) __syncthreads();  // the previous chunk's records
        stage_chunk(v, c0, n, org, srow, sperm, [&](int j, int, int ax, R t) { peskin4(t, sw + 12 * j + 4 * ax); });
        if (c0 == s + part * CAP) cp_async_wait_all();  // the tile
        __syncthreads();
        for (int q0 = 2 * warp; q0 < n; q0 += 2 * nw) {  // uniform per warp: shuffles below
            const int q = q0 + h;
            R U[3] = {R(0), R(0), R(0)};
            const int row0 = q < n ? srow[q] : -1;
            if (row0 >= 0) {
                const R *w = sw + 12 * q;
                const R wyz = w[4 + b] * w[8 + c];
                const int row = row0 + TS_Y * b + TS_Z * c;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    R t = R(0);
#pragma unroll
                    for (int a = 0; a < 4; ++a) t += w[a] * tile[d][row + a];
                    U[d] = wyz * t;
                }
            }
            R Us[3];
            sum16(U, Us);
            double dmax = 0.0;
            if (row0 >= 0 && (lane & 15) == 0) dmax = move_vertex<INTEG>(v, sperm[q], Us[0], Us[1], Us[2]);
            if (v.adapt) adapt_max(v.adapt, dmax);
        }
    }
}

// FP32 interpolation: one thread per vertex.  The bin's 11^3 neighbourhood
// of u is staged once as (ux, uy, uz, 0) per node, so each stencil node is
// one 16-byte shared load; the weights stay in registers and each thread
// sums its vertex's 64 terms itself (no shuffles, the same order for every
// vertex).
//
// A 16-byte load is served eight lanes at a time, without conflict when their
// records fall in the eight 16-byte banks.  All lanes load at the same offset
// from their vertex's first record, so the bin's vertices are sorted by that
// record's index mod 8 in shared memory and lane l takes one of class l mod
// 8: four cycles per load instead of about ten.  The fullest class sets the
// number of lanes (1.39 times the vertices on the pipe).
//
// Bound by shared-memory wavefronts (62.5 M -> 47.3 M on the 128 x 128 x 512
// vessel, 77 % of the kernel's cycles; conflicts 29.8 M -> 8.9 M).  Vessel 238 ->
// 194 us, 1000 x 208 x 208 pipe 953 -> 776 us; five CTAs per SM 785, seven 806
// (spills).
//
// Staging.  With a tensor map of u (4-D: x, y, z, component) one thread
// copies the box x in [ox - 4, ox + 12), y in [oy - 1, oy + 10), z in
// [oz - 1, oz + 10), all three components, into shared memory with a single
// tensor copy (x starts 16-byte aligned: ox is a multiple of 8; coordinates
// outside the lattice read as zero, the resting wall beyond a non-periodic
// edge); the threads then rearrange it into the node records, in place (each
// first reads its nodes' values into registers).  A bin whose neighbourhood
// wraps around a periodic edge, and every bin without a tensor map, is
// staged node by node with 4-byte asynchronous copies.
constexpr int IT_Y = TILE, IT_Z = TILE * TILE;  // node record strides of the interpolation tile
constexpr int UBOX_X = 16;                      // x extent of the tensor copy (nodes)
constexpr unsigned UBOX_BYTES = 3u * UBOX_X * TILE * TILE * 4u;
constexpr int INTERP_SMEM = UBOX_BYTES > 16u * TILE3 ? (int)UBOX_BYTES : 16 * TILE3;
__device__ __forceinline__ void tma_load_4d(void *dst, const void *map, int c0, int c1, int c2, int c3, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_addr(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

constexpr int IT_CHUNK = 256;  // vertices sorted at a time, one per thread
template <int INTEG>
__global__ void __launch_bounds__(IT_CHUNK, 6) interpolate_v4_kernel(View<float> v, const __grid_constant__ CUtensorMap umap) {
    wait_previous();
    drop_dead_lines(v);
    const int k = bin_of(v, blockIdx.x);
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1];
    if (s == e) return;
    __shared__ __align__(128) unsigned char tile_raw[INTERP_SMEM];
    __shared__ int jtab[3][TILE];  // wrapped lattice coordinate, -1 beyond a non-periodic edge
    __shared__ __align__(8) uint64_t bar;
    __shared__ float4 srec[IT_CHUNK];  // sorted vertices: fractions and first record, then their velocities
    __shared__ int count[8];           // vertices of the chunk per class
    float4 *tile = reinterpret_cast<float4 *>(tile_raw);
    if (threadIdx.x < 8) count[threadIdx.x] = 0;
    int org[3];
    bin_origin(v, k, org);
    // the tensor copy serves a neighbourhood that does not wrap
    bool boxed = v.u_tmap != nullptr;
    for (int d = 0; d < 3; ++d) {
        const int dims = d == 0 ? v.nx : (d == 1 ? v.ny : v.nz);
        if (v.per[d] && (org[d] - 1 < 0 || org[d] + BLK + 1 >= dims)) boxed = false;
    }
    if (boxed && v.stalled_wait_test) {
        // failure-path test: wait on a barrier that nothing arrives at (no
        // copy issued); the bounded wait runs out and the CTA reports it
        if (threadIdx.x == 0) {
            mbar_init(&bar, 1);
            fence_mbar_init();
        }
        __syncthreads();
        const bool ok = threadIdx.x == 0 ? mbar_wait(&bar, 0u, 2000000ull) : true;
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) atomicOr(v.status, ST_TIMEOUT);
            return;
        }
    }
    if (boxed && threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        fence_async_smem();
        mbar_expect_tx(&bar, UBOX_BYTES);
        tma_load_4d(tile_raw, &umap, org[0] - 4, org[1] - 1, org[2] - 1, 0, &bar);
    }
    if (!boxed) {
        if (threadIdx.x < 3 * TILE) {
            const int d = threadIdx.x / TILE, l = threadIdx.x % TILE;
            const int dims = d == 0 ? v.nx : (d == 1 ? v.ny : v.nz);
            int j = org[d] - 1 + l;
            if (v.per[d]) j = wrap(j, dims);
            else if (j < 0 || j >= dims) j = -1;
            jtab[d][l] = j;
        }
        __syncthreads();
        const size_t N = (size_t)v.N;
        // asynchronous copies (no register round trip: all of a thread's loads
        // are in flight at once); nodes beyond a non-periodic edge are a
        // resting wall
        for (int q = threadIdx.x; q < TILE3; q += blockDim.x) {
            const int l0 = q % TILE, l1 = (q / TILE) % TILE, l2 = q / (TILE * TILE);
            const int jx = jtab[0][l0], jy = jtab[1][l1], jz = jtab[2][l2];
            float4 *dst = tile + q;
            if ((jx | jy | jz) >= 0) {
                const size_t n = (size_t)jx + (size_t)v.nx * ((size_t)jy + (size_t)v.ny * jz);
                cp_async4(&dst->x, v.u + n);
                cp_async4(&dst->y, v.u + N + n);
                cp_async4(&dst->z, v.u + 2 * N + n);
            } else {
                *dst = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
    // chunks of equal size; the first one's records are requested and sorted
    // before the tile is staged, so their latency overlaps the staging
    const int n = e - s, nch = (n + IT_CHUNK - 1) / IT_CHUNK, csz = (n + nch - 1) / nch;
    const int lane = threadIdx.x & 31;
    int n0 = 0, f0 = 0, slots = 0;  // this lane's class: vertices, first position; lanes of the chunk
    int own = -1, at = -1;          // this thread's vertex and its place in srec
    auto sort_chunk = [&](int p) {
        int i = -1, row = -1;
        float t[3] = {0.f, 0.f, 0.f};
        if ((int)threadIdx.x < csz && p + (int)threadIdx.x < e) {
            i = v.perm[p + threadIdx.x];
            if (index_ok(i >= 0 && i < v.nv, v.status)) {
                bool ok = true;
                int r = 0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int b = v.anc_i[3 * (size_t)i + d] - org[d];
                    ok &= b >= 0 && b < BLK;  // (else the vertex left the lattice; the domain status is raised)
                    r += b * (d == 0 ? 1 : (d == 1 ? IT_Y : IT_Z));
                    t[d] = v.anc_t[3 * (size_t)i + d];
                }
                row = ok ? r : -1;
            }
        }
        // the lanes of a class count together
        unsigned peers = __ballot_sync(0xffffffffu, row >= 0);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const unsigned bal = __ballot_sync(0xffffffffu, row & o);
            peers &= row & o ? bal : ~bal;
        }
        const int leader = __ffs(peers) - 1;
        int rank = 0;
        if (row >= 0 && lane == leader) rank = atomicAdd(count + (row & 7), __popc(peers));
        rank = __shfl_sync(0xffffffffu, rank, leader & 31) + __popc(peers & ((1u << lane) - 1u));
        __syncthreads();
        n0 = count[lane & 7];
        f0 = n0;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, f0, o, 8);
            if ((lane & 7) >= o) f0 += x;
        }
        f0 -= n0;
        slots = 8 * __reduce_max_sync(0xffffffffu, n0);
        at = __shfl_sync(0xffffffffu, f0, row & 7) + rank;
        own = row >= 0 ? i : -1;
        if (row >= 0) {
            srec[at] = make_float4(t[0], t[1], t[2], __int_as_float(row));
            // the move's loads (offsets; the previous velocity for Adams-Bashforth;
            // the offsets of the last force evaluation for the adaptive
            // separation) are requested into L1 before the stencil sums, whose
            // shared loads would otherwise hide nothing of their latency
            prefetch_l1(v.off + 3 * (size_t)i);
            if (INTEG == 2) prefetch_l1(v.Uprev + 3 * (size_t)i);
            if (v.off_eval) prefetch_l1(v.off_eval + 3 * (size_t)i);
        }
    };
    __syncthreads();  // (the counts; the barrier is initialised)
    sort_chunk(s);
    if (boxed) {
        const bool ok = mbar_wait(&bar, 0);
        if (__syncthreads_or(!ok)) {  // the copy did not complete in time: report, let it land, leave
            if (threadIdx.x == 0) {
                atomicOr(v.status, ST_TIMEOUT);
                mbar_wait(&bar, 0);
            }
            __syncthreads();
            return;
        }
        // rearrange [component][z][y][x - ox + 4] into node records, in place
        constexpr int PER = (TILE3 + 255) / 256;
        const float *box = reinterpret_cast<const float *>(tile_raw);
        float4 r[PER];
        TileWalk tw(threadIdx.x, blockDim.x);
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int q = threadIdx.x + 256 * m;
            if (q < TILE3) {
                const int b0 = tw.l0 + 3 + UBOX_X * (tw.l1 + TILE * tw.l2);
                r[m] = make_float4(box[b0], box[b0 + UBOX_X * TILE * TILE], box[b0 + 2 * UBOX_X * TILE * TILE], 0.f);
            }
            tw.next();
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < PER; ++m) {
            const int q = threadIdx.x + 256 * m;
            if (q < TILE3) tile[q] = r[m];
        }
    } else {
        cp_async_wait_all();
    }
    float dmax = 0.f;  // adaptive separation: this thread's largest displacement
    for (int p = s; p < e; p += csz) {
        if (p != s) {
            __syncthreads();  // the previous chunk is done with the records
            if (threadIdx.x < 8) count[threadIdx.x] = 0;
            __syncthreads();
            sort_chunk(p);
        }
        __syncthreads();  // the records, and the tile before the first chunk
        for (int q = threadIdx.x; q < slots; q += IT_CHUNK) {
            if ((q >> 3) >= n0) continue;
            const float4 rec = srec[f0 + (q >> 3)];
            float w[3][4];
            peskin4(rec.x, w[0]);
            peskin4(rec.y, w[1]);
            peskin4(rec.z, w[2]);
            const float4 *first = tile + __float_as_int(rec.w);
            float U0 = 0.f, U1 = 0.f, U2 = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float wyz = w[1][b] * w[2][c];
                    const float4 *row = first + IT_Y * b + IT_Z * c;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const float wa = wyz * w[0][a];
                        const float4 t = row[a];
                        U0 += wa * t.x;
                        U1 += wa * t.y;
                        U2 += wa * t.z;
                    }
                }
            srec[f0 + (q >> 3)] = make_float4(U0, U1, U2, 0.f);
        }
        // the moves, in the bin's order (neighbouring ids: coalesced accesses;
        // from the sorted lanes the 101 x 83 x 119 chamber with Adams-Bashforth
        // took 41 instead of 28 us)
        __syncthreads();
        if (own >= 0) {
            const float4 U = srec[at];
            dmax = fmaxf(dmax, move_vertex<INTEG>(v, own, U.x, U.y, U.z));
        }
    }
    if (v.adapt) adapt_max(v.adapt, (double)dmax);  // (FP64 once per thread, adaptive runs only)
}

// Peskin weights and their derivatives d/dt for the fraction t
template <typename R>
__device__ __forceinline__ void peskin4_d(R t, R *w, R *dw) {
    const R q = sqrt_r(R(1) + R(4) * t - R(4) * t * t);
    const R qp = (R(2) - R(4) * t) / q;
    w[0] = (R(3) - R(2) * t - q) * R(0.125);
    w[1] = (R(3) - R(2) * t + q) * R(0.125);
    w[2] = (R(1) + R(2) * t + q) * R(0.125);
    w[3] = (R(1) + R(2) * t - q) * R(0.125);
    dw[0] = (R(-2) - qp) * R(0.125);
    dw[1] = (R(-2) + qp) * R(0.125);
    dw[2] = (R(2) + qp) * R(0.125);
    dw[3] = (R(2) - qp) * R(0.125);
}

// Adjoint of the coupling operators at the vertices (differentiation form):
// for each vertex v of a bin, with the lattice field A staged like the
// velocity in interpolate_kernel,
//   out_interp[v]  = sum_x w(X_v, x) A(x)                  (interpolation)
//   out_grad[v]   += sum_x (A(x) . B[v]) grad_X w(X_v, x)  (position derivative)
// grad_X w = (w'_x w_y w_z, w_x w'_y w_z, w_x w_y w'_z).  Either output may
// be null (B is then unused).  out_grad may alias B: a vertex reads B[v]
// before its own write.
constexpr int VF_CAP = 16;  // vertices per chunk
template <typename R>
__global__ void __launch_bounds__(256) vertex_field_kernel(View<R> v, const R *A, const R *B, R *out_grad,
                                                           R *out_interp, int parts) {
    wait_previous();
    constexpr int CAP = VF_CAP;
    const int k = bin_of(v, blockIdx.x % v.nbins), part = blockIdx.x / v.nbins;  // CTA part takes chunks part, part + parts, ...
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1];
    if (s + part * CAP >= e) return;
    __shared__ R tile[3][TILE_SMEM];
    __shared__ int srow[CAP], sperm[CAP];
    __shared__ R sw[24 * CAP], sB[3 * CAP];
    __shared__ int jtab[3][TILE];
    int org[3];
    bin_origin(v, k, org);
    if (threadIdx.x < 3 * TILE) {
        const int d = threadIdx.x / TILE, l = threadIdx.x % TILE;
        const int dims = d == 0 ? v.nx : (d == 1 ? v.ny : v.nz);
        int j = org[d] - 1 + l;
        if (v.per[d]) j = wrap(j, dims);
        else if (j < 0 || j >= dims) j = -1;
        jtab[d][l] = j;
    }
    __syncthreads();
    stage_tile(v, A, jtab, tile);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int h = lane >> 4, b = lane & 3, c = (lane >> 2) & 3;
    for (int c0 = s + part * CAP; c0 < e; c0 += parts * CAP) {
        const int n = min(CAP, e - c0);
        if (c0 != s + part * CAP) __syncthreads();  // the previous chunk's records
        stage_chunk(v, c0, n, org, srow, sperm, [&](int j, int i, int ax, R t) {
            peskin4_d(t, sw + 24 * j + 4 * ax, sw + 24 * j + 12 + 4 * ax);
            sB[3 * j + ax] = B ? B[3 * (size_t)i + ax] : R(0);
        });
        if (c0 == s + part * CAP) cp_async_wait_all();  // the tile
        __syncthreads();
        for (int q0 = 2 * warp; q0 < n; q0 += 2 * nw) {  // uniform per warp: shuffles below
            const int q = q0 + h;
            R UG[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
            const int row0 = q < n ? srow[q] : -1;
            if (row0 >= 0) {
                const R *w = sw + 24 * q, *dw = w + 12;
                const R Bv[3] = {sB[3 * q], sB[3 * q + 1], sB[3 * q + 2]};
                const R wy = w[4 + b], wz = w[8 + c], dwy = dw[4 + b], dwz = dw[8 + c];
                const int row = row0 + TS_Y * b + TS_Z * c;
                // along x first: sum_a w_a A and sum_a w'_a (A . B)
                R tx[3] = {R(0), R(0), R(0)}, dx = R(0);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const R A0 = tile[0][row + a], A1 = tile[1][row + a], A2 = tile[2][row + a];
                    tx[0] += w[a] * A0;
                    tx[1] += w[a] * A1;
                    tx[2] += w[a] * A2;
                    dx += dw[a] * (A0 * Bv[0] + A1 * Bv[1] + A2 * Bv[2]);
                }
                const R wyz = wy * wz, sx = tx[0] * Bv[0] + tx[1] * Bv[1] + tx[2] * Bv[2];
                for (int d = 0; d < 3; ++d) UG[d] = wyz * tx[d];
                UG[3] = dx * wyz;
                UG[4] = sx * (dwy * wz);
                UG[5] = sx * (wy * dwz);
            }
            R S[6];
            sum16(UG, S);
            if (row0 >= 0 && (lane & 15) == 0) {
                const size_t vid = (size_t)sperm[q];
                for (int d = 0; d < 3; ++d) {
                    if (out_interp) out_interp[3 * vid + d] = S[d];
                    if (out_grad) out_grad[3 * vid + d] += S[3 + d];
                }
            }
        }
    }
}

// FP32 form of vertex_field_kernel: one thread per vertex over a float4
// tile, as in interpolate_v4_kernel
__global__ void __launch_bounds__(256) vertex_field_v4_kernel(View<float> v, const float *A, const float *B,
                                                              float *out_grad, float *out_interp) {
    wait_previous();
    const int k = bin_of(v, blockIdx.x);
    if (HEMO_BOUNDS_CHECK && k < 0) return;
    const int s = v.start[k], e = v.start[k + 1];
    if (s == e) return;
    __shared__ float4 tile[TILE_SMEM];
    __shared__ int jtab[3][TILE];
    int org[3];
    bin_origin(v, k, org);
    if (threadIdx.x < 3 * TILE) {
        const int d = threadIdx.x / TILE, l = threadIdx.x % TILE;
        const int dims = d == 0 ? v.nx : (d == 1 ? v.ny : v.nz);
        int j = org[d] - 1 + l;
        if (v.per[d]) j = wrap(j, dims);
        else if (j < 0 || j >= dims) j = -1;
        jtab[d][l] = j;
    }
    __syncthreads();
    const size_t N = (size_t)v.N;
    TileWalk tw(threadIdx.x, blockDim.x);
    for (int q = threadIdx.x; q < TILE3; q += blockDim.x, tw.next()) {  // (asynchronous: all loads in flight at once)
        const int jx = jtab[0][tw.l0], jy = jtab[1][tw.l1], jz = jtab[2][tw.l2];
        float4 *dst = tile + tw.l0 + TS_Y * tw.l1 + TS_Z * tw.l2;
        if ((jx | jy | jz) >= 0) {
            const size_t n = (size_t)jx + (size_t)v.nx * ((size_t)jy + (size_t)v.ny * jz);
            cp_async4(&dst->x, A + n);
            cp_async4(&dst->y, A + N + n);
            cp_async4(&dst->z, A + 2 * N + n);
        } else {
            *dst = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    cp_async_wait_all();
    __syncthreads();
    for (int j = s + threadIdx.x; j < e; j += blockDim.x) {
        const int i = v.perm[j];
        float w[3][4], dw[3][4];
        int r0 = 0;
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int b = v.anc_i[3 * (size_t)i + d] - org[d];
            ok &= b >= 0 && b < BLK;
            r0 += b * (d == 0 ? 1 : (d == 1 ? TS_Y : TS_Z));
            peskin4_d(v.anc_t[3 * (size_t)i + d], w[d], dw[d]);
        }
        if (!ok) continue;
        const float B0 = B ? B[3 * (size_t)i] : 0.f, B1 = B ? B[3 * (size_t)i + 1] : 0.f, B2 = B ? B[3 * (size_t)i + 2] : 0.f;
        float U0 = 0.f, U1 = 0.f, U2 = 0.f, G0 = 0.f, G1 = 0.f, G2 = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float wyz = w[1][b] * w[2][c], dyz = dw[1][b] * w[2][c], ydz = w[1][b] * dw[2][c];
                const float4 *row = tile + r0 + TS_Y * b + TS_Z * c;
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const float4 t = row[a];
                    const float wa = w[0][a] * wyz;
                    U0 += wa * t.x;
                    U1 += wa * t.y;
                    U2 += wa * t.z;
                    const float sAB = t.x * B0 + t.y * B1 + t.z * B2;
                    G0 += sAB * dw[0][a] * wyz;
                    G1 += sAB * w[0][a] * dyz;
                    G2 += sAB * w[0][a] * ydz;
                }
            }
        if (out_interp) {
            out_interp[3 * (size_t)i] = U0;
            out_interp[3 * (size_t)i + 1] = U1;
            out_interp[3 * (size_t)i + 2] = U2;
        }
        if (out_grad) {
            out_grad[3 * (size_t)i] += G0;
            out_grad[3 * (size_t)i + 1] += G1;
            out_grad[3 * (size_t)i + 2] += G2;
        }
    }
}

// four consecutive components per thread: 16-byte loads and stores in FP32
// (a thread per vertex, with strided 4- and 8-byte accesses: 219 us on the pipe's
// 12.6 M vertices; one component per thread 254, this 206)
template <typename R>
__global__ void __launch_bounds__(256) verts_out_kernel(View<R> v, double *X, double *F) {
    wait_previous();
    const unsigned q0 = 4u * (blockIdx.x * 256u + threadIdx.x), n = 3u * (unsigned)v.nv;
    if (q0 >= n) return;
    const bool vec = sizeof(R) == 4 && q0 + 4 <= n && (((uintptr_t)X | (uintptr_t)F) & 15) == 0;
    R o[4] = {}, f[4] = {};
    if (vec) {
        if (X) ld4_any(v.off + q0, o);
        if (F) ld4_any(v.Fv + q0, f);
    } else {
        for (unsigned k = 0; k < 4 && q0 + k < n; ++k) {
            if (X) o[k] = v.off[q0 + k];
            if (F) f[k] = v.Fv[q0 + k];
        }
    }
    double x[4] = {};
    if (X)
        for (unsigned k = 0; k < 4 && q0 + k < n; ++k) {
            const unsigned q = q0 + k, i = q / 3, d = q - 3 * i;
            x[k] = v.ctr[3 * (size_t)v.vcell[i] + d] + (double)o[k];
        }
    if (vec) {
        if (X) {
            reinterpret_cast<double2 *>(X + q0)[0] = make_double2(x[0], x[1]);
            reinterpret_cast<double2 *>(X + q0)[1] = make_double2(x[2], x[3]);
        }
        if (F) {
            reinterpret_cast<double2 *>(F + q0)[0] = make_double2((double)f[0], (double)f[1]);
            reinterpret_cast<double2 *>(F + q0)[1] = make_double2((double)f[2], (double)f[3]);
        }
    } else {
        for (unsigned k = 0; k < 4 && q0 + k < n; ++k) {
            if (X) X[q0 + k] = x[k];
            if (F) F[q0 + k] = (double)f[k];
        }
    }
}

template <typename R>
__global__ void set_vertices_kernel(View<R> v, const double *X) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= v.nv) return;
    const int c = v.vcell[i];
    for (int d = 0; d < 3; ++d) v.off[3 * (size_t)i + d] = R(X[3 * (size_t)i + d] - v.ctr[3 * c + d]);
}

}  // namespace

template <typename R>
void launch_bins(const View<R> &v, cudaStream_t st, bool stable) {
    cudaMemsetAsync(v.counts, 0, sizeof(int) * v.nbins, st);
    launch_next(anchor_count_kernel<R>, nblocks(v.nv, 256), 256, 0, st, v);
    launch_next(scan_kernel, 1, 1024, 0, st, v.counts, v.start, v.cursor, v.nbins, nullptr, 0, 0);
    if (stable) {
        launch_next(scatter_kernel, nblocks(v.nv, 256), 256, 0, st, v.key, v.cursor, v.perm_raw, v.nv, v.status);
        launch_next(sort_bins_kernel, nblocks((long long)v.nbins * 32, 128), 128, 0, st, v.start, v.perm_raw, v.perm, v.nbins);
    } else {
        launch_next(scatter_kernel, nblocks(v.nv, 256), 256, 0, st, v.key, v.cursor, v.perm, v.nv, v.status);
    }
}

template <typename R>
void launch_bin_ranges(const View<R> &v, cudaStream_t st) {
    const int nbins = v.nbins + (v.le ? 1 : 0);  // (+ the Lees-Edwards bin)
    if (nbins <= SMALL_BINS && v.nv <= SMALL_NV) {
        launch_next(scan_scatter_kernel, 1, 1024, 0, st, v.counts, v.start, nbins, v.key, v.perm, v.nv, v.status);
        return;
    }
    launch_next(scan_kernel, 1, 1024, 0, st, v.counts, v.start, v.cursor, nbins, v.order, v.nbins, v.nv / v.nbins);
    launch_next(scatter_kernel, nblocks(v.nv, 256), 256, 0, st, v.key, v.cursor, v.perm, v.nv, v.status);
}

template <typename R>
void launch_spread(const View<R> &v, cudaStream_t st) {
    if constexpr (std::is_same<R, float>::value) launch_next(spread_tile_f32_kernel, v.nbins, SP_CHUNK, 0, st, v);
    else launch_next(spread_tile_kernel, 3 * v.nbins, SP64_THREADS, 0, st, v);
    // (across a periodic edge the tiles' positions are those of whole blocks only;
    // the general gather for every block of such a lattice: FP32 channel 128 x 64 x
    // 253 288 us a step, 128 x 64 x 256 269.  For the edge layers alone, with
    // spread_gather3_kernel for the rest, 284, but the second launch costs small
    // lattices more: 61 x 64 x 253 151 -> 155, 45 x 39 x 61 in FP64 186 -> 196 us)
    const int dims[3] = {v.nx, v.ny, v.nz};
    bool regular = true;
    for (int d = 0; d < 3; ++d) regular &= v.nb[d] >= 3 && (!v.per[d] || dims[d] % BLK == 0);
    if (regular) launch_next(spread_gather3_kernel<R>, v.nbins, 256, 0, st, v);
    else launch_next(spread_gather_kernel<R>, v.nbins, 256, 0, st, v);
}

template <typename R, int INTEG>
void launch_interpolate_as(const View<R> &v, cudaStream_t st) {
    if constexpr (std::is_same<R, float>::value) {
        // the tensor map describes the step's u array only (the adjoint's
        // recomputation keeps u per step elsewhere)
        View<float> w = v;
        CUtensorMap map;
        if (v.u_tmap && v.u_tmap_base == (const void *)v.u) {
            std::memcpy(&map, v.u_tmap, sizeof(map));
        } else {
            std::memset(&map, 0, sizeof(map));
            w.u_tmap = nullptr;
        }
        launch_next(interpolate_v4_kernel<INTEG>, v.nbins, IT_CHUNK, 0, st, w, map);
    }
    else launch_next(interpolate_kernel<R, INTEG>, v.nbins * FP64_BIN_PARTS, 256, 0, st, v, FP64_BIN_PARTS);
}

template <typename R>
void launch_interpolate(const View<R> &v, cudaStream_t st) {
    if (v.integ == 2) launch_interpolate_as<R, 2>(v, st);
    else if (v.integ == 1) launch_interpolate_as<R, 1>(v, st);
    else launch_interpolate_as<R, 0>(v, st);
}

template <typename R>
void launch_hold_bins(const View<R> &v, cudaStream_t st) {
    if (v.nv) launch_next(hold_bins_kernel<R>, nblocks(v.nv, 256), 256, 0, st, v);
}

void launch_adapt_decide(unsigned long long *adapt, double tol, int every, cudaStream_t st) {
    launch_next(adapt_decide_kernel, 1, 1, 0, st, adapt, tol, every);
}

template <typename R>
void launch_vertex_field(const View<R> &v, const R *field, const R *vec, R *out_grad, R *out_interp, cudaStream_t st) {
    if constexpr (std::is_same<R, float>::value)
        launch_next(vertex_field_v4_kernel, v.nbins, 256, 0, st, v, field, vec, out_grad, out_interp);
    else
        launch_next(vertex_field_kernel<R>, v.nbins * FP64_BIN_PARTS, 256, 0, st, v, field, vec, out_grad, out_interp, FP64_BIN_PARTS);
}

template <typename R>
void launch_verts_out(const View<R> &v, double *X, double *F, cudaStream_t st) {
    if (v.nv) launch_next(verts_out_kernel<R>, nblocks(3LL * v.nv, 1024), 256, 0, st, v, X, F);
}

template <typename R>
void launch_set_vertices(const View<R> &v, const double *X, cudaStream_t st) {
    if (v.nv) set_vertices_kernel<R><<<nblocks(v.nv, 256), 256, 0, st>>>(v, X);
}

#define HEMO_INST(R)                                                                      \
    template void launch_bins<R>(const View<R> &, cudaStream_t, bool);                    \
    template void launch_bin_ranges<R>(const View<R> &, cudaStream_t);                     \
    template void launch_spread<R>(const View<R> &, cudaStream_t);                        \
    template void launch_interpolate<R>(const View<R> &, cudaStream_t);                   \
    template void launch_hold_bins<R>(const View<R> &, cudaStream_t);                     \
    template void launch_verts_out<R>(const View<R> &, double *, double *, cudaStream_t); \
    template void launch_vertex_field<R>(const View<R> &, const R *, const R *, R *, R *, cudaStream_t); \
    template void launch_set_vertices<R>(const View<R> &, const double *, cudaStream_t);
HEMO_INST(double)
HEMO_INST(float)

}  // namespace hemo

// ===========================================================================
// Vertex binning without any device allocation.
//
// Some callers cannot let a library allocate device memory: code that runs
// inside another framework's memory budget (a caching allocator that owns
// all of the GPU's memory), latency-critical loops in which cudaMalloc's
// implicit device synchronisation is not acceptable, or tools that hold
// vertex positions in their own buffers and no simulation handle.  For them
// hemo_bin_vertices_noalloc runs the same binning kernels as the step on
// caller-owned inputs and outputs, with its scratch (block counts, block
// cursors, unsorted permutation) in the file-scope array below.  The array
// is part of the loaded module: every GPU that loads the library holds its
// 5 MiB until the process exits.
// ===========================================================================
#include <mutex>

namespace hemo {

namespace {

constexpr int NOALLOC_MAX_VERTICES = 1 << 20;  // 1,048,576 vertices
constexpr int NOALLOC_MAX_BINS = 1 << 17;      // 131,072 blocks of 8^3 nodes

// [0, MAX_BINS): counts; [MAX_BINS, 2 MAX_BINS): cursors; then the unsorted
// permutation (MAX_VERTICES entries)
static __device__ __align__(256) int g_bin_scratch[2 * NOALLOC_MAX_BINS + NOALLOC_MAX_VERTICES];

// Device address of g_bin_scratch per device; in host code the symbol is
// only a host-side stand-in, so its address is taken once per device with
// cudaGetSymbolAddress while that device is current.
constexpr int NOALLOC_MAX_DEVICES = 64;
int *g_bin_scratch_dev[NOALLOC_MAX_DEVICES] = {};
std::mutex g_bin_scratch_mutex;

// key and count of each vertex from absolute FP64 positions (same floor,
// wrap and clamp rule as the step's anchor kernel)
__global__ void abs_key_count_kernel(const double *X, int nv, int nx, int ny, int nz, int px, int py, int pz,
                                     int nb0, int nb1, int *key, int *counts) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nv) return;
    const int dims[3] = {nx, ny, nz};
    const int per[3] = {px, py, pz};
    int b[3];
    for (int d = 0; d < 3; ++d) {
        int j = (int)floor(X[3 * (size_t)i + d]);
        if (per[d]) j = wrap(j, dims[d]);
        const int jc = j < 0 ? 0 : (j >= dims[d] ? dims[d] - 1 : j);
        b[d] = jc / BLK;
    }
    const int k = b[0] + nb0 * (b[1] + nb1 * b[2]);
    key[i] = k;
    atomicAdd(counts + k, 1);
}

int noalloc_fail(int code, const char *msg) {
    set_last_error(msg);  // reported by hemo_last_error()
    return code;
}

}  // namespace

}  // namespace hemo

extern "C" int hemo_bin_vertices_noalloc(const double *verts, int nv, int nx, int ny, int nz, const int32_t *periodic,
                                         int32_t *key, int32_t *perm, int32_t *start, void *cuda_stream) {
    using namespace hemo;
    if (nx < 1 || ny < 1 || nz < 1 || nv < 0 || !periodic || !start || (nv > 0 && (!verts || !key || !perm)))
        return noalloc_fail(HEMO_ERR_ARG, "hemo_bin_vertices_noalloc: bad sizes or null pointer");
    if (nv > NOALLOC_MAX_VERTICES)
        return noalloc_fail(HEMO_ERR_ARG, "hemo_bin_vertices_noalloc: more than 1,048,576 vertices");
    // block counts in 64 bits; each factor is checked before the product so
    // that no intermediate can overflow
    const long long nb0 = (long long)nx / BLK + (nx % BLK != 0), nb1 = (long long)ny / BLK + (ny % BLK != 0),
                    nb2 = (long long)nz / BLK + (nz % BLK != 0);
    if (nb0 > NOALLOC_MAX_BINS || nb1 > NOALLOC_MAX_BINS || nb2 > NOALLOC_MAX_BINS || nb0 * nb1 > NOALLOC_MAX_BINS ||
        nb0 * nb1 * nb2 > NOALLOC_MAX_BINS)
        return noalloc_fail(HEMO_ERR_ARG, "hemo_bin_vertices_noalloc: more than 131,072 lattice blocks of 8^3 nodes");
    const int nbins = (int)(nb0 * nb1 * nb2);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES)
        return noalloc_fail(HEMO_ERR_CUDA, "hemo_bin_vertices_noalloc: no usable current device");
    int *scratch;
    {
        std::lock_guard<std::mutex> lock(g_bin_scratch_mutex);
        if (!g_bin_scratch_dev[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_bin_scratch);
            if (e != cudaSuccess || !p) return noalloc_fail(HEMO_ERR_CUDA, "hemo_bin_vertices_noalloc: cudaGetSymbolAddress failed");
            g_bin_scratch_dev[dev] = (int *)p;
        }
        scratch = g_bin_scratch_dev[dev];
    }
    int *counts = scratch, *cursor = scratch + NOALLOC_MAX_BINS, *perm_raw = scratch + 2 * NOALLOC_MAX_BINS;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // the array keeps the previous call's contents: the counts must start at zero
    if (cudaMemsetAsync(counts, 0, sizeof(int) * nbins, st) != cudaSuccess)
        return noalloc_fail(HEMO_ERR_CUDA, "hemo_bin_vertices_noalloc: clearing the counts failed");
    if (nv > 0)
        abs_key_count_kernel<<<(nv + 255) / 256, 256, 0, st>>>(verts, nv, nx, ny, nz, periodic[0] != 0, periodic[1] != 0,
                                                               periodic[2] != 0, (int)nb0, (int)nb1, key, counts);
    scan_kernel<<<1, 1024, 0, st>>>(counts, start, cursor, nbins, nullptr, 0, 0);
    if (nv > 0) {
        scatter_kernel<<<(nv + 255) / 256, 256, 0, st>>>(key, cursor, perm_raw, nv, nullptr);
        sort_bins_kernel<<<(int)(((long long)nbins * 32 + 127) / 128), 128, 0, st>>>(start, perm_raw, perm, nbins);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return noalloc_fail(HEMO_ERR_CUDA, cudaGetErrorString(e));
    return HEMO_OK;
}
