// Device primitives used by the index builder and the seeding pipeline: prefix scans and a
// stable LSD radix sort of (u64 key, u32 value) pairs.
#include "common.cuh"

namespace {

constexpr int SCAN_T = 256;      // threads per scan block
constexpr int SCAN_I = 16;       // items per thread
constexpr size_t SCAN_TILE = (size_t)SCAN_T * SCAN_I;

struct OpSum {
    template <class T> __device__ __forceinline__ T operator()(T a, T b) const { return a + b; }
    template <class T> static __device__ __forceinline__ T id() { return T(0); }
};
struct OpMax {
    template <class T> __device__ __forceinline__ T operator()(T a, T b) const { return a > b ? a : b; }
    template <class T> static __device__ __forceinline__ T id() { return T(0); }
};

template <class T, class Op>
__device__ __forceinline__ T warp_incl(T v, Op op) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T o = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v = op(v, o);
    }
    return v;
}

// Block-wide exclusive scan of one value per thread; returns the exclusive prefix and the total.
template <class T, class Op>
__device__ __forceinline__ T block_excl(T v, T &total, Op op) {
    __shared__ T ws[SCAN_T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = warp_incl(v, op);
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < SCAN_T / 32 ? ws[lane] : Op::template id<T>();
        T wi = warp_incl(w, op);
        if (lane < SCAN_T / 32) ws[lane] = wi;   // inclusive over warps
    }
    __syncthreads();
    T warp_pre = warp == 0 ? Op::template id<T>() : ws[warp - 1];
    total = ws[SCAN_T / 32 - 1];
    T ex = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) ex = Op::template id<T>();
    __syncthreads();
    return op(warp_pre, ex);
}

// A thread's SCAN_I items of a full tile in 32-byte accesses (whole sectors; one item at a time, the lanes
// of a load lie 64 or 128 bytes apart and each sector is asked for several times).
template <class T>
__device__ __forceinline__ void load_items(const T *p, T v[SCAN_I]) {
    constexpr int PER = 32 / sizeof(T);
#pragma unroll
    for (int i = 0; i < SCAN_I / PER; ++i) {
        u64 a, b, c, d;
        asm volatile("ld.global.v4.u64 {%0,%1,%2,%3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p + PER * i));
        const u64 x[4] = {a, b, c, d};
#pragma unroll
        for (int j = 0; j < PER; ++j)
            v[PER * i + j] = sizeof(T) == 8 ? (T)x[j & 3] : (T)(x[(j / 2) & 3] >> (32 * (j & 1)));
    }
}
template <class T>
__device__ __forceinline__ void store_items(T *p, const T v[SCAN_I]) {
    constexpr int PER = 32 / sizeof(T);
#pragma unroll
    for (int i = 0; i < SCAN_I / PER; ++i) {
        u64 x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            x[j] = sizeof(T) == 8 ? (u64)v[PER * i + j]
                                  : (u64)(u32)v[PER * i + (2 * j) % PER] | ((u64)(u32)v[PER * i + (2 * j + 1) % PER] << 32);
        asm volatile("st.global.v4.u64 [%0], {%1,%2,%3,%4};" ::"l"(p + PER * i), "l"(x[0]), "l"(x[1]), "l"(x[2]), "l"(x[3])
                     : "memory");
    }
}
__device__ __forceinline__ bool sectors(const void *p) { return ((uintptr_t)p & 31) == 0; }

// With n_dev (device) only the first min(n, *n_dev) items take part: tiles past them read and write
// nothing but an identity partial.
template <class T, class Op>
__global__ void k_scan_reduce(const T *__restrict__ in, size_t n, const u64 *n_dev, T *__restrict__ part, Op op) {
    if (n_dev && *n_dev < n) n = (size_t)*n_dev;
    if (blockIdx.x * SCAN_TILE >= n) {
        if (threadIdx.x == 0) part[blockIdx.x] = Op::template id<T>();
        return;
    }
    size_t base = blockIdx.x * SCAN_TILE + (size_t)threadIdx.x * SCAN_I;
    T acc = Op::template id<T>();
    if (base + SCAN_I <= n && sectors(in)) {
        T v[SCAN_I];
        load_items(in + base, v);
#pragma unroll
        for (int i = 0; i < SCAN_I; ++i) acc = op(acc, v[i]);
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_I; ++i)
            if (base + i < n) acc = op(acc, in[base + i]);
    }
    T tot;
    block_excl(acc, tot, op);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// Scans one tile; carry = scanned partial of this tile (exclusive), or identity for one tile.
template <class T, class Op, bool INCL>
__global__ void k_scan_apply(const T *in, T *out, size_t n, const u64 *n_dev, const T *__restrict__ carry, T *total, Op op) {
    if (n_dev && *n_dev < n) n = (size_t)*n_dev;
    if (blockIdx.x * SCAN_TILE >= n && !(total && blockIdx.x == gridDim.x - 1)) return;
    size_t base = blockIdx.x * SCAN_TILE + (size_t)threadIdx.x * SCAN_I;
    T v[SCAN_I];
    T acc = Op::template id<T>();
    const bool full = base + SCAN_I <= n;
    if (full && sectors(in)) {
        load_items(in + base, v);
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_I; ++i) v[i] = base + i < n ? in[base + i] : Op::template id<T>();
    }
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) acc = op(acc, v[i]);
    T tot;
    T pre = block_excl(acc, tot, op);
    T c = carry ? carry[blockIdx.x] : Op::template id<T>();
    pre = op(c, pre);
#pragma unroll
    for (int i = 0; i < SCAN_I; ++i) {
        const T nx = op(pre, v[i]);
        v[i] = INCL ? nx : pre;
        pre = nx;
    }
    if (full && sectors(out)) {
        store_items(out + base, v);
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_I; ++i)
            if (base + i < n) out[base + i] = v[i];
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = op(c, tot);
}

size_t level_blocks(size_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

template <class T, class Op, bool INCL>
int scan_impl(const T *in, T *out, size_t n, T *total, void *tmp, cudaStream_t st, Op op, const u64 *n_dev = nullptr) {
    if (n == 0) return MB_OK;
    size_t nb = level_blocks(n);
    if (nb == 1) {
        k_scan_apply<T, Op, INCL><<<1, SCAN_T, 0, st>>>(in, out, n, n_dev, nullptr, total, op);
        MB_KCHECK();
        return MB_OK;
    }
    T *part = (T *)tmp;
    void *rest = (void *)((char *)tmp + ((nb * sizeof(u64) + 255) & ~(size_t)255));
    k_scan_reduce<T, Op><<<(unsigned)nb, SCAN_T, 0, st>>>(in, n, n_dev, part, op);
    MB_KCHECK();
    // exclusive scan of the tile sums gives each tile's carry
    MB_TRY((scan_impl<T, Op, false>(part, part, nb, nullptr, rest, st, op)));
    k_scan_apply<T, Op, INCL><<<(unsigned)nb, SCAN_T, 0, st>>>(in, out, n, n_dev, part, total, op);
    MB_KCHECK();
    return MB_OK;
}

// exclusive sum; total: of all inputs (written by the last tile)
template <class T>
int scan_excl_total(const T *in, T *out, size_t n, T *total, void *tmp, cudaStream_t st, const u64 *n_dev) {
    if (n == 0) {
        if (total) MB_CK(cudaMemsetAsync(total, 0, sizeof(T), st));
        return MB_OK;
    }
    return scan_impl<T, OpSum, false>(in, out, n, total, tmp, st, OpSum(), n_dev);
}

}  // namespace

size_t scan_tmp_bytes(size_t n) {
    size_t b = 0;
    size_t nb = level_blocks(n);
    while (nb > 1) {
        b += ((nb * sizeof(u64) + 255) & ~(size_t)255);
        nb = level_blocks(nb);
    }
    return b + 256;
}

int scan_exclusive_u64(const u64 *in, u64 *out, size_t n, u64 *total, void *tmp, cudaStream_t st, const u64 *n_dev) {
    return scan_excl_total<u64>(in, out, n, total, tmp, st, n_dev);
}

int scan_exclusive_u32(const u32 *in, u32 *out, size_t n, u32 *total, void *tmp, cudaStream_t st) {
    return scan_excl_total<u32>(in, out, n, total, tmp, st, nullptr);
}

int scan_inclusive_max_u32(const u32 *in, u32 *out, size_t n, void *tmp, cudaStream_t st, const u64 *n_dev) {
    return scan_impl<u32, OpMax, true>(in, out, n, nullptr, tmp, st, OpMax(), n_dev);
}

// ============================================================================ radix sort
namespace {
constexpr int RS_T = 256;        // threads (8 warps)
constexpr int RS_I = 16;         // items per thread
constexpr size_t RS_TILE = (size_t)RS_T * RS_I;

// n_dev (device, may be null): the number of items to sort when it is below n (the tiles past it
// count nothing and move nothing).
__device__ __forceinline__ size_t items(size_t n, const u64 *n_dev) { return n_dev && *n_dev < n ? (size_t)*n_dev : n; }

template <class K>
__global__ void __launch_bounds__(RS_T) k_radix_up(const K *__restrict__ keys, size_t n, const u64 *n_dev, int shift,
                                                   u32 mask, u32 *__restrict__ hist, size_t tiles) {
    __shared__ u32 h[256];
    n = items(n, n_dev);
    h[threadIdx.x] = 0;
    __syncthreads();
    size_t base = blockIdx.x * RS_TILE;
#pragma unroll 4
    for (int it = 0; it < RS_I; ++it) {
        size_t idx = base + (size_t)it * RS_T + threadIdx.x;
        if (idx < n) atomicAdd(&h[(u32)(keys[idx] >> shift) & mask], 1u);
    }
    __syncthreads();
    hist[(size_t)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

// One tile: every item's place among the tile's items of the same or a smaller digit, the tile put in
// that order in shared memory, then written out, so that the items of a digit (16 on average) go out as
// one run.  Each warp owns a contiguous run of 32 * RS_I items; items keep their order inside a warp
// (iteration-major, lane-minor), warps keep theirs inside the tile, tiles theirs inside a digit: the
// scatter is stable.  Bound: the copy of 12 bytes per item; writing each item from its lane instead
// (partial sectors all over the digits) took 5 to 6 ms per pass of 200M items, this about 1.7 ms.
// Without VALS an item is a word, its key in the high half and its value in the low one; with K = u32 such
// words are made from keys and vals.
struct RadixTile {
    u64 key[RS_TILE];
    u32 val[RS_TILE];
    u32 wh[RS_T / 32][256];   // per warp and digit: items, then their first place in the tile
    u32 to[256];              // per digit: where its run goes, less its first place in the tile
};
template <class K, bool VALS>
__global__ void __launch_bounds__(RS_T, 3) k_radix_down(const K *__restrict__ keys, const u32 *__restrict__ vals,
                                                        u64 *__restrict__ okeys, u32 *__restrict__ ovals, size_t n,
                                                        const u64 *n_dev, int shift, u32 mask,
                                                        const u32 *__restrict__ offs, size_t tiles) {
    extern __shared__ __align__(16) unsigned char smem[];
    RadixTile &S = *reinterpret_cast<RadixTile *>(smem);
    constexpr bool JOIN = sizeof(K) == 4;
    n = items(n, n_dev);
    const size_t tile0 = blockIdx.x * RS_TILE;
    if (tile0 >= n) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < (RS_T / 32) * 256; i += RS_T) (&S.wh[0][0])[i] = 0;
    const size_t base = tile0 + (size_t)warp * 32 * RS_I + lane;
    u64 k[RS_I];
    u32 rank[RS_I / 2];   // 16 bits each
#pragma unroll
    for (int it = 0; it < RS_I; ++it) {
        const size_t at = base + 32 * it;
        k[it] = at < n ? (JOIN ? (u64)keys[at] << 32 | vals[at] : (u64)keys[at]) : 0;
    }
    __syncthreads();
    const u32 lt = (1u << lane) - 1u;
#pragma unroll
    for (int it = 0; it < RS_I; ++it) {
        const bool ok = base + 32 * it < n;
        const u32 d = ok ? ((u32)(k[it] >> shift) & mask) : 256u;
        const u32 peers = __match_any_sync(0xffffffffu, d);
        const u32 b = ok ? S.wh[warp][d] : 0;
        const u32 rk = b + __popc(peers & lt);
        rank[it / 2] = it & 1 ? rank[it / 2] | (rk << 16) : rk;
        __syncwarp();
        if (ok && (peers & lt) == 0) S.wh[warp][d] = b + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        const u32 d = threadIdx.x;
        u32 cnt = 0;
#pragma unroll
        for (int w = 0; w < RS_T / 32; ++w) {
            const u32 t = S.wh[w][d];
            S.wh[w][d] = cnt;
            cnt += t;
        }
        u32 tot;
        const u32 first = block_excl(cnt, tot, OpSum());
#pragma unroll
        for (int w = 0; w < RS_T / 32; ++w) S.wh[w][d] += first;
        S.to[d] = offs[(size_t)d * tiles + blockIdx.x] - first;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < RS_I; ++it)
        if (base + 32 * it < n) {
            const u32 at = S.wh[warp][(u32)(k[it] >> shift) & mask] + ((rank[it / 2] >> (16 * (it & 1))) & 0xFFFFu);
            S.key[at] = k[it];
            if (VALS) S.val[at] = vals[base + 32 * it];
        }
    __syncthreads();
    const u32 cnt = (u32)(n - tile0 < RS_TILE ? n - tile0 : RS_TILE);
    for (u32 i = threadIdx.x; i < cnt; i += RS_T) {
        const u64 x = S.key[i];
        const u32 at = S.to[(u32)(x >> shift) & mask] + i;
        okeys[at] = x;
        if (VALS) ovals[at] = S.val[i];
    }
}

// out[at[t]] = v[t]
__global__ void k_permute(const u32 *__restrict__ at, const u32 *__restrict__ v, size_t n, u32 *__restrict__ out) {
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < n; t += (size_t)gridDim.x * blockDim.x)
        out[at[t]] = v[t];
}
// The same for words (place, value) of a permutation of [0, n), in order of place / PERM_WIN: window w of
// `out` takes exactly the words of the same numbers, so a block puts them in place in shared memory.
constexpr int PERM_BITS = 12;
constexpr u32 PERM_WIN = 1u << PERM_BITS;
__global__ void __launch_bounds__(256) k_permute_windows(const u64 *__restrict__ words, size_t n, u32 *__restrict__ out) {
    __shared__ u32 win[PERM_WIN];
    const size_t first = blockIdx.x * (size_t)PERM_WIN;
    const u32 len = (u32)(n - first < PERM_WIN ? n - first : PERM_WIN);
#pragma unroll 4
    for (u32 t = threadIdx.x; t < len; t += 256) {
        const u64 w = words[first + t];
        win[(u32)(w >> 32) & (PERM_WIN - 1)] = (u32)w;
    }
    __syncthreads();
    for (u32 t = threadIdx.x; t < len; t += 256) out[first + t] = win[t];
}
}  // namespace

// out[at[t]] = v[t], `at` a permutation of [0, n), n <= 2^bits.  Single words written all over memory move a
// sector each, or within what L2 holds a slot of its write rate each (200M ranks: 7.5 ms; after one radix pass
// on the place 4.6 ms).  From 2^24 items on the items are therefore sorted by place down to windows that fit
// shared memory, two passes up to 2^28 items and three above (200M ranks: 4.2 ms in all).
// a, b: room for n words each (vals and `v` may lie in b), tmp: radix_tmp_bytes(n).
int permute_u32(const u32 *at, const u32 *v, size_t n, int bits, u32 *out, u64 *a, u64 *b, void *tmp, cudaStream_t st) {
    if (n < (size_t)1 << 24 || n >= (1ULL << 32)) {
        k_permute<<<grid_for(n, 256), 256, 0, st>>>(at, v, n, out);
        MB_KCHECK();
        return MB_OK;
    }
    const size_t tiles = (n + RS_TILE - 1) / RS_TILE;
    u32 *hist = (u32 *)tmp;
    void *stmp = (char *)tmp + (((256 * tiles * sizeof(u32)) + 255) & ~(size_t)255);
    MB_CK(cudaFuncSetAttribute(k_radix_down<u32, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixTile)));
    MB_CK(cudaFuncSetAttribute(k_radix_down<u64, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixTile)));
    for (int sh = PERM_BITS; sh < bits; sh += 8) {
        const u32 mask = bits - sh < 8 ? (1u << (bits - sh)) - 1u : 255u;
        const bool first = sh == PERM_BITS;
        if (first) k_radix_up<u32><<<(unsigned)tiles, RS_T, 0, st>>>(at, n, nullptr, sh, mask, hist, tiles);
        else k_radix_up<u64><<<(unsigned)tiles, RS_T, 0, st>>>(b, n, nullptr, 32 + sh, mask, hist, tiles);
        MB_KCHECK();
        MB_TRY(scan_exclusive_u32(hist, hist, 256 * tiles, nullptr, stmp, st));
        if (first)
            k_radix_down<u32, false><<<(unsigned)tiles, RS_T, sizeof(RadixTile), st>>>(at, v, a, nullptr, n, nullptr, 32 + sh,
                                                                                       mask, hist, tiles);
        else
            k_radix_down<u64, false><<<(unsigned)tiles, RS_T, sizeof(RadixTile), st>>>(b, nullptr, a, nullptr, n, nullptr,
                                                                                       32 + sh, mask, hist, tiles);
        MB_KCHECK();
        u64 *t = a; a = b; b = t;
    }
    k_permute_windows<<<(unsigned)((n + PERM_WIN - 1) / PERM_WIN), 256, 0, st>>>(b, n, out);
    MB_KCHECK();
    return MB_OK;
}

size_t radix_tmp_bytes(size_t n) {
    size_t tiles = (n + RS_TILE - 1) / RS_TILE;
    size_t h = ((256 * tiles * sizeof(u32)) + 255) & ~(size_t)255;
    return h + scan_tmp_bytes(256 * tiles);
}

int radix_sort_pairs(u64 *keys, u32 *vals, u64 *keys_alt, u32 *vals_alt, size_t n, const BitRange *ranges,
                     int nranges, void *tmp, cudaStream_t st, const u64 *n_dev, bool *in_alt) {
    if (in_alt) *in_alt = false;
    if (n <= 1) return MB_OK;
    if (n >= (1ULL << 32)) {
        mb_set_error("radix_sort_pairs: %zu items exceed 2^32-1", n);
        return MB_ERR_ARG;
    }
    size_t tiles = (n + RS_TILE - 1) / RS_TILE;
    MB_CK(cudaFuncSetAttribute(k_radix_down<u64, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixTile)));
    u32 *hist = (u32 *)tmp;
    void *stmp = (char *)tmp + (((256 * tiles * sizeof(u32)) + 255) & ~(size_t)255);
    u64 *ka = keys, *kb = keys_alt;
    u32 *va = vals, *vb = vals_alt;
    int passes = 0;
    for (int r = 0; r < nranges; ++r) {
        for (int sh = ranges[r].lo; sh < ranges[r].hi; sh += 8) {
            int w = ranges[r].hi - sh < 8 ? ranges[r].hi - sh : 8;
            u32 mask = (1u << w) - 1u;
            k_radix_up<u64><<<(unsigned)tiles, RS_T, 0, st>>>(ka, n, n_dev, sh, mask, hist, tiles);
            MB_KCHECK();
            MB_TRY(scan_exclusive_u32(hist, hist, 256 * tiles, nullptr, stmp, st));
            k_radix_down<u64, true><<<(unsigned)tiles, RS_T, sizeof(RadixTile), st>>>(ka, va, kb, vb, n, n_dev, sh, mask, hist, tiles);
            MB_KCHECK();
            u64 *tk = ka; ka = kb; kb = tk;
            u32 *tv = va; va = vb; vb = tv;
            ++passes;
        }
    }
    if (in_alt) {
        *in_alt = passes & 1;
    } else if (passes & 1) {
        MB_CK(cudaMemcpyAsync(keys, ka, n * sizeof(u64), cudaMemcpyDeviceToDevice, st));
        MB_CK(cudaMemcpyAsync(vals, va, n * sizeof(u32), cudaMemcpyDeviceToDevice, st));
    }
    return MB_OK;
}
