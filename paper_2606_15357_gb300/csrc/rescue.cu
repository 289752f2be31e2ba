// Mate-rescue prefilter of Section 2.7 (mb_rescue_prefilter): for a read P and a reference window
// R, M_t = #{(i, j) : P[i, i+q) = R[j, j+q), j - i = t}, and the result is max_t M_t.
//
// One warp per (read, window) pair, bit-parallel along each diagonal.  The warp writes, for each
// base a, the bit masks P_a (bit i = [P[i] = a]) and R_a (bit j = [R[j] = a], behind a zero pad so
// that negative diagonals read zeros) into its slice of shared memory, by ballots.  Lane l takes
// the diagonals t = t0 + l, t0 + l + 32, ...; on diagonal t the word D_k = OR_a P_a[k] & (R_a
// shifted by t) has bit i set where P[i] = R[i+t] (an N is in no mask, so it matches nothing), a
// q-mer match at i is a run of q set bits starting at i (q - 1 shifted ANDs, the next word
// carried in), and M_t is the popcount of those run starts.  64 positions of a diagonal cost
// about 30 integer operations instead of 64 code compares.
//
// Reads of at most 256 bases (k_qmer_words, the usual case) go without the base masks: the read and the
// window are kept as two code bits and a validity bit per base, 32 bases per word.
#include <algorithm>
#include <vector>
#include "common.cuh"

namespace {

// 64 bits of the padded mask m starting at bit b
__device__ __forceinline__ u64 bits_at(const u64 *__restrict__ m, u32 b) {
    const u32 w = b >> 6, s = b & 63;
    const u64 lo = m[w];
    return s ? (lo >> s) | (m[w + 1] << (64 - s)) : lo;
}

// Words per base of a pair's masks: P (np words), R (pad np + nr + np + 1 words).
__host__ __device__ __forceinline__ u32 words_p(u32 m) { return (m + 63) / 64; }
__host__ __device__ __forceinline__ u32 words_r(u32 m, u32 w) { return 2 * words_p(m) + (w + 63) / 64 + 1; }

// masks of x (len bases) at bit offset `shift` of 4 arrays of `stride` words (already zero)
__device__ __forceinline__ void build_masks(const u8 *__restrict__ x, u32 len, u64 *__restrict__ M, u32 stride,
                                            u32 shift, u32 lane) {
    u32 *M32 = reinterpret_cast<u32 *>(M);
    for (u32 c = 0; c * 32 < len; ++c) {
        const u32 i = c * 32 + lane;
        const u32 b = i < len ? x[i] : 4u;
#pragma unroll
        for (u32 a = 0; a < 4; ++a) {
            const u32 bal = __ballot_sync(0xffffffffu, b == a);
            if (lane == a) M32[2 * stride * a + (shift >> 5) + c] = bal;   // shift is a multiple of 64
        }
    }
}

__global__ void k_qmer_diag_max(const u8 *__restrict__ reads, const u64 *__restrict__ roff,
                                const u8 *__restrict__ wins, const u64 *__restrict__ woff, u32 npairs, u32 q,
                                u32 slice_words, u32 *__restrict__ best) {
    extern __shared__ u64 sm[];
    const u32 lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    u64 *S = sm + (size_t)wib * slice_words;
    const u32 nw = (gridDim.x * blockDim.x) >> 5;
    for (u32 p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < npairs; p += nw) {
        const u64 r0 = roff[p], w0 = woff[p];
        const u32 m = (u32)(roff[p + 1] - r0), w = (u32)(woff[p + 1] - w0);
        const u32 np = words_p(m), sr = words_r(m, w);
        u64 *Pm = S, *Rm = S + 4 * np;
        for (u32 k = lane; k < 4 * (np + sr); k += 32) S[k] = 0;
        __syncwarp();
        build_masks(reads + r0, m, Pm, np, 0, lane);
        build_masks(wins + w0, w, Rm, sr, 64 * np, lane);
        __syncwarp();
        const int mp = m >= q ? (int)(m - q + 1) : 0, wr = w >= q ? (int)(w - q + 1) : 0;
        u32 top = 0;
        if (mp > 0 && wr > 0) {
            for (int t = -(mp - 1) + (int)lane; t <= wr - 1; t += 32) {
                const u32 base = (u32)((int)(64 * np) + t);   // bit of R_a for j = t (>= 1)
                auto diag = [&](u32 k) -> u64 {
                    u64 d = 0;
#pragma unroll
                    for (u32 a = 0; a < 4; ++a) d |= Pm[a * np + k] & bits_at(Rm + a * sr, base + 64 * k);
                    return d;
                };
                u32 cnt = 0;
                u64 dn = diag(0);
                for (u32 k = 0; k < np; ++k) {
                    const u64 d = dn;
                    dn = k + 1 < np ? diag(k + 1) : 0;
                    u64 run = d;
                    for (u32 s = 1; s < q; ++s) run &= (d >> s) | (dn << (64 - s));
                    cnt += __popcll(run);
                }
                top = max(top, cnt);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
        if (lane == 0) best[p] = top;
        __syncwarp();   // the masks are rewritten for the next pair
    }
}

// ---------------------------------------------------------------------------- reads of up to 256 bases
// One warp per pair.  The read's NP words (low code bits, high code bits, valid) stay in registers of
// every lane; the window's words sit in shared memory, behind NP zero words.  Lane s takes the
// diagonals whose offset (t + 32 NP) is s modulo 32: for all of them the window is shifted by the same
// s bits, so each window word W is shifted once (three funnel shifts) and compared with all NP read
// words, word k then belonging to diagonal W - k.  A diagonal's words arrive in order, one per W: the
// word before it (prev) gets its runs of q matches now that the bits after it are known, by doubling
// (q = 7: x & x >> 1, & >> 2, & >> 3), and its count moves one place up.  About 15 operations per 32
// positions of a diagonal; the earlier form took about 120 per 64 (four base masks with two shared-
// memory loads each, q - 1 shifts).  Integer-bound: 1M pairs of 100-150 by 600 bases 11.0 -> 3.1 ms.
__device__ __forceinline__ u32 bits4(u32 x) { return ((x & 0x01010101u) * 0x10204080u) >> 28; }   // bit 0 of four bytes

struct Planes {
    u32 lo, hi, ok;
};
// The three planes of x[0, n), n <= 32, from the aligned words that hold its bytes.
__device__ __forceinline__ Planes planes_of(const u8 *__restrict__ x, u32 n) {
    Planes p{0, 0, 0};
    const u32 *a = reinterpret_cast<const u32 *>((uintptr_t)x & ~(uintptr_t)3);
    const u32 mis = (u32)((uintptr_t)x & 3), last = n ? (mis + n - 1) / 4 : 0;   // last aligned word holding a byte
    u32 w = n ? __ldg(a) : 0u;
#pragma unroll
    for (u32 q = 0; q < 8; ++q) {
        if (4 * q >= n) break;
        const u32 nx = q + 1 <= last ? __ldg(a + q + 1) : 0u;
        const u32 v = __funnelshift_r(w, nx, 8 * mis);
        w = nx;
        p.lo |= bits4(v) << (4 * q);
        p.hi |= bits4(v >> 1) << (4 * q);
        u32 t = v & 0xFCFCFCFCu;   // above 3: an N
        t |= t >> 4;
        t |= t >> 2;
        p.ok |= (bits4(t | t >> 1) ^ 15u) << (4 * q);
    }
    p.ok &= n >= 32 ? ~0u : (1u << n) - 1u;
    return p;
}

// Bits of d that start q set bits, dn being the word after it; s1..s4: the doubling's steps (0: none).
__device__ __forceinline__ u32 runs(u32 d, u32 dn, u32 s1, u32 s2, u32 s3, u32 s4) {
    d &= __funnelshift_r(d, dn, s1);
    dn &= dn >> s1;
    d &= __funnelshift_r(d, dn, s2);
    dn &= dn >> s2;
    d &= __funnelshift_r(d, dn, s3);
    if (s4) {
        dn &= dn >> s3;
        d &= __funnelshift_r(d, dn, s4);
    }
    return d;
}

template <int NP, bool Q7>
__global__ void __launch_bounds__(256) k_qmer_words(const u8 *__restrict__ reads, const u64 *__restrict__ roff,
                                                    const u8 *__restrict__ wins, const u64 *__restrict__ woff,
                                                    u32 npairs, u32 q, uint4 step, u32 win_words,
                                                    u32 *__restrict__ best) {
    extern __shared__ u32 smw[];   // per warp: three planes of win_words words
    const u32 lane = threadIdx.x & 31;
    u32 *const lo = smw + (threadIdx.x >> 5) * 3 * win_words, *const hi = lo + win_words, *const ok = hi + win_words;
    const u32 nw = (gridDim.x * blockDim.x) >> 5;
    const u32 s1 = Q7 ? 1u : step.x, s2 = Q7 ? 2u : step.y, s3 = Q7 ? 3u : step.z, s4 = Q7 ? 0u : step.w;
    for (u32 p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < npairs; p += nw) {
        const u64 r0 = roff[p], w0 = woff[p];
        const u32 m = (u32)(roff[p + 1] - r0), w = (u32)(woff[p + 1] - w0);
        u32 top = 0;
        if (m >= q && w >= q) {
            const u32 nr = (w + 31) / 32;
            // words 0..nr-1 of the window and NP of the read, one per lane and round
            u32 pl[NP], ph[NP], pv[NP];
            for (u32 c = 0; c < nr + NP; c += 32) {
                const u32 t = c + lane;
                const bool win = t < nr;
                const u32 at = 32 * (win ? t : t - nr), of = win ? w : (t < nr + NP ? m : 0u);
                const Planes v = planes_of((win ? wins + w0 : reads + r0) + at, at < of ? min(of - at, 32u) : 0u);
                if (win) {
                    lo[NP + t] = v.lo;
                    hi[NP + t] = v.hi;
                    ok[NP + t] = v.ok;
                }
#pragma unroll
                for (int k = 0; k < NP; ++k)
                    if (nr + k >= c && nr + k < c + 32) {   // the same for all lanes
                        pl[k] = __shfl_sync(0xffffffffu, v.lo, (int)(nr + k - c));
                        ph[k] = __shfl_sync(0xffffffffu, v.hi, (int)(nr + k - c));
                        pv[k] = __shfl_sync(0xffffffffu, v.ok, (int)(nr + k - c));
                    }
            }
            if (lane < NP) ok[lane] = 0;         // the zero words before the window, and two after it
            if (lane < 2) ok[NP + nr + lane] = 0;
            __syncwarp();
            u32 prev[NP], cnt[NP + 1];
#pragma unroll
            for (int k = 0; k < NP; ++k) prev[k] = cnt[k] = 0;
            cnt[NP] = 0;
            u32 a = lo[NP - 1], b = hi[NP - 1], c = ok[NP - 1];
            // every diagonal's last word is done NP steps after the window's last one
#pragma unroll 2
            for (u32 W = NP - 1; W < 2 * NP + nr; ++W) {
                u32 cur[NP];
                if (W < NP + nr) {
                    const u32 a2 = lo[W + 1], b2 = hi[W + 1], c2 = ok[W + 1];
                    const u32 sl = __funnelshift_r(a, a2, lane), sh = __funnelshift_r(b, b2, lane),
                              sv = __funnelshift_r(c, c2, lane);
                    a = a2;
                    b = b2;
                    c = c2;
#pragma unroll
                    for (int k = 0; k < NP; ++k) cur[k] = ~((pl[k] ^ sl) | (ph[k] ^ sh)) & pv[k] & sv;
                } else {
#pragma unroll
                    for (int k = 0; k < NP; ++k) cur[k] = 0;
                }
#pragma unroll
                for (int k = NP; k >= 1; --k)
                    cnt[k] = cnt[k - 1] + __popc(runs(prev[k - 1], k < NP ? cur[k] : 0u, s1, s2, s3, s4));
                top = max(top, cnt[NP]);
                cnt[0] = 0;
#pragma unroll
                for (int k = 0; k < NP; ++k) prev[k] = cur[k];
            }
        }
        top = __reduce_max_sync(0xffffffffu, top);
        if (lane == 0) best[p] = top;
        __syncwarp();   // the window's words are rewritten for the next pair
    }
}

// mx (zero before): the longest read and window, npairs less the first pair whose offsets decrease (0: none),
// and the ends of both arrays, so that one copy takes all to the host.
__global__ void k_pair_sizes(const u64 *__restrict__ roff, const u64 *__restrict__ woff, u32 npairs,
                             unsigned long long *__restrict__ mx) {
    u64 a = 0, b = 0;
    u32 first = npairs;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        mx[3] = roff[npairs];
        mx[4] = woff[npairs];
    }
    for (u32 p = blockIdx.x * blockDim.x + threadIdx.x; p < npairs; p += gridDim.x * blockDim.x) {
        const u64 r0 = roff[p], r1 = roff[p + 1], w0 = woff[p], w1 = woff[p + 1];
        if (r1 < r0 || w1 < w0) {
            first = min(first, p);
        } else {
            a = max(a, r1 - r0);
            b = max(b, w1 - w0);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
        b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
        first = min(first, __shfl_xor_sync(0xffffffffu, first, o));
    }
    if ((threadIdx.x & 31) == 0) {
        if (a) atomicMax(mx, (unsigned long long)a);
        if (b) atomicMax(mx + 1, (unsigned long long)b);
        if (first < npairs) atomicMax(mx + 2, (unsigned long long)(npairs - first));
    }
}

template <int NP>
int launch_words(const u8 *reads, const u64 *roff, const u8 *wins, const u64 *woff, u32 npairs, u32 q, u64 wmax, int sms,
                 int smem_max, u32 *best, cudaStream_t st) {
    const u32 words = (u32)((wmax + 31) / 32) + NP + 2;
    const size_t smem = 8 * 3 * (size_t)words * 4;
    const void *f = q == 7 ? (const void *)k_qmer_words<NP, true> : (const void *)k_qmer_words<NP, false>;
    // (always the device's maximum: the attribute is the kernel's, and another thread's call with smaller windows
    // must not lower it before this launch)
    if (smem > 48 * 1024) MB_CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, 256, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    u32 s[4] = {0, 0, 0, 0};   // run lengths 1, 1 + s0, ...: each step at most doubles
    for (u32 r = 1, i = 0; r < q; ++i) {
        s[i] = r < q - r ? r : q - r;
        r += s[i];
    }
    const unsigned blocks = (unsigned)std::min<u64>((u64)sms * per_sm, ((u64)npairs + 7) / 8);
    const uint4 step = make_uint4(s[0], s[1], s[2], s[3]);
    if (q == 7) k_qmer_words<NP, true><<<blocks, 256, smem, st>>>(reads, roff, wins, woff, npairs, q, step, words, best);
    else k_qmer_words<NP, false><<<blocks, 256, smem, st>>>(reads, roff, wins, woff, npairs, q, step, words, best);
    MB_KCHECK();
    return MB_OK;
}

}  // namespace

extern "C" int mb_rescue_prefilter(const uint8_t *reads, const uint64_t *read_off, const uint8_t *wins,
                                   const uint64_t *win_off, uint32_t n_pairs, uint32_t q, void *stream,
                                   uint32_t *best) {
    if (!read_off || !win_off || !best || (n_pairs && (!reads || !wins))) {
        mb_set_error("mb_rescue_prefilter: null argument");
        return MB_ERR_ARG;
    }
    if (q == 0) q = 7;
    if (q > 15) {
        mb_set_error("mb_rescue_prefilter: q = %u, at most 15", q);
        return MB_ERR_ARG;
    }
    if (n_pairs == 0) return MB_OK;
    cudaStream_t st = (cudaStream_t)stream;
    // the longest read and window, and the ends of both arrays: offsets in host memory are read there,
    // in device memory by a kernel (copying them out and looping over them took 1.3 ms for 1M pairs)
    u64 mmax = 0, wmax = 0, rend = 0, wend = 0;
    u32 bad = n_pairs;
    const bool rdev = mb_is_device_ptr(read_off), wdev = mb_is_device_ptr(win_off);
    DevBuf br, bw, bro, bwo, bb, bsz;
    const void *dr, *dw, *dro, *dwo;
    MB_TRY(mb_stage_in(read_off, ((size_t)n_pairs + 1) * 8, st, bro, &dro));
    MB_TRY(mb_stage_in(win_off, ((size_t)n_pairs + 1) * 8, st, bwo, &dwo));
    if (!rdev && !wdev) {
        MB_CK(cudaStreamSynchronize(st));   // what the stream still writes there: the staged copies have it
        for (u32 p = 0; p < n_pairs && bad == n_pairs; ++p) {
            if (read_off[p + 1] < read_off[p] || win_off[p + 1] < win_off[p]) bad = p;
            else {
                mmax = std::max<u64>(mmax, read_off[p + 1] - read_off[p]);
                wmax = std::max<u64>(wmax, win_off[p + 1] - win_off[p]);
            }
        }
        rend = read_off[n_pairs];
        wend = win_off[n_pairs];
    } else {
        MB_TRY(bsz.alloc(40, st));
        unsigned long long *mx = bsz.as<unsigned long long>();
        MB_CK(cudaMemsetAsync(mx, 0, 40, st));
        k_pair_sizes<<<grid_for(n_pairs, 256, 152 * 4), 256, 0, st>>>((const u64 *)dro, (const u64 *)dwo, n_pairs, mx);
        MB_KCHECK();
        u64 v[5];
        MB_CK(cudaMemcpyAsync(v, mx, sizeof v, cudaMemcpyDeviceToHost, st));
        MB_CK(cudaStreamSynchronize(st));
        mmax = v[0];
        wmax = v[1];
        bad = n_pairs - (u32)v[2];
        rend = v[3];
        wend = v[4];
    }
    if (bad < n_pairs) {
        mb_set_error("mb_rescue_prefilter: offsets decrease at pair %u", bad);
        return MB_ERR_ARG;
    }
    // mask words per warp: 4 bases x (P words + padded R words) of the longest read and window
    const u64 np = (mmax + 63) / 64, nr = (wmax + 63) / 64;
    const u64 slice = 4 * (np + 2 * np + nr + 1);
    const size_t per_warp = (size_t)slice * 8;
    int dev = 0, smem_max = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (per_warp > (size_t)smem_max) {
        mb_set_error("mb_rescue_prefilter: a read of %llu and a window of %llu bases need %zu bytes of "
                     "shared memory, more than %d",
                     (unsigned long long)mmax, (unsigned long long)wmax, per_warp, smem_max);
        return MB_ERR_ARG;
    }
    int warps = (int)std::min<size_t>(8, (size_t)smem_max / per_warp);
    const size_t smem = per_warp * warps;
    if (smem > 48 * 1024)
        MB_CK(cudaFuncSetAttribute(k_qmer_diag_max, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_qmer_diag_max, warps * 32, smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const u64 blocks = std::min<u64>((u64)sms * per_sm, ((u64)n_pairs + warps - 1) / warps);

    MB_TRY(mb_stage_in(reads, rend, st, br, &dr));
    MB_TRY(mb_stage_in(wins, wend, st, bw, &dw));
    u32 *db = best;
    const bool bdev = mb_is_device_ptr(best);
    if (!bdev) {
        MB_TRY(bb.alloc((size_t)n_pairs * 4, st));
        db = bb.as<u32>();
    }
    KTimer kt("rescue", st);
    kt.start();
    // up to eight read words of 32 bases in registers, and windows whose words fit the shared memory of a
    // block of eight warps; else the masks, which have room for any size accepted above
    const u32 words = (u32)((mmax + 31) / 32);
    if (words <= 8 && 8 * 3 * ((wmax + 31) / 32 + 10) * 4 <= (u64)smem_max) {
        const u8 *xr = (const u8 *)dr, *xw = (const u8 *)dw;
        const u64 *xo = (const u64 *)dro, *yo = (const u64 *)dwo;
        if (words <= 2) MB_TRY(launch_words<2>(xr, xo, xw, yo, n_pairs, q, wmax, sms, smem_max, db, st));
        else if (words == 3) MB_TRY(launch_words<3>(xr, xo, xw, yo, n_pairs, q, wmax, sms, smem_max, db, st));
        else if (words == 4) MB_TRY(launch_words<4>(xr, xo, xw, yo, n_pairs, q, wmax, sms, smem_max, db, st));
        else if (words == 5) MB_TRY(launch_words<5>(xr, xo, xw, yo, n_pairs, q, wmax, sms, smem_max, db, st));
        else MB_TRY(launch_words<8>(xr, xo, xw, yo, n_pairs, q, wmax, sms, smem_max, db, st));
    } else {
        k_qmer_diag_max<<<(unsigned)blocks, warps * 32, smem, st>>>((const u8 *)dr, (const u64 *)dro, (const u8 *)dw,
                                                                    (const u64 *)dwo, n_pairs, q, (u32)slice, db);
        MB_KCHECK();
    }
    kt.stop();
    if (!bdev) MB_CK(cudaMemcpyAsync(best, db, (size_t)n_pairs * 4, cudaMemcpyDeviceToHost, st));
    MB_CK(cudaStreamSynchronize(st));
    return MB_OK;
}
