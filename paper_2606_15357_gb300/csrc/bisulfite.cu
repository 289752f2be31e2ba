// Section 2.9 on the GPU: the strand rule of bisulfite hits (mb_bs_filter) and the T-to-C split of seed
// matches (mb_bs_split).
//
// A seed found on the 3-base index matches the converted read against the converted reference,
// so a read C over a reference T (read 1, C->T) or a read G over a reference A (read 2, G->A)
// matches there although the original bases differ.  Each kept hit of a seed is compared with the
// original reference under it and cut at every such position; the pieces of at least min_len bases
// are the output.
//
// A warp takes a tile of up to 256 hits, finds the tile's first record by one binary search and then reads
// the records 32 at a time, each hit finding its record among them in shared memory.  Only the read's C (or
// G) positions can cut, and conversion leaves few: they are marked once per record, and a hit reads the
// reference there only.  The pieces are counted per tile, the tiles' counts scanned, and the tiles
// written (a hit found uncut while counting reads no reference again).  14M hits: the two passes of the
// split 2.0 -> 1.2 ms against one thread per hit with a search over all records and a byte-by-byte
// comparison each.
#include "common.cuh"

namespace {

constexpr u32 TILE = 256;        // hits per tile at most
constexpr u32 MARKS = 8;         // words of cut marks per record: seeds of up to 256 bases
constexpr u32 NO_MARKS = 1u << 31;
enum { BS_FILTER = 0, BS_COUNT = 1, BS_WRITE = 2 };
enum { HIT_NONE = 0, HIT_WHOLE = 1, HIT_CUT = 2 };

struct BsArgs {
    const mb_smem *sm;
    u64 nsm;
    const u32 *hits;
    const u8 *keep;       // split: hits to split (null: all)
    u64 nh;
    const u8 *ref;
    u64 M;                // |R|; the text is CT(R) GA(R) rc(GA(R)) rc(CT(R)) $
    const u8 *seq;
    const u64 *off;
    const u8 *mate;
    u32 min_len;
    u32 per_tile;         // hits per tile
    u64 *tile;            // pieces of each tile, then of the tiles before it
    u8 *kind;             // per hit: no piece, one uncut piece, or pieces to find again when writing
    mb_piece *out;
    u64 cap;
    u8 *kept;             // filter: the result
};

struct BsRecords {        // the 32 records a warp looks at
    u32 end[32];          // hits of the tile before the end of record q
    u32 qbeg[32], len[32], read[32];
    u32 mate[32];         // 0, 1 or 2; bit 31: longer than the marks reach
    u32 mark[MARKS][32];  // bit t: the read's base t of the seed can cut
};

__device__ __forceinline__ u32 comp_code(u32 b) { return b < 4 ? 3u - b : 4u; }

// hit_off of record m, the first record's taken as 0 and the one past the last as nh: record m owns the
// hits from its offset to the next one's.
__device__ __forceinline__ u64 first_hit(const BsArgs &a, u64 m) {
    return m == 0 ? 0 : m < a.nsm ? __ldg(&a.sm[m].hit_off) : a.nh;
}

template <int MODE>
__global__ void __launch_bounds__(256) k_bs_tiles(BsArgs a) {
    __shared__ BsRecords shared[8];
    BsRecords &R = shared[threadIdx.x >> 5];
    const u32 FULL = 0xffffffffu, lane = threadIdx.x & 31;
    const u64 nt = (a.nh + a.per_tile - 1) / a.per_tile, nwarps = ((u64)gridDim.x * blockDim.x) >> 5;
    for (u64 tl = (blockIdx.x * (u64)blockDim.x + threadIdx.x) >> 5; tl < nt; tl += nwarps) {
        const u64 h0 = tl * a.per_tile, h1 = h0 + a.per_tile < a.nh ? h0 + a.per_tile : a.nh;
        u64 m0 = 0, hi = a.nsm;   // the last record that starts at or before h0
        while (hi - m0 > 1) {
            const u64 mid = (m0 + hi) >> 1;
            if (first_hit(a, mid) <= h0) m0 = mid;
            else hi = mid;
        }
        u64 at = MODE == BS_WRITE ? a.tile[tl] : 0;   // the next piece's place, or the pieces counted
        u32 done = 0;                                 // hits of the tile worked off
        const u32 all = (u32)(h1 - h0);
        for (; done < all && m0 < a.nsm; m0 += 32) {
            const u64 m = m0 + lane;
            const u64 e = m < a.nsm ? first_hit(a, m + 1) : a.nh;
            __syncwarp();
            R.end[lane] = e <= h0 ? 0u : (e - h0 < all ? (u32)(e - h0) : all);
            if (m < a.nsm) {
                const uint2 rq = *reinterpret_cast<const uint2 *>(&a.sm[m].read);   // read, qbeg
                const u32 len = a.sm[m].qend - rq.y, mt = a.mate ? a.mate[rq.x] : 0u;
                R.len[lane] = len;
                R.mate[lane] = mt;
                if (MODE != BS_FILTER) {
                    R.read[lane] = rq.x;
                    R.qbeg[lane] = rq.y;
                    const bool cuts = mt == 1 || mt == 2, fits = len <= 32 * MARKS;
                    if (cuts && !fits) R.mate[lane] = mt | NO_MARKS;
                    if (cuts && fits && e > h0 && first_hit(a, m) < h1) {   // a record of hits in this tile
                        const u8 *P = a.seq + a.off[rq.x] + rq.y;
                        for (u32 w = 0; 32 * w < len; ++w) {
                            u32 bits = 0;
                            const u32 k = len - 32 * w < 32 ? len - 32 * w : 32u;
                            for (u32 t = 0; t < k; ++t) bits |= (P[32 * w + t] == mt ? 1u : 0u) << t;   // C = 1 (read 1), G = 2 (read 2)
                            R.mark[w][lane] = bits;
                        }
                    }
                }
            }
            __syncwarp();
            const u32 upto = R.end[31];
            for (u32 t0 = done; t0 < upto; t0 += 32) {
                const u32 t = t0 + lane;
                const bool on = t < upto;
                u32 q = 0;
                if (on) {
#pragma unroll
                    for (u32 b = 16; b; b >>= 1)
                        if (R.end[q + b - 1] <= t) q += b;
                }
                const u64 h = h0 + t;
                const u32 pos = on ? a.hits[h] : 0u, L = R.len[q], M = (u32)a.M;
                // the copy holding pos, and whether the hit lies inside it
                const u32 g = M ? pos / M : 0u;
                const u32 x = pos - g * M;
                const bool whole = L ? (u64)x + L <= a.M : x != 0;
                const u32 mt = R.mate[q] & ~NO_MARKS;
                if (MODE == BS_FILTER) {
                    const bool ok = mt == 1 ? (g == 0 || g == 2) : mt == 2 ? (g == 1 || g == 3) : true;
                    if (on) a.kept[h] = whole && ok ? 1 : 0;
                    continue;
                }
                const bool use = on && (!a.keep || a.keep[h]) && L && g < 4 && whole;
                const u32 cut_ref = mt == 1 ? 3u : 0u;   // a read C over a reference T, a read G over a reference A
                // calls emit(b, e) for every piece [b, e) of the seed, in order
                auto pieces = [&](auto emit) {
                    u32 start = 0;
                    auto cut_at = [&](u32 p) {
                        const u32 r = g < 2 ? (u32)a.ref[x + p] : comp_code(a.ref[a.M - 1 - (x + p)]);
                        if (r != cut_ref) return;
                        if (p - start >= a.min_len) emit(start, p);
                        start = p + 1;
                    };
                    if (R.mate[q] & NO_MARKS) {
                        const u8 *P = a.seq + a.off[R.read[q]] + R.qbeg[q];
                        for (u32 p = 0; p < L; ++p)
                            if (P[p] == mt) cut_at(p);
                    } else if (mt == 1 || mt == 2) {
                        for (u32 w = 0; 32 * w < L; ++w)
                            for (u32 bits = R.mark[w][q]; bits; bits &= bits - 1) cut_at(32 * w + __ffs((int)bits) - 1);
                    }
                    if (L - start >= a.min_len) emit(start, L);
                };
                u32 cnt = 0;
                const u8 kind = MODE == BS_WRITE && on ? a.kind[h] : (u8)HIT_CUT;
                if (kind == HIT_WHOLE) {
                    cnt = 1;
                } else if (use && kind == HIT_CUT) {
                    bool uncut = true;
                    pieces([&](u32 b, u32 e2) {
                        ++cnt;
                        uncut = uncut && b == 0 && e2 == L;
                    });
                    if (MODE == BS_COUNT) a.kind[h] = cnt == 0 ? HIT_NONE : (cnt == 1 && uncut ? HIT_WHOLE : HIT_CUT);
                } else if (MODE == BS_COUNT && on) {
                    a.kind[h] = HIT_NONE;
                }
                u32 incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u32 v = __shfl_up_sync(FULL, incl, o);
                    if (lane >= (u32)o) incl += v;
                }
                if (MODE == BS_WRITE && cnt) {
                    u64 to = at + incl - cnt;
                    auto write = [&](u32 b, u32 e2) {
                        if (to < a.cap) a.out[to] = mb_piece{h, R.read[q], R.qbeg[q] + b, R.qbeg[q] + e2, pos + b};
                        ++to;
                    };
                    if (kind == HIT_WHOLE) write(0u, L);
                    else pieces(write);
                }
                at += __shfl_sync(FULL, incl, 31);
            }
            if (upto > done) done = upto;
        }
        if (MODE == BS_COUNT && lane == 0) a.tile[tl] = at;
    }
}

// Tiles of 256 hits, or as small as gives every SM's 32 warps one: with 256 always, the split of 18,000 hits
// took 0.230 ms against 0.148 for a thread per hit, now 0.093; 209,000 hits 0.246, 0.157 and 0.124; the
// same from 600,000 hits on.  (A quarter of the warps instead: 209,000 hits 0.232 ms.)
u32 tile_size(u64 hits) {
    u32 t = 32;
    while (t < TILE && hits > (u64)t * 152 * 32) t *= 2;
    return t;
}
unsigned tile_grid(u64 tiles) { return grid_for(tiles * 32, 256, 152u * 8u); }

}  // namespace

extern "C" int mb_bs_filter(const mb_index *idx, const mb_smem *smem, uint64_t n_smem, const uint8_t *mate,
                            const uint32_t *hits, uint64_t n_hits, void *stream, uint8_t *keep) {
    if (!idx || (n_hits && (!smem || !hits || !keep))) return MB_ERR_ARG;
    if (n_hits == 0) return MB_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DevBuf bsm, bmate, bhits, bkeep;
    const void *dsm = nullptr, *dmate = nullptr, *dhits = nullptr;
    MB_TRY(mb_stage_in(smem, n_smem * sizeof(mb_smem), st, bsm, &dsm));
    if (mate) {
        mb_smem last;
        MB_CK(cudaMemcpyAsync(&last, (const mb_smem *)dsm + n_smem - 1, sizeof last, cudaMemcpyDeviceToHost, st));
        MB_CK(cudaStreamSynchronize(st));
        MB_TRY(mb_stage_in(mate, (size_t)last.read + 1, st, bmate, &dmate));
    }
    MB_TRY(mb_stage_in(hits, n_hits * 4, st, bhits, &dhits));
    u8 *dk = keep;
    const bool kdev = mb_is_device_ptr(keep);
    if (!kdev) {
        MB_TRY(bkeep.alloc(n_hits, st));
        dk = bkeep.as<u8>();
    }
    u64 M = 0, n = 0, prim = 0;
    mb_index_info(idx, &n, &prim, &M);
    // the 3-base index holds four copies of |R| = M/2 bases
    u64 quarter = M / 2;
    const u32 per = tile_size(n_hits);
    const BsArgs a{(const mb_smem *)dsm, n_smem, (const u32 *)dhits, nullptr, n_hits, nullptr, quarter, nullptr, nullptr,
                   (const u8 *)dmate, 0, per, nullptr, nullptr, nullptr, 0, dk};
    k_bs_tiles<BS_FILTER><<<tile_grid((n_hits + per - 1) / per), 256, 0, st>>>(a);
    MB_KCHECK();
    if (!kdev) MB_CK(cudaMemcpyAsync(keep, dk, n_hits, cudaMemcpyDeviceToHost, st));
    MB_CK(cudaStreamSynchronize(st));
    return MB_OK;
}

extern "C" int mb_bs_split(const mb_index *idx, const uint8_t *ref, const uint8_t *seq, const uint64_t *off,
                           uint32_t n_reads, const uint8_t *mate, const mb_smem *smem, uint64_t n_smem,
                           const uint32_t *hits, const uint8_t *keep, uint64_t n_hits, const mb_opts *opts,
                           void *stream, mb_piece *out, uint64_t cap, uint64_t *n_out) {
    if (!idx || !n_out || (n_hits && (!ref || !seq || !off || !smem || !hits || !n_smem))) {
        mb_set_error("mb_bs_split: null argument");
        return MB_ERR_ARG;
    }
    *n_out = 0;
    if (!(mb_index_flags(idx) & MB_BS3)) {
        mb_set_error("mb_bs_split: the index is not a bisulfite (MB_BS3) index");
        return MB_ERR_ARG;
    }
    if (n_hits == 0) return MB_OK;
    cudaStream_t st = (cudaStream_t)stream;
    u64 n = 0, prim = 0, r3 = 0;
    MB_TRY(mb_index_info(idx, &n, &prim, &r3));
    const u64 M = r3 / 2;   // the index holds CT(R) GA(R): |R3| = 2 |R|
    const u32 min_len = opts && opts->min_len ? opts->min_len : 19;

    u64 o_last = 0;
    MB_CK(cudaMemcpyAsync(&o_last, off + n_reads, 8, cudaMemcpyDefault, st));
    MB_CK(cudaStreamSynchronize(st));
    DevBuf bref, bseq, boff, bmate, bsm, bhits, bkeep, bcnt, btmp, bout;
    const void *dref, *dseq, *doff, *dmate = nullptr, *dsm, *dhits, *dkeep = nullptr;
    MB_TRY(mb_stage_in(ref, M, st, bref, &dref));
    MB_TRY(mb_stage_in(seq, o_last, st, bseq, &dseq));
    MB_TRY(mb_stage_in(off, ((size_t)n_reads + 1) * 8, st, boff, &doff));
    if (mate) MB_TRY(mb_stage_in(mate, n_reads, st, bmate, &dmate));
    MB_TRY(mb_stage_in(smem, n_smem * sizeof(mb_smem), st, bsm, &dsm));
    MB_TRY(mb_stage_in(hits, n_hits * 4, st, bhits, &dhits));
    if (keep) MB_TRY(mb_stage_in(keep, n_hits, st, bkeep, &dkeep));
    const u32 per = tile_size(n_hits);
    const u64 tiles = (n_hits + per - 1) / per;
    MB_TRY(bcnt.alloc(tiles * 8 + 64 + n_hits, st));
    u64 *cnt = bcnt.as<u64>(), *dtotal = cnt + tiles;
    BsArgs a{(const mb_smem *)dsm, n_smem, (const u32 *)dhits, (const u8 *)dkeep, n_hits, (const u8 *)dref, M,
             (const u8 *)dseq, (const u64 *)doff, (const u8 *)dmate, min_len, per, cnt, (u8 *)(dtotal + 8), nullptr, 0, nullptr};
    k_bs_tiles<BS_COUNT><<<tile_grid(tiles), 256, 0, st>>>(a);
    MB_KCHECK();
    MB_TRY(btmp.alloc(scan_tmp_bytes(tiles), st));
    MB_TRY(scan_exclusive_u64(cnt, cnt, tiles, dtotal, btmp.p, st));
    u64 total = 0;
    MB_CK(cudaMemcpyAsync(&total, dtotal, 8, cudaMemcpyDeviceToHost, st));
    MB_CK(cudaStreamSynchronize(st));
    *n_out = total;
    if (total > cap) return MB_ERR_CAPACITY;
    if (total == 0) return MB_OK;
    if (!out) return MB_ERR_ARG;
    mb_piece *dout = out;
    const bool odev = mb_is_device_ptr(out);
    if (!odev) {
        MB_TRY(bout.alloc(total * sizeof(mb_piece), st));
        dout = bout.as<mb_piece>();
    }
    a.out = dout;
    a.cap = total;
    k_bs_tiles<BS_WRITE><<<tile_grid(tiles), 256, 0, st>>>(a);
    MB_KCHECK();
    if (!odev) MB_CK(cudaMemcpyAsync(out, dout, total * sizeof(mb_piece), cudaMemcpyDeviceToHost, st));
    MB_CK(cudaStreamSynchronize(st));
    return MB_OK;
}
