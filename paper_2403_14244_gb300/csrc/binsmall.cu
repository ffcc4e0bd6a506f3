// Binning of few Gaussians (rectangle footprints), in two or three launches instead
// of the fourteen of sort.cu's counting-sort route. Each of those is a chain of
// latencies on one or a few CTAs when there is little to sort (4,096 Gaussians on
// 256 x 256 pixels: 5 to 22 us a launch). Here no block waits on another, nothing is
// zeroed beforehand, and what is done twice is cheap:
//   k_small_rank   up to kRankMax Gaussians: the depth rank of each, by counting the
//                  keys before it;
//   k_small_sort, k_small_merge   more: chunks of 1024 sorted by one CTA each, then the
//                  rank of each Gaussian by a binary search in every other chunk, and per
//                  tile row a bitmap over the depth order of the rectangles that span it;
//   k_small_place  one CTA per strip of up to eight tiles of a tile row: the strip's tile
//                  ranges and, in depth order, the entries of its tiles, from the row's
//                  bitmap (up to kRankMax Gaussians: from all rectangles).
// 4,096 Gaussians on 256 x 256 pixels: 12 us against 41 for the general route; 16,384: 22 against
// 45. The entries per tile row, which give a strip its first slot, are summed by the merge: with
// the parts of every 256 Gaussians added up again by every strip, 32,768 Gaussians at 3840 x 2160
// took 150 us with 16-pixel tiles and 632 with 8-pixel tiles, now 119 and 396 (and the general
// route takes the latter: bin_small_ok).
// Writes what launch_bin_sort writes: order, ranges, vals and the status words (the
// same values: the stable depth order, rectangles row by row).
#include <mutex>

#include "binning.cuh"

namespace igs {
namespace {

constexpr int kRankThreads = 256;            // 8 warps, each comparing an eighth of every staged tile of keys
constexpr int kRankWarps = kRankThreads / 32;
constexpr uint32_t kRankTile = 4096;         // keys staged at a time
constexpr int64_t kRankMax = 4096;
constexpr uint32_t kChunk = 1024;            // Gaussians of a sorted chunk
constexpr int kMergeThreads = 256;           // Gaussians ranked by a block of the merge (of one chunk)
constexpr uint32_t kMergeStage = 8;          // chunks staged at a time
constexpr int kPlaceThreads = 512;
constexpr int kPlaceWarps = kPlaceThreads / 32;
constexpr uint32_t kStrip = 8;               // most tiles of a strip
// Positions of the depth order a thread takes per round of the placement: a word of the row's
// bitmap, or eight rectangles. (A round costs some 4,000 warp instructions whatever it finds:
// with a byte of the bitmap per thread, five rounds made 17 us of 20,000 Gaussians.)
constexpr uint32_t kEachBits = 32, kEachRects = 8;
constexpr uint32_t kListMax = 6144;          // items of a block's list (Gaussians in 26 bits)
static_assert(kBinSmallMax <= 65535ll * kPlaceThreads, "a thread's tile counters have 16 bits");
static_assert(kBinSmallMax <= 1 << 26, "a list item's Gaussian has 26 bits");
constexpr uint32_t kNoTiles = 1u << 16;      // rect.x of a Gaussian without tiles (rows 1..0; rect.y = 0)

// A block ranks 32 Gaussians, one per lane (n^2 comparisons: 7 us at 4,096, where the
// sort and the merge take 12; 65 us at 20,000, where they take 16): rank = the keys smaller than its own,
// or equal with a smaller index (the stable order). order[rank] = index and
// srect[rank] = its rectangle (culled Gaussians, whose keys are the largest: no tiles).
__global__ void __launch_bounds__(kRankThreads) k_small_rank(const uint32_t* __restrict__ key,
                                                             const uint2* __restrict__ rect,
                                                             const uint32_t* __restrict__ count, uint32_t n,
                                                             uint32_t* __restrict__ order,
                                                             uint2* __restrict__ srect) {
    pdl_wait();
    __shared__ uint4 s_k[kRankTile / 4];
    __shared__ uint32_t s_cnt[kRankWarps][32];
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t i0 = blockIdx.x * 32, i = i0 + lane;
    const uint32_t ki = i < n ? key[i] : 0xFFFFFFFFu;
    uint32_t before = 0;
    for (uint32_t base = 0; base < n; base += kRankTile) {
        if (base) __syncthreads();
        uint32_t* s = reinterpret_cast<uint32_t*>(s_k);
        // past the end: the largest key at an index above every i, before nothing
        for (uint32_t k = threadIdx.x; k < kRankTile; k += kRankThreads) s[k] = base + k < n ? key[base + k] : 0xFFFFFFFFu;
        __syncthreads();
        // the warp's keys in groups of 32; all of a group lie below the block's Gaussians, above them, or are them
        constexpr uint32_t kPer = kRankTile / kRankWarps;
        const uint32_t end = min(kPer, n > base + w * kPer ? n - (base + w * kPer) : 0u);
        for (uint32_t g = 0; g < end; g += 32) {
            const uint32_t j0 = base + w * kPer + g;
            const uint4* q = s_k + (w * kPer + g) / 4;
            if (j0 < i0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint4 v = q[k];
                    before += (v.x <= ki) + (v.y <= ki) + (v.z <= ki) + (v.w <= ki);
                }
            } else if (j0 > i0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint4 v = q[k];
                    before += (v.x < ki) + (v.y < ki) + (v.z < ki) + (v.w < ki);
                }
            } else {
                const uint32_t* e = reinterpret_cast<const uint32_t*>(q);
                for (uint32_t k = 0; k < 32; ++k) before += e[k] < ki || (e[k] == ki && k < lane);
            }
        }
    }
    s_cnt[w][lane] = before;
    __syncthreads();
    if (w != 0 || i >= n) return;
    uint32_t rank = 0;
#pragma unroll
    for (int k = 0; k < kRankWarps; ++k) rank += s_cnt[k][lane];
    order[rank] = i;
    srect[rank] = count[i] ? rect[i] : make_uint2(kNoTiles, 0u);
}

// Block c sorts Gaussians [1024 c, 1024 c + 1024) by (key, index): a bitonic network,
// one Gaussian per thread, exchanges within a warp by shuffles. skey holds whole chunks
// (past the end: the largest key). The row bitmaps and totals of the merge are zeroed on the way.
__global__ void __launch_bounds__(kChunk) k_small_sort(const uint32_t* __restrict__ key, uint32_t n,
                                                       uint32_t* __restrict__ skey, uint32_t* __restrict__ sid,
                                                       uint32_t* __restrict__ bits, uint32_t words) {
    pdl_wait();
    __shared__ u64 s_x[2][kChunk];
    const uint32_t t = threadIdx.x, i = blockIdx.x * kChunk + t;
    for (uint32_t c = i; c < words; c += gridDim.x * kChunk) bits[c] = 0u;
    u64 v = ((u64)(i < n ? key[i] : 0xFFFFFFFFu) << 32) | i;  // past the end: after every Gaussian
    int buf = 0;
#pragma unroll 1
    for (uint32_t k = 2; k <= kChunk; k <<= 1) {
#pragma unroll 1
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            u64 o;
            if (j >= 32) {
                s_x[buf][t] = v;
                __syncthreads();
                o = s_x[buf][t ^ j];
                buf ^= 1;  // (the next exchange writes the other buffer: one barrier each)
            } else {
                o = __shfl_xor_sync(0xffffffffu, v, j);
            }
            const bool low = ((t & j) == 0) == ((t & k) == 0);  // whether this thread keeps the smaller item
            if ((v < o) != low) v = o;
        }
    }
    skey[i] = (uint32_t)(v >> 32);
    if (i < n) sid[i] = (uint32_t)v;
}

// Rank of every Gaussian = its place in its chunk + in every other chunk the keys
// before its own: those not larger in the chunks of lower indices, the smaller ones
// in the others (ties in depth go by index). The chunks' keys are staged eight at a
// time, and a thread searches four at once; a warp's Gaussians are neighbours in their
// chunk's order, so its lanes search nearly the same places. Every kept rectangle then
// sets its rank's bit in the zeroed bitmap of each tile row it spans (row_words words
// a row), and the block adds the entries of its Gaussians per tile row to the zeroed
// row_total[rows] (below 2^32: at most kBinSmallMax rectangles of 2048 tiles a row).
__global__ void __launch_bounds__(kMergeThreads) k_small_merge(const uint32_t* __restrict__ skey,
                                                               const uint32_t* __restrict__ sid, uint32_t n,
                                                               const uint2* __restrict__ rect,
                                                               const uint32_t* __restrict__ count,
                                                               uint32_t* __restrict__ order,
                                                               uint2* __restrict__ srect, uint32_t* __restrict__ bits,
                                                               uint32_t row_words, uint32_t* __restrict__ row_total,
                                                               uint32_t rows) {
    pdl_wait();
    __shared__ uint32_t s_row[kBinSmallRows];
    __shared__ uint4 s_k4[kMergeStage][kChunk / 4];
    const uint32_t e = blockIdx.x * kMergeThreads + threadIdx.x;  // (below the padded length of skey)
    const uint32_t mine = blockIdx.x * kMergeThreads / kChunk, chunks = (n + kChunk - 1) / kChunk;
    const uint32_t k = skey[e];
    uint32_t rank = e % kChunk;
    for (uint32_t y = threadIdx.x; y < rows; y += kMergeThreads) s_row[y] = 0u;  // (barriers below)
    for (uint32_t c0 = 0; c0 < chunks; c0 += kMergeStage) {
        const uint32_t nc = min(kMergeStage, chunks - c0);
        if (c0) __syncthreads();
        for (uint32_t q = threadIdx.x; q < nc * (kChunk / 4); q += kMergeThreads)
            (&s_k4[0][0])[q] = reinterpret_cast<const uint4*>(skey + (size_t)c0 * kChunk)[q];
        __syncthreads();
        for (uint32_t q0 = 0; q0 < nc; q0 += 4) {
            uint32_t at[4] = {0u, 0u, 0u, 0u}, top[4];  // keys <= top are counted
#pragma unroll
            for (int q = 0; q < 4; ++q) top[q] = c0 + q0 + q < mine ? k : k - 1u;
#pragma unroll
            for (uint32_t step = kChunk; step > 0; step >>= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t* a = reinterpret_cast<const uint32_t*>(s_k4[q0 + q]);
                    if (at[q] + step <= kChunk && a[at[q] + step - 1] <= top[q]) at[q] += step;
                }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t c = c0 + q0 + q;
                const bool counts = q0 + q < nc && c != mine && !(c > mine && k == 0u);  // (no key is below 0)
                rank += counts ? at[q] : 0u;
            }
        }
    }
    if (e < n) {
        const uint32_t g = sid[e];
        order[rank] = g;
        const uint2 r = count[g] ? rect[g] : make_uint2(kNoTiles, 0u);
        srect[rank] = r;
        const uint32_t y0 = r.x >> 16, y1 = r.y >> 16, width = (r.y & 0xFFFFu) - (r.x & 0xFFFFu) + 1;
        for (uint32_t y = y0; y <= y1; ++y) {
            atomicOr(&bits[(size_t)y * row_words + (rank >> 5)], 1u << (rank & 31));
            atomicAdd(&s_row[y], width);
        }
    }
    __syncthreads();
    for (uint32_t y = threadIdx.x; y < rows; y += kMergeThreads)
        if (s_row[y]) atomicAdd(&row_total[y], s_row[y]);
}

__device__ __forceinline__ u64 block_sum64(u64 v, u64* s_part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    u64 t = 0;
#pragma unroll
    for (int k = 0; k < kPlaceWarps; ++k) t += s_part[k];
    return t;
}

// Status words of the frame, by one block: what the general route's kernels write.
__device__ __forceinline__ void small_status(const uint32_t* __restrict__ key, uint32_t n, u64 total,
                                             uint64_t capacity, u64* s_part, uint32_t* __restrict__ info) {
    bool wrap = false;
    uint32_t kept = 0;
    uint32_t any = 0u, all = 0xFFu;  // OR and AND of the top bytes of the keys that are not culled
    for (uint32_t i = threadIdx.x; i < n; i += kPlaceThreads) {
        const uint32_t k = key[i];
        if (k == 0xFFFFFFFFu) continue;
        ++kept;
        wrap |= (k & 0xFFFFFFu) == 0xFFFFFFu || (k >> 24) == 0xFFu;
        any |= k >> 24;
        all &= k >> 24;
    }
    const bool wraps = __syncthreads_or(wrap);
    any = __reduce_or_sync(0xffffffffu, any);
    all = __reduce_and_sync(0xffffffffu, all);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = any | ((u64)all << 32);
    __syncthreads();
    any = 0u;
    all = 0xFFu;
    for (int w = 0; w < kPlaceWarps; ++w) {
        any |= (uint32_t)s_part[w];
        all &= (uint32_t)(s_part[w] >> 32);
    }
    const uint32_t mixed = any & ~all;  // bits in which two top bytes differ
    const uint32_t kept_all = (uint32_t)block_sum64(kept, s_part);
    const uint32_t m32 = (uint32_t)min(total, (u64)0xFFFFFFFFu);
    if (threadIdx.x >= kInfoWords) return;
    uint32_t v = 0u;
    switch (threadIdx.x) {
        case kInfoM: case kInfoNeed: case kInfoTileTotal: v = m32; break;
        case kInfoKept: v = kept_all; break;
        case kInfoErr: v = total > capacity ? (uint32_t)IGS_ERR_CAPACITY : 0u; break;
        case kInfoAbort: v = total > capacity ? 1u : 0u; break;
        case kInfoKeyWrap: v = wraps ? 1u : 0u; break;
        case kInfoSkipTop: v = !wraps && mixed == 0u ? 1u : 0u; break;
        default: break;
    }
    info[threadIdx.x] = v;
}

// Block (y, s): tiles [s per, (s + 1) per) of tile row y (the strip, at most eight). The
// rectangles that meet the strip, in depth order, go into a list in shared memory: a round
// of positions of the depth order at a time, those that span the row first
// (from the row's bitmap (BITS) or from the rectangles themselves), then those of them
// that meet the strip. On the way the block counts the entries of each of its tiles, of
// the row's tiles before the strip, and of the rows before y (its first slot) and of the
// frame (the capacity check): from row_total[tiles_y], or again from the
// rectangles. Then every warp walks a part of the list and writes its tiles' entries.
// A strip met by more than kListMax rectangles is listed and placed again in shorter
// rounds. Block (tiles_y, 0) writes the status words.
template <bool BITS>
__global__ void __launch_bounds__(kPlaceThreads) k_small_place(
    const uint32_t* __restrict__ order, const uint2* __restrict__ srect, const uint32_t* __restrict__ key,
    const uint32_t* __restrict__ bits, uint32_t row_words, const uint32_t* __restrict__ row_total, uint32_t n,
    uint32_t tiles_x, uint32_t tiles_y, uint32_t per, uint64_t capacity, uint2* __restrict__ ranges,
    uint32_t* __restrict__ vals, uint32_t* __restrict__ tile_order, uint32_t* __restrict__ info) {
    pdl_wait();
    constexpr uint32_t kEach = BITS ? kEachBits : kEachRects;
    extern __shared__ uint32_t s_list[];   // [kListMax] Gaussian | first tile << 26 | last tile << 29
    uint32_t* s_raw = s_list + kListMax;   // [kEach kPlaceThreads] a round's positions that span the row, then items
    __shared__ uint32_t s_warp[2][kPlaceWarps];
    __shared__ u64 s_part[kPlaceWarps];
    __shared__ uint32_t s_cnt[kStrip], s_slot[kStrip], s_wcnt[kPlaceWarps][kStrip];
    constexpr uint32_t kMiss = 1u << 26;  // a span (1, 0): no tile of the strip
    const uint32_t y = blockIdx.x, xa = blockIdx.y * per, xb = min(tiles_x, xa + per), strip = xb - xa;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5, lt = (1u << lane) - 1u;
    if (y == tiles_y && xa > 0) return;
    if (threadIdx.x < kStrip) s_cnt[threadIdx.x] = 0u;
    u64 before = 0, total = 0;
    if constexpr (BITS) {
        for (uint32_t i = threadIdx.x; i < tiles_y; i += kPlaceThreads) {
            const uint32_t v = row_total[i];
            total += v;
            if (i < y) before += v;
        }
    } else {
        for (uint32_t p = threadIdx.x; p < n; p += kPlaceThreads) {
            const uint2 r = srect[p];
            const uint32_t y0 = r.x >> 16, y1 = r.y >> 16;
            if (y0 > y1) continue;
            const uint32_t width = (r.y & 0xFFFFu) - (r.x & 0xFFFFu) + 1, stop = min(y1 + 1, y);
            total += width * (y1 - y0 + 1);
            if (stop > y0) before += width * (stop - y0);
        }
    }
    if (y == tiles_y) {
        small_status(key, n, block_sum64(total, s_part), capacity, s_part, info);
        return;
    }
    // Exclusive prefix of a per-warp count over the block's warps, and their sum (one barrier;
    // `buf` alternates).
    auto warp_prefix = [&](uint32_t v, int buf, uint32_t& sum) -> uint32_t {
        if (lane == 31) s_warp[buf][w] = v;
        __syncthreads();
        uint32_t incl = lane < kPlaceWarps ? s_warp[buf][lane] : 0u;
#pragma unroll
        for (int o = 1; o < kPlaceWarps; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        sum = __shfl_sync(0xffffffffu, incl, kPlaceWarps - 1);
        const uint32_t before_me = __shfl_sync(0xffffffffu, incl, w == 0 ? 0 : w - 1);
        return w == 0 ? 0u : before_me;
    };
    // One round: appends the rectangles of positions [base, base + kEach threads) that meet the
    // strip to the list after `listed` items; returns the new length (items past the list's end
    // are counted, not written). With `counting`, counts their tiles and the row's tiles before the strip.
    u64 cnt03 = 0, cnt47 = 0;  // 16 bits per tile of the strip
    auto round = [&](uint32_t base, uint32_t threads, uint32_t listed, bool counting) -> uint32_t {
        const uint32_t p0 = base + kEach * threadIdx.x;
        uint32_t m = 0;  // this thread's positions that span the row
        if (p0 < n && threadIdx.x < threads) {
            if constexpr (BITS) {
                m = bits[(size_t)y * row_words + (p0 >> 5)];
            } else {
#pragma unroll
                for (uint32_t k = 0; k < kEach; k += 2) {  // (pairs: 16-byte loads, all in flight)
                    const uint4 r = p0 + k + 2 <= n ? *reinterpret_cast<const uint4*>(srect + p0 + k)
                                                    : make_uint4(p0 + k < n ? srect[p0 + k].x : kNoTiles,
                                                                 p0 + k < n ? srect[p0 + k].y : 0u, kNoTiles, 0u);
                    if ((r.x >> 16) <= y && y <= (r.y >> 16)) m |= 1u << k;
                    if ((r.z >> 16) <= y && y <= (r.w >> 16)) m |= 2u << k;
                }
            }
        }
        uint32_t incl = __popc(m);
        const uint32_t mine = incl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        uint32_t raw;
        uint32_t at = warp_prefix(incl, 0, raw) + incl - mine;
        for (; m; m &= m - 1) s_raw[at++] = p0 + __ffs(m) - 1;
        __syncthreads();
        // the warp's part of the round's positions: which meet the strip, and in which tiles
        const uint32_t part = ((raw + kPlaceWarps - 1) / kPlaceWarps + 31) & ~31u;
        const uint32_t i0 = min(raw, w * part), i1 = min(raw, i0 + part);
        uint32_t met = 0;
#pragma unroll 2
        for (uint32_t b = i0; b < i1; b += 32) {
            const uint32_t i = b + lane;
            bool in = false;
            if (i < i1) {
                const uint32_t p = s_raw[i];
                const uint2 r = srect[p];
                const uint32_t x0 = r.x & 0xFFFFu, x1 = r.y & 0xFFFFu;
                in = x0 < xb && x1 >= xa;
                const uint32_t a0 = max(x0, xa) - xa, b0 = min(x1, xb - 1) - xa;
                s_raw[i] = in ? order[p] | (a0 << 26) | (b0 << 29) : kMiss;
                if (counting) {
                    if (x0 < xa) before += min(x1 + 1, xa) - x0;
                    if (in) {
                        const uint32_t t = (2u << b0) - (1u << a0);  // bits a0 .. b0
                        cnt03 += ((t & 15u) * 0x0000200040008001ull) & 0x0001000100010001ull;  // bit k to 16 k
                        cnt47 += ((t >> 4) * 0x0000200040008001ull) & 0x0001000100010001ull;
                    }
                }
            }
            met += __popc(__ballot_sync(0xffffffffu, in));
        }
        uint32_t all;
        uint32_t to = listed + warp_prefix(met, 1, all);
#pragma unroll 2
        for (uint32_t b = i0; b < i1; b += 32) {
            const uint32_t it = b + lane < i1 ? s_raw[b + lane] : kMiss;
            const bool in = ((it >> 26) & 7u) <= (it >> 29);
            const uint32_t hit = __ballot_sync(0xffffffffu, in);
            const uint32_t d = to + __popc(hit & lt);
            if (in && d < kListMax) s_list[d] = it;
            to += __popc(hit);
        }
        return listed + all;
    };
    uint32_t listed = 0;
    for (uint32_t base = 0; base < n; base += kEach * kPlaceThreads) {
        if (base) __syncthreads();  // the last round's positions are no longer read
        listed = round(base, kPlaceThreads, listed, true);
    }
    const u64 total_all = block_sum64(total, s_part);
    const u64 before_all = block_sum64(before, s_part);
#pragma unroll
    for (uint32_t t = 0; t < kStrip; ++t) {
        if (t >= strip) break;
        const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)((t < 4 ? cnt03 : cnt47) >> (16 * (t & 3))) & 0xFFFFu);
        if (lane == 0 && c) atomicAdd(&s_cnt[t], c);
    }
    __syncthreads();
    if (threadIdx.x < strip) {
        uint32_t s = (uint32_t)before_all;
        for (uint32_t t = 0; t < threadIdx.x; ++t) s += s_cnt[t];
        const uint32_t c = s_cnt[threadIdx.x], tile = y * tiles_x + xa + threadIdx.x;
        s_slot[threadIdx.x] = s;
        ranges[tile] = c ? make_uint2(s, s + c) : make_uint2(0u, 0u);
        if (tile_order) tile_order[tile] = tile;  // as they come
    }
    if (total_all > capacity || listed == 0) return;  // (uniform over the block)
    // the list of m items, from every tile's next slot on: a warp counts its part's entries per tile, takes
    // its slots after the earlier warps' and writes
    auto place = [&](uint32_t m) {
        const uint32_t part = ((m + kPlaceWarps - 1) / kPlaceWarps + 31) & ~31u;
        const uint32_t i0 = min(m, w * part), i1 = min(m, i0 + part);
        uint32_t c = 0;  // lane t: the part's entries in tile t
        for (uint32_t b = i0; b < i1; b += 32) {
            const uint32_t it = b + lane < i1 ? s_list[b + lane] : kMiss;
            const uint32_t lo = (it >> 26) & 7u, hi = it >> 29;
            for (uint32_t t = 0; t < strip; ++t) {
                const uint32_t hit = __ballot_sync(0xffffffffu, lo <= t && t <= hi);
                if (lane == t) c += __popc(hit);
            }
        }
        if (lane < kStrip) s_wcnt[w][lane] = c;
        __syncthreads();
        uint32_t slot = 0;  // lane t: the warp's next slot in tile t
        if (lane < strip) {
            slot = s_slot[lane];
            for (uint32_t v = 0; v < w; ++v) slot += s_wcnt[v][lane];
        }
        for (uint32_t b = i0; b < i1; b += 32) {
            const uint32_t it = b + lane < i1 ? s_list[b + lane] : kMiss;
            const uint32_t lo = (it >> 26) & 7u, hi = it >> 29;
            for (uint32_t t = 0; t < strip; ++t) {
                const bool in = lo <= t && t <= hi;
                const uint32_t hit = __ballot_sync(0xffffffffu, in);
                const uint32_t first = __shfl_sync(0xffffffffu, slot, t);
                if (in) vals[first + __popc(hit & lt)] = it & 0x3FFFFFFu;
                if (lane == t) slot += __popc(hit);
            }
        }
        return slot;
    };
    __syncthreads();  // the list and the slots are written
    if (listed <= kListMax) {
        place(listed);
        return;
    }
    constexpr uint32_t kShort = kListMax / kEach;  // threads whose positions fit the list
    for (uint32_t base = 0; base < n; base += kEach * kShort) {
        const uint32_t m = round(base, kShort, 0u, false);
        __syncthreads();  // the list is complete
        const uint32_t slot = place(m);
        __syncthreads();  // every warp has read the list and its tile's slot
        if (w == kPlaceWarps - 1 && lane < strip) s_slot[lane] = slot;  // (the last warp's next slots are the block's)
        __syncthreads();
    }
}

}  // namespace

// Lets the placement use its largest shared memory, once per device; never lowers it.
static cudaError_t place_opt_in(int bytes) {
    static std::mutex mu;
    static bool done[128] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 128) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(k_small_place<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

bool bin_small_ok(const igs_frame& f, int footprint) {
    return footprint == 0 && f.n > 0 && f.n <= kBinSmallMax && f.sort_chunks > 0 && f.tiles_y <= kBinSmallRows &&
           f.n * f.tiles_x * f.tiles_y <= kBinSmallCells;
}

cudaError_t launch_bin_small(const igs_frame& f, const SortScratch& s, cudaStream_t st) {
    cudaError_t e;
#define CK(x) do { if ((e = (x)) != cudaSuccess) { g_failed_call = #x " (binsmall.cu:" IGS_STR(__LINE__) ")"; return e; } } while (0)
    const uint32_t n = (uint32_t)f.n, tx = (uint32_t)f.tiles_x, ty = (uint32_t)f.tiles_y;
    const uint2* rect = reinterpret_cast<const uint2*>(f.rect);
    uint2* srect = s.walk_rect;
    // skey: the 8 n bytes of ditems_a hold n rounded up to 1024 words above kRankMax Gaussians
    uint32_t *skey = reinterpret_cast<uint32_t*>(s.ditems_a), *sid = reinterpret_cast<uint32_t*>(s.ditems_b);
    // the row bitmaps and, after them, the rows' totals: 4 (n / 32 + 2) bytes per tile row of the 4 walk_chunks
    // bytes per row of walk_h1 (at least 32 KB up to kBinSmallRows rows)
    const uint32_t row_words = (uint32_t)ceil_div(f.n, 32);
    uint32_t *bits = s.walk_h1, *row_total = s.walk_h1 + (size_t)row_words * ty;
    const bool rank = f.n <= kRankMax;
    if (rank) {
        CK(launch_pdl(k_small_rank, dim3((unsigned)ceil_div(f.n, 32)), dim3(kRankThreads), 0, st, f.depth_key, rect,
                      f.count, n, f.order, srect));
    } else {
        if ((int64_t)row_words + 1 > s.walk_chunks) return cudaErrorInvalidValue;  // (never: bin_small_ok)
        CK(launch_pdl(k_small_sort, dim3((unsigned)ceil_div(f.n, kChunk)), dim3(kChunk), 0, st, f.depth_key, n, skey,
                      sid, bits, (row_words + 1) * ty));
        count_launches();
        CK(cudaGetLastError());
        CK(launch_pdl(k_small_merge, dim3((unsigned)ceil_div(f.n, kMergeThreads)), dim3(kMergeThreads), 0, st, skey, sid,
                      n, rect, f.count, f.order, srect, bits, row_words, row_total, ty));
    }
    count_launches();
    CK(cudaGetLastError());
    // strips of eight tiles, narrower where they would leave SMs without a block
    uint32_t per = kStrip;
    while (per > 2 && (int64_t)ty * ceil_div(f.tiles_x, per) < 152) per /= 2;
    const size_t smem = (size_t)(kListMax + (rank ? kEachRects : kEachBits) * kPlaceThreads) * 4;
    if (smem > 40 * 1024) CK(place_opt_in((int)smem));
    CK(launch_pdl(rank ? k_small_place<false> : k_small_place<true>, dim3(ty + 1, (unsigned)ceil_div(f.tiles_x, per)),
                  dim3(kPlaceThreads), smem, st, f.order, srect, f.depth_key, bits, row_words, row_total, n, tx, ty, per,
                  (uint64_t)f.capacity,
                  reinterpret_cast<uint2*>(f.ranges), f.vals, s.tile_order, f.info));
    count_launches();
    CK(cudaGetLastError());
#undef CK
    return cudaSuccess;
}

}  // namespace igs
