// Front-to-back compositing (Eq. 4), shared by the one-view forward kernel
// (blend.cu) and the multi-view kernels (batch.cu), so all produce bit-identical
// pixels. Internal to libigs.
#pragma once

#include "common.cuh"

namespace igs {
namespace {

// A record's first float4 is (u, v, w2, pmax), its second (r, g, b, o); the
// exponent of a pixel is w2 d^2 and pmax = log2(o / alpha_min) + margin bounds
// it: a larger exponent gives alpha < alpha_min.
struct Dist {
    float dx, dy, d2, pw;
};

// Squared distance and exponent of one (pixel, entry) pair, each step rounded
// once in a fixed order, so that forward and backward take the same decisions.
__device__ __forceinline__ Dist eval_dist(float px, float py, float4 a) {
    Dist r;
    r.dx = __fsub_rn(px, a.x);
    r.dy = __fsub_rn(py, a.y);
    r.d2 = __fmaf_rn(r.dx, r.dx, __fmul_rn(r.dy, r.dy));
    r.pw = __fmul_rn(a.z, r.d2);
    return r;
}

// Whether the entry can reach a pixel centre in [xlo, xhi] x [ylo, yhi] (first
// and last centres of a block of rows): the exponent test at the centre nearest
// to (u, v). Each rounded step of eval_dist is monotone in |dx| and |dy|, so that
// centre has the smallest exponent of the block and a false answer never drops
// a pair that the per-pixel test would keep.
__device__ __forceinline__ bool may_reach(float4 a, float xlo, float xhi, float ylo, float yhi) {
    const float cx = fminf(fmaxf(floorf(a.x) + 0.5f, xlo), xhi);
    const float cy = fminf(fmaxf(floorf(a.y) + 0.5f, ylo), yhi);
    return !(eval_dist(cx, cy, a).pw > a.w);
}

// One CTA of TS*TS threads composites one tile (one thread per pixel), staging
// B entries at a time in shared memory (s_a, s_c hold B float4 each), and leaves
// the batch loop once every pixel has stopped. Each warp owns an 8 x 4 block of
// the tile (compact blocks are reached by fewer entries than whole rows, and
// their pixels stop at similar depths) and walks, in order, only the staged
// entries that may reach it (one ballot per 32 entries). Writes img (planar,
// `plane` floats per channel, row stride `width`). The batch path's persistent
// blend; pixels are bit for bit those of blend_block_fwd.
template <int TS, int B>
__device__ __forceinline__ void blend_tile_fwd(int tx, int ty, int width, int height, uint2 rg,
                                               const uint32_t* __restrict__ vals, const float4* __restrict__ rec,
                                               float alpha_min, float alpha_max, float t_min, const float* bg,
                                               float4* s_a, float4* s_c, float* __restrict__ img) {
    constexpr int NT = TS * TS;
    constexpr int BPR = TS / 8;  // 8 x 4 warp blocks per block row of the tile
    static_assert(B <= NT, "staging batch larger than the tile");
    static_assert(TS >= 8 && TS <= 32, "the tile holds whole 8 x 4 warp blocks");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int bx = tx * TS + (w % BPR) * 8, by = ty * TS + (w / BPR) * 4;  // the warp's block
    const int x = bx + (lane & 7), y = by + (lane >> 3);
    const bool inside = x < width && y < height;
    const float px = (float)x + 0.5f, py = (float)y + 0.5f;
    // pixel centres of this warp's block
    const float bx0 = (float)bx + 0.5f, bx1 = bx0 + 7.f;
    const float by0 = (float)by + 0.5f, by1 = by0 + 3.f;
    float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
    bool done = !inside;
    // Software-pipelined staging: thread t < B stages entry b0 + t of every
    // batch, its ids fetched two batches ahead and its records one batch ahead,
    // so that a long walk does not wait out two dependent gathers per batch.
    const bool stager = threadIdx.x < B;
    uint32_t g_nxt = 0;
    float4 a_cur = make_float4(0.f, 0.f, 0.f, 0.f), c_cur = a_cur;
    if (stager) {
        const uint32_t j0 = rg.x + threadIdx.x, j1 = j0 + B;
        if (j0 < rg.y) {
            const uint32_t g = vals[j0];
            a_cur = rec[2 * g];
            c_cur = rec[2 * g + 1];
        }
        if (j1 < rg.y) g_nxt = vals[j1];
    }
    for (uint32_t b0 = rg.x; b0 < rg.y; b0 += B) {
        if (__syncthreads_count(done) == NT) break;
        if (stager) {
            const uint32_t j = b0 + threadIdx.x;
            if (j < rg.y) {
                s_a[threadIdx.x] = a_cur;
                s_c[threadIdx.x] = c_cur;
            }
            if (j + B < rg.y) {  // the next batch's record, then the id of the one after it
                a_cur = rec[2 * g_nxt];
                c_cur = rec[2 * g_nxt + 1];
            }
            if (j + 2 * B < rg.y) g_nxt = vals[j + 2 * B];
        }
        __syncthreads();
        const int nb = (int)min((uint32_t)B, rg.y - b0);
        for (int c0 = 0; c0 < nb; c0 += 32) {
            if (__all_sync(0xffffffffu, done)) break;
            const bool reach = c0 + lane < nb && may_reach(s_a[c0 + lane], bx0, bx1, by0, by1);
            uint32_t bits = __ballot_sync(0xffffffffu, reach);
            while (bits && !done) {
                const int k = c0 + __ffs(bits) - 1;
                bits &= bits - 1;
                const float4 a = s_a[k];
                const float pw = eval_dist(px, py, a).pw;
                if (pw > a.w) continue;
                const float4 c = s_c[k];
                const float alpha = fminf(alpha_max, __fmul_rn(c.w, fast_exp2(-pw)));
                if (alpha < alpha_min) continue;
                const float Tn = T * (1.f - alpha);
                if (Tn < t_min) {
                    done = true;
                    break;
                }
                const float w = alpha * T;
                C0 = fmaf(c.x, w, C0);
                C1 = fmaf(c.y, w, C1);
                C2 = fmaf(c.z, w, C2);
                T = Tn;
            }
        }
    }
    if (!inside) return;
    const size_t pix = (size_t)y * width + x, plane = (size_t)width * height;
    img[pix] = fmaf(T, bg[0], C0);
    img[plane + pix] = fmaf(T, bg[1], C1);
    img[2 * plane + pix] = fmaf(T, bg[2], C2);
}

// ---- one warp per 8 x 8 pixel block ----
//
// The blend is bound by instruction issue, so the walk is laid out to need few
// instructions per (pixel, entry) pair: a lane holds two pixels of one column
// (rows r and r + 4), whose distances, exponents and transmittances go through
// packed two-lane FP32 steps (each lane rounded as its scalar _rn counterpart);
// the entries that reach the block are compacted into a queue in shared memory,
// operands duplicated as the packed steps want them, and walked without
// branches. A pixel that has stopped carries an alpha threshold of infinity.
// Against one thread per pixel, two warps per block and a branch per rule:
// 202 -> 141 us for a 1080p view of 1M clustered Gaussians, 237 -> 191 us for
// the 3M training views (32-pixel tiles), 32 mixed views of 2M in one chain
// 11.1 -> 9.4 ms. The first issues 3.4 of 4 instructions a clock while it runs. A training
// view of 1.5M issues in 74 % of the slots while a scheduler has a warp, waiting most
// on other warps and on the FP32 pipes, and in 64 % of all slots of the launch: the
// rest is its drain, long walks of few warps; L2 is at 10 % of its rate. One warp
// per CTA: a block's slot is free as soon as its own walk ends (two warps per
// CTA: 376 against 366 us for the whole 1080p frame).
struct __align__(16) FwdEntry {
    float4 p;  // (-u, -u, -v, -v)
    float4 q;  // (-w2, -w2, -pmax, list position + 1 as bits)
    float4 c;  // (r, g, b, o): the colour record as it is
};
constexpr uint32_t kQueue = 64;  // entries of a block's queue (a ring)

// A warp's entries on their way: batches of 32 list positions, one entry per
// lane. A batch's ids are requested kIdAhead batches before its records, and
// those kRecAhead batches before the batch is tested, all by asynchronous
// copies whose slots only the lane itself reads: a walk that mostly misses its
// block takes some 250 cycles a batch, and both loads may come from HBM. (With
// one batch between an id and its record, the sparse walks of the 3M training
// views, up to 7,000 positions, waited out a memory latency per batch.)
constexpr uint32_t kRecAhead = 3, kIdAhead = 4, kIdSlots = 8;
static_assert(kRecAhead + kIdAhead < kIdSlots && (kIdSlots & (kIdSlots - 1)) == 0, "ids live until their batch is tested");
struct Stager {
    float4 rec[kRecAhead][2][32];
    uint32_t id[kIdSlots][32];
};
// Position(j): address of the id of the walk's j-th entry; j < total.
template <typename IdOf>
__device__ __forceinline__ void stage_ids(Stager& S, uint32_t batch, uint32_t total, uint32_t lane, IdOf id_of) {
    const uint32_t j = batch * 32 + lane;
    if (j < total) cp_async4(&S.id[batch & (kIdSlots - 1)][lane], id_of(j));
}
__device__ __forceinline__ void stage_records(Stager& S, uint32_t batch, uint32_t slot, uint32_t total, uint32_t lane,
                                              const float4* __restrict__ rec) {
    if (batch * 32 + lane >= total) return;
    const float4* r = rec + 2 * (size_t)S.id[batch & (kIdSlots - 1)][lane];
    cp_async16(&S.rec[slot][0][lane], r);
    cp_async16(&S.rec[slot][1][lane], r + 1);
}
// The copies of the first batches; one commit group per batch from here on.
template <typename IdOf>
__device__ __forceinline__ void stage_begin(Stager& S, uint32_t total, uint32_t lane, const float4* __restrict__ rec,
                                            IdOf id_of) {
#pragma unroll
    for (uint32_t b = 0; b < kRecAhead; ++b) stage_ids(S, b, total, lane, id_of);
    cp_async_commit();
#pragma unroll
    for (uint32_t b = kRecAhead; b < kRecAhead + kIdAhead; ++b) stage_ids(S, b, total, lane, id_of);
    cp_async_commit();
    cp_async_wait<1>();
#pragma unroll
    for (uint32_t b = 0; b < kRecAhead; ++b) {
        stage_records(S, b, b, total, lane, rec);
        cp_async_commit();
    }
}

struct FwdQueue {
    FwdEntry e[kQueue];
    Stager st;
};
// Resident one-warp CTAs per SM asked of the compiler (72 registers a thread; 27 and 28 take the same
// time), as many as an SM's 228 KB of shared memory holds, 1 KB of it the system's for each.
constexpr int kFwdMinCtas = 28;
static_assert(kFwdMinCtas * (sizeof(FwdQueue) + 1024) <= 228 * 1024, "resident CTAs per SM");

__device__ __forceinline__ float2 pk_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 pk_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 pk_add(float2 a, float2 b) { return __fadd2_rn(a, b); }

// The warp's two pixels per lane and what they have composited.
struct FwdPixels {
    float2 px, py;     // centres: px the same twice
    float2 T;
    float2 thr;        // alpha threshold: alpha_min, or infinity once stopped
    float C[2][3];
    float D[2][3];     // colour composited since the last cut (walk segments, after the first cut)
    uint32_t last[2];  // last blended list position + 1
};

// One pixel of a pair: blend the entry with the given alpha, T (1 - alpha) and
// alpha T, by the comparisons of Eq. 4's rules in their order (skip, stop, blend),
// as predicated instructions: nothing is added where the entry is not blended.
// SUM: the entry's colour is added to D too.
template <bool SUM>
__device__ __forceinline__ void fwd_blend_one(float npw, float npmax, float alpha, float Tn, float w, const float4& c,
                                              uint32_t pos1, float t_min, float& T, float& thr, float (&C)[3],
                                              float (&D)[3], uint32_t& last) {
    if constexpr (SUM)
        asm("{\n\t"
            ".reg .pred near, in, stop, go;\n\t"
            "setp.geu.f32 near, %9, %10;\n\t"             // !(w2 d^2 > pmax)
            "setp.ge.and.f32 in, %11, %1, near;\n\t"      // alpha >= threshold
            "setp.lt.and.f32 stop|go, %12, %18, in;\n\t"  // T (1 - alpha) < t_min, or blended
            "@stop mov.f32 %1, 0f7F800000;\n\t"
            "@go fma.rn.f32 %2, %14, %13, %2;\n\t"
            "@go fma.rn.f32 %3, %15, %13, %3;\n\t"
            "@go fma.rn.f32 %4, %16, %13, %4;\n\t"
            "@go fma.rn.f32 %6, %14, %13, %6;\n\t"
            "@go fma.rn.f32 %7, %15, %13, %7;\n\t"
            "@go fma.rn.f32 %8, %16, %13, %8;\n\t"
            "@go mov.f32 %0, %12;\n\t"
            "@go mov.u32 %5, %17;\n\t"
            "}"
            : "+f"(T), "+f"(thr), "+f"(C[0]), "+f"(C[1]), "+f"(C[2]), "+r"(last), "+f"(D[0]), "+f"(D[1]), "+f"(D[2])
            : "f"(npw), "f"(npmax), "f"(alpha), "f"(Tn), "f"(w), "f"(c.x), "f"(c.y), "f"(c.z), "r"(pos1), "f"(t_min));
    else
        asm("{\n\t"
            ".reg .pred near, in, stop, go;\n\t"
            "setp.geu.f32 near, %6, %7;\n\t"
            "setp.ge.and.f32 in, %8, %1, near;\n\t"
            "setp.lt.and.f32 stop|go, %9, %15, in;\n\t"
            "@stop mov.f32 %1, 0f7F800000;\n\t"
            "@go fma.rn.f32 %2, %11, %10, %2;\n\t"
            "@go fma.rn.f32 %3, %12, %10, %3;\n\t"
            "@go fma.rn.f32 %4, %13, %10, %4;\n\t"
            "@go mov.f32 %0, %9;\n\t"
            "@go mov.u32 %5, %14;\n\t"
            "}"
            : "+f"(T), "+f"(thr), "+f"(C[0]), "+f"(C[1]), "+f"(C[2]), "+r"(last)
            : "f"(npw), "f"(npmax), "f"(alpha), "f"(Tn), "f"(w), "f"(c.x), "f"(c.y), "f"(c.z), "r"(pos1), "f"(t_min));
}

// Walk U queued entries from e on: their alphas first (independent of one
// another), then the pixels' transmittances entry by entry.
template <int U, bool SUM>
__device__ __forceinline__ void fwd_walk_some(const FwdEntry* e, float alpha_max, float t_min, FwdPixels& s) {
    float2 npw[U], alpha[U], oma[U];
    float4 c[U];
    float npmax[U];
    uint32_t pos1[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
        const float4 p = e[k].p, q = e[k].q;
        c[k] = e[k].c;
        npmax[k] = q.z;
        pos1[k] = __float_as_uint(q.w);
        const float2 dx = pk_add(s.px, make_float2(p.x, p.y));
        const float2 dy = pk_add(s.py, make_float2(p.z, p.w));
        npw[k] = pk_mul(make_float2(q.x, q.y), pk_fma(dx, dx, pk_mul(dy, dy)));
        alpha[k] = make_float2(fminf(alpha_max, __fmul_rn(c[k].w, fast_exp2(npw[k].x))),
                               fminf(alpha_max, __fmul_rn(c[k].w, fast_exp2(npw[k].y))));
        oma[k] = pk_fma(alpha[k], make_float2(-1.f, -1.f), make_float2(1.f, 1.f));
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
        const float2 Tn = pk_mul(s.T, oma[k]), w = pk_mul(alpha[k], s.T);
        fwd_blend_one<SUM>(npw[k].x, npmax[k], alpha[k].x, Tn.x, w.x, c[k], pos1[k], t_min, s.T.x, s.thr.x, s.C[0],
                           s.D[0], s.last[0]);
        fwd_blend_one<SUM>(npw[k].y, npmax[k], alpha[k].y, Tn.y, w.y, c[k], pos1[k], t_min, s.T.y, s.thr.y, s.C[1],
                           s.D[1], s.last[1]);
    }
}

// Walk cnt queued entries from e on (no wrap within them). Four entries' alphas are
// independent work between two steps of the transmittance chain, which is what a
// long walk waits for once few warps are left (two and eight measured alike, within 1 %).
constexpr int kFwdUnroll = 4;
template <bool SUM>
__device__ __forceinline__ void fwd_walk(const FwdEntry* e, int cnt, float alpha_max, float t_min, FwdPixels& s) {
    int k = 0;
#pragma unroll 1
    for (; k + kFwdUnroll <= cnt; k += kFwdUnroll) fwd_walk_some<kFwdUnroll, SUM>(e + k, alpha_max, t_min, s);
#pragma unroll 1
    for (; k < cnt; ++k) fwd_walk_some<1, SUM>(e + k, alpha_max, t_min, s);
}

// One warp composites the 8 x 8 block at pixel (bx, by), walking the tile's
// entries rg in batches of 32, one entry per lane (Stager). The entries that
// reach the block are queued, and walked in multiples of kFwdUnroll once 32 are
// queued. SEG: the walk is cut into segments for the backward (SegLayout),
// `block` naming this block. Writes what blend_tile_fwd writes.
template <bool SEG>
__device__ __forceinline__ void blend_block_fwd(int bx, int by, int width, int height, uint2 rg,
                                                const uint32_t* __restrict__ vals, const float4* __restrict__ rec,
                                                float alpha_min, float alpha_max, float t_min, const float* bg,
                                                FwdQueue& Q, float* __restrict__ img, float* __restrict__ T_final,
                                                uint32_t* __restrict__ n_contrib, const SegLayout seg = SegLayout{},
                                                uint32_t block = 0) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t n = rg.y > rg.x ? rg.y - rg.x : 0u;
    vals += rg.x;
    const auto id_of = [vals](uint32_t j) { return vals + j; };
    stage_begin(Q.st, n, lane, rec, id_of);
    const int x = bx + (int)(lane & 7), y0 = by + (int)(lane >> 3), y1 = y0 + 4;
    const float inf = __int_as_float(0x7f800000);
    FwdPixels s;
    s.px = make_float2((float)x + 0.5f, (float)x + 0.5f);
    s.py = make_float2((float)y0 + 0.5f, (float)y1 + 0.5f);
    s.T = make_float2(1.f, 1.f);
    s.thr = make_float2(x < width && y0 < height ? alpha_min : inf, x < width && y1 < height ? alpha_min : inf);
#pragma unroll
    for (int i = 0; i < 2; ++i) s.C[i][0] = s.C[i][1] = s.C[i][2] = s.D[i][0] = s.D[i][1] = s.D[i][2] = 0.f;
    s.last[0] = s.last[1] = 0;
    // segment state (warp-uniform): where the open segment starts, the segments closed, the last one's slot,
    // and the list positions between cuts
    uint32_t seg_lo = 0, seg_n = 0, seg_last = kSegNone;
    uint32_t stride = seg.stride;
    bool seg_stop = false;
    uint32_t reserved = kSegNone;  // lane 0: the pool slot taken for the next close (its atomic is in flight meanwhile)
    const bool segs = SEG && seg.slots != 0;
    uint32_t head = 0, queued = 0;  // the ring's first entry (a multiple of kFwdUnroll) and entries (warp-uniform)
    uint32_t slot = 0;              // the records' slot of the current batch
    auto walk = [&](uint32_t cnt) {  // the first cnt queued entries; whether every pixel has stopped
        __syncwarp();
        const uint32_t first = min(cnt, kQueue - head);
        if (SEG && seg_n > 0) {  // past the first cut: the open segment's own colour too
            fwd_walk<true>(Q.e + head, (int)first, alpha_max, t_min, s);
            if (first < cnt) fwd_walk<true>(Q.e, (int)(cnt - first), alpha_max, t_min, s);
        } else {
            fwd_walk<false>(Q.e + head, (int)first, alpha_max, t_min, s);
            if (first < cnt) fwd_walk<false>(Q.e, (int)(cnt - first), alpha_max, t_min, s);
        }
        queued -= cnt;
        head = queued ? (head + cnt) & (kQueue - 1) : 0u;
        return __all_sync(0xffffffffu, s.thr.x == inf && s.thr.y == inf);  // (also: the entries may be overwritten)
    };
    bool done = __all_sync(0xffffffffu, s.thr.x == inf && s.thr.y == inf);
    for (uint32_t b = 0; b * 32 < n && !done; ++b) {
        const uint32_t b0 = b * 32;
        if constexpr (SEG) {
            if (segs && b0 > 0 && (b0 & (stride - 1)) == 0) {
                if (queued && walk(queued)) break;
                // close the open segment here if it holds blends: each pixel's T is that after every
                // entry before b0, and the segment's own colour is kept until the walk has ended and
                // the colour behind the cut can be summed
                const uint32_t hi = __reduce_max_sync(0xffffffffu, max(s.last[0], s.last[1]));
                if (hi <= seg_lo) {
                    seg_lo = b0;  // nothing blended since the last cut
                } else if (!seg_stop) {
                    uint32_t pool_slot = kSegNone;
                    if (lane == 0) {
                        if (reserved == kSegNone) reserved = atomicAdd(&seg.ctrl->slots_used, 1u);
                        if (reserved < seg.fine || (b0 & (kSegStride - 1)) == 0) {
                            pool_slot = reserved;
                            if (pool_slot < seg.slots) reserved = atomicAdd(&seg.ctrl->slots_used, 1u);
                        }
                    }
                    pool_slot = __shfl_sync(0xffffffffu, pool_slot, 0);
                    if (pool_slot == kSegNone) {
                        stride = kSegStride;  // the slots left are for longer pieces
                    } else if (pool_slot >= seg.slots) {
                        seg_stop = true;  // pool full: the block's last segment takes the rest
                    } else {
                        if (lane == 0) seg.items[pool_slot] = make_uint4(block, seg_lo, hi, seg_last);
                        const float(&own)[2][3] = seg_n == 0 ? s.C : s.D;  // the first segment's colour is all there is
                        float4* st = seg.state(pool_slot) + lane;
                        st[0] = make_float4(s.T.x, own[0][0], own[0][1], own[0][2]);
                        st[32] = make_float4(s.T.y, own[1][0], own[1][1], own[1][2]);
#pragma unroll
                        for (int i = 0; i < 2; ++i) s.D[i][0] = s.D[i][1] = s.D[i][2] = 0.f;
                        ++seg_n;
                        seg_last = pool_slot;
                        seg_lo = b0;
                    }
                }
            }
        }
        cp_async_wait<kRecAhead - 1>();  // this lane's record of this batch, its id kRecAhead batches on
        const float4 a = Q.st.rec[slot][0][lane];
        const float bx0 = (float)bx + 0.5f, by0 = (float)by + 0.5f;
        const bool reach = b0 + lane < n && may_reach(a, bx0, bx0 + 7.f, by0, by0 + 7.f);
        const uint32_t bits = __ballot_sync(0xffffffffu, reach);
        if (reach) {
            FwdEntry& e = Q.e[(head + queued + __popc(bits & ((1u << lane) - 1u))) & (kQueue - 1)];
            e.p = make_float4(-a.x, -a.x, -a.y, -a.y);
            e.q = make_float4(-a.z, -a.z, -a.w, __uint_as_float(b0 + lane + 1));
            e.c = Q.st.rec[slot][1][lane];
        }
        stage_records(Q.st, b + kRecAhead, slot, n, lane, rec);
        stage_ids(Q.st, b + kRecAhead + kIdAhead, n, lane, id_of);
        cp_async_commit();
        slot = slot == kRecAhead - 1 ? 0u : slot + 1;
        queued += __popc(bits);
        if (queued >= 32) done = walk(queued & ~(uint32_t)(kFwdUnroll - 1));
    }
    cp_async_wait<0>();
    if (queued && !done) walk(queued);
    if constexpr (SEG) {
        if (segs) {
            const uint32_t hi = __reduce_max_sync(0xffffffffu, max(s.last[0], s.last[1]));
            if (lane == 0) {
                seg.last[block] = make_uint4(seg_n, hi > seg_lo ? seg_lo : kSegNone, hi, 0u);
                if (reserved != kSegNone && reserved < seg.slots)
                    seg.items[reserved] = make_uint4(kSegNone, 0u, 0u, kSegNone);  // taken, not used
            }
            __syncwarp();
            // the saved colours become the colour composited behind each cut: the background through
            // the last segment's T and the segments behind the cut, from the back (as the difference
            // of the colours up to the end and up to the cut, the little that shines through from
            // behind a nearly opaque front would keep few of its digits)
            if (seg_n > 0) {
                float S[2][3];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) S[h][ch] = fmaf(h ? s.T.y : s.T.x, bg[ch], s.D[h][ch]);
                for (uint32_t slot_i = seg_last; slot_i != kSegNone;) {
                    float4* st = seg.state(slot_i) + lane;
                    const uint32_t before = lane == 0 ? seg.items[slot_i].w : 0u;  // (lane 0 wrote it)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 v = st[32 * h];
                        st[32 * h] = make_float4(v.x, S[h][0], S[h][1], S[h][2]);
                        S[h][0] += v.y;
                        S[h][1] += v.z;
                        S[h][2] += v.w;
                    }
                    slot_i = __shfl_sync(0xffffffffu, before, 0);
                }
            }
        }
    }
    const size_t plane = (size_t)width * height;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int y = h ? y1 : y0;
        if (x >= width || y >= height) continue;
        const size_t pix = (size_t)y * width + x;
        const float T = h ? s.T.y : s.T.x;
        img[pix] = fmaf(T, bg[0], s.C[h][0]);
        img[plane + pix] = fmaf(T, bg[1], s.C[h][1]);
        img[2 * plane + pix] = fmaf(T, bg[2], s.C[h][2]);
        if (T_final) T_final[pix] = T;
        if (n_contrib) n_contrib[pix] = s.last[h];
    }
}

}  // namespace
}  // namespace igs
