// Per-tile front-to-back compositing (Eq. 4) and its adjoint.
//
// One warp per 8 x 8 pixel block of a binning tile, two pixels per lane. The
// tile's entries (already in front-to-back order) pass by in batches of 32, those
// that can reach the block at all (w2 d^2 <= pmax at the nearest pixel centre) are
// queued in shared memory, and each pixel walks the queue with
//   alpha = min(alpha_max, o * 2^(-w2 d^2)),  w2 = log2(e) / (2 s^2)   (Eq. 8)
//   skip if alpha < alpha_min; stop (without blending) if T (1 - alpha) < t_min
//   C += c alpha T; T *= (1 - alpha)
// and the warp leaves the list as soon as every pixel has stopped.
// The backward pass walks each pixel's blended entries in reverse from n_contrib,
// recovering T_k = T_{k+1} / (1 - alpha_k) from the saved T_final, and reduces the
// per-pixel gradient terms of each entry over the warp before one vector atomic
// per (entry, 4 floats).
#include "blendtile.cuh"
#include "warp.cuh"

namespace igs {
namespace {

// Zeros to n4 float4 at p (none if p is null), spread over the grid: the
// forward blend of a training step clears the 2D gradient for the adjoint that
// follows. The blend is bound by instruction issue and leaves HBM mostly idle,
// so the stores cost it a few instructions per thread, not a pass of their own.
__device__ __forceinline__ void clear_slice(float4* __restrict__ p, uint64_t n4) {
    if (!p) return;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (uint64_t)gridDim.x * blockDim.x)
        p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---- backward: one warp per 8 x 8 pixel block ----
//
// Like the forward (blendtile.cuh), the reverse walk is bound by instruction
// issue: two pixels of one column per lane on packed FP32 steps, the reached
// entries compacted into a queue and walked without branches. The entry's own
// factors (d alpha / d power = -ln 2 o g, d power / d(u, v) = -2 w2 (dx, dy))
// are the same for every pixel, so the walk sums dalpha g times (dx, dy, d^2, 1)
// and the factors are applied once per entry, after the warp reduction. The
// reduction of the seven terms (31 of about 90 instructions per entry) is the
// largest part left. 398 -> 297 us for a 1080p view of 1M clustered Gaussians,
// 458 -> 333 us for the 3M training views, 133 -> 85 us at 30K Gaussians and
// 401 x 299 pixels (there latency-bound: 2000 blocks).
struct BwdQueue {
    FwdEntry e[kQueue];   // q.w: the list position's bits (not + 1)
    Stager st;
    float red[32][8];     // reduced terms of the entries of one walk
    uint32_t id[kQueue];  // the queued entries' Gaussians
};

// The colour composited behind the current entry, S, enters the adjoint only
// through G . S (G = dL/dC), so a pixel carries that scalar, negated:
// nGS = -G . (T_final bg) at the start, then nGS -= w T (G . c) per blended entry.
struct BwdPixels {
    float2 px, py;  // centres: px the same twice
    float2 T, nGS;
    float G[2][3];
    uint32_t nc[2];
};

__device__ __forceinline__ float fast_rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// (A pixel that did not blend an entry multiplies its T by fast_rcp(1), thousands of times
// in a long walk. That this is 1 exactly is not promised by the instruction's error bound
// of one ulp; it holds on this hardware, and a test holds it: selects for T cost 1 % of the
// backward, 299 us a 1080p view of 1M Gaussians without and 302 with.)
//
// The adjoint of one entry at the warp's 64 pixels, summed over the warp: lane
// 4 v holds term v of (dalpha g (dx, dy, d^2, 1), dr, dg, db, -). With FINITE
// (every G of the warp and every distance is finite), a pixel that did not blend
// the entry enters the sums with zero factors; otherwise its terms are left out by selects.
template <bool FINITE>
__device__ __forceinline__ float bwd_entry(const FwdEntry& en, const BlendParams& P, BwdPixels& s, int lane) {
    const float4 p = en.p, q = en.q, c = en.c;
    const float2 dx = pk_add(s.px, make_float2(p.x, p.y));
    const float2 dy = pk_add(s.py, make_float2(p.z, p.w));
    const float2 d2 = pk_fma(dx, dx, pk_mul(dy, dy));
    const float2 npw = pk_mul(make_float2(q.x, q.y), d2);
    const uint32_t pos = __float_as_uint(q.w);
    const float2 g = make_float2(fast_exp2(npw.x), fast_exp2(npw.y));
    const float2 og = make_float2(__fmul_rn(c.w, g.x), __fmul_rn(c.w, g.y));
    const float ax = fminf(P.alpha_max, og.x), ay = fminf(P.alpha_max, og.y);
    const bool in0 = pos < s.nc[0] && !(npw.x < q.z) && ax >= P.alpha_min;
    const bool in1 = pos < s.nc[1] && !(npw.y < q.z) && ay >= P.alpha_min;
    const float2 alpha = make_float2(in0 ? ax : 0.f, in1 ? ay : 0.f);
    const float2 oma = pk_fma(alpha, make_float2(-1.f, -1.f), make_float2(1.f, 1.f));  // >= 1 - alpha_max > 0
    const float2 inv = make_float2(fast_rcp(oma.x), fast_rcp(oma.y));
    const float2 Tk = pk_mul(s.T, inv);  // transmittance before this entry
    const float2 wT = pk_mul(alpha, Tk);
    s.T = Tk;
    float v[8];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        if (FINITE)
            v[4 + ch] = fmaf(wT.x, s.G[0][ch], wT.y * s.G[1][ch]);
        else
            v[4 + ch] = (in0 ? wT.x * s.G[0][ch] : 0.f) + (in1 ? wT.y * s.G[1][ch] : 0.f);
    }
    const float2 Gc = make_float2(fmaf(s.G[0][2], c.z, fmaf(s.G[0][1], c.y, s.G[0][0] * c.x)),
                                  fmaf(s.G[1][2], c.z, fmaf(s.G[1][1], c.y, s.G[1][0] * c.x)));
    const float2 da = pk_mul(pk_fma(Tk, Gc, pk_mul(s.nGS, inv)), g);  // dalpha g
    if (in0) s.nGS.x = fmaf(-wT.x, Gc.x, s.nGS.x);
    if (in1) s.nGS.y = fmaf(-wT.y, Gc.y, s.nGS.y);
    const float dg0 = in0 && og.x <= P.alpha_max ? da.x : 0.f;  // alpha not clamped
    const float dg1 = in1 && og.y <= P.alpha_max ? da.y : 0.f;
    v[3] = dg0 + dg1;
    if (FINITE) {
        v[0] = v[3] * dx.x;  // (dx is the same for both pixels)
        v[1] = fmaf(dg0, dy.x, dg1 * dy.y);
        v[2] = fmaf(dg0, d2.x, dg1 * d2.y);
    } else {
        v[0] = (in0 ? dg0 * dx.x : 0.f) + (in1 ? dg1 * dx.y : 0.f);
        v[1] = (in0 ? dg0 * dy.x : 0.f) + (in1 ? dg1 * dy.y : 0.f);
        v[2] = (in0 ? dg0 * d2.x : 0.f) + (in1 ? dg1 * d2.y : 0.f);
    }
    v[7] = 0.f;
    return warp_reduce8(v, lane);
}

// Walk cnt <= 32 queued entries from ring slot `head` on, then add each one's
// terms to its Gaussian's row of g2d (two float4 atomics per entry).
template <bool FINITE>
__device__ __forceinline__ void bwd_walk(BwdQueue& Q, uint32_t head, uint32_t cnt, const BlendParams& P, BwdPixels& s,
                                         int lane, float4* __restrict__ g2d) {
    __syncwarp();
#pragma unroll 2
    for (uint32_t k = 0; k < cnt; ++k) {
        const float r = bwd_entry<FINITE>(Q.e[(head + k) & (kQueue - 1)], P, s, lane);
        if ((lane & 3) == 0) Q.red[k][lane >> 2] = r;
    }
    __syncwarp();
    for (uint32_t t = (uint32_t)lane; t < 2 * cnt; t += 32) {
        const uint32_t k = t >> 1, h = t & 1u, at = (head + k) & (kQueue - 1);
        float4 acc = *reinterpret_cast<const float4*>(&Q.red[k][4 * h]);
        if (h == 0) {
            const float ocl = -kLn2 * Q.e[at].c.w, k2 = ocl * (2.f * Q.e[at].q.x);  // q.x = -w2
            acc.x *= k2;
            acc.y *= k2;
            acc.z *= ocl;
        }
        if (acc.x != 0.f || acc.y != 0.f || acc.z != 0.f || acc.w != 0.f)
            atomicAdd(&g2d[2 * (size_t)Q.id[at] + h], acc);
    }
    __syncwarp();
}

// One warp walks the entries rg of its 8 x 8 block at pixel (bx, by) from the last
// one any of its pixels blended to the first, or, for a walk segment, list positions
// [seg_lo, seg_hi) from the pixels' saved state at seg_hi (seg_state: 64 pixels
// (T, colour behind); nullptr: the final state). Staged like blend_block_fwd.
__device__ __forceinline__ void blend_block_bwd(int bx, int by, uint2 rg, const uint32_t* __restrict__ vals,
                                                const float4* __restrict__ rec, const BlendParams& P,
                                                const float* __restrict__ dL, const float* __restrict__ T_final,
                                                const uint32_t* __restrict__ n_contrib, float4* __restrict__ g2d,
                                                BwdQueue& Q, uint32_t seg_lo = 0, uint32_t seg_hi = kSegNone,
                                                const float4* __restrict__ seg_state = nullptr) {
    const uint32_t lane = threadIdx.x & 31;
    const int x = bx + (int)(lane & 7), y0 = by + (int)(lane >> 3);
    const size_t plane = (size_t)P.width * P.height;
    BwdPixels s;
    s.px = make_float2((float)x + 0.5f, (float)x + 0.5f);
    s.py = make_float2((float)y0 + 0.5f, (float)(y0 + 4) + 0.5f);
    float T[2], nGS[2];
    bool finite = true;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int y = y0 + 4 * i;
        float* G = s.G[i];
        G[0] = G[1] = G[2] = 0.f;
        T[i] = 1.f;
        s.nc[i] = 0;
        if (x < P.width && y < P.height) {
            const size_t pix = (size_t)y * P.width + x;
            G[0] = dL[pix];
            G[1] = dL[plane + pix];
            G[2] = dL[2 * plane + pix];
            T[i] = T_final[pix];
            s.nc[i] = n_contrib[pix];
        }
        finite &= isfinite(G[0]) && isfinite(G[1]) && isfinite(G[2]);
        nGS[i] = -(T[i] * (G[0] * P.bg[0] + G[1] * P.bg[1] + G[2] * P.bg[2]));
        if (seg_state) {  // pixel index in the block: row * 8 + column = lane + 32 i
            const float4 v = seg_state[lane + 32 * i];
            T[i] = v.x;
            nGS[i] = -(G[0] * v.y + G[1] * v.z + G[2] * v.w);
        }
    }
    s.T = make_float2(T[0], T[1]);
    s.nGS = make_float2(nGS[0], nGS[1]);
    finite = __all_sync(0xffffffffu, finite);
    const uint32_t n = rg.y > rg.x ? rg.y - rg.x : 0u;
    // nothing blended at or past hi; the walk takes positions hi - 1 - j, j < total
    const uint32_t hi = min(min(__reduce_max_sync(0xffffffffu, max(s.nc[0], s.nc[1])), seg_hi), n);
    const uint32_t total = hi > seg_lo ? hi - seg_lo : 0u;
    vals += rg.x;
    const auto id_of = [vals, hi](uint32_t j) { return vals + (hi - 1 - j); };
    stage_begin(Q.st, total, lane, rec, id_of);
    uint32_t head = 0, queued = 0, slot = 0;
    auto walk = [&](uint32_t cnt) {
        if (finite)
            bwd_walk<true>(Q, head, cnt, P, s, lane, g2d);
        else
            bwd_walk<false>(Q, head, cnt, P, s, lane, g2d);
        head = (head + cnt) & (kQueue - 1);
        queued -= cnt;
    };
    const float bx0 = (float)bx + 0.5f, by0 = (float)by + 0.5f;
    for (uint32_t b = 0; b * 32 < total; ++b) {
        const uint32_t j = b * 32 + lane;
        cp_async_wait<kRecAhead - 1>();  // this lane's record of this batch, its id kRecAhead batches on
        const float4 a = Q.st.rec[slot][0][lane];
        const bool reach = j < total && may_reach(a, bx0, bx0 + 7.f, by0, by0 + 7.f);
        const uint32_t bits = __ballot_sync(0xffffffffu, reach);
        // (a centre so far away that its squared distance overflows: no product with zero from here on)
        finite = finite && !__any_sync(0xffffffffu, reach && !(fabsf(a.x) + fabsf(a.y) < 1e15f));
        if (reach) {
            const uint32_t at = (head + queued + __popc(bits & ((1u << lane) - 1u))) & (kQueue - 1);
            FwdEntry& e = Q.e[at];
            e.p = make_float4(-a.x, -a.x, -a.y, -a.y);
            e.q = make_float4(-a.z, -a.z, -a.w, __uint_as_float(hi - 1 - j));
            e.c = Q.st.rec[slot][1][lane];
            Q.id[at] = Q.st.id[b & (kIdSlots - 1)][lane];
        }
        stage_records(Q.st, b + kRecAhead, slot, total, lane, rec);
        stage_ids(Q.st, b + kRecAhead + kIdAhead, total, lane, id_of);
        cp_async_commit();
        slot = slot == kRecAhead - 1 ? 0u : slot + 1;
        queued += __popc(bits);
        if (queued >= 32) walk(32);
    }
    cp_async_wait<0>();
    if (queued) walk(queued);
    __syncwarp();
}

// Sub-tile kernels: one CTA per 8 x 8 pixel block of a TS x TS binning tile,
// walking the binning tile's entries; each block stops on its own (its
// pixels' last contributors), and entries that miss it cost one reach test.
// Per pixel the walk, the arithmetic and the result are those of the whole-tile
// kernels.
template <int TS>
__global__ void __launch_bounds__(32, kFwdMinCtas) k_blend_fwd_sub(
    const uint2* __restrict__ ranges, const uint32_t* __restrict__ vals, const float4* __restrict__ rec, BlendParams P,
    float* __restrict__ img, float* __restrict__ T_final, uint32_t* __restrict__ n_contrib,
    const uint32_t* __restrict__ info, SegLayout seg, const uint32_t* __restrict__ tile_order,
    float4* __restrict__ clear, uint64_t clear4) {
    pdl_wait();
    constexpr int SUB = TS / 8;
    __shared__ FwdQueue s_q;
    clear_slice(clear, clear4);
    if (info[kInfoAbort]) return;
    const int q = (int)(blockIdx.x % (SUB * SUB));
    const uint32_t tiles = (uint32_t)(P.tiles_x * P.tiles_y);
    uint32_t t = blockIdx.x / (SUB * SUB);  // in starting order
    if (tile_order && (t = tile_order[t]) >= tiles) return;  // (a frame whose binning never ordered its tiles)
    const int tile = (int)t;
    const int tx = tile % P.tiles_x, ty = tile / P.tiles_x;
    blend_block_fwd<TS != 8>((tx * SUB + q % SUB) * 8, (ty * SUB + q / SUB) * 8, P.width, P.height, ranges[tile], vals,
                             rec, P.alpha_min, P.alpha_max, P.t_min, P.bg, s_q, img, T_final,
                             n_contrib, seg, (uint32_t)(tile * SUB * SUB + q));
}

// The backward of a block's whole walk (8-pixel tiles; larger ones when the
// frame has no room for walk segments).
constexpr int kBwdMinCtas = 24;  // resident one-warp CTAs per SM asked of the compiler
static_assert(kBwdMinCtas * (sizeof(BwdQueue) + 1024) <= 228 * 1024, "resident CTAs per SM");
template <int TS>
__global__ void __launch_bounds__(32, kBwdMinCtas) k_blend_bwd_sub(
    const uint2* __restrict__ ranges, const uint32_t* __restrict__ vals, const float4* __restrict__ rec, BlendParams P,
    const float* __restrict__ dL, const float* __restrict__ T_final, const uint32_t* __restrict__ n_contrib,
    float4* __restrict__ g2d, const uint32_t* __restrict__ info) {
    pdl_wait();
    constexpr int SUB = TS / 8;
    __shared__ BwdQueue s_q;
    if (info[kInfoAbort]) return;
    const int tile = blockIdx.x / (SUB * SUB), q = blockIdx.x % (SUB * SUB);
    const int tx = tile % P.tiles_x, ty = tile / P.tiles_x;
    blend_block_bwd((tx * SUB + q % SUB) * 8, (ty * SUB + q / SUB) * 8, ranges[tile], vals, rec, P, dL, T_final,
                    n_contrib, g2d, s_q);
}

// The backward over walk segments: one-warp CTAs, all resident, take work from
// one counter: first the segments the forward closed, then each block's last
// segment (its whole walk when it closed none). A piece walks at most 1024
// list positions, or 256 (SegLayout), unless the pool ran out, so no block's long
// walk sets the kernel's length.
template <int TS>
__global__ void __launch_bounds__(32, kBwdMinCtas) k_blend_bwd_segs(const uint2* __restrict__ ranges,
                                                           const uint32_t* __restrict__ vals,
                                                           const float4* __restrict__ rec, BlendParams P,
                                                           const float* __restrict__ dL,
                                                           const float* __restrict__ T_final,
                                                           const uint32_t* __restrict__ n_contrib,
                                                           float4* __restrict__ g2d,
                                                           const uint32_t* __restrict__ info, SegLayout seg) {
    pdl_wait();
    constexpr int SUB = TS / 8;
    __shared__ BwdQueue s_q;
    if (info[kInfoAbort]) return;
    const uint32_t items = min(seg.ctrl->slots_used, seg.slots);  // closed segments, by pool slot
    const uint32_t total = items + seg.blocks;                       // then each block's last segment
    for (;;) {
        uint32_t u = 0;
        if (threadIdx.x == 0) u = atomicAdd(&seg.ctrl->next, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= total) break;
        uint32_t block, lo, hi, slot = kSegNone;
        if (u < items) {
            const uint4 it = seg.items[u];
            if (it.x == kSegNone) continue;  // a slot taken ahead and not used
            block = it.x;
            lo = it.y;
            hi = it.z;
            slot = u;
        } else {
            block = u - items;
            const uint4 l = seg.last[block];
            if (l.y == kSegNone) continue;  // its last segment holds no blend
            lo = l.y;
            hi = l.z;
        }
        const int tile = (int)(block / (SUB * SUB)), q = (int)(block % (SUB * SUB));
        const int tx = tile % P.tiles_x, ty = tile / P.tiles_x;
        blend_block_bwd((tx * SUB + q % SUB) * 8, (ty * SUB + q / SUB) * 8, ranges[tile], vals, rec, P, dL, T_final,
                        n_contrib, g2d, s_q, lo, hi, slot == kSegNone ? nullptr : seg.state(slot));
    }
}

}  // namespace

// Walk segments of the sub-tile blends of frame f (off for 8-pixel tiles and
// when the frame's depth-item buffers cannot hold a useful pool).
SegLayout frame_segments(const igs_frame& f) {
    if (f.tile != 16 && f.tile != 32) return SegLayout{};
    const SortScratch s = sort_scratch(f);
    const int64_t sub = f.tile / 8;
    return seg_layout(s.seg_base, s.seg_bytes, s.seg_base2, s.seg_bytes2, (int64_t)f.tiles_x * f.tiles_y * sub * sub);
}

cudaError_t launch_blend_fwd(const igs_frame& f, const BlendParams& bp, float* img, cudaStream_t st, float* clear_g2d) {
    const unsigned tiles = (unsigned)(f.tiles_x * f.tiles_y);
    auto clear = reinterpret_cast<float4*>(clear_g2d);
    const uint64_t clear4 = clear_g2d ? 2 * (uint64_t)f.n : 0;  // [n][8] floats
    if (tiles == 0) {  // nothing to blend; the gradient is still cleared for the adjoint
        if (!clear || clear4 == 0) return cudaSuccess;
        ZeroRanges z = {};
        z.ptr[0] = clear;
        z.bytes[0] = clear4 * 16;
        z.count = 1;
        return launch_zero(z, st);
    }
    auto rg = reinterpret_cast<const uint2*>(f.ranges);
    auto rec = reinterpret_cast<const float4*>(f.rec);
    const SegLayout seg = frame_segments(f);
    cudaError_t e = cudaSuccess;
    if (seg.slots) {  // a fresh list of segments for this forward
        ZeroRanges z = {};
        z.ptr[0] = seg.ctrl;
        z.bytes[0] = sizeof(SegCtrl);
        z.count = 1;
        if ((e = launch_zero(z, st)) != cudaSuccess) return e;
    }
    const uint32_t* tile_order = f.n > 0 ? sort_scratch(f).tile_order : nullptr;  // (an empty scene bins nothing)
    const int64_t sub = f.tile / 8;
    const dim3 grid((unsigned)((int64_t)tiles * sub * sub)), block(32);
    switch (f.tile) {
        case 8: e = launch_pdl(k_blend_fwd_sub<8>, grid, block, 0, st, rg, f.vals, rec, bp, img, f.T_final, f.n_contrib, f.info, seg, tile_order, clear, clear4); break;
        case 16: e = launch_pdl(k_blend_fwd_sub<16>, grid, block, 0, st, rg, f.vals, rec, bp, img, f.T_final, f.n_contrib, f.info, seg, tile_order, clear, clear4); break;
        case 32: e = launch_pdl(k_blend_fwd_sub<32>, grid, block, 0, st, rg, f.vals, rec, bp, img, f.T_final, f.n_contrib, f.info, seg, tile_order, clear, clear4); break;
        default: return cudaErrorInvalidValue;
    }
    count_launches();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The segmented backward: one-warp CTAs, kBwdMinCtas resident per SM.
constexpr unsigned kSegCtas = 152 * kBwdMinCtas;

cudaError_t launch_blend_bwd(const igs_frame& f, const BlendParams& bp, const float* dL, float* g2d, cudaStream_t st) {
    const unsigned tiles = (unsigned)(f.tiles_x * f.tiles_y);
    if (tiles == 0) return cudaSuccess;
    auto rg = reinterpret_cast<const uint2*>(f.ranges);
    auto rec = reinterpret_cast<const float4*>(f.rec);
    auto g = reinterpret_cast<float4*>(g2d);
    const SegLayout seg = frame_segments(f);
    cudaError_t e = cudaSuccess;
    switch (f.tile) {
        case 8: e = launch_pdl(k_blend_bwd_sub<8>, dim3(tiles), dim3(32), 0, st, rg, f.vals, rec, bp, dL, f.T_final, f.n_contrib, g, f.info); break;
        case 16:
            if (seg.slots)
                e = launch_pdl(k_blend_bwd_segs<16>, dim3(kSegCtas), dim3(32), 0, st, rg, f.vals, rec, bp, dL, f.T_final, f.n_contrib, g, f.info, seg);
            else
                e = launch_pdl(k_blend_bwd_sub<16>, dim3(tiles * 4), dim3(32), 0, st, rg, f.vals, rec, bp, dL, f.T_final, f.n_contrib, g, f.info);
            break;
        case 32:
            if (seg.slots)
                e = launch_pdl(k_blend_bwd_segs<32>, dim3(kSegCtas), dim3(32), 0, st, rg, f.vals, rec, bp, dL, f.T_final, f.n_contrib, g, f.info, seg);
            else
                e = launch_pdl(k_blend_bwd_sub<32>, dim3(tiles * 16), dim3(32), 0, st, rg, f.vals, rec, bp, dL, f.T_final, f.n_contrib, g, f.info);
            break;
        default: return cudaErrorInvalidValue;
    }
    count_launches();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The backward's work counter of frame f (zeroed with the 2D gradient before
// each backward), or nullptr when the frame has no walk segments.
void* blend_bwd_counter(const igs_frame& f) {
    const SegLayout seg = frame_segments(f);
    return seg.slots ? &seg.ctrl->next : nullptr;
}

const uint32_t* blend_segments_used(const igs_frame& f) {
    const SegLayout seg = frame_segments(f);
    return seg.slots ? &seg.ctrl->slots_used : nullptr;
}

}  // namespace igs
