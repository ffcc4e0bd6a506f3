// Octree initialisation of 3D Gaussians (Sec. 3.1: an Octree for 3D, as the
// QuadTree for 2D; colour = the cell average, sigma = half the cell width), from
// a coloured point set.
//
// Cells of level l (0 = the whole cube) are cubes of side side / 2^l, id =
// (8^l - 1) / 7 + Morton index (x lowest). Each holds the exact integer sums n,
// S1_c, S2_c of its points' colours quantised to 12 bits. The greedy growth
// (split the splittable leaf of largest error first, while the non-empty leaves
// stay within the budget) splits a prefix of the order (error descending, id
// ascending) over the splittable cells: a cell's error is never below a child's
// (the children partition its points) and its id is smaller, so every cell
// comes after its ancestors, and the greedy stops at the first cell of the
// order whose split (adding its non-empty children minus one) does not fit.
// The prefix is found by a radix selection on the 64-bit key (8 bits at a time,
// histograms weighted by the leaves each split adds), and then on the id among
// equal keys, by one cluster of CTAs that holds every key in shared memory (or by one
// CTA: few cells, or a device or partition of one that does not hold the cluster). The
// leaves are then emitted in id order, a CTA per chunk of cells placed after the
// leaves of the chunks before it. (2M points, seven levels, a budget of 500K: 752 us
// before, 478 with all that follows here, of which the kernels 286.)
//
// The counts (4 bytes a cell) sit apart from the colour sums (48): deciding what
// splits and where a leaf goes reads the counts alone, and the sums of empty cells
// are never read (with both in one 56-byte record, the seven sums over the levels took
// 88 us, counting the leaves 29; now 44 and 11).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"

namespace igs {
namespace {

struct OctSums {
    unsigned long long s1[3], s2[3];
};

__host__ __device__ inline long long oct_off(int l) { return (((long long)1 << (3 * l)) - 1) / 7; }

__device__ __forceinline__ uint32_t oct_morton(uint32_t x, uint32_t y, uint32_t z, int L) {
    uint32_t m = 0;
    for (int b = 0; b < L; ++b)
        m |= (((x >> b) & 1u) << (3 * b)) | (((y >> b) & 1u) << (3 * b + 1)) | (((z >> b) & 1u) << (3 * b + 2));
    return m;
}

struct OctParams {
    float lo[3];
    float inv;            // 2^L / side (FP32)
    double y00;           // 1 / (2 sqrt(pi)), for the SH DC coefficient
    double cell[8];       // per level: side / 2^l
    float log_half[8];    // per level: log(side / 2^(l+1)) (param_mode 1) or side / 2^(l+1)
    float op_value;       // stored opacity (logit with param_mode 1)
    int L, C, sh;
    long long k_max;
};

// (2M points: 14M atomics at random cells, 100 us, near the L2's atomic rate.)
__global__ void k_oct_base(const float* __restrict__ pts, const float* __restrict__ cols, long long npts,
                           OctParams P, uint32_t* __restrict__ cnt, OctSums* __restrict__ sums) {
    const int top = (1 << P.L) - 1;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npts;
         i += (long long)gridDim.x * blockDim.x) {
        const float px = pts[3 * i], py = pts[3 * i + 1], pz = pts[3 * i + 2];
        if (!isfinite(px) || !isfinite(py) || !isfinite(pz)) continue;
        const float p3[3] = {px, py, pz};
        uint32_t ix[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float t = floorf(__fmul_rn(__fsub_rn(p3[a], P.lo[a]), P.inv));
            ix[a] = t < 0.f ? 0u : (t > (float)top ? (uint32_t)top : (uint32_t)t);
        }
        const long long id = oct_off(P.L) + oct_morton(ix[0], ix[1], ix[2], P.L);
        atomicAdd(&cnt[id], 1u);
        OctSums* c = sums + id;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            const float v = fminf(fmaxf(cols[3 * i + ch], 0.f), 1.f);
            const unsigned long long q = (unsigned long long)rintf(__fmul_rn(v, 4096.f));
            atomicAdd(&c->s1[ch], q);
            atomicAdd(&c->s2[ch], q * q);
        }
    }
}

// Cells [0, 8^l) of level l from their children: eight lanes per cell, one child
// each. Every lane of a warp calls it (cell: this lane's cell, `on` if there is one).
__device__ __forceinline__ void oct_sum_children(uint32_t* __restrict__ cnt, OctSums* __restrict__ sums, int l,
                                                 long long cell, int child, bool on) {
    uint32_t n = 0;
    unsigned long long v[6] = {0, 0, 0, 0, 0, 0};
    if (on) {
        const long long k = oct_off(l + 1) + 8 * cell + child;
        n = cnt[k];
        if (n) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c] = sums[k].s1[c];
                v[3 + c] = sums[k].s2[c];
            }
        }
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        n += __shfl_xor_sync(0xffffffffu, n, o);
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
    }
    if (!on) return;
    const long long id = oct_off(l) + cell;
    if (child == 0) cnt[id] = n;
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(sums + id);  // s1, s2: six words
#pragma unroll
    for (int c = 0; c < 6; ++c)
        if (child == c) dst[c] = v[c];
}

__global__ void __launch_bounds__(256) k_oct_up(uint32_t* __restrict__ cnt, OctSums* __restrict__ sums, int l) {
    const long long t = blockIdx.x * 256ll + threadIdx.x, cell = t >> 3;
    oct_sum_children(cnt, sums, l, cell, (int)(t & 7), cell < (1LL << (3 * l)));
}

// Levels `from` .. 0 by one CTA, a level after another (each is read by the next).
constexpr int kOctTopLevel = 2;  // 64 cells and fewer
__global__ void __launch_bounds__(1024) k_oct_up_top(uint32_t* __restrict__ cnt, OctSums* __restrict__ sums, int from) {
    for (int l = from; l >= 0; --l) {
        const int cells = 1 << (3 * l);
        for (int t = threadIdx.x; t < ((8 * cells + 31) & ~31); t += 1024)
            oct_sum_children(cnt, sums, l, t >> 3, t & 7, (t >> 3) < cells);
        __syncthreads();  // (one CTA: its barrier orders its own global writes)
    }
}

constexpr int kOctThreads = 256;
constexpr int kOctChunk = kOctThreads * 8;  // cells per CTA of the emission
constexpr int kOctPasses = 11;              // 8 digits of the key, then 3 of the id (ids < 2^24)

// Error of a cell: max(0, sum_c (S2_c - S1_c^2 / n)) in double, one rounding per
// step in channel order (0 for an empty cell, and for one point, where every step is exact).
__device__ __forceinline__ double oct_err(uint32_t cnt, const OctSums& c) {
    if (cnt < 2) return 0.0;
    const double n = (double)cnt;
    double e = 0.0;
    for (int ch = 0; ch < 3; ++ch) {
        const double s1 = (double)c.s1[ch];
        e = __dadd_rn(e, __dsub_rn((double)c.s2[ch], __ddiv_rn(__dmul_rn(s1, s1), n)));
    }
    return e > 0.0 ? e : 0.0;
}

// The largest l with (8^l - 1) / 7 <= id, i.e. 8^l <= 7 id + 1 (ids < 2^24).
__device__ __forceinline__ int oct_level(long long id) { return (31 - __clz((int)(7u * (uint32_t)id + 1u))) / 3; }

// Errors (as bits, ordered like the value: they are not negative) and increments of
// the cells above the finest level: the leaves a split of the cell adds (non-empty
// children - 1), or 0xFF if it cannot split (fewer than 2 points).
__global__ void __launch_bounds__(256) k_oct_err(const uint32_t* __restrict__ cnt, const OctSums* __restrict__ sums,
                                                 long long items, unsigned long long* __restrict__ err,
                                                 uint8_t* __restrict__ inc8) {
    const long long id = blockIdx.x * 256ll + threadIdx.x;
    if (id >= items) return;
    const uint32_t n = cnt[id];
    uint32_t inc = 0xFFu;
    if (n >= 2) {
        const int l = oct_level(id);
        const uint32_t* k = cnt + oct_off(l + 1) + 8 * (id - oct_off(l));
        uint32_t kids = 0;
#pragma unroll
        for (int d = 0; d < 8; ++d) kids += k[d] > 0;
        inc = kids - 1;
    }
    err[id] = n >= 2 ? (unsigned long long)__double_as_longlong(oct_err(n, sums[id])) : 0ull;
    inc8[id] = (uint8_t)inc;
}

// The selection's state between passes. X = max{X : 1 + W(X) > k_max}, W(X) the
// increments of the splittable cells with key >= X, is found 8 bits at a time
// from the top: `above` = 1 + the increments of keys whose fixed high bits exceed
// `prefix`. Then, among keys == X, the first id (in id order) whose cumulative
// increments no longer fit k_max - above is found the same way on the id bits.
struct OctSel {
    unsigned long long prefix;  // key bits fixed so far; X once the key passes end
    long long above;
    unsigned long long idp;     // id bits fixed so far
    long long below;            // increments of keys == X with ids below the fixed id bits
    long long ihi;              // the last id of key X that splits
    int done;                   // no pass left to run
    int all;                    // every splittable cell splits
};

// The selection and the split flags, by one cluster of kSelCtas CTAs. Each holds an
// equal share of the cells above the finest level: their keys, key = min(error, the
// ancestors' errors), which keeps every child after its parent in the order whatever
// the rounding, and their increments. A pass counts the CTA's increments per digit in
// shared memory, sums the cluster's histograms over distributed shared memory (every
// CTA the same sums in the same order) and fixes the digit, in every CTA alike. Each
// warp keeps a list of its cells that the digits so far leave in question, so that the
// passes after the first two go over a few of them. 83 us at seven levels, most of it
// reading the ancestors' errors and the first passes; 16 SMs' worth of shared memory is
// what the keys need. (As two launches per pass, a histogram over all CTAs and a pick by
// one, the eleven passes took 108 us and the keys, a launch per level, 66; without the
// lists this kernel took 111.)
constexpr int kSelCtas = 16, kSelThreads = 1024;
constexpr long long kSelShare = (299593 + kSelCtas - 1) / kSelCtas;  // cells of levels 0 .. 6 (L <= 7)
constexpr int kSelSpan = (int)((kSelShare + kSelThreads / 32 - 1) / (kSelThreads / 32));  // cells per warp
constexpr size_t kSelSmem = (size_t)kSelShare * 9 + 1 + (size_t)kSelSpan * (kSelThreads / 32) * 2;
// Up to this many levels (4681 cells above the finest) one CTA is the better form: 20,000 points on
// 4 and 5 levels take 145 and 172 us in all, 174 and 192 with the cluster; on 6 and 7 levels 315 and 1437
// against 218 and 262, which is what a device without room for the cluster takes.
constexpr int kSelOneLevels = 5;
static_assert(kSelShare <= 65536 && kSelShare % 2 == 1, "16-bit lists, placed after the odd bytes of the increments");
static_assert(kSelSmem + 4096 <= 227 * 1024, "shared memory of a CTA");
//
// Without CLUSTER, one CTA does it all: the keys are formed in place of the errors, a level
// after another, and a pass goes over every cell in global memory.
template <bool CLUSTER>
__global__ void __launch_bounds__(kSelThreads) k_oct_select(const uint32_t* __restrict__ cnt,
                                                            unsigned long long* __restrict__ err,
                                                            const uint8_t* __restrict__ inc8, long long items,
                                                            long long k_max, uint8_t* __restrict__ split) {
    extern __shared__ unsigned long long s_key[];                       // [kSelShare]
    uint8_t* s_inc = reinterpret_cast<uint8_t*>(s_key + kSelShare);     // [kSelShare]
    uint16_t* s_list = reinterpret_cast<uint16_t*>(s_inc + kSelShare + 1);  // [warps][kSelSpan]: candidates
    __shared__ uint32_t s_h[256], s_scan[256], s_tot[256], s_warp[8];
    __shared__ OctSel s;
    __shared__ int s_b;
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();  // (of one CTA, without CLUSTER)
    const int t = threadIdx.x, lane = t & 31;
    const long long first = CLUSTER ? (long long)cluster.block_rank() * kSelShare : 0;
    const int mine = CLUSTER ? (int)max(0ll, min(kSelShare, items - first)) : (int)items;
    auto key_of = [&](int i) { return CLUSTER ? s_key[i] : err[i]; };
    auto inc_of = [&](int i) { return (uint32_t)(CLUSTER ? s_inc[i] : inc8[i]); };
    const int w0 = (t >> 5) * kSelSpan, w1 = min(mine, w0 + kSelSpan);  // this warp's cells
    uint16_t* list = s_list + w0;
    int left = 0;  // its candidates: cells whose split adds leaves, and whose key the digits so far allow
    if constexpr (!CLUSTER) {
        for (int l = 1; oct_off(l) < items; ++l) {  // (the parents' keys are complete)
            for (long long m = t; m < (1ll << (3 * l)); m += kSelThreads)
                err[oct_off(l) + m] = min(err[oct_off(l) + m], err[oct_off(l - 1) + (m >> 3)]);
            __syncthreads();
        }
    }
    for (int i0 = CLUSTER ? w0 : w1; i0 < w1; i0 += 32) {
        const int i = i0 + lane;
        bool cand = false;
        if (i < w1) {
            long long id = first + i;
            const uint32_t c = inc8[id];
            unsigned long long k = err[id];
            for (int l = oct_level(id); l > 0; --l) {  // up the ancestors
                id = oct_off(l - 1) + ((id - oct_off(l)) >> 3);
                k = min(k, err[id]);
            }
            s_key[i] = k;
            s_inc[i] = (uint8_t)c;
            cand = c != 0 && c != 0xFFu;
        }
        const uint32_t on = __ballot_sync(0xffffffffu, cand);
        if (cand) list[left + __popc(on & ((1u << lane) - 1u))] = (uint16_t)i;
        left += __popc(on);
    }
    if (t == 0) s = OctSel{};
    const bool root = cnt[0] > 0;
    for (int pass = 0; pass < kOctPasses; ++pass) {
        if (t < 256) s_h[t] = 0u;
        if (t == 0) s_b = pass < 8 ? 0 : 256;
        __syncthreads();
        if (s.done) break;  // (the same in every CTA)
        const unsigned long long prefix = s.prefix, idp = s.idp;
        const bool key = pass < 8;
        const int sh = 8 * (key ? 7 - pass : 10 - pass);
        const unsigned long long hi = key && pass == 0 ? 0ull : (~0ull << (sh + 8));
        int kept = 0;
        // the warp's list, or every 32nd run of 32 cells
        for (int j0 = CLUSTER ? 0 : t & ~31; j0 < (CLUSTER ? left : mine); j0 += CLUSTER ? 32 : kSelThreads) {
            uint32_t c = 0, d = 0;
            int i = 0;
            if (j0 + lane < (CLUSTER ? left : mine)) {
                i = CLUSTER ? list[j0 + lane] : j0 + lane;
                const unsigned long long k = key_of(i), id = (unsigned long long)(first + i);
                const bool in = key ? (k & hi) == prefix : k == prefix && (id & hi) == idp;
                d = (uint32_t)((key ? k : id) >> sh) & 0xFFu;
                if (in) c = inc_of(i);
                if (!CLUSTER && c == 0xFFu) c = 0;
            }
            uint32_t on = __ballot_sync(0xffffffffu, c != 0);
            // the list shrinks in place: what is written lies at or below what every lane has read
            if (CLUSTER && c) list[kept + __popc(on & ((1u << lane) - 1u))] = (uint16_t)i;
            kept += __popc(on);
            // the errors' top digits (sign and exponent) are few: a digit that many lanes share is added once
#pragma unroll
            for (int rep = 0; rep < 2 && on; ++rep) {
                const uint32_t lead = __shfl_sync(0xffffffffu, d, __ffs(on) - 1);
                const bool same = c != 0 && d == lead;
                const uint32_t sum = __reduce_add_sync(0xffffffffu, same ? c : 0u);
                if (lane == 0) atomicAdd(&s_h[lead], sum);
                if (same) c = 0;
                on = __ballot_sync(0xffffffffu, c != 0);
            }
            if (c) atomicAdd(&s_h[d], c);
        }
        left = kept;
        if constexpr (CLUSTER) {
            cluster.sync();  // every CTA's histogram is complete
            if (t < 256) {
                uint32_t h = 0;  // (all increments together are below 7 x 299593)
#pragma unroll
                for (int r = 0; r < kSelCtas; ++r) h += cluster.map_shared_rank(s_h, r)[t];
                s_tot[t] = h;
            }
            cluster.sync();  // no CTA reads another's histogram any more
        } else {
            __syncthreads();
            if (t < 256) s_tot[t] = s_h[t];
            __syncthreads();
        }
        // thread t < 256 holds one bin (bin 255 - t for the key, taken from the top; bin t for the id); an
        // inclusive scan gives each the increments at and above it (key) or at and below it (id)
        const int bin = key ? 255 - t : t;
        uint32_t v = t < 256 ? s_tot[bin] : 0u;
        if (t < 256) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
                if ((t & 31) >= o) v += u;
            }
            if ((t & 31) == 31) s_warp[t >> 5] = v;
        }
        __syncthreads();
        if (t < 256) {
            for (int q = 0; q < (t >> 5); ++q) v += s_warp[q];
            s_scan[t] = v;
        }
        __syncthreads();
        long long above = s.above;
        if (pass == 0) {
            above = 1;
            // 1 + W(0): the leaves if every splittable cell split
            if (!root || 1 + (long long)s_scan[255] <= k_max) {
                __syncthreads();
                if (t == 0) s.all = s.done = 1;
                continue;  // (the next pass's barrier shows it)
            }
        }
        if (t < 256) {
            if (key) {
                // the highest digit at which above + the increments at and above it exceed k_max (0 if none)
                if (bin >= 1 && above + v > k_max) atomicMax(&s_b, bin);
            } else {
                // the lowest digit at which the increments of key X, in id order, leave k_max - above
                if (s.below + v > k_max - above) atomicMin(&s_b, bin);
            }
        }
        __syncthreads();
        if (t == 0) {
            const int d = s_b;
            if (key) {
                s.prefix |= (unsigned long long)d << sh;
                s.above = above + (long long)s_scan[255 - d] - (long long)s_tot[d];  // + the increments above digit d
            } else if (d == 256) {  // every cell of key X fits
                s.ihi = items - 1;
                s.done = 1;
            } else {
                s.idp |= (unsigned long long)d << sh;
                s.below += (long long)s_scan[d] - (long long)s_tot[d];  // + the increments below digit d
                if (pass == kOctPasses - 1) {
                    s.ihi = (long long)s.idp - 1;  // idp: the first id whose increment does not fit
                    s.done = 1;
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();
    for (int i = t; i < mine; i += kSelThreads) {
        const long long id = first + i;
        bool sp = false;
        if (root && inc_of(i) != 0xFFu)
            sp = s.all != 0 || key_of(i) > s.prefix || (key_of(i) == s.prefix && id <= s.ihi);
        split[id] = sp ? 1 : 0;
    }
}

// Whether cell id holds a Gaussian: non-empty, its parent split (or the root), and
// itself not split (or the finest level).
__device__ __forceinline__ bool oct_leaf(const uint32_t* __restrict__ cnt, const uint8_t* __restrict__ split,
                                         long long id, long long cells, int L, int* lvl, long long* mor) {
    if (id >= cells || cnt[id] == 0) return false;
    const int l = oct_level(id);
    const long long m = id - oct_off(l);
    *lvl = l;
    *mor = m;
    const bool parent_split = l == 0 || split[oct_off(l - 1) + (m >> 3)];
    return parent_split && (l == L || !split[id]);
}

__device__ __forceinline__ long long oct_block_sum(long long v, long long* s_tmp) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_tmp[threadIdx.x >> 5] = v;
    __syncthreads();
    long long t = 0;
    for (int i = 0; i < kOctThreads / 32; ++i) t += s_tmp[i];
    return t;
}

// Leaves per chunk of kOctChunk cells.
__global__ void __launch_bounds__(kOctThreads) k_oct_count(const uint32_t* __restrict__ cnt,
                                                           const uint8_t* __restrict__ split, int L,
                                                           uint32_t* __restrict__ chunk_leaves) {
    __shared__ long long s_tmp[kOctThreads / 32];
    const long long cells = oct_off(L + 1), c0 = (long long)blockIdx.x * kOctChunk;
    long long n = 0;
    for (int j = threadIdx.x; j < kOctChunk; j += kOctThreads) {
        int l;
        long long m;
        n += oct_leaf(cnt, split, c0 + j, cells, L, &l, &m);
    }
    n = oct_block_sum(n, s_tmp);
    if (threadIdx.x == 0) chunk_leaves[blockIdx.x] = (uint32_t)n;
}

// The non-empty leaves in id order, one Gaussian each: a CTA per chunk, placed
// after the leaves of the chunks before it. The chunk's leaves are listed first and
// then taken one per thread: about a fifth of the cells are leaves, and FP64 steps
// (which this part issues at a small fraction of the FP32 rate) cost a warp the same
// whether one lane needs them or all (cell by cell the emission took 189 us, now 45). The
// mean of a channel, S1 / (4096 n) rounded to double and then to float, is formed
// in FP32 where n < 4096 and colours are plain: numerator and denominator are then
// FP32 numbers, and their quotient lies at least 2^-49 of its size from any midpoint of
// two floats that it does not hit, so rounding it through a double changes nothing.
__global__ void __launch_bounds__(kOctThreads) k_oct_emit(const uint32_t* __restrict__ cnt,
                                                         const OctSums* __restrict__ sums,
                                                         const uint8_t* __restrict__ split,
                                                         const uint32_t* __restrict__ chunk_leaves, OctParams P,
                                                         float4* __restrict__ out_ms, float* __restrict__ out_op,
                                                         float* __restrict__ out_col, int32_t* __restrict__ count) {
    __shared__ long long s_tmp[kOctThreads / 32];
    __shared__ int s_warp[2][kOctThreads / 32];
    __shared__ uint16_t s_leaf[kOctChunk];  // the chunk's leaves, relative to its first cell
    __shared__ float s_dc[3 * kOctThreads];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t mine = chunk_leaves[blockIdx.x];
    long long before = 0;
    for (unsigned b = threadIdx.x; b < blockIdx.x; b += kOctThreads) before += chunk_leaves[b];
    const long long base = oct_block_sum(before, s_tmp);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *count = (int32_t)min(base + (long long)mine, P.k_max);
    if (base >= P.k_max || mine == 0) return;  // uniform over the CTA
    const long long cells = oct_off(P.L + 1), c0 = (long long)blockIdx.x * kOctChunk;
    int listed = 0;
    for (int j0 = 0, buf = 0; j0 < kOctChunk; j0 += kOctThreads, buf ^= 1) {
        int l;
        long long m;
        const bool leaf = oct_leaf(cnt, split, c0 + j0 + threadIdx.x, cells, P.L, &l, &m);
        const uint32_t bal = __ballot_sync(0xffffffffu, leaf);
        if (lane == 0) s_warp[buf][w] = __popc(bal);
        __syncthreads();
        int at = listed;
        for (int i = 0; i < kOctThreads / 32; ++i) {
            if (i < w) at += s_warp[buf][i];
            listed += s_warp[buf][i];
        }
        if (leaf) s_leaf[at + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(j0 + threadIdx.x);
    }
    __syncthreads();
    const long long total = min((long long)listed, P.k_max - base);
    for (long long k0 = 0; k0 < total; k0 += kOctThreads) {
        const long long k = k0 + threadIdx.x;
        if (k < total) {
            const long long id = c0 + s_leaf[k], pos = base + k;
            const int l = oct_level(id);
            const long long m = id - oct_off(l);
            const uint32_t n = cnt[id];
            const OctSums& s = sums[id];
            uint32_t c3[3] = {0u, 0u, 0u};
            for (int b = 0; b < l; ++b)
                for (int a = 0; a < 3; ++a) c3[a] |= (uint32_t)((m >> (3 * b + a)) & 1) << b;
            const double cs = P.cell[l];
            out_ms[pos] = make_float4((float)__dadd_rn((double)P.lo[0], __dmul_rn((double)c3[0] + 0.5, cs)),
                                      (float)__dadd_rn((double)P.lo[1], __dmul_rn((double)c3[1] + 0.5, cs)),
                                      (float)__dadd_rn((double)P.lo[2], __dmul_rn((double)c3[2] + 0.5, cs)),
                                      P.log_half[l]);
            out_op[pos] = P.op_value;
            float* dc = s_dc + 3 * threadIdx.x;
            if (P.sh < 0 && n < 4096u) {
                for (int ch = 0; ch < 3; ++ch) dc[ch] = __fdiv_rn((float)s.s1[ch], 4096.f * (float)n);
            } else {
                for (int ch = 0; ch < 3; ++ch) {
                    const double mean = __ddiv_rn((double)s.s1[ch], __dmul_rn(4096.0, (double)n));
                    dc[ch] = P.sh < 0 ? (float)mean : (float)__ddiv_rn(__dsub_rn(mean, 0.5), P.y00);
                }
            }
        }
        __syncthreads();
        // these leaves hold positions [base + k0, ...): their colour rows are one contiguous
        // range, written by the whole CTA (DC from shared memory, the rest 0)
        const int rows = (int)min((long long)kOctThreads, total - k0);
        float* dst = out_col + (size_t)P.C * (size_t)(base + k0);
        for (int i = threadIdx.x; i < rows * P.C; i += kOctThreads) {
            const int r = i / P.C, q = i - r * P.C;
            dst[i] = q < 3 ? s_dc[3 * r + q] : 0.f;
        }
        __syncthreads();  // s_dc is rewritten by the next round
    }
}

}  // namespace

// Scratch: cell counts and sums, errors and increments of the cells above the finest
// level, split flags, leaves per emission chunk.
struct OctWork {
    OctSums* sums;
    uint32_t* cnt;
    unsigned long long* err;
    uint8_t *inc8, *split;
    uint32_t* chunk_leaves;
    size_t bytes;
};

OctWork oct_work(int L, void* base) {
    const size_t cells = (size_t)oct_off(L + 1), items = (size_t)oct_off(L);
    const size_t chunks = (cells + kOctChunk - 1) / kOctChunk;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const uintptr_t w = reinterpret_cast<uintptr_t>(base);
    OctWork o;
    size_t at = 0;
    o.sums = reinterpret_cast<OctSums*>(w + at);
    at += up(cells * sizeof(OctSums));
    o.cnt = reinterpret_cast<uint32_t*>(w + at);
    at += up(cells * 4);
    o.err = reinterpret_cast<unsigned long long*>(w + at);
    at += up(items * 8);
    o.inc8 = reinterpret_cast<uint8_t*>(w + at);
    at += up(items + 1);
    o.split = reinterpret_cast<uint8_t*>(w + at);
    at += up(items + 1);
    o.chunk_leaves = reinterpret_cast<uint32_t*>(w + at);
    at += up(chunks * 4);
    o.bytes = at;
    return o;
}

size_t octree_work_bytes(int L) {
    if (L < 0 || L > 7) return 0;
    return oct_work(L, nullptr).bytes;
}

// Whether the device holds the selection's cluster (with what the current context has of it): its
// shared memory and its size (above the portable eight) are opted into, once per device.
static bool sel_cluster_fits(const cudaLaunchConfig_t& cfg) {
    static std::mutex mu;
    static bool done[128] = {};
    int dev = 0, clusters = 0;
    auto ok = [](cudaError_t e) {
        if (e != cudaSuccess) cudaGetLastError();  // (the other form needs neither)
        return e == cudaSuccess;
    };
    if (!ok(cudaGetDevice(&dev)) || dev < 0 || dev >= 128) return false;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!done[dev]) {
            if (!ok(cudaFuncSetAttribute(k_oct_select<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSelSmem)) ||
                !ok(cudaFuncSetAttribute(k_oct_select<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)))
                return false;
            done[dev] = true;
        }
    }
    return ok(cudaOccupancyMaxActiveClusters(&clusters, k_oct_select<true>, &cfg)) && clusters > 0;
}

cudaError_t launch_octree_init(const float* pts, const float* cols, long long npts, const float lo[3], float side,
                               int L, long long k_max, float opacity, int sh_degree, int param_mode, float* out_ms,
                               float* out_op, float* out_col, int32_t* count, void* work, cudaStream_t st) {
    const long long cells = oct_off(L + 1), items = oct_off(L);
    const OctWork o = oct_work(L, work);
    OctParams P;
    for (int a = 0; a < 3; ++a) P.lo[a] = lo[a];
    P.inv = (float)((double)(1 << L) / (double)side);
    P.y00 = 0.5 / std::sqrt(3.14159265358979323846);
    for (int l = 0; l < 8; ++l) {
        const double half = 0.5 * (double)side / (double)(1 << l);
        P.log_half[l] = param_mode == 1 ? (float)std::log(half) : (float)half;
        P.cell[l] = (double)side / (double)(1 << l);
    }
    P.op_value = param_mode == 1 ? (float)std::log((double)opacity / (1.0 - (double)opacity)) : opacity;
    P.L = L;
    P.sh = sh_degree;
    P.C = sh_degree < 0 ? 3 : 3 * (sh_degree + 1) * (sh_degree + 1);
    P.k_max = k_max;
    // the finest level is counted into (its counts and sums zeroed), the others are written
    cudaError_t e = cudaMemsetAsync(o.sums + oct_off(L), 0, sizeof(OctSums) * ((size_t)1 << (3 * L)), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(o.cnt + oct_off(L), 0, 4 * ((size_t)1 << (3 * L)), st);
    if (e != cudaSuccess) return e;
    int launches = 0;
    if (npts > 0) {
        k_oct_base<<<(unsigned)std::min<long long>(ceil_div(npts, 256), 152 * 8), 256, 0, st>>>(pts, cols, npts, P,
                                                                                                o.cnt, o.sums);
        ++launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    for (int l = L - 1; l > kOctTopLevel; --l) {
        k_oct_up<<<(unsigned)ceil_div(8LL << (3 * l), 256), 256, 0, st>>>(o.cnt, o.sums, l);
        ++launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (L > 0) {
        k_oct_up_top<<<1, 1024, 0, st>>>(o.cnt, o.sums, std::min(L - 1, kOctTopLevel));
        k_oct_err<<<(unsigned)ceil_div(items, 256), 256, 0, st>>>(o.cnt, o.sums, items, o.err, o.inc8);
        launches += 2;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kSelCtas);
        cfg.blockDim = dim3(kSelThreads);
        cfg.dynamicSmemBytes = kSelSmem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kSelCtas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (L > kSelOneLevels && sel_cluster_fits(cfg))
            e = cudaLaunchKernelEx(&cfg, k_oct_select<true>, (const uint32_t*)o.cnt, o.err, (const uint8_t*)o.inc8,
                                   items, k_max, o.split);
        else {
            k_oct_select<false><<<1, kSelThreads, 0, st>>>(o.cnt, o.err, o.inc8, items, k_max, o.split);
            e = cudaGetLastError();
        }
        ++launches;
        if (e != cudaSuccess) return e;
    }
    const unsigned chunks = (unsigned)ceil_div(cells, kOctChunk);
    k_oct_count<<<chunks, kOctThreads, 0, st>>>(o.cnt, o.split, L, o.chunk_leaves);
    k_oct_emit<<<chunks, kOctThreads, 0, st>>>(o.cnt, o.sums, o.split, o.chunk_leaves, P, reinterpret_cast<float4*>(out_ms),
                                               out_op, out_col, count);
    launches += 2;
    count_launches(launches);
    return cudaGetLastError();
}

}  // namespace igs
