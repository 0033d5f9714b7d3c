// Adaptive octree construction for the Laplace FMM (Sec. 6.4.1), as plain
// data-parallel kernels around the task-parallel traversal:
//   1. bounding cube of the points (min/max reduction);
//   2. 63-bit Morton codes, 21 bits per axis, q = min(2^21-1, floor((x-lo)*2^21/side));
//   3. stable LSD radix sort of (code, input index), 8 passes of 8 bits, so
//      equal codes keep input order: the digit counts of all passes are taken
//      with the codes, and a pass is one kernel whose tiles hand their digit
//      prefixes on (decoupled look-back, Merrill and Garland 2016);
//   4. level-synchronous refinement: a cell of level l with more than
//      leaf_size points (and l < 21) splits into its non-empty octants, found
//      by search in the sorted codes; child cells are numbered breadth first by
//      a scan of the per-cell child counts.  One kernel refines all levels, with
//      a barrier of its running blocks between them;
//   5. gather of the points into Morton order.
// A build is 14 launches in the mixed form, 13 in FP64 (no leaf-local coordinates), and a memset,
// whatever the set (five launches per radix pass and five per level made 85); most of a small set's build time was launches and the 7 x 20
// dependent loads of one thread searching the root cell.  Build time before ->
// now: 3,001 points 0.64 -> 0.16 ms, Plummer 60,001 0.85 -> 0.23 ms, uniform 2^20
// 0.96 -> 0.47 ms.  A small set is bound by the chain of launches and barriers,
// a large one by the latency of the eight dependent passes.
// The geometry is computed in FP64 with every operation rounded separately
// (no contraction), so cell centres and codes are reproducible bit for bit.
#include <cuda_runtime.h>

#include "fmm_internal.h"

namespace gtap {
namespace fmm {
namespace {

constexpr int kRsBlock = 256;

// A wait that runs out marks the build as failed.  The other waits of the build then end at once and the
// kernels behind it do no work on keys that were never written: a failed build takes one wait's limit,
// not one for each.
__device__ __forceinline__ bool build_failed(const int* flags) { return *(const volatile int*)(flags + 1) != 0; }

// Bounding cube: per-block min/max, and the last block to finish reduces those and
// writes box = {lo x, lo y, lo z, side, scale, 0} and the root cell.
__global__ void __launch_bounds__(256) k_bbox(const double* pos, long long n, double* part, unsigned* done, double* box,
                                              Dbl4* geom, int4* info, int4* lat, int* lstart, int* flags) {
    __shared__ double sh[6][256];
    __shared__ bool last;
    const int t = threadIdx.x;
    double mn[3] = {pos[0], pos[1], pos[2]}, mx[3] = {pos[0], pos[1], pos[2]};
    for (long long i = blockIdx.x * (long long)blockDim.x + t; i < n; i += (long long)gridDim.x * blockDim.x)
        for (int d = 0; d < 3; ++d) {
            const double v = pos[3 * i + d];
            mn[d] = fmin(mn[d], v);
            mx[d] = fmax(mx[d], v);
        }
    auto reduce = [&] {
        for (int d = 0; d < 3; ++d) { sh[d][t] = mn[d]; sh[3 + d][t] = mx[d]; }
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if (t < o)
                for (int d = 0; d < 3; ++d) {
                    sh[d][t] = fmin(sh[d][t], sh[d][t + o]);
                    sh[3 + d][t] = fmax(sh[3 + d][t], sh[3 + d][t + o]);
                }
            __syncthreads();
        }
    };
    reduce();
    if (t < 6) {
        __stcg(&part[blockIdx.x * 6 + t], sh[t][0]);
        __threadfence();
    }
    __syncthreads();
    if (t == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int d = 0; d < 3; ++d) { mn[d] = sh[d][0]; mx[d] = sh[3 + d][0]; }
    __syncthreads();
    for (int b = t; b < (int)gridDim.x; b += blockDim.x)
        for (int d = 0; d < 3; ++d) {
            mn[d] = fmin(mn[d], __ldcg(&part[6 * b + d]));
            mx[d] = fmax(mx[d], __ldcg(&part[6 * b + 3 + d]));
        }
    reduce();
    if (t != 0) return;
    double side = 0.0;
    for (int d = 0; d < 3; ++d) side = fmax(side, __dsub_rn(sh[3 + d][0], sh[d][0]));
    if (!(side > 0.0)) side = 1.0;
    const double half = __dmul_rn(side, 0.5);
    double c[3];
    for (int d = 0; d < 3; ++d) {
        const double lo = __dsub_rn(__dmul_rn(__dadd_rn(sh[d][0], sh[3 + d][0]), 0.5), half);
        box[d] = lo;
        c[d] = __dadd_rn(lo, half);
    }
    box[3] = side;
    box[4] = __ddiv_rn(2097152.0, side);
    box[5] = 0.0;   // largest |charge|: the gather's
    geom[0] = make_dbl4(c[0], c[1], c[2], half);
    info[0] = make_int4(0, (int)n, -1, 0);
    lat[0] = make_int4(1 << 21, 1 << 21, 1 << 21, 0);
    lstart[0] = 0;
    lstart[1] = 1;
    for (int i = 0; i < 4; ++i) flags[i] = 0;
}

__device__ __forceinline__ unsigned long long spread21(unsigned long long v) {
    v &= 0x1FFFFFull;
    v = (v | (v << 32)) & 0x1F00000000FFFFull;
    v = (v | (v << 16)) & 0x1F0000FF0000FFull;
    v = (v | (v << 8)) & 0x100F00F00F00F00Full;
    v = (v | (v << 4)) & 0x10C30C30C30C30C3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__device__ __forceinline__ unsigned long long compact21(unsigned long long v) {
    v &= 0x1249249249249249ull;
    v = (v | (v >> 2)) & 0x10C30C30C30C30C3ull;
    v = (v | (v >> 4)) & 0x100F00F00F00F00Full;
    v = (v | (v >> 8)) & 0x1F0000FF0000FFull;
    v = (v | (v >> 16)) & 0x1F00000000FFFFull;
    v = (v | (v >> 32)) & 0x1FFFFFull;
    return v;
}

constexpr int kPasses = 8;   // of 8 bits

// Codes, and the digit counts of every pass (the counts do not depend on the order of the keys).
__global__ void __launch_bounds__(kRsBlock) k_codes(const double* pos, long long n, const double* box,
                                                    unsigned long long* keys, uint32_t* vals, unsigned* counts) {
    __shared__ unsigned h[kPasses][256];
    for (int p = 0; p < kPasses; ++p) h[p][threadIdx.x] = 0;
    __syncthreads();
    const double lo[3] = {box[0], box[1], box[2]}, scale = box[4];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        unsigned long long q[3];
        for (int d = 0; d < 3; ++d) {
            double f = floor(__dmul_rn(__dsub_rn(pos[3 * i + d], lo[d]), scale));
            f = fmin(fmax(f, 0.0), 2097151.0);
            q[d] = (unsigned long long)f;
        }
        const unsigned long long key = spread21(q[0]) | (spread21(q[1]) << 1) | (spread21(q[2]) << 2);
        keys[i] = key;
        vals[i] = (uint32_t)i;
#pragma unroll
        for (int p = 0; p < kPasses; ++p) atomicAdd(&h[p][(unsigned)(key >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = 0; p < kPasses; ++p)
        if (h[p][threadIdx.x]) atomicAdd(&counts[p * 256 + threadIdx.x], h[p][threadIdx.x]);
}

// Look-back word of (tile, digit): value:40 | state:2 (1 the tile's own count,
// 2 the count up to and including the tile) | pass + 1:8 from bit 48.
constexpr unsigned long long kLbValue = (1ull << 40) - 1;

// One radix pass.  Tiles are taken in the order of a ticket, so every earlier
// tile is running or done and the look-back waits only for work in progress.
// Inside a tile a warp ranks its own 32 * ITEMS consecutive keys (match by
// digit, counters private to the warp), so equal digits keep their order.
template <int ITEMS>
__global__ void __launch_bounds__(kRsBlock) k_rs_pass(const unsigned long long* kin, const uint32_t* vin,
                                                      unsigned long long* kout, uint32_t* vout, long long n, int pass,
                                                      const unsigned* counts, unsigned* ticket,
                                                      unsigned long long* look, int* flags) {
    constexpr int kWarps = kRsBlock / 32;
    __shared__ unsigned cnt[kWarps][256];   // per warp: running digit counts, then the warp's first output position
    __shared__ unsigned tile_sh, wsum[kWarps];
    __shared__ bool failed;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) {
        tile_sh = atomicAdd(ticket, 1u);
        failed = build_failed(flags);
    }
    for (int i = 0; i < kWarps; ++i) cnt[i][t] = 0;
    __syncthreads();
    if (failed) return;
    const unsigned tile = tile_sh;
    const int shift = 8 * pass;
    const long long base = (long long)tile * (kRsBlock * ITEMS) + w * (32 * ITEMS) + lane;
    unsigned long long key[ITEMS];
    unsigned rank[ITEMS];
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const long long i = base + 32 * k;
        key[k] = i < n ? kin[i] : ~0ull;
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const bool valid = base + 32 * k < n;
        const unsigned d = valid ? (unsigned)(key[k] >> shift) & 255u : 256u + lane;   // a lane past the end matches none
        const unsigned m = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(m) - 1;
        unsigned old = 0;
        if (valid && lane == leader) { old = cnt[w][d]; cnt[w][d] = old + __popc(m); }
        old = __shfl_sync(0xffffffffu, old, leader);
        rank[k] = old + __popc(m & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    // thread t owns digit t: the tile's count, then its prefix over the earlier tiles
    unsigned own = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
        const unsigned c = cnt[i][t];
        cnt[i][t] = own;
        own += c;
    }
    volatile unsigned long long* lb = look;
    const unsigned long long tag = (unsigned long long)(pass + 1) << 48;
    lb[(size_t)tile * 256 + t] = tag | ((tile == 0 ? 2ull : 1ull) << 40) | own;
    // first position of the digit: the counts of the smaller digits (block scan)
    const unsigned total = counts[pass * 256 + t];
    unsigned incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    unsigned first = incl - total;
    for (int i = 0; i < w; ++i) first += wsum[i];
    unsigned long long before = 0;
    bool ok = true;
    if (tile > 0) {
        for (long long p = (long long)tile - 1; p >= 0 && ok; --p) {
            unsigned long long v = 0;
            int it = 0;
            do {
                v = lb[(size_t)p * 256 + t];
                ok = (v >> 48) == (tag >> 48);
                if (!ok) {
                    __nanosleep(20);
                    if ((it & 255) == 255 && build_failed(flags)) break;
                }
            } while (!ok && ++it < (1 << 20));
            before += v & kLbValue;
            if ((v >> 40 & 3ull) == 2ull) break;
        }
        if (!ok) flags[1] = 1;   // an earlier tile never reported: the build fails
        else lb[(size_t)tile * 256 + t] = tag | (2ull << 40) | ((before + own) & kLbValue);
    }
#pragma unroll
    for (int i = 0; i < kWarps; ++i) cnt[i][t] += first + (unsigned)before;
    if (__syncthreads_or(!ok)) return;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const long long i = base + 32 * k;
        if (i < n) {
            const unsigned pos = cnt[w][(unsigned)(key[k] >> shift) & 255u] + rank[k];
            if (pos < n) {
                kout[pos] = key[k];
                vout[pos] = vin[i];
            }
        }
    }
}

// The state of the blocks that refine together, zeroed before the kernel.
struct LvState {
    unsigned started;   // blocks that have started
    unsigned members;   // those that take part
    unsigned met;       // their arrivals at barriers so far
};
constexpr int kLvGather = 1 << 10;   // looks at `started` (50 us) before the first block goes on with fewer

// The blocks that refine together: all that start within about 50 us of the first.  They run, so they may
// wait for one another, and a later block leaves.  (A cooperative launch waits until every block has
// room: beside a served session that fills the chip but for a few blocks, until the session ends.)
// Returns this block's number among them, or -1.
__device__ __forceinline__ int join_members(LvState* st, int* members) {
    __shared__ int rank_sh, members_sh;
    if (threadIdx.x == 0) {
        const unsigned r = atomicAdd(&st->started, 1u);
        unsigned n = 0;
        if (r == 0) {
            volatile unsigned* started = &st->started;
            for (int it = 0; it < kLvGather && *started < gridDim.x; ++it) __nanosleep(32);
            n = *started;   // (a block that starts from here on has a number of at least n)
            atomicExch(&st->members, n);
        } else {
            volatile unsigned* m = &st->members;
            for (int it = 0; it < (1 << 22); ++it) {
                n = *m;
                if (n != 0) break;
                __nanosleep(32);
            }
        }
        rank_sh = r < n ? (int)r : -1;
        members_sh = (int)n;
    }
    __syncthreads();
    *members = members_sh;
    return rank_sh;
}

// The members meet: `target` arrivals in all.  The wait is bounded; a block that
// gives up marks the build as failed.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, int* flags) {
    __shared__ int met;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        met = 0;
        for (int it = 0; it < (1 << 22); ++it) {
            if (*(volatile unsigned*)count >= target) { met = 1; break; }
            if ((it & 1023) == 1023 && build_failed(flags)) break;
            __nanosleep(32);
        }
        __threadfence();
        if (!met) flags[1] = 1;
    }
    __syncthreads();
    return met != 0;
}

// First k in [a, b) whose code has an octant digit >= o: three probes a step.
__device__ __forceinline__ int octant_bound(const unsigned long long* codes, int a, int b, int shift, int o) {
    while (a < b) {
        const int q = (b - a) / 4, m1 = a + q, m2 = a + 2 * q, m3 = a + 3 * q;
        const bool l1 = (int)((__ldg(codes + m1) >> shift) & 7ull) < o;
        const bool l2 = (int)((__ldg(codes + m2) >> shift) & 7ull) < o;
        const bool l3 = (int)((__ldg(codes + m3) >> shift) & 7ull) < o;
        if (!l1) b = m1;
        else if (!l2) { a = m1 + 1; b = m2; }
        else if (!l3) { a = m2 + 1; b = m3; }
        else a = m3 + 1;
    }
    return a;
}

// Refinement of every level.  A member block owns a contiguous range of the level's
// cells, 8 lanes to a cell (one per octant): first the octant boundaries and the
// block's child count, then, after a barrier, the children from the prefix over
// the blocks.
constexpr int kLvBlock = 256;

__global__ void __launch_bounds__(kLvBlock) k_levels(const unsigned long long* codes, int4* info, Dbl4* geom, int4* lat,
                                                     int* lstart, const double* box, int* bounds, int leaf, int cap,
                                                     int* block_sums, LvState* state, int* flags) {
    __shared__ int red[kLvBlock / 32], total_sh, base_sh;
    const int t = threadIdx.x, lane = t & 31, o = t & 7, grp = t >> 3;
    const unsigned gshift = (unsigned)(lane & ~7);
    if (build_failed(flags)) return;
    int members;
    const int rank = join_members(state, &members);
    if (rank < 0) return;
    unsigned* barrier = &state->met;
    unsigned meet = 0;
    int l = 0;
    for (; l < kMaxLevel; ++l) {
        const int lo = __ldcg(lstart + l), hi = __ldcg(lstart + l + 1);
        if (lo == hi) break;
        const int per = (hi - lo + members - 1) / members;
        const int c0 = min(hi, lo + rank * per), c1 = min(hi, c0 + per);
        const int shift = 3 * (20 - l);
        int mine = 0;   // children counted by this group (on its lane 0)
        for (int c = c0 + grp; c - grp < c1; c += kLvBlock / 8) {
            int b0 = 0, b1 = 0;
            if (c < c1) {
                const int4 in = __ldcg(info + c);
                if (in.y > leaf) {
                    b0 = o ? octant_bound(codes, in.x, in.x + in.y, shift, o) : in.x;
                    b1 = in.x + in.y;   // the last octant's end
                }
            }
            const int next = __shfl_down_sync(0xffffffffu, b0, 1, 8);
            if (o < 7) b1 = next;
            if (c < c1) {
                bounds[9 * (size_t)(c - lo) + o] = b0;
                if (o == 7) bounds[9 * (size_t)(c - lo) + 8] = b1;
            }
            const unsigned m = (__ballot_sync(0xffffffffu, b1 > b0) >> gshift) & 255u;
            if (o == 0) mine += __popc(m);
        }
        const int ws = (int)__reduce_add_sync(0xffffffffu, (unsigned)mine);
        if (lane == 0) red[t >> 5] = ws;
        __syncthreads();
        if (t == 0) {
            int s = 0;
            for (int i = 0; i < kLvBlock / 32; ++i) s += red[i];
            __stcg(block_sums + rank, s);
        }
        if (!grid_barrier(barrier, ++meet * (unsigned)members, flags)) return;
        // children before this block's, and in all
        int before = 0, all = 0;
        for (int i = t; i < members; i += kLvBlock) {
            const int v = __ldcg(block_sums + i);
            all += v;
            if (i < rank) before += v;
        }
        before = (int)__reduce_add_sync(0xffffffffu, (unsigned)before);
        all = (int)__reduce_add_sync(0xffffffffu, (unsigned)all);
        if (t == 0) { total_sh = 0; base_sh = 0; }
        __syncthreads();
        if (lane == 0) { atomicAdd(&total_sh, all); atomicAdd(&base_sh, before); }
        __syncthreads();
        if (total_sh > cap - hi) {   // the same decision in every block
            if (rank == 0 && t == 0) flags[0] = 1;
            return;
        }
        if (rank == 0 && t == 0) __stcg(lstart + l + 2, hi + total_sh);
        const int cl = l + 1;
        const double cell = __ddiv_rn(box[3], (double)(1ull << cl));
        const double half = __dmul_rn(cell, 0.5);
        const int cshift = 3 * (21 - cl), sh = kMaxLevel - cl;
        int next_child = hi + base_sh;
        for (int c = c0 + grp; c - grp < c1; c += kLvBlock / 8) {
            int b0 = 0, b1 = 0;
            if (c < c1) {
                b0 = bounds[9 * (size_t)(c - lo) + o];
                b1 = bounds[9 * (size_t)(c - lo) + o + 1];
            }
            const unsigned m = (__ballot_sync(0xffffffffu, b1 > b0) >> gshift) & 255u;
            const int nch = __popc(m);
            // exclusive prefix of nch over the 32 cells of this round
            int excl = 0, warp_total = 0;
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int v = __shfl_sync(0xffffffffu, nch, 8 * g);
                if (g < (lane >> 3)) excl += v;
                warp_total += v;
            }
            __syncthreads();
            if (lane == 0) red[t >> 5] = warp_total;
            __syncthreads();
            int round_total = 0;
            for (int i = 0; i < kLvBlock / 32; ++i) {
                if (i < (t >> 5)) excl += red[i];
                round_total += red[i];
            }
            const int cf = next_child + excl;
            next_child += round_total;
            if (nch > 0 && o == 0) {
                int4 in = __ldcg(info + c);
                in.z = cf;
                in.w = (l << 8) | nch;
                __stcg(info + c, in);
            }
            if (b1 > b0) {
                const int ch = cf + __popc(m & ((1u << o) - 1u));
                const unsigned long long pre = __ldg(codes + b0) >> cshift;
                const unsigned long long jx = compact21(pre), jy = compact21(pre >> 1), jz = compact21(pre >> 2);
                lat[ch] = make_int4((int)((2 * jx + 1) << sh), (int)((2 * jy + 1) << sh), (int)((2 * jz + 1) << sh), cl);
                geom[ch] = make_dbl4(__dadd_rn(box[0], __dmul_rn(__dadd_rn((double)jx, 0.5), cell)),
                                     __dadd_rn(box[1], __dmul_rn(__dadd_rn((double)jy, 0.5), cell)),
                                     __dadd_rn(box[2], __dmul_rn(__dadd_rn((double)jz, 0.5), cell)), half);
                __stcg(info + ch, make_int4(b0, b1 - b0, -1, cl << 8));
            }
        }
        if (!grid_barrier(barrier, ++meet * (unsigned)members, flags)) return;
    }
    // level l is empty (or past the deepest): the start entries after it equal its own
    if (rank == 0 && l < kMaxLevel) {
        const int v = __ldcg(lstart + l);
        for (int k = l + 2 + t; k <= kMaxLevel + 1; k += kLvBlock) lstart[k] = v;
    }
}

// (also the largest |charge| to 20 bits, in box[5]: the high words of non-negative doubles keep their order)
__global__ void k_gather(const double* pos, const double* q, const uint32_t* order, long long n, Dbl4* pts, int* flags,
                         double* box) {
    unsigned qm = 0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const uint32_t i = order[k];
        if (i >= n) { flags[1] = 1; continue; }   // a sort that gave up leaves entries unwritten: any number
        pts[k] = make_dbl4(pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2], q[i]);
        qm = max(qm, (unsigned)__double2hiint(q[i]) & 0x7FFFFFFFu);
    }
    __shared__ unsigned block_max;
    if (threadIdx.x == 0) block_max = 0;
    __syncthreads();
    qm = __reduce_max_sync(0xffffffffu, qm);
    if ((threadIdx.x & 31) == 0) atomicMax(&block_max, qm);
    __syncthreads();
    unsigned* top = reinterpret_cast<unsigned*>(box + 5) + 1;
    if (threadIdx.x == 0 && block_max > *(volatile unsigned*)top) atomicMax(top, block_max);
}

// One warp per cell: leaf points relative to the leaf centre, in FP32.
__global__ void k_leaf_local(const Dbl4* pts, const Dbl4* geom, const int4* info, int n_cells, float4* ploc) {
    const int lane = threadIdx.x & 31;
    const int warp = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)(((long long)gridDim.x * blockDim.x) >> 5);
    for (int c = warp; c < n_cells; c += nw) {
        const int4 in = info[c];
        if (in.z >= 0) continue;
        const Dbl4 g = geom[c];
        for (int k = in.x + lane; k < in.x + in.y; k += 32) {
            const Dbl4 p = pts[k];
            ploc[k] = make_float4((float)(p.x - g.x), (float)(p.y - g.y), (float)(p.z - g.z), (float)p.w);
        }
    }
}

int grid_for(long long n, int block, int cap) {
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

// Keys per tile: 4096 from 2^18 points up; a smaller set takes 1024, for enough tiles to fill the chip.
static int rs_items(long long n) { return n >= (1ll << 18) ? 16 : 4; }

// Zeroed scratch of a build: the bounding-box, barrier and ticket counters (64 words), the digit counts of every
// pass, then the look-back words of a pass (tagged with the pass, so one zeroing serves all).
constexpr size_t kRsCounters = 64 * sizeof(unsigned), kRsCounts = kPasses * 256 * sizeof(unsigned);
size_t tree_work_bytes(long long n) {
    const long long tile = kRsBlock * rs_items(n), tiles = (n + tile - 1) / tile;
    return kRsCounters + kRsCounts + 256 * sizeof(unsigned long long) * (size_t)tiles;
}

// Structural check of the cell records before any kernel follows their links:
// flags[1] = 1 on a malformed record; flags[2] = leaves; flags[3] = largest leaf.
// The cell count is read from lstart[kMaxLevel + 1], never above `cap`.
__global__ void k_check_tree(const int4* info, const int* lstart, int cap, long long n, int* flags) {
    const int n_cells = min(lstart[kMaxLevel + 1], cap);
    int bad = 0, leaves = 0, big = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_cells; i += gridDim.x * blockDim.x) {
        const int4 c = info[i];
        const int level = c.w >> 8, nch = c.w & 0xFF;
        bool ok = c.x >= 0 && c.y >= 1 && (long long)c.x + c.y <= n && level >= 0 && level <= kMaxLevel;
        if (c.z >= 0) {
            ok = ok && c.z > i && nch >= 1 && nch <= 8 && (long long)c.z + nch <= n_cells;
            if (ok)
                for (int j = 0; j < nch; ++j) ok = ok && (info[c.z + j].w >> 8) == level + 1;
        } else {
            ok = ok && c.z == -1 && nch == 0;
            if (ok) {
                ++leaves;
                big = max(big, c.y);
            }
        }
        if (!ok) bad = 1;
    }
    bad = __reduce_or_sync(0xffffffffu, (unsigned)bad);
    leaves = (int)__reduce_add_sync(0xffffffffu, (unsigned)leaves);
    big = (int)__reduce_max_sync(0xffffffffu, (unsigned)big);
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicOr(&flags[1], 1);
        if (leaves) atomicAdd(&flags[2], leaves);
        if (big) atomicMax(&flags[3], big);
    }
}

cudaError_t launch_gather(const double* pos, const double* q, const uint32_t* order, long long n, Dbl4* pts, int* flags,
                          double* box, cudaStream_t s) {
    k_gather<<<grid_for(n, 256, 4096), 256, 0, s>>>(pos, q, order, n, pts, flags, box);
    return cudaGetLastError();
}

cudaError_t launch_tree(TreeBufs& b, int sms, cudaStream_t s) {
    const long long n = b.n;
    cudaError_t e = cudaMemsetAsync(b.work, 0, tree_work_bytes(n), s);
    if (e != cudaSuccess) return e;
    unsigned* counters = static_cast<unsigned*>(b.work);   // [0] box, [4..6] LvState, [8 + pass] tile tickets
    unsigned* counts = reinterpret_cast<unsigned*>(static_cast<char*>(b.work) + kRsCounters);
    unsigned long long* look = reinterpret_cast<unsigned long long*>(static_cast<char*>(b.work) + kRsCounters + kRsCounts);
    k_bbox<<<grid_for(n, 256 * 4, kBoxParts), 256, 0, s>>>(b.pos, n, b.bbox_part, counters, b.box, b.geom, b.info, b.lat,
                                                          b.lstart, b.flags);
    k_codes<<<grid_for(n, kRsBlock, 4 * sms), kRsBlock, 0, s>>>(b.pos, n, b.box, b.keys[0], b.vals[0], counts);
    const int items = rs_items(n);
    const unsigned tiles = (unsigned)((n + kRsBlock * items - 1) / (kRsBlock * items));
    int cur = 0;
    for (int pass = 0; pass < kPasses; ++pass) {
        if (items == 16)
            k_rs_pass<16><<<tiles, kRsBlock, 0, s>>>(b.keys[cur], b.vals[cur], b.keys[cur ^ 1], b.vals[cur ^ 1], n, pass,
                                                     counts, counters + 8 + pass, look, b.flags);
        else
            k_rs_pass<4><<<tiles, kRsBlock, 0, s>>>(b.keys[cur], b.vals[cur], b.keys[cur ^ 1], b.vals[cur ^ 1], n, pass,
                                                    counts, counters + 8 + pass, look, b.flags);
        cur ^= 1;
    }
    b.codes = b.keys[cur];
    b.order = b.vals[cur];
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_levels<<<b.refine_blocks, kLvBlock, 0, s>>>(b.codes, b.info, b.geom, b.lat, b.lstart, b.box, b.bounds, b.leaf,
                                                  b.cap_cells, b.block_sums, reinterpret_cast<LvState*>(counters + 4),
                                                  b.flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_gather(b.pos, b.q, b.order, n, b.pts, b.flags, b.box, s)) != cudaSuccess) return e;
    k_check_tree<<<grid_for(b.cap_cells, 256, 1216), 256, 0, s>>>(b.info, b.lstart, b.cap_cells, n, b.flags);
    return cudaGetLastError();
}

cudaError_t launch_leaf_local(const TreeBufs& b, int n_cells, cudaStream_t s) {
    k_leaf_local<<<grid_for((long long)n_cells * 32, 256, 4096), 256, 0, s>>>(b.pts, b.geom, b.info, n_cells, b.ploc);
    return cudaGetLastError();
}

}  // namespace fmm
}  // namespace gtap
