// Leaf evaluation of the FMM (Sec. 6.4.1): P2P sums the near field over the lists
// grouped by target leaf, then L2P adds every point's far field and writes phi.
//
// A leaf's near list is cut into runs of at most `chunk` source leaves, one
// block per run: the lists are very uneven (in a Plummer set of 60,001 points a
// large outer leaf meets thousands of small leaves of the core, and its one
// block ran 0.8 ms after all others had finished), and a small set has fewer
// leaves than the chip has SMs.  A run's sums are added by FP64 atomics to `near`
// (sorted point order, zeroed first); phi is written once, by L2P.
#include <cuda_runtime.h>

#include "fmm_arith.cuh"
#include "fmm_internal.h"

namespace gtap {
namespace fmm {
namespace {

// ---------------------------------------------------------------------------
// Points much closer than their leaf's extent are not resolved by the mixed form's FP32 coordinates
// relative to leaf centres: such a distance is off, or zero for distinct points, and the near sum
// wrong, infinite or NaN.  The near sum of a target that one such pair dominates exceeds what well
// separated points add up to (about half of q_max / h for each of them, h the leaf's half side);
// it is taken again from the FP64 coordinates.  Below the limit a pair with the largest charge is more
// than h / (kCloseSum + near points) apart, and its FP32 distance good to a few 1e-4.
constexpr float kCloseSum = 1024.f;

// The near sum of sorted point `own` of leaf c in FP64, by a warp.  (Points of one leaf at the same place do
// not interact in the mixed form.)
static __device__ __noinline__ double near_fp64(const EvalBufs& e, int c, int own) {
    const int lane = threadIdx.x & 31;
    const Dbl4 p = e.pts[own];
    double sum = 0.0;
    for (int j = e.p2p_off[c]; j < e.p2p_off[c + 1]; ++j) {
        const int4 si = e.info[e.p2p_src[j]];
        for (int k = si.x + lane; k < si.x + si.y; k += 32) {
            const Dbl4 q = e.pts[k];
            const double dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z, r2 = fma(dz, dz, fma(dy, dy, dx * dx));
            if (r2 > 0.0) sum = fma(q.w, rsqrt(r2), sum);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    return sum;
}

// L2P: one block per leaf, one thread per point, nested Horner sums.
constexpr int kL2pBlock = 64;
static_assert(kL2pBlock >= kMaxLeaf, "one thread per point");

template <class R>
__global__ void __launch_bounds__(kL2pBlock, 32) k_l2p(EvalBufs e, const double* near) {
    __shared__ R lsm[n_coef(kMaxOrder)];
    const int c = blockIdx.x;
    const int4 in = e.info[c];
    if (in.z >= 0) return;
    const int p = e.p, nt = e.nt;
    for (int i = threadIdx.x; i < nt; i += kL2pBlock) lsm[i] = (R)e.L[(size_t)c * nt + i];
    __syncthreads();
    const Dbl4 g = e.geom[c];
    const int i = threadIdx.x, k = in.x + min(i, in.y - 1);
    if ((i & ~31) >= in.y) return;   // (a warp without a point; lanes past the last repeat it)
    R x, y, z;
    if constexpr (sizeof(R) == 4) {
        const float4 pl = e.ploc[k];
        x = pl.x; y = pl.y; z = pl.z;
    } else {
        const Dbl4 pt = e.pts[k];
        x = __dsub_rn(pt.x, g.x); y = __dsub_rn(pt.y, g.y); z = __dsub_rn(pt.z, g.z);
    }
    R sx = 0;
    for (int a = p; a >= 0; --a) {
        R sy = 0;
        for (int b = p - a; b >= 0; --b) {
            R sz = 0;
            for (int cc = p - a - b; cc >= 0; --cc) sz = sz * z + lsm[cidx(a, b, cc)];
            sy = sy * y + sz;
        }
        sx = sx * x + sy;
    }
    double nk = near[k];
    if constexpr (sizeof(R) == 4) {
        // the limit of a normal sum, compared by the double's high word
        const int entries = e.p2p_off[c + 1] - e.p2p_off[c];
        const float limit = (kCloseSum + (float)kMaxLeaf * (float)entries) * e.close_unit * (float)(1 << (in.w >> 8));
        const unsigned limit_hi = (__float_as_uint(limit) >> 3) + (896u << 20);
        for (unsigned m = __ballot_sync(0xffffffffu, ((unsigned)__double2hiint(nk) & 0x7FFFFFFFu) > limit_hi); m != 0u; m &= m - 1u) {
            const int o = __ffs((int)m) - 1;
            const double v = near_fp64(e, c, __shfl_sync(0xffffffffu, k, o));
            if ((i & 31) == o) nk = v;
        }
    }
    if (i < in.y) e.phi[e.order[k]] = nk + (double)sx;
}

// ---------------------------------------------------------------------------
// Runs of the near lists: {leaf, first entry, last entry}.
__global__ void k_p2p_runs(const int4* info, const int* off, int n_cells, int chunk, int4* runs, int* n_runs) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n_cells || info[c].z >= 0) return;
    const int s0 = off[c], s1 = off[c + 1];
    if (s0 == s1) return;
    int r = atomicAdd(n_runs, (s1 - s0 + chunk - 1) / chunk);
    for (int s = s0; s < s1; s += chunk) runs[r++] = make_int4(c, s, min(s1, s + chunk), 0);
}

// Packed FP32 pairs (two lanes of a 64-bit register): one f32x2 instruction
// does the work of two FP32 ones.
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
    return (unsigned long long)__float_as_uint(lo) | ((unsigned long long)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float lo_f32(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi_f32(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ unsigned long long sub_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// 1/sqrt(x), the hardware approximation; infinite for zero and subnormal x (see near_fp64)
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int kP2pBlock = 128;

constexpr int kSrcBatch = 1024;   // source points staged at once, from up to 32 source leaves
constexpr int kTargets = 2;         // target points per thread

// Mixed form, one block per run.  Threads are (group of kTargets target points,
// source part): a thread keeps its targets in registers and walks every
// parts-th pair of source points, so a pair's two 16-byte shared loads serve
// 2 kTargets interactions, and the finer split of the 128 threads leaves fewer
// of them without work than one target per thread did.  Bound by FP32 issue (68 %
// of it used) before the reciprocal square roots (16 a cycle and SM: 1.05 of the
// 1.89 ms at N = 2^20 uniform).  Leaf evaluation, one target per thread and one
// block per list -> this: 2^20 uniform 2.31 -> 1.89 ms, Plummer 2.53 -> 2.26 ms,
// Plummer 60,001 0.86 -> 0.24 ms.  Four targets per thread measure the same; one
// warp per run without the staging in the target's frame measured 2.8 ms.
__global__ void __launch_bounds__(kP2pBlock) k_p2p_mixed(EvalBufs e, const int4* runs, const int* n_runs, double* near) {
    __shared__ __align__(16) float sp[4 * kSrcBatch];   // pair records {x0 x1 y0 y1 z0 z1 q0 q1}
    __shared__ float red[kTargets][kP2pBlock];
    __shared__ int bpre[33], bfirst[32], bself;
    __shared__ float boff[32][3];
    if ((int)blockIdx.x >= *n_runs) return;
    const int t = threadIdx.x, lane = t & 31;
    const int4 run = runs[blockIdx.x];
    const int c = run.x;
    const int4 in = e.info[c];
    const Dbl4 g = e.geom[c];
    const int count = in.y, slots = (count + kTargets - 1) / kTargets, parts = kP2pBlock / slots;
    const int part = t / slots, slot = t - part * slots;
    const bool active = part < parts;
    // a target past the last repeats it; its sum is not used
    float4 tg[kTargets];
#pragma unroll
    for (int h = 0; h < kTargets; ++h) tg[h] = e.ploc[in.x + min(slot + h * slots, count - 1)];
    Acc<float> acc[kTargets];
    const ulonglong2* pr = reinterpret_cast<const ulonglong2*>(sp);
    for (int cur = run.y; cur < run.z;) {
        __syncthreads();
        if (t < 32) {
            const int j = cur + lane;
            int cnt = 0, first = 0;
            bool self = false;
            Dbl4 gs = make_dbl4(0, 0, 0, 0);
            if (j < run.z) {
                const int sc = e.p2p_src[j];
                const int4 si = e.info[sc];
                self = sc == c;
                cnt = self ? 0 : si.y;   // the leaf itself has its own pass
                first = si.x;
                gs = e.geom[sc];
            }
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            // the fitting entries are a prefix of the lanes; a leaf holds <= 64 points
            const int nfit = max(1, __popc(__ballot_sync(0xffffffffu, j < run.z && incl <= kSrcBatch)));
            const unsigned sm = __ballot_sync(0xffffffffu, self && lane < nfit);
            bpre[lane + 1] = incl;
            bfirst[lane] = first;
            boff[lane][0] = (float)__dsub_rn(gs.x, g.x);
            boff[lane][1] = (float)__dsub_rn(gs.y, g.y);
            boff[lane][2] = (float)__dsub_rn(gs.z, g.z);
            if (lane == 0) { bpre[0] = 0; bself = nfit | (sm ? 64 : 0); }
        }
        __syncthreads();
        const int nfit = bself & 63;
        const bool self = (bself & 64) != 0;
        const int total = bpre[nfit];
        // the source points in the target leaf's frame, as pair records
        for (int i = t, s = 0; i < total; i += kP2pBlock) {
            while (bpre[s + 1] <= i) ++s;
            const float4 l = e.ploc[bfirst[s] + i - bpre[s]];
            float* d = sp + i / 2 * 8 + (i & 1);
            d[0] = l.x + boff[s][0]; d[2] = l.y + boff[s][1]; d[4] = l.z + boff[s][2]; d[6] = l.w;
        }
        if (t == 0 && (total & 1)) {   // an odd tail is padded with a far, chargeless point
            float* d = sp + total / 2 * 8 + 1;
            d[0] = d[2] = d[4] = 1e18f;
            d[6] = 0.f;
        }
        __syncthreads();
        if (active) {
            // each batch is summed plainly and added to the compensated totals
            const int npairs = (total + 1) >> 1;
            unsigned long long x[kTargets], y[kTargets], z[kTargets], sum[kTargets];
#pragma unroll
            for (int h = 0; h < kTargets; ++h) {
                x[h] = pack_f32x2(tg[h].x, tg[h].x);
                y[h] = pack_f32x2(tg[h].y, tg[h].y);
                z[h] = pack_f32x2(tg[h].z, tg[h].z);
                sum[h] = 0ull;
            }
#pragma unroll 2
            for (int m = part; m < npairs; m += parts) {
                const ulonglong2 xy = pr[2 * m], zq = pr[2 * m + 1];
#pragma unroll
                for (int h = 0; h < kTargets; ++h) {
                    const unsigned long long dx = sub_f32x2(x[h], xy.x), dy = sub_f32x2(y[h], xy.y), dz = sub_f32x2(z[h], zq.x);
                    const unsigned long long r2 = fma_f32x2(dz, dz, fma_f32x2(dy, dy, mul_f32x2(dx, dx)));
                    sum[h] = fma_f32x2(zq.y, pack_f32x2(rsqrt_ftz(lo_f32(r2)), rsqrt_ftz(hi_f32(r2))), sum[h]);
                }
            }
#pragma unroll
            for (int h = 0; h < kTargets; ++h) acc[h].add(lo_f32(sum[h]) + hi_f32(sum[h]));
        }
        if (self && active) {
            // the leaf's own points: a target's own copy has exactly the same local
            // coordinates (r^2 == 0), and only this pass tests for it
            float own[kTargets] = {};
            for (int j = part; j < count; j += parts) {
                const float4 s = e.ploc[in.x + j];
#pragma unroll
                for (int h = 0; h < kTargets; ++h) {
                    const float dx = tg[h].x - s.x, dy = tg[h].y - s.y, dz = tg[h].z - s.z;
                    const float r2 = dx * dx + dy * dy + dz * dz;
                    own[h] += (r2 > 0.f) ? s.w * rsqrtf(r2) : 0.f;
                }
            }
#pragma unroll
            for (int h = 0; h < kTargets; ++h) acc[h].add(own[h]);
        }
        cur += nfit;
    }
#pragma unroll
    for (int h = 0; h < kTargets; ++h) red[h][t] = Ops<float>::sub(acc[h].s, acc[h].c);
    __syncthreads();
    // one thread per target sums the parts
    for (int i = t; i < count; i += kP2pBlock) {
        const int h = i / slots, sl = i - h * slots;
        Acc<float> tot;
        for (int q = 0; q < parts; ++q) tot.add(red[h][q * slots + sl]);
        atomicAdd(&near[in.x + i], (double)tot.s - (double)tot.c);
    }
}

// 1/sqrt(x) in FP64 from the FP32 approximation and one step of Householder's
// third-order iteration,  e = 1 - x y^2,  y (1 + e/2 + 3 e^2 / 8)  (the first
// terms of (1 - e)^(-1/2); the next is below 2^-63 of y): 5 FP64 operations.
// The FP64 pipe (2 lanes a cycle and SM) is what the P2P waits for, so the
// conversions to and from FP32 are integer shifts.  x outside the normal FP32
// range takes the library function.
__device__ __forceinline__ double rsqrt_fp64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    // biased exponent in [897, 1150]: x >= 2^-126 and x < 2^128
    if (hi - (897u << 20) >= (254u << 20)) return rsqrt(x);
    const unsigned f = __float_as_uint(rsqrt_ftz(__uint_as_float(__funnelshift_l(lo, hi - (896u << 20), 3))));
    const double y = __hiloint2double((int)((f >> 3) + (896u << 20)), (int)(f << 29));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// FP64 form, one block per run, by symmetry: for leaves A < B the reciprocal
// distance of a point pair serves both sums, 13 FP64 operations for two
// interactions instead of 24.  (The near relation is symmetric: the list of A
// names B whenever the list of B names A, and the entry with B < A is skipped.)
// Groups of kGroup lanes hold as many targets of A; the points of all the run's
// leaves form one sequence, cut into equal parts, and a group walks its part
// with lane l at position s + l - (kGroup - 1) in step s.  The running sum of a
// source point moves down one lane a step, so no two lanes add to one point and
// lane 0 adds the finished sum to `near`.  One sequence instead of a loop per
// leaf, and groups of 4 rather than 8, keep the lanes of a warp in step.
// Points are read from L1/L2: the FP64 pipe takes ~200 cycles a step and warp.
// Leaf evaluation, one-sided sums -> this: N = 2^20 uniform 128 -> 73 ms, Plummer
// 115 -> 69 ms, Plummer 60,001 19.2 -> 6.7 ms.
constexpr int kGroup = 4;
constexpr int kMaxRun64 = 64;     // source leaves in one run, at most

__global__ void __launch_bounds__(kP2pBlock) k_p2p_fp64(EvalBufs e, const int4* runs, const int* n_runs, double* near) {
    __shared__ int pre[kMaxRun64 + 1], first[kMaxRun64], own;
    if ((int)blockIdx.x >= *n_runs) return;
    const int t = threadIdx.x, lane = t & 31, gl = lane % kGroup, grp = t / kGroup;
    const unsigned gmask = ((1u << kGroup) - 1u) << (lane - gl);
    const int4 run = runs[blockIdx.x];
    const int c = run.x, m = run.z - run.y;
    const int4 in = e.info[c];
    if (t == 0) { own = 0; pre[0] = 0; }
    __syncthreads();
    if (t < kMaxRun64) {
        int n = 0;
        if (t < m) {
            const int sc = e.p2p_src[run.y + t];
            const int4 si = e.info[sc];
            first[t] = si.x;
            n = sc > c ? si.y : 0;
            if (sc == c) own = 1;
        }
        pre[t + 1] = n;
    }
    __syncthreads();
    if (t < 32) {   // inclusive prefix of the 64 counts, two per lane
        const int n0 = pre[2 * t + 1], n1 = pre[2 * t + 2];
        int incl = n0 + n1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncwarp();
        pre[2 * t + 1] = incl - n1;
        pre[2 * t + 2] = incl;
    }
    __syncthreads();
    const int total = pre[kMaxRun64];
    const int count = in.y, tiles = (count + kGroup - 1) / kGroup, slots = (kP2pBlock / kGroup) / tiles;
    const int tile = grp % tiles, slot = grp / tiles;
    if (slot >= slots) return;
    const int i = tile * kGroup + gl;
    const bool target = i < count;
    const int ki = in.x + min(i, count - 1);
    const Dbl4 pt = e.pts[ki];
    double acc = 0.0;
    if (own) {
        for (int k = slot; k < count; k += slots) {
            if (in.x + k == ki) continue;
            const Dbl4 s = e.pts[in.x + k];
            const double dx = pt.x - s.x, dy = pt.y - s.y, dz = pt.z - s.z;
            acc = fma(s.w, rsqrt_fp64(fma(dz, dz, fma(dy, dy, dx * dx))), acc);
        }
        __syncwarp(gmask);
    }
    const int p0 = (int)((long long)total * slot / slots), p1 = (int)((long long)total * (slot + 1) / slots);
    if (p0 < p1) {
        int lo = 0, hi = m - 1;   // the last leaf that starts at or before p0 (it holds p0)
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= p0) lo = mid; else hi = mid - 1;
        }
        int leaf = lo, pos = p0 + gl - (kGroup - 1);
        double mine = 0.0;        // the running sum of source point `pos`
        for (; pos - gl < p1; ++pos) {
            const bool valid = pos >= p0 && pos < p1;
            const int at = max(p0, min(pos, p1 - 1));
            while (at >= pre[leaf + 1]) ++leaf;
            const int k = first[leaf] + at - pre[leaf];
            const Dbl4 p = e.pts[k];
            const double dx = pt.x - p.x, dy = pt.y - p.y, dz = pt.z - p.z;
            const double ir = rsqrt_fp64(fma(dz, dz, fma(dy, dy, dx * dx)));
            // (selected, not weighted by zero: an infinite charge or 1/r stays where it belongs)
            acc = valid ? fma(p.w, ir, acc) : acc;
            mine = target ? fma(pt.w, ir, mine) : mine;
            if (gl == 0 && valid) atomicAdd(&near[k], mine);
            const double down = __shfl_down_sync(gmask, mine, 1, kGroup);
            mine = (gl == kGroup - 1 || pos + 1 < p0) ? 0.0 : down;
        }
    }
    if (target) atomicAdd(&near[ki], acc);
}

}  // namespace

// Source leaves per run: about eight runs for each SM, but at least 16, and at
// most 256 in the mixed form (a typical whole list; a split one repeats its
// set-up) or kMaxRun64 in FP64 (where the set-up is nothing beside the arithmetic).
static int p2p_chunk(bool mixed, long long n_p2p, int sms) {
    const long long want = n_p2p / (8ll * (sms > 0 ? sms : 1)), most = mixed ? 256 : kMaxRun64;
    return (int)(want < 16 ? 16 : want > most ? most : want);
}

// Scratch: the run count (16 bytes), the near sums of n points, the runs.
static size_t near_bytes(long long n) { return ((size_t)n * sizeof(double) + 15) / 16 * 16; }

size_t p2p_scratch_bytes(bool mixed, long long n, long long n_p2p, int n_leaves, int sms) {
    return 16 + near_bytes(n) + sizeof(int4) * (size_t)(n_p2p / p2p_chunk(mixed, n_p2p, sms) + n_leaves + 1);
}

cudaError_t launch_leaf_eval(const EvalBufs& e, bool mixed, long long n_p2p, int n_leaves, int sms, void* scratch,
                             cudaStream_t s) {
    const int chunk = p2p_chunk(mixed, n_p2p, sms);
    char* base = static_cast<char*>(scratch);
    int* n_runs = reinterpret_cast<int*>(base);
    double* near = reinterpret_cast<double*>(base + 16);
    int4* runs = reinterpret_cast<int4*>(base + 16 + near_bytes(e.n));
    cudaError_t err = cudaMemsetAsync(base, 0, 16 + near_bytes(e.n), s);
    if (err != cudaSuccess) return err;
    k_p2p_runs<<<(e.n_cells + 127) / 128, 128, 0, s>>>(e.info, e.p2p_off, e.n_cells, chunk, runs, n_runs);
    const unsigned grid = (unsigned)(n_p2p / chunk + n_leaves);   // at least the number of runs
    if (mixed) {
        k_p2p_mixed<<<grid, kP2pBlock, 0, s>>>(e, runs, n_runs, near);
        k_l2p<float><<<e.n_cells, kL2pBlock, 0, s>>>(e, near);
    } else {
        k_p2p_fp64<<<grid, kP2pBlock, 0, s>>>(e, runs, n_runs, near);
        k_l2p<double><<<e.n_cells, kL2pBlock, 0, s>>>(e, near);
    }
    return cudaGetLastError();
}

}  // namespace fmm
}  // namespace gtap
