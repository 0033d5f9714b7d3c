// Data-parallel FMM kernels around the traversal (Sec. 6.4.1): upward pass
// (P2M at leaves, M2M level by level), M2L over the interaction list grouped
// by target cell, and downward pass (L2L level by level); the leaf kernels
// (L2P and P2P) are in fmm_leaf.cu.  Cartesian Taylor expansions of total
// order p about the cell centres:
//   P2M  M_a  = sum_j q_j (x_j - c)^a
//   M2M  M_a(c) += sum_{b <= a} C(a, b) (c' - c)^(a-b) M_b(c')      (child c')
//   M2L  L_b(A) += sum_{|a|+|b| <= p} (-1)^|a| C(a+b, b) T_{a+b}(c_A - c_B) M_a(B)
//   L2L  L_g(c') += sum_{b >= g} C(b, g) (c' - c)^(b-g) L_b(c)       (child c')
//   L2P  phi_i  = sum_b L_b (x_i - c)^b
//   P2P  phi_i += sum_{j != i} q_j / |x_i - x_j|
// with T_n = d^n(1/r)/n! from the recurrence in fmm_internal.h.  R is the
// arithmetic type: double, or float for the mixed form, where the per-target
// sums of M2L and P2P are compensated (Kahan) and the translations into the
// top levels stay in double.
#include <cuda_runtime.h>

#include <algorithm>

#include "fmm_arith.cuh"
#include "fmm_internal.h"
#include "scan.cuh"

namespace gtap {
namespace fmm {
namespace {

// M2M and L2L between a cell and its children work in the scaled variables
// M_a / a!, b! L_b and d^n / n!, where a shift is a plain correlation: one
// multiply-add per term, no binomials.  One warp per child, a lane per output
// coefficient; the displacement's scaled monomials come from three short power
// tables.  One thread per coefficient for all eight children, binomials read
// with every term and the monomials built by one thread per child took 25 us a
// level, whatever its size; a small set's passes are bound by that chain.
constexpr int kShiftBlock = 256;   // 8 warps

// Scaled powers d_x^k / k! of every child's displacement: pw[child][axis][k].
template <class R>
__device__ __forceinline__ void shift_powers(const EvalBufs& e, const Dbl4& g, int cf, int nch, R* pw) {
    const int t = threadIdx.x, j = t / 3, axis = t % 3, p1 = kMaxOrder + 1;
    if (j < nch) {
        const Dbl4 gc = e.geom[cf + j];
        const R d = (R)(axis == 0 ? __dsub_rn(gc.x, g.x) : axis == 1 ? __dsub_rn(gc.y, g.y) : __dsub_rn(gc.z, g.z));
        R v = 1;
        pw[t * p1] = v;
        for (int k = 1; k <= e.p; ++k) {
            v = v * d / (R)k;
            pw[t * p1 + k] = v;
        }
    }
}

// Warp j fills mono[i] = d^n / n! of child j for every coefficient.
template <class R>
__device__ __forceinline__ void shift_monomials(const EvalBufs& e, const R* pw, R* mono) {
    const int lane = threadIdx.x & 31, p1 = kMaxOrder + 1;
    const R* w = pw + 3 * p1 * (threadIdx.x >> 5);
    for (int i = lane; i < e.nt; i += 32) {
        const short3 n = e.tab.mi[i];
        mono[i] = w[n.x] * w[p1 + n.y] * w[2 * p1 + n.z];
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// P2M: one block per leaf.  Point powers in shared memory, one thread per
// coefficient summing over the leaf's points in order.
template <class R>
__global__ void k_p2m(EvalBufs e) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int p = e.p, nt = e.nt, p1 = p + 1;
    R* pw = reinterpret_cast<R*>(sm_raw);              // [kMaxLeaf][3][p1]
    R* qv = pw + kMaxLeaf * 3 * p1;                    // [kMaxLeaf]
    short3* mi = reinterpret_cast<short3*>(qv + kMaxLeaf);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) mi[i] = e.tab.mi[i];
    for (int c = blockIdx.x; c < e.n_cells; c += gridDim.x) {
        const int4 in = e.info[c];
        if (in.z >= 0) continue;
        const Dbl4 g = e.geom[c];
        __syncthreads();
        for (int k = threadIdx.x; k < in.y; k += blockDim.x) {
            R d[3];
            if constexpr (sizeof(R) == 4) {
                const float4 pl = e.ploc[in.x + k];
                d[0] = pl.x; d[1] = pl.y; d[2] = pl.z;
                qv[k] = pl.w;
            } else {
                const Dbl4 pt = e.pts[in.x + k];
                d[0] = __dsub_rn(pt.x, g.x); d[1] = __dsub_rn(pt.y, g.y); d[2] = __dsub_rn(pt.z, g.z);
                qv[k] = pt.w;
            }
            for (int a = 0; a < 3; ++a) {
                R v = 1;
                pw[(k * 3 + a) * p1] = v;
                for (int j = 1; j <= p; ++j) { v = Ops<R>::mul(v, d[a]); pw[(k * 3 + a) * p1 + j] = v; }
            }
        }
        __syncthreads();
        for (int a = threadIdx.x; a < nt; a += blockDim.x) {
            const short3 m = mi[a];
            Acc<R> acc;
            for (int k = 0; k < in.y; ++k) {
                const R t = Ops<R>::mul(Ops<R>::mul(Ops<R>::mul(qv[k], pw[(k * 3) * p1 + m.x]), pw[(k * 3 + 1) * p1 + m.y]),
                                        pw[(k * 3 + 2) * p1 + m.z]);
                acc.add(t);
            }
            e.M[(size_t)c * nt + a] = (double)acc.s - (double)acc.c;
        }
    }
}

// M2M for the parents of one level: one block per cell, leaves leave at once.
template <class R>
__global__ void __launch_bounds__(kShiftBlock) k_m2m(EvalBufs e, int lo) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int nt = e.nt, c = lo + (int)blockIdx.x, t = threadIdx.x, lane = t & 31, j = t >> 5;
    const int4 in = e.info[c];
    if (in.z < 0) return;
    const int nch = in.w & 0xFF, cf = in.z;
    R* pw = reinterpret_cast<R*>(sm_raw);              // [8][3][kMaxOrder + 1]
    R* mono = pw + 24 * (kMaxOrder + 1) + j * nt;      // [8][nt], this warp's row
    R* mc = pw + 24 * (kMaxOrder + 1) + (8 + j) * nt;  // [8][nt]
    R* part = pw + 24 * (kMaxOrder + 1) + 16 * nt;     // [8][nt]
    shift_powers(e, e.geom[c], cf, nch, pw);
    if (j < nch)
        for (int i = lane; i < nt; i += 32) mc[i] = (R)(e.M[(size_t)(cf + j) * nt + i] * __ldg(e.tab.lscale + i));
    __syncthreads();
    if (j < nch) {
        shift_monomials(e, pw, mono);
        for (int a = lane; a < nt; a += 32) {
            const int t1 = __ldg(e.tab.m2m_off + a + 1);
            R s = 0;
#pragma unroll 4
            for (int i = __ldg(e.tab.m2m_off + a); i < t1; ++i) {
                const unsigned u = __ldg(e.tab.m2m_terms + i);
                s += mono[u >> 16] * mc[u & 0xFFFFu];
            }
            part[j * nt + a] = s;
        }
    }
    __syncthreads();
    for (int a = t; a < nt; a += kShiftBlock) {
        Acc<R> acc;
        for (int k = 0; k < nch; ++k) acc.add(part[k * nt + a]);
        e.M[(size_t)c * nt + a] = ((double)acc.s - (double)acc.c) * __ldg(e.tab.fact + a);
    }
}

// ---------------------------------------------------------------------------
// M2L: one block per target cell; sources in batches of kSB.  The Taylor
// coefficients of every source displacement are built degree by degree in
// shared memory, then each thread owns one item (a run of <= kM2lChunk terms
// of one output coefficient) and accumulates it over all sources.
constexpr int kSB = 8;

template <class R>
__global__ void k_m2l(EvalBufs e) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int p = e.p, nt = e.nt;
    R* T = reinterpret_cast<R*>(sm_raw);               // [kSB][nt]
    R* Ms = T + kSB * nt;                              // [kSB][nt]
    R* dv = Ms + kSB * nt;                             // [kSB][4]: dx, dy, dz, 1/r^2
    R* accs = dv + kSB * 4;                            // [n_items]
    R* c1 = accs + e.tab.n_m2l_items;                  // [p + 1]
    R* c2 = c1 + (p + 1);
    DerivEntry* der = reinterpret_cast<DerivEntry*>(c2 + (p + 1) + ((p + 1) & 1) + 2);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) der[i] = e.tab.deriv[i];
    for (int k = threadIdx.x; k <= p; k += blockDim.x) {
        c1[k] = k ? (R)(2.0 * k - 1.0) / (R)k : (R)0;
        c2[k] = k ? (R)(k - 1.0) / (R)k : (R)0;
    }
    // this thread's item, its terms cached in registers
    const int it = threadIdx.x;
    const bool has_item = it < e.tab.n_m2l_items;
    int len = 0;
    R cf[kM2lChunk];
    uint8_t ta[kM2lChunk], tb[kM2lChunk];
    if (has_item) {
        const ItemEntry ie = e.tab.m2l_items[it];
        len = ie.len;
#pragma unroll
        for (int j = 0; j < kM2lChunk; ++j) {
            if (j < len) {
                const TermEntry te = e.tab.m2l_terms[ie.first + j];
                cf[j] = Ops<R>::coef(te);
                ta[j] = te.a;
                tb[j] = te.b;
            } else {
                cf[j] = 0; ta[j] = 0; tb[j] = 0;
            }
        }
    }
    for (int c = blockIdx.x; c < e.n_cells; c += gridDim.x) {
        const int s0 = e.m2l_off[c], s1 = e.m2l_off[c + 1];
        if (s0 == s1) continue;
        const Dbl4 g = e.geom[c];
        Acc<R> acc;
        for (int b0 = s0; b0 < s1; b0 += kSB) {
            const int nb = min(kSB, s1 - b0);
            __syncthreads();
            for (int i = threadIdx.x; i < nb * nt; i += blockDim.x) {
                const int s = i / nt, a = i - s * nt;
                Ms[i] = (R)e.M[(size_t)e.m2l_src[b0 + s] * nt + a];
            }
            if ((int)threadIdx.x < nb) {
                const Dbl4 gs = e.geom[e.m2l_src[b0 + threadIdx.x]];
                const R x = (R)__dsub_rn(g.x, gs.x), y = (R)__dsub_rn(g.y, gs.y), z = (R)__dsub_rn(g.z, gs.z);
                const R r2 = x * x + y * y + z * z;
                R* d = dv + threadIdx.x * 4;
                d[0] = x; d[1] = y; d[2] = z; d[3] = (R)1 / r2;
                T[threadIdx.x * nt] = Ops<R>::rsq(r2);
            }
            __syncthreads();
            for (int k = 1; k <= p; ++k) {
                const int i0 = n_coef(k - 1), cnt = n_coef(k) - i0;
                for (int w = threadIdx.x; w < nb * cnt; w += blockDim.x) {
                    const int s = w / cnt, i = i0 + (w - s * cnt);
                    const DerivEntry de = der[i];
                    const R* Ts = T + s * nt;
                    const R* d = dv + s * 4;
                    R s1v = 0, s2v = 0;
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (de.e1[q] >= 0) s1v += d[q] * Ts[de.e1[q]];
                        if (de.e2[q] >= 0) s2v += Ts[de.e2[q]];
                    }
                    T[s * nt + i] = -(c1[k] * s1v + c2[k] * s2v) * d[3];
                }
                __syncthreads();
            }
            if (has_item) {
                for (int s = 0; s < nb; ++s) {
                    R part = 0;
#pragma unroll
                    for (int j = 0; j < kM2lChunk; ++j)
                        if (j < len) part += cf[j] * T[s * nt + tb[j]] * Ms[s * nt + ta[j]];
                    acc.add(part);
                }
            }
        }
        if (has_item) accs[it] = Ops<R>::sub(acc.s, acc.c);
        __syncthreads();
        for (int b = threadIdx.x; b < nt; b += blockDim.x) {
            Acc<R> sum;
            for (int i = e.tab.m2l_item_off[b]; i < e.tab.m2l_item_off[b + 1]; ++i) sum.add(accs[i]);
            e.L[(size_t)c * nt + b] = (double)sum.s - (double)sum.c;
        }
    }
}

// M2L with the expansion in registers, one warp per target cell and one source
// cell per lane.  In the scaled variables
//   Tt_n = n! T_n,   Mt_a = (-1)^|a| M_a / a!,   Lt_b = b! L_b
// the translation is a plain correlation, Lt_b = sum_a Tt_{a+b} Mt_a.
//
// 1/r is harmonic: Tt_{n+2ex} + Tt_{n+2ey} + Tt_{n+2ez} = 0.  So every index
// with z >= 2 folds onto indices with z in {0, 1},
//   Tt_{(x, y, z)} = (-1)^m sum_j C(m, j) Tt_{(x+2j, y+2(m-j), z-2m)},  m = z / 2,
// the multipole is folded once per cell (k_fold_m), Lt is accumulated for z in
// {0, 1} only (its truncated sum is harmonic as well) and unfolded once per
// target.  (p+1)^2 coefficients instead of (p+1)(p+2)(p+3)/6: at p = 6, 49
// instead of 84, 532 multiply-adds a pair instead of 924, and a recurrence over
// 49 coefficients (plus 15 sums for z = 2) instead of 84.
// The order P is a template parameter so that every index is a constant and
// the compiler keeps Tt and Lt in registers.
// coefficients with z in {0, 1}: order k starts at k^2, its z = 0 entries by y, then z = 1 by y
__host__ __device__ constexpr int n_harm(int p) { return (p + 1) * (p + 1); }
__host__ __device__ constexpr int hidx(int a, int b, int c) {
    return (a + b + c) * (a + b + c) + (c ? (a + b + c) + 1 + b : b);
}
// z = 2 entries of the derivative table, after the n_harm(p) others
__host__ __device__ constexpr int n_harm2(int p) { return p * (p - 1) / 2; }
__host__ __device__ constexpr int tidx(int p, int a, int b, int c) {
    return c < 2 ? hidx(a, b, c) : n_harm(p) + (a + b + 1) * (a + b) / 2 + b;
}
__host__ __device__ constexpr int row_stride(int p) { return (n_harm(p) + 3) / 4 * 4; }

// Row `cell` of Ms: the folded multipole sum_{m, j} (-1)^m C(m, j) Mt, in FP64,
// rounded once to the row's type; the factors (-1)^|a| / a! come from a
// per-coefficient table (an FP64 divide is a long sequence on the FP64 pipe,
// the narrowest pipe of this GPU).  Row n_cells is zero: the source of idle lanes.
template <int P, class R>
__global__ void k_fold_m(const double* __restrict__ M, int n_cells, const double* __restrict__ mscale,
                         R* __restrict__ Ms) {
    constexpr int N = n_coef(P), H = n_harm(P), S = row_stride(P);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)(n_cells + 1) * S;
         i += (long long)gridDim.x * blockDim.x) {
        const int cell = (int)(i / S), h = (int)(i - (long long)cell * S);
        double v = 0.0;
        if (h < H && cell < n_cells) {
            int k = 0;
            while ((k + 1) * (k + 1) <= h) ++k;
            const int r = h - k * k, c = r > k ? 1 : 0, b = c ? r - k - 1 : r, a = k - b - c;
            const double* Mc = M + (size_t)cell * N;
            for (int m = 0; 2 * m <= a + b; ++m) {
                double binom = 1.0;   // C(m, j)
                for (int j = 0; j <= m; ++j) {
                    const int ax = a - 2 * j, bx = b - 2 * (m - j);
                    if (ax >= 0 && bx >= 0) {
                        const int id = cidx(ax, bx, c + 2 * m);
                        const double t = binom * (Mc[id] * __ldg(mscale + id));
                        v += (m & 1) ? -t : t;
                    }
                    binom = binom * (double)(m - j) / (double)(j + 1);
                }
            }
        }
        Ms[i] = (R)v;
    }
}

// Tt_n of the displacement (x, y, z) for z-index 0, 1 and 2, by
//   |n| r^2 Tt_n = -(2|n|-1) sum_i n_i x_i Tt_{n-e_i} - (|n|-1) sum_i n_i (n_i-1) Tt_{n-2e_i}.
// T[i * LD] is coefficient i (LD = 32: a lane's column of a shared table).
template <int P, int LD, class R>
__device__ __forceinline__ void taylor_harmonic(R x, R y, R z, R ir, R ir2, R* T) {
    R ax[P + 1], by[P + 1];
#pragma unroll
    for (int k = 1; k <= P; ++k) { ax[k] = (R)k * x; by[k] = (R)k * y; }
    T[0] = ir;
#pragma unroll
    for (int k = 1; k <= P; ++k) {
        const R ck = (R)(-(2.0 * k - 1.0) / (double)k) * ir2, dk = (R)(-((double)k - 1.0) / (double)k) * ir2;
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int b = 0; b <= k - c; ++b) {
                const int a = k - b - c;
                R s1 = 0, s2 = 0;
                if (a > 0) s1 += ax[a] * T[LD * hidx(a - 1, b, c)];
                if (b > 0) s1 += by[b] * T[LD * hidx(a, b - 1, c)];
                if (c > 0) s1 += z * T[LD * hidx(a, b, c - 1)];
                if (a > 1) s2 += (R)(a * (a - 1)) * T[LD * hidx(a - 2, b, c)];
                if (b > 1) s2 += (R)(b * (b - 1)) * T[LD * hidx(a, b - 2, c)];
                T[LD * hidx(a, b, c)] = (a > 1 || b > 1) ? ck * s1 + dk * s2 : ck * s1;
            }
    }
#pragma unroll
    for (int k = 2; k <= P; ++k)
#pragma unroll
        for (int b = 0; b <= k - 2; ++b)
            T[LD * tidx(P, k - 2 - b, b, 2)] = -(T[LD * hidx(k - b, b, 0)] + T[LD * hidx(k - 2 - b, b + 2, 0)]);
}

// L_b += sum_a Tt_{a+b} row_a over one source row (V: the vector type of its loads).
template <int P, int LD, class R, class V>
__device__ __forceinline__ void m2l_accumulate(const R* T, const R* __restrict__ row, R* L) {
    constexpr int W = (int)(sizeof(V) / sizeof(R));
    R mv[W];
#pragma unroll
    for (int k1 = 0; k1 <= P; ++k1)
#pragma unroll
        for (int c1 = 0; c1 < 2; ++c1)
#pragma unroll
            for (int b1 = 0; b1 <= k1 - c1; ++b1) {
                const int a1 = k1 - b1 - c1, ia = hidx(a1, b1, c1);
                if (ia % W == 0) {
                    const V v = __ldg(reinterpret_cast<const V*>(row) + ia / W);
                    memcpy(mv, &v, sizeof(V));
                }
                const R m = mv[ia % W];
#pragma unroll
                for (int k2 = 0; k2 <= P - k1; ++k2)
#pragma unroll
                    for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
                        for (int b2 = 0; b2 <= k2 - c2; ++b2) {
                            const int a2 = k2 - b2 - c2;
                            R& l = L[hidx(a2, b2, c2)];
                            l += T[LD * tidx(P, a1 + a2, b1 + b2, c1 + c2)] * m;
                        }
            }
}

// One round of a butterfly reduction that halves the vector: the lane keeps the
// half its bit O selects and gives the other to its partner.
template <int O, int N, class R>
__device__ __forceinline__ void butterfly_halve(R* v, int* base) {
    const bool up = (threadIdx.x & O) != 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const R mine = up ? v[i + N] : v[i], give = up ? v[i] : v[i + N];
        v[i] = mine + __shfl_xor_sync(0xffffffffu, give, O);
    }
    if (up) *base += N;
}

// Sum the 32 lanes' partial expansions: a butterfly that halves the vector each
// round leaves every lane with PAD / 32 finished sums (62 shuffles at p = 6; one
// full reduction per coefficient would take 245), which go to `out` (shared, PAD
// entries).  Then the warp unfolds and writes L_b = Lt_b / b! in FP64.
template <int P, class R>
__device__ __forceinline__ void m2l_finish(R (&L)[n_harm(P)], R* out, const EvalBufs& e, int tgt) {
    constexpr int N = n_coef(P), H = n_harm(P), PAD = (H + 31) / 32 * 32;
    const int lane = threadIdx.x & 31;
    R v[PAD];
#pragma unroll
    for (int i = 0; i < PAD; ++i) v[i] = i < H ? L[i] : (R)0;
    int base = 0;
    butterfly_halve<16, PAD / 2>(v, &base);
    butterfly_halve<8, PAD / 4>(v, &base);
    butterfly_halve<4, PAD / 8>(v, &base);
    butterfly_halve<2, PAD / 16>(v, &base);
    butterfly_halve<1, PAD / 32>(v, &base);
#pragma unroll
    for (int i = 0; i < PAD / 32; ++i) out[base + i] = v[i];
    __syncwarp();
    for (int i = lane; i < N; i += 32) {
        const short3 n = e.tab.mi[i];
        const int m = n.z >> 1, c = n.z & 1;
        double s = 0.0, binom = (m & 1) ? -1.0 : 1.0;   // (-1)^m C(m, j)
        for (int j = 0; j <= m; ++j) {
            s += binom * (double)out[hidx(n.x + 2 * j, n.y + 2 * (m - j), c)];
            binom = (m == 3) ? (j == 0 || j == 1 ? -3.0 : -1.0) : (m == 2) ? (j == 0 ? 2.0 : 1.0) : binom;
        }
        e.L[(size_t)tgt * N + i] = s * __ldg(e.tab.lscale + i);
    }
}

constexpr int kM2lWarps = 4;

// Bound by FP32 issue and by the lanes' uncoalesced row reads (208 B a source).
// 49 + 64 expansion and derivative registers fit 128, so 4 blocks (16 warps)
// stay resident (24 bytes spill); over 84 coefficients it took 168 registers at 3 blocks.
// N = 2^20 uniform, p = 6: 2.29 -> 1.70 ms (fold included); Plummer 3.88 -> 2.86 ms.
// Error against the FP64 form there: 9.2e-7 -> 7.6e-7 and 1.4e-6 -> 1.1e-6.
template <int P>
__global__ void __launch_bounds__(32 * kM2lWarps, 4) k_m2l_reg(EvalBufs e, const float* __restrict__ Ms) {
    constexpr int H = n_harm(P), S = row_stride(P);
    __shared__ float sums[kM2lWarps][(H + 31) / 32 * 32];
    const int lane = threadIdx.x & 31;
    const int tgt = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
    if (tgt >= e.n_cells) return;
    const int s0 = e.m2l_off[tgt], s1 = e.m2l_off[tgt + 1];
    if (s0 == s1) return;
    // exact integer displacement on the level-21 lattice, one FP32 scaling
    const int4 lt = e.lat[tgt];
    const float u = e.lat_unit;
    const int far = e.m2l_src[s0];   // an idle lane's displacement: any valid one, times the zero row
    float L[H];
#pragma unroll
    for (int i = 0; i < H; ++i) L[i] = 0.f;
    for (int base = s0; base < s1; base += 32) {
        const int s = base + lane;
        const int src = s < s1 ? e.m2l_src[s] : far;
        const int4 ls = __ldg(e.lat + src);
        const float x = (float)(lt.x - ls.x) * u, y = (float)(lt.y - ls.y) * u, z = (float)(lt.z - ls.z) * u;
        const float ir = rsqrtf(x * x + y * y + z * z);
        float T[H + n_harm2(P) + 1];
        taylor_harmonic<P, 1>(x, y, z, ir, ir * ir, T);
        m2l_accumulate<P, 1, float, float4>(T, Ms + (size_t)(s < s1 ? src : e.n_cells) * S, L);
    }
    m2l_finish<P>(L, sums[threadIdx.x >> 5], e, tgt);
}

// FP64: the local expansion stays in registers, the Taylor coefficients of each
// lane's source go to the lane's column of a shared-memory table.  The FP64
// pipe, not the shared-memory bandwidth, bounds this kernel (N = 2^20 uniform:
// 87.0 -> 49.1 ms, Plummer 151 -> 85.8 ms with the harmonic form).
template <int P>
__global__ void __launch_bounds__(32 * kM2lWarps) k_m2l_reg64(EvalBufs e, const double* __restrict__ Ms) {
    constexpr int H = n_harm(P), S = row_stride(P), NT = H + n_harm2(P);
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    double* T = reinterpret_cast<double*>(sm_raw) + (size_t)wib * NT * 32 + lane;   // T[i * 32]
    const int tgt = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
    if (tgt >= e.n_cells) return;
    const int s0 = e.m2l_off[tgt], s1 = e.m2l_off[tgt + 1];
    if (s0 == s1) return;
    const Dbl4 g = e.geom[tgt];
    const int far = e.m2l_src[s0];
    double L[H];
#pragma unroll
    for (int i = 0; i < H; ++i) L[i] = 0.0;
    for (int base = s0; base < s1; base += 32) {
        const int s = base + lane;
        const int src = s < s1 ? e.m2l_src[s] : far;
        const Dbl4 gs = e.geom[src];
        const double x = __dsub_rn(g.x, gs.x), y = __dsub_rn(g.y, gs.y), z = __dsub_rn(g.z, gs.z);
        const double r2 = x * x + y * y + z * z;
        taylor_harmonic<P, 32>(x, y, z, rsqrt(r2), 1.0 / r2, T);
        m2l_accumulate<P, 32, double, double2>(T, Ms + (size_t)(s < s1 ? src : e.n_cells) * S, L);
    }
    __syncwarp();   // the warp's table becomes the buffer of the lane sums
    m2l_finish<P>(L, T - lane, e, tgt);
}

// L2L from the cells of one level into their children: one block per cell.
template <class R>
__global__ void __launch_bounds__(kShiftBlock) k_l2l(EvalBufs e, int lo) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int nt = e.nt, c = lo + (int)blockIdx.x, t = threadIdx.x, lane = t & 31, j = t >> 5;
    const int4 in = e.info[c];
    if (in.z < 0) return;
    const int nch = in.w & 0xFF, cf = in.z;
    R* pw = reinterpret_cast<R*>(sm_raw);              // [8][3][kMaxOrder + 1]
    R* lp = pw + 24 * (kMaxOrder + 1);                 // [nt]
    R* mono = lp + nt + j * nt;                        // [8][nt], this warp's row
    shift_powers(e, e.geom[c], cf, nch, pw);
    for (int i = t; i < nt; i += kShiftBlock) lp[i] = (R)(e.L[(size_t)c * nt + i] * __ldg(e.tab.fact + i));
    __syncthreads();
    if (j >= nch) return;
    shift_monomials(e, pw, mono);
    for (int g = lane; g < nt; g += 32) {
        const int t1 = __ldg(e.tab.l2l_off + g + 1);
        R s = 0;
#pragma unroll 4
        for (int i = __ldg(e.tab.l2l_off + g); i < t1; ++i) {
            const unsigned u = __ldg(e.tab.l2l_terms + i);
            s += mono[u >> 16] * lp[u & 0xFFFFu];
        }
        e.L[(size_t)(cf + j) * nt + g] += (double)s * __ldg(e.tab.lscale + g);
    }
}

// ---------------------------------------------------------------------------
// Counting sort of a list by target.  The traversal appends the child pairs of
// one split pair together, so a warp's 32 entries often share a target: the
// lanes of one target (found with __match_any_sync) make one atomic between
// them.  The warp-uniform loop keeps all 32 lanes in every collective.
__global__ void k_group_count(const unsigned long long* list, long long count, int* cnt) {
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long w = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); w < count; w += stride) {
        const long long i = w + lane;
        const int tg = (i < count) ? (int)(list[i] >> 32) : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, tg);
        if (tg >= 0 && lane == __ffs(grp) - 1) atomicAdd(&cnt[tg], __popc(grp));
    }
}

__global__ void k_group_fill(const unsigned long long* list, long long count, const int* off, int* cursor, int* src) {
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long w = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); w < count; w += stride) {
        const long long i = w + lane;
        const unsigned long long v = (i < count) ? list[i] : 0ull;
        const int tg = (i < count) ? (int)(v >> 32) : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, tg);
        const int leader = __ffs(grp) - 1;
        int base = 0;
        if (tg >= 0 && lane == leader) base = atomicAdd(&cursor[tg], __popc(grp));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (tg >= 0) src[off[tg] + base + __popc(grp & ((1u << lane) - 1u))] = (int)(v & 0xFFFFFFFFull);
    }
}

int grid_for(long long n, int block, int cap) {
    long long g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

template <class R>
size_t p2m_smem(int p, int nt) { return sizeof(R) * (kMaxLeaf * 3 * (p + 1) + kMaxLeaf) + sizeof(short3) * nt + 16; }
template <class R>
size_t m2m_smem(int nt) { return sizeof(R) * (24 * (kMaxOrder + 1) + 24 * nt); }
template <class R>
size_t l2l_smem(int nt) { return sizeof(R) * (24 * (kMaxOrder + 1) + 9 * nt); }
template <class R>
size_t m2l_smem(int p, int nt, int items) {
    return sizeof(R) * (2 * kSB * nt + 4 * kSB + items + 2 * (p + 1) + ((p + 1) & 1) + 2) + sizeof(DerivEntry) * nt + 16;
}
template <class K>
cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <class R>
cudaError_t upward_level(const EvalBufs& e, int l, cudaStream_t s) {
    const int lo = e.lstart[l], hi = e.lstart[l + 1];
    if (hi > lo) k_m2m<R><<<hi - lo, kShiftBlock, m2m_smem<R>(e.nt), s>>>(e, lo);   // at most 33 KB: no opt-in
    return cudaGetLastError();
}

template <class R>
cudaError_t downward_level(const EvalBufs& e, int l, cudaStream_t s) {
    const int lo = e.lstart[l], hi = e.lstart[l + 1];
    if (hi > lo) k_l2l<R><<<hi - lo, kShiftBlock, l2l_smem<R>(e.nt), s>>>(e, lo);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_upward(const EvalBufs& e, bool mixed, int fp64_levels, cudaStream_t s) {
    cudaError_t err;
    const int grid = grid_for(e.n_cells, 1, 1 << 20);
    if (mixed) {
        const size_t sm = p2m_smem<float>(e.p, e.nt);
        if ((err = set_smem(k_p2m<float>, sm)) != cudaSuccess) return err;
        k_p2m<float><<<grid, 128, sm, s>>>(e);
    } else {
        const size_t sm = p2m_smem<double>(e.p, e.nt);
        if ((err = set_smem(k_p2m<double>, sm)) != cudaSuccess) return err;
        k_p2m<double><<<grid, 128, sm, s>>>(e);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    for (int l = e.n_levels - 2; l >= 0; --l) {
        err = (!mixed || l < fp64_levels) ? upward_level<double>(e, l, s) : upward_level<float>(e, l, s);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

template <int P>
cudaError_t launch_m2l_reg(const EvalBufs& e, float* ms, cudaStream_t s) {
    k_fold_m<P, float><<<grid_for((e.n_cells + 1ll) * row_stride(P), 256, 4096), 256, 0, s>>>(e.M, e.n_cells, e.tab.mscale, ms);
    k_m2l_reg<P><<<grid_for((long long)e.n_cells * 32, 32 * kM2lWarps, 1 << 30), 32 * kM2lWarps, 0, s>>>(e, ms);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_m2l_reg64(const EvalBufs& e, double* ms, cudaStream_t s) {
    k_fold_m<P, double><<<grid_for((e.n_cells + 1ll) * row_stride(P), 256, 4096), 256, 0, s>>>(e.M, e.n_cells, e.tab.mscale, ms);
    const size_t sm = sizeof(double) * std::max(n_harm(P) + n_harm2(P), (n_harm(P) + 31) / 32) * 32 * kM2lWarps;
    cudaError_t err = set_smem(k_m2l_reg64<P>, sm);
    if (err != cudaSuccess) return err;
    k_m2l_reg64<P><<<grid_for((long long)e.n_cells * 32, 32 * kM2lWarps, 1 << 30), 32 * kM2lWarps, sm, s>>>(e, ms);
    return cudaGetLastError();
}

// Scratch for the folded multipoles: FP32 rows (mixed) or FP64 rows, one per cell and a zero row, in bytes.
size_t m2l_scratch_bytes(int p, int n_cells, bool mixed) {
    return ((size_t)n_cells + 1) * row_stride(p) * (mixed ? sizeof(float) : sizeof(double));
}

cudaError_t launch_m2l(const EvalBufs& e, bool mixed, cudaStream_t s) {
    cudaError_t err;
    if (e.m2l_ms != nullptr && e.p <= 6) {
        float* f32 = static_cast<float*>(e.m2l_ms);
        double* f64 = static_cast<double*>(e.m2l_ms);
        switch (e.p) {
        case 1: return mixed ? launch_m2l_reg<1>(e, f32, s) : launch_m2l_reg64<1>(e, f64, s);
        case 2: return mixed ? launch_m2l_reg<2>(e, f32, s) : launch_m2l_reg64<2>(e, f64, s);
        case 3: return mixed ? launch_m2l_reg<3>(e, f32, s) : launch_m2l_reg64<3>(e, f64, s);
        case 4: return mixed ? launch_m2l_reg<4>(e, f32, s) : launch_m2l_reg64<4>(e, f64, s);
        case 5: return mixed ? launch_m2l_reg<5>(e, f32, s) : launch_m2l_reg64<5>(e, f64, s);
        default: return mixed ? launch_m2l_reg<6>(e, f32, s) : launch_m2l_reg64<6>(e, f64, s);
        }
    }
    const int grid = grid_for(e.n_cells, 1, 1 << 20);
    const int block = (e.tab.n_m2l_items + 31) / 32 * 32;
    if (mixed) {
        const size_t sm = m2l_smem<float>(e.p, e.nt, e.tab.n_m2l_items);
        if ((err = set_smem(k_m2l<float>, sm)) != cudaSuccess) return err;
        k_m2l<float><<<grid, block, sm, s>>>(e);
    } else {
        const size_t sm = m2l_smem<double>(e.p, e.nt, e.tab.n_m2l_items);
        if ((err = set_smem(k_m2l<double>, sm)) != cudaSuccess) return err;
        k_m2l<double><<<grid, block, sm, s>>>(e);
    }
    return cudaGetLastError();
}

cudaError_t launch_downward(const EvalBufs& e, bool mixed, int fp64_levels, cudaStream_t s) {
    for (int l = 0; l + 1 < e.n_levels; ++l) {
        cudaError_t err = (!mixed || l < fp64_levels) ? downward_level<double>(e, l, s) : downward_level<float>(e, l, s);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

cudaError_t launch_group(const unsigned long long* list, long long count, int n_cells, int* cnt, int* off, int* cursor,
                         int* src, int* tile_sums, cudaStream_t s) {
    cudaError_t err;
    if ((err = cudaMemsetAsync(cnt, 0, sizeof(int) * (size_t)n_cells, s)) != cudaSuccess) return err;
    if ((err = cudaMemsetAsync(cursor, 0, sizeof(int) * (size_t)n_cells, s)) != cudaSuccess) return err;
    if (count > 0) k_group_count<<<grid_for(count, 256, 4096), 256, 0, s>>>(list, count, cnt);
    if ((err = scan::exclusive(cnt, off, nullptr, n_cells, tile_sums, off + n_cells, s)) != cudaSuccess) return err;
    if (count > 0) k_group_fill<<<grid_for(count, 256, 4096), 256, 0, s>>>(list, count, off, cursor, src);
    return cudaGetLastError();
}

}  // namespace fmm
}  // namespace gtap
