// Thread-mode task programs written as explicit continuation state machines
// (the lowering Sec. 5.2 describes: locals that cross a join live in the task
// record and a switch on the resume point re-enters the function).
//
// Result slots are addressed as (byte offset in the parent record) / 8.
#pragma once
#include "gtap_device.cuh"
#include "sort_networks.cuh"

namespace gtap {

// ---------------------------------------------------------------------------
// fib(n) with a task at every call (Sec. 6.3 "Fibonacci"), or with a
// sequential cutoff (Sec. 6.3.2): a call with n below the cutoff is a leaf
// task that computes fib(n) by the serial recursion inside its lane.
// record: [16] n, route | cutoff << 8  [24] l  [32] r
struct FibSpawn { int32_t n; int32_t rc; };
constexpr uint32_t kFibSlotL = 3, kFibSlotR = 4;

// The serial recursion fib(n) = fib(n-1) + fib(n-2) with an explicit stack of
// pending calls (n < 64, so at most n + 1 entries).
static __device__ __noinline__ long long fib_serial(int n) {
    int stack[64];
    int sp = 0;
    long long acc = 0;
    stack[sp++] = n;
    while (sp > 0) {
        const int m = stack[--sp];
        if (m < 2) { acc += m; continue; }
        stack[sp++] = m - 1;
        stack[sp++] = m - 2;
    }
    return acc;
}

__device__ __forceinline__ void fib_step(TaskCtx& c) {
    const FibSpawn a = c.load<FibSpawn>();
    const int route = a.rc & 0xFF, cutoff = a.rc >> 8;
    // route 1 (DAQ with three queues, Sec. 6.3.2): recursive calls, leaves, continuations
    const int qrec = 0, qleaf = route ? 1 : 0, qcont = route ? 2 : 0;
    if (c.pc() == 0) {
        if (a.n < 2 || a.n < cutoff) { c.ret((unsigned long long)fib_serial(a.n)); return; }
        const int n1 = a.n - 1, n2 = a.n - 2;
        c.spawn(T_FIB, kFibSlotL, (n1 >= 2 && n1 >= cutoff) ? qrec : qleaf, FibSpawn{n1, a.rc});
        c.spawn(T_FIB, kFibSlotR, (n2 >= 2 && n2 >= cutoff) ? qrec : qleaf, FibSpawn{n2, a.rc});
        c.join(1, qcont);
    } else {
        const long long l = (long long)c.word<kFibSlotL>();
        const long long r = (long long)c.word<kFibSlotR>();
        c.ret((unsigned long long)(l + r));
    }
}

// ---------------------------------------------------------------------------
// N-Queens by bitmask backtracking, one task per placed row (Sec. 6.3), or
// with a cutoff depth (Sec. 6.3.1): a board with `depth` rows placed is a leaf
// task that finishes the search serially in its lane.
// record: [16] cols, diag_l, diag_r, row | n << 8 | route << 16 | depth << 24  [32] acc (u64, children add into it)
struct NqSpawn { uint32_t cols, dl, dr, meta; unsigned long long acc; unsigned long long pad; };
constexpr uint32_t kNqSlotAcc = 4;

// Serial backtracking from a partial board: one (cols, dl, dr, remaining
// candidates) frame per placed row, at most 16 rows.
static __device__ __noinline__ unsigned long long nq_serial(int n, int row, uint32_t cols, uint32_t dl, uint32_t dr) {
    if (row == n) return 1ull;
    const uint32_t full = (n >= 32) ? 0xFFFFFFFFu : ((1u << n) - 1u);
    uint32_t sc[17], sl[17], sr[17], sa[17];
    int top = 0;
    sc[0] = cols; sl[0] = dl; sr[0] = dr; sa[0] = ~(cols | dl | dr) & full;
    unsigned long long sols = 0;
    const int rows_left = n - row;
    while (top >= 0) {
        const uint32_t avail = sa[top];
        if (avail == 0) { --top; continue; }
        const uint32_t bit = avail & (0u - avail);
        sa[top] = avail ^ bit;
        if (top + 1 == rows_left) { ++sols; continue; }
        const uint32_t c2 = sc[top] | bit, l2 = (sl[top] | bit) << 1, r2 = (sr[top] | bit) >> 1;
        ++top;
        sc[top] = c2; sl[top] = l2; sr[top] = r2; sa[top] = ~(c2 | l2 | r2) & full;
    }
    return sols;
}

__device__ __forceinline__ void nqueens_step(TaskCtx& c) {
    if (c.pc() == 0) {
        const uint4 a = c.load<uint4>();
        const int row = (int)(a.w & 0xFF), n = (int)((a.w >> 8) & 0xFF), route = (int)((a.w >> 16) & 0xFF);
        const int depth = (int)(a.w >> 24);
        if (row == n) { c.ret(1ull); return; }
        if (depth > 0 && row >= depth) { c.ret(nq_serial(n, row, a.x, a.y, a.z)); return; }
        const uint32_t full = (n >= 32) ? 0xFFFFFFFFu : ((1u << n) - 1u);
        uint32_t avail = ~(a.x | a.y | a.z) & full;
        if (avail == 0) { c.ret(0ull); return; }
        const uint32_t meta = (uint32_t)(row + 1) | (a.w & 0xFFFFFF00u);
        // DAQ: route 1 = queue depth mod n_queues; route 2 = recursive tasks q0, cutoff leaves q1
        const int qchild = route == 1 ? (row + 1) : (route == 2 ? ((depth > 0 && row + 1 >= depth) ? 1 : 0) : 0);
        while (avail) {
            const uint32_t bit = avail & (0u - avail);
            avail ^= bit;
            NqSpawn s{a.x | bit, (a.y | bit) << 1, (a.z | bit) >> 1, meta, 0ull, 0ull};
            c.spawn(T_NQUEENS, kNqSlotAcc, qchild, s, kFlagAccumulate);
        }
        c.join(1, route == 1 ? row : 0);
    } else {
        c.ret(c.word<kNqSlotAcc>());
    }
}

// ---------------------------------------------------------------------------
// Unbalanced hashed tree.  SplitMix64 (Steele, Lea, Flood 2014): advance the
// state by the golden-ratio increment, then apply the xor-shift-multiply
// finaliser.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    unsigned long long z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned long long uts_child_id(unsigned long long p, uint32_t i) {
    return splitmix64(p ^ (0x9E3779B97F4A7C15ull * (unsigned long long)(i + 1)));
}
__device__ __forceinline__ uint32_t uts_arity(unsigned long long v, uint32_t m, unsigned long long thr) {
    return splitmix64(v ^ 0xD1B54A32D192ED03ull) < thr ? m : 0u;
}
// A node's result packs (nodes << 32 | leaves) of its subtree; sums of packed
// values add both fields as long as each stays below 2^32.
constexpr unsigned long long kUtsNode = 1ull << 32;

// record: [16] id  [24] threshold  [32] m|route<<8  [36] arity (0xFFFFFFFF: compute)  [40] acc
struct UtsSpawn { unsigned long long id, thr; uint32_t m_route, arity; unsigned long long acc; };
constexpr uint32_t kUtsSlotAcc = 5;
// range record: [16] parent id  [24] threshold  [32] m|route<<8  [36] lo  [40] hi  [44] pad  [48] acc
struct UtsRangeSpawn { unsigned long long id, thr; uint32_t m_route, lo, hi, pad; unsigned long long acc; };
constexpr uint32_t kUtsRangeSlotAcc = 6;
constexpr int kUtsFan = 8;   // children staged per step; wider nodes fork range tasks

__device__ __forceinline__ int uts_child_queue(unsigned long long cid, uint32_t m, unsigned long long thr, int route) {
    if (!route) return 0;
    return uts_arity(cid, m, thr) ? 0 : 1;  // nodes with children -> q0, leaves -> q1
}

// Spawn children [lo, hi) of node `id`: directly when few, else as range tasks.
__device__ __forceinline__ void uts_spawn_children(TaskCtx& c, unsigned long long id, unsigned long long thr,
                                                   uint32_t m_route, uint32_t lo, uint32_t hi, uint32_t slot) {
    const uint32_t m = m_route & 0xFF;
    const int route = (int)((m_route >> 8) & 0xFF);
    const uint32_t n = hi - lo;
    if (n <= (uint32_t)kUtsFan) {
        for (uint32_t i = lo; i < hi; ++i) {
            const unsigned long long cid = uts_child_id(id, i);
            c.spawn(T_UTS, slot, uts_child_queue(cid, m, thr, route), UtsSpawn{cid, thr, m_route, 0xFFFFFFFFu, 0ull},
                    kFlagAccumulate);
        }
    } else {
        const uint32_t per = (n + kUtsFan - 1) / kUtsFan;
        for (uint32_t s = lo; s < hi; s += per) {
            const uint32_t e = min(hi, s + per);
            c.spawn(T_UTS_RANGE, slot, 0, UtsRangeSpawn{id, thr, m_route, s, e, 0u, 0ull}, kFlagAccumulate);
        }
    }
}

// The root record carries the seed and flag kUtsHashRoot: its id is splitmix64(seed).
constexpr uint32_t kUtsHashRoot = 1u << 16;

__device__ __forceinline__ void uts_step(TaskCtx& c) {
    const UtsSpawn a = c.load<UtsSpawn>();
    const int route = (int)((a.m_route >> 8) & 0xFF);
    if (c.pc() == 0) {
        unsigned long long id = a.id;
        uint32_t mr = a.m_route;
        if (mr & kUtsHashRoot) { id = splitmix64(id); mr &= 0xFFFFu; }
        const uint32_t arity = (a.arity != 0xFFFFFFFFu) ? a.arity : uts_arity(id, mr & 0xFF, a.thr);
        if (arity == 0) { c.ret(kUtsNode | 1ull); return; }
        uts_spawn_children(c, id, a.thr, mr, 0, arity, kUtsSlotAcc);
        c.join(1, route ? 2 : 0);
    } else {
        c.ret(a.acc + kUtsNode);
    }
}

__device__ __forceinline__ void uts_range_step(TaskCtx& c) {
    const UtsRangeSpawn a = c.load<UtsRangeSpawn>();
    if (c.pc() == 0) {
        uts_spawn_children(c, a.id, a.thr, a.m_route, a.lo, a.hi, kUtsRangeSlotAcc);
        c.join(1, (a.m_route >> 8) ? 2 : 0);
    } else {
        c.ret(a.acc);
    }
}

// ---------------------------------------------------------------------------
// Adaptive trapezoid integration, thread mode (Program 1(a)).  Explicitly
// rounded double operations (no contraction into fused multiply-add), so the
// result is the same bit pattern as a plain IEEE evaluation on the host.
__device__ __forceinline__ double runge_fn(double x) {
    return __ddiv_rn(1.0, __dadd_rn(1.0, __dmul_rn(__dmul_rn(25.0, x), x)));
}
__device__ __forceinline__ double trap_rn(double a, double b) {
    return __dmul_rn(__dmul_rn(__dsub_rn(b, a), __dadd_rn(runge_fn(a), runge_fn(b))), 0.5);
}
// record: [16] a  [24] b  [32] eps  [40] l  [48] r
struct IntegSpawn { double a, b, eps; double pad; };
constexpr uint32_t kIntSlotL = 5, kIntSlotR = 6;

__device__ __forceinline__ void integrate_step(TaskCtx& c) {
    if (c.pc() == 0) {
        const IntegSpawn s = c.load<IntegSpawn>();
        const double m = __dmul_rn(0.5, __dadd_rn(s.a, s.b));
        const double coarse = trap_rn(s.a, s.b);
        const double fine = __dadd_rn(trap_rn(s.a, m), trap_rn(m, s.b));
        if (fabs(__dsub_rn(fine, coarse)) < s.eps) {
            const double v = __ddiv_rn(__dsub_rn(__dmul_rn(4.0, fine), coarse), 3.0);
            c.ret((unsigned long long)__double_as_longlong(v));
            return;
        }
        c.spawn(T_INTEGRATE, kIntSlotL, 0, IntegSpawn{s.a, m, s.eps, 0.0});
        c.spawn(T_INTEGRATE, kIntSlotR, 0, IntegSpawn{m, s.b, s.eps, 0.0});
        c.join(1, 0);
    } else {
        const double l = __longlong_as_double((long long)c.word<kIntSlotL>());
        const double r = __longlong_as_double((long long)c.word<kIntSlotR>());
        c.ret((unsigned long long)__double_as_longlong(__dadd_rn(l, r)));
    }
}

}  // namespace gtap

namespace gtap {

// ---------------------------------------------------------------------------
// k-clique counting by orientation (Sec. 6.4.2).  For a DAG edge (u, v),
// C = N+(u) n N+(v); count(S, 1) = |S|, count(S, j) = sum over w in S of
// count(S n N+(w), j - 1).  A set of at most `thr` (<= 64) vertices is counted
// where it is found, by its pairs or its 64-bit adjacency rows; a larger one is a
// task that forks over its branch range (the paper's split on the spawn-time
// estimate |C|), or counts its pairs when they are all that is left (see the
// warp-cooperative passes below).
//
// Sets of the first level, C = N+(u) n N+(v), are spawned unmaterialised:
// the record names P = N+(u), the vertex w = v and |C|, and the child writes C
// to the scratch arena when it first runs.  The edge-range tasks then only
// count, and the expensive intersections are spread over the set tasks that
// idle lanes steal (k = 4, scale 20: 874 -> 769 ms), while waiting first-level
// tasks hold no scratch.  Deeper sets are materialised by the spawning lane:
// that keeps the lanes expanding the frontier busy, and with DAQ choosing the
// fullest queue, cheap unmaterialised spawns at every level let the waiting
// frontier outgrow the frame pool (k = 5, scale 18, 1 GiB pool).
//
// Records (64 bytes):
//   KC range [16] root, lo, hi, pad   [32] acc  [40] local
//   KC set   [16] root, j  [24] set pointer  [32] len, lo  [40] hi, own  [48] acc  [56] local
//   own = kKcLazy: not materialised yet; set/len are P = N+(u), lo is w = v, hi is |C|
//   own = 1: materialised set in a recycled scratch block, freed by this task when its subtree is done
//   own = 0: a branch range of a set owned by an ancestor (or a set in never-recycled scratch)
struct KcRangeSpawn { uint32_t root, lo, hi, pad; unsigned long long acc, local; };
struct KcSetSpawn { uint32_t root, j; unsigned long long set; uint32_t len, lo, hi, own; unsigned long long acc, local; };
constexpr uint32_t kKcRangeSlotAcc = 4, kKcRangeLocal = 40;
constexpr uint32_t kKcSetSlotAcc = 6, kKcSetLocal = 56;
constexpr uint32_t kKcSetPtr = 24, kKcSetLenLo = 32, kKcSetHiOwn = 40;
constexpr uint32_t kKcLazy = 2;
constexpr int kKcFan = 8;          // children per split
constexpr int kKcMaxThr = 64;      // sets counted by 64-bit rows

// The root environment is immutable during a batch run (read-only path, L1);
// in a served session the poller writes root slots while the kernel runs, so
// it is read through L2 there.
__device__ __forceinline__ gtap_kclique_args kc_env(const KParams& P, uint32_t root) {
    return P.serving ? ld_obj<gtap_kclique_args>(P.root_desc[root].env)
                     : ld_obj_ro<gtap_kclique_args>(P.root_desc[root].env);
}

// Read-only adjacency (never written during a run): non-coherent cached loads.
struct AdjLoad { __device__ int operator()(const int* p) const { return __ldg(p); } };
// Sets in the scratch arena are written during the run: loads through L2.
struct SetLoad { __device__ int operator()(const int* p) const { return __ldcg(p); } };

// |a n b| for sorted lists; the first `cap` common elements go to out (if not null).
template <class LA, class LB>
static __device__ int kc_intersect(const int* a, int na, LA la, const int* b, int nb, LB lb, int* out, int cap) {
    int cnt = 0;
    if (na == 0 || nb == 0) return 0;
    if ((long long)na * 8 < nb) {
        // gallop the short list's elements through the long one
        int lo = 0;
        for (int i = 0; i < na && lo < nb; ++i) {
            const int x = la(a + i);
            int step = 1, hi = lo;
            while (hi < nb && lb(b + hi) < x) { lo = hi + 1; hi = lo + step; step <<= 1; }
            if (hi > nb) hi = nb;
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (lb(b + mid) < x) lo = mid + 1; else hi = mid; }
            if (lo < nb && lb(b + lo) == x) { if (out && cnt < cap) out[cnt] = x; ++cnt; ++lo; }
        }
    } else if ((long long)nb * 8 < na) {
        int lo = 0;
        for (int i = 0; i < nb && lo < na; ++i) {
            const int x = lb(b + i);
            int step = 1, hi = lo;
            while (hi < na && la(a + hi) < x) { lo = hi + 1; hi = lo + step; step <<= 1; }
            if (hi > na) hi = na;
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (la(a + mid) < x) lo = mid + 1; else hi = mid; }
            if (lo < na && la(a + lo) == x) { if (out && cnt < cap) out[cnt] = x; ++cnt; ++lo; }
        }
    } else {
        // branch-free merge: lanes of a warp with different data take the same path
        // every iteration (only the trip counts differ)
        int i = 0, j = 0;
        while (i < na && j < nb) {
            const int x = la(a + i), y = lb(b + j);
            if (x == y) {
                if (out && cnt < cap) out[cnt] = x;
                ++cnt;
            }
            i += (x <= y) ? 1 : 0;
            j += (y <= x) ? 1 : 0;
        }
    }
    return cnt;
}

// The j-cliques (j >= 2) of a set of ns <= 64 members that start at member `first`, from the
// set's adjacency rows (bit b of row[a]: member b is an out-neighbour of member a).
static __device__ unsigned long long kc_count_rows(const unsigned long long* row, int ns, int j, int first) {
    if (ns < j) return 0;
    const unsigned long long m0 = row[first];
    if (j == 2) return (unsigned)__popcll(m0);
    if (j == 3) {
        unsigned long long t = 0;
        for (unsigned long long w = m0; w; w &= w - 1) t += (unsigned)__popcll(m0 & row[__ffsll((long long)w) - 1]);
        return t;
    }
    // depth-first over choices; M = candidates at a level, R = those not yet tried there
    unsigned long long M[16], R[16];
    if (__popcll(m0) < j - 1) return 0;
    M[0] = m0;
    R[0] = m0;
    int l = 0;
    unsigned long long total = 0;
    while (l >= 0) {
        if (R[l] == 0) { --l; continue; }
        const int a = __ffsll((long long)R[l]) - 1;
        R[l] &= R[l] - 1;
        const unsigned long long mn = M[l] & row[a];
        const int rem = j - l - 2;   // still to choose after `first`, l others and a
        if (rem == 2) {
            for (unsigned long long w = mn; w; w &= w - 1) total += (unsigned)__popcll(mn & row[__ffsll((long long)w) - 1]);
        } else if (__popcll(mn) >= rem) {
            ++l;
            M[l] = mn;
            R[l] = mn;
        }
    }
    return total;
}

// ---------------------------------------------------------------------------
// Pivoting (Sec. 6.4.2, the second k-clique algorithm).  A candidate set of at
// most 64 vertices is encoded as 64-bit adjacency rows: bit b of row a says
// that members a and b are adjacent (in either direction of the DAG).  The
// pivot search counts the cliques of the set that contain exactly r more
// vertices: at a node (S, r still to choose, p pivots) the pivot x is the
// member of S with the most neighbours in S (lowest position on ties); the
// branches are x and the members of S not adjacent to x, in position order;
// branch w recurses on S n N(w) without the earlier branch vertices, w counted
// as a pivot when it is x and as chosen otherwise.  An empty S adds C(p, r);
// r = 0 adds 1 (only the all-pivot path leads to a leaf); a node with fewer
// than r members and pivots together adds nothing.
struct LocalRows { const unsigned long long* r; __device__ unsigned long long operator()(int i) const { return r[i]; } };
struct ScratchRows { const unsigned long long* r; __device__ unsigned long long operator()(int i) const { return __ldcg(r + i); } };

__device__ __forceinline__ unsigned long long kp_binom(int n, int r) {
    if (r < 0 || r > n) return 0ull;
    unsigned long long c = 1;
    for (int i = 1; i <= r; ++i) c = c * (unsigned long long)(n - r + i) / (unsigned long long)i;   // n <= 64, r <= 16
    return c;
}

template <class R>
__device__ __forceinline__ int kp_pivot(R row, unsigned long long S) {
    int best = -1, bx = 0;
    for (unsigned long long t = S; t; t &= t - 1) {
        const int x = __ffsll((long long)t) - 1;
        const int c = __popcll(row(x) & S);
        if (c > best) { best = c; bx = x; }
    }
    return bx;
}

constexpr int kKpStack = 66;   // every child set is smaller than its parent's: depth <= 64 + 1

template <class R>
static __device__ __noinline__ unsigned long long kp_count(R row, unsigned long long S0, int r0, int p0) {
    unsigned long long st_s[kKpStack], st_rem[kKpStack];
    unsigned char st_r[kKpStack], st_p[kKpStack], st_x[kKpStack];
    int top = -1;
    unsigned long long total = 0;
    auto enter = [&](unsigned long long S, int r, int p) {
        if (r < 0) return;
        if (r == 0) { total += 1; return; }
        if (__popcll(S) + p < r) return;
        if (S == 0) { total += kp_binom(p, r); return; }
        const int x = kp_pivot(row, S);
        ++top;
        st_s[top] = S;
        st_rem[top] = S & ~row(x);
        st_r[top] = (unsigned char)r;
        st_p[top] = (unsigned char)p;
        st_x[top] = (unsigned char)x;
    };
    enter(S0, r0, p0);
    while (top >= 0) {
        const unsigned long long rem = st_rem[top];
        if (rem == 0) { --top; continue; }
        const int w = __ffsll((long long)rem) - 1;
        st_rem[top] = rem & (rem - 1);
        const unsigned long long branches = st_s[top] & ~row(st_x[top]);
        const unsigned long long Sw = row(w) & st_s[top] & ~(branches & ((1ull << w) - 1ull));
        if (w == (int)st_x[top]) enter(Sw, st_r[top], st_p[top] + 1);
        else enter(Sw, st_r[top] - 1, st_p[top]);
    }
    return total;
}

// Adjacency rows of the candidate set S[0 .. ns) (ns <= 64, sorted by id), both
// directions: each DAG edge inside S is found from its earlier endpoint's
// out-list, then mirrored.
static __device__ void kp_rows(const int* S, int ns, const int64_t* off, const int* adj, unsigned long long* row) {
    for (int a = 0; a < ns; ++a) {
        const long long b0 = (long long)__ldg(reinterpret_cast<const long long*>(off) + S[a]);
        const int len = (int)((long long)__ldg(reinterpret_cast<const long long*>(off) + S[a] + 1) - b0);
        const int* nb = adj + b0;
        unsigned long long bits = 0;
        int i = 0, b = 0;
        if (len > 4 * ns) {
            int lo = 0;
            for (b = 0; b < ns && lo < len; ++b) {
                const int x = S[b];
                int hi = len;
                while (lo < hi) { const int mid = (lo + hi) >> 1; if (__ldg(nb + mid) < x) lo = mid + 1; else hi = mid; }
                if (lo < len && __ldg(nb + lo) == x) { bits |= 1ull << b; ++lo; }
            }
        } else {
            while (i < len && b < ns) {
                const int x = __ldg(nb + i), y = S[b];
                if (x < y) ++i;
                else if (y < x) ++b;
                else { bits |= 1ull << b; ++i; ++b; }
            }
        }
        row[a] = bits;
    }
    // mirror: adding the mirror of a mirrored bit changes nothing, so one pass in place is enough
    for (int b = 0; b < ns; ++b)
        for (unsigned long long t = row[b]; t; t &= t - 1) row[__ffsll((long long)t) - 1] |= 1ull << b;
}

// r-cliques of the candidate set S[0 .. ns) by the pivot search, in the lane.
static __device__ __noinline__ unsigned long long kp_count_small(const int* S, int ns, int r, const int64_t* off,
                                                                 const int* adj) {
    if (r == 1) return (unsigned long long)ns;
    if (ns < r) return 0;
    unsigned long long row[kKcMaxThr];
    kp_rows(S, ns, off, adj, row);
    const unsigned long long full = (ns == 64) ? ~0ull : ((1ull << ns) - 1ull);
    return kp_count(LocalRows{row}, full, r, 0);
}

// Candidate sets in the scratch arena: a set that fits one block is recycled
// when the set task that owns it is done with it.
__device__ __forceinline__ int* kc_scratch_alloc(TaskCtx& c, int n, bool* pooled) {
    return reinterpret_cast<int*>(scratch_alloc(c.P, (uint64_t)n * 4, pooled, c.type(), c.worker));
}

__device__ __forceinline__ int kc_queue(const gtap_kclique_args& e, int depth) { return e.route ? depth : 0; }
__device__ __forceinline__ long long kc_off(const gtap_kclique_args& e, long long v) {
    return __ldg(reinterpret_cast<const long long*>(e.off) + v);
}

// Bitset-encoded split (Sec. 6.4.2, pivoting): a candidate set too heavy for
// one lane (more than split_threshold members, at most 64) is encoded as its
// adjacency rows in a recycled scratch block, and a task over its pivot's
// branch range is forked; that task splits the range over child tasks (each
// re-applies the test) or runs its branches itself.
// Record: [16] root  [20] r:8 | p:8 | lo:8 | hi:8  [24] rows  [32] S  [40] branches (0: not chosen yet)
//         [48] x:8 | own:8 | depth:8  [56] acc
struct KpSpawn { uint32_t root, meta; unsigned long long rows, S, vp; uint32_t xo, pad; unsigned long long acc; };
constexpr uint32_t kKpSlotAcc = 7;
constexpr uint32_t kKpRows = 24, kKpBranches = 40, kKpXo = 48;

__device__ __forceinline__ bool kp_spawn_split(TaskCtx& c, const gtap_kclique_args& e, uint32_t root, const int* S,
                                               int ns, int r, int depth, uint32_t slot) {
    unsigned long long row[kKcMaxThr];
    kp_rows(S, ns, e.off, e.adj, row);
    bool pooled;
    unsigned long long* blk = reinterpret_cast<unsigned long long*>(scratch_alloc(c.P, (uint64_t)ns * 8, &pooled, c.type(), c.worker));
    if (!blk) return false;
    for (int a = 0; a < ns; ++a) __stcg(blk + a, row[a]);
    const unsigned long long full = (ns == 64) ? ~0ull : ((1ull << ns) - 1ull);
    c.spawn(T_KCLIQUE_PIV, slot, kc_queue(e, depth),
            KpSpawn{root, (uint32_t)r | (255u << 24), (unsigned long long)blk, full, 0ull,
                    (pooled ? 1u : 0u) << 8 | ((uint32_t)depth << 16), 0u, 0ull},
            kFlagAccumulate);
    return true;
}

static __device__ void kclique_piv_step(TaskCtx& c) {
    const KpSpawn a = c.load<KpSpawn>();
    const unsigned long long* rows = reinterpret_cast<const unsigned long long*>(a.rows);
    const bool own = ((a.xo >> 8) & 0xFF) != 0;
    if (c.pc() != 0) {
        if (own) scratch_free(c.P, rows, c.type(), c.worker);
        c.ret(a.acc);
        return;
    }
    const gtap_kclique_args e = kc_env(c.P, a.root);
    const ScratchRows row{rows};
    const int r = (int)(a.meta & 0xFF), p = (int)((a.meta >> 8) & 0xFF);
    const int depth = (int)((a.xo >> 16) & 0xFF);
    unsigned long long vp = a.vp;
    int x = (int)(a.xo & 0xFF);
    if (vp == 0) {
        // first run on this set: choose the pivot; the branches are x and its non-neighbours
        x = kp_pivot(row, a.S);
        vp = a.S & ~row(x);
        st_cg64(c.frame + kKpBranches, vp);
    }
    const int nb = __popcll(vp);
    const int lo = (int)((a.meta >> 16) & 0xFF), hi = min((int)(a.meta >> 24), nb);
    if (hi - lo > kKcFan) {
        const int per = (hi - lo + kKcFan - 1) / kKcFan;
        for (int s0 = lo; s0 < hi; s0 += per)
            c.spawn(T_KCLIQUE_PIV, kKpSlotAcc, kc_queue(e, depth + 1),
                    KpSpawn{a.root, (uint32_t)r | ((uint32_t)p << 8) | ((uint32_t)s0 << 16) | ((uint32_t)min(hi, s0 + per) << 24),
                            a.rows, a.S, vp, (uint32_t)x | ((uint32_t)(depth + 1) << 16), 0u, 0ull},
                    kFlagAccumulate);
        if (own) {
            // the owner frees the rows once its children are done
            st_cg64(c.frame + kKpXo, (unsigned long long)((uint32_t)x | (1u << 8) | ((uint32_t)depth << 16)));
        }
        c.join(1, kc_queue(e, depth));
        return;
    }
    // branches lo .. hi-1 (in bit order) in this lane
    unsigned long long total = 0;
    unsigned long long t = vp;
    for (int i = 0; i < lo; ++i) t &= t - 1;
    for (int i = lo; i < hi; ++i) {
        const int w = __ffsll((long long)t) - 1;
        t &= t - 1;
        const unsigned long long Sw = row(w) & a.S & ~(vp & ((1ull << w) - 1ull));
        total += (w == x) ? kp_count(row, Sw, r, p + 1) : kp_count(row, Sw, r - 1, p);
    }
    if (own) scratch_free(c.P, rows, c.type(), c.worker);
    c.ret(total);
}

// Pivoting on candidate sets of more than 64 vertices (multi-word bitsets).
// The first run of an edge's node materialises C = P n N+(w) and the rows of
// the subgraph C induces (ceil(|C| / 64) words per member, both directions)
// in one scratch allocation; every node keeps its own set S and branch set
// (the pivot and its non-neighbours) in a small block.  A node chooses its
// pivot on its first run; a node with more than kKcFan branches splits the
// branch range over child tasks; otherwise it runs its branches: a branch set
// of at most 64 members is compacted to 64-bit rows and counted in the lane,
// a larger one becomes a child node.
// Record: [16] root  [20] r:8 | p:8 | W:8 | flags:8 (1 lazy, 2 owns rows, 4 owns set, 8 branches chosen,
//         16 rows block pooled, 32 set block pooled)
//         (16/32: the rows / set block is a recycled one-block buffer; 64/128: a recycled large chunk)
//         [24] rows (lazy: P = N+(u))  [32] set block (lazy: w | |P| << 32)
//         [40] lo:16 | hi:16 | x:16 | depth:8 (lazy: |C| in lo/hi)  [48] local  [56] acc
struct KpbSpawn { uint32_t root, meta; unsigned long long rows, set, range, local, acc; };
constexpr uint32_t kKpbSlotAcc = 7;
constexpr uint32_t kKpbMeta = 16, kKpbRows = 24, kKpbSet = 32, kKpbRange = 40, kKpbLocal = 48;
constexpr int kKpbMaxW = 16;   // members up to 1024 (the DAG's out-lists are at most 8192, C is much smaller in practice)
constexpr uint32_t kKpbLazy = 1, kKpbOwnRows = 2, kKpbOwnSet = 4, kKpbChosen = 8, kKpbRowsPooled = 16, kKpbSetPooled = 32,
                   kKpbRowsLarge = 64, kKpbSetLarge = 128;

// Release the blocks a node owns (each block once: a root's set lies inside its rows block).
__device__ __forceinline__ void kpb_release(TaskCtx& c, uint32_t flags, const void* rows, const void* setb) {
    if (flags & kKpbOwnSet) scratch_free_kind(c.P, setb, (flags & kKpbSetPooled) ? 1 : ((flags & kKpbSetLarge) ? 2 : 0),
                                              c.type(), c.worker);
    if (flags & kKpbOwnRows) scratch_free_kind(c.P, rows, (flags & kKpbRowsPooled) ? 1 : ((flags & kKpbRowsLarge) ? 2 : 0),
                                               c.type(), c.worker);
}

__device__ __forceinline__ unsigned long long kpb_range(uint32_t lo, uint32_t hi, uint32_t x, uint32_t depth) {
    return (unsigned long long)(lo & 0xFFFF) | ((unsigned long long)(hi & 0xFFFF) << 16) |
           ((unsigned long long)(x & 0xFFFF) << 32) | ((unsigned long long)(depth & 0xFF) << 48);
}

// A branch set of at most 64 members as a compact 64-bit subgraph, then the pivot count.
__device__ __forceinline__ unsigned long long kpb_count_compact(const unsigned long long* rows, int W,
                                                                 const unsigned long long* Sw, int r, int p) {
    int m[kKcMaxThr];
    int c = 0;
    for (int t = 0; t < W; ++t)
        for (unsigned long long b = Sw[t]; b; b &= b - 1) m[c++] = t * 64 + __ffsll((long long)b) - 1;
    unsigned long long row[kKcMaxThr];
    for (int i = 0; i < c; ++i) {
        const unsigned long long* ri = rows + (size_t)m[i] * W;
        unsigned long long bits = 0;
        for (int j = 0; j < c; ++j)
            if ((__ldcg(ri + (m[j] >> 6)) >> (m[j] & 63)) & 1ull) bits |= 1ull << j;
        row[i] = bits;
    }
    const unsigned long long full = (c == 64) ? ~0ull : ((1ull << c) - 1ull);
    return kp_count(LocalRows{row}, full, r, p);
}

static __device__ void kclique_pivb_step(TaskCtx& c) {
    const KpbSpawn a = c.load<KpbSpawn>();
    uint32_t flags = a.meta >> 24;
    const int r = (int)(a.meta & 0xFF), p = (int)((a.meta >> 8) & 0xFF);
    int W = (int)((a.meta >> 16) & 0xFF);
    if (c.pc() != 0) {
        kpb_release(c, flags, reinterpret_cast<const void*>(a.rows), reinterpret_cast<const void*>(a.set));
        c.ret(a.acc + a.local);
        return;
    }
    const gtap_kclique_args e = kc_env(c.P, a.root);
    unsigned long long* rows = reinterpret_cast<unsigned long long*>(a.rows);
    unsigned long long* setb = reinterpret_cast<unsigned long long*>(a.set);
    uint32_t depth = (uint32_t)((a.range >> 48) & 0xFF);
    uint32_t lo = (uint32_t)(a.range & 0xFFFF), hi = (uint32_t)((a.range >> 16) & 0xFFFF);
    uint32_t x = (uint32_t)((a.range >> 32) & 0xFFFF);
    unsigned long long S[kKpbMaxW], V[kKpbMaxW];
    if (flags & kKpbLazy) {
        // materialise C = P n N+(w) and the rows of the subgraph it induces, in one allocation
        const int* P = reinterpret_cast<const int*>(a.rows);
        const int w = (int)(a.set & 0xFFFFFFFFull), np = (int)(a.set >> 32);
        const int cn = (int)lo;
        W = (cn + 63) / 64;
        if (W > kKpbMaxW) { c.fail(GTAP_ERR_INVALID_ARG, (unsigned long long)cn); return; }
        const uint64_t words = (uint64_t)cn * W + 2 * (uint64_t)W;
        int kind;
        char* blk = scratch_alloc_kind(c.P, words * 8 + (uint64_t)cn * 4, &kind, c.type(), c.worker);
        if (!blk) return;
        rows = reinterpret_cast<unsigned long long*>(blk);
        setb = rows + (size_t)cn * W;
        int* C = reinterpret_cast<int*>(setb + 2 * W);
        const long long ow = kc_off(e, w);
        kc_intersect(P, np, AdjLoad{}, e.adj + ow, (int)(kc_off(e, w + 1) - ow), AdjLoad{}, C, cn);
        for (uint64_t i = 0; i < (uint64_t)cn * W; ++i) __stcg(rows + i, 0ull);
        // DAG edges inside C from each member's out-list, set in both rows
        for (int i = 0; i < cn; ++i) {
            const int y = __ldcg(C + i);
            const long long oy = kc_off(e, y);
            const int ny = (int)(kc_off(e, y + 1) - oy);
            int u0 = 0, v0 = 0;
            while (u0 < ny && v0 < cn) {
                const int s0 = __ldg(e.adj + oy + u0), t0 = __ldcg(C + v0);
                if (s0 < t0) ++u0;
                else if (t0 < s0) ++v0;
                else {
                    unsigned long long* ri = rows + (size_t)i * W + (v0 >> 6);
                    __stcg(ri, __ldcg(ri) | (1ull << (v0 & 63)));
                    unsigned long long* rj = rows + (size_t)v0 * W + (i >> 6);
                    __stcg(rj, __ldcg(rj) | (1ull << (i & 63)));
                    ++u0; ++v0;
                }
            }
        }
        for (int t = 0; t < W; ++t) {
            const int rem_bits = cn - t * 64;
            S[t] = rem_bits >= 64 ? ~0ull : ((1ull << rem_bits) - 1ull);
            __stcg(setb + t, S[t]);   // read by the child tasks of a split branch range
        }
        // the set block lies inside the rows allocation: freeing the rows frees it (one free per block)
        flags = kKpbOwnRows | (kind == 1 ? kKpbRowsPooled : 0u) | (kind == 2 ? kKpbRowsLarge : 0u);
        lo = 0;
        hi = 0xFFFF;
        // what the resume needs: the blocks to free
        st_cg64(c.frame + kKpbRows, (unsigned long long)rows);
        st_cg64(c.frame + kKpbSet, (unsigned long long)setb);
        st_cg32(c.frame + kKpbMeta, (uint32_t)r | ((uint32_t)p << 8) | ((uint32_t)W << 16) | (flags << 24));
    } else {
        for (int t = 0; t < W; ++t) S[t] = __ldcg(setb + t);
    }
    if (!(flags & kKpbChosen)) {
        // the pivot: most neighbours inside S, lowest position on ties; the branches: x and its non-neighbours
        int best = -1;
        for (int t = 0; t < W; ++t)
            for (unsigned long long b = S[t]; b; b &= b - 1) {
                const int y = t * 64 + __ffsll((long long)b) - 1;
                int cnt = 0;
                for (int q = 0; q < W; ++q) cnt += __popcll(__ldcg(rows + (size_t)y * W + q) & S[q]);
                if (cnt > best) { best = cnt; x = (uint32_t)y; }
            }
        for (int t = 0; t < W; ++t) {
            V[t] = S[t] & ~__ldcg(rows + (size_t)x * W + t);
            __stcg(setb + W + t, V[t]);
        }
        flags |= kKpbChosen;
    } else {
        for (int t = 0; t < W; ++t) V[t] = __ldcg(setb + W + t);
    }
    int nb = 0;
    for (int t = 0; t < W; ++t) nb += __popcll(V[t]);
    hi = min(hi, (uint32_t)nb);
    if (hi - lo > (uint32_t)kKcFan) {
        const uint32_t per = (hi - lo + kKcFan - 1) / kKcFan;
        for (uint32_t s0 = lo; s0 < hi; s0 += per)
            c.spawn(T_KCLIQUE_PIVB, kKpbSlotAcc, kc_queue(e, (int)depth + 1),
                    KpbSpawn{a.root, (uint32_t)r | ((uint32_t)p << 8) | ((uint32_t)W << 16) | (kKpbChosen << 24),
                             (unsigned long long)rows, (unsigned long long)setb,
                             kpb_range(s0, min(hi, s0 + per), x, depth + 1), 0ull, 0ull},
                    kFlagAccumulate);
        st_cg32(c.frame + kKpbMeta, (uint32_t)r | ((uint32_t)p << 8) | ((uint32_t)W << 16) | (flags << 24));
        c.join(1, kc_queue(e, (int)depth));
        return;
    }
    // branches lo .. hi-1 of V, in bit order
    unsigned long long local = 0;
    int idx = 0;
    for (int t = 0; t < W && idx < (int)hi; ++t) {
        for (unsigned long long b = V[t]; b && idx < (int)hi; b &= b - 1, ++idx) {
            if (idx < (int)lo) continue;
            const int bit = __ffsll((long long)b) - 1;
            const int w = t * 64 + bit;
            const bool is_x = (uint32_t)w == x;
            const int r2 = is_x ? r : r - 1, p2 = is_x ? p + 1 : p;
            if (r2 < 0) continue;
            if (r2 == 0) { local += 1; continue; }
            // S_w = row(w) n S without the branch vertices before w
            unsigned long long Sw[kKpbMaxW];
            int cnt = 0;
            for (int q = 0; q < W; ++q) {
                const unsigned long long before = q < t ? V[q] : (q == t ? (V[q] & ((1ull << bit) - 1ull)) : 0ull);
                Sw[q] = __ldcg(rows + (size_t)w * W + q) & S[q] & ~before;
                cnt += __popcll(Sw[q]);
            }
            if (cnt + p2 < r2) continue;
            if (cnt == 0) { local += kp_binom(p2, r2); continue; }
            if (cnt <= kKcMaxThr) { local += kpb_count_compact(rows, W, Sw, r2, p2); continue; }
            int kind;
            unsigned long long* nb2 = reinterpret_cast<unsigned long long*>(scratch_alloc_kind(c.P, (uint64_t)W * 16, &kind, c.type(), c.worker));
            if (!nb2) return;
            for (int q = 0; q < W; ++q) __stcg(nb2 + q, Sw[q]);
            c.spawn(T_KCLIQUE_PIVB, kKpbSlotAcc, kc_queue(e, (int)depth + 1),
                    KpbSpawn{a.root, (uint32_t)r2 | ((uint32_t)p2 << 8) | ((uint32_t)W << 16) |
                                         ((kKpbOwnSet | (kind == 1 ? kKpbSetPooled : 0u) | (kind == 2 ? kKpbSetLarge : 0u)) << 24),
                             (unsigned long long)rows, (unsigned long long)nb2, kpb_range(0, 0xFFFF, 0, depth + 1), 0ull, 0ull},
                    kFlagAccumulate);
        }
    }
    if (c.nspawned == 0) {
        kpb_release(c, flags, rows, setb);
        c.ret(local);
        return;
    }
    st_cg64(c.frame + kKpbLocal, local);
    st_cg32(c.frame + kKpbMeta, (uint32_t)r | ((uint32_t)p << 8) | ((uint32_t)W << 16) | (flags << 24));
    c.join(1, kc_queue(e, (int)depth));
}

template <bool SCRATCH>
__device__ __forceinline__ int kc_ld(const int* p) { return SCRATCH ? __ldcg(p) : __ldg(p); }

template <bool SCRATCH>
__device__ __forceinline__ bool kc_contains(const int* L, int n, int x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (kc_ld<SCRATCH>(L + mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo < n && kc_ld<SCRATCH>(L + lo) == x;
}

__device__ __forceinline__ int kc_index_of(const int* C, int n, int x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (C[mid] < x) lo = mid + 1; else hi = mid;
    }
    return (lo < n && C[lo] == x) ? lo : -1;
}

// Warp-cooperative passes (orientation).  A step runs in three parts: each lane
// begins its own task and, where the work is intersections, leaves a request;
// all 32 lanes of the warp, with a task or without, then take the requests one
// after another, together; each lane finishes its task (spawn, join, return).
// Lanes with short and long adjacency lists no longer wait for each other, and
// the lanes of a warp that holds few tasks, as at the start and the end of a run,
// help with them instead of standing idle.
//
// Kinds of requests:
//   kKcEdges     DAG edges [lo, hi): per edge C = N+(u) n N+(v)
//   kKcBranches  branches [lo, hi) of a set S (len members, in scratch): per branch C = S n N+(w)
//   kKcPairs     a set of at most kKcSetMax members with one more vertex to choose after each
//                branch: the DAG edges inside it.  The set is S in scratch, or (lazy) A n B,
//                which is then never written to memory.
// For edges and branches a C of at most `thr` members is counted (its pairs when need == 2,
// from the 64-bit rows of the subgraph it induces when more); a larger one goes back to the
// owner lane (di / dc, at most hi - lo of them), which spawns it.  (The last sets below a
// branch, need == 2, are counted up to kKcSetMax members: written to scratch and queued, their
// number outgrew the arena at k = 5, scale 20.)
// Lanes of one warp may run tasks of different roots (batched or served graphs), so every
// request carries its graph.
//
// Counting the pairs of a set needs no rows: a hit is counted when a member's out-neighbour is
// found in the set, which is searched in shared memory.  (Per-lane merges of
// a set's branches, two branches a task, left the lanes waiting for one L2 load after another,
// in 57 tasks for a set of 92 members.)  Orientation and the 4-clique count of an R-MAT graph of
// scale 17: 31.8 -> 11.8 ms; 400 served requests, a quarter of them such counts at scales
// 10..14: 90 -> 65 ms.  Bound by issue: about 30 instructions for each list element searched.
constexpr int kKcEdges = 1, kKcBranches = 2, kKcPairs = 3;
// (the largest sets of an R-MAT graph of scale 20 hold between 256 and 512 members: its 4-clique
// count takes 218 ms with 512 here, 364 ms with 256 and the rest by the per-lane path.  Denser graphs
// have larger sets, which fork over their branches, one lane each, in full batches: 4-cliques of K_700
// 79 ms, of K_900 165 ms; with every set by the per-lane path it was 82 and 203 ms)
constexpr int kKcSetMax = 512;
// Per-warp area: the set, then the rows of a small set or 32 members' lists.
struct KcArea {
    int set[kKcSetMax];
    union {
        unsigned long long rows[kKcMaxThr];
        struct {
            const int* ptr[33];
            int len[33];
        } m;
    };
};
constexpr int kKcCoopSmem = (int)((sizeof(KcArea) + 15) / 16 * 16);

static_assert(kKcSetMax == 512, "kc_warp_pairs selects searches of up to 2 * 256 members");

struct KcReq {
    int kind = 0;
    int need = 0, thr = 0;
    uint32_t lo = 0, hi = 0, len = 0, own = 0;
    const int* set = nullptr;            // S in scratch, or the list A of a lazy set
    const int* list = nullptr;           // lazy set: the list B
    int nlist = 0;
    const long long* off = nullptr;
    const int* adj = nullptr;
    const int* src = nullptr;
    bool warp_task = false;              // a task of this kind is served by the warp: hold few at a time
    unsigned long long local = 0;        // the owner's count
    int nd = 0;                          // sets too large to count here: item and size
    uint32_t di[kKcFan];
    int dc[kKcFan];
};

__device__ __forceinline__ const int* kc_from(const void* p, int owner) {
    return reinterpret_cast<const int*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(p), owner));
}

// C = S n L by the warp (S the shorter sorted list, split over the lanes; L
// searched where it is: a copy of it in shared memory measured slower), in order
// in the area up to kKcSetMax members.  Returns |C|.
template <bool SSET, bool LSET>
__device__ __forceinline__ int kc_warp_collect(KcArea& w, const int* S, int ns, const int* L, int nl) {
    const int lane = threadIdx.x & 31;
    int cn = 0;
    for (int b = 0; b < ns; b += 32) {
        int x = 0;
        bool in = false;
        if (b + lane < ns) {
            x = kc_ld<SSET>(S + b + lane);
            in = kc_contains<LSET>(L, nl, x);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        const int p = cn + __popc(bal & lanemask_lt());
        if (in && p < kKcSetMax) w.set[p] = x;   // ascending: S is sorted, lanes in order
        cn += __popc(bal);
    }
    __syncwarp();
    return cn;
}
template <bool ASET>
__device__ __forceinline__ int kc_warp_intersect(KcArea& w, const int* A, int na, const int* B, int nb) {
    return (na <= nb) ? kc_warp_collect<ASET, false>(w, A, na, B, nb) : kc_warp_collect<false, ASET>(w, B, nb, A, na);
}

// The elements of m members' lists (w.m, closed by an endless one) as one sequence, lane l at
// elements l, l + 32, ...; an element is loaded a round before it is searched in the set, which
// is padded to 2 * HALF.  Returns this lane's hits.
// HALF 0: the search is a loop over `half`.
template <int HALF>
__device__ __forceinline__ unsigned kc_pair_rounds(const KcArea& w, int m, int rounds, int half = HALF) {
    const int lane = threadIdx.x & 31;
    int r = 0, o = lane, ln = w.m.len[0];
    const int* list = w.m.ptr[0];
    auto next = [&] {   // the element at the lane's place, or -1 past the end
        while (o >= ln) {
            o -= ln;
            ++r;
            ln = w.m.len[r];
            list = w.m.ptr[r];
        }
        const int x = r < m ? __ldg(list + o) : -1;
        if (r < m) o += 32;
        return x;
    };
    unsigned hits = 0;
    int x = next();
    for (int i = 0; i < rounds; ++i) {
        const int nx = next();
        int p = 0;   // the first member not less than x
        if constexpr (HALF == 0) {
            for (int h = half; h > 0; h >>= 1)
                if (w.set[p + h - 1] < x) p += h;
        } else {
#pragma unroll
            for (int h = HALF; h > 0; h >>= 1)
                if (w.set[p + h - 1] < x) p += h;
        }
        hits += w.set[p] == x ? 1u : 0u;
        x = nx;
    }
    return hits;
}

// This lane's share of the DAG edges inside the set w.set[0, cn) that leave members [lo, hi).
template <bool COMPACT>
__device__ __forceinline__ unsigned kc_warp_pairs(KcArea& w, int cn, int lo, int hi, const long long* off, const int* adj) {
    const int lane = threadIdx.x & 31;
    const int half = cn > 1 ? 1 << (31 - __clz(cn - 1)) : 1;   // half the padded size (which is >= 2)
    for (int i = cn + lane; i < 2 * half; i += 32) w.set[i] = 0x7FFFFFFF;
    __syncwarp();
    unsigned hits = 0;
    for (int base = lo; base < hi; base += 32) {
        // every lane prepares one member's list
        const int m = min(32, hi - base);
        int n = 0;
        if (lane < m) {
            const int v = w.set[base + lane];
            const long long o = __ldg(off + v);
            n = (int)(__ldg(off + v + 1) - o);
            w.m.ptr[lane] = adj + o;
            w.m.len[lane] = n;
        }
        if (lane == 0) { w.m.ptr[m] = adj; w.m.len[m] = 0x7FFFFFFF; }
        const int rounds = ((int)__reduce_add_sync(0xffffffffu, (unsigned)n) + 31) / 32;
        __syncwarp();
        if constexpr (COMPACT) {
            hits += kc_pair_rounds<0>(w, m, rounds, half);
        } else {
            switch (half) {
            case 1: hits += kc_pair_rounds<1>(w, m, rounds); break;
            case 2: hits += kc_pair_rounds<2>(w, m, rounds); break;
            case 4: hits += kc_pair_rounds<4>(w, m, rounds); break;
            case 8: hits += kc_pair_rounds<8>(w, m, rounds); break;
            case 16: hits += kc_pair_rounds<16>(w, m, rounds); break;
            case 32: hits += kc_pair_rounds<32>(w, m, rounds); break;
            case 64: hits += kc_pair_rounds<64>(w, m, rounds); break;
            case 128: hits += kc_pair_rounds<128>(w, m, rounds); break;
            default: hits += kc_pair_rounds<256>(w, m, rounds); break;
            }
        }
        __syncwarp();
    }
    return hits;
}

// This lane's share of the cliques of `need` vertices (>= 3) in the set cbuf[0, cn), cn <= 64:
// the warp builds the 64-bit rows, then a lane counts the cliques that start at its members.
__device__ __forceinline__ unsigned long long kc_warp_rows(KcArea& w, int cn, int need, const long long* off,
                                                           const int* adj) {
    const int lane = threadIdx.x & 31;
    const int* cbuf = w.set;
    unsigned long long* rows = w.rows;
    for (int base = 0; base < cn; base += 32) {
        long long ptr = 0;
        int n = 0;
        if (base + lane < cn) {
            const int v = cbuf[base + lane];
            ptr = __ldg(off + v);
            n = (int)(__ldg(off + v + 1) - ptr);
        }
        const int m = min(32, cn - base);
        for (int r = 0; r < m; ++r) {
            const int* list = adj + __shfl_sync(0xffffffffu, ptr, r);
            const int ln = __shfl_sync(0xffffffffu, n, r);
            unsigned long long bits = 0;
            for (int b = lane; b < ln; b += 32) {
                const int idx = kc_index_of(cbuf, cn, __ldg(list + b));
                if (idx >= 0) bits |= 1ull << idx;
            }
            const unsigned r0 = __reduce_or_sync(0xffffffffu, (unsigned)bits);
            const unsigned r1 = __reduce_or_sync(0xffffffffu, (unsigned)(bits >> 32));
            if (lane == 0) rows[base + r] = ((unsigned long long)r1 << 32) | r0;
        }
    }
    __syncwarp();
    unsigned long long total = 0;
    for (int a = lane; a < cn; a += 32) total += kc_count_rows(rows, cn, need, a);
    __syncwarp();   // the rows are rewritten by the next item
    return total;
}

// The requests of the warp's lanes, by all 32 lanes (converged).
// COMPACT: one search loop for every set size, for kernels that hold other programs too.
template <bool COMPACT>
static __device__ __noinline__ void kc_warp_requests(KcArea& w, KcReq& q) {
    const int lane = threadIdx.x & 31;
    for (unsigned m = __ballot_sync(0xffffffffu, q.kind != 0); m != 0u; m &= m - 1u) {
        const int owner = __ffs((int)m) - 1;
        const int kind = __shfl_sync(0xffffffffu, q.kind, owner);
        const int need = __shfl_sync(0xffffffffu, q.need, owner), thr = __shfl_sync(0xffffffffu, q.thr, owner);
        const uint32_t lo = __shfl_sync(0xffffffffu, q.lo, owner), hi = __shfl_sync(0xffffffffu, q.hi, owner);
        const int len = (int)__shfl_sync(0xffffffffu, q.len, owner);
        const int* set = kc_from(q.set, owner);
        const long long* off = reinterpret_cast<const long long*>(kc_from(q.off, owner));
        const int* adj = kc_from(q.adj, owner);
        unsigned long long mine = 0;
        if (kind == kKcPairs) {
            const int* list = kc_from(q.list, owner);
            int cn = len;
            if (list != nullptr) {
                cn = kc_warp_intersect<false>(w, set, len, list, __shfl_sync(0xffffffffu, q.nlist, owner));
                mine = kc_warp_pairs<COMPACT>(w, cn, 0, cn, off, adj);
            } else {
                for (int i = lane; i < cn; i += 32) w.set[i] = __ldcg(set + i);
                __syncwarp();
                mine = kc_warp_pairs<COMPACT>(w, cn, (int)lo, (int)hi, off, adj);
            }
        } else {
            // at most kKcFan items: lane i prepares item lo + i
            const int* src = kc_from(q.src, owner);
            const int items = (int)(hi - lo);
            long long oa = 0, ob = 0;
            int na = len, nb = 0;
            if (lane < items) {
                int v;
                if (kind == kKcEdges) {
                    const int u = __ldg(src + lo + lane);
                    v = __ldg(adj + lo + lane);
                    oa = __ldg(off + u);
                    na = (int)(__ldg(off + u + 1) - oa);
                } else {
                    v = __ldcg(set + lo + lane);
                }
                ob = __ldg(off + v);
                nb = (int)(__ldg(off + v + 1) - ob);
            }
            int nd = 0;
            for (int i = 0; i < items; ++i) {
                const int ina = __shfl_sync(0xffffffffu, na, i), inb = __shfl_sync(0xffffffffu, nb, i);
                const int* A = adj + __shfl_sync(0xffffffffu, oa, i);
                const int* B = adj + __shfl_sync(0xffffffffu, ob, i);
                const int cn = kind == kKcEdges ? kc_warp_intersect<false>(w, A, ina, B, inb)
                                                : kc_warp_intersect<true>(w, set, ina, B, inb);
                if (cn < need) continue;
                if (cn > thr && (kind == kKcEdges || need != 2 || cn > kKcSetMax)) {
                    if (lane == owner) { q.di[nd] = lo + (uint32_t)i; q.dc[nd] = cn; }
                    ++nd;
                } else if (need == 2) {
                    mine += kc_warp_pairs<COMPACT>(w, cn, 0, cn, off, adj);
                } else {
                    mine += kc_warp_rows(w, cn, need, off, adj);
                }
            }
            if (lane == owner) q.nd = nd;
        }
        // the owner's count: the sum over the lanes
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
        if (lane == owner) q.local = mine;
        __syncwarp();
    }
}

// Whether a root's tasks ask the warp: orientation with at least two more vertices to choose after
// an edge.  Pivoting and the triangle count run in their own lanes, 32 tasks a step.
__device__ __forceinline__ bool kc_warp_root(const gtap_kclique_args& e) {
    return e.algorithm != GTAP_KCLIQUE_PIVOT && e.k > 3;
}

// First part of the range step: returns true with a request for the warp, or false when the
// step is complete.
static __device__ bool kclique_range_begin(TaskCtx& c, KcReq& q) {
    const KcRangeSpawn a = c.load<KcRangeSpawn>();
    const gtap_kclique_args& e = kc_env(c.P, a.root);
    // (beside roots whose tasks ask the warp, a triangle count's are held few at a time as well: a claim of
    // 32 would take theirs too; 3-, 4- and 5-cliques of one R-MAT graph of scale 13 in one run 2.8 against 4.8 ms)
    q.warp_task = kc_warp_root(e) || (e.algorithm != GTAP_KCLIQUE_PIVOT && c.P.warp_roots == kWarpRootsBatch);
    if (c.pc() != 0) { c.ret(a.acc + a.local); return false; }
    const uint32_t n = a.hi - a.lo;
    if (n > (uint32_t)kKcFan) {
        const uint32_t per = (n + kKcFan - 1) / kKcFan;
        for (uint32_t s = a.lo; s < a.hi; s += per)
            c.spawn(T_KCLIQUE_ROOT, kKcRangeSlotAcc, kc_queue(e, 0), KcRangeSpawn{a.root, s, min(a.hi, s + per), 0u, 0ull, 0ull},
                    kFlagAccumulate);
        c.join(1, kc_queue(e, 0));
        return false;
    }
    const int thr = e.split_threshold;
    const int need = e.k - 2;
    const bool pivot = e.algorithm == GTAP_KCLIQUE_PIVOT;
    if (!pivot && need >= 2) {
        q.kind = kKcEdges;
        q.need = need;
        q.thr = thr;
        q.lo = a.lo;
        q.hi = a.hi;
        q.off = reinterpret_cast<const long long*>(e.off);
        q.adj = e.adj;
        q.src = e.src;
        return true;
    }
    unsigned long long local = 0;
    int C[kKcMaxThr];
    for (uint32_t ei = a.lo; ei < a.hi; ++ei) {
        const int u = __ldg(e.src + ei), v = __ldg(e.adj + ei);
        const long long ou = kc_off(e, u), ov = kc_off(e, v);
        const int nu = (int)(kc_off(e, u + 1) - ou), nv = (int)(kc_off(e, v + 1) - ov);
        const int cn = kc_intersect(e.adj + ou, nu, AdjLoad{}, e.adj + ov, nv, AdjLoad{}, need == 1 ? nullptr : C, kKcMaxThr);
        if (need == 1) { local += (unsigned)cn; continue; }
        if (cn < need) continue;
        // pivoting
        if (cn <= thr) {
            local += kp_count_small(C, cn, need, e.off, e.adj);
            continue;
        }
        if (cn <= kKcMaxThr) {
            if (!kp_spawn_split(c, e, a.root, C, cn, need, 1, kKcRangeSlotAcc)) return false;
            continue;
        }
        // more than 64 members: a pivot node over multi-word bitsets, materialised when it runs
        c.spawn(T_KCLIQUE_PIVB, kKcRangeSlotAcc, kc_queue(e, 1),
                KpbSpawn{a.root, (uint32_t)need | (kKpbLazy << 24), (unsigned long long)(e.adj + ou),
                         (unsigned long long)(uint32_t)v | ((unsigned long long)(uint32_t)nu << 32),
                         kpb_range((uint32_t)cn, (uint32_t)cn, 0, 1), 0ull, 0ull},
                kFlagAccumulate);
    }
    if (c.nspawned == 0) { c.ret(local); return false; }
    st_cg64(c.frame + kKcRangeLocal, local);
    c.join(1, kc_queue(e, 0));
    return false;
}

// Last part of the range step: the sets too large to count there become set tasks, which
// materialise N+(u) n N+(v) when they run and add their count into this task's accumulator.
static __device__ void kclique_range_finish(TaskCtx& c, const KcReq& q) {
    const KcRangeSpawn a = c.load<KcRangeSpawn>();
    const gtap_kclique_args& e = kc_env(c.P, a.root);
    for (int i = 0; i < q.nd; ++i) {
        const uint32_t ei = q.di[i];
        const int u = __ldg(e.src + ei), v = __ldg(e.adj + ei);
        const long long ou = kc_off(e, u);
        const int nu = (int)(kc_off(e, u + 1) - ou);
        c.spawn(T_KCLIQUE_SET, kKcRangeSlotAcc, kc_queue(e, 1),
                KcSetSpawn{a.root, (uint32_t)q.need, (unsigned long long)(e.adj + ou), (uint32_t)nu, (uint32_t)v,
                           (uint32_t)q.dc[i], kKcLazy, 0ull, 0ull},
                kFlagAccumulate);
    }
    if (c.nspawned == 0) { c.ret(q.local); return; }
    st_cg64(c.frame + kKcRangeLocal, q.local);
    c.join(1, kc_queue(e, 0));
}

static __device__ bool kclique_set_begin(TaskCtx& c, KcReq& q) {
    const KcSetSpawn a = c.load<KcSetSpawn>();
    const gtap_kclique_args& e = kc_env(c.P, a.root);
    // (branches of a set beyond kKcSetMax that need one more vertex are counted by their own lane)
    q.warp_task = kc_warp_root(e) && (a.j > 2 || (a.own == kKcLazy ? a.hi : a.len) <= (uint32_t)kKcSetMax);
    if (c.pc() != 0) {
        // an owner frees its set once every task that reads it is done
        if (a.own == 1u) scratch_free(c.P, reinterpret_cast<const int*>(a.set), c.type(), c.worker);
        c.ret(a.acc + a.local);
        return false;
    }
    const int* set = reinterpret_cast<const int*>(a.set);
    uint32_t len = a.len, lo = a.lo, hi = a.hi, own = a.own;
    const bool pivot = e.algorithm == GTAP_KCLIQUE_PIVOT;
    const int need = (int)a.j - 1;
    q.off = reinterpret_cast<const long long*>(e.off);
    q.adj = e.adj;
    if (!pivot && need == 1 && (own == kKcLazy ? hi : len) <= (uint32_t)kKcSetMax) {
        q.kind = kKcPairs;
        q.set = set;
        q.len = len;
        q.lo = lo;
        q.hi = hi;
        q.own = own;
        if (own == kKcLazy) {
            const int w = (int)a.lo;
            const long long ow = kc_off(e, w);
            q.list = e.adj + ow;
            q.nlist = (int)(kc_off(e, w + 1) - ow);
        }
        return true;
    }
    if (own == kKcLazy) {
        // materialise S = P n N+(w) (|S| = hi > thr, known from the spawn)
        const int w = (int)a.lo;
        const long long ow = kc_off(e, w);
        const int nw = (int)(kc_off(e, w + 1) - ow);
        bool pooled;
        int* S = kc_scratch_alloc(c, (int)a.hi, &pooled);
        if (!S) return false;
        kc_intersect(set, (int)a.len, SetLoad{}, e.adj + ow, nw, AdjLoad{}, S, (int)a.hi);
        set = S;
        len = a.hi;
        lo = 0;
        own = pooled ? 1u : 0u;
        // what the resume needs: the set to free
        st_cg64(c.frame + kKcSetPtr, (unsigned long long)S);
        st_cg64(c.frame + kKcSetLenLo, (unsigned long long)len);
        st_cg64(c.frame + kKcSetHiOwn, (unsigned long long)hi | ((unsigned long long)own << 32));
    }
    const int depth = e.k - 2 - (int)a.j + 1;
    const uint32_t n = hi - lo;
    if (n > (uint32_t)kKcFan) {
        const uint32_t per = (n + kKcFan - 1) / kKcFan;
        for (uint32_t s = lo; s < hi; s += per)
            c.spawn(T_KCLIQUE_SET, kKcSetSlotAcc, kc_queue(e, depth),
                    KcSetSpawn{a.root, a.j, (unsigned long long)set, len, s, min(hi, s + per), 0u, 0ull, 0ull},
                    kFlagAccumulate);
        c.join(1, kc_queue(e, depth));
        return false;
    }
    const int thr = e.split_threshold;
    if (!pivot && need >= 2) {
        q.kind = kKcBranches;
        q.need = need;
        q.thr = thr;
        q.set = set;
        q.len = len;
        q.lo = lo;
        q.hi = hi;
        q.own = own;
        return true;
    }
    // a branch range of a set of more than kKcSetMax members (need == 1), or pivoting
    unsigned long long local = 0;
    int C[kKcMaxThr];
    for (uint32_t i = lo; i < hi; ++i) {
        const int w = __ldcg(set + i);
        const long long ow = kc_off(e, w);
        const int nw = (int)(kc_off(e, w + 1) - ow);
        const int cn = kc_intersect(set, (int)len, SetLoad{}, e.adj + ow, nw, AdjLoad{}, need == 1 ? nullptr : C, kKcMaxThr);
        if (need == 1) { local += (unsigned)cn; continue; }
        if (cn < need) continue;
        if (cn <= thr) {
            local += kp_count_small(C, cn, need, e.off, e.adj);
            continue;
        }
        if (cn <= kKcMaxThr) {
            if (!kp_spawn_split(c, e, a.root, C, cn, need, depth + 1, kKcSetSlotAcc)) return false;
            continue;
        }
        bool pooled;
        int* S = kc_scratch_alloc(c, cn, &pooled);
        if (!S) return false;
        kc_intersect(set, (int)len, SetLoad{}, e.adj + ow, nw, AdjLoad{}, S, cn);
        c.spawn(T_KCLIQUE_SET, kKcSetSlotAcc, kc_queue(e, depth + 1),
                KcSetSpawn{a.root, (uint32_t)need, (unsigned long long)S, (uint32_t)cn, 0u, (uint32_t)cn, pooled ? 1u : 0u,
                           0ull, 0ull},
                kFlagAccumulate);
    }
    if (c.nspawned == 0) {
        if (own == 1u) scratch_free(c.P, set, c.type(), c.worker);
        c.ret(local);
        return false;
    }
    st_cg64(c.frame + kKcSetLocal, local);
    c.join(1, kc_queue(e, depth));
    return false;
}

static __device__ void kclique_set_finish(TaskCtx& c, const KcReq& q) {
    const KcSetSpawn a = c.load<KcSetSpawn>();
    const gtap_kclique_args& e = kc_env(c.P, a.root);
    const int depth = e.k - 2 - (int)a.j + 1;
    // deeper sets are materialised here, by the spawning lane (see the header)
    for (int i = 0; i < q.nd; ++i) {
        const int w = __ldcg(q.set + q.di[i]);
        const long long ow = kc_off(e, w);
        const int nw = (int)(kc_off(e, w + 1) - ow);
        bool pooled;
        int* S = kc_scratch_alloc(c, q.dc[i], &pooled);
        if (!S) return;
        kc_intersect(q.set, (int)q.len, SetLoad{}, e.adj + ow, nw, AdjLoad{}, S, q.dc[i]);
        c.spawn(T_KCLIQUE_SET, kKcSetSlotAcc, kc_queue(e, depth + 1),
                KcSetSpawn{a.root, (uint32_t)q.need, (unsigned long long)S, (uint32_t)q.dc[i], 0u, (uint32_t)q.dc[i],
                           pooled ? 1u : 0u, 0ull, 0ull},
                kFlagAccumulate);
    }
    if (c.nspawned == 0) {
        if (q.own == 1u) scratch_free(c.P, q.set, c.type(), c.worker);
        c.ret(q.local);
        return;
    }
    st_cg64(c.frame + kKcSetLocal, q.local);
    c.join(1, kc_queue(e, depth));
}

}  // namespace gtap

namespace gtap {

// ---------------------------------------------------------------------------
// Thread-mode Cilksort (Sec. 6.3: sort halves in parallel and merge with a
// forked parallel merge; Sec. 6.3.2 routes recursive, serial-sort and
// serial-merge tasks to three DAQ queues).  One lane is one task, so a leaf
// sorts or merges its keys alone (these lanes touch unrelated data: the
// accesses of a warp are not coalesced, the structural cost the paper names).
// Buffers: 0 = dst, 1 = tmp; sort leaves read src.
// Records:  TSORT  [16] root, into  [24] lo, hi (u32)
//           TMERGE [16] root, from  [24] a0, a1, b0, b1  [40] out
struct CsSortSpawn { uint32_t root, into, lo, hi; };
struct CsMergeSpawn { uint32_t root, from, a0, a1, b0, b1, out, pad; };
constexpr uint32_t kCsSlot = 7;       // void results: accumulate 0, nothing written
constexpr int kCsMaxSortCut = 256;

__device__ __forceinline__ gtap_cilksort_args cs_env(const KParams& P, uint32_t root) {
    return P.serving ? ld_obj<gtap_cilksort_args>(P.root_desc[root].env)
                     : ld_obj_ro<gtap_cilksort_args>(P.root_desc[root].env);
}
__device__ __forceinline__ uint32_t* cs_buf(const gtap_cilksort_args& e, uint32_t b) { return b ? e.tmp : e.dst; }
__device__ __forceinline__ int cs_queue(const gtap_cilksort_args& e, int kind) { return e.route ? kind : 0; }

// Serial sort leaf: the lane's keys in registers through a bitonic network of 32
// or 64 (shorter ranges padded with the largest key).  An insertion sort in
// local memory took a dependent load and store per move, and every lane of a
// warp waited for the longest.
// (With the windowed merges and the wider search below: 300,007 keys, three
// queues, 2.37 -> 1.35 ms; what is left is the chain of forks and joins.)
template <int N>
static __device__ __noinline__ void cs_sort_network(const uint32_t* src, uint32_t* out, int n) {
    uint32_t k[N];
#pragma unroll
    for (int i = 0; i < N; ++i) k[i] = i < n ? __ldcg(src + i) : 0xFFFFFFFFu;
    sort_registers<N>(k);
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < n) __stcg(out + i, k[i]);
}
static __device__ __noinline__ void cs_sort_insertion(const uint32_t* src, uint32_t* out, int n) {
    uint32_t k[kCsMaxSortCut];
    for (int i = 0; i < n; ++i) {
        const uint32_t x = __ldcg(src + i);
        int j = i;
        while (j > 0 && k[j - 1] > x) { k[j] = k[j - 1]; --j; }
        k[j] = x;
    }
    for (int i = 0; i < n; ++i) __stcg(out + i, k[i]);
}
__device__ __forceinline__ void cs_sort_leaf(const uint32_t* src, uint32_t* out, int n) {
    if (n <= 32) cs_sort_network<32>(src, out, n);
    else if (n <= 64) cs_sort_network<64>(src, out, n);
    else cs_sort_insertion(src, out, n);   // a sort_cutoff above the default
}

// Serial merge leaf: eight outputs a step, the lowest eight of the next eight
// keys of either run (a two-finger merge waits for one L2 load per output).  The
// keys taken from A are those not above their partner in reversed B.  A key past
// a run's end reads as the largest value; once one of those ties with a real
// key, all that is left has that value.
static __device__ __noinline__ void cs_merge_leaf(const uint32_t* A, uint32_t na, const uint32_t* B, uint32_t nb,
                                                  uint32_t* out) {
    constexpr uint32_t kW = 8;
    const unsigned long long n = (unsigned long long)na + nb;
    unsigned long long i = 0, j = 0;
    for (unsigned long long done = 0; done < n; done += kW) {
        uint32_t x[kW], y[kW];
#pragma unroll
        for (uint32_t k = 0; k < kW; ++k) {
            x[k] = i + k < na ? __ldcg(A + i + k) : 0xFFFFFFFFu;
            y[k] = j + k < nb ? __ldcg(B + j + k) : 0xFFFFFFFFu;
        }
        uint32_t taken = 0;
#pragma unroll
        for (uint32_t k = 0; k < kW; ++k) taken += x[k] <= y[kW - 1 - k] ? 1u : 0u;
        lowest_of_two_sorted<(int)kW>(x, y);
#pragma unroll
        for (uint32_t k = 0; k < kW; ++k)
            if (done + k < n) __stcg(out + done + k, x[k]);
        i += taken;
        j += kW - taken;
    }
}

__device__ __forceinline__ void cs_merge_spawn(TaskCtx& c, const gtap_cilksort_args& e, uint32_t root, uint32_t from,
                                               uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, uint32_t out) {
    const bool leaf = (a1 - a0) + (b1 - b0) <= e.merge_cutoff;
    c.spawn(T_TMERGE, kCsSlot, cs_queue(e, leaf ? 2 : 0), CsMergeSpawn{root, from, a0, a1, b0, b1, out, 0u},
            kFlagAccumulate);
}

__device__ __forceinline__ void cilksort_sort_step(TaskCtx& c) {
    const CsSortSpawn a = c.load<CsSortSpawn>();
    const gtap_cilksort_args e = cs_env(c.P, a.root);
    const uint32_t n = a.hi - a.lo, mid = a.lo + n / 2;
    if (c.pc() == 0) {
        if (n <= e.sort_cutoff) {
            cs_sort_leaf(e.src + a.lo, cs_buf(e, a.into) + a.lo, (int)n);
            c.ret(0ull);
            return;
        }
        const uint32_t other = 1u - a.into;
        const uint32_t h0 = mid - a.lo, h1 = a.hi - mid;
        c.spawn(T_TSORT, kCsSlot, cs_queue(e, h0 <= e.sort_cutoff ? 1 : 0), CsSortSpawn{a.root, other, a.lo, mid}, kFlagAccumulate);
        c.spawn(T_TSORT, kCsSlot, cs_queue(e, h1 <= e.sort_cutoff ? 1 : 0), CsSortSpawn{a.root, other, mid, a.hi}, kFlagAccumulate);
        c.join(1, 0);
    } else if (c.pc() == 1) {
        // the halves are sorted in the other buffer: merge them back into this task's buffer
        cs_merge_spawn(c, e, a.root, 1u - a.into, a.lo, mid, mid, a.hi, a.lo);
        c.join(2, 0);
    } else {
        c.ret(0ull);
    }
}

__device__ __forceinline__ void cilksort_merge_step(TaskCtx& c) {
    const CsMergeSpawn a = c.load<CsMergeSpawn>();
    if (c.pc() != 0) { c.ret(0ull); return; }
    const gtap_cilksort_args e = cs_env(c.P, a.root);
    const uint32_t* X = cs_buf(e, a.from);
    uint32_t* Y = cs_buf(e, 1u - a.from);
    uint32_t a0 = a.a0, a1 = a.a1, b0 = a.b0, b1 = a.b1;
    if ((a1 - a0) + (b1 - b0) <= e.merge_cutoff) {
        cs_merge_leaf(X + a0, a1 - a0, X + b0, b1 - b0, Y + a.out);
        c.ret(0ull);
        return;
    }
    if (a1 - a0 < b1 - b0) { uint32_t t = a0; a0 = b0; b0 = t; t = a1; a1 = b1; b1 = t; }
    const uint32_t ma = a0 + (a1 - a0) / 2;
    const uint32_t x = __ldcg(X + ma);
    // first position of B whose key is not less than x: seven probes a step, one round
    // trip for eight times fewer candidates
    uint32_t lo = b0, hi = b1;
    while (lo < hi) {
        const uint32_t span = hi - lo;
        uint32_t less = 0;   // probes below x: they are the first ones, B is sorted
#pragma unroll
        for (uint32_t p = 0; p < 7; ++p) less += __ldcg(X + lo + (uint32_t)((unsigned long long)span * (p + 1) / 8)) < x ? 1u : 0u;
        const uint32_t nlo = less > 0 ? lo + (uint32_t)((unsigned long long)span * less / 8) + 1 : lo;
        hi = less < 7 ? lo + (uint32_t)((unsigned long long)span * (less + 1) / 8) : hi;
        lo = nlo;
    }
    const uint32_t at = a.out + (ma - a0) + (lo - b0);
    __stcg(Y + at, x);
    cs_merge_spawn(c, e, a.root, a.from, a0, ma, b0, lo, a.out);
    cs_merge_spawn(c, e, a.root, a.from, ma + 1, a1, lo, b1, at + 1);
    c.join(1, 0);
}

}  // namespace gtap
