// Per-run reset: re-zero the deques and control words, re-arm the pool's
// chunk queue, write the root records and push each root to a worker's deque
// (Sec. 4: storage is preallocated; a run only re-initialises it).
#include "launch.h"
#include "gtap_device.cuh"

namespace gtap {

__global__ void reset_kernel(KParams P, int init_queues) {
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nth = (size_t)gridDim.x * blockDim.x;
    const uint32_t Q = P.n_queues;
    const uint32_t cap = P.ring_mask + 1;
    // a slot no ticket of the last run reached still holds its own index (megabytes of them for a 1 GiB pool)
    const bool all = init_queues || P.ctl->used_known == 0;
    auto rearm = [&](unsigned long long* seq, uint64_t mask, unsigned long long used) {
        if (seq == nullptr) return;
        const uint64_t n = all || used > mask ? mask + 1 : used;
        for (size_t i = tid; i < n; i += nth) seq[i] = i;
    };
    rearm(P.cq_seq, P.ncq_mask, P.ctl->cq_used);
    rearm(P.sq_seq, P.sq_mask, P.ctl->sq_used);
    rearm(P.lq_seq, P.lq_mask, P.ctl->lq_used);
    if (tid < 16) P.ctl->sums[tid] = 0;
    if (P.gq != nullptr) {
        // central queue: slot i holds root i (published: sequence i + 1), the rest are free (sequence i)
        for (size_t i = tid; i <= P.gq_mask; i += nth) {
            const bool root = i < P.n_roots;
            P.gq[i] = ((unsigned long long)(uint32_t)(i + (root ? 1 : 0)) << 32) | (root ? (uint32_t)i : 0u);
        }
    }
    if (P.fstate != nullptr)
        for (size_t i = tid; i < P.n_frames; i += nth) P.fstate[i] = (i < P.n_roots) ? 3u : 0u;
    // root records
    for (size_t r = tid; r < P.n_roots; r += nth) {
        const RootDesc& d = P.root_desc[r];
        char* f = frame_ptr(P, (uint32_t)r);
        FrameHdr h;
        h.w0 = d.type & 0xFFu;
        h.pending = 0;
        h.parent = kRootBit | (uint32_t)r;
        h.w3 = 0;
        *reinterpret_cast<FrameHdr*>(f) = h;
        for (int i = 0; i < kRootPayloadBytes / 4; ++i)
            reinterpret_cast<uint32_t*>(f + kHdrBytes)[i] = reinterpret_cast<const uint32_t*>(d.payload)[i];
        RootEntry e;
        e.result[0] = 0; e.result[1] = 0; e.done = 0; e.type = d.type; e.req = r;
        P.roots[r] = e;
    }
    // deques: worker w owns roots w, w + W, w + 2W, ...
    for (size_t w = tid; w < P.n_workers; w += nth) {
        uint32_t cnt[kMaxQueues];
        for (uint32_t q = 0; q < Q; ++q) cnt[q] = 0;
        for (size_t r = w; P.gq == nullptr && r < P.n_roots; r += P.n_workers) {
            const uint32_t q = P.root_desc[r].queue % Q;
            P.rings[((size_t)w * Q + q) * cap + cnt[q]] = (uint32_t)r;
            ++cnt[q];
        }
        for (uint32_t q = 0; q < Q; ++q) {
            QState s;
            s.count = (int)cnt[q];
            s.head = 0;
            s.lock = 0;
            s.tail0 = cnt[q];
            P.qs[(size_t)w * Q + q] = s;
        }
    }
    if (tid == 0) {
        P.ctl->roots_remaining.v = P.n_roots;
        P.ctl->abort_flag.v = 0;
        P.ctl->bump.v = P.n_roots;
        P.ctl->cq_enq.v = 0;
        P.ctl->cq_deq.v = 0;
        P.ctl->cq_avail.v = 0;
        P.ctl->sc_enq.v = 0;
        P.ctl->sc_deq.v = 0;
        P.ctl->sc_avail.v = 0;
        P.ctl->lc_enq.v = 0;
        P.ctl->lc_deq.v = 0;
        P.ctl->lc_avail.v = 0;
        P.ctl->out_tail.v = 0;
        P.ctl->admitted.v = 0;
        P.ctl->scratch_top.v = 0;
        P.ctl->inflight.v = 0;
        P.ctl->gq_enq.v = P.gq ? P.n_roots : 0;
        P.ctl->gq_deq.v = 0;
        P.ctl->gq_avail.v = P.gq ? P.n_roots : 0;
        P.ctl->report_done = 0;
        P.ctl->err.code = 0;
        P.ctl->err.task_type = -1;
        P.ctl->err.worker = -1;
        P.ctl->err.detail = 0;
    }
}

cudaError_t launch_reset(const KParams& P, int init_queues, cudaStream_t s) {
    reset_kernel<<<304, 256, 0, s>>>(P, init_queues);
    return cudaGetLastError();
}

// Thread t sums word t % 16 over every 16th worker row of its block's share; the
// last block to finish writes the report.
constexpr int kReportBlocks = 32, kReportThreads = 256;

__global__ void __launch_bounds__(kReportThreads) report_kernel(KParams P, uint32_t n_roots, RunReport* report,
                                                                RootEntry* roots) {
    __shared__ unsigned long long sh[kReportThreads];
    __shared__ bool last;
    const int t = threadIdx.x;
    const uint32_t rows = kReportThreads / 16;
    const unsigned long long* st = reinterpret_cast<const unsigned long long*>(P.stats);
    unsigned long long sum = 0;
    for (uint32_t w = blockIdx.x * rows + t / 16; w < P.n_workers; w += gridDim.x * rows) sum += st[(size_t)w * 16 + t % 16];
    sh[t] = sum;
    // root results, 16 bytes a thread
    const uint4* src = reinterpret_cast<const uint4*>(P.roots);
    for (uint32_t i = blockIdx.x * kReportThreads + t; i < 2 * n_roots; i += gridDim.x * kReportThreads)
        reinterpret_cast<uint4*>(roots)[i] = src[i];
    __syncthreads();
    if (t < 16) {
        for (uint32_t k = 1; k < rows; ++k) sum += sh[t + 16 * k];
        atomicAdd(&P.ctl->sums[t], sum);
        __threadfence();
    }
    __syncthreads();
    if (t == 0) last = atomicAdd(&P.ctl->report_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (t < 16) report->sums[t] = ld_cg64(&P.ctl->sums[t]);
    if (t == 0) {
        report->bump = P.ctl->bump.v;
        report->scratch_top = P.ctl->scratch_top.v;
        report->err = P.ctl->err;
        P.ctl->cq_used = max(P.ctl->cq_enq.v, P.ctl->cq_deq.v);
        P.ctl->sq_used = max(P.ctl->sc_enq.v, P.ctl->sc_deq.v);
        P.ctl->lq_used = max(P.ctl->lc_enq.v, P.ctl->lc_deq.v);
        P.ctl->used_known = 1;
    }
}

cudaError_t launch_report(const KParams& P, uint32_t n_roots, RunReport* report, RootEntry* roots, cudaStream_t s) {
    static_assert(sizeof(WorkerStats) == 128 && sizeof(RootEntry) == 32, "the report reads 16 words a worker and 2 x 16 bytes a root");
    report_kernel<<<kReportBlocks, kReportThreads, 0, s>>>(P, n_roots, report, roots);
    return cudaGetLastError();
}

}  // namespace gtap
