// Several sparse instances in one launch: the batch kernel (mars_solve_batch)
// and the persistent serving kernel. Both run the sliced-ELL job of
// sell_job.cuh with its magnetisations in shared memory, the slot width,
// coupling format and degree chosen per job.
#include "sell_job.cuh"

#include <algorithm>
#include <cstdlib>

namespace mars {
namespace {

constexpr int kKeepSmem = 16 * 1024;  // of a block's shared memory, for the static part (allow_smem)

// One job of a batched launch with its own slot width (1 or 2, job.rt),
// coupling format and degree under the CTA's two-slot bookkeeping. Regular
// instances of degree 4 or 6 (square and cubic lattices) have their coupling
// loop unrolled in the shapes such instances take: format 1 only beyond 32767
// spins, where one slot is all that fits.
template <int NT>
__device__ void run_batch_job(const BatchJob& job, float* m, SlotState<2, NT / 32>& S)
{
    const int deg = NT == 1024 ? job.in.regular_deg : 0;
    const int key = job.rt * 4 + job.fmt;
    if constexpr (NT == 1024) {
        if (deg == 4 || deg == 6) {
            switch (key) {
            case 4 + 1: return deg == 4 ? run_job<1, NT, 1, 4, 2>(job.in, job.s, m, S) : run_job<1, NT, 1, 6, 2>(job.in, job.s, m, S);
            case 4 + 2: return deg == 4 ? run_job<1, NT, 2, 4, 2>(job.in, job.s, m, S) : run_job<1, NT, 2, 6, 2>(job.in, job.s, m, S);
            case 4 + 3: return deg == 4 ? run_job<1, NT, 3, 4, 2>(job.in, job.s, m, S) : run_job<1, NT, 3, 6, 2>(job.in, job.s, m, S);
            case 8 + 2: return deg == 4 ? run_job<2, NT, 2, 4, 2>(job.in, job.s, m, S) : run_job<2, NT, 2, 6, 2>(job.in, job.s, m, S);
            case 8 + 3: return deg == 4 ? run_job<2, NT, 3, 4, 2>(job.in, job.s, m, S) : run_job<2, NT, 3, 6, 2>(job.in, job.s, m, S);
            }
        }
    }
    switch (key) {
    case 4 + 3: run_job<1, NT, 3, 0, 2>(job.in, job.s, m, S); break;
    case 4 + 2: run_job<1, NT, 2, 0, 2>(job.in, job.s, m, S); break;
    case 4 + 1: run_job<1, NT, 1, 0, 2>(job.in, job.s, m, S); break;
    case 4 + 0: run_job<1, NT, 0, 0, 2>(job.in, job.s, m, S); break;
    case 8 + 3: run_job<2, NT, 3, 0, 2>(job.in, job.s, m, S); break;
    case 8 + 2: run_job<2, NT, 2, 0, 2>(job.in, job.s, m, S); break;
    case 8 + 1: run_job<2, NT, 1, 0, 2>(job.in, job.s, m, S); break;
    default: run_job<2, NT, 0, 0, 2>(job.in, job.s, m, S); break;
    }
}

// Several instances in one persistent launch: CTAs work through the job list
// in order, each job's replica queue drained by every CTA before it moves on
// (a job is a CTA's current work until its queue is empty). Shared memory is
// sized for the most demanding job; slot width and coupling format are chosen
// per job.
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) sparse_sell_batch_kernel(const BatchJob* jobs, int njobs,
                                                                       int* cursor)
{
    extern __shared__ __align__(16) float m[];
    __shared__ SlotState<2, NT / 32> S;
    __shared__ BatchJob s_jobcopy;  // the current job's descriptors, read from shared memory
    __shared__ int s_job;
    for (;;) {
        if (threadIdx.x == 0) {
            int j = *((volatile int*)cursor);
            while (j < njobs && *((volatile int*)jobs[j].s.work_counter) >= jobs[j].s.R) {
                atomicMax(cursor, j + 1);
                ++j;
            }
            s_job = j < njobs ? j : -1;
        }
        __syncthreads();
        const int j = s_job;
        if (j < 0) break;
        {
            const int* src = reinterpret_cast<const int*>(jobs + j);
            int* dst = reinterpret_cast<int*>(&s_jobcopy);
            for (int w = threadIdx.x; w < (int)(sizeof(BatchJob) / sizeof(int)); w += blockDim.x)
                dst[w] = src[w];
        }
        __syncthreads();
        run_batch_job<NT>(s_jobcopy, m, S);
        __syncthreads();
    }
}

// Persistent serving kernel: CTAs take replicas from the jobs published in the
// ring, oldest first; when none is left, thread 0 polls the ring's tail
// (about 2 us apart, at most idle_polls times) and the CTA exits when nothing
// new arrives. Descriptors written by the host's copies are read through
// volatile loads (past L1), after the tail that published them. Several launches
// may work on one ring: a CTA inside a long replica outlives the others' idle
// time, and the host replaces those (serve_ring_ensure_kernel).
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) serve_ring_kernel(ServeRing* ring, int idle_polls, int32_t* passed,
                                                                  int32_t* gone)
{
    extern __shared__ __align__(16) float m[];
    __shared__ SlotState<2, NT / 32> S;
    __shared__ BatchJob s_jobcopy;
    __shared__ int s_job;
    for (;;) {
        if (threadIdx.x == 0) {
            int found = -1;
            for (int poll = 0; poll <= idle_polls; ++poll) {
                int c = *reinterpret_cast<volatile int*>(&ring->cursor);
                const int tail = *reinterpret_cast<volatile int*>(&ring->tail);
                __threadfence();
                while (c < tail) {
                    const int k = c % kRingCap;
                    const int taken = *reinterpret_cast<volatile int*>(&ring->slots[k].taken);
                    const int R = *reinterpret_cast<volatile int*>(&ring->jobs[k].s.R);
                    if (taken < R) break;
                    atomicMax(&ring->cursor, c + 1);
                    *reinterpret_cast<volatile int*>(passed + k) = 1;
                    ++c;
                }
                if (c < tail) {
                    found = c;
                    break;
                }
                if (*reinterpret_cast<volatile int*>(&ring->stop)) break;
                __nanosleep(2000);
            }
            s_job = found;
        }
        __syncthreads();
        const int j = s_job;
        if (j < 0) break;
        {
            const volatile int* src = reinterpret_cast<const volatile int*>(ring->jobs + j % kRingCap);
            int* dst = reinterpret_cast<int*>(&s_jobcopy);
            for (int w = threadIdx.x; w < (int)(sizeof(BatchJob) / sizeof(int)); w += blockDim.x)
                dst[w] = src[w];
        }
        __syncthreads();
        run_batch_job<NT>(s_jobcopy, m, S);
        __syncthreads();
    }
    if (threadIdx.x == 0) *reinterpret_cast<volatile int*>(gone + blockIdx.x) = 1;
}

}  // namespace

namespace {
const void* pick_batch(int nt)
{
    return nt == 1024 ? (const void*)sparse_sell_batch_kernel<1024> : (const void*)sparse_sell_batch_kernel<512>;
}
}  // namespace

// Launch shape of a batch: per job its slots per CTA (one with few replicas,
// as in a solve of its own; else two, where two replicas' magnetisations fit on
// chip: six graphs and lattices of 64 to 512 replicas took 107 ms with two
// slots each and 62 with one) and its coupling format; shared memory of the
// most demanding job.
bool plan_sparse_batch(const DevInstance* ins, const int* reps, const bool* even, int count, int device, BatchPlan* p,
                       int* fmts, int* rts)
{
    int sms = 1, optin = 48 * 1024;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    const size_t budget = (size_t)optin - kKeepSmem;
    const int rt_set = env_int("MARS_SELL_RT", -1);
    int nt = env_int("MARS_SELL_THREADS", 1024);
    if (nt != 512 && nt != 1024) nt = 1024;
    auto m_bytes = [&](int n, int c) { return align16((size_t)(n + 1) * c * sizeof(float)); };
    size_t smem = 0;
    for (int j = 0; j < count; ++j) {
        const DevInstance& in = ins[j];
        if (in.dense || !in.slices || (!in.sell_pm1 && !in.sell_gen)) return false;
        int rt = rt_set >= 0 ? (rt_set >= 2 ? 2 : 1) : few_replicas(in, reps[j], sms, even[j], nt) ? 1 : 2;
        while (rt > 1 && m_bytes(in.n, rt) > budget) rt /= 2;
        if (m_bytes(in.n, rt) > budget) return false;
        const size_t table = half_table_bytes(in);
        int fmt = in.sell_pm1 ? 1 : 0;
        if (in.sell16) fmt = 3;
        if (in.sell16 && env_int("MARS_SELL_SMEM_TABLE", 1) && m_bytes(in.n, rt) + table <= budget) fmt = 2;
        fmts[j] = fmt;
        rts[j] = rt;
        smem = std::max(smem, m_bytes(in.n, rt) + (fmt == 2 ? table : 0));
    }
    p->rt = 2;
    p->threads = nt;
    p->smem = smem;
    const void* k = pick_batch(nt);
    allow_smem(k, kKeepSmem);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nt, smem);
    p->grid = sms * std::max(per_sm, 1);
    return true;
}

cudaError_t launch_sparse_batch(const BatchJob* jobs, int count, int* cursor, const BatchPlan& p,
                                cudaStream_t st)
{
    const void* k = pick_batch(p.threads);
    cudaError_t e = allow_smem(k, kKeepSmem);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&jobs, (void*)&count, (void*)&cursor};
    return cudaLaunchKernel(k, dim3(p.grid), dim3(p.threads), args, p.smem, st);
}

bool plan_serve_ring(int device, RingPlan* p)
{
    int sms = 1, optin = 48 * 1024;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    p->rt = 2;
    p->threads = 1024;
    p->smem = (size_t)optin - kKeepSmem;
    const void* k = (const void*)serve_ring_kernel<1024>;
    if (allow_smem(k, kKeepSmem) != cudaSuccess) return false;
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, p->threads, p->smem);
    p->grid = sms * std::max(per_sm, 1);
    return true;
}

int ring_job_format(const DevInstance& in, const RingPlan& p, int* rt)
{
    if (in.dense || !in.slices || (!in.sell_pm1 && !in.sell_gen)) return -1;
    auto m_bytes = [&](int c) { return align16((size_t)(in.n + 1) * c * sizeof(float)); };
    *rt = m_bytes(2) <= p.smem ? 2 : 1;
    const size_t mb = m_bytes(*rt);
    if (mb > p.smem) return -1;
    const size_t table = half_table_bytes(in);
    if (in.sell16 && mb + table <= p.smem) return 2;
    if (in.sell16) return 3;
    return in.sell_pm1 ? 1 : 0;
}

cudaError_t launch_serve_ring(ServeRing* ring, const RingPlan& p, int ctas, int idle_polls, int32_t* passed,
                              int32_t* gone, cudaStream_t st)
{
    if (p.threads != 1024) return cudaErrorInvalidValue;
    const void* k = (const void*)serve_ring_kernel<1024>;
    cudaError_t e = allow_smem(k, kKeepSmem);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&ring, (void*)&idle_polls, (void*)&passed, (void*)&gone};
    return cudaLaunchKernel(k, dim3(ctas), dim3(p.threads), args, p.smem, st);
}

}  // namespace mars
