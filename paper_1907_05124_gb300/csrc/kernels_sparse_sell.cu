// Sparse MARS descent, fast path: sliced-ELL couplings and on-chip replicas.
//
// Same method and same schedule as kernels_sparse.cu (Section 3, Algorithm 1:
// sequential sweeps reproduced level by level), with a layout built for the
// SM instead of a plain CSR walk:
//
//  * Within a level the runtime sorts spins by degree and cuts them into
//    slices of 32 consecutive new labels (any order inside a level gives the
//    sequential sweep's values, since those spins share no coupling). A
//    slice's couplings are stored slot-major, padded to the slice's largest
//    degree: entry d of row q sits at off + 32*d + q. A warp walks one slice,
//    lane q owns row q, and each of its loads is one coalesced 128-byte line.
//    Padding points at a dummy spin whose magnetisation is held at 0.
//  * +-1 couplings are one 32-bit word: column | sign bit. General weights
//    are a (column, value) pair.
//  * A thread owns one spin for all RT replicas of the tile: one coupling
//    load, one RT-wide shared-memory gather, RT multiply-adds.
//
// The tile's magnetisations m[i*RT + k] live in shared memory for the whole
// descent; the dummy row n is zero. Only the sweeps' parallel steps need a
// block barrier. When not even one replica's m fits on chip, the same job
// runs with m in a global-memory slab per CTA (kernels_sparse_slab.cu).
#include "sell_job.cuh"

#include <algorithm>
#include <cstdlib>

namespace mars {
namespace {

constexpr int kKeepSmem = 12 * 1024;  // of a block's shared memory, for the static part (allow_smem)

template <int RT, int NT, int FMT, int DEG>
__global__ void __launch_bounds__(NT, 1024 / NT) sparse_sell_kernel(DevInstance in, DevSolve s)
{
    extern __shared__ __align__(16) float m[];  // (n+1)*RT, then the staged table (FMT 2)
    __shared__ SlotState<RT, NT / 32> S;
    run_job<RT, NT, FMT, DEG>(in, s, m, S);
}

template <int RT, int NT>
const void* pick_nt(int fmt, int deg)
{
    if (fmt == 2)
        return deg == 4 ? (const void*)sparse_sell_kernel<RT, NT, 2, 4>
             : deg == 6 ? (const void*)sparse_sell_kernel<RT, NT, 2, 6>
                        : (const void*)sparse_sell_kernel<RT, NT, 2, 0>;
    if (fmt == 0) return (const void*)sparse_sell_kernel<RT, NT, 0, 0>;
    if constexpr (NT >= 512) {
        if constexpr (NT == 1024) {
            if (deg == 4 || deg == 6) {
                if (fmt == 3)
                    return deg == 4 ? (const void*)sparse_sell_kernel<RT, NT, 3, 4>
                                    : (const void*)sparse_sell_kernel<RT, NT, 3, 6>;
                return deg == 4 ? (const void*)sparse_sell_kernel<RT, NT, 1, 4>
                                : (const void*)sparse_sell_kernel<RT, NT, 1, 6>;
            }
        }
        return fmt == 3 ? (const void*)sparse_sell_kernel<RT, NT, 3, 0> : (const void*)sparse_sell_kernel<RT, NT, 1, 0>;
    }
    return nullptr;
}

// Regular instances of degree 4 or 6 (square and cubic lattices) get a fully
// unrolled coupling loop. CTAs of 128 and 256 threads take the formats that
// small instances have (0 and 2) and one or two slots.
const void* pick(int rt, int nt, int fmt, int deg)
{
    switch (nt) {
    case 128: return rt == 1 ? pick_nt<1, 128>(fmt, deg) : rt == 2 ? pick_nt<2, 128>(fmt, deg) : nullptr;
    case 256: return rt == 1 ? pick_nt<1, 256>(fmt, deg) : rt == 2 ? pick_nt<2, 256>(fmt, deg) : nullptr;
    case 512: return rt == 1 ? pick_nt<1, 512>(fmt, deg) : rt == 2 ? pick_nt<2, 512>(fmt, deg) : pick_nt<4, 512>(fmt, deg);
    case 1024:
        return rt == 1 ? pick_nt<1, 1024>(fmt, deg) : rt == 2 ? pick_nt<2, 1024>(fmt, deg) : pick_nt<4, 1024>(fmt, deg);
    }
    return nullptr;
}

}  // namespace

// Launch shape: replica slots per CTA (RT) and threads per CTA.
//
// Slots: two amortise the coupling loads, one ends sooner. A solve lasts as long as
// its longest replica, which two slots slow down, until there are so many replicas,
// or replicas so even (fixed sweeps, a low k_max), that it is bound by all of them.
// Descents on a GB300, ms with one / two slots, k_max = 1000: 2-D L = 64, R = 320
// 2.39 / 2.72, R = 512 2.69 / 2.87, R = 600 3.00 / 2.88; L = 100, R = 512 6.03 / 6.53;
// 3-D L = 21, R = 320 10.4 / 12.9, R = 512 13.9 / 13.3; random graphs n = 20000 of
// degree 6, R = 320 66 / 74, R = 512 79 / 76; degree 24, n = 5000, R = 320 85 / 100.
// The degree-6 graph with k_max = 100: R = 320 9.4 / 10.4, R = 400 11.8 / 10.8,
// R = 512 14.9 / 11.0; three fixed sweeps, R = 456: 0.70 / 0.52. Even replicas of small
// instances are bound by latency as long as an SM has few threads at work: k_max = 100,
// n = 301, degree 9, R = 512 (430 threads an SM) 1.56 / 1.64; n = 600, degree 6, R = 512
// (860) 1.59 / 1.68; n = 2000, degree 12, R = 320 (1080) 3.34 / 3.16.
//
// Threads: no more than one per spin of the largest level. A sweep of a small
// instance is a few hundred cycles per level, much of it the barrier over
// warps that had nothing to do. R = 64, L = 12, ms with 128 / 256 / 512 / 1024
// threads: 0.274 / 0.286 / 0.321 / 0.394; R = 256, L = 32: 1.72 / 1.10 / 0.87 /
// 1.05; L = 64, R = 320: 6.3 / 3.7 / 2.7 / 2.0. General couplings are read through the
// L1, which shrinks by the shared memory of every CTA the SM can hold: 1024 threads
// instead of 512 leave room for a table of 192 kB (n = 2000, degree 12, R = 64 17.3 /
// 9.7 ms, R = 320 25.8 / 13.2) and cost 1 % where it does not fit (degree 20, 56.0 /
// 56.8); of 128 and 256 threads small instances have the use all the same (n = 1000,
// degree 12, R = 64 7.3 ms with 256, 7.9 with 1024).
//
// The instance's launch shape (mars_autotune, mars_set_shape), else
// MARS_SELL_RT / MARS_SELL_THREADS / MARS_SELL_SMEM_TABLE, override both.
bool plan_sparse_sell(const DevInstance& in, int R, int device, bool even, SparsePlan* p)
{
    if (!in.slices || (!in.sell_pm1 && !in.sell_gen)) return false;
    int sms = 1, optin = 48 * 1024;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    const size_t budget = (size_t)optin - kKeepSmem;
    const LaunchShape& sh = in.shape;
    const int rt_set = sh.sell_rt >= 0 ? sh.sell_rt : env_int("MARS_SELL_RT", -1);
    const int nt_set = sh.sell_threads >= 0 ? sh.sell_threads : env_int("MARS_SELL_THREADS", -1);
    int nt = nt_set;
    if (nt < 0)
        for (nt = 128; nt < 1024 && nt < 32 * in.max_slices;) nt *= 2;
    if (nt_set < 0 && nt == 512 && !in.sell_pm1) nt = 1024;
    int rt = rt_set >= 0 ? rt_set : few_replicas(in, R, sms, even, nt) ? 1 : 2;
    const int smem_table = sh.sell_smem_table >= 0 ? sh.sell_smem_table : env_int("MARS_SELL_SMEM_TABLE", 1);
    if (rt != 1 && rt != 2 && rt != 4) rt = 1;
    if (nt != 512 && nt != 1024 && nt != 256 && nt != 128) nt = 512;
    auto m_bytes = [&](int c) { return align16((size_t)(in.n + 1) * c * sizeof(float)); };
    const size_t table = half_table_bytes(in);
    // Halfword couplings staged on chip when they fit beside the magnetisations.
    int fmt = in.sell_pm1 ? 1 : 0;
    if (in.sell16 && smem_table) {
        int c = rt;
        while (c > 1 && m_bytes(c) + table > budget) c /= 2;
        if (m_bytes(c) + table <= budget) {
            fmt = 2;
            rt = c;
        }
    }
    const int rt_asked = rt_set >= 0 ? rt : 2;
    if (fmt != 2) {
        while (rt > 1 && m_bytes(rt) > budget) rt /= 2;
        if (m_bytes(rt) > budget) {
            // Not even one replica fits on chip: per-CTA slabs of global
            // memory, the asked slot width, one 1024-thread CTA per SM.
            const int sfmt = in.sell_pm1 ? 1 : 0;
            const int sdeg = sfmt == 1 && env_int("MARS_SELL_UNROLL", 1) ? in.regular_deg : 0;
            const void* k = pick_sell_slab(rt_asked, sfmt, sdeg);
            if (!k) return false;
            int per_sm = 1;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 1024, 0);
            p->rt = rt_asked;
            p->onchip = 0;
            p->threads = 1024;
            p->entry = sfmt;
            p->smem = 0;
            p->sell = 1;
            p->deg = sdeg;
            p->grid = std::max(1, std::min((R + rt_asked - 1) / rt_asked, sms * std::max(per_sm, 1)));
            p->scratch_floats = (size_t)p->grid * sell_slab_floats(in.n, rt_asked);
            return true;
        }
        if (in.sell16 && env_int("MARS_SELL_HALF_L1", 1)) fmt = 3;  // halfwords through L1
    }
    if (nt < 512 && (rt > 2 || (fmt != 0 && fmt != 2))) nt = 512;  // pick's small shapes
    p->rt = rt;
    p->onchip = 1;
    p->threads = nt;
    p->entry = fmt;
    p->smem = m_bytes(rt) + (fmt == 2 ? table : 0);
    p->sell = 1;
    const int deg = env_int("MARS_SELL_UNROLL", 1) ? in.regular_deg : 0;
    p->deg = deg;
    const void* k = pick(rt, nt, fmt, deg);
    if (!k) return false;
    allow_smem(k, kKeepSmem);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nt, p->smem);
    if (per_sm < 1) per_sm = 1;
    const int ntiles = (R + rt - 1) / rt;
    p->grid = std::max(1, std::min(ntiles, sms * per_sm));
    p->scratch_floats = 0;
    return true;
}

cudaError_t launch_sparse_sell(const DevInstance& in, const DevSolve& s, const SparsePlan& p,
                               cudaStream_t st)
{
    const void* k = p.onchip ? pick(p.rt, p.threads, p.entry, p.deg) : pick_sell_slab(p.rt, p.entry, p.deg);
    if (!k) return cudaErrorInvalidValue;
    cudaError_t e = allow_smem(k, kKeepSmem);
    if (e != cudaSuccess) return e;
    DevInstance a = in;
    DevSolve b = s;
    void* args[] = {&a, &b};
    return cudaLaunchKernel(k, dim3(p.grid), dim3(p.threads), args, p.smem, st);
}

}  // namespace mars
