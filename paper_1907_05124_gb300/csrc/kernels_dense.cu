// Dense MARS descent (Section 3, Algorithm 1) in FP32 on the SIMT cores.
//
// One warp carries one replica through the whole descent. A sweep visits the
// spins one after another (Gauss-Seidel: every spin shares a coupling with
// every other, so there is no parallelism inside one replica's sweep); the
// warp spreads each local field Phi_a = sum_b J_ab s_b over its 32 lanes and
// reduces it with shuffles, in compensated arithmetic (see Dot2). The
// replicas' magnetisations stay in shared memory. J is copied there as a whole
// when it fits, else row by row, once per CTA (dense_staged_kernel); beyond
// that every warp reads it through the read-only cache. Synchronous sweeps give
// a replica several warps (dense_sync_kernel). This is the plain FP32 path the
// tensor-core path is checked against.
#include "device_common.cuh"
#include "schedule.cuh"
#include "tc_primitives.cuh"
#include "mars_internal.h"

#include <algorithm>

namespace mars {
namespace {

constexpr int kDenseWarps = 4;
// Row buffers of the staged kernel's ring (fewer when shared memory is short;
// 16 instead of 4 were no faster at n = 256 and 512).
constexpr int kMaxStages = 4;

// Compensated dot product (Ogita, Rump, Oishi, "Accurate sum and dot
// product", SIAM J. Sci. Comput. 2005, algorithm Dot2): every product's
// rounding error comes from an FMA, every sum's from TwoSum, and the errors
// are carried in a second float. The result is as accurate as a dot product
// evaluated in twice the working precision and then rounded, so the local
// field of a dense row does not lose ulps to a 32-lane tree of n terms.
// Explicit-rounding intrinsics keep the compiler from fusing the error terms.
struct Dot2 {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add_product(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        const float pe = __fmaf_rn(a, b, -p);
        add_pair(p, pe);
    }
    __device__ __forceinline__ void add_pair(float v, float err)
    {
        const float t = __fadd_rn(s, v);
        const float z = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z));
        s = t;
        c = __fadd_rn(c, __fadd_rn(e, err));
    }
    __device__ __forceinline__ float warp_total()
    {
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            const float s2 = __shfl_xor_sync(0xffffffffu, s, m);
            const float c2 = __shfl_xor_sync(0xffffffffu, c, m);
            add_pair(s2, c2);
        }
        return __fadd_rn(s, c);
    }
};


// Two Dot2 sums side by side, every operation on both in one instruction
// (packed FP32); each half's values are Dot2's. Where Dot2's issue is the bound
// this takes 3 to 12 % less time (synchronous n = 4096 491 against 558 ns a
// spin); with one warp per scheduler it is 1 to 5 % slower.
struct Dot2x2 {
    float2 s = {0.f, 0.f}, c = {0.f, 0.f};
    __device__ __forceinline__ void add_product(float2 a, float2 b)
    {
        const float2 p = mul2(a, b);
        add_pair(p, fma2(a, b, mul2(p, make_float2(-1.f, -1.f))));
    }
    __device__ __forceinline__ void add_pair(float2 v, float2 err)
    {
        const float2 t = add2(s, v);
        const float2 z = sub2(t, s);
        const float2 e = add2(sub2(s, sub2(t, z)), sub2(v, z));
        s = t;
        c = add2(c, add2(e, err));
    }
};

template <bool LDG>
__device__ __forceinline__ float4 load4(const float4* p)
{
    if constexpr (LDG) return __ldg(p);
    return *p;
}

// Phi_a = sum_b J_ab m_b (+ h_a) of one row over the warp. Four Dot2 sums, one
// per float4 component (two packed pairs), and two float4 loads per lane per
// step keep several loads in flight; the sums and then the lanes are merged
// with the same error-free additions, so the result keeps Dot2's accuracy.
// n4 = n / 4 when the row and m are 16-byte aligned, else 0 (scalar loop). LDG:
// the row is in global memory (read-only path), else in shared memory.
template <bool LDG>
__device__ __forceinline__ float row_field(const float* __restrict__ Jrow, const float* m, int n,
                                           int n4, int lane, float h)
{
    Dot2x2 lo, hi;  // components x, y and z, w
    const float4* J4 = reinterpret_cast<const float4*>(Jrow);
    const float4* m4 = reinterpret_cast<const float4*>(m);
    int k = lane;
#pragma unroll 2
    for (; k + 32 < n4; k += 64) {
        const float4 j0 = load4<LDG>(J4 + k), j1 = load4<LDG>(J4 + k + 32);
        const float4 x0 = m4[k], x1 = m4[k + 32];
        lo.add_product(make_float2(j0.x, j0.y), make_float2(x0.x, x0.y));
        hi.add_product(make_float2(j0.z, j0.w), make_float2(x0.z, x0.w));
        lo.add_product(make_float2(j1.x, j1.y), make_float2(x1.x, x1.y));
        hi.add_product(make_float2(j1.z, j1.w), make_float2(x1.z, x1.w));
    }
    if (k < n4) {
        const float4 j0 = load4<LDG>(J4 + k);
        const float4 x0 = m4[k];
        lo.add_product(make_float2(j0.x, j0.y), make_float2(x0.x, x0.y));
        hi.add_product(make_float2(j0.z, j0.w), make_float2(x0.z, x0.w));
    }
    Dot2 acc[2];
    acc[0].s = lo.s.x;
    acc[0].c = lo.c.x;
    acc[1].s = hi.s.x;
    acc[1].c = hi.c.x;
#pragma unroll 4
    for (int b = 4 * n4 + lane; b < n; b += 32)
        acc[0].add_product(LDG ? __ldg(Jrow + b) : Jrow[b], m[b]);
    acc[0].add_pair(h, 0.f);
    acc[0].add_pair(lo.s.y, lo.c.y);
    acc[1].add_pair(hi.s.y, hi.c.y);
    acc[0].add_pair(acc[1].s, acc[1].c);
    return acc[0].warp_total();
}

// One replica's place in the schedule (Algorithm 1's outer loop, schedule.cuh).
struct Level {
    double T = 0.0;
    float invT = 0.f;
    bool act = false;
    int levels = 0, sweeps = 0, capped = 0, lvl_sweeps = 0;

    // the first level, or the given one (the FP32 polish)
    __device__ void start(const DevSolve& s, int r)
    {
        if (s.t_first) {
            T = s.t_first[r];
            act = T > 0.0;
        } else {
            act = sched_first(s, (double)s.t0[r], &T);
        }
        invT = act ? sched_inv_t(T) : 0.f;
        levels = act ? 1 : 0;
    }
    // after a sweep whose largest change was d: stay, cool, or stop
    __device__ void after_sweep(const DevSolve& s, float d)
    {
        ++sweeps;
        ++lvl_sweeps;
        const bool fixed = sched_fixed(s, T);
        const bool level_done = fixed ? lvl_sweeps >= s.fixed_sweeps : (d <= s.d_min || lvl_sweeps >= s.k_max);
        if (!level_done) return;
        if (!fixed && !(d <= s.d_min)) ++capped;
        lvl_sweeps = 0;
        if (!s.one_level && sched_advance(s, &T)) {
            ++levels;
            invT = sched_inv_t(T);
        } else {
            act = false;
        }
    }
};

// Noisy mean-field annealing after a synchronous sweep that left the raw
// field Phi_a = sum_b J_ab s_b + h_a of every spin in phi[a]: each lane updates
// its spins a = first, first + step, ... with the normalised field and its noise
// (iteration lv.sweeps of replica r), s_a <- alpha shat_a + (1 - alpha) s_a.
// Returns the sweep's largest change (every lane).
__device__ float nmfa_finish_sweep(const DevInstance& in, const DevSolve& s, int r, const Level& lv,
                                   float* m, const float* phi, int first, int step)
{
    float d = 0.f;
    for (int a = first; a < in.n; a += step) {
        const float xi = s.nmfa_sigma > 0.f
                             ? nmfa_normal(s.seed, s.stream, (uint32_t)r, (uint32_t)lv.sweeps,
                                           (uint32_t)__ldg(in.new2old + a))
                             : 0.f;
        const float v = nmfa_update(phi[a], __ldg(in.inv_norm + a), xi, s.nmfa_sigma, lv.invT,
                                    s.nmfa_alpha, m[a]);
        d = fmaxf(d, fabsf(v - m[a]));
        m[a] = v;
    }
    return warp_reduce_strided<1>(d, MaxOp());
}

__device__ __forceinline__ void init_m(const DevInstance& in, const DevSolve& s, int r, float* m,
                                       int lane)
{
    const int n = in.n;
    for (int a = lane; a < n; a += 32) {
        const int o = __ldg(in.new2old + a);
        m[a] = s.m0 ? __ldg(s.m0 + (size_t)r * n + o) : draw_m0(s.seed, s.stream, r, o);
    }
}

// Sign-round, outputs and the replica's energy (pairs a < b once plus the
// field). The lanes stride along row a, so every load of the row is
// coalesced; integer J sums exactly in int64. With skip_energy the library
// evaluates the energies exactly afterwards (launch_energy) and none is summed
// here.
__device__ void finish_replica(const DevInstance& in, const DevSolve& s, int r, const float* m,
                               int lane, const Level& lv)
{
    const int n = in.n;
    for (int a = lane; a < n; a += 32) {
        const int o = __ldg(in.new2old + a);
        s.sigma[(size_t)r * n + o] = (int8_t)(m[a] >= 0.f ? 1 : -1);
        if (s.m_final) s.m_final[(size_t)r * n + o] = m[a];
    }
    long long ei = 0;
    double ef = 0.0;
    for (int a = 0; a < n && !s.skip_energy; ++a) {
        const int sa = m[a] >= 0.f ? 1 : -1;
        if (in.integer) {
            const int8_t* row = in.J_i8 + (size_t)a * n;
            int acc = 0;  // at most n / 32 terms of magnitude <= 128 per lane
            for (int b = a + 1 + lane; b < n; b += 32) acc += m[b] >= 0.f ? (int)row[b] : -(int)row[b];
            ei += (long long)(acc * sa);
            if (in.h && lane == 0) ei += (long long)__ldg(in.h + a) * sa;
        } else {
            const double* row = in.J_f64 + (size_t)a * n;
            double acc = 0.0;
            for (int b = a + 1 + lane; b < n; b += 32) acc += m[b] >= 0.f ? row[b] : -row[b];
            ef += acc * sa;
            if (in.h_f64 && lane == 0) ef += __ldg(in.h_f64 + a) * sa;
        }
    }
    ei = warp_reduce_strided<1>(ei, SumOp());
    ef = warp_reduce_strided<1>(ef, SumOp());
    if (lane == 0) {
        s.energy[r] = in.integer ? (double)ei : ef;
        s.energy_i64[r] = in.integer ? ei : 0;
        if (s.add_counts) {
            s.sweeps[r] += lv.sweeps;
            s.capped[r] += lv.capped;
        } else {
            s.sweeps[r] = lv.sweeps;
            s.levels[r] = lv.levels;
            s.capped[r] = lv.capped;
        }
    }
}

// The next row's cache lines are requested into L1 while this row's field is
// summed (a prefetch is a hint and never faults).
__device__ __forceinline__ void prefetch_row_l1(const float* row, int n, int lane)
{
    for (int o = lane * 32; o < n; o += 32 * 32)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(row + o));
}

// Fallback for n too large for the staged kernel's shared memory: every warp
// reads the rows through the read-only cache, and m lives in shared memory
// (ONCHIP) or in a global scratch row.
template <bool ONCHIP, bool JACOBI>
__global__ void __launch_bounds__(kDenseWarps * 32) dense_descent_kernel(DevInstance in, DevSolve s,
                                                                         int /*stages*/)
{
    extern __shared__ __align__(128) float smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.x * kDenseWarps + warp;
    if (r >= s.R) return;  // whole warp leaves; the kernel has no block barrier
    const int n = in.n;
    // rows (and m) start on 16-byte boundaries when n % 4 == 0: float4 path
    const int n4 = (n & 3) == 0 ? n >> 2 : 0;
    const int per = n * (JACOBI ? 2 : 1);
    float* m = ONCHIP ? smem + (size_t)warp * per : s.m_scratch + (size_t)r * per;
    float* mn = JACOBI ? m + n : m;
    init_m(in, s, r, m, lane);
    __syncwarp();
    Level lv;
    lv.start(s, r);
    while (lv.act) {
        float d = 0.f;
        for (int a = 0; a < n; ++a) {
            prefetch_row_l1(in.Jf + (size_t)(a + 1 < n ? a + 1 : 0) * n, n, lane);
            const float p = row_field<true>(in.Jf + (size_t)a * n, m, n, n4, lane,
                                            in.h && lane == 0 ? __ldg(in.h + a) : 0.f);
            // NMFA keeps the raw field; its update follows the sweep
            const float sn = JACOBI && s.nmfa ? p : -tanhf(p * lv.invT);
            if (!(JACOBI && s.nmfa)) d = fmaxf(d, fabsf(sn - m[a]));
            __syncwarp();
            if (lane == 0) mn[a] = sn;
            __syncwarp();
        }
        if (JACOBI) {
            if (s.nmfa) {
                d = nmfa_finish_sweep(in, s, r, lv, m, mn, lane, 32);
            } else {
                for (int a = lane; a < n; a += 32) m[a] = mn[a];
            }
            __syncwarp();
        }
        // the lanes' merges may differ in the last bit: lane 0's spins were kept
        lv.after_sweep(s, __shfl_sync(0xffffffffu, d, 0));
    }
    finish_replica(in, s, r, m, lane, lv);
}

// Wait for a row stage's barrier phase. Every lane polls; the wait gives up
// when another warp has given up (abort flag) or after kSpinLimit polls, when
// it raises the flag and records the timeout in the status word.
__device__ __forceinline__ bool stage_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                           int32_t* status)
{
    for (uint32_t i = 0; i < tc::kSpinLimit; ++i) {
        if (tc::mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    atomicExch(status, tc::kErrTimeout);
    return false;
}

// One spin of a replica's sweep: its new value from row a (in shared memory),
// or the raw field for NMFA, whose update follows the sweep.
template <bool JACOBI>
__device__ __forceinline__ void sweep_spin(const DevInstance& in, const DevSolve& s, const Level& lv, const float* row,
                                           const float* m, float* mn, int a, int n4, int lane, float& d)
{
    const float p = row_field<false>(row, m, in.n, n4, lane, in.h && lane == 0 ? __ldg(in.h + a) : 0.f);
    const float sn = JACOBI && s.nmfa ? p : -tanhf(p * lv.invT);
    if (!(JACOBI && s.nmfa)) d = fmaxf(d, fabsf(sn - m[a]));
    __syncwarp();
    if (lane == 0) mn[a] = sn;
}

// The end of a replica's synchronous sweep: the new state becomes the state.
__device__ __forceinline__ void finish_jacobi(const DevInstance& in, const DevSolve& s, int r, const Level& lv, float* m,
                                              const float* mn, int lane, float& d)
{
    if (s.nmfa) {
        d = nmfa_finish_sweep(in, s, r, lv, m, mn, lane, 32);
    } else {
        for (int a = lane; a < in.n; a += 32) m[a] = mn[a];
    }
    __syncwarp();
}

// A row buffer of the ring: row a starts (a n) mod 4 floats into it, where the
// 16-byte pieces that hold the row begin (bulk copies move whole pieces; J is
// padded by one).
__host__ __device__ inline int row_floats(int n) { return (n & 3) == 0 ? n : ((n + 3) & ~3) + 4; }
__device__ __forceinline__ int row_shift(int a, int n) { return (int)(((unsigned)a * (unsigned)n) & 3u); }
__device__ __forceinline__ void load_row(float* buf, const float* J, int a, int n, uint64_t* full)
{
    const int sh = row_shift(a, n);
    const uint32_t bytes = (uint32_t)((sh + n + 3) & ~3) * sizeof(float);
    tc::mbar_arrive_expect_tx(full, bytes);
    tc::bulk_load(buf, J + ((size_t)a * n - sh), bytes, full);
}

// Staged kernel: each row J[a,:] is fetched into shared memory once per CTA.
// RESIDENT (`stages` == n): all of J stays there and every warp runs its
// replica's sweeps by itself. Otherwise the kDenseWarps replicas of a CTA sweep
// the spins in lockstep and the rows pass through a ring of `stages` buffers,
// filled by bulk copies (cp.async.bulk, completion on a `full` mbarrier per
// stage); every warp releases a stage on its `empty` mbarrier once its field is
// summed, and a fifth warp refills it with the row `stages` spins ahead (a
// replica's warp that did so held the others up at every spin). The rows wrap
// from n - 1 to 0, so the pipeline runs across sweeps; the CTA stops when none
// of its replicas is active and drains the copies still in flight before it
// exits. Warps past R take part in the pipeline only.
//
// What bounds it: with one warp per scheduler, a spin's latency (the row's Dot2
// terms, the 5-level merge of the lanes, tanhf), not the copies; from n of
// about 2048, or several warps per scheduler, Dot2's issue. Time per spin on a
// GB300, ns: all of J on chip, n = 64, R = 256 305 (593 through the ring with a
// replica's warp refilling it); ring, n = 256, R = 512 524 (695), n = 1024,
// R = 256 826 (1080), n = 4096, R = 512 1967 (4682).
template <bool JACOBI, bool RESIDENT>
__global__ void __launch_bounds__((kDenseWarps + 1) * 32) dense_staged_kernel(DevInstance in, DevSolve s,
                                                                        int stages)
{
    extern __shared__ __align__(128) float smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.x * kDenseWarps + warp;
    const bool live = warp < kDenseWarps && r < s.R;
    const int n = in.n, n4 = (n & 3) == 0 ? n >> 2 : 0;
    const int per = n * (JACOBI ? 2 : 1), rb = row_floats(n);
    constexpr bool resident = RESIDENT;  // stages == n
    const size_t jfloats = resident ? ((size_t)n * n + 3) & ~(size_t)3 : (size_t)stages * rb;
    float* rows = smem;
    float* m = smem + jfloats + (size_t)warp * per;
    float* mn = JACOBI ? m + n : m;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + jfloats + (size_t)kDenseWarps * per);
    uint64_t* empty = full + stages;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + stages);

    if (threadIdx.x == 0) {
        for (int k = 0; k < (resident ? 1 : stages); ++k) {
            tc::mbar_init(&full[k], 1);
            tc::mbar_init(&empty[k], kDenseWarps);
        }
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (resident) {  // all rows on one barrier
            const uint32_t bytes = (uint32_t)jfloats * sizeof(float);
            tc::mbar_arrive_expect_tx(&full[0], bytes);
            tc::bulk_load(rows, in.Jf, bytes, &full[0]);
        } else {
            for (int k = 0; k < stages; ++k) load_row(rows + (size_t)k * rb, in.Jf, k, n, &full[k]);
        }
    }
    Level lv;
    if (live) {
        init_m(in, s, r, m, lane);
        lv.start(s, r);
    }
    __syncwarp();

    if constexpr (resident) {
        const bool ok = stage_wait(&full[0], 0, abort_flag, s.status);
        if (__syncthreads_and(ok)) {
            while (lv.act) {
                float d = 0.f;
                for (int a = 0; a < n; ++a) {
                    sweep_spin<JACOBI>(in, s, lv, rows + (size_t)a * n, m, mn, a, n4, lane, d);
                    __syncwarp();
                }
                if (JACOBI) finish_jacobi(in, s, r, lv, m, mn, lane, d);
                lv.after_sweep(s, __shfl_sync(0xffffffffu, d, 0));  // lane 0's spins were kept
            }
        }
        if (live) finish_replica(in, s, r, m, lane, lv);
        return;
    }
    int st = 0;        // stage of the next row to consume
    uint32_t ph = 0;   // its barrier parity
    auto next_stage = [&]() {
        if (++st == stages) {
            st = 0;
            ph ^= 1u;
        }
    };
    bool any = __syncthreads_or(lv.act) != 0;
    while (any) {
        float d = 0.f;
        if (warp == kDenseWarps) {  // the producer: row a's buffer takes the row `stages` after it
            if (lane == 0)  // whose st and ph alone follow
                for (int a = 0; a < n; ++a) {
                    if (!stage_wait(&empty[st], ph, abort_flag, s.status)) break;
                    const int next = a + stages < n ? a + stages : a + stages - n;
                    load_row(rows + (size_t)st * rb, in.Jf, next, n, &full[st]);
                    next_stage();
                }
            __syncwarp();
        } else {
            for (int a = 0; a < n; ++a) {
                if (!__all_sync(0xffffffffu, stage_wait(&full[st], ph, abort_flag, s.status))) break;
                if (lv.act)
                    sweep_spin<JACOBI>(in, s, lv, rows + (size_t)st * rb + row_shift(a, n), m, mn, a, n4, lane, d);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&empty[st]);
                next_stage();
            }
        }
        if (JACOBI && lv.act) finish_jacobi(in, s, r, lv, m, mn, lane, d);
        if (lv.act) lv.after_sweep(s, __shfl_sync(0xffffffffu, d, 0));  // lane 0's spins were kept
        any = __syncthreads_or(lv.act) != 0 && !*abort_flag;
    }
    // the last copy into each buffer: up to `stages` are ahead of the last row
    // consumed, and after a timeout too none may land in an exited CTA's memory
    if (warp == kDenseWarps && lane == 0)
        for (int q = 0; q < stages; ++q) tc::mbar_wait(&full[q], q < st ? ph ^ 1u : ph, s.status);
    __syncthreads();
    if (live) finish_replica(in, s, r, m, lane, lv);
}

// Synchronous sweeps: every spin's field comes from the same
// state, so the spins of a replica are summed by several warps at once. A CTA
// carries REPS replicas and 16 / REPS warps for each; warp (ph, rep) takes the
// rows ph, ph + 16 / REPS, ... of its replica, so a row is read from shared
// memory by the REPS warps that need it, and a seventeenth warp keeps the ring
// of row buffers filled. With one warp per replica (the staged kernel above)
// the same sweeps ran at one warp per scheduler: n = 1024, R = 400 took 1.09 us a
// spin on a GB300, and 0.36 here; n = 4096, R = 256 4.6, and 0.49.
//
// A row's `full` barrier goes by its number modulo sync_barriers, a multiple of
// the warps per replica, not by its buffer: a wait by parity is sound only for
// one who has seen the barrier's fill before, and with that count the row before
// on a barrier was the same warp's. (With one barrier per buffer it was another
// warp's row whenever the buffers were no multiple of the warps: a warp could
// take the barrier's last but one fill for its own, and with fewer buffers than
// warps always did.)
constexpr int kSyncWarps = 16;

// At least one barrier per buffer, so that a barrier's last row has been read
// before the producer arms it again.
__host__ __device__ constexpr int sync_barriers(int stages, int reps)
{
    const int phases = kSyncWarps / reps;
    return (stages + phases - 1) / phases * phases;
}

template <int REPS>
__global__ void __launch_bounds__((kSyncWarps + 1) * 32) dense_sync_kernel(DevInstance in, DevSolve s, int stages)
{
    constexpr int kPhases = kSyncWarps / REPS;
    extern __shared__ __align__(128) float smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rep = warp % REPS, phase = warp / REPS;
    const int r = blockIdx.x * REPS + rep;
    const bool worker = warp < kSyncWarps, live = worker && r < s.R;
    const int n = in.n, n4 = (n & 3) == 0 ? n >> 2 : 0, rb = row_floats(n);
    float* rows = smem;
    float* m = smem + (size_t)stages * rb + (size_t)rep * 2 * n;
    float* mn = m + n;
    const int bars = sync_barriers(stages, REPS);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)stages * rb + (size_t)REPS * 2 * n);
    uint64_t* empty = full + bars;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + stages);
    __shared__ float s_d[REPS][kPhases];
    if (threadIdx.x == 0) {
        for (int k = 0; k < bars; ++k) tc::mbar_init(&full[k], 1);
        for (int k = 0; k < stages; ++k) tc::mbar_init(&empty[k], REPS);  // the warps of the row's phase
        *abort_flag = 0;
        tc::fence_barrier_init();
    }
    Level lv;
    if (live) {
        for (int a = phase * 32 + lane; a < n; a += 32 * kPhases) {
            const int o = __ldg(in.new2old + a);
            m[a] = s.m0 ? __ldg(s.m0 + (size_t)r * n + o) : draw_m0(s.seed, s.stream, r, o);
        }
        lv.start(s, r);
    }
    bool any = __syncthreads_or(lv.act) != 0;
    int st = 0, fb = 0;         // buffer and `full` barrier of row 0 of the next sweep
    uint32_t ph = 0, fp = 0;    // and their parities
    // a sweep's turns through both, and a worker's way from row to row: no division
    // inside the sweeps
    const int n_st = n % stages, n_fb = n % bars, phase_st = phase % stages, step_st = kPhases % stages;
    const uint32_t t_st = (uint32_t)(n / stages), t_fb = (uint32_t)(n / bars);
    int issued = 0, fb0 = 0;    // the producer: the sweep's rows issued, and where they began
    uint32_t fp0 = 0;
    bool first = true;
    while (any) {
        float d = 0.f;
        if (!worker) {
            // the producer: rows 0 .. n - 1, each once its buffer's last row has
            // been read (the first `stages` rows find theirs empty)
            int q = st, b = fb;
            uint32_t qp = ph;
            fb0 = fb;
            fp0 = fp;
            issued = 0;
            if (lane == 0) {
                for (int a = 0; a < n; ++a) {
                    if (!(first && a < stages) && !stage_wait(&empty[q], qp ^ 1u, abort_flag, s.status)) break;
                    load_row(rows + (size_t)q * rb, in.Jf, a, n, &full[b]);
                    issued = a + 1;
                    if (++q == stages) {
                        q = 0;
                        qp ^= 1u;
                    }
                    if (++b == bars) b = 0;
                }
            }
            __syncwarp();
        } else {
            int q = st + phase_st, b = fb + phase;
            uint32_t bp = fp;
            if (q >= stages) q -= stages;
            if (b >= bars) {
                b -= bars;
                bp ^= 1u;
            }
            for (int a = phase; a < n; a += kPhases) {
                if (!__all_sync(0xffffffffu, stage_wait(&full[b], bp, abort_flag, s.status))) break;
                if (lv.act)
                    sweep_spin<true>(in, s, lv, rows + (size_t)q * rb + row_shift(a, n), m, mn, a, n4, lane, d);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&empty[q]);
                q += step_st;
                if (q >= stages) q -= stages;
                b += kPhases;
                if (b >= bars) {
                    b -= bars;
                    bp ^= 1u;
                }
            }
        }
        st += n_st;
        ph ^= (t_st + (st >= stages)) & 1u;
        if (st >= stages) st -= stages;
        fb += n_fb;
        fp ^= (t_fb + (fb >= bars)) & 1u;
        if (fb >= bars) fb -= bars;
        first = false;
        __syncthreads();  // every row of the sweep has been read, every field written
        if (lv.act) {
            const int at = phase * 32 + lane, step = 32 * kPhases;
            if (s.nmfa) {
                d = nmfa_finish_sweep(in, s, r, lv, m, mn, at, step);
            } else {
                for (int a = at; a < n; a += step) m[a] = mn[a];
            }
            if (lane == 0) s_d[rep][phase] = d;
        }
        any = __syncthreads_or(*abort_flag) == 0;
        if (lv.act) {
            float dd = 0.f;
#pragma unroll
            for (int k = 0; k < kPhases; ++k) dd = fmaxf(dd, s_d[rep][k]);
            lv.after_sweep(s, dd);
        }
        any = __syncthreads_or(lv.act) != 0 && any;
    }
    // No copy is in flight: every row of the last sweep was read. After a timeout it
    // was not, and none may land in an exited CTA's memory.
    if (warp == kSyncWarps && lane == 0 && *abort_flag)
        for (int k = max(issued - stages, 0); k < issued; ++k)
            tc::mbar_wait(&full[(fb0 + k) % bars], fp0 ^ (uint32_t)((fb0 + k) / bars & 1), s.status);
    __syncthreads();
    if (live && phase == 0) finish_replica(in, s, r, m, lane, lv);
}

// What the plan leaves of a block's shared memory (allow_smem).
int keep_smem(const DensePlan& p) { return p.sync_reps ? 2048 : p.stages ? 0 : 4096; }

const void* pick(const DensePlan& p, bool jacobi)
{
    if (p.sync_reps)
        return p.sync_reps == 4 ? (const void*)dense_sync_kernel<4>
             : p.sync_reps == 2 ? (const void*)dense_sync_kernel<2>
                                : (const void*)dense_sync_kernel<1>;
    if (p.stages && p.resident)
        return jacobi ? (const void*)dense_staged_kernel<true, true> : (const void*)dense_staged_kernel<false, true>;
    if (p.stages)
        return jacobi ? (const void*)dense_staged_kernel<true, false> : (const void*)dense_staged_kernel<false, false>;
    if (p.onchip) return jacobi ? (const void*)dense_descent_kernel<true, true>
                                : (const void*)dense_descent_kernel<true, false>;
    return jacobi ? (const void*)dense_descent_kernel<false, true>
                  : (const void*)dense_descent_kernel<false, false>;
}

}  // namespace

DensePlan plan_dense(const DevInstance& in, int R, int jacobi, int device)
{
    int optin = 48 * 1024;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    DensePlan p;
    p.warps_per_block = kDenseWarps;
    p.grid = (R + kDenseWarps - 1) / kDenseWarps;
    const size_t per_warp = (size_t)in.n * sizeof(float) * (jacobi ? 2 : 1);
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    const int rb = row_floats(in.n);
    if (jacobi && in.n >= 64) {
        // Several warps per replica: the fewer replicas, the more of them.
        // Rows under way: two per phase (16 kB at least) where they fit.
        const int reps = R >= 2 * sms ? 4 : R >= sms ? 2 : 1;
        auto bytes = [&](int stages) {
            return ((size_t)stages * rb + (size_t)2 * reps * in.n) * sizeof(float) +
                   (sync_barriers(stages, reps) + stages) * sizeof(uint64_t) + 16;
        };
        int stages = std::min(2 * kSyncWarps / reps, in.n);
        while (stages > 2 && bytes(stages) + 2048 > (size_t)optin) --stages;
        if (bytes(stages) + 2048 <= (size_t)optin) {
            p.sync_reps = reps;
            p.stages = stages;
            p.smem = bytes(stages);
            p.threads = (kSyncWarps + 1) * 32;
            p.grid = (R + reps - 1) / reps;
            return p;
        }
    }
    {
        auto bytes = [&](int stages) {
            const size_t j = stages == in.n ? ((size_t)in.n * in.n + 3) & ~(size_t)3 : (size_t)stages * rb;
            return j * sizeof(float) + per_warp * kDenseWarps + 2 * stages * sizeof(uint64_t) + 16;
        };
        // All of J on chip when that keeps every CTA resident at once.
        if (bytes(in.n) <= (size_t)optin && p.grid <= sms * (int)((size_t)optin / (bytes(in.n) + 1024)))
            p.stages = in.n;
        for (int stages = std::min(kMaxStages, in.n); stages >= 2 && !p.stages;
             --stages)
            if (bytes(stages) <= (size_t)optin) p.stages = stages;
        if (p.stages) {
            p.resident = p.stages == in.n;
            p.smem = bytes(p.stages);
            p.threads = (kDenseWarps + 1) * 32;
        }
    }
    if (p.stages) return p;
    p.onchip = per_warp * kDenseWarps <= (size_t)optin - 4096;
    p.smem = p.onchip ? per_warp * kDenseWarps : 0;
    p.scratch_floats = p.onchip ? 0 : (size_t)R * in.n * (jacobi ? 2 : 1);
    return p;
}

cudaError_t launch_dense(const DevInstance& in, const DevSolve& s, const DensePlan& p,
                         cudaStream_t st)
{
    const void* k = pick(p, s.jacobi != 0);
    if (p.smem > 48 * 1024) {
        cudaError_t e = allow_smem(k, keep_smem(p));
        if (e != cudaSuccess) return e;
    }
    DevInstance a = in;
    DevSolve b = s;
    int stages = p.stages;
    void* args[] = {&a, &b, &stages};
    return cudaLaunchKernel(k, dim3(p.grid), dim3(p.threads), args, p.smem, st);
}

}  // namespace mars
