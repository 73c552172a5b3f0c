// One sliced-ELL descent job (Section 3, Algorithm 1), shared by the sparse
// kernels: the coupling formats, the RT-wide replica vectors, the per-CTA
// slot bookkeeping and run_job, which drains one instance's replica queue on
// a CTA. The kernels differ only in where the magnetisations m[i*RT + k]
// live: shared memory (kernels_sparse_sell.cu) or a slab of global memory
// per CTA (kernels_sparse_slab.cu); run_job addresses them through a plain
// pointer either way.
#pragma once

#include "best_reduce.cuh"
#include "device_common.cuh"
#include "schedule.cuh"
#include "mars_internal.h"

#include <climits>
#include <cstdlib>

namespace mars {
namespace {


// tanh(x) = sign(x) (1 - 2 / (1 + e^{2|x|})), with e^{2|x|} = 2^{2|x| log2 e}
// from the SFU's ex2.approx and the quotient from its rcp.approx. Absolute
// error below 2.5e-7 over all of R (checked against FP64 tanh through the C
// ABI by the fields-only test); saturates to +-1 when 2|x| log2 e overflows.
__device__ __forceinline__ float tanh_sfu(float x)
{
    // Below |x| = 4e-3, tanh(x) = x to within
    // x^3/3 <= 2.2e-8, which also keeps the sign of tiny fields that the
    // difference 1 - 2/(1+e) would round away.
    const float a = fabsf(x) * 2.8853900817779268f;
    float e, r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(a));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
    const float big = copysignf(fmaf(-2.0f, r, 1.0f), x);
    return fabsf(x) < 4e-3f ? x : big;
}

template <int RT>
struct Vec;
template <>
struct Vec<1> {
    using T = float;
    __device__ static T load(const float* p) { return *p; }
    __device__ static void store(float* p, T v) { *p = v; }
    __device__ static float get(const T& v, int) { return v; }
    __device__ static void set(T& v, int, float x) { v = x; }
};
template <>
struct Vec<2> {
    using T = float2;
    __device__ static T load(const float* p) { return *reinterpret_cast<const float2*>(p); }
    __device__ static void store(float* p, T v) { *reinterpret_cast<float2*>(p) = v; }
    __device__ static float get(const T& v, int k) { return k == 0 ? v.x : v.y; }
    __device__ static void set(T& v, int k, float x) { if (k == 0) v.x = x; else v.y = x; }
};
template <>
struct Vec<4> {
    using T = float4;
    __device__ static T load(const float* p) { return *reinterpret_cast<const float4*>(p); }
    __device__ static void store(float* p, T v) { *reinterpret_cast<float4*>(p) = v; }
    __device__ static float get(const T& v, int k)
    {
        return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
    }
    __device__ static void set(T& v, int k, float x)
    {
        if (k == 0) v.x = x; else if (k == 1) v.y = x; else if (k == 2) v.z = x; else v.w = x;
    }
};

// Coupling formats. 0: (column, float bits) pairs; 1: +-1 words, column |
// sign << 31; 2: +-1 halfwords, column | sign << 15, two to a word, staged in
// shared memory for the whole kernel; 3: the same words read from global
// memory through L1. A slice's entries are slot-major (DevInstance): entry d of
// a lane's row is 32 d further on, in formats 2 and 3 a pair of entries.
template <int FMT>
struct Couplings;
template <>
struct Couplings<0> {
    const int2* e;
};
template <>
struct Couplings<1> {
    const uint32_t* e;
};
template <>
struct Couplings<2> {
    const uint32_t* e;  // shared memory
};
template <>
struct Couplings<3> {
    const uint32_t* e;
};

// acc += w m for one gathered row of W replicas and w = +-1, the sign of `sg`.
// The product is exact, so this rounds as an FMA does.
template <int W>
__device__ __forceinline__ void add_signed(float (&acc)[W], const float* p, uint32_t sg)
{
    if constexpr (W == 1) {
        acc[0] += __uint_as_float(__float_as_uint(p[0]) ^ (sg & 0x80000000u));
    } else {
        const float w = __uint_as_float((sg & 0x80000000u) | 0x3f800000u);
        const float2 ww = make_float2(w, w);
#pragma unroll
        for (int k = 0; k < W; k += 2) {
            const float2 v = fma2(ww, make_float2(p[k], p[k + 1]), make_float2(acc[k], acc[k + 1]));
            acc[k] = v.x;
            acc[k + 1] = v.y;
        }
    }
}

template <int W>
__device__ __forceinline__ void add_weighted(float (&acc)[W], const float* p, float w)
{
#pragma unroll
    for (int k = 0; k < W; ++k) acc[k] = fmaf(w, p[k], acc[k]);
}

// The W replicas' magnetisations of row c (W = 1: one slot of a wider tile).
template <int RT, int W>
__device__ __forceinline__ void gather(float (&v)[W], const float* m, uint32_t c)
{
    if constexpr (W == 1) {
        v[0] = m[c * RT];
    } else {
        const typename Vec<W>::T x = Vec<W>::load(m + c * RT);
#pragma unroll
        for (int k = 0; k < W; ++k) v[k] = Vec<W>::get(x, k);
    }
}

// NP pairs of +-1 couplings: their words, then every gather, then the sums in
// the couplings' order, so that one round trip serves them all.
template <int RT, int W, int NP>
__device__ __forceinline__ void field_pairs(float (&acc)[W], const uint32_t (&w)[NP], const float* m)
{
    float v[2 * NP][W];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        gather<RT, W>(v[2 * p], m, w[p] & 0x7fffu);
        gather<RT, W>(v[2 * p + 1], m, (w[p] >> 16) & 0x7fffu);
    }
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        add_signed<W>(acc, v[2 * p], w[p] << 16);
        add_signed<W>(acc, v[2 * p + 1], w[p]);
    }
}

// Local fields of one row for W replicas: acc += sum over its couplings, in
// their order. e0: the lane's first entry; DEG: the degree when it is known.
template <int RT, int W, int FMT, int DEG>
__device__ __forceinline__ void row_field(float (&acc)[W], const Couplings<FMT>& ent, int e0, int deg, const float* m)
{
    if constexpr (FMT == 2 || FMT == 3) {
        const uint32_t* e = ent.e + e0;
        auto word = [&](int p) { return FMT == 2 ? e[32 * p] : __ldg(e + 32 * p); };
        if constexpr (DEG > 0) {
            static_assert(DEG % 2 == 0, "pairs");
            uint32_t w[DEG / 2];
#pragma unroll
            for (int p = 0; p < DEG / 2; ++p) w[p] = word(p);
            field_pairs<RT, W>(acc, w, m);
        } else {
            // batches of four pairs, the next batch's words loaded before this
            // one's gathers are summed; then two pairs, then one
            constexpr int B = W > 2 ? 2 : 4;
            const int np = (deg + 1) >> 1;
            int p = 0;
            if (np >= B) {
                uint32_t w[B];
#pragma unroll
                for (int q = 0; q < B; ++q) w[q] = word(q);
                for (p = B; p + B <= np; p += B) {
                    uint32_t nw[B];
#pragma unroll
                    for (int q = 0; q < B; ++q) nw[q] = word(p + q);
                    field_pairs<RT, W>(acc, w, m);
#pragma unroll
                    for (int q = 0; q < B; ++q) w[q] = nw[q];
                }
                field_pairs<RT, W>(acc, w, m);
            }
            if (B > 2 && p + 2 <= np) {
                const uint32_t w[2] = {word(p), word(p + 1)};
                field_pairs<RT, W>(acc, w, m);
                p += 2;
            }
            if (p < np) {
                const uint32_t w[1] = {word(p)};
                field_pairs<RT, W>(acc, w, m);
            }
        }
    } else if constexpr (FMT == 1) {
        const uint32_t* e = ent.e + e0;
        const int n = DEG > 0 ? DEG : deg;
#pragma unroll(DEG > 0 ? DEG : 4)
        for (int q = 0; q < n; ++q) {
            const uint32_t w = __ldg(e + 32 * q);
            float v[W];
            gather<RT, W>(v, m, w & 0x7fffffffu);
            add_signed<W>(acc, v, w);
        }
    } else {
        const int2* e = ent.e + e0;
#pragma unroll 4
        for (int q = 0; q < deg; ++q) {
            const int2 w = __ldg(e + 32 * q);
            float v[W];
            gather<RT, W>(v, m, (uint32_t)w.x);
            add_weighted<W>(acc, v, __int_as_float(w.y));
        }
    }
}

// -tanh(x) for the negated argument nx = -x (tanh_sfu; both halves of its
// formula are odd), for W replicas.
template <int W>
__device__ __forceinline__ void neg_tanh(float (&sn)[W], const float (&nx)[W])
{
    if constexpr (W == 1) {
        sn[0] = tanh_sfu(nx[0]);
    } else {
#pragma unroll
        for (int k = 0; k < W; k += 2) {
            float2 e, r;
            const float a0 = fabsf(nx[k]) * 2.8853900817779268f, a1 = fabsf(nx[k + 1]) * 2.8853900817779268f;
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(a0));
            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(a1));
            e = add2(e, make_float2(1.0f, 1.0f));
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(e.x));
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(e.y));
            const float2 b = fma2(make_float2(-2.0f, -2.0f), r, make_float2(1.0f, 1.0f));
            sn[k] = fabsf(nx[k]) < 4e-3f ? nx[k] : copysignf(b.x, nx[k]);
            sn[k + 1] = fabsf(nx[k + 1]) < 4e-3f ? nx[k + 1] : copysignf(b.y, nx[k + 1]);
        }
    }
}

// The end of a row's update for W replicas: from its neighbours' sum, the new
// values, the largest change folded into d, and the store.
template <int RT, int W>
__device__ __forceinline__ void finish_row(float (&acc)[W], const float (&old)[W], float* m, int i, const float* h,
                                           const float (&ninvT)[W], float (&d)[W])
{
    float nx[W], sn[W];
    if (h) {
        const float hv = __ldg(h + i);
#pragma unroll
        for (int k = 0; k < W; ++k) acc[k] += hv;
    }
#pragma unroll
    for (int k = 0; k < W; ++k) nx[k] = acc[k] * ninvT[k];
    neg_tanh<W>(sn, nx);
#pragma unroll
    for (int k = 0; k < W; ++k) d[k] = fmaxf(d[k], fabsf(sn[k] - old[k]));
    if constexpr (W == 1) {
        m[i * RT] = sn[0];
    } else {
        typename Vec<W>::T v;
#pragma unroll
        for (int k = 0; k < W; ++k) Vec<W>::set(v, k, sn[k]);
        Vec<W>::store(m + i * RT, v);
    }
}

// A row of known degree with everything it reads already on its way, so that a
// thread can have two rows of a level under way (they share no coupling). With
// one slot, L = 100, R = 400: 5.4 -> 4.9 ms; with two it was slower (7.9 -> 8.1).
template <int RT, int W, int FMT, int DEG>
struct RowLoads {
    uint32_t w[DEG / 2];
    float v[DEG][W], old[W];
    __device__ __forceinline__ void words(const Couplings<FMT>& ent, int e0)
    {
#pragma unroll
        for (int p = 0; p < DEG / 2; ++p) w[p] = FMT == 2 ? ent.e[e0 + 32 * p] : __ldg(ent.e + e0 + 32 * p);
    }
    __device__ __forceinline__ void gathers(const float* m, int i)
    {
#pragma unroll
        for (int p = 0; p < DEG / 2; ++p) {
            gather<RT, W>(v[2 * p], m, w[p] & 0x7fffu);
            gather<RT, W>(v[2 * p + 1], m, (w[p] >> 16) & 0x7fffu);
        }
        gather<RT, W>(old, m, (uint32_t)i);
    }
    __device__ __forceinline__ void finish(float* m, int i, const float* h, const float (&ninvT)[W], float (&d)[W])
    {
        float acc[W];
#pragma unroll
        for (int k = 0; k < W; ++k) acc[k] = 0.f;
#pragma unroll
        for (int p = 0; p < DEG / 2; ++p) {
            add_signed<W>(acc, v[2 * p], w[p] << 16);
            add_signed<W>(acc, v[2 * p + 1], w[p]);
        }
        finish_row<RT, W>(acc, old, m, i, h, ninvT, d);
    }
};

// One row's update for W replicas (slots k0 .. k0 + W - 1 of the tile when
// m points at slot k0 of row 0): s_i <- -tanh(Phi_i / T), the largest change
// folded into d.
template <int RT, int W, int FMT, int DEG>
__device__ __forceinline__ void update_row(const Couplings<FMT>& ent, int e0, int deg, float* m, int i, const float* h,
                                           const float (&ninvT)[W], float (&d)[W])
{
    float acc[W], old[W];
#pragma unroll
    for (int k = 0; k < W; ++k) acc[k] = 0.f;
    gather<RT, W>(old, m, (uint32_t)i);
    row_field<RT, W, FMT, DEG>(acc, ent, e0, deg, m);
    finish_row<RT, W>(acc, old, m, i, h, ninvT, d);
}

// The levels of one sweep in order, each a parallel step over the CTA's warps
// (32-row slices), with a barrier after all but the last.
template <int RT, int W, int NT, int FMT, int DEG>
__device__ __forceinline__ void sweep_levels(const DevInstance& in, const Couplings<FMT>& ent, const int4* slices,
                                             float* m, const float (&ninvT)[W], float (&d)[W])
{
    constexpr int kWarps = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int s0 = 0, s1 = __ldg(in.lvl_slice + 1);  // this level's slices; level 0 starts at 0
    int r0 = 0, r1 = DEG > 0 ? __ldg(in.lvl_start + 1) : 0;
    for (int l = 0; l < in.nlev; ++l) {
        // the next level's bounds arrive while this one runs
        const int ln = l + 2 <= in.nlev ? l + 2 : in.nlev;
        const int s2 = __ldg(in.lvl_slice + ln);
        const int r2 = DEG > 0 ? __ldg(in.lvl_start + ln) : 0;
        if constexpr (DEG > 0) {
            // every slice has degree DEG: its rows and couplings follow from its number
            constexpr int kE = FMT >= 2 ? 16 * DEG : 32 * DEG;
            int i = r0 + 32 * warp + lane;
            if constexpr (FMT >= 2 && RT == 1) {
                int sl = s0 + warp;
                for (; i + 32 * kWarps < r1; sl += 2 * kWarps, i += 64 * kWarps) {
                    RowLoads<RT, W, FMT, DEG> a, b;
                    a.words(ent, sl * kE + lane);
                    b.words(ent, (sl + kWarps) * kE + lane);
                    a.gathers(m, i);
                    b.gathers(m, i + 32 * kWarps);
                    a.finish(m, i, in.h, ninvT, d);
                    b.finish(m, i + 32 * kWarps, in.h, ninvT, d);
                }
                if (i < r1) update_row<RT, W, FMT, DEG>(ent, sl * kE + lane, DEG, m, i, in.h, ninvT, d);
            } else {
                for (int sl = s0 + warp; sl < s1; sl += kWarps, i += 32 * kWarps)
                    if (i < r1) update_row<RT, W, FMT, DEG>(ent, sl * kE + lane, DEG, m, i, in.h, ninvT, d);
            }
        } else {
            for (int sl = s0 + warp; sl < s1; sl += kWarps) {
                const int4 c = FMT == 2 ? slices[sl] : __ldg(slices + sl);  // row0, rows, degree, offset
                if (lane >= c.y) continue;
                const bool half = FMT >= 2 || (FMT == 1 && in.sell16);  // .z holds two numbers
                const int deg = half ? c.z & 0xffff : c.z;
                const int e0 = FMT >= 2 ? ((c.w + 32 * (int)((uint32_t)c.z >> 16)) >> 1) + lane : c.w + lane;
                update_row<RT, W, FMT, 0>(ent, e0, deg, m, c.x + lane, in.h, ninvT, d);
            }
        }
        if (l + 1 < in.nlev) __syncthreads();
        s0 = s1;
        s1 = s2;
        r0 = r1;
        r1 = r2;
    }
}

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Floats of one CTA's slab of magnetisations in global memory: (n + 1) * rt
// (the dummy row n included), rounded up to 16 bytes so that every slab
// starts on a 16-byte boundary.
__host__ __device__ inline size_t sell_slab_floats(int n, int rt)
{
    return align16((size_t)(n + 1) * rt * sizeof(float)) / sizeof(float);
}

// Bytes of the slice table and the +-1 halfword couplings (format 2).
inline size_t half_table_bytes(const DevInstance& in)
{
    return (size_t)in.nslices * sizeof(int4) + (size_t)in.sell16_len * sizeof(uint32_t);
}

// Whether a solve of R replicas takes one slot per CTA of nt threads
// (plan_sparse_sell); `even`: its replicas take about as many sweeps each
// (even_sweeps), and then the threads at work on an SM decide.
inline bool few_replicas(const DevInstance& in, int R, int sms, bool even, int nt)
{
    if (R <= 2 * sms) return true;
    return (even ? (int64_t)R * nt <= (int64_t)960 * sms : 2 * R <= 7 * sms) && in.nnz <= (int64_t)16 * in.n;
}

inline int env_int(const char* name, int dflt)
{
    const char* v = std::getenv(name);
    return v && *v ? std::atoi(v) : dflt;
}

// Per-CTA bookkeeping of the RT replica slots, in shared memory.
template <int RT, int NW>
struct SlotState {
    double T[RT];
    float invT[RT];
    int rep[RT], fresh[RT], done[RT];
    int lvl_sweeps[RT], sweeps[RT], levels[RT], capped[RT], active[RT];
    uint32_t dred[2][NW][RT];  // per-warp largest changes (float bits), by sweep parity
    long long ei[NW][RT];
    double ef[NW][RT];
};

// Run one instance's replica queue on this CTA until the queue is empty and
// every slot has drained. Called by the whole CTA (it contains barriers). The
// slot bookkeeping S may be sized for more slots (RTS) than the job uses.
template <int RT, int NT, int FMT, int DEG = 0, int RTS = RT>
__device__ void run_job(const DevInstance& in, const DevSolve& s, float* m, SlotState<RTS, NT / 32>& S)
{
    static_assert(RT <= RTS, "the slot bookkeeping holds the job's slots");
    constexpr int kThreads = NT;
    constexpr int kWarps = NT / 32;
    using V = Vec<RT>;
    double* const s_T = S.T;
    float* const s_invT = S.invT;
    int* const s_rep = S.rep;
    int* const s_fresh = S.fresh;
    int* const s_done = S.done;
    int* const s_lvl_sweeps = S.lvl_sweeps;
    int* const s_sweeps = S.sweeps;
    int* const s_levels = S.levels;
    int* const s_capped = S.capped;
    int* const s_active = S.active;
    auto& s_dred = S.dred;
    auto& s_ei = S.ei;
    auto& s_ef = S.ef;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = in.n;
    __shared__ int s_last[RT];  // serving ring: this slot finished its job's last replica
    Couplings<FMT> ent;
    const int4* slices = in.slices;
    if constexpr (FMT == 0) ent.e = in.sell_gen;
    if constexpr (FMT == 1) ent.e = in.sell_pm1;
    if constexpr (FMT == 3) ent.e = in.sell16;
    if constexpr (FMT == 2) {
        // Stage the slice table and the couplings in shared memory, after the
        // magnetisations; they serve every replica this CTA runs.
        unsigned char* base = reinterpret_cast<unsigned char*>(m);
        int4* ss = reinterpret_cast<int4*>(base + align16((size_t)(n + 1) * RT * sizeof(float)));
        uint32_t* se = reinterpret_cast<uint32_t*>(ss + in.nslices);
        for (int q = tid; q < in.nslices; q += kThreads) ss[q] = __ldg(in.slices + q);
        for (int64_t q = tid; q < in.sell16_len; q += kThreads) se[q] = __ldg(in.sell16 + q);
        slices = ss;
        ent.e = se;
        __syncthreads();
    }

    // Each of the RT slots takes replicas from the queue s.tile_rep[0..R) (longest
    // start temperatures first) until it is empty: when a slot's replica ends,
    // the slot is finalised and refilled at once, so no slot idles while work
    // remains.
    if (tid == 0) {
        for (int k = 0; k < RT; ++k) {
            const int q = atomicAdd(s.work_counter, 1);
            const int r = q < s.R ? s.tile_rep[q] : -1;
            s_rep[k] = r;
            s_fresh[k] = r >= 0;
            s_done[k] = 0;
            s_active[k] = 0;
        }
    }
    __syncthreads();

    for (;;) {
        // ---- fresh slots: start state (caller m0 or the draw) and first level --
        bool fresh[RT], any_fresh = false;
#pragma unroll
        for (int k = 0; k < RT; ++k) { fresh[k] = s_fresh[k] != 0; any_fresh |= fresh[k]; }
        if (any_fresh) {
            for (int idx = tid; idx < (n + 1) * RT; idx += kThreads) {
                const int i = idx / RT, k = idx % RT;
                if (!fresh[k]) continue;
                const int r = s_rep[k];
                float v = 0.f;
                if (i < n) {
                    const int o = __ldg(in.new2old + i);
                    v = s.m0 ? __ldg(s.m0 + (size_t)r * n + o) : draw_m0(s.seed, s.stream, r, o);
                }
                m[idx] = v;
            }
            __syncthreads();
            if (tid < RT && fresh[tid]) {
                double T;
                const bool act = sched_first(s, (double)s.t0[s_rep[tid]], &T);
                s_T[tid] = T;
                s_invT[tid] = act ? sched_inv_t(T) : 0.f;
                s_active[tid] = act;
                s_done[tid] = !act;  // no level with T > 0: the result is sign(m0)
                s_levels[tid] = act ? 1 : 0;
                s_lvl_sweeps[tid] = 0;
                s_sweeps[tid] = 0;
                s_capped[tid] = 0;
                s_fresh[tid] = 0;
            }
            __syncthreads();
        }

        // ---- finished slots: sign-round, outputs, exact energy; then refill ----
        bool done[RT], any_done = false;
#pragma unroll
        for (int k = 0; k < RT; ++k) { done[k] = s_done[k] != 0; any_done |= done[k]; }
        if (any_done) {
            long long ei[RT];
            double ef[RT];
            int rep[RT];
#pragma unroll
            for (int k = 0; k < RT; ++k) { ei[k] = 0; ef[k] = 0.0; rep[k] = s_rep[k]; }
            for (int i = tid; i < n; i += kThreads) {
                const int o = __ldg(in.new2old + i);
                const typename V::T mi = V::load(m + i * RT);
#pragma unroll
                for (int k = 0; k < RT; ++k) {
                    if (!done[k]) continue;
                    const float mv = V::get(mi, k);
                    s.sigma[(size_t)rep[k] * n + o] = (int8_t)(mv >= 0.f ? 1 : -1);
                    if (s.m_final) s.m_final[(size_t)rep[k] * n + o] = mv;
                }
                const int e0 = __ldg(in.row_ptr + i), e1 = __ldg(in.row_ptr + i + 1);
                for (int e = e0; e < e1; ++e) {
                    const int j = __ldg(in.col + e);
                    if (j <= i) continue;
                    const typename V::T mj = V::load(m + j * RT);
                    if (in.integer) {
                        const int w = (int)__ldg(in.val_i8 + e);
#pragma unroll
                        for (int k = 0; k < RT; ++k)
                            if (done[k])
                                ei[k] += (V::get(mi, k) >= 0.f) == (V::get(mj, k) >= 0.f) ? w : -w;
                    } else {
                        const double w = __ldg(in.val_f64 + e);
#pragma unroll
                        for (int k = 0; k < RT; ++k)
                            if (done[k])
                                ef[k] += (V::get(mi, k) >= 0.f) == (V::get(mj, k) >= 0.f) ? w : -w;
                    }
                }
#pragma unroll
                for (int k = 0; k < RT; ++k) {
                    if (!done[k]) continue;
                    const int si = V::get(mi, k) >= 0.f ? 1 : -1;
                    if (in.integer) {
                        if (in.h) ei[k] += (long long)__ldg(in.h + i) * si;
                    } else if (in.h_f64) {
                        ef[k] += __ldg(in.h_f64 + i) * si;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < RT; ++k) {
                const long long a = warp_reduce_strided<1>(ei[k], SumOp());
                const double b = warp_reduce_strided<1>(ef[k], SumOp());
                if (lane == 0) { s_ei[warp][k] = a; s_ef[warp][k] = b; }
            }
            if (s.finished) __threadfence();  // this thread's outputs, before the completion count
            __syncthreads();
            if (tid < RT && done[tid]) {
                const int r = rep[tid];
                long long ti = 0;
                double tf = 0.0;
                for (int w = 0; w < kWarps; ++w) { ti += s_ei[w][tid]; tf += s_ef[w][tid]; }
                s.energy[r] = in.integer ? (double)ti : tf;
                s.energy_i64[r] = in.integer ? ti : 0;
                s.sweeps[r] = s_sweeps[tid];
                s.levels[r] = s_levels[tid];
                s.capped[r] = s_capped[tid];
                if (s.finished) {
                    __threadfence();
                    s_last[tid] = atomicAdd(s.finished, 1) + 1 == s.R;
                }
            }
            __syncthreads();
            if (s.finished) {
                // The CTA that finishes a served job's last replica selects its
                // best replica and tells the host (every CTA fenced its outputs
                // before counting them).
                bool last = false;
#pragma unroll
                for (int k = 0; k < RT; ++k) last |= done[k] && s_last[k] != 0;
                if (last) {
                    __threadfence();
                    best_reduce<kThreads>(s, n, in.integer, s.best_out, s.res);
                    __threadfence_system();
                    __syncthreads();
                    if (tid == 0) *reinterpret_cast<volatile int32_t*>(s.done_flag) = 1;
                }
                __syncthreads();
#pragma unroll
                for (int k = 0; k < RT; ++k)
                    if (tid == k) s_last[k] = 0;
            }
            if (tid == 0) {
                for (int k = 0; k < RT; ++k) {
                    if (!done[k]) continue;
                    const int q = atomicAdd(s.work_counter, 1);
                    const int r = q < s.R ? s.tile_rep[q] : -1;
                    s_rep[k] = r;
                    s_fresh[k] = r >= 0;
                    s_done[k] = 0;
                }
            }
            __syncthreads();
            continue;
        }

        bool act[RT], any_act = false;
#pragma unroll
        for (int k = 0; k < RT; ++k) { act[k] = s_active[k] != 0; any_act |= act[k]; }
        if (!any_act) break;  // every slot is empty: the queue ran dry

        // ---- sweeps until a slot's level ends --------------------------------
        // A thread updates its spin for all RT replicas from one coupling load
        // and RT-wide gathers (a dead slot's values are computed and never
        // used). When a single slot is left (the queue ran dry) it takes a
        // one-replica path, so a straggler's sweep costs what a one-replica
        // sweep costs. Every thread applies the stopping rule to every slot
        // itself, from the warps' largest changes: a sweep has one barrier per
        // level and no other.
        int live = 0, only = 0;
        float ninvT[RT], dmin[RT];
        int ls[RT], limit[RT], done_now[RT];
#pragma unroll
        for (int k = 0; k < RT; ++k) {
            ninvT[k] = act[k] ? -s_invT[k] : 0.f;
            live += act[k];
            only = act[k] ? k : only;
            const bool fixed = sched_fixed(s, s_T[k]);
            ls[k] = act[k] ? s_lvl_sweeps[k] : 0;
            limit[k] = act[k] ? (fixed ? s.fixed_sweeps : s.k_max) : INT_MAX;
            dmin[k] = act[k] && !fixed ? s.d_min : -1.f;  // changes are >= 0
            done_now[k] = 0;
        }
        int sweeps = 0, par = 0;
        float dd[RT];
        for (bool more = true; more; par ^= 1) {
            float d[RT];
#pragma unroll
            for (int k = 0; k < RT; ++k) d[k] = 0.f;
            if (RT > 1 && live == 1) {
                float d1[1] = {0.f}, n1[1] = {ninvT[0]};
#pragma unroll
                for (int k = 1; k < RT; ++k)
                    if (only == k) n1[0] = ninvT[k];
                sweep_levels<RT, 1, NT, FMT, DEG>(in, ent, slices, m + only, n1, d1);
#pragma unroll
                for (int k = 0; k < RT; ++k)
                    if (only == k) d[k] = d1[0];
            } else {
                sweep_levels<RT, RT, NT, FMT, DEG>(in, ent, slices, m, ninvT, d);
            }
#pragma unroll
            for (int k = 0; k < RT; ++k) {
                // non-negative floats order like their bits
                const uint32_t v = __reduce_max_sync(0xffffffffu, __float_as_uint(d[k]));
                if (lane == 0) s_dred[par][warp][k] = v;
            }
            __syncthreads();  // the last level's spins and the warps' changes
            ++sweeps;
#pragma unroll
            for (int k = 0; k < RT; ++k) {
                const uint32_t v = lane < kWarps ? s_dred[par][lane][k] : 0u;
                dd[k] = __uint_as_float(__reduce_max_sync(0xffffffffu, v));
                ls[k] += 1;
                done_now[k] = dd[k] <= dmin[k] || ls[k] >= limit[k];
                more &= !done_now[k];
            }
        }
        // the levels that ended: cool, or finish (the slots' sweeps so far)
        __syncthreads();  // every thread has read the slots' state
#pragma unroll
        for (int k = 0; k < RT; ++k) {
            if (tid != k || !act[k]) continue;
            s_sweeps[k] += sweeps;
            double T = s_T[k];
            int l = ls[k];
            if (done_now[k]) {
                if (!sched_fixed(s, T) && !(dd[k] <= s.d_min)) s_capped[k] += 1;
                l = 0;
                if (sched_advance(s, &T)) {
                    s_T[k] = T;
                    s_levels[k] += 1;
                    s_invT[k] = sched_inv_t(T);
                } else {
                    s_active[k] = 0;
                    s_done[k] = 1;
                }
            }
            s_lvl_sweeps[k] = l;
        }
        __syncthreads();
    }
}
}  // namespace
}  // namespace mars
