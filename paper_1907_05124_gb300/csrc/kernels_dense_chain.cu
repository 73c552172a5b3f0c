// The in-panel chain of the tensor-core descent (kernels_dense_tc.cu), with
// the sequential steps and the folding of their results on different warps.
//
// A panel's 128 spins are updated one after the other (Section 3, Algorithm 1),
// each new value changing the fields of every later spin. Per replica the steps
// form a chain of dependent tanhs; the folds are plain FMAs that only have to
// stay ahead of it. So, for the RPC replicas of a CTA:
//
//  * Warp 0 runs the chain, one replica per lane, eight steps (a run) at a
//    time. It holds the fields of the run's and the next run's spins in
//    registers and folds each new spin into those itself.
//  * The helper warps own the fields of the later spins (4 spins x TR replicas
//    a lane, in registers) and, when the chain feeds the next panel, that
//    panel's fields. After every run the chain raises an mbarrier, and they
//    fold its eight new values in. A run's spins are handed to the chain
//    through shared memory a run ahead, without the last run's values, which
//    the chain adds itself: it does not wait for the helpers' way there and
//    back (about 420 cycles).
//
// Every field takes its FMAs in the order of the spins, and the step folds its
// last term into the tanh's argument exactly as chain_body does, so the results
// are bit for bit chain_body's.
//
// What bounds it: issue on the chain's scheduler. By clock stamps (N = 8192) a step
// takes 64 cycles in a panel's first run, which has no last run's values to fold
// (FMA, ex2, add, rcp, FMA, select, FMA depend on one another), and about 86 in the
// others; waiting for hand-overs takes 140 a run, so a panel's steps take 12,300 to
// 12,800 cycles, and 15,700 where 32 replicas feed the next panel. chain_body keeps
// 32 / RPW lanes on a replica, every one computing the step, so with all
// replicas active two warps per scheduler issue about 260 cycles a step.
// Measured on a GB300 at N = 8192, a sweep with 4096 replicas active: 1.96 ms
// with chain_body's kernel, 1.47 with this one (1024 active: 0.99, 0.78).
#include "device_common.cuh"
#include "mars_internal.h"
#include "tc_primitives.cuh"

#include <cuda_bf16.h>
#include <cuda_fp8.h>

namespace mars {
namespace {

constexpr int kBM = 128;   // spins of a panel
constexpr int kGrp = 32;   // spins of a helper warp
constexpr int kRun = 8;    // steps of a run; the chain holds the fields of two runs' spins
constexpr int kRuns = kBM / kRun;

template <int RPC>
struct ChainShape {
    // replicas of one helper lane's tile and helper warps: 4 groups of 32
    // spins x kRG replica groups
    static constexpr int TR = RPC >= 16 ? 4 : 2;
    static constexpr int kRG = RPC / (4 * TR);
    static constexpr int kHelpers = 4 * kRG;
    // The other warps help to load and store only; those whose number is a
    // multiple of 4 issue on the chain's scheduler and take no folds.
    static constexpr int kWarps = RPC >= 16 ? 12 : 8;
    static constexpr int kLd = RPC + 1;  // row stride of the transposed arrays
};

template <int RPC, bool NEXT>
struct SplitChainSmem {
    static constexpr int kJ = kBM * kBM * (int)sizeof(float);
    static constexpr int kBlocks = NEXT ? 2 : 1;
    static constexpr int kT = kBM * ChainShape<RPC>::kLd * (int)sizeof(float);  // fields, old spins, old low-precision
    static constexpr int kV = kBM * RPC * (int)sizeof(float);                   // deltas, new spins (NEXT)
    static constexpr int kBars = 2 * kRuns + 1;
    static constexpr int kBytes = kBlocks * kJ + (NEXT ? 2 : 1) * kV + 3 * kT + kBars * 8 + 16;
};

template <int N>
struct Int {
    static constexpr int value = N;
};

// A helper lane's tile: the fields of 4 spins for TR replicas.
template <int TR>
struct FieldTile {
    float v[4][TR];
    // += J[a][4 spins] x x[a][TR replicas]
    __device__ __forceinline__ void fold(const float* J, const float* x)
    {
        const float4 j = *reinterpret_cast<const float4*>(J);
        const float w[4] = {j.x, j.y, j.z, j.w};
        if constexpr (TR == 4) {
            const float4 d = *reinterpret_cast<const float4*>(x);
            const float2 d0 = make_float2(d.x, d.y), d1 = make_float2(d.z, d.w);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 ww = make_float2(w[i], w[i]);
                const float2 a = fma2(ww, d0, make_float2(v[i][0], v[i][1]));
                const float2 b = fma2(ww, d1, make_float2(v[i][2], v[i][3]));
                v[i][0] = a.x;
                v[i][1] = a.y;
                v[i][2] = b.x;
                v[i][3] = b.y;
            }
        } else {
            const float2 d = *reinterpret_cast<const float2*>(x);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 a = fma2(make_float2(w[i], w[i]), d, make_float2(v[i][0], v[i][1]));
                v[i][0] = a.x;
                v[i][1] = a.y;
            }
        }
    }
};

// One CTA: the chain of panel p for replica slots [blockIdx.x RPC, + RPC).
// The arguments are panel_chain_kernel's. G and gx_in are not __restrict__:
// the compiler may move loads through a restricted pointer to const above the
// wait that makes them valid.
template <int RPC, bool NEXT, bool FP8>
__global__ void __launch_bounds__(ChainShape<RPC>::kWarps * 32, 1)
    split_chain_kernel(TcState t, int p, const float* G, const float* gx_in, float* gx_out, int g_early)
{
    using L = SplitChainSmem<RPC, NEXT>;
    using C = ChainShape<RPC>;
    constexpr int kThreads = C::kWarps * 32, LD = C::kLd, TR = C::TR;
    extern __shared__ __align__(16) unsigned char chain_smem[];
    float* Jb = reinterpret_cast<float*>(chain_smem);   // J[p][p] (symmetric)
    float* Jn = Jb + kBM * kBM;                          // NEXT: J[p][p+1], row a = this panel's spin
    float* dl = reinterpret_cast<float*>(chain_smem + L::kBlocks * L::kJ);  // [spin][RPC] deltas
    float* sv = dl + kBM * RPC;                          // NEXT: [spin][RPC] new spins
    float* F = dl + (NEXT ? 2 : 1) * kBM * RPC;          // [spin][LD] fields, then the new spins
    float2* so = reinterpret_cast<float2*>(F + kBM * LD);  // [spin][LD] old spins and their low-precision values
    uint64_t* bars = reinterpret_cast<uint64_t*>(chain_smem + L::kBytes - L::kBars * 8 - 8);
    uint64_t* prog = bars;           // [16] run k is done
    uint64_t* hand = bars + kRuns;   // [16] run k's fields are in F, with the spins of runs 0 .. k - 3
    uint64_t* jbar = hand + kRuns;   // J blocks loaded
    __shared__ int s_ok;
    __shared__ uint32_t s_live;  // the CTA's active replicas
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int slot0 = blockIdx.x * RPC, p0 = p * kBM;
    if (tid == 0) {
        for (int k = 0; k < kRuns; ++k) {
            tc::mbar_init(&prog[k], 1);
            tc::mbar_init(&hand[k], C::kRG);
        }
        tc::mbar_init(jbar, 1);
        tc::fence_barrier_init();
        tc::mbar_arrive_expect_tx(jbar, L::kBlocks * L::kJ);
        tc::bulk_load(Jb, t.Jdiag + (size_t)p * kBM * kBM, L::kJ, jbar);
        if (NEXT) tc::bulk_load(Jn, t.Jsup + (size_t)p * kBM * kBM, L::kJ, jbar);
    }
    // Programmatic launch: what the previous kernels do not write is read
    // before the wait (see chain_body): this panel's old spins, the level
    // state and, with g_early, the fields.
    const int r = lane % RPC;  // warp 0: this lane's replica (RPC < 32: lanes share one)
    const int slot = slot0 + r;
    const bool valid = slot < t.R && t.active[slot];
    const float invT = valid ? t.invT[slot] : 0.f;  // idle replicas compute and store nothing
    // A piece is 4 spins of one replica; a warp takes 8 pieces of 4 replicas,
    // whose transposed stores fall in 32 different banks.
    constexpr int kPieces = RPC * (kBM / 4);
    constexpr int kPer = (kPieces + kThreads - 1) / kThreads;
    auto piece = [&](int e, int& rr, int& a4) {
        const int q = e >> 5, l = e & 31;  // RPC / 4 replica groups x 4 spin groups
        rr = (q >> 2) * 4 + (l >> 3);
        a4 = ((q & 3) * 8 + (l & 7)) * 4;
    };
    {
        float4 v[kPer];
        uint2 lo[kPer];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int e = tid + k * kThreads;
            if (e >= kPieces) break;
            int rr, a4;
            piece(e, rr, a4);
            const int s = slot0 + rr < t.R ? slot0 + rr : 0;
            const size_t idx = (size_t)s * t.n_pad + p0 + a4;
            v[k] = *reinterpret_cast<const float4*>(t.S + idx);
            if (FP8)
                lo[k] = make_uint2(*reinterpret_cast<const uint32_t*>(t.S8 + idx), 0u);
            else
                lo[k] = *reinterpret_cast<const uint2*>(t.Sb + idx);
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int e = tid + k * kThreads;
            if (e >= kPieces) break;
            int rr, a4;
            piece(e, rr, a4);
            float f[4];
            if (FP8) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    __nv_fp8_e4m3 q;
                    q.__x = (__nv_fp8_storage_t)((lo[k].x >> (8 * i)) & 0xffu);
                    f[i] = float(q);
                }
            } else {
                f[0] = __uint_as_float(lo[k].x << 16);
                f[1] = __uint_as_float(lo[k].x & 0xffff0000u);
                f[2] = __uint_as_float(lo[k].y << 16);
                f[3] = __uint_as_float(lo[k].y & 0xffff0000u);
            }
            so[(a4 + 0) * LD + rr] = make_float2(v[k].x, f[0]);
            so[(a4 + 1) * LD + rr] = make_float2(v[k].y, f[1]);
            so[(a4 + 2) * LD + rr] = make_float2(v[k].z, f[2]);
            so[(a4 + 3) * LD + rr] = make_float2(v[k].w, f[3]);
        }
    }
    if (!g_early) {
        tc::pdl_wait();
        tc::pdl_launch_dependents();
    }
    // The fields: split-K partials in split order, the previous panel's part
    // and h, summed in FP32 in that order.
    {
        float4 f[kPer];
        // NS splits of K pieces at a time: all their loads are in flight
        // before the first sum (a round trip is about 1000 cycles)
        auto gather = [&](auto ns, auto at_once) {
            constexpr int NS = decltype(ns)::value, K = decltype(at_once)::value;
#pragma unroll
            for (int k0 = 0; k0 < kPer; k0 += K) {
                float4 q[K][NS];
#pragma unroll
                for (int k = k0; k < k0 + K && k < kPer; ++k) {
                    const int e = tid + k * kThreads;
                    if (e >= kPieces) break;
                    int rr, a4;
                    piece(e, rr, a4);
                    const float* src = G + (size_t)(slot0 + rr < t.R ? slot0 + rr : 0) * kBM + a4;
#pragma unroll
                    for (int sp = 0; sp < NS; ++sp)
                        q[k - k0][sp] = __ldcg(reinterpret_cast<const float4*>(src + (size_t)sp * t.R_pad * kBM));
                }
#pragma unroll
                for (int k = k0; k < k0 + K && k < kPer; ++k) {
                    f[k] = q[k - k0][0];
#pragma unroll
                    for (int sp = 1; sp < NS; ++sp) {
                        f[k].x += q[k - k0][sp].x;
                        f[k].y += q[k - k0][sp].y;
                        f[k].z += q[k - k0][sp].z;
                        f[k].w += q[k - k0][sp].w;
                    }
                }
            }
        };
        switch (t.splitk) {  // a power of two
        case 1: gather(Int<1>(), Int<kPer>()); break;
        case 2: gather(Int<2>(), Int<kPer>()); break;
        case 4: gather(Int<4>(), Int<kPer>()); break;
        case 8: gather(Int<8>(), Int<2>()); break;
        default: gather(Int<16>(), Int<1>()); break;
        }
        if (g_early) {
            tc::pdl_wait();
            tc::pdl_launch_dependents();
        }
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int e = tid + k * kThreads;
            if (e >= kPieces) break;
            int rr, a4;
            piece(e, rr, a4);
            if (gx_in) {
                const int s = slot0 + rr < t.R ? slot0 + rr : 0;
                const float4 q = __ldcg(reinterpret_cast<const float4*>(gx_in + (size_t)s * kBM + a4));
                f[k].x += q.x;
                f[k].y += q.y;
                f[k].z += q.z;
                f[k].w += q.w;
            }
            if (t.h) {
                const int a = p0 + a4;
                if (a + 0 < t.n) f[k].x += __ldg(t.h + a + 0);
                if (a + 1 < t.n) f[k].y += __ldg(t.h + a + 1);
                if (a + 2 < t.n) f[k].z += __ldg(t.h + a + 2);
                if (a + 3 < t.n) f[k].w += __ldg(t.h + a + 3);
            }
            F[(a4 + 0) * LD + rr] = f[k].x;
            F[(a4 + 1) * LD + rr] = f[k].y;
            F[(a4 + 2) * LD + rr] = f[k].z;
            F[(a4 + 3) * LD + rr] = f[k].w;
        }
    }
    if (warp == 0) {
        if (lane == 0) s_ok = tc::mbar_wait(jbar, 0, t.counters + 2) ? 1 : 0;
        const uint32_t act = __ballot_sync(0xffffffffu, valid && lane < RPC);
        if (lane == 0) s_live = act;
    }
    __syncthreads();
    const uint32_t live = s_live;
    if (!live || !s_ok) return;  // all idle, or the host reports the error

    if (warp == 0) {
        constexpr float kK = 2.8853900817779268f;      // 2 log2(e)
        constexpr float kKinv = 0.34657359027997264f;  // 1 / K
        constexpr float kSmallZ = 4e-3f * kK;          // |y| < 4e-3: tanh(y) = y to 2.2e-8
        const float kinv = kK * invT;
        const float dold = valid ? t.d[slot] : 0.f;    // used at the very end
        float dloc = 0.f;
        // g: the fields of this run's and the next run's spins. The next run's
        // miss the last run's values when they arrive; a step adds two of the
        // 16 pending ones (the last run's, then this run's), in order.
        float g[2 * kRun], old[kRun], cur[kRun];
#pragma unroll
        for (int i = 0; i < 2 * kRun; ++i) g[i] = F[i * LD + r];
#pragma unroll
        for (int i = 0; i < kRun; ++i) old[i] = cur[i] = 0.f;
        auto pend = [&](const float4 (&row)[2], float x) {  // += J[.][next run's spins] x
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float4 w = row[u];
                float* q = g + kRun + 4 * u;
                const float2 xx = make_float2(x, x);
                const float2 lo = fma2(make_float2(w.x, w.y), xx, make_float2(q[0], q[1]));
                const float2 hi = fma2(make_float2(w.z, w.w), xx, make_float2(q[2], q[3]));
                q[0] = lo.x;
                q[1] = lo.y;
                q[2] = hi.x;
                q[3] = hi.y;
            }
        };
        // pending value k of a run: row a0 + k - 8 at the next run's columns.
        // Every operand is loaded a step ahead of its use: a warp issues in
        // order, so a load's latency would land on the chain.
        auto row_of = [&](const float* J0, int k, float4 (&w)[2]) {
            const float* src = J0 + (k - kRun) * kBM + kRun;
            w[0] = *reinterpret_cast<const float4*>(src);
            w[1] = *reinterpret_cast<const float4*>(src + 4);
        };
        float z = kinv * g[0];  // J[-1][0] = 0
        float2 c_s = so[r];
        float jp = Jb[1];
        float4 jr[2] = {*reinterpret_cast<const float4*>(Jb), *reinterpret_cast<const float4*>(Jb + 4)};
        float4 pa[2], pb[2];  // the step's two pending rows
        pa[0] = pa[1] = pb[0] = pb[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        // One run; the first has no values of a last run pending. The step's
        // tanh is started before, and the next one's argument formed right
        // after, everything that may wait.
        auto steps = [&](int run, auto first) {
            constexpr bool kFirst = decltype(first)::value != 0;
            const int a0 = run * kRun;
            // the block from spin a0 on; past the panel's end (last run) values
            // are read from the arrays behind and not used
            const float* J0 = Jb + a0 * kBM + a0;
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const int a = a0 + i;
                const bool wrap = i + 1 == kRun;
                float e, rc;
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z));
                // the next step's operands
                const int an = !wrap ? a + 1 : run + 1 < kRuns ? a0 + kRun : a0;
                const float* Jx = wrap ? Jb + an * kBM + an : J0;  // the next step's block
                const int in = wrap ? 0 : i + 1;
                const float2 n_s = so[an * LD + r];
                const float n_jp = Jx[in * kBM + in + 1];
                float4 jn[2], qa[2], qb[2];
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (4 * u + 3 > in + 1) jn[u] = *reinterpret_cast<const float4*>(Jx + in * kBM + 4 * u);
                if (!kFirst || in >= kRun / 2 || wrap) {
                    row_of(Jx, 2 * in, qa);
                    row_of(Jx, 2 * in + 1, qb);
                }
                // the pending values but this step's own
                if (i >= kRun / 2) pend(pa, cur[2 * i - kRun]);
                else if (!kFirst) pend(pa, old[2 * i]);
                // spin a + 1 takes its last term in its argument
                const float cz = kinv * jp, bz = kinv * fmaf(-jp, c_s.y, g[i + 1]);
                asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(1.0f + e));
                if (i >= kRun / 2) {
                    if (!wrap) pend(pb, cur[2 * i + 1 - kRun]);
                } else if (!kFirst) {
                    pend(pb, old[2 * i + 1]);
                }
                const float big = fmaf(2.0f, rc, -1.0f);
                const float sn = fabsf(z) < kSmallZ ? -kKinv * z : big;
                z = fmaf(cz, sn, bz);
                const float delta = sn - c_s.y;
                dloc = fmaxf(dloc, fabsf(sn - c_s.x));
                F[a * LD + r] = sn;
                dl[a * RPC + r] = delta;
                if (NEXT) sv[a * RPC + r] = sn;
                const float* row = reinterpret_cast<const float*>(jr);
                if (i + 2 < kRun) {
                    if ((i & 1) != 0) g[i + 2] = fmaf(row[i + 2], delta, g[i + 2]);
#pragma unroll
                    for (int q = (i + 3) & ~1; q < kRun; q += 2) {
                        const float2 v = fma2(make_float2(row[q], row[q + 1]), make_float2(delta, delta),
                                              make_float2(g[q], g[q + 1]));
                        g[q] = v.x;
                        g[q + 1] = v.y;
                    }
                }
                cur[i] = delta;
                if (wrap) pend(pb, delta);
                c_s = n_s;
                jp = n_jp;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (4 * u + 3 > in + 1) jr[u] = jn[u];
                    pa[u] = qa[u];
                    pb[u] = qb[u];
                }
            }
            __syncwarp();
            tc::mbar_arrive_if(&prog[run], lane == 0);
        };
        bool ok = true;
        steps(0, Int<1>());
#pragma unroll 1
        for (int run = 1; run + 1 < kRuns; ++run) {
            // the run's spins move up; the next one's fields arrive
            if (run > 1 && ok) ok = tc::mbar_spin(&hand[run + 1], 0, t.counters + 2);
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                g[i] = g[kRun + i];
                g[kRun + i] = F[((run + 1) * kRun + i) * LD + r];
                old[i] = cur[i];
            }
            steps(run, Int<0>());
        }
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            g[i] = g[kRun + i];
            old[i] = cur[i];
        }
        steps(kRuns - 1, Int<0>());
        if (valid && lane < RPC) t.d[slot] = fmaxf(dold, dloc);
    } else if (warp % 4 != 0 && warp - 1 - warp / 4 < C::kHelpers) {
        const int h = warp - 1 - warp / 4;            // helper number
        const int sg = h & 3, rg = h >> 2;            // its group of 32 spins and of replicas
        const int q4 = 4 * (lane & 7), r4 = (rg * 4 + (lane >> 3)) * TR;
        const int mine = 4 * sg + (lane & 7) / 2;     // the run of this lane's spins
        FieldTile<TR> f, gn;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < TR; ++c) {
                f.v[i][c] = F[(kGrp * sg + q4 + i) * LD + r4 + c];  // of runs 0 .. 2: not used
                gn.v[i][c] = 0.f;
            }
        for (int k = 0; k < kRuns; ++k) {
            const bool diag = k + 3 <= 4 * sg + 3;  // the warp still folds into this panel
            if (!NEXT && !diag) break;
            if (!__all_sync(0xffffffffu, tc::mbar_spin(&prog[k], 0, t.counters + 2))) break;
            if (diag) {
#pragma unroll
                for (int i = 0; i < kRun; ++i)
                    f.fold(Jb + (kRun * k + i) * kBM + kGrp * sg + q4, dl + (kRun * k + i) * RPC + r4);
                if (k + 3 >= 4 * sg) {  // run k + 3 is the warp's: hand it over
                    if (mine == k + 3) {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int c = 0; c < TR; ++c) F[(kGrp * sg + q4 + i) * LD + r4 + c] = f.v[i][c];
                    }
                    __syncwarp();
                    tc::mbar_arrive_if(&hand[k + 3], lane == 0);
                }
            }
            if (NEXT) {
#pragma unroll
                for (int i = 0; i < kRun; ++i)
                    gn.fold(Jn + (kRun * k + i) * kBM + kGrp * sg + q4, sv + (kRun * k + i) * RPC + r4);
            }
        }
        if (NEXT) {
#pragma unroll
            for (int c = 0; c < TR; ++c) {
                if ((live >> (r4 + c)) & 1u)
                    *reinterpret_cast<float4*>(gx_out + (size_t)(slot0 + r4 + c) * kBM + kGrp * sg + q4) =
                        make_float4(gn.v[0][c], gn.v[1][c], gn.v[2][c], gn.v[3][c]);
            }
        }
    }
    __syncthreads();
    // the new spins and their low-precision copies
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int e = tid + k * kThreads;
        if (e >= kPieces) break;
        int rr, a4;
        piece(e, rr, a4);
        const int s = slot0 + rr;
        if (!((live >> rr) & 1u)) continue;
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = F[(a4 + i) * LD + rr];
        const size_t idx = (size_t)s * t.n_pad + p0 + a4;
        if (p0 + a4 + 3 < t.n) {
            *reinterpret_cast<float4*>(t.S + idx) = make_float4(v[0], v[1], v[2], v[3]);
            if (FP8) {
                uint32_t w = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) w |= (uint32_t)__nv_fp8_e4m3(v[i]).__x << (8 * i);
                *reinterpret_cast<uint32_t*>(t.S8 + idx) = w;
            } else {
                __nv_bfloat162 w[2] = {__floats2bfloat162_rn(v[0], v[1]), __floats2bfloat162_rn(v[2], v[3])};
                *reinterpret_cast<uint2*>(t.Sb + idx) = *reinterpret_cast<uint2*>(w);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (p0 + a4 + i >= t.n) continue;
                t.S[idx + i] = v[i];
                if (FP8)
                    t.S8[idx + i] = __nv_fp8_e4m3(v[i]).__x;
                else
                    t.Sb[idx + i] = __float2bfloat16_rn(v[i]);
            }
        }
    }
}

template <int RPC, bool NEXT, bool FP8>
cudaError_t launch_as(const TcState& t, int p, const float* G, const float* gx_in, float* gx_out, int ge,
                      cudaStream_t st)
{
    constexpr int smem = SplitChainSmem<RPC, NEXT>::kBytes;
    const void* k = (const void*)split_chain_kernel<RPC, NEXT, FP8>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    TcState tt = t;
    void* args[] = {&tt, &p, &G, &gx_in, &gx_out, &ge};
    return launch_pdl(k, dim3((t.R + RPC - 1) / RPC), dim3(ChainShape<RPC>::kWarps * 32), args, smem, st);
}

template <bool NEXT, bool FP8>
cudaError_t launch_rpc(const TcState& t, int p, int rpc, const float* G, const float* gx_in, float* gx_out, int ge,
                       cudaStream_t st)
{
    switch (rpc) {
    case 8: return launch_as<8, NEXT, FP8>(t, p, G, gx_in, gx_out, ge, st);
    case 16: return launch_as<16, NEXT, FP8>(t, p, G, gx_in, gx_out, ge, st);
    case 32: return launch_as<32, NEXT, FP8>(t, p, G, gx_in, gx_out, ge, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_tc_split_chain(const TcState& t, int p, int rpc, const float* G, const float* gx_in,
                                  float* gx_out, bool g_early, cudaStream_t st)
{
    if (t.splitk < 1 || t.splitk > kChainMaxSplit || t.R_pad % rpc != 0) return cudaErrorInvalidValue;
    const bool next = gx_out != nullptr;
    if (next && !t.Jsup) return cudaErrorInvalidValue;
    const int ge = g_early ? 1 : 0;
    if (t.S8)
        return next ? launch_rpc<true, true>(t, p, rpc, G, gx_in, gx_out, ge, st)
                    : launch_rpc<false, true>(t, p, rpc, G, gx_in, gx_out, ge, st);
    return next ? launch_rpc<true, false>(t, p, rpc, G, gx_in, gx_out, ge, st)
                : launch_rpc<false, false>(t, p, rpc, G, gx_in, gx_out, ge, st);
}

}  // namespace mars
