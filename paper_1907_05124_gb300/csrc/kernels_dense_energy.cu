// Exact energies of many spin vectors of one dense instance (Section 2, Eq. 2
// with each pair counted once), as integer matrix products on tensor cores.
//
// Every coupling is an integer: J_ab itself for integer instances, else
// J_ab / 2^e0 (exact_sum.cuh), cut into signed 7-bit digits. The energy of a
// vector is then sum_d 128^d P_d with
//   P_d = sum_a s_a D_a,  D_a = sum_{b>a} digit_d(J_ab) s_b,
// and D for 128 vectors and 128 rows is a BF16 matrix product whose every sum
// is an integer below 4096 x 127 < 2^19 (longer rows are summed in runs), exact
// in the FP32 accumulator. Integer sums do not depend on their order, so the
// result is the exact sum, rounded once.
//
// A CTA takes 128 vectors (the MMA's rows) against 128-row tiles of J, 64
// columns a step. Each step all threads cut the couplings into digits, four
// digit planes at a time, straight from J into swizzled shared memory (no second
// copy of J, no work at ingest) and one of them issues the planes' MMAs, which
// run while the next step's digits are cut; the next step's couplings are
// already on their way. After a run of a row tile's columns, each thread weights
// one vector's D_a (its TMEM lane) with that vector's own spins. The tiles of
// one vector group are dealt to the CTAs of a cluster, whose partial sums meet
// in distributed shared memory, so the pass needs no scratch in device memory.
//
// What bounds it: the integer instructions that cut and place the digits, and the
// barrier of every step (n = 4096, 2048 vectors: ALU pipe 52 % busy, an instruction
// issued in 44 % of the cycles, barrier the first stall, tensor pipe 16 %; with 8
// warps, or with the loaded spins tested before the step, a third to a half slower).
// Measured on a GB300, FP32-valued Gaussian couplings (8 planes) and +-1:
// n = 8192, 4096 vectors 7.6 and 1.3 ms; n = 2048, 512 vectors 0.23 and 0.07
// ms. The byte-wise dp4a kernel this replaced (36 lanes a clock and SM) took
// 38.6 and 5.6 ms, 1.10 and 0.22 ms; only below n about 500 is it the faster
// by 0 to 9 us.
#include "device_common.cuh"
#include "exact_sum.cuh"
#include "mars_internal.h"
#include "tc_primitives.cuh"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

namespace mars {
namespace {

namespace cg = cooperative_groups;

constexpr int kTile = 128;            // vectors of a CTA, rows of a J tile
constexpr int kStep = 64;             // columns of a step: one 128-byte swizzled row of BF16
constexpr int kEThreads = 512;
constexpr int kChunks = kTile * kStep / 8 / kEThreads;  // 8-column chunks of a step per thread
constexpr int kRowStep = kEThreads / (kStep / 8);       // rows between a thread's chunks
constexpr int kDigit = 7;             // bits of a digit
constexpr int kMaxPlanes = (220 + kDigit) / kDigit;  // exact_span's limit
constexpr int kGroup = 4;             // digit planes made from one read of a tile
constexpr int kOp = kTile * kStep * 2;  // bytes of one operand tile
constexpr int kRun = 32;              // tiles of a row summed before they are weighted: D < 4096 x 127
constexpr int kParts = kEThreads / kTile;  // threads that weight a vector's rows of a tile
constexpr int kShortPass = 6;  // steps of a pass that takes no cluster (an integer instance below n = 256)
constexpr int kSpinLd = 132;           // bytes of a vector's spins of a row tile in shared memory

template <bool INT>
constexpr int kPlanesAtOnce = INT ? 1 : kGroup;
template <bool INT>
constexpr size_t kBuffer = (size_t)(1 + kPlanesAtOnce<INT>) * kOp;  // the vectors' and the planes' operands

// The digits (one per plane) of two couplings as BF16 pairs: a digit's bits are
// put into the significand of +-128, whose sign is its coupling's, and the
// +-128 are taken off (exactly). `flip` holds the signs.
template <int PLANES>
__device__ __forceinline__ void digit_pairs(uint32_t w0, uint32_t w1, uint32_t flip, uint32_t (&out)[PLANES])
{
    const uint32_t bias = 0x43004300u ^ flip;
    uint32_t both = 0;
#pragma unroll
    for (int p = 0; p < PLANES; ++p) {
        both = p & 1 ? both >> kDigit : __byte_perm(w0 >> (kDigit * p), w1 >> (kDigit * p), 0x5410);
        const uint32_t biased = (both & 0x007f007fu) | bias;
        const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&biased),
                                         *reinterpret_cast<const __nv_bfloat162*>(&bias));
        out[p] = *reinterpret_cast<const uint32_t*>(&d);
    }
}

// x >> k and x << k, 0 for k > 31 (what the instructions do; in C++ not defined).
__device__ __forceinline__ uint32_t shr_all(uint32_t x, int k)
{
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(k));
    return r;
}
__device__ __forceinline__ uint32_t shl_all(uint32_t x, int k)
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(k));
    return r;
}

// Bits [28 g, 28 g + 28) of |v| / 2^e0, the digits of plane group g, in the low
// bits. With SUBNORMAL false there are no subnormal couplings (the caller looks
// at e0), and the implicit bit that zeros get here lies below the window.
template <bool SUBNORMAL>
__device__ __forceinline__ uint32_t digit_window(double v, int e0, int g)
{
    const uint32_t top = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    int ex = (int)((top >> 20) & 0x7ffu);
    uint32_t hi = (top & 0xfffffu) | 0x100000u;
    if constexpr (SUBNORMAL) {
        if (ex == 0) hi &= 0xfffffu;
        ex = max(ex, 1);
    }
    const int sh = kDigit * kGroup * g + 1075 + e0 - ex;  // the significand's bit at the window's start
    return shl_all(shr_all(__funnelshift_rc(lo, hi, (uint32_t)max(sh, 0)), max(sh - 32, 0)), max(-sh, 0));
}

__device__ __forceinline__ void fence_proxy_async_shared()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

template <bool INT>
__global__ void __launch_bounds__(kEThreads, 1) dense_energy_kernel(DevInstance in, const int8_t* __restrict__ spins,
                                                                    int count, double* e_out, long long* e_i64,
                                                                    int32_t* status, int planes)
{
    constexpr int kP = kPlanesAtOnce<INT>;
    constexpr uint32_t kCols = kP * kTile;
    extern __shared__ unsigned char esm_raw[];
    unsigned char* esm = (unsigned char*)(((uintptr_t)esm_raw + 1023) & ~(uintptr_t)1023);  // same place in every CTA
    unsigned char* sA = esm + 2 * kBuffer<INT>;                           // [128][kSpinLd] spins of the row tile
    long long* sum = reinterpret_cast<long long*>(sA + kTile * kSpinLd);  // [planes][128]
    uint64_t* done = reinterpret_cast<uint64_t*>(sum + planes * kTile);   // [2] a buffer's MMAs have completed
    __shared__ uint32_t s_tmem;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), size = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = in.n, r0 = (blockIdx.x / size) * kTile;
    const bool hcol = !INT && in.h_f64 != nullptr;  // the field as a coupling to a spin n held at +1
    const int T = (n + (hcol ? 1 : 0) + kTile - 1) / kTile;
    // tiles (ta, tb >= ta) in row order; this CTA's contiguous share
    const long long ntiles = (long long)T * (T + 1) / 2;
    const long long t_begin = ntiles * rank / size, t_end = ntiles * (rank + 1) / size;
    for (int q = tid; q < planes * kTile; q += kEThreads) sum[q] = 0;
    if (tid == 0) {
        tc::mbar_init(&done[0], 1);
        tc::mbar_init(&done[1], 1);
        tc::fence_barrier_init();
    }
    if (warp == 0) tc::tmem_alloc(&s_tmem, kCols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = s_tmem;

    // Chunks of 8 columns: this thread's are rows row0, row0 + kRowStep, ... at the
    // same 8 columns of a step (of the couplings and of the vectors alike).
    const int c8 = tid & 7, row0 = tid >> 3;
    const bool even = (n & 1) == 0, words = in.identity && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(spins) & 3) == 0;
    const bool jwords = (n & 3) == 0;
    double jv[INT ? 1 : kChunks][8];
    uint32_t ji[INT ? kChunks : 1][2];
    uint32_t sv[kChunks][2];

    auto spin_word = [&](int r, int b) -> uint32_t {  // spins b .. b + 3 of vector r as bytes
        uint32_t w = 0;
        if (r0 + r >= count) return 0;
        if (words && b < n) {
            return __ldg(reinterpret_cast<const uint32_t*>(spins + (size_t)(r0 + r) * n + b));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int v = 0;
            if (b + i < n) {
                v = spins[(size_t)(r0 + r) * n + __ldg(in.new2old + b + i)];
            } else if (hcol && b + i == n) {
                v = 1;
            }
            w |= ((uint32_t)v & 0xffu) << (8 * i);
        }
        return w;
    };
    // A step's couplings and spins, into registers: nothing here looks at what
    // was loaded, so that all of it is under way while the last step is summed.
    auto fetch = [&](int ta, int col) {
        const int b = col + 8 * c8;
#pragma unroll
        for (int u = 0; u < kChunks; ++u) {
            const int row = row0 + kRowStep * u, a = ta * kTile + row;
            sv[u][0] = spin_word(row, b);
            sv[u][1] = spin_word(row, b + 4);
            if constexpr (INT) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t w = 0;
                    const int bb = b + 4 * h;
                    if (a < n && bb < n) {
                        const int8_t* src = in.J_i8 + (size_t)a * n + bb;
                        if (jwords) {
                            w = __ldg(reinterpret_cast<const uint32_t*>(src));
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (bb + i < n) w |= ((uint32_t)src[i] & 0xffu) << (8 * i);
                        }
                    }
                    ji[u][h] = w;
                }
            } else {
                const double* src = in.J_f64 + (size_t)a * n + b;
                if (a < n && b > a && b + 8 <= n && even) {
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        const double2 v = __ldg(reinterpret_cast<const double2*>(src + i));
                        jv[u][i] = v.x;
                        jv[u][i + 1] = v.y;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        double v = 0.0;
                        if (a < n && b + i > a) {
                            if (b + i < n) v = __ldg(src + i);
                            else if (hcol && b + i == n) v = __ldg(in.h_f64 + a);
                        }
                        jv[u][i] = v;
                    }
                }
            }
        }
    };
    // the fetched step as operands of buffer `buf` (K-major, 128-byte swizzle)
    auto cut = [&](int buf, int group, int ta, int col, auto sub_tag) {
        [[maybe_unused]] constexpr bool sub = decltype(sub_tag)::value;
        unsigned char* base = esm + buf * kBuffer<INT>;
#pragma unroll
        for (int u = 0; u < kChunks; ++u) {
            const int row = row0 + kRowStep * u;
            const uint32_t at = (uint32_t)row * 128u + (uint32_t)((c8 ^ (row & 7)) * 16);
            const int b = col + 8 * c8;
            uint32_t upper[2] = {~0u, ~0u};  // bytes of the pairs b > a
            if (INT && col < (ta + 1) * kTile) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int skip = ta * kTile + row + 1 - (b + 4 * h);  // leading columns at or below the diagonal
                    upper[h] = skip <= 0 ? ~0u : skip < 4 ? ~0u << (8 * skip) : 0u;
                }
            }
            if (ta == 0 && group == 0) {  // the first row of tiles sees every spin: each is +-1
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int there = r0 + row < count ? n - (b + 4 * h) : 0;
                    const uint32_t bytes = there >= 4 ? ~0u : there > 0 ? ~0u >> (32 - 8 * there) : 0u;
                    if ((__vabsss4(sv[u][h]) ^ 0x01010101u) & bytes) atomicExch(status, (int)kDevBadIndex);
                }
            }
            uint32_t o[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {  // +-1 bytes to BF16; 0 stays 0
                const uint32_t w = sv[u][h >> 1] >> (16 * (h & 1));
                const uint32_t x = __byte_perm(w, 0, 0x4140);  // the two bytes in the low bytes of the halves
                o[h] = ((x & 0x00010001u) * 0x3f80u) | ((x & 0x00800080u) << 8);
            }
            *reinterpret_cast<uint4*>(base + at) = make_uint4(o[0], o[1], o[2], o[3]);
            uint32_t d[4][kP];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                uint32_t w0, w1, sign;
                if constexpr (INT) {
                    const uint32_t w = (ji[u][h >> 1] & upper[h >> 1]) >> (16 * (h & 1));
                    const int v0 = (int)(int8_t)(w & 0xffu), v1 = (int)(int8_t)((w >> 8) & 0xffu);
                    w0 = (uint32_t)abs(v0);
                    w1 = (uint32_t)abs(v1);
                    sign = ((uint32_t)v0 >> 31 << 15) | ((uint32_t)v1 & 0x80000000u);
                } else {
                    const double v0 = jv[u][2 * h], v1 = jv[u][2 * h + 1];
                    w0 = digit_window<sub>(v0, in.exact_e0, group);
                    w1 = digit_window<sub>(v1, in.exact_e0, group);
                    sign = ((uint32_t)__double2hiint(v0) >> 31 << 15) | ((uint32_t)__double2hiint(v1) & 0x80000000u);
                }
                digit_pairs<kP>(w0, w1, sign, d[h]);
            }
#pragma unroll
            for (int p = 0; p < kP; ++p)
                *reinterpret_cast<uint4*>(base + (1 + p) * kOp + at) = make_uint4(d[0][p], d[1][p], d[2][p], d[3][p]);
        }
    };

    const bool subnormal = !INT && in.exact_e0 < -1010;  // else a zero's implicit bit is 65 or more below 2^e0
    uint32_t step = 0;  // buffers filled so far: step s uses buffer s % 2, its phase s / 2
    bool ok = true;
    for (int p0 = 0; p0 < planes && ok; p0 += kP) {
        const int np = min(kP, planes - p0);
        long long t = t_begin;
        int ta = 0, tb = 0;  // tile t's place: rows of T, T - 1, ... tiles
        {
            long long left = t;
            while (ta < T && left >= T - ta) left -= T - ta++;
            tb = ta + (int)left;
        }
        if (t < t_end) fetch(ta, tb * kTile);
        while (t < t_end && ok) {
            // a run of one row tile's columns in this CTA's share
            const int row_tile = ta;
            const int run = (int)min((long long)min(T - tb, kRun), t_end - t);
            const int cols = 2 * run;  // steps
            int col = tb * kTile;
            t += run;
            tb += run;
            if (tb == T) tb = ++ta;
            for (int k = 0; k < cols && ok; ++k, ++step) {
                const int buf = (int)(step & 1u);
                // the MMAs that read this buffer last have completed
                const bool free = step < 2 || tc::mbar_wait(&done[buf], ((step >> 1) - 1) & 1u, status);
                if (subnormal) cut(buf, p0 / kP, row_tile, col, std::true_type{});
                else cut(buf, p0 / kP, row_tile, col, std::false_type{});
                col += kStep;
                // the next step, or the next run's first
                if (k + 1 < cols) fetch(row_tile, col);
                else if (t < t_end) fetch(ta, tb * kTile);
                fence_proxy_async_shared();
                ok = __syncthreads_or(!free) == 0;
                if (tid == 0 && ok) {
                    tc::tc_fence_after();
                    const uint32_t base = tc::smem_addr(esm + buf * kBuffer<INT>);
                    for (int p = 0; p < np; ++p)
#pragma unroll
                        for (int q = 0; q < kStep / 16; ++q)
                            tc::mma_bf16(tmem + p * kTile, tc::smem_desc_sw128(base + q * 32),
                                         tc::smem_desc_sw128(base + (1 + p) * kOp + q * 32),
                                         tc::idesc_bf16_f32(kTile, kTile), (k | q) != 0);
                    tc::mma_commit(&done[buf]);
                }
            }
            // the row tile's own spins, for this thread's vector: kParts threads
            // share a vector (TMEM lane), each taking some of the rows
            const int r = (warp & 3) * 32 + lane, part = warp >> 2;
            for (int q = tid; q < kTile * (kTile / 4); q += kEThreads) {
                const int v = q / (kTile / 4), w = q % (kTile / 4), a = row_tile * kTile + 4 * w;
                *reinterpret_cast<uint32_t*>(sA + v * kSpinLd + 4 * w) = a < n ? spin_word(v, a) : 0u;
            }
            const bool last = ok && tc::mbar_wait(&done[(step - 1) & 1u], ((step - 1) >> 1) & 1u, status);
            ok = __syncthreads_or(!last) == 0;
            tc::tc_fence_after();
            if (ok) {
                for (int p = 0; p < np; ++p) {
                    int e = 0;  // 32 x 4096 x 127 < 2^31
#pragma unroll
                    for (int c0 = 0; c0 < kTile / kParts; c0 += 32) {
                        float v[32];
                        const int at = part * (kTile / kParts) + c0;
                        tc::tmem_ld_32cols(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(p * kTile + at), v);
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const uint32_t s4 = *reinterpret_cast<const uint32_t*>(sA + r * kSpinLd + at + i);
#pragma unroll
                            for (int q = 0; q < 4; ++q) e += __float2int_rn(v[i + q]) * (int)(int8_t)(s4 >> (8 * q));
                        }
                    }
                    atomicAdd(reinterpret_cast<unsigned long long*>(&sum[(p0 + p) * kTile + r]),
                              (unsigned long long)(long long)e);
                }
            }
            tc::tc_fence_before();
            __syncthreads();  // TMEM and the spins may be overwritten
        }
    }
    if (INT && in.h && ok) {  // integer fields (up to 2^24) do not fit a digit
        const int r = tid % kTile;
        long long v = 0;
        if (r0 + r < count)
            for (int a = tid / kTile + (kEThreads / kTile) * rank; a < n; a += (kEThreads / kTile) * size)
                v += (long long)__ldg(in.h + a) * (int)spins[(size_t)(r0 + r) * n + __ldg(in.new2old + a)];
        atomicAdd(reinterpret_cast<unsigned long long*>(&sum[r]), (unsigned long long)v);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tmem, kCols);
    cl.sync();
    if (rank == 0 && tid < kTile && r0 + tid < count) {
        ExactAcc x;
        x.clear();
        long long total = 0;
        for (int p = 0; p < planes; ++p) {
            total = 0;
            for (int q = 0; q < size; ++q) total += cl.map_shared_rank(sum, q)[p * kTile + tid];
            if constexpr (!INT) {
                // total 2^(7 p), |total| < 2^38, in 32-bit limbs
                const bool neg = total < 0;
                const unsigned long long m = (unsigned long long)(neg ? -total : total);
                const int bit = kDigit * p, l0 = bit >> 5, sh = bit & 31;
                const unsigned long long lo = m << sh, hi = sh ? m >> (64 - sh) : 0ull;
                const long long d0 = (long long)(lo & 0xffffffffull), d1 = (long long)(lo >> 32), d2 = (long long)hi;
#pragma unroll
                for (int l = 0; l < kExactLimbs; ++l) {
                    const long long d = (l == l0 ? d0 : 0) + (l == l0 + 1 ? d1 : 0) + (l == l0 + 2 ? d2 : 0);
                    x.d[l] += neg ? -d : d;
                }
            }
        }
        e_out[r0 + tid] = INT ? (double)total : x.round(in.exact_e0);
        if (e_i64) e_i64[r0 + tid] = INT ? total : 0;
    }
    cl.sync();  // the other CTAs' sums stay until rank 0 has read them
}

template <bool INT>
cudaError_t launch_as(const DevInstance& in, const int8_t* spins, int32_t count, double* e, long long* e_i64,
                      int32_t* status, int planes, cudaStream_t st, int max_cluster)
{
    auto bytes = [](int np) {
        return 1024 + 2 * kBuffer<INT> + (size_t)kTile * kSpinLd + (size_t)np * kTile * sizeof(long long) +
               2 * sizeof(uint64_t);
    };
    const size_t smem = bytes(planes);
    const void* k = (const void*)dense_energy_kernel<INT>;
    // the limit is the process's: that of the largest pass, for every pass
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(kMaxPlanes));
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);  // clusters of 16
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kEThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // CTAs per vector group: the cluster size (up to 16 where the GPU is this
    // solve's alone, more than the portable 8) with the fewest waves per share of the tiles, the smaller one on a tie.
    // A cluster keeps inside one GPC, so the driver says how many fit at once. It
    // takes 5 us to say so, which up to kShortPass steps would not win back.
    // n = 2048, 512 vectors: 0.41 ms with up to 8 CTAs, 0.23 ms with 16.
    const int groups = (count + kTile - 1) / kTile, T = in.n / kTile + 1;
    const long long steps = (long long)T * (T + 1) * ((planes + kPlanesAtOnce<INT> - 1) / kPlanesAtOnce<INT>);
    int cs = 1;
    long long cost = 0;
    if (T == 1 || steps <= kShortPass) max_cluster = 0;  // one CTA per group
    for (int c = 1; c <= max_cluster && (long long)c <= (long long)T * (T + 1) / 2; c *= 2) {
        attr[0].val.clusterDim.x = (unsigned)c;
        cfg.gridDim = dim3((unsigned)(groups * c));
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            continue;
        }
        const long long now = (long long)((groups + fit - 1) / fit) * (16 / c);  // waves x sixteenths of the tiles
        if (cost == 0 || now < cost) {
            cost = now;
            cs = c;
        }
    }
    attr[0].val.clusterDim.x = (unsigned)cs;
    cfg.gridDim = dim3((unsigned)(groups * cs));
    DevInstance a = in;
    void* args[] = {&a, &spins, &count, &e, &e_i64, &status, &planes};
    return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace

cudaError_t launch_dense_energy(const DevInstance& in, const int8_t* spins, int32_t count, double* e,
                                long long* e_i64, int32_t* status, cudaStream_t st, int max_cluster)
{
    if (count <= 0) return cudaSuccess;
    if (in.integer) return launch_as<true>(in, spins, count, e, e_i64, status, 1, st, max_cluster);
    const int planes = std::min(kMaxPlanes, std::max(1, (in.exact_bits + kDigit - 1) / kDigit));
    return launch_as<false>(in, spins, count, e, e_i64, status, planes, st, max_cluster);
}

}  // namespace mars
