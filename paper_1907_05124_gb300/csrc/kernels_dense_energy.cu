// Exact energies of many spin vectors of one dense instance (Section 2, Eq. 2
// with each pair counted once), as a tiled integer quadratic form.
//
// Every coupling is an integer: J_ab itself for integer instances, else
// J_ab / 2^e0 (exact_sum.cuh), a two's complement number cut into bytes. The
// energy of a vector is then sum_d 256^d P_d with
//   P_d = sum_{a<b} byte_d(J_ab) s_a s_b,
// one small-integer quadratic form per byte plane (a single signed plane for
// integer instances), which dp4a sums four pairs at a time. Integer sums do
// not depend on their order, so the result is the exact sum, rounded once.
//
// Work: 128 x 128 tiles (ta <= tb) of J against RT spin vectors. A tile's
// bytes are made once in shared memory, straight from J (double -> bytes costs
// about 80 instructions per four couplings and four planes; no second copy of
// J, no work at ingest), and serve RT vectors. A warp owns 32 rows x 32
// vectors, a lane 4 x 8 of them: 12 16-byte loads feed 128 dp4a. The tiles of
// one vector group are dealt to the CTAs of a cluster, whose partial sums meet
// in distributed shared memory, so the pass needs no scratch in device memory.
//
// What bounds it: dp4a, which a GB300 SM issues at about 36 lanes a clock, and
// with 32 vectors the cutting of doubles into bytes (half of a tile's 16 us).
// Measured on a GB300 at n = 8192, 4096 vectors: 40.8 ms for FP32-valued
// Gaussian couplings (7 planes) and 5.7 ms for +-1, where the kernel this
// replaced (a thread per row of J, uncoalesced, every term added into eight
// 64-bit limbs) took about 1,490 and 160 ms; n = 2048, 512 vectors: 1.1 against
// 9.9 ms.
#include "device_common.cuh"
#include "exact_sum.cuh"
#include "mars_internal.h"

#include <cooperative_groups.h>

#include <algorithm>

namespace mars {
namespace {

namespace cg = cooperative_groups;

constexpr int kTile = 128;        // rows and columns of a J tile
constexpr int kStride = 144;      // bytes of a tile row in shared memory: rows 0..7 hit distinct banks
constexpr int kEThreads = 512;
constexpr int kMaxPlanes = 28;    // (220 bits + sign) in bytes, exact_span's limit
constexpr int kGroup = 4;         // byte planes made from one read of a tile
constexpr int kFlush = 8192;      // tiles a 32-bit partial may take: 8192 x 4 x 128 x 255 < 2^31

// byte * spin dot products: the top plane's bytes are signed, the others not.
template <bool SIGNED>
__device__ __forceinline__ int dot4(int a, int s, int acc)
{
    if constexpr (SIGNED) {
        asm("dp4a.s32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(a), "r"(s));
    } else {
        asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(acc) : "r"(a), "r"(s));
    }
    return acc;
}

// A lane's 4 rows x 8 vectors over bytes [16 k0, 16 k1) of the tile rows, then
// the rows' own spins: e[j] += sum_i s_{a_i, j} (row_i . vector_j).
template <bool SIGNED>
__device__ __forceinline__ void tile_dot(const unsigned char* J, const unsigned char* S, const unsigned char* A,
                                         int k0, int k1, int (&e)[8])
{
    int acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0;
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
        int4 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const int4*>(J + 8 * i * kStride + 16 * k);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int4 v = *reinterpret_cast<const int4*>(S + 4 * j * kStride + 16 * k);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i][j] = dot4<SIGNED>(w[i].x, v.x, acc[i][j]);
                acc[i][j] = dot4<SIGNED>(w[i].y, v.y, acc[i][j]);
                acc[i][j] = dot4<SIGNED>(w[i].z, v.z, acc[i][j]);
                acc[i][j] = dot4<SIGNED>(w[i].w, v.w, acc[i][j]);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) e[j] += acc[i][j] * (int)(signed char)A[4 * j * kStride + 8 * i];
}

// Bits [8 p0, 8 p0 + 32) of the two's complement integer v / 2^e0: the bytes of
// four planes at once.
__device__ __forceinline__ uint32_t plane_bytes(double v, int e0, int p0)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7ffu);
    long long sm = (long long)(bits & ((1ull << 52) - 1));
    if (ex) sm |= 1ll << 52;
    if (bits >> 63) sm = -sm;
    const int sh = 8 * p0 - ((ex ? ex : 1) - 1075 - e0);
    return sh >= 0 ? (uint32_t)(sm >> min(sh, 63)) : sh > -32 ? (uint32_t)((uint32_t)sm << -sh) : 0u;
}

// RT: spin vectors of a CTA, 128 or 32. With 128 the 16 warps are 4 row blocks
// x 4 vector blocks and a warp takes the planes of a group in turn; with 32
// they are 4 row blocks x 4 units, a unit being one plane of the group
// (couplings in FP64) or a quarter of the tile's columns (integer couplings).
template <int RT, bool INT>
__global__ void __launch_bounds__(kEThreads, 1) dense_energy_kernel(DevInstance in, const int8_t* __restrict__ spins,
                                                                    int count, double* e_out, long long* e_i64,
                                                                    int32_t* status, int planes)
{
    constexpr int kG = INT ? 1 : kGroup;
    constexpr bool kWide = RT == 128;
    extern __shared__ __align__(16) unsigned char esm[];
    unsigned char* sJ = esm;                             // [kG][128][kStride]
    unsigned char* sS = sJ + kG * kTile * kStride;       // [RT][kStride], the tile's columns' spins
    unsigned char* sA = sS + RT * kStride;               // [RT][kStride], its rows' spins
    long long* sum = reinterpret_cast<long long*>(sA + RT * kStride);  // [planes][RT]
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), size = (int)cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = in.n, r0 = (blockIdx.x / size) * RT;
    const bool hcol = !INT && in.h_f64 != nullptr;  // the field as a coupling to a spin n held at +1
    const int T = (n + (hcol ? 1 : 0) + kTile - 1) / kTile;
    const long long ntiles = (long long)T * (T + 1) / 2;
    for (int q = tid; q < planes * RT; q += kEThreads) sum[q] = 0;
    __syncthreads();

    const int ab = warp & 3, unit = warp >> 2;
    const int ag = lane & 7, rg = lane >> 3;
    const int rb = kWide ? unit : 0;
    const unsigned char* Jl = sJ + (ab * 32 + ag) * kStride;        // this lane's first row
    const unsigned char* Sl = sS + (rb * 32 + rg) * kStride;        // its first vector
    const unsigned char* Al = sA + (rb * 32 + rg) * kStride + ab * 32 + ag;

    // four spins of vector r as bytes, from new label b0 (0 past the end): one
    // word when the labels are the caller's and rows keep 4-byte alignment
    const bool words = in.identity && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(spins) & 3) == 0;
    auto spin_word = [&](int r, int b0, bool col) -> uint32_t {
        uint32_t w = 0;
        if (words && b0 < n) {
            if (r0 + r < count) {
                w = __ldg(reinterpret_cast<const uint32_t*>(spins + (size_t)(r0 + r) * n + b0));
                if (__vabsss4(w) != 0x01010101u) atomicExch(status, (int)kDevBadIndex);
            }
            return w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int b = b0 + i;
            int v = 0;
            if (b < n) {
                if (r0 + r < count) {
                    v = spins[(size_t)(r0 + r) * n + __ldg(in.new2old + b)];
                    if (v != 1 && v != -1) atomicExch(status, (int)kDevBadIndex);
                }
            } else if (col && hcol && b == n) {
                v = 1;
            }
            w |= ((uint32_t)v & 0xffu) << (8 * i);
        }
        return w;
    };
    // J[a][b0 .. b0+3] above the diagonal (0 elsewhere)
    auto int_word = [&](int a, int b0) -> uint32_t {
        uint32_t w = 0;
        if (a >= n || b0 >= n) return 0;
        if ((n & 3) == 0) {
            w = __ldg(reinterpret_cast<const uint32_t*>(in.J_i8 + (size_t)a * n + b0));
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (b0 + i <= a) w &= ~(0xffu << (8 * i));
            return w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (b0 + i < n && b0 + i > a) w |= ((uint32_t)in.J_i8[(size_t)a * n + b0 + i] & 0xffu) << (8 * i);
        return w;
    };
    auto f64_at = [&](int a, int b) -> double {
        if (a >= n || b <= a) return 0.0;
        return b < n ? __ldg(in.J_f64 + (size_t)a * n + b) : hcol && b == n ? __ldg(in.h_f64 + a) : 0.0;
    };

    for (int p0 = 0; p0 < planes; p0 += kG) {
        constexpr int kE = kWide ? kG : 1;
        int e[kE][8];
#pragma unroll
        for (int g = 0; g < kE; ++g)
#pragma unroll
            for (int j = 0; j < 8; ++j) e[g][j] = 0;
        // this lane's partial sums to shared memory
        auto flush = [&]() {
#pragma unroll
            for (int g = 0; g < kE; ++g) {
                const int p = p0 + (kWide ? g : INT ? 0 : unit);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    long long v = e[g][j];
                    v += shfl_xor(v, 1);
                    v += shfl_xor(v, 2);
                    v += shfl_xor(v, 4);
                    if (ag == 0 && p < planes)
                        atomicAdd(reinterpret_cast<unsigned long long*>(&sum[p * RT + rb * 32 + rg + 4 * j]),
                                  (unsigned long long)v);
                    e[g][j] = 0;
                }
            }
        };
        int held = 0;
        for (long long t = rank; t < ntiles; t += size) {
            int tb = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
            while ((long long)(tb + 1) * (tb + 2) / 2 <= t) ++tb;
            while ((long long)tb * (tb + 1) / 2 > t) --tb;
            const int ta = (int)(t - (long long)tb * (tb + 1) / 2);
            __syncthreads();  // the previous tile has been read
#pragma unroll 4
            for (int q = tid; q < RT * (kTile / 4); q += kEThreads) {
                const int r = q / (kTile / 4), w = q % (kTile / 4);
                *reinterpret_cast<uint32_t*>(sS + r * kStride + 4 * w) = spin_word(r, tb * kTile + 4 * w, true);
                *reinterpret_cast<uint32_t*>(sA + r * kStride + 4 * w) = spin_word(r, ta * kTile + 4 * w, false);
            }
            // 8 words of 4 couplings per thread; in FP64 the loads of half of
            // them are in flight before the first is cut into bytes
            const int w = tid % (kTile / 4), row0 = tid / (kTile / 4), b0 = tb * kTile + 4 * w;
            unsigned char* dst = sJ + row0 * kStride + 4 * w;
            if constexpr (INT) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    *reinterpret_cast<uint32_t*>(dst + 16 * u * kStride) = int_word(ta * kTile + row0 + 16 * u, b0);
            } else {
#pragma unroll 1
                for (int u = 0; u < 8; u += 4) {
                    double v[4][4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int i = 0; i < 4; ++i) v[q][i] = f64_at(ta * kTile + row0 + 16 * (u + q), b0 + i);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t c[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) c[i] = plane_bytes(v[q][i], in.exact_e0, p0);
                        // 4 x 4 byte transpose: couplings -> planes
                        const uint32_t lo0 = __byte_perm(c[0], c[1], 0x5140), lo1 = __byte_perm(c[2], c[3], 0x5140);
                        const uint32_t hi0 = __byte_perm(c[0], c[1], 0x7362), hi1 = __byte_perm(c[2], c[3], 0x7362);
                        unsigned char* o = dst + 16 * (u + q) * kStride;
                        *reinterpret_cast<uint32_t*>(o) = __byte_perm(lo0, lo1, 0x5410);
                        *reinterpret_cast<uint32_t*>(o + kTile * kStride) = __byte_perm(lo0, lo1, 0x7632);
                        *reinterpret_cast<uint32_t*>(o + 2 * kTile * kStride) = __byte_perm(hi0, hi1, 0x5410);
                        *reinterpret_cast<uint32_t*>(o + 3 * kTile * kStride) = __byte_perm(hi0, hi1, 0x7632);
                    }
                }
            }
            __syncthreads();
            if constexpr (INT) {
                if constexpr (kWide) tile_dot<true>(Jl, Sl, Al, 0, 8, e[0]);
                else tile_dot<true>(Jl, Sl, Al, 2 * unit, 2 * unit + 2, e[0]);
            } else if constexpr (kWide) {
#pragma unroll
                for (int g = 0; g < kG; ++g) {
                    if (p0 + g < planes - 1) tile_dot<false>(Jl + g * kTile * kStride, Sl, Al, 0, 8, e[g]);
                    else if (p0 + g == planes - 1) tile_dot<true>(Jl + g * kTile * kStride, Sl, Al, 0, 8, e[g]);
                }
            } else {
                if (p0 + unit < planes - 1) tile_dot<false>(Jl + unit * kTile * kStride, Sl, Al, 0, 8, e[0]);
                else if (p0 + unit == planes - 1) tile_dot<true>(Jl + unit * kTile * kStride, Sl, Al, 0, 8, e[0]);
            }
            if (++held == kFlush) {
                flush();
                held = 0;
            }
        }
        flush();
    }
    if (INT && in.h) {  // integer fields (up to 2^24) do not fit a byte plane
        constexpr int kPer = kEThreads / RT;
        const int r = tid % RT;
        long long v = 0;
        if (r0 + r < count)
            for (int a = tid / RT + kPer * rank; a < n; a += kPer * size)
                v += (long long)__ldg(in.h + a) * (int)spins[(size_t)(r0 + r) * n + __ldg(in.new2old + a)];
        __syncthreads();
        atomicAdd(reinterpret_cast<unsigned long long*>(&sum[r]), (unsigned long long)v);
    }
    cl.sync();
    if (rank == 0 && tid < RT && r0 + tid < count) {
        ExactAcc x;
        x.clear();
        long long total = 0;
        for (int p = 0; p < planes; ++p) {
            total = 0;
            for (int q = 0; q < size; ++q) total += cl.map_shared_rank(sum, q)[p * RT + tid];
            if constexpr (!INT) {
                const bool neg = total < 0;
                const unsigned long long m = (unsigned long long)(neg ? -total : total) << (8 * (p & 3));
                const long long lo = (long long)(m & 0xffffffffull), hi = (long long)(m >> 32);
                const int l0 = p >> 2;
#pragma unroll
                for (int l = 0; l < kExactLimbs; ++l)
                    x.d[l] += (l == l0 ? (neg ? -lo : lo) : 0) + (l == l0 + 1 ? (neg ? -hi : hi) : 0);
            }
        }
        e_out[r0 + tid] = INT ? (double)total : x.round(in.exact_e0);
        if (e_i64) e_i64[r0 + tid] = INT ? total : 0;
    }
    cl.sync();  // the other CTAs' sums stay until rank 0 has read them
}

template <int RT, bool INT>
cudaError_t launch_as(const DevInstance& in, const int8_t* spins, int32_t count, double* e, long long* e_i64,
                      int32_t* status, int planes, int sms, cudaStream_t st)
{
    const size_t smem = (size_t)(INT ? 1 : kGroup) * kTile * kStride + 2 * (size_t)RT * kStride +
                        (size_t)planes * RT * sizeof(long long);
    const void* k = (const void*)dense_energy_kernel<RT, INT>;
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
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
    // CTAs per vector group: the cluster size with the fewest waves per share
    // of the tiles, the smaller one on a tie. A cluster keeps inside one GPC,
    // so the driver says how many fit at once (128 CTAs in clusters of 8 take
    // two waves on 152 SMs).
    const int groups = (count + RT - 1) / RT, T = in.n / kTile + 1;
    int cs = 1;
    long long cost = 0;
    for (int c = 1; c <= 8 && (long long)c <= (long long)T * (T + 1) / 2; c *= 2) {
        attr[0].val.clusterDim.x = (unsigned)c;
        cfg.gridDim = dim3((unsigned)(groups * c));
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            continue;
        }
        const long long now = (long long)((groups + fit - 1) / fit) * (8 / c);  // waves x eighths of the tiles
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
                                long long* e_i64, int32_t* status, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int planes = in.integer ? 1 : std::min(kMaxPlanes, std::max(1, (in.exact_bits + 1 + 7) / 8));
    // 128 vectors per CTA amortise a tile's bytes four times better; below
    // about half a GPU of such CTAs (8 to a cluster) 32 spread further.
    // n = 8192, Gaussian, ms with 32 / 128: 256 vectors 8.7 / 20.5, 1024
    // 17.1 / 20.5, 1216 25.8 / 20.4, 4096 67.9 / 40.8.
    const bool wide = (count + 127) / 128 * 8 > sms / 2;
    if (in.integer)
        return wide ? launch_as<128, true>(in, spins, count, e, e_i64, status, planes, sms, st)
                    : launch_as<32, true>(in, spins, count, e, e_i64, status, planes, sms, st);
    return wide ? launch_as<128, false>(in, spins, count, e, e_i64, status, planes, sms, st)
                : launch_as<32, false>(in, spins, count, e, e_i64, status, planes, sms, st);
}

}  // namespace mars
