// Forward of a linear layer on a few rows (at most 16) for sm_100a:  out[m, o] = sum_k inp[m, k] W[o, k]
//
// Every weight is used for a handful of rows, so the product is a stream of the weights and, for the
// sizes of one layer (a few megabytes over 148 SMs), not even that: what counts is the chain of
// latencies of one CTA. The tcgen05 kernels pay for descriptors, TMA (about 900 cycles to the first
// tile), MMAs that take 70 cycles each however few columns they have, the commit and the TMEM read
// one after the other. Here a CTA takes 16 weight rows and all of K: each of its eight warps loads
// 32-wide pieces of K straight from global memory into registers (16 bytes per lane; the lane's
// eight k go to both operands alike, so the order of k inside a piece does not matter), several of
// them in flight at once, multiplies with warp-level MMAs (m16n8k16: weights x rows) and the eight
// partial sums meet in shared memory, always in the same order. The weights are requested into L2
// before the kernel waits for the one before it. Where K is long and there are few features, the
// CTAs of a cluster share K and read each other's sums.
//
// Chained launches, 8 rows, against gemm_kernel: 768 -> 768 1.8 us (6.7), 768 -> 3072 2.5 us (7.8),
// 3072 -> 768 3.2 us (19.9), 768 -> 50304 14.5 us (17.2; 77 MB of weights take 12 us).
#pragma once
#include "gemm_sm100.cuh"

namespace nb {

constexpr int kRowsThreads = 256;
constexpr int kRowsWarps = 8;
constexpr int kRowsFeatures = 16;  // weight rows per CTA (SwiGLU: 16 gate + 16 up)
constexpr int kRowsMax = 16;
constexpr int kRowsMaxSplit = 8;

struct RowsParams {
    const __nv_bfloat16 *inp, *weight, *bias;
    __nv_bfloat16 *out, *pre;
    int M, K, N;      // N: weight rows (SwiGLU: 2 H)
    int swiglu_h;
    int ksplit;       // CTAs of a cluster that share K
};

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 ld_stream(const __nv_bfloat16 *p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// NT: groups of eight rows. At least two CTAs have to fit an SM (128 registers a thread), or the next
// launch of the chain cannot start while this one runs: 16 rows, or gate and up rows, with one CTA (138
// and 168 registers, more pieces of K in flight) took 6.0 us against 3.6 (16 rows, 3072 -> 768), 4.2
// against 2.9 (768 -> 3072), 10.3 against 4.2 (8 rows, SwiGLU, 4096 -> 1024). MANY: there are several
// CTAs of work per SM: fewer pieces of K in flight per thread and four CTAs on an SM (8 rows,
// 768 -> 50304: 14.5 us against 22.7 us with two, five or six have too few registers, 15.7 and 17.1 us;
// 16 rows, 1024 -> 8192: 4.6 us against 5.8 us with two and 6.1 us with three).
template <int NT, int EPI, bool MANY>
__global__ void __launch_bounds__(kRowsThreads, MANY ? 4 : 2)
rows_kernel(const RowsParams p)
{
    constexpr int SETS = EPI == kEpiSwiglu ? 2 : 1;  // gate and up rows
    constexpr int U = MANY ? (NT == 2 ? 2 : 3) : (SETS == 2 || NT == 2) ? 3 : 6;  // pieces of K in flight
    constexpr int LD = 18;  // floats from one row's sixteen partial sums to the next
    __shared__ float part[SETS][kRowsWarps][NT * 8][LD];
    const int warp = static_cast<int>(threadIdx.x >> 5), lane = static_cast<int>(threadIdx.x & 31);
    const int g = lane >> 2, t = lane & 3;
    const int rank = static_cast<int>(blockIdx.x) % p.ksplit;
    const int f0 = static_cast<int>(blockIdx.x) / p.ksplit * kRowsFeatures;
    const int pieces = (p.K + 31) / 32;  // of K, 32 wide
    const int pc0 = pieces * rank / p.ksplit, pc1 = pieces * (rank + 1) / p.ksplit;
    const int k0 = pc0 * 32, k1 = min(pc1 * 32, p.K);
    const int span = EPI == kEpiSwiglu ? p.swiglu_h : p.N;
    // rows beyond the end are read as the last one and never stored
    const __nv_bfloat16 *wrow[SETS][2];
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            wrow[s][h] = p.weight + static_cast<long long>(s * p.swiglu_h + min(f0 + g + 8 * h, span - 1)) * p.K + t * 8;
    const __nv_bfloat16 *xrow[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) xrow[n] = p.inp + static_cast<long long>(min(n * 8 + g, p.M - 1)) * p.K + t * 8;

    // the CTA's weights into L2: a hint, nothing is read before the wait below
    if (threadIdx.x < SETS * kRowsFeatures) {
        const int s = threadIdx.x / kRowsFeatures, f = min(f0 + static_cast<int>(threadIdx.x) % kRowsFeatures, span - 1);
        const __nv_bfloat16 *w = p.weight + static_cast<long long>(s * p.swiglu_h + f) * p.K + k0;
        if (k1 > k0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(w), "r"((k1 - k0) * 2) : "memory");
    }
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    // two neighbouring features of one row per thread at the end; their bias is fetched with the operands
    // (fetched when it is needed it adds an L2 latency to the chain)
    constexpr int ITEMS = NT * 8 * (kRowsFeatures / 2);
    static_assert(ITEMS <= kRowsThreads, "one item per thread");
    const int m = static_cast<int>(threadIdx.x) / (kRowsFeatures / 2), f = (static_cast<int>(threadIdx.x) % (kRowsFeatures / 2)) * 2;
    const bool mine = static_cast<int>(threadIdx.x) < ITEMS && (p.ksplit == 1 || m % p.ksplit == rank) && m < p.M &&
                      f0 + f < span;
    float bias[SETS][2];
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
        bias[s][0] = bias[s][1] = 0.0f;
        if (!MANY && mine && p.bias != nullptr) {  // only 2-byte aligned: element by element
            bias[s][0] = __bfloat162float(p.bias[s * p.swiglu_h + f0 + f]);
            bias[s][1] = __bfloat162float(p.bias[s * p.swiglu_h + f0 + f + 1]);
        }
    }

    float acc[SETS][NT][4];
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[s][n][k] = 0.0f;

    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int c0 = pc0 + warp; c0 < pc1; c0 += kRowsWarps * U) {
        uint4 a[U][SETS][2], b[U][NT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = (c0 + u * kRowsWarps) * 32;
            const bool in = k + t * 8 < k1;  // K is a multiple of 8: a lane's piece exists or does not
#pragma unroll
            for (int s = 0; s < SETS; ++s)
#pragma unroll
                for (int h = 0; h < 2; ++h) a[u][s][h] = in ? ld_stream(wrow[s][h] + k) : zero;
#pragma unroll
            for (int n = 0; n < NT; ++n)
                b[u][n] = in ? ptx::ld_global_v4(xrow[n] + k) : zero;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int s = 0; s < SETS; ++s)
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    mma_16816(acc[s][n], a[u][s][0].x, a[u][s][1].x, a[u][s][0].y, a[u][s][1].y, b[u][n].x, b[u][n].y);
                    mma_16816(acc[s][n], a[u][s][0].z, a[u][s][1].z, a[u][s][0].w, a[u][s][1].w, b[u][n].z, b[u][n].w);
                }
    }
    // accumulator: features g, g + 8 of rows 2t, 2t + 1
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            part[s][warp][n * 8 + 2 * t][g] = acc[s][n][0];
            part[s][warp][n * 8 + 2 * t + 1][g] = acc[s][n][1];
            part[s][warp][n * 8 + 2 * t][g + 8] = acc[s][n][2];
            part[s][warp][n * 8 + 2 * t + 1][g + 8] = acc[s][n][3];
        }
    __syncthreads();
    float z[SETS][2];
    const bool split = p.ksplit > 1;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
        z[s][0] = z[s][1] = 0.0f;
        if (static_cast<int>(threadIdx.x) < ITEMS)
#pragma unroll
            for (int w = 0; w < kRowsWarps; ++w) {
                const float2 v = *reinterpret_cast<const float2 *>(&part[s][w][m][f]);
                z[s][0] += v.x;
                z[s][1] += v.y;
            }
    }
    if (split) {
        // the CTA's sums stand where warp 0's were (each thread overwrites what it alone has read);
        // rank r finishes the rows m with m % ksplit == r
#pragma unroll
        for (int s = 0; s < SETS; ++s)
            if (static_cast<int>(threadIdx.x) < ITEMS) *reinterpret_cast<float2 *>(&part[s][0][m][f]) = make_float2(z[s][0], z[s][1]);
        ptx::cluster_sync();
        if (mine)
#pragma unroll
            for (int s = 0; s < SETS; ++s) {
                z[s][0] = z[s][1] = 0.0f;
                const uint32_t at = ptx::smem_u32(&part[s][0][m][f]);
                for (int r = 0; r < p.ksplit; ++r) {
                    float2 v;
                    ptx::ld_cluster_f32x2(ptx::mapa(at, static_cast<uint32_t>(r)), v);
                    z[s][0] += v.x;
                    z[s][1] += v.y;
                }
            }
        ptx::cluster_sync();  // nobody leaves while a peer may still read its sums
    }
    if (!mine) return;
    const int col = f0 + f;
    if (MANY && p.bias != nullptr)  // other CTAs of the SM cover the latency, and registers are scarce
#pragma unroll
        for (int s = 0; s < SETS; ++s) {
            bias[s][0] = __bfloat162float(p.bias[s * p.swiglu_h + col]);
            bias[s][1] = __bfloat162float(p.bias[s * p.swiglu_h + col + 1]);
        }
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
        z[s][0] += bias[s][0];
        z[s][1] += bias[s][1];
    }
    const long long row = m;
    uint32_t o;
    if (EPI == kEpiStore) {
        o = ptx::pack_bf16x2(z[0][0], z[0][1]);
    } else if (EPI == kEpiGelu) {
        *reinterpret_cast<uint32_t *>(p.pre + row * p.N + col) = ptx::pack_bf16x2(z[0][0], z[0][1]);
        o = ptx::pack_bf16x2(gelu_fwd(z[0][0]), gelu_fwd(z[0][1]));
    } else {
        *reinterpret_cast<uint32_t *>(p.pre + row * p.N + col) = ptx::pack_bf16x2(z[0][0], z[0][1]);
        *reinterpret_cast<uint32_t *>(p.pre + row * p.N + p.swiglu_h + col) = ptx::pack_bf16x2(z[SETS - 1][0], z[SETS - 1][1]);
        o = ptx::pack_bf16x2(silu_fwd(z[0][0]) * z[SETS - 1][0], silu_fwd(z[0][1]) * z[SETS - 1][1]);
    }
    *reinterpret_cast<uint32_t *>(p.out + row * span + col) = o;
}

}  // namespace nb
