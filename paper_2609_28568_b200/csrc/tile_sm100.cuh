// Small-problem GEMM for sm_100a: one output tile per CTA, K split over a thread-block cluster.
//
// The persistent kernels (gemm_kernel, layer_bwd_kernel) work in 256-row or 256-column tiles. A
// problem of a few hundred rows has a handful of those: most SMs idle, each busy one works through
// all of K by itself (512 tensor-core cycles per 64 of K, whatever part of the tile is padding), and
// the epilogue of a 256-wide tile is exposed at the end. What bounds such a problem is latency, so
// here a CTA takes a 128 x BN tile (BN = 32 / 64 / 128, or 192 without a split), and where there are far fewer tiles than SMs
// the CTAs of a cluster share a tile's K range: each accumulates its part in TMEM and sends every
// other CTA that one's slice of the columns through distributed shared memory, and after a barrier
// of the cluster adds the parts it got in rank order (a fixed order: products do not vary; the bias
// gradient's partial sums meet in shared memory in any order) and runs the epilogue on its slice.
//
//   warp 0      TMA producer
//   warp 1      MMA issuer, TMEM allocation
//   warps 2..9  before they wait for the previous kernel of the stream they ask for the first weight
//               tiles of the CTA to be brought into L2 (a hint: nothing is read into the SM); then
//               epilogue: TMEM -> registers -> bias / activation -> the warp's box in the drained
//               pipeline stages -> whole rows of the box to global memory (no TMA store to wait for:
//               a shorter chain), or, for fp32 weight gradients, TMA stores / reduce-adds
//
// The A tile's slot holds only the rows that exist when there are fewer than 128 (a_slot): the
// tensor core then multiplies whatever follows in shared memory for the other rows, which touches
// no valid row of the result.
//
// Chained launches against the persistent kernels: forward 1024 rows 768 -> 2304 6.2 us (8.7),
// 1024 rows 3072 -> 768 11.4 us (18.5), 128 rows 768 -> 768 4.4 us (7.3); dinp 2048 rows 3072 -> 768
// 13.1 us (18.5); backward 512 rows 768 x 768 5.5 us (14.1 with the clearing of dweight, 8.3 without).
#pragma once
#include "gemm_sm100.cuh"

namespace nb {

constexpr int kTileMaxStages = 16;
constexpr int kTileThreads = 320;
constexpr int kTilePrefetch = 1;  // weight k-blocks each epilogue warp asks for ahead of time

struct TileJob {
    int M, N;
    int tiles_m, tiles_n;
    int kblocks;        // ceil(K / 64)
    int kblocks_ext;    // k-blocks of the adapter term (A2 . B2^T), after the last one of the base product
    uint32_t a_slot;    // bytes of one A tile in shared memory (a multiple of 1024): what its boxes deliver
    int stages;
    int ctas;           // CTAs of this job: tiles (x cluster size where K is split)
    float alpha;
    const __nv_bfloat16 *bias;
    __nv_bfloat16 *D;
    long long d_ld;
    __nv_bfloat16 *E;   // pre-activation: written (GELU, SwiGLU) or read (gelu' of the producer)
    long long e_ld;
    int swiglu_h;
    int reduce;         // fp32 result: 1 reduce-add, 0 overwrite
    float *dbias;       // fp32 result: column sums of dz, [M], or null
    int dbias_add;      // add to what dbias holds
    int wait_ext;       // of this job's operands the launch before this one (trigger_late) makes only A2:
                        // only the adapter term's loads wait for it
};

struct TileParams {
    TileJob job[2];
    int cluster;        // CTAs per cluster; job 0 splits K over it, job 1 does not
    int trigger_late;   // the next launch may start once everything before this one is done, no sooner
    int *status;
    unsigned long long timeout_ns;
};

struct TileMaps {  // one job's tensor maps
    const CUtensorMap *A, *B, *A2, *B2, *D;
};

template <int BN>
struct TileGeom {
    static constexpr uint32_t B_BYTES = BN * kBlockK * 2;
    static constexpr uint32_t TMEM_COLS = BN == 192 ? 256 : BN;  // a power of two
    // behind the stages: slices received from the cluster (only where K is split), then the bias /
    // partial-sum line and the barriers
    static constexpr uint32_t RECV_BYTES = (kBlockM + 1) * BN * 4;
    static constexpr uint32_t LINE_BYTES = BN > 128 ? BN * 4 : 512;
    static constexpr uint32_t TAIL_BYTES = LINE_BYTES + 512;
};

// offsets inside the barrier block
//   8 s          full[s]          8 (16 + s)  empty[s]
//   8 * 32       accumulator complete
//   8 * 34       TMEM base address (4 bytes), abort flag (4 bytes)
constexpr uint32_t kTileBarAcc = 8 * 32, kTileTmemSlot = 8 * 34, kTileAbort = 8 * 34 + 4;

// Sixteen columns of this thread's row.
__device__ __forceinline__ void tile_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    ptx::tmem_ld_32x16_wait(taddr, r);
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Eight consecutive columns of one row through the epilogue: the result, and for GELU z.
template <int EPI>
__device__ __forceinline__ void tile_math8(const TileJob &j, const float *v, uint32_t bias_s, int col_in_tile,
                                           const uint4 &e, uint4 &out, uint4 &pre)
{
    uint32_t w[4];
    if (EPI == kEpiMulGeluGrad) {
        const uint32_t x[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[k] = pack_f2_bf16x2(mul_gelu_bwd2(ptx::make_f2(v[2 * k], v[2 * k + 1]),
                                                ptx::make_f2_bits(x[k] << 16, x[k] & 0xffff0000u)));
    } else {
        float4 b0, b1;
        ptx::ld_shared_f32x4(bias_s + 4u * static_cast<uint32_t>(col_in_tile), b0);
        ptx::ld_shared_f32x4(bias_s + 4u * static_cast<uint32_t>(col_in_tile) + 16u, b1);
        const ptx::f2 al = ptx::make_f2(j.alpha, j.alpha);
        ptx::f2 z[4];
        z[0] = ptx::fma2(ptx::make_f2(v[0], v[1]), al, ptx::make_f2(b0.x, b0.y));
        z[1] = ptx::fma2(ptx::make_f2(v[2], v[3]), al, ptx::make_f2(b0.z, b0.w));
        z[2] = ptx::fma2(ptx::make_f2(v[4], v[5]), al, ptx::make_f2(b1.x, b1.y));
        z[3] = ptx::fma2(ptx::make_f2(v[6], v[7]), al, ptx::make_f2(b1.z, b1.w));
        if (EPI == kEpiGelu) {
            pre = make_uint4(pack_f2_bf16x2(z[0]), pack_f2_bf16x2(z[1]), pack_f2_bf16x2(z[2]), pack_f2_bf16x2(z[3]));
#pragma unroll
            for (int k = 0; k < 4; ++k) z[k] = gelu_fwd2(z[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = pack_f2_bf16x2(z[k]);
    }
    out = make_uint4(w[0], w[1], w[2], w[3]);
}

// A warp's 32 x COLS results leave through its own piece of shared memory, so that a store covers
// whole rows of the piece and not 16 bytes of each of 32 rows (with those, the epilogue of a 128 x 128
// tile took longer than its twelve k-blocks). 16-byte chunk c of row r lies at r * COLS * 2 +
// ((c ^ swizzle(r)) << 4).
template <int COLS>
struct WarpBox {
    static constexpr int CH = COLS / 8;             // chunks per row: 2, 4 or 8
    static constexpr uint32_t BYTES = 32 * COLS * 2;
    static __device__ __forceinline__ uint32_t pos(int r, int c)
    {
        const int x = CH == 8 ? (r & 7) : CH == 4 ? ((r >> 1) & 3) : ((r >> 2) & 1);
        return static_cast<uint32_t>(r * (COLS * 2) + ((c ^ x) << 4));
    }
    // rows [0, rows) of the box to `dst` (its first row and column), columns below `cols` only
    static __device__ __forceinline__ void flush(uint32_t box, __nv_bfloat16 *dst, long long ld, int rows, int cols,
                                                 int lane)
    {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < CH; ++i) {
            const int r = i * (32 / CH) + lane / CH, c = lane % CH;
            uint4 v;
            ptx::ld_shared_v4(box + pos(r, c), v.x, v.y, v.z, v.w);
            if (r < rows && c * 8 < cols) *reinterpret_cast<uint4 *>(dst + r * ld + c * 8) = v;
        }
    }
};

// One CTA's work on one tile. `tile` counts the job's tiles (row tiles fastest), `rank` is this
// CTA's share of K among `cluster` (1: all of K). Every thread of the CTA calls it.
template <int BN, bool A_MN, bool B_MN, int EPI>
__device__ __forceinline__ void tile_body(const TileJob &j, const TileMaps &t, uint32_t smem, int tile, int rank,
                                          int cluster, const TileParams &p)
{
    int *const status = p.status;
    const unsigned long long timeout_ns = p.timeout_ns;
    using G = TileGeom<BN>;
    const int warp = static_cast<int>(threadIdx.x >> 5);
    const int lane = static_cast<int>(threadIdx.x & 31);
    const int stages = j.stages;
    const uint32_t off_b = static_cast<uint32_t>(stages) * j.a_slot;
    const uint32_t off_recv = off_b + static_cast<uint32_t>(stages) * G::B_BYTES;
    const uint32_t off_line = off_recv + (cluster > 1 ? G::RECV_BYTES : 0u);
    const uint32_t line = smem + off_line;          // floats: bias of the tile / dbias partial sums
    const uint32_t bar0 = line + G::LINE_BYTES;
    auto full_bar = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(s); };
    auto empty_bar = [&](int s) { return bar0 + 8u * static_cast<uint32_t>(kTileMaxStages + s); };
    const uint32_t acc_bar = bar0 + kTileBarAcc;
    const uint32_t abort_addr = bar0 + kTileAbort;

    const int m_blk = tile % j.tiles_m, n_blk = tile / j.tiles_m;
    const int m0 = m_blk * kBlockM;
    constexpr int n_span = EPI == kEpiSwiglu ? BN / 2 : BN;  // columns of the result per tile
    const int n0 = n_blk * n_span;
    const int rows = min(kBlockM, j.M - m0);
    const int kb0 = j.kblocks * rank / cluster, kb1 = j.kblocks * (rank + 1) / cluster;
    const int kb_end = kb1 + (rank == cluster - 1 ? j.kblocks_ext : 0);
    const bool sum_dz = EPI == kEpiF32 && j.dbias != nullptr && n_blk == 0;

    const bool smem_ok = (smem & 1023u) == 0;
    if (!smem_ok && threadIdx.x == 0 && atomicCAS(status, 0, kStatusBadSmem) == 0)
        status[2] = static_cast<int>(blockIdx.x);

    if (warp == 0) {
        // one lane per stage: a lane after the other would spend longer here than a k-block takes
        if (lane < stages) {
            ptx::mbar_init(full_bar(lane), 1);
            // the tensor core has read the stage; with the bias gradient one epilogue warp has too
            ptx::mbar_init(empty_bar(lane), sum_dz ? 2 : 1);
        }
        if (lane == 31) {
            ptx::mbar_init(acc_bar, 1);
            ptx::st_shared_u32_volatile(abort_addr, 0);
        }
        ptx::fence_barrier_init();
        if (lane == 30) {
            ptx::prefetch_tmap(t.A);
            ptx::prefetch_tmap(t.B);
            if (EPI == kEpiF32) ptx::prefetch_tmap(t.D);
        }
        __syncwarp();
    }
    if (warp == 1) {
        ptx::tmem_alloc<1>(bar0 + kTileTmemSlot, G::TMEM_COLS);
        ptx::tmem_relinquish<1>();
    }
    // B boxes: a K-major tile is one box of BN rows (SwiGLU: the gate and the up rows), an MN-major
    // tile one box per 64 columns
    constexpr int B_BOXES = EPI == kEpiSwiglu ? 2 : B_MN ? BN / 64 : 1;
    constexpr uint32_t B_BOX_BYTES = G::B_BYTES / B_BOXES;
    auto b_row = [&](int i) { return EPI == kEpiSwiglu ? i * j.swiglu_h + n0 : n0; };
    if (warp >= 2 && EPI != kEpiF32) {
        // B is the weight: its tiles may be brought into L2 while the previous kernel still runs (issued
        // by one thread this took longer than the rest of the set-up)
        if (ptx::elect_one()) {
#pragma unroll
            for (int r = 0; r < kTilePrefetch; ++r) {
                const int kb = kb0 + warp - 2 + r * kEpiWarps;
                if (kb >= kb1) break;
#pragma unroll
                for (int i = 0; i < B_BOXES; ++i) {
                    if (B_MN) ptx::tma_prefetch_2d(t.B, n0 + i * 64, kb * kBlockK);
                    else ptx::tma_prefetch_2d(t.B, kb * kBlockK, b_row(i));
                }
            }
        }
        __syncwarp();
    }
    ptx::tc_fence_before();
    if (cluster > 1) ptx::cluster_sync();  // the peers' barriers are initialised before anyone sends to them
    else __syncthreads();
    ptx::tc_fence_after();
    // nothing above read or wrote global memory: it may overlap the previous kernel's tail
    if (!p.trigger_late) ptx::grid_launch_dependents();
    if (!j.wait_ext) ptx::grid_dependency_wait();
    if (p.trigger_late) ptx::grid_launch_dependents();
    const uint32_t tmem = ptx::ld_shared_u32_volatile(bar0 + kTileTmemSlot);
    const WaitCtx wctx{abort_addr, status, timeout_ns};
    const WaitCtx wctx_epi{abort_addr, status, 2 * timeout_ns};

    // the loads of one k-block into its stage
    auto issue = [&](int kb, int stage) {
        const bool ext = kb >= kb1;
        if (ext && j.wait_ext) ptx::grid_dependency_wait();
        const CUtensorMap *mapA = ext ? t.A2 : t.A;
        const CUtensorMap *mapB = ext ? t.B2 : t.B;
        const int k0 = (ext ? kb - kb1 : kb) * kBlockK;
        const uint32_t fb = full_bar(stage);
        ptx::mbar_expect_tx(fb, j.a_slot + G::B_BYTES);
        const uint32_t sa = smem + static_cast<uint32_t>(stage) * j.a_slot;
        const uint32_t sb = smem + off_b + static_cast<uint32_t>(stage) * G::B_BYTES;
#pragma unroll
        for (int i = 0; i < B_BOXES; ++i) {
            if (B_MN) ptx::tma_load_2d(sb + i * B_BOX_BYTES, mapB, fb, n0 + i * 64, k0);
            else ptx::tma_load_2d(sb + i * B_BOX_BYTES, mapB, fb, k0, b_row(i));
        }
        if (A_MN) {
#pragma unroll
            for (int i = 0; i < 2; ++i) ptx::tma_load_2d(sa + i * 8192u, mapA, fb, m0 + i * 64, k0);
        } else {
            ptx::tma_load_2d(sa, mapA, fb, k0, m0);
        }
    };
    // The first fill of the ring is shared among all warps but the MMA issuer's: issuing one box takes
    // a thread about 130 cycles, so a k-block's loads take one thread longer than the tensor core
    // takes to consume them.
    if (smem_ok && warp != 1) {
        if (ptx::elect_one()) {
            const int kb_fill = min(kb_end, kb0 + stages);
            for (int kb = kb0 + (warp == 0 ? 0 : warp - 1); kb < kb_fill; kb += kTileThreads / 32 - 1) issue(kb, kb - kb0);
        }
        __syncwarp();
    }

    if (!smem_ok) {
        // fall through to the common exit
    } else if (warp == 0) {
        // ------------------------------------------------------------ TMA producer: what the ring did not hold
        if (ptx::elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = kb0 + stages; kb < kb_end; ++kb) {
                if (!wait_barrier(wctx, empty_bar(stage), phase, 100 + stage)) break;
                issue(kb, stage);
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (ptx::elect_one()) {
            constexpr uint32_t idesc = make_idesc(kBlockM, BN, A_MN, B_MN);
            constexpr uint32_t a_step = A_MN ? (2048u >> 4) : (32u >> 4);
            constexpr uint32_t b_step = B_MN ? (2048u >> 4) : (32u >> 4);
            int stage = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int kb = kb0; kb < kb_end; ++kb) {
                ok = wait_barrier(wctx, full_bar(stage), phase, 300 + stage);
                if (!ok) break;
                ptx::tc_fence_after();
                const uint32_t sa = smem + static_cast<uint32_t>(stage) * j.a_slot;
                const uint32_t sb = smem + off_b + static_cast<uint32_t>(stage) * G::B_BYTES;
                const uint64_t adesc = A_MN ? make_smem_desc(sa, 8192, 1024) : make_smem_desc(sa, 16, 1024);
                const uint64_t bdesc = B_MN ? make_smem_desc(sb, 8192, 1024) : make_smem_desc(sb, 16, 1024);
#pragma unroll
                for (int k = 0; k < kBlockK / kUmmaK; ++k)
                    ptx::umma_bf16<1>(tmem, adesc + static_cast<uint64_t>(k * a_step),
                                      bdesc + static_cast<uint64_t>(k * b_step), idesc,
                                      (kb > kb0 || k > 0) ? 1u : 0u);
                ptx::umma_commit<1>(empty_bar(stage));
                if (++stage == stages) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (ok) ptx::umma_commit<1>(acc_bar);
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..9)
        // Warp w reads TMEM lanes 32 (w % 4) .. +31 (rows of the tile); two warps share a lane quarter
        // and take half of the columns each.
        const int q = warp & 3;
        const int hf = (warp - 2) >> 2;
        const int et = static_cast<int>(threadIdx.x) - 64;
        constexpr int HC = BN / 2;  // columns per warp
        const bool live = q * 32 < rows;
        const uint32_t t_acc = tmem + (static_cast<uint32_t>(q * 32) << 16);
        const int row = q * 32 + lane;
        const bool row_ok = row < rows;
        const long long grow = m0 + row;

        if constexpr (EPI == kEpiF32) {
            // ---------------- fp32 weight gradient
            if (sum_dz) {
                // Column sums of dz from the A tiles (two boxes of 64 k-rows x 64 m, swizzled). A warp
                // owns whole stages, so that the waits and shared-memory latencies of neighbouring
                // k-blocks overlap (all eight warps on one k-block after the other took 1.8 us longer
                // than the products at 512 rows), and so that it sees every phase of its stages'
                // barriers in turn. Lane (cc, kr) adds up eight consecutive m over k rows kr + 2 i.
                const int cc = lane & 15, kr0 = lane >> 4;
                ptx::f2 acc[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[k] = ptx::make_f2(0.0f, 0.0f);
                if (et < kBlockM) ptx::st_shared_f32(line + 4u * et, 0.0f);
                ptx::named_bar_sync(1, kEpiThreads);
                bool ok = true;
                uint32_t phase = 0;
                for (int base = kb0; base < kb_end; base += stages, phase ^= 1u)
                    for (int stage = warp - 2; stage < stages && base + stage < kb_end; stage += kEpiWarps) {
                        if (ok) {
                            bool w = true;
                            if (lane == 0) w = wait_barrier(wctx_epi, full_bar(stage), phase, 600 + stage);
                            ok = __shfl_sync(0xffffffffu, w ? 1 : 0, 0) != 0;
                            __syncwarp();
                        }
                        if (ok) {
                            const uint32_t sa = smem + static_cast<uint32_t>(stage) * j.a_slot +
                                                static_cast<uint32_t>(cc >> 3) * 8192u;
#pragma unroll 8
                            for (int r = 0; r < 32; ++r) {
                                const uint32_t kr = static_cast<uint32_t>(kr0 + 2 * r);
                                uint32_t x[4];
                                ptx::ld_shared_v4(sa + kr * 128u + (((cc & 7u) ^ (kr & 7u)) << 4), x[0], x[1], x[2], x[3]);
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    acc[k] = ptx::add2(acc[k], ptx::make_f2_bits(x[k] << 16, x[k] & 0xffff0000u));
                            }
                        }
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(empty_bar(stage));
                    }
                float sum[8];
#pragma unroll
                for (int k = 0; k < 4; ++k) ptx::split_f2(acc[k], sum[2 * k], sum[2 * k + 1]);
                // lanes l and l ^ 16 hold the same columns
#pragma unroll
                for (int k = 0; k < 8; ++k) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], 16);
                if (lane < 16)
#pragma unroll
                    for (int k = 0; k < 8; ++k) atomicAdd_shared_f32(line + 4u * (cc * 8 + k), sum[k]);
                ptx::named_bar_sync(1, kEpiThreads);
                // this CTA has summed all of K for its 128 columns: nobody else adds to them
                if (ok && et < rows) {
                    float *d = j.dbias + m0 + et;
                    const float v = ptx::ld_shared_f32(line + 4u * et);
                    *d = j.dbias_add ? *d + v : v;
                }
            }
            bool ok = true;
            if (lane == 0) ok = wait_barrier(wctx_epi, acc_bar, 0, 400);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            ptx::tc_fence_after();
            // Every stage has been consumed by the tensor core (and, after the barrier above, by the
            // bias-gradient sums): the boxes are staged there.
            if (live && ok) {
                constexpr int BOXES = HC / 32;
                const uint32_t stg = smem + static_cast<uint32_t>(warp - 2) * BOXES * 4096u;
                const uint32_t sw = static_cast<uint32_t>(lane & 7);
#pragma unroll
                for (int h = 0; h < HC / 16; ++h) {
                    float v[16];
                    tile_ld16(t_acc + static_cast<uint32_t>(hf * HC + h * 16), v);
                    const uint32_t fb = stg + static_cast<uint32_t>(h >> 1) * 4096u + static_cast<uint32_t>(lane) * 128u;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        ptx::st_shared_v4(fb + ((static_cast<uint32_t>((h & 1) * 4 + i) ^ sw) << 4),
                                          __float_as_uint(v[i * 4]), __float_as_uint(v[i * 4 + 1]),
                                          __float_as_uint(v[i * 4 + 2]), __float_as_uint(v[i * 4 + 3]));
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (ptx::elect_one()) {
#pragma unroll
                    for (int b = 0; b < BOXES; ++b) {
                        const int x = n0 + hf * HC + b * 32;
                        if (x < j.N) {
                            if (j.reduce) ptx::tma_reduce_add_2d(t.D, stg + b * 4096u, x, m0 + q * 32);
                            else ptx::tma_store_2d(t.D, stg + b * 4096u, x, m0 + q * 32);
                        }
                    }
                    ptx::bulk_commit_group();
                }
                __syncwarp();
            }
            ptx::bulk_wait_group<0>();
        } else {
            // ---------------- bf16 results
            if (EPI != kEpiMulGeluGrad) {
                for (int i = et; i < BN; i += kEpiThreads) {
                    int col = n0 + i;
                    bool in = col < j.N;
                    if (EPI == kEpiSwiglu) {
                        in = n0 + (i % n_span) < j.swiglu_h;
                        col = (i < n_span ? 0 : j.swiglu_h) + n0 + (i % n_span);
                    }
                    ptx::st_shared_f32(line + 4u * i, (j.bias != nullptr && in) ? __bfloat162float(j.bias[col]) : 0.0f);
                }
                ptx::named_bar_sync(1, kEpiThreads);
            }
            if (cluster == 1) {
                constexpr int PIECES = HC / 8;  // eight columns each
                uint4 e[EPI == kEpiMulGeluGrad ? PIECES : 1];
                if (EPI == kEpiMulGeluGrad) {  // the pre-activation is fetched while the tensor core works
#pragma unroll
                    for (int i = 0; i < PIECES; ++i) {
                        const int col = n0 + hf * HC + i * 8;
                        e[i] = make_uint4(0, 0, 0, 0);
                        if (row_ok && col < j.N)
                            e[i] = ptx::ld_global_v4(j.E + grow * j.e_ld + col);
                    }
                }
                bool ok = true;
                if (lane == 0) ok = wait_barrier(wctx_epi, acc_bar, 0, 400);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                ptx::tc_fence_after();
                if (live && ok) {
                    if constexpr (EPI == kEpiSwiglu) {
                        // this warp: gate columns hf * HC / 2 .. and the matching up columns
                        constexpr int SC = HC / 2;
                        static_assert(SC == 32, "SwiGLU tiles are 64 gate + 64 up columns");
                        using Box = WarpBox<SC>;
                        const uint32_t box = smem + static_cast<uint32_t>(q * 2 + hf) * 3u * Box::BYTES;
                        float gg[16], uu[16];
#pragma unroll
                        for (int i = 0; i < SC / 8; ++i) {
                            const int cl = hf * SC + i * 8;
                            if ((i & 1) == 0) {
                                tile_ld16(t_acc + static_cast<uint32_t>(cl), gg);
                                tile_ld16(t_acc + static_cast<uint32_t>(n_span + cl), uu);
                            }
                            uint32_t wo[4], wg[4], wu[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                float g[2], u[2], o[2];
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const int c = 2 * k + h;
                                    g[h] = gg[(i & 1) * 8 + c] + ptx::ld_shared_f32(line + 4u * (cl + c));
                                    u[h] = uu[(i & 1) * 8 + c] + ptx::ld_shared_f32(line + 4u * (n_span + cl + c));
                                    o[h] = silu_fwd(g[h]) * u[h];
                                }
                                wo[k] = ptx::pack_bf16x2(o[0], o[1]);
                                wg[k] = ptx::pack_bf16x2(g[0], g[1]);
                                wu[k] = ptx::pack_bf16x2(u[0], u[1]);
                            }
                            const uint32_t at = Box::pos(lane, i);
                            ptx::st_shared_v4(box + at, wo[0], wo[1], wo[2], wo[3]);
                            ptx::st_shared_v4(box + Box::BYTES + at, wg[0], wg[1], wg[2], wg[3]);
                            ptx::st_shared_v4(box + 2 * Box::BYTES + at, wu[0], wu[1], wu[2], wu[3]);
                        }
                        const int col = n0 + hf * SC;
                        const long long r0 = m0 + q * 32;
                        Box::flush(box, j.D + r0 * j.d_ld + col, j.d_ld, rows - q * 32, j.swiglu_h - col, lane);
                        Box::flush(box + Box::BYTES, j.E + r0 * j.e_ld + col, j.e_ld, rows - q * 32, j.swiglu_h - col, lane);
                        Box::flush(box + 2 * Box::BYTES, j.E + r0 * j.e_ld + j.swiglu_h + col, j.e_ld, rows - q * 32,
                                   j.swiglu_h - col, lane);
                    } else {
                        // boxes of 64 columns (32, 16 where the warp's share is no multiple of that)
                        constexpr int CW = HC % 64 == 0 ? 64 : HC % 32 == 0 ? 32 : 16;
                        using Box = WarpBox<CW>;
                        constexpr int PLANES = EPI == kEpiGelu ? 2 : 1;
                        const uint32_t box0 = smem + static_cast<uint32_t>((q * 2 + hf) * (HC / CW)) * PLANES * Box::BYTES;
                        const long long r0 = m0 + q * 32;
#pragma unroll
                        for (int b = 0; b < HC / CW; ++b) {
                            const uint32_t box = box0 + static_cast<uint32_t>(b) * PLANES * Box::BYTES;
#pragma unroll
                            for (int h = 0; h < CW / 16; ++h) {
                                float v[16];
                                const int c0 = hf * HC + b * CW + h * 16;  // column in the tile
                                tile_ld16(t_acc + static_cast<uint32_t>(c0), v);
#pragma unroll
                                for (int i = 0; i < 2; ++i) {
                                    uint4 o, z;
                                    tile_math8<EPI>(j, &v[i * 8], line, c0 + i * 8,
                                                    e[EPI == kEpiMulGeluGrad ? (b * CW + h * 16) / 8 + i : 0], o, z);
                                    const uint32_t at = box + Box::pos(lane, h * 2 + i);
                                    ptx::st_shared_v4(at, o.x, o.y, o.z, o.w);
                                    if (EPI == kEpiGelu) ptx::st_shared_v4(at + Box::BYTES, z.x, z.y, z.z, z.w);
                                }
                            }
                            const int col = n0 + hf * HC + b * CW;
                            if (EPI == kEpiGelu)
                                Box::flush(box + Box::BYTES, j.E + r0 * j.e_ld + col, j.e_ld, rows - q * 32, j.N - col, lane);
                            Box::flush(box, j.D + r0 * j.d_ld + col, j.d_ld, rows - q * 32, j.N - col, lane);
                        }
                    }
                }
            } else if constexpr (EPI != kEpiSwiglu && BN <= 128) {
                // K is split: slice d of BN / cluster columns goes to rank d, laid out there as
                // [sender][group of four columns][row], so that a warp's store fills 512 bytes; a
                // group is 129 rows long, so that neighbouring groups of a row lie in other banks. The
                // network between the SMs is the slow part, so the CTA's own slice stays off it: 128
                // columns over two CTAs 8.4 -> 6.9 us (128 rows, 768 -> 768), 13.5 -> 11.7 us (1024
                // rows, 3072 -> 768, a form it no longer takes), 32 columns over two 5.2 -> 4.5 us. Plain stores and one barrier of the
                // cluster; st.async with the bytes counted on the receiver's mbarrier took 0.1 to 0.5 us
                // longer (64 rows, 768 -> 768: 3.80 -> 3.65 us; 519 rows, 3072 -> 1024: 12.0 -> 11.4), bulk
                // copies from shared memory to shared memory another 0.6 us.
                const int sl = BN / cluster;
                auto slice_pos = [&](int sender, int r, int c) {
                    return static_cast<uint32_t>(((sender * (sl / 4) + c / 4) * (kBlockM + 1) + r) * 16);
                };
                bool ok = true;
                if (lane == 0) ok = wait_barrier(wctx_epi, acc_bar, 0, 400);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                ptx::tc_fence_after();
                if (live && ok) {
#pragma unroll
                    for (int h = 0; h < HC / 16; ++h) {
                        float v[16];
                        tile_ld16(t_acc + static_cast<uint32_t>(hf * HC + h * 16), v);
                        if (row_ok)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int cl = hf * HC + h * 16 + i * 4;
                                const int d = cl / sl;
                                const uint32_t at = smem + off_recv + slice_pos(rank, row, cl - d * sl);
                                const uint32_t x0 = __float_as_uint(v[i * 4]), x1 = __float_as_uint(v[i * 4 + 1]),
                                               x2 = __float_as_uint(v[i * 4 + 2]), x3 = __float_as_uint(v[i * 4 + 3]);
                                if (d == rank) ptx::st_shared_v4(at, x0, x1, x2, x3);
                                else ptx::st_cluster_v4(ptx::mapa(at, d), x0, x1, x2, x3);
                            }
                    }
                }
                __syncwarp();
                ptx::cluster_arrive();
                // eight columns of one row per item, neighbouring items along the row
                const int pieces = sl / 8;
                const int items = rows * pieces;
                const int cbase = rank * sl;
                uint4 e0 = make_uint4(0, 0, 0, 0);
                if (EPI == kEpiMulGeluGrad && et < items) {
                    const int col = n0 + cbase + (et % pieces) * 8;
                    if (col < j.N)
                        e0 = ptx::ld_global_v4(j.E + static_cast<long long>(m0 + et / pieces) * j.e_ld + col);
                }
                ptx::cluster_wait();  // every part has arrived
                for (int it = et; ok && it < items; it += kEpiThreads) {
                    const int rw = it / pieces, piece = it % pieces;
                    const int cl = cbase + piece * 8;
                    const int col = n0 + cl;
                    float v[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = 0.0f;
                    for (int s = 0; s < cluster; ++s) {
                        float4 a, b;
                        ptx::ld_shared_f32x4(smem + off_recv + slice_pos(s, rw, piece * 8), a);
                        ptx::ld_shared_f32x4(smem + off_recv + slice_pos(s, rw, piece * 8 + 4), b);
                        v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
                        v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
                    }
                    if (col < j.N) {
                        uint4 e = e0;
                        if (EPI == kEpiMulGeluGrad && it != et)
                            e = ptx::ld_global_v4(j.E + static_cast<long long>(m0 + rw) * j.e_ld + col);
                        uint4 o, z;
                        tile_math8<EPI>(j, v, line, cl, e, o, z);
                        const long long r = static_cast<long long>(m0) + rw;
                        *reinterpret_cast<uint4 *>(j.D + r * j.d_ld + col) = o;
                        if (EPI == kEpiGelu) *reinterpret_cast<uint4 *>(j.E + r * j.e_ld + col) = z;
                    }
                }
            }
        }
    }

    // ---------------------------------------------------------------- common exit
    __syncwarp();
    constexpr bool SPLIT = EPI != kEpiF32 && EPI != kEpiSwiglu && BN <= 128;
    if (SPLIT && cluster > 1 && (warp < 2 || !smem_ok)) ptx::cluster_sync();  // the epilogue's warps have passed it
    ptx::tc_fence_before();
    __syncthreads();
    if (ptx::ld_shared_u32_volatile(abort_addr) != 0) {
        // A wait expired somewhere: give copies and MMAs still in flight time to land. (A peer sends nothing
        // after the cluster's barrier.)
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
        __syncwarp();
    }
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc<1>(tmem, G::TMEM_COLS);
    }
}

// One product (forward, or dinp alone).
template <int BN, bool B_MN, int EPI>
__global__ void __launch_bounds__(kTileThreads, BN >= 128 ? 1 : 2)
tile_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
            const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
            const __grid_constant__ TileParams p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const TileMaps t{&tmA, &tmB, &tmA2, &tmB2, nullptr};
    const int c = static_cast<int>(blockIdx.x);
    tile_body<BN, false, B_MN, EPI>(p.job[0], t, ptx::smem_u32(smem_raw), c / p.cluster, c % p.cluster, p.cluster, p);
}

// Two products that read the same tensor. The CTAs of job 0 form a bf16 result (A by rows, B
// MN-major, adapter term possible), those of job 1 an fp32 one (both operands MN-major, all of its K
// in one CTA, so nothing has to start from zero and nothing is summed in a varying order) and, with
// it, column sums of its A operand:
//   a layer's backward       dinp = dz . W                      dweight (+)= dz^T . inp, dbias
//   an adapter's backward    u = scale dy . B                   dB (+)= dy^T . t
//                            dinp = dy . W + u . A              dA (+)= u^T . inp
template <int BN, bool GELU_GRAD>
__global__ void __launch_bounds__(kTileThreads, BN == 128 && GELU_GRAD ? 1 : 2)  // two where the planner may count on two
tile_pair_kernel(const __grid_constant__ CUtensorMap tmA0,  // boxes of up to 128 rows
                 const __grid_constant__ CUtensorMap tmB0,  // 64 x 64 boxes, as all that follow
                 const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmB2,
                 const __grid_constant__ CUtensorMap tmA1, const __grid_constant__ CUtensorMap tmB1,
                 const __grid_constant__ CUtensorMap tmD1,  // fp32, 32 x 32 boxes
                 const __grid_constant__ TileParams p)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const int c = static_cast<int>(blockIdx.x);
    const int n0 = p.job[0].ctas;
    if (c < n0) {
        const TileMaps t{&tmA0, &tmB0, &tmA2, &tmB2, nullptr};
        tile_body<BN, false, true, GELU_GRAD ? kEpiMulGeluGrad : kEpiStore>(
            p.job[0], t, ptx::smem_u32(smem_raw), c / p.cluster, c % p.cluster, p.cluster, p);
    } else if (c - n0 < p.job[1].ctas) {
        const TileMaps t{&tmA1, &tmB1, nullptr, nullptr, &tmD1};
        tile_body<BN, true, true, kEpiF32>(p.job[1], t, ptx::smem_u32(smem_raw), c - n0, 0, 1, p);
    }
}

}  // namespace nb
