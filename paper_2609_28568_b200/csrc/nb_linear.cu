// Host side of the nb_linear C ABI: argument checks, TMA descriptors, kernel selection, launches.
// Declarations and argument documentation live in include/nb_linear.h.
#include "nb_linear.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <unordered_map>

#include "elementwise.cuh"
#include "gemm_sm100.cuh"
#include "layer_bwd_sm100.cuh"
#include "lora_udb_sm100.cuh"
#include "rows_sm100.cuh"
#include "tile_sm100.cuh"

namespace {

using namespace nb;

constexpr int kMaxDevices = 64;
constexpr unsigned long long kDefaultTimeoutNs = 2000000000ull;  // 2 s per wait

std::atomic<long long> g_launches{0};
const bool g_use_pdl = [] {
    const char *e = getenv("NB_PDL");  // debugging aid: NB_PDL=0 turns dependent launch off
    return !(e && e[0] == '0');
}();
thread_local std::string g_err;
thread_local cudaStream_t g_stream = nullptr;

int fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

#define NB_CUDA(call)                                                                        \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return fail(NB_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_));        \
    } while (0)

// ----------------------------------------------------------------------------- per-device state
struct TmapKey {
    const void *ptr;
    uint64_t rows, cols, ld;
    uint32_t box_cols, box_rows, dtype;
    bool operator==(const TmapKey &o) const
    {
        return ptr == o.ptr && rows == o.rows && cols == o.cols && ld == o.ld && box_cols == o.box_cols &&
               box_rows == o.box_rows && dtype == o.dtype;
    }
};
struct TmapKeyHash {
    size_t operator()(const TmapKey &k) const
    {
        uint64_t h = reinterpret_cast<uint64_t>(k.ptr) * 0x9E3779B97F4A7C15ull;
        h ^= (k.rows + 0x7F4A7C15ull) * 0xBF58476D1CE4E5B9ull;
        h ^= (k.cols + 0x165667B1ull) * 0x94D049BB133111EBull;
        h ^= (k.ld + 0x2545F491ull) * 0xD6E8FEB86659FD93ull;
        h ^= (static_cast<uint64_t>(k.box_cols) << 40) ^ (static_cast<uint64_t>(k.box_rows) << 20) ^
             k.dtype;
        return static_cast<size_t>(h ^ (h >> 29));
    }
};

struct PlanKey {
    int64_t BT, C, OC;
    int pairs;
    bool gelu_grad, fresh;
    bool operator==(const PlanKey &o) const
    {
        return BT == o.BT && C == o.C && OC == o.OC && pairs == o.pairs && gelu_grad == o.gelu_grad && fresh == o.fresh;
    }
};
// The plans of the sizes used last: a model's layers at a few row counts. A program whose row count is new on every call replaces
// the one that was not used for longest, and finds those of its other layers again.
struct PlanCache {
    static constexpr int kSlots = 64;
    PlanKey keys[kSlots];
    uint64_t used[kSlots];  // 0: empty
    LayerBwdParams plans[kSlots];
    uint64_t clock;
};

struct DeviceState {
    bool init = false;
    int num_sms = 0;
    int *status = nullptr;   // 16 ints on the device
    void *workspace = nullptr;
    size_t workspace_bytes = 0;
    std::unordered_map<TmapKey, CUtensorMap, TmapKeyHash> tmaps;
    PlanCache plans{};
};

std::mutex g_mu;
DeviceState g_dev[kMaxDevices];

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

int get_state(DeviceState **out)
{
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(NB_ERR_UNSUPPORTED, "device index %d", dev);
    DeviceState &s = g_dev[dev];
    if (!s.init) {
        cudaDeviceProp prop;
        NB_CUDA(cudaGetDeviceProperties(&prop, dev));
        if (prop.major != 10)
            return fail(NB_ERR_UNSUPPORTED,
                        "device %d is sm_%d%d; this library only runs on sm_100 (B200)", dev,
                        prop.major, prop.minor);
        s.num_sms = prop.multiProcessorCount;
        NB_CUDA(cudaMalloc(reinterpret_cast<void **>(&s.status), 64));
        NB_CUDA(cudaMemset(s.status, 0, 64));
        if (!g_encode) {
            void *fn = nullptr;
            cudaDriverEntryPointQueryResult qres;
            NB_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
            if (qres != cudaDriverEntryPointSuccess || !fn)
                return fail(NB_ERR_CUDA, "cuTensorMapEncodeTiled is not available in this driver");
            g_encode = reinterpret_cast<EncodeTiledFn>(fn);
        }
        s.init = true;
    }
    *out = &s;
    return NB_OK;
}

// Row-major [rows, cols] tensor, tiles of box_rows x box_cols with the 128-byte swizzle.
// dtype: 0 bf16, 1 fp32. The innermost box extent is always 128 bytes (64 bf16 / 32 fp32).
// ld: elements from one row to the next (0: dense, = cols); a column slice of a wider tensor is a
// view with ld > cols, and what lies beyond its cols reads as zero and is never written.
int get_tmap(DeviceState &s, CUtensorMap *out, const void *ptr, uint64_t rows, uint64_t cols,
             uint32_t dtype, uint32_t box_rows, uint64_t ld = 0)
{
    const uint32_t esz = dtype == 0 ? 2u : 4u;
    const uint32_t box_cols = 128u / esz;
    if (ld == 0) ld = cols;
    if (ld < cols || (ld * esz) % 16 != 0)
        return fail(NB_ERR_UNSUPPORTED, "row stride of %llu elements is not a multiple of 16 bytes",
                    static_cast<unsigned long long>(ld));
    TmapKey key{ptr, rows, cols, ld, box_cols, box_rows, dtype};
    auto it = s.tmaps.find(key);
    if (it != s.tmaps.end()) {
        *out = it->second;
        return NB_OK;
    }
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * esz};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    // The encoder does not write every byte of the opaque descriptor: start from zeros, otherwise
    // stack garbage ends up in fields the TMA unit reads.
    alignas(64) CUtensorMap m;
    memset(&m, 0, sizeof(m));
    CUresult r = g_encode(&m, dtype == 0 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                          2, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return fail(NB_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d) for [%llu, %llu] at %p",
                    static_cast<int>(r), static_cast<unsigned long long>(rows),
                    static_cast<unsigned long long>(cols), ptr);
    if (s.tmaps.size() > 8192) s.tmaps.clear();
    s.tmaps.emplace(key, m);
    *out = m;
    return NB_OK;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_dims(int64_t BT, int64_t C, int64_t OC)
{
    if (BT < 0 || C <= 0 || OC <= 0) return fail(NB_ERR_INVALID_ARG, "negative or zero dimension");
    if (BT >= (1ll << 31) || C >= (1ll << 31) || OC >= (1ll << 31) || BT * OC >= (1ll << 40) ||
        BT * C >= (1ll << 40))
        return fail(NB_ERR_UNSUPPORTED, "dimension too large");
    if (C % 8 != 0 || OC % 8 != 0)
        return fail(NB_ERR_UNSUPPORTED, "C (%lld) and OC (%lld) must be multiples of 8",
                    static_cast<long long>(C), static_cast<long long>(OC));
    return NB_OK;
}

// Programmatic dependent launch is used unless it is switched off, or the stream is being captured
// and this launch has more than one dependency (see launch_gemm).
bool dependent_launch_allowed(cudaStream_t stream)
{
    if (!g_use_pdl) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t *deps = nullptr;
    size_t ndeps = 0;
    if (cudaStreamGetCaptureInfo(stream, &cs, nullptr, nullptr, &deps, &ndeps) != cudaSuccess) {
        (void)cudaGetLastError();
        cs = cudaStreamCaptureStatusNone;
    }
    return !(cs == cudaStreamCaptureStatusActive && ndeps != 1);
}

// ----------------------------------------------------------------------------- GEMM launch
struct GemmArgs {
    const void *A;  uint64_t a_rows, a_cols;   // global tensor of the A operand (bf16)
    const void *B;  uint64_t b_rows, b_cols;   // global tensor of the B operand (bf16)
    void *D;        uint64_t d_rows, d_cols;  uint32_t d_dtype;
    const void *E;  uint64_t e_rows, e_cols;   // second bf16 tensor (pre-activation / aux) or null
    int M, N, K;
    const void *bias;
    int swiglu_h;
    int reduce;
    int splits;
    float *dbias;  // wgrad: bias gradient fused into the pass over dz, or null
    bool wait_ext;      // small-problem kernel only: TileJob::wait_ext, TileParams::trigger_late
    bool trigger_late;
    // adapter term D += A2 . B2^T over k2 columns (k2 <= 64), read after the main k range
    const void *A2; uint64_t a2_rows, a2_cols;
    const void *B2; uint64_t b2_rows, b2_cols;
    int k2;
    float alpha = 1.0f;   // D = alpha * acc (+ bias)
    uint64_t a_ld, b_ld, d_ld, a2_ld;  // row strides in elements of A, B, D, A2 when they are column slices (0: dense)
    float2 *stats; // forward with softmax statistics: [M, stats_ld]
    int stats_ld;
    int v_real;
    int debug_stop_kb;                  // nb_debug_gemm_timeout only: see GemmParams; 0 = unset (-1 is passed on)
    unsigned long long debug_timeout_ns;  //   and its shortened wait limit
};

template <class Cfg>
int launch_gemm(DeviceState &s, const GemmArgs &a, cudaStream_t stream)
{
    static bool attr_set[kMaxDevices] = {};
    static int max_clusters[kMaxDevices] = {};
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (!attr_set[dev]) {
        NB_CUDA(cudaFuncSetAttribute(gemm_kernel<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(Cfg::SMEM_BYTES)));
        max_clusters[dev] = s.num_sms / Cfg::CG;
        if (Cfg::CG == 2) {  // how many CTA pairs can be resident at once
            cudaLaunchConfig_t qc = {};
            qc.gridDim = dim3(static_cast<unsigned>(s.num_sms));
            qc.blockDim = dim3(Cfg::THREADS);
            qc.dynamicSmemBytes = Cfg::SMEM_BYTES;
            cudaLaunchAttribute qa[1];
            qa[0].id = cudaLaunchAttributeClusterDimension;
            qa[0].val.clusterDim.x = 2;
            qa[0].val.clusterDim.y = 1;
            qa[0].val.clusterDim.z = 1;
            qc.attrs = qa;
            qc.numAttrs = 1;
            int n = 0;
            NB_CUDA(cudaOccupancyMaxActiveClusters(&n, gemm_kernel<Cfg>, &qc));
            if (n < 1) return fail(NB_ERR_CUDA, "no CTA pair of this kernel fits on the device");
            if (n < max_clusters[dev]) max_clusters[dev] = n;
        }
        attr_set[dev] = true;
    }
    CUtensorMap tA, tB, tD, tE;
    int rc;
    // operands are fetched as 64 x 64 boxes (192-wide tiles: 128 and 96 rows of 64); results (and the aux tile) move as 128-row chunks
    if ((rc = get_tmap(s, &tA, a.A, a.a_rows, a.a_cols, 0, Cfg::A_BOX_ROWS, a.a_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tB, a.B, a.b_rows, a.b_cols, 0, Cfg::B_BOX_ROWS, a.b_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tD, a.D, a.d_rows, a.d_cols, a.d_dtype, Cfg::OUT_BOX_ROWS, a.d_ld)) != NB_OK) return rc;
    if (a.E) {
        if ((rc = get_tmap(s, &tE, a.E, a.e_rows, a.e_cols, 0, Cfg::OUT_BOX_ROWS)) != NB_OK) return rc;
    } else {
        tE = tD;
    }
    CUtensorMap tA2 = tA, tB2 = tB;
    if (a.A2 && a.B2 && a.k2 > 0) {
        if ((rc = get_tmap(s, &tA2, a.A2, a.a2_rows, a.a2_cols, 0, Cfg::A_BOX_ROWS, a.a2_ld)) != NB_OK) return rc;
        if ((rc = get_tmap(s, &tB2, a.B2, a.b2_rows, a.b2_cols, 0, Cfg::B_BOX_ROWS)) != NB_OK) return rc;
    }
    GemmParams p;
    memset(&p, 0, sizeof(p));
    p.M = a.M;
    p.N = a.N;
    p.K = a.K;
    p.tiles_m = (a.M + Cfg::TILE_M - 1) / Cfg::TILE_M;
    const int n_span = (Cfg::EPI == kEpiSwiglu) ? a.swiglu_h : a.N;
    const int n_tile = (Cfg::EPI == kEpiSwiglu) ? 128 : Cfg::BLOCK_N;
    p.tiles_n = (n_span + n_tile - 1) / n_tile;
    p.kblocks = (a.K + kBlockK - 1) / kBlockK;
    int splits = a.splits < 1 ? 1 : a.splits;
    if (splits > p.kblocks) splits = p.kblocks;
    p.kblocks_per_split = (p.kblocks + splits - 1) / splits;
    p.splits = (p.kblocks + p.kblocks_per_split - 1) / p.kblocks_per_split;
    // rasterisation: units walk `group_m` row tiles for each column tile before moving to the next
    // column tile. Many column tiles (the head): a tall group keeps the weight tiles' reuse in L2;
    // few column tiles: a short group keeps the row tiles' (measured on B200, 1-2 % either way)
    p.kblocks_ext = (a.A2 && a.B2 && a.k2 > 0 && p.splits == 1) ? (a.k2 + kBlockK - 1) / kBlockK : 0;
    p.alpha = a.alpha;
    p.group_m = (p.tiles_n >= 64 ? 64 : p.tiles_n <= 4 ? 4 : 16) / Cfg::CG;
    p.swiglu_h = a.swiglu_h;
    p.reduce = a.reduce;
    p.bias = static_cast<const __nv_bfloat16 *>(a.bias);
    p.dbias = a.dbias;
    p.stats = a.stats;
    p.stats_ld = a.stats_ld;
    p.v_real = a.v_real;
    p.status = s.status;
    p.timeout_ns = a.debug_timeout_ns ? a.debug_timeout_ns : kDefaultTimeoutNs;
    p.debug_stop_kb = a.debug_stop_kb > 0 ? a.debug_stop_kb : -1;
    const long long units = 1ll * p.tiles_m * p.tiles_n * p.splits;
    if (units <= 0 || units >= (1ll << 31)) return fail(NB_ERR_UNSUPPORTED, "tile count out of range");
    const int clusters = static_cast<int>(units < max_clusters[dev] ? units : max_clusters[dev]);

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(clusters * Cfg::CG));
    cfg.blockDim = dim3(Cfg::THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = Cfg::CG;
    attrs[0].val.clusterDim.y = 1;
    attrs[0].val.clusterDim.z = 1;
    // programmatic dependent launch: the kernel's set-up overlaps the previous kernel's tail; the
    // kernel itself waits for that kernel before it touches global memory
    attrs[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attrs;
    // While a stream is being captured into a graph, a launch that follows a wait on another
    // stream has more than one dependency; with the programmatic attribute all of them became
    // programmatic edges and the kernel then waited for only one (observed: a consumer started
    // before its cross-stream producer had finished). Such a launch keeps full dependencies.
    cfg.numAttrs = dependent_launch_allowed(stream) ? 2 : 1;
    NB_CUDA(cudaLaunchKernelEx(&cfg, gemm_kernel<Cfg>, tA, tB, tD, tE, tA2, tB2, p));
    ++g_launches;
    return NB_OK;
}

// Kernel configurations: <CTAs per tile, BLOCK_N, stages, staging buffers, A MN-major, B MN-major,
// epilogue>. The pair forms (256-row tiles) are used whenever there is more than one 128-row block;
// the single-CTA forms serve small row counts.
using FwdStore1 = GemmCfg<1, 256, 4, 2, false, false, kEpiStore>;
using FwdGelu1 = GemmCfg<1, 256, 3, 4, false, false, kEpiGelu>;
using FwdSwiglu1 = GemmCfg<1, 256, 3, 3, false, false, kEpiSwiglu>;
using DgradStore1 = GemmCfg<1, 256, 4, 2, false, true, kEpiStore>;
using DgradMulGelu1 = GemmCfg<1, 256, 2, 2, false, true, kEpiMulGeluGrad>;
using WgradF32_1 = GemmCfg<1, 256, 3, 4, true, true, kEpiF32>;
using WgradBf16_1 = GemmCfg<1, 256, 4, 2, true, true, kEpiStore>;
using FwdStore2 = GemmCfg<2, 256, 6, 2, false, false, kEpiStore>;
using FwdStoreStats1 = GemmCfg<1, 256, 4, 2, false, false, kEpiStoreStats>;
using FwdStoreStats2 = GemmCfg<2, 256, 6, 2, false, false, kEpiStoreStats>;
using FwdGelu2 = GemmCfg<2, 256, 5, 4, false, false, kEpiGelu>;
// 192-wide pair tiles, where these make fewer or shorter waves (narrower_tiles)
using FwdStore2N = GemmCfg<2, 192, 6, 2, false, false, kEpiStore>;
using FwdGelu2N = GemmCfg<2, 192, 5, 4, false, false, kEpiGelu>;
using FwdSwiglu2 = GemmCfg<2, 256, 5, 3, false, false, kEpiSwiglu>;
using DgradStore2 = GemmCfg<2, 256, 6, 2, false, true, kEpiStore>;
using DgradMulGelu2 = GemmCfg<2, 256, 4, 2, false, true, kEpiMulGeluGrad>;
using WgradF32_2 = GemmCfg<2, 256, 5, 4, true, true, kEpiF32>;
using WgradF32Bias1 = GemmCfg<1, 256, 3, 4, true, true, kEpiF32, true>;
using WgradF32Bias2 = GemmCfg<2, 256, 5, 4, true, true, kEpiF32, true>;
using WgradBf16_2 = GemmCfg<2, 256, 6, 2, true, true, kEpiStore>;
// Narrow results (N <= 64: the rank-r products of the adapter layer). A 256-wide tile would spend
// 4-16x the tensor-core time on padding; a 64-wide one leaves these products bound by the read of
// their tall operand, so they run one CTA per tile with a deep ring.
using FwdStoreNarrow = GemmCfg<1, 64, 7, 2, false, false, kEpiStore>;
using DgradStoreNarrow = GemmCfg<1, 64, 7, 2, false, true, kEpiStore>;
using WgradF32Narrow = GemmCfg<1, 64, 7, 2, true, true, kEpiF32>;
constexpr int kNarrowN = 64;

// ----------------------------------------------------------------------------- elementwise kernels
// Launches a kernel that begins with chained_start.
template <class... P, class... A>
int launch_chained(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = dependent_launch_allowed(stream) ? 1 : 0;
    NB_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    return NB_OK;
}

// ----------------------------------------------------------------------------- clearing
// Zeroes up to two fp32 arrays in stream order (clear_kernel).
int launch_clear(const DeviceState &s, void *a, int64_t na, void *b, int64_t nb_, cudaStream_t stream)
{
    if (!b) nb_ = 0;
    const long long vec = (na > nb_ ? na : nb_) / 4;
    long long blocks = (vec + 1023) / 1024;  // four stores per thread, up to four blocks per SM
    if (blocks > 4ll * s.num_sms) blocks = 4ll * s.num_sms;
    if (blocks < 1) blocks = 1;
    // not counted in g_launches, as the memsets it replaces were not
    return launch_chained(clear_kernel, dim3(static_cast<unsigned>(blocks)), 256, stream, static_cast<float *>(a),
                          static_cast<long long>(na), static_cast<float *>(b), static_cast<long long>(nb_));
}

// ----------------------------------------------------------------------------- small problems
// Launch configuration: cluster size along x, and dependent launch where it is allowed.
void small_launch_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attrs)[2], int ctas, int threads, int cluster,
                         uint32_t smem_bytes, cudaStream_t stream)
{
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(static_cast<unsigned>(ctas));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    unsigned n = 0;
    if (cluster > 1) {
        attrs[n].id = cudaLaunchAttributeClusterDimension;
        attrs[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attrs[n].val.clusterDim.y = 1;
        attrs[n].val.clusterDim.z = 1;
        ++n;
    }
    if (dependent_launch_allowed(stream)) {
        attrs[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attrs[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = attrs;
    cfg.numAttrs = n;
}

constexpr uint32_t kTileSmemTwo = 113u * 1024u;  // two CTAs on an SM
constexpr uint32_t kTileSmemOne = 220u * 1024u;

// The ring of a job in BN-wide tiles: bytes of an A tile, stages, the CTA's shared memory. `longest`: the most
// k-blocks a CTA works through. two: sized for two CTAs on an SM, where that leaves two stages
// (pair_fits_twice asks whether it does).
struct TileRing {
    uint32_t a_slot;
    int stages;
    uint32_t bytes;
};
template <int BN>
TileRing tile_ring(int M, int epi, bool a_mn, int cluster, int longest, bool two)
{
    using G = TileGeom<BN>;
    TileRing r;
    // a K-major A tile is one box; a single row tile of fewer than 128 rows is fetched (and kept) as
    // just those rows
    r.a_slot = (!a_mn && M < kBlockM ? static_cast<uint32_t>((M + 7) / 8 * 8) : kBlockM) * 128u;
    const uint32_t recv = cluster > 1 ? G::RECV_BYTES : 0u;
    const uint32_t stage = r.a_slot + G::B_BYTES;
    auto fit = [&](uint32_t budget) { return static_cast<int>((budget - recv - G::TAIL_BYTES) / stage); };
    int st = fit(two ? kTileSmemTwo : kTileSmemOne);
    if (st < 2) st = fit(kTileSmemOne);
    if (st > kTileMaxStages) st = kTileMaxStages;
    if (st > longest) st = longest;
    // the result is staged in the drained stages' memory: 4 bytes an element (fp32, or bf16 result and
    // pre-activation) or 2, for the 32-row quarters that hold rows; SwiGLU: three planes of half a tile
    const uint32_t quarters = M < kBlockM ? static_cast<uint32_t>((M + 31) / 32) : 4u;
    const uint32_t elem = epi == kEpiF32 || epi == kEpiGelu ? 4u : epi == kEpiSwiglu ? 3u : 2u;
    const uint32_t staged = (epi == kEpiF32 ? 4u : quarters) * 32u * BN * elem;
    const int min_st = cluster > 1 ? 1 : static_cast<int>((staged + stage - 1) / stage);
    if (st < min_st) st = min_st;
    r.stages = st;
    r.bytes = static_cast<uint32_t>(st) * stage + recv + G::TAIL_BYTES;
    // the tensor core reads 128 rows from every A slot
    const uint32_t reach = static_cast<uint32_t>(st - 1) * r.a_slot + kBlockM * 128u;
    if (r.bytes < reach) r.bytes = reach;
    return r;
}

// Fills a job (and the shared memory it needs) for D[M, N] in BN-wide tiles, K split over `cluster`.
template <int BN>
void fill_tile_job(TileJob &j, uint32_t &smem_bytes, const GemmArgs &a, int epi, bool a_mn, int cluster, bool two)
{
    memset(&j, 0, sizeof(j));
    const bool swiglu = epi == kEpiSwiglu;
    j.M = a.M;
    j.N = a.N;
    j.tiles_m = (a.M + kBlockM - 1) / kBlockM;
    const int span = swiglu ? BN / 2 : BN, n = swiglu ? a.swiglu_h : a.N;
    j.tiles_n = (n + span - 1) / span;
    j.kblocks = (a.K + kBlockK - 1) / kBlockK;
    j.kblocks_ext = (a.A2 && a.B2 && a.k2 > 0) ? (a.k2 + kBlockK - 1) / kBlockK : 0;
    j.ctas = j.tiles_m * j.tiles_n * cluster;
    j.alpha = a.alpha;
    j.bias = static_cast<const __nv_bfloat16 *>(a.bias);
    j.D = static_cast<__nv_bfloat16 *>(a.D);
    j.d_ld = static_cast<long long>(a.d_ld ? a.d_ld : a.d_cols);
    j.E = static_cast<__nv_bfloat16 *>(const_cast<void *>(a.E));
    j.e_ld = static_cast<long long>(a.e_cols);
    j.swiglu_h = a.swiglu_h;
    j.reduce = a.reduce;
    j.wait_ext = a.wait_ext && j.kblocks_ext > 0;
    const TileRing r = tile_ring<BN>(a.M, epi, a_mn, cluster, (j.kblocks + cluster - 1) / cluster + j.kblocks_ext, two);
    j.a_slot = r.a_slot;
    j.stages = r.stages;
    smem_bytes = r.bytes;
}

template <int BN, bool B_MN, int EPI>
int launch_tile(DeviceState &s, const GemmArgs &a, int cluster, cudaStream_t stream)
{
    static bool attr_set[kMaxDevices] = {};
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (!attr_set[dev]) {
        NB_CUDA(cudaFuncSetAttribute(tile_kernel<BN, B_MN, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(kTileSmemOne)));
        attr_set[dev] = true;
    }
    TileParams p;
    memset(&p, 0, sizeof(p));
    uint32_t smem_bytes = 0;
    fill_tile_job<BN>(p.job[0], smem_bytes, a, EPI, false, cluster, false);
    p.cluster = cluster;
    p.trigger_late = a.trigger_late;
    p.status = s.status;
    p.timeout_ns = kDefaultTimeoutNs;
    const uint32_t a_box = p.job[0].a_slot / 128u;
    const uint32_t b_box = B_MN || EPI == kEpiSwiglu ? 64u : static_cast<uint32_t>(BN);
    CUtensorMap tA, tB, tA2, tB2;
    int rc;
    if ((rc = get_tmap(s, &tA, a.A, a.a_rows, a.a_cols, 0, a_box, a.a_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tB, a.B, a.b_rows, a.b_cols, 0, b_box, a.b_ld)) != NB_OK) return rc;
    tA2 = tA;
    tB2 = tB;
    if (p.job[0].kblocks_ext > 0) {
        if ((rc = get_tmap(s, &tA2, a.A2, a.a2_rows, a.a2_cols, 0, a_box, a.a2_ld)) != NB_OK) return rc;
        if ((rc = get_tmap(s, &tB2, a.B2, a.b2_rows, a.b2_cols, 0, b_box)) != NB_OK) return rc;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attrs[2];
    small_launch_config(cfg, attrs, p.job[0].ctas, kTileThreads, cluster, smem_bytes, stream);
    NB_CUDA(cudaLaunchKernelEx(&cfg, tile_kernel<BN, B_MN, EPI>, tA, tB, tA2, tB2, p));
    ++g_launches;
    return NB_OK;
}

// Two products in one launch (tile_pair_kernel): `d` a bf16 result with a B operand that is read
// MN-major (null: none), `w` an fp32 one with both operands MN-major (dbias optional).
template <int BN, bool GELU_GRAD>
int launch_tile_pair(DeviceState &s, const GemmArgs *d, const GemmArgs &w, int accumulate, int cluster, bool two,
                     cudaStream_t stream)
{
    static bool attr_set[kMaxDevices] = {};
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (!attr_set[dev]) {
        NB_CUDA(cudaFuncSetAttribute(tile_pair_kernel<BN, GELU_GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(kTileSmemOne)));
        attr_set[dev] = true;
    }
    TileParams p;
    memset(&p, 0, sizeof(p));
    uint32_t smem_d = 0, smem_w = 0;
    fill_tile_job<BN>(p.job[1], smem_w, w, kEpiF32, true, 1, two);
    p.job[1].reduce = accumulate ? 1 : 0;
    p.job[1].dbias = w.dbias;
    p.job[1].dbias_add = accumulate ? 1 : 0;
    p.cluster = cluster;
    p.trigger_late = w.trigger_late;
    p.status = s.status;
    p.timeout_ns = kDefaultTimeoutNs;
    CUtensorMap tA0, tB0, tA2, tB2, tA1, tB1, tD1;
    int rc;
    if ((rc = get_tmap(s, &tA1, w.A, w.a_rows, w.a_cols, 0, 64, w.a_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tB1, w.B, w.b_rows, w.b_cols, 0, 64, w.b_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tD1, w.D, w.d_rows, w.d_cols, 1, 32)) != NB_OK) return rc;
    tA0 = tA1;  // never read without d, nor the second pair without an adapter term
    tB0 = tB1;
    if (d) {
        fill_tile_job<BN>(p.job[0], smem_d, *d, GELU_GRAD ? kEpiMulGeluGrad : kEpiStore, false, cluster, two);
        const uint32_t a_box = p.job[0].a_slot / 128u;
        if ((rc = get_tmap(s, &tA0, d->A, d->a_rows, d->a_cols, 0, a_box, d->a_ld)) != NB_OK) return rc;
        if ((rc = get_tmap(s, &tB0, d->B, d->b_rows, d->b_cols, 0, 64, d->b_ld)) != NB_OK) return rc;
        tA2 = tA0;
        tB2 = tB0;
        if (p.job[0].kblocks_ext > 0) {
            if ((rc = get_tmap(s, &tA2, d->A2, d->a2_rows, d->a2_cols, 0, a_box, d->a2_ld)) != NB_OK) return rc;
            if ((rc = get_tmap(s, &tB2, d->B2, d->b2_rows, d->b2_cols, 0, 64)) != NB_OK) return rc;
        }
    } else {
        tA2 = tA0;
        tB2 = tB0;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attrs[2];
    int ctas = p.job[0].ctas + p.job[1].ctas;
    ctas = (ctas + cluster - 1) / cluster * cluster;
    small_launch_config(cfg, attrs, ctas, kTileThreads, cluster, smem_d > smem_w ? smem_d : smem_w, stream);
    NB_CUDA(cudaLaunchKernelEx(&cfg, tile_pair_kernel<BN, GELU_GRAD>, tA0, tB0, tA2, tB2, tA1, tB1, tD1, p));
    ++g_launches;
    return NB_OK;
}

// A forward product on at most kRowsMax rows. K is shared among a cluster when it is long (48 CTAs
// of 16 features took 7.9 us for K = 3072, and 2.7 us for K = 768), as far as two CTAs per SM go.
int rows_split(int sms, int groups, int K)
{
    int split = 1;
    while (split < kRowsMaxSplit && K >= 1024 * split && groups * split <= sms) split *= 2;
    return split;
}
// Several CTAs of features per SM: the form with four of them on an SM. Not for the gate and up rows of 9 to 16
// rows: too few registers (1024 -> 16384 12.6 us, with two CTAs 8.6).
bool rows_many(int sms, int M, int span, bool swiglu)
{
    return span > 3 * sms * kRowsFeatures && !(swiglu && M > 8);
}
template <int NT, int EPI, bool MANY>
int launch_rows(DeviceState &s, const GemmArgs &a, cudaStream_t stream)
{
    RowsParams p;
    memset(&p, 0, sizeof(p));
    p.inp = static_cast<const __nv_bfloat16 *>(a.A);
    p.weight = static_cast<const __nv_bfloat16 *>(a.B);
    p.bias = static_cast<const __nv_bfloat16 *>(a.bias);
    p.out = static_cast<__nv_bfloat16 *>(a.D);
    p.pre = static_cast<__nv_bfloat16 *>(const_cast<void *>(a.E));
    p.M = a.M;
    p.K = a.K;
    p.N = a.N;
    p.swiglu_h = a.swiglu_h;
    const int groups = ((EPI == kEpiSwiglu ? a.swiglu_h : a.N) + kRowsFeatures - 1) / kRowsFeatures;
    p.ksplit = rows_split(s.num_sms, groups, a.K);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attrs[2];
    small_launch_config(cfg, attrs, groups * p.ksplit, kRowsThreads, p.ksplit, 0, stream);
    NB_CUDA(cudaLaunchKernelEx(&cfg, rows_kernel<NT, EPI, MANY>, p));
    ++g_launches;
    return NB_OK;
}

template <int EPI>
int launch_rows_auto(DeviceState &s, const GemmArgs &a, cudaStream_t stream)
{
    const bool many = rows_many(s.num_sms, a.M, EPI == kEpiSwiglu ? a.swiglu_h : a.N, EPI == kEpiSwiglu);
    if (a.M <= 8) return many ? launch_rows<1, EPI, true>(s, a, stream) : launch_rows<1, EPI, false>(s, a, stream);
    if constexpr (EPI != kEpiSwiglu)
        if (many) return launch_rows<2, EPI, true>(s, a, stream);
    return launch_rows<2, EPI, false>(s, a, stream);
}

// What the forms of a product take, in microseconds: a fit to chained launches on B200 (1..2048 rows,
// 768..3072 columns), good to about 15 %. They decide between kernels of very different shape, so
// where two are close either will do.
//
// A CTA of the small-problem kernel: launch, set-up and epilogue, then 64-wide k-blocks. A k-block
// costs the MMA issuer about 300 cycles whatever BN is, and more when many SMs load at once.
struct SmallPlan {
    int bn = 0, cluster = 1;  // bn == 0: the persistent kernels
    bool two = false;         // tile_pair_kernel: ring sized for two CTAs on an SM
    double us = 0;
};
constexpr double kLaunchUs = 1.0;

double small_cta_us(int bn, double kblocks, int rows, int ctas, bool two)
{
    const double part = (rows < kBlockM ? rows : kBlockM) / 128.0 * bn / 64.0;
    const double stage_kb = 16.0 + bn / 8.0;
    const double mma = bn > 128 ? 0.00105 * bn : 0.152;  // 2 bn cycles per k-block take over from the issue
    return 1.45 + 0.5 * part + kblocks * ((two ? (bn == 128 ? 0.30 : 0.18) : mma) + 1e-5 * ctas * stage_kb);
}
// Adding up the parts of a cluster that shares K; the network between the SMs slows down where more
// than half of them use it (768 columns from 3072, 128-wide tiles over two: 72 CTAs 10.5 us, 96 11.7).
double small_exchange_us(int bn, int rows, int ctas)
{
    const double part = (rows < kBlockM ? rows : kBlockM) / 128.0 * bn / 64.0;
    return 0.6 + part * (1.2 + (ctas > 74 ? 0.015 * (ctas - 74) : 0.0));
}
// gemm_kernel: waves of 128 (256) x 256 tiles, 512 tensor-core cycles per k-block
double persistent_us(int sms, int M, int N, int kblocks)
{
    const int tm = M > kBlockM ? 2 * kBlockM : kBlockM;
    const long long tiles = 1ll * ((M + tm - 1) / tm) * ((N + 255) / 256);
    const int slots = M > kBlockM ? sms / 2 : sms;
    return 5.3 + 0.27 * kblocks * static_cast<double>((tiles + slots - 1) / slots);
}

// Tile width and K split for one product D[M, N] over `kblocks`. The tiles have to fit the chip in one
// wave; with more of them the persistent kernels, which overlap one tile's epilogue with the next
// one's main loop, are as fast or faster (1024 rows, 768 -> 3072: 192 tiles of 128 columns 11.5 us,
// persistent 9.2 us, 128 tiles of 192 columns 8.0 us; 256 columns never beat the persistent kernel).
// `other` is what the alternative takes; split: 0 any split of K, else that one.
SmallPlan plan_single(int sms, int M, int N, int kblocks, bool allow32, int split, int min_bn, double other)
{
    SmallPlan best;
    best.us = other;
    for (int bn : {32, 64, 128, 192}) {
        if (bn < min_bn || (bn == 32 && !allow32) || (bn > 128 && (min_bn || split > 1))) continue;
        const long long tiles = 1ll * ((M + kBlockM - 1) / kBlockM) * ((N + bn - 1) / bn);
        if (tiles > sms) continue;
        for (int cl = split ? split : 1; cl <= (split ? split : bn > 128 ? 1 : 8); cl *= 2) {
            // a cluster lies within one GPC: not every SM finds a place in clusters of 4 or 8
            if (tiles * cl > sms * (cl >= 8 ? 0.86 : cl >= 4 ? 0.95 : 1.0) || bn / cl < 8 || (cl > 1 && 2 * cl > kblocks)) break;
            const double us = kLaunchUs + small_cta_us(bn, (kblocks + cl - 1) / cl, M, static_cast<int>(tiles * cl), false) +
                              (cl > 1 ? small_exchange_us(bn, M, static_cast<int>(tiles * cl)) : 0.0);
            if (us < best.us) best = SmallPlan{bn, cl, false, us};
        }
    }
    return best;
}

// Whether two CTAs of tile_pair_kernel fit an SM: by the shared memory of both jobs' rings (with K split,
// 128-wide tiles of more than 56 rows do not: the slices received take 66 KB), and by registers (gelu' in 128-wide
// tiles takes 156 a thread; 102 are what two CTAs leave).
template <int BN>
bool pair_fits_twice(int M, int longest, int cluster, int Mw, int kw, bool gelu)
{
    if (BN == 128 && gelu) return false;
    return tile_ring<BN>(Mw, kEpiF32, true, 1, kw, true).bytes <= kTileSmemTwo &&
           (M == 0 || tile_ring<BN>(M, gelu ? kEpiMulGeluGrad : kEpiStore, false, cluster, longest, true).bytes <= kTileSmemTwo);
}

// The same for a bf16 product D[M, N] (M == 0: none) and an fp32 product [Mw, Nw] over kw k-blocks in
// one launch; `other` is what the alternative takes, `split` as above; gelu: the bf16 product times gelu'.
SmallPlan plan_pair(int sms, int M, int N, int kblocks, int split, int Mw, int Nw, int kw, bool dbias, bool gelu, double other, bool only64)
{
    SmallPlan best;
    best.us = other;
    for (int bn = 64; bn <= (only64 ? 64 : 128); bn *= 2) {
        const long long nd = M > 0 ? 1ll * ((M + kBlockM - 1) / kBlockM) * ((N + bn - 1) / bn) : 0;
        const long long nw = 1ll * ((Mw + kBlockM - 1) / kBlockM) * ((Nw + bn - 1) / bn);
        if (nd + nw > 16ll * sms) continue;
        for (int cl = nd && split ? split : 1; cl <= (!nd ? 1 : split ? split : 8); cl *= 2) {
            if (bn / cl < 8 || (cl > 1 && 2 * cl > kblocks)) break;
            for (int two = 0; two <= 1; ++two) {
                const int longest = (kblocks + cl - 1) / cl;
                const double slots = sms * (two ? 2.0 : 1.0);
                const double n = static_cast<double>(nd * cl + nw);
                // job 0's clusters come first and have to find their places; job 1's tiles fill up behind them
                if (cl >= 8 ? n > 0.86 * slots : cl > 1 && nd * cl > 0.95 * slots) continue;
                const int crowd = static_cast<int>(n < slots ? n : slots);
                const double td = nd ? small_cta_us(bn, longest, M, crowd, two != 0) +
                                           (cl > 1 ? small_exchange_us(bn, M, static_cast<int>(nd * cl)) : 0.0) : 0.0;
                // the bias gradient's warps own a stage each: the fewer stages, the longer they hold them
                const double tw = small_cta_us(bn, kw, Mw, crowd, two != 0) + (dbias ? kw * (two ? 0.18 : bn == 128 ? 0.115 : 0.05) : 0.0);
                double us = td > tw ? td : tw;
                if (n > slots) {
                    const double line = (nd * cl * td + nw * tw) / slots + tw;
                    if (line > us) us = line;
                }
                // three stages each: from eight k-blocks of dweight on, short rings that wait for each other (1003
                // rows, 776 -> 1416: 18 us against 12.6); up to four, one CTA's stores run under the other's
                // loads (130 rows, 4096 -> 1024: 9.5 us against 12.8; 256 rows, 4096 x 4096: 36.8 against 42.8)
                if (two && bn == 128 && kw > 4) us *= 1.0 + 0.1 * (kw < 8 ? kw - 4 : 4);
                us += kLaunchUs;
                if (us < best.us) best = SmallPlan{bn, cl, two != 0, us};
            }
        }
    }
    // Where two do not fit, the form runs one per SM with the whole ring, and the estimate of two is a second one of
    // that: where its tiles take more than a wave it lies nearer than the first one, which adds a whole last tile. 700
    // drawn problems, the chosen form against the fastest: 2.6 % with it on average, 2.5 % without, but without it eleven
    // small ones lose 3 to 11 % (100 rows, 1536 -> 1536 with gelu': 64-wide tiles 9.4 us, 128-wide ones 8.4; 519 rows,
    // 3072 -> 768: layer_bwd_kernel 15.8, 128-wide tiles 13.2).
    if (best.two) {
        const int longest = (kblocks + best.cluster - 1) / best.cluster;
        best.two = best.bn == 64 ? pair_fits_twice<64>(M, longest, best.cluster, Mw, kw, gelu)
                                 : pair_fits_twice<128>(M, longest, best.cluster, Mw, kw, gelu);
    }
    return best;
}

// The split of K for dinp. It fixes the order of the sums, so it depends on the problem alone and not
// on which other gradients are asked for in the same call; above 256 rows, where the weight gradient's
// tiles join dinp's in the persistent kernel, there is none. At most four CTAs share K: eight find no place
// in a GPC among the weight gradient's tiles (128 rows, 768 -> 3072, both products: 9.3 us with eight, 7.4
// with four; 64 rows, 768 -> 2304: 7.7 and 5.9; dinp alone 6.3 and 6.6). Where those tiles fill the chip
// twice over, the clusters take no more than 32 places (256 rows, 4096 x 4096: 53 us with two CTAs
// sharing K, 37 without; 200 rows, 1024 -> 6144: 20.9 with four, 18.7 with two, 21.4 without).
int dinp_split(int sms, int M, int N, int kblocks)
{
    if (M > 2 * kBlockM) return 1;
    const SmallPlan pl = plan_single(sms, M, N, kblocks, false, 0, 0, 1e9);
    int split = pl.bn ? (pl.cluster < 4 ? pl.cluster : 4) : 1;
    const int cols = (N + kBlockM - 1) / kBlockM;
    if ((kblocks + 1) / 2 * cols > 2 * sms)
        while (split > 1 && (M + kBlockM - 1) / kBlockM * cols * split > 32) split /= 2;
    return split;
}

template <bool B_MN, int EPI>
int launch_tile_plan(DeviceState &s, const GemmArgs &a, const SmallPlan &pl, cudaStream_t stream)
{
    if constexpr (!B_MN)
        if (pl.bn == 32) return launch_tile<32, B_MN, EPI>(s, a, pl.cluster, stream);
    if (pl.bn == 64) return launch_tile<64, B_MN, EPI>(s, a, pl.cluster, stream);
    if (pl.bn == 192) return launch_tile<192, B_MN, EPI>(s, a, 1, stream);
    return launch_tile<128, B_MN, EPI>(s, a, pl.cluster, stream);
}

int launch_tile_pair_plan(DeviceState &s, const GemmArgs *d, const GemmArgs &w, bool gelu_grad, int accumulate,
                          const SmallPlan &pl, cudaStream_t stream)
{
    if (gelu_grad)
        return pl.bn == 64 ? launch_tile_pair<64, true>(s, d, w, accumulate, pl.cluster, pl.two, stream)
                           : launch_tile_pair<128, true>(s, d, w, accumulate, pl.cluster, pl.two, stream);
    return pl.bn == 64 ? launch_tile_pair<64, false>(s, d, w, accumulate, pl.cluster, pl.two, stream)
                       : launch_tile_pair<128, false>(s, d, w, accumulate, pl.cluster, pl.two, stream);
}

int kblocks_of(int64_t K) { return static_cast<int>((K + kBlockK - 1) / kBlockK); }

bool use_pairs(int M)
{
    static const int force = [] {
        const char *e = getenv("NB_CTA_GROUP");  // debugging aid: 1 or 2 forces one form
        return e ? atoi(e) : 0;
    }();
    if (force == 1) return false;
    if (force == 2) return true;
    return M > kBlockM;
}

template <class C1, class C2>
int launch_gemm_auto(DeviceState &s, const GemmArgs &a, cudaStream_t stream)
{
    return use_pairs(a.M) ? launch_gemm<C2>(s, a, stream) : launch_gemm<C1>(s, a, stream);
}

// Split-K factor for wgrad: the one whose waves of (tiles x splits) units over `slots` resident
// tiles take the least time, counting a fixed cost per unit (epilogue and pipeline ramp, about six
// k-blocks' worth). Every (m, n, k-range) is covered exactly once whatever the choice.
int choose_splits(int tiles, int kblocks, int slots)
{
    const int kUnitOverhead = 6;
    int best = 1;
    long long best_cost = -1;
    const int max_splits = kblocks / 4 > 1 ? kblocks / 4 : 1;
    for (int sp = 1; sp <= max_splits && sp <= 128; ++sp) {
        const int kps = (kblocks + sp - 1) / sp;
        const int eff = (kblocks + kps - 1) / kps;  // splits that are not empty
        const long long units = 1ll * tiles * eff;
        const long long waves = (units + slots - 1) / slots;
        const long long cost = waves * (kps + kUnitOverhead);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = eff;
        }
    }
    return best;
}

int ensure_workspace(DeviceState &s, size_t bytes, cudaStream_t stream = nullptr)
{
    if (s.workspace_bytes >= bytes) return NB_OK;
    // growing synchronises the device and frees memory that kernels of a graph under
    // construction may refer to: refuse instead of failing inside the runtime
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (stream != nullptr && cudaStreamIsCapturing(stream, &cs) != cudaSuccess) (void)cudaGetLastError();
    if (cs != cudaStreamCaptureStatusNone)
        return fail(NB_ERR_UNSUPPORTED,
                    "the workspace would have to grow to %zu bytes during stream capture; call "
                    "nb_workspace_reserve before capturing", bytes);
    if (s.workspace) {
        NB_CUDA(cudaDeviceSynchronize());
        NB_CUDA(cudaFree(s.workspace));
        s.workspace = nullptr;
        s.workspace_bytes = 0;
    }
    const size_t want = (bytes + (1u << 20) - 1) & ~static_cast<size_t>((1u << 20) - 1);
    NB_CUDA(cudaMalloc(&s.workspace, want));
    s.workspace_bytes = want;
    return NB_OK;
}

int launch_dbias(DeviceState &s, float *dbias, const void *dz, int64_t BT, int64_t OC, int accumulate,
                 cudaStream_t stream)
{
    if (!accumulate) {
        const int crc = launch_clear(s, dbias, OC, nullptr, 0, stream);
        if (crc != NB_OK) return crc;
    }
    if (BT == 0) return NB_OK;
    const int col_blocks = static_cast<int>((OC + kDbiasCols - 1) / kDbiasCols);
    // about three blocks per SM: with six (or one) the same kernel was 15-25 % slower on the stack's
    // shapes (measured: 16.6 us against 19.2 us for 16384 x 2304)
    long long want_row_blocks = (3ll * s.num_sms + col_blocks - 1) / col_blocks;
    long long rows_per_block = (BT + want_row_blocks - 1) / want_row_blocks;
    rows_per_block = ((rows_per_block + 127) / 128) * 128;  // a block sweeps 128 rows per iteration
    if (rows_per_block < 128) rows_per_block = 128;
    const long long row_blocks = (BT + rows_per_block - 1) / rows_per_block;
    if (row_blocks > 65535) return fail(NB_ERR_UNSUPPORTED, "BT too large for the dbias grid");
    dim3 grid(col_blocks, static_cast<unsigned>(row_blocks));
    const int rc = launch_chained(dbias_kernel, grid, kDbiasThreads, stream, dbias, static_cast<const __nv_bfloat16 *>(dz), BT,
                                  static_cast<int>(OC), static_cast<int>(rows_per_block));
    if (rc != NB_OK) return rc;
    ++g_launches;
    return NB_OK;
}

int elementwise_grid(const DeviceState &s, long long nvec)
{
    long long blocks = (nvec + 255) / 256;
    const long long cap = 16ll * s.num_sms;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

// dweight[M_, N_] (+)= dz^T . inp over BT rows, fp32, with the split-K factor chosen per shape;
// dz [BT, M_], inp [BT, N_]. dbias (or null) is summed inside the same kernel.
int run_wgrad_f32(DeviceState &s, const void *dz, const void *inp, void *dweight, float *dbias,
                  int64_t BT, int64_t M_, int64_t N_, int accumulate, cudaStream_t stream,
                  uint64_t inp_ld = 0)
{
    GemmArgs a{};
    a.A = dz; a.a_rows = BT; a.a_cols = M_;
    a.B = inp; a.b_rows = BT; a.b_cols = N_; a.b_ld = inp_ld;
    a.D = dweight; a.d_rows = M_; a.d_cols = N_; a.d_dtype = 1;
    a.M = static_cast<int>(M_); a.N = static_cast<int>(N_); a.K = static_cast<int>(BT);
    const bool narrow = dbias == nullptr && a.N <= kNarrowN;
    const bool pairs = !narrow && use_pairs(a.M);
    const int tile_m = pairs ? 2 * kBlockM : kBlockM;
    const int tile_n = narrow ? kNarrowN : 256;
    const int tiles = ((a.M + tile_m - 1) / tile_m) * ((a.N + tile_n - 1) / tile_n);
    const int kblocks = (a.K + kBlockK - 1) / kBlockK;
    const int slots = s.num_sms / (pairs ? 2 : 1);  // tiles resident at once
    const int splits = choose_splits(tiles, kblocks, slots);
    a.splits = splits;
    a.reduce = (accumulate || splits > 1) ? 1 : 0;
    const bool clear_w = !accumulate && splits > 1, clear_b = !accumulate && dbias != nullptr;
    int rc;
    if (clear_w && (rc = launch_clear(s, dweight, M_ * N_, clear_b ? dbias : nullptr, M_, stream)) != NB_OK) return rc;
    if (clear_b && !clear_w && (rc = launch_clear(s, dbias, M_, nullptr, 0, stream)) != NB_OK) return rc;
    if (dbias) {  // the bias gradient rides along: reducer warps sum dz while it is in shared memory
        a.dbias = dbias;
        return launch_gemm_auto<WgradF32Bias1, WgradF32Bias2>(s, a, stream);
    }
    if (narrow) return launch_gemm<WgradF32Narrow>(s, a, stream);
    return launch_gemm_auto<WgradF32_1, WgradF32_2>(s, a, stream);
}

// u = bf16(scale * dy . B) and dB (+)= dy^T . t of one adapted projection from one pass over dy
// (lora_udb_sm100.cuh). u and t may be column slices of wider tensors (row strides u_ld, t_ld).
// x and dlora_a both non-NULL: the A gradient dlora_a [r, C] (+)= u^T . x rides on the same launch
// (only with the whole of u in one call: u_ld == r).
int launch_lora_udb(DeviceState &s, const void *dy, const void *lora_b, const void *t, uint64_t t_ld, void *dlora_b,
                    void *u, uint64_t u_ld, float scale, int64_t BT, int64_t OC, int64_t r, int accumulate,
                    cudaStream_t stream, const void *x = nullptr, void *dlora_a = nullptr, int64_t C = 0)
{
    static bool attr_set[kMaxDevices] = {};
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (!attr_set[dev]) {
        NB_CUDA(cudaFuncSetAttribute(lora_udb_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(kUdbSmemBytes)));
        attr_set[dev] = true;
    }
    const bool want_da = x != nullptr && dlora_a != nullptr;
    CUtensorMap tDy, tB, tT, tDb, tX, tDa;
    int rc;
    if ((rc = get_tmap(s, &tDy, dy, BT, OC, 0, 64)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tB, lora_b, OC, r, 0, 64)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tT, t, BT, r, 0, 64, t_ld)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tDb, dlora_b, OC, r, 1, 32)) != NB_OK) return rc;
    if (want_da) {
        if ((rc = get_tmap(s, &tX, x, BT, C, 0, 64)) != NB_OK) return rc;
        if ((rc = get_tmap(s, &tDa, dlora_a, r, C, 1, 32)) != NB_OK) return rc;
    } else {
        tX = tDy;   // never dereferenced
        tDa = tDb;
    }
    // every panel reduce-adds its share, so a fresh gradient starts from zero
    if (!accumulate && (rc = launch_clear(s, dlora_b, OC * r, want_da ? dlora_a : nullptr, r * C, stream)) != NB_OK) return rc;
    UdbParams p;
    memset(&p, 0, sizeof(p));
    p.BT = static_cast<int>(BT);
    p.OC = static_cast<int>(OC);
    p.r = static_cast<int>(r);
    p.panels = static_cast<int>((BT + 127) / 128);
    p.tiles = static_cast<int>((OC + 127) / 128);
    p.want_db = 1;
    p.want_da = want_da ? 1 : 0;
    p.C = static_cast<int>(C);
    p.xtiles = want_da ? static_cast<int>((C + 127) / 128) : 0;
    p.alpha = scale;
    p.u = static_cast<__nv_bfloat16 *>(u);
    p.u_ld = static_cast<int>(u_ld);
    p.after_clear = accumulate ? 0 : 1;
    p.status = s.status;
    p.timeout_ns = kDefaultTimeoutNs;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(p.panels < s.num_sms ? p.panels : s.num_sms));
    cfg.blockDim = dim3(kUdbThreads);
    cfg.dynamicSmemBytes = kUdbSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = dependent_launch_allowed(stream) ? 1 : 0;
    NB_CUDA(cudaLaunchKernelEx(&cfg, lora_udb_kernel, tDy, tB, tT, tDb, tX, tDa, p));
    ++g_launches;
    return NB_OK;
}

// ----------------------------------------------------------------------------- one launch per layer backward
int env_int(const char *name, int dflt)
{
    const char *e = getenv(name);
    return (e && *e) ? atoi(e) : dflt;
}

constexpr double kNarrowD = 0.6;  // in the level share of the work; backward_us takes 0.7 for the chain of one such tile
bool layer_bwd_narrow(int d_tiles, int d_kblocks, int w_tiles, int w_kblocks, int P)
{
    return d_tiles * 4 <= P && d_kblocks >= 36 && d_kblocks >= 12 + 2 * d_tiles &&
           static_cast<double>(d_kblocks) * P > 1.0 * d_tiles * d_kblocks + 1.0 * w_tiles * w_kblocks;
}

// What a unit costs beside its k-blocks, in k-blocks of 0.33 us, from the times at which the pairs of twelve launches ended
// (2021 and 4096 rows): a W unit's fp32 boxes, 128 KB an SM, take up to 2.3 us of the main loop they leave under, a D unit's
// bf16 boxes 0.4, and gelu' some arithmetic on top. (5 to 7 for a W unit measure alike; 3, as before, leaves the pairs with
// several of them 3 to 5 us behind the others.)
constexpr int kCostD = 1, kCostDGelu = 2, kCostW = 5;
constexpr int kMaxChunk = 64;  // k-blocks
constexpr int kLbTries = 4;    // forms that are cut; 0.4 us each
constexpr int kCostClear = 8;  // the launch that clears a fresh dweight, 2.5 to 3 us on the chain
constexpr int kMinPiece = 2;  // k-blocks of a W unit that are worth a cut

// The W units that are left after the whole rounds, as one line of k-blocks: `full` of them in units of kbc, the rest in
// units of last.
struct LbLine {
    long long total, full;
    int kbc, last;
};
struct LbCut {
    double most = 0.0, sum = 0.0, end = 0.0;  // cost of the dearest pair, of all of them, of the last one
};
// Cuts the line into a range per pair (begin: P + 1 borders) such that no pair's cost (cD for the first d_tail of them, a range,
// kCostW for each unit that it touches) exceeds `limit`; a range ends with a unit or at least kMinPiece k-blocks from either end of
// one (whole: with a unit), and the last pair takes what is left. Units that fit whole are taken at once.
LbCut cut_line(const LbLine &l, int P, int d_tail, double cD, double limit, bool whole, int *begin)
{
    LbCut c;
    long long x = 0, left = l.full > 0 ? l.kbc : l.last;  // of the unit that x is in
    for (int q = 0; q < P; ++q) {
        begin[q] = static_cast<int>(x);
        double cost = q < d_tail ? cD : 0.0;
        const long long most = q == P - 1 ? 1ll << 40 : static_cast<long long>(limit - cost);
        long long spent = 0;
        while (x < l.total) {
            const long long end = x < l.full ? l.full : l.total;
            const int unit = x < l.full ? l.kbc : l.last;
            const long long room = most - spent - kCostW;
            if (room < left) {
                const long long take = room < left - kMinPiece ? room : left - kMinPiece;
                if (!whole && take >= kMinPiece) {
                    x += take;
                    left -= take;
                    spent += kCostW + take;
                }
                break;
            }
            long long n = 1;
            if (left == unit) {
                n = (most - spent) / (unit + kCostW);
                if (n > (end - x) / unit) n = (end - x) / unit;
            }
            x += n * left;
            spent += n * (kCostW + left);
            left = x < l.full ? l.kbc : l.last;
        }
        cost += static_cast<double>(spent);
        if (cost > c.most) c.most = cost;
        c.sum += cost;
        c.end = cost;
    }
    begin[P] = static_cast<int>(l.total);
    return c;
}

// A schedule of the W units for the geometry that p holds, found in one pass: about two of them a pair, none shorter than 32
// k-blocks, and ranges of the line that each level the cost of the pairs still to be served (k-blocks and 3 a unit, 8 for a D unit with
// gelu'), ending at a multiple of four k-blocks of a unit or at its end. W rounds are taken back until the pairs with a tail D
// tile have a range as well. It says which sizes have a schedule (more rounds than the order mask holds: none).
int level_layer_bwd(LayerBwdParams &p, bool gelu_grad)
{
    constexpr double eW = 3.0;
    const int P = p.num_pairs;
    const double cD = p.d_kblocks * (p.d_w == 128 ? kNarrowD : 1.0) + (gelu_grad ? 8 : 3);
    int chunks = (2 * P + p.w_tiles - 1) / p.w_tiles;
    const int max_chunks = p.w_kblocks / 32 > 1 ? p.w_kblocks / 32 : 1;
    if (chunks > max_chunks) chunks = max_chunks;
    p.w_kbc = (p.w_kblocks + chunks - 1) / chunks;
    chunks = (p.w_kblocks + p.w_kbc - 1) / p.w_kbc;
    const long long w_units = 1ll * chunks * p.w_tiles;
    if (w_units >= (1ll << 24)) return fail(NB_ERR_UNSUPPORTED, "too many work units");
    p.w_units = static_cast<int>(w_units);
    p.w_last_len = p.w_kblocks - (chunks - 1) * p.w_kbc;
    const int even_units = p.w_last_len == p.w_kbc ? p.w_units : p.w_units - p.w_tiles;
    const long long ragged = 1ll * (p.w_units - even_units) * p.w_last_len;
    long long full = 0;
    for (p.w_rounds = even_units / P;; --p.w_rounds) {
        full = 1ll * (even_units - p.w_rounds * P) * p.w_kbc;
        const double mean = static_cast<double>(full + ragged) / P;
        if (p.w_rounds == 0 || (p.d_tail == 0 ? full + ragged == 0 || mean >= 8.0 : mean + cD * p.d_tail / P - cD >= 8.0)) break;
    }
    const long long total = full + ragged;
    if (total >= (1ll << 30)) return fail(NB_ERR_UNSUPPORTED, "weight-gradient tail too long");
    if (p.d_rounds + p.w_rounds > kLbMaxRounds) return fail(NB_ERR_UNSUPPORTED, "more than %d rounds", kLbMaxRounds);
    p.w_tail_full = static_cast<int>(full);
    long long x = 0, units = p.w_units - 1ll * p.w_rounds * P;  // still on the line, the one that x is in among them
    long long left = full > 0 ? p.w_kbc : p.w_last_len;         // of that one
    for (int q = 0; q < P; ++q) {
        p.w_tail_begin[q] = static_cast<int>(x);
        const double line_cost = static_cast<double>(total - x) + eW * static_cast<double>(units + P - q - 1);
        double rem = (line_cost + cD * (p.d_tail > q ? p.d_tail - q : 0)) / (P - q) - (q < p.d_tail ? cD : 0.0);
        while (x < total && rem >= eW + 4) {
            const int unit = x < full ? p.w_kbc : p.w_last_len;
            if (rem - eW < static_cast<double>(left)) {
                const long long take = static_cast<long long>(rem - eW) / 4 * 4;
                x += take;
                left -= take;
                break;
            }
            long long n = 1;  // units that end here: this one's rest, or whole ones as many as fit
            if (left == unit && unit >= 4) {
                n = static_cast<long long>(rem / (eW + unit));
                const long long have = ((x < full ? full : total) - x) / unit;
                if (n > have) n = have;
            }
            x += n * left;
            units -= n;
            rem -= static_cast<double>(n) * (eW + static_cast<double>(left));
            left = x < full ? p.w_kbc : p.w_last_len;
        }
    }
    for (int q = P; q <= kMaxPairs; ++q) p.w_tail_begin[q] = static_cast<int>(total);
    return NB_OK;
}

// What the error of a schedule's weight gradient goes with: the squares of the lengths of its sums (products of one sign, whose
// running sum grows with the length) and their cubes (products of either sign, where it grows with the root of it), each as
// often as the tile has elements of dweight.
struct LbSums {
    double squares = 0.0, cubes = 0.0;
    int longest = 0;
    void add(int len, double elements)
    {
        squares += elements * len * len;
        cubes += elements * len * len * len;
        if (len > longest) longest = len;
    }
    // (with room for tiles that are cut differently: alike in both sums, errors measured up to 1.2 of each other)
    bool no_worse_than(const LbSums &o) const
    {
        return squares <= 0.85 * o.squares && cubes <= 0.75 * o.cubes && longest <= o.longest;
    }
};
LbSums sums_of(const LayerBwdParams &p, int w_chain)
{
    LbSums s;
    // elements of the tiles of the units before j, in order
    auto elements_to = [&](unsigned j) {
        const unsigned t = j % p.w_tiles, m = t / p.w_tiles_n, n = t % p.w_tiles_n;
        const int rows = p.OC - 256 * static_cast<int>(m) < 256 ? p.OC - 256 * static_cast<int>(m) : 256;
        return static_cast<double>(j / p.w_tiles) * p.OC * p.C + 256.0 * m * p.C + 256.0 * rows * n;  // (n is not the last column's end)
    };
    unsigned j = 0;  // the unit that the line is in, after the rounds' units
    double before = 0.0;
    auto piece = [&](int len, unsigned units, bool ends) {
        const LbUnit u{1, 0, 0, 0, len};
        const int part = chain_len(u, w_chain);
        const double after = elements_to(j + units), elements = after - before;
        if (ends) {
            before = after;
            j += units;
        }
        s.add(part, elements * (len / part));
        if (len % part) s.add(len % part, elements);
    };
    if (p.w_rounds) piece(p.w_kbc, static_cast<unsigned>(p.w_rounds) * p.num_pairs, true);
    int left = p.w_tail_full > 0 ? p.w_kbc : p.w_last_len;  // of the unit
    for (int q = 0, x = 0; q < p.num_pairs; ++q) {
        while (x < p.w_tail_begin[q + 1]) {
            const int unit = x < p.w_tail_full ? p.w_kbc : p.w_last_len;
            int end = p.w_tail_begin[q + 1];
            if (x < p.w_tail_full && end > p.w_tail_full) end = p.w_tail_full;
            const int len = left < end - x ? left : end - x;
            const int n = left == unit && end - x > unit ? (end - x) / unit : 1;
            piece(len, n, len == left);
            x += n * len;
            left = len < left ? left - len : x < p.w_tail_full ? p.w_kbc : p.w_last_len;
        }
    }
    return s;
}

// The schedule of layer_bwd_kernel for P CTA pairs (layer_bwd_sm100.cuh describes the unit list). Costs are counted in
// k-blocks of tensor-core time (kCostD, kCostW above); every pair should end up with the same cost.
//  1. Whole rounds (one unit per pair) are dealt first; W rounds are spread evenly among D rounds.
//  2. The last D round is partial: pairs [0, d_tail) take one more tile. The W units left over are laid out as one line of
//     k-blocks and cut into P ranges at the lowest limit on a pair's cost at which cut_line finds a place for all of it.
//  3. K = BT of the weight gradient is cut into chunks, as many as give two W units per pair or fewer, of 16 to kMaxChunk k-blocks
//     where that leaves a choice. For each number of chunks and each number of W rounds that leaves the pairs with a tail
//     D tile about level, the cost of a pair is estimated; the kLbTries cheapest are cut and the one with the cheapest dearest pair
//     is taken.
//  4. Units that are longer than the one-pass schedule's sums are summed in parts (w_chain).
// Against the one-pass schedule (level_layer_bwd; chains of single launches, below the power cap, accumulating, us): 4096 rows,
// 768 -> 768 16.4 -> 14.4, 768 -> 2304 27.0 -> 26.1, 768 -> 3072 33.3 -> 31.4, 1024 -> 6144 78.9 -> 74.9; 8192 rows, 768 -> 3072
// 62.8 -> 60.2; 16384 rows, 768 -> 768 36.6 -> 36.1, 768 -> 2304 91.2 -> 89.8 (no difference in a step at the cap). Chunks of up to
// 256 k-blocks cost 16384 rows, 768 -> 3072 4 % (the pairs drift apart).
// fresh: dweight starts from nothing. Where every W unit is a tile's whole K it is stored and the clearing launch saved (2021 rows,
// 768 -> 2304 19.5 -> 17.7 us, 768 -> 3072 22.3 -> 19.9; 1100 rows, 1024 -> 4096 26.0 -> 23.5), which is worth kCostClear.
// narrow (as it is launched): D tiles are 128 columns wide (layer_bwd_narrow; not with gelu') where the 256-wide ones are
// at most a quarter of the pairs, K is long, and a single one takes longer than a pair's share of all the work: 1500 rows,
// 768 -> 3072, 18 tiles of 48 k-blocks, 18.9 -> 16.4 us; 1024 rows, 1024 -> 6144, 32.5 -> 24.4 us. With
// more tiles the operand traffic of halved ones costs more than the shorter chain gives (2021 rows,
// 768 -> 2304, 24 tiles: 16.0 -> 19.4 us). A 128-wide k-block is counted as 0.6 of a 256-wide one.
// Returns NB_ERR_UNSUPPORTED when the shape needs more rounds than the order mask holds (level_layer_bwd).
int plan_layer_bwd(LayerBwdParams &p, int64_t BT, int64_t C, int64_t OC, int P, bool gelu_grad, bool narrow, bool fresh)
{
    memset(&p, 0, sizeof(p));
    if (P < 1 || P > kMaxPairs) return fail(NB_ERR_UNSUPPORTED, "CTA pair count %d out of range", P);
    p.BT = static_cast<int>(BT);
    p.C = static_cast<int>(C);
    p.OC = static_cast<int>(OC);
    p.num_pairs = P;
    p.d_tiles_m = static_cast<int>((BT + 255) / 256);
    p.d_tiles_n = static_cast<int>((C + 255) / 256);
    p.d_kblocks = static_cast<int>((OC + kBlockK - 1) / kBlockK);
    p.w_tiles_n = p.d_tiles_n;
    p.d_w = 256;
    p.w_tiles_m = static_cast<int>((OC + 255) / 256);
    p.w_tiles = p.w_tiles_m * p.w_tiles_n;
    p.w_kblocks = static_cast<int>((BT + kBlockK - 1) / kBlockK);
    if (narrow && !gelu_grad && layer_bwd_narrow(p.d_tiles_m * p.d_tiles_n, p.d_kblocks, p.w_tiles, p.w_kblocks, P)) {
        p.d_w = 128;
        p.d_tiles_n = static_cast<int>((C + 127) / 128);
    }
    if (1ll * p.d_tiles_m * p.d_tiles_n >= (1 << 24)) return fail(NB_ERR_UNSUPPORTED, "too many work units");
    p.d_tiles = p.d_tiles_m * p.d_tiles_n;
    p.d_group_m = (p.d_tiles_n >= 64 ? 64 : p.d_tiles_n <= 4 ? 4 : 16) / 2;
    p.d_rounds = p.d_tiles / P;
    p.d_tail = p.d_tiles % P;
    const double cD = p.d_kblocks * (p.d_w == 128 ? kNarrowD : 1.0) + (gelu_grad ? kCostDGelu : kCostD);
    // stands where the search below has nothing, as for a head whose tail D tiles leave room for more rounds than there are
    const int rc = level_layer_bwd(p, gelu_grad);
    if (rc != NB_OK) return rc;
    const LbSums level = sums_of(p, p.w_kblocks);

    struct Form {
        LbLine line;
        long long units;  // on the line
        int chunks, rounds;
        double estimate;  // of what it costs, in the terms of `price`, less the clearing if it may be saved
    } forms[kLbTries];
    int n_forms = 0;
    int max_chunks = (2 * P + p.w_tiles - 1) / p.w_tiles;
    if (max_chunks > p.w_kblocks / 16) max_chunks = p.w_kblocks / 16;
    if (max_chunks < 1) max_chunks = 1;
    // The dearest pair counts and, where the chip is at its power limit, what all of them do. (A judgement, not a fit: with 0.25 or
    // 1 in the place of 0.5, 3 to 5 % of 3000 drawn sizes get another plan.)
    auto price = [&](double most, double sum, int rounds, int kbc) { return most + 0.5 * sum / P + 1.5 * rounds * (kbc + kCostW); };
    for (int want = 1; want <= max_chunks; ++want) {
        const int kbc = (p.w_kblocks + want - 1) / want;
        const int chunks = (p.w_kblocks + kbc - 1) / kbc;
        // the same length again, or one that is too long (the shortest is always tried: it may be both)
        if (want < max_chunks && (chunks != want || kbc > kMaxChunk)) continue;
        const long long w_units = 1ll * chunks * p.w_tiles;
        if (w_units >= (1ll << 24)) break;
        // the units of the last chunk may be shorter than the others: they all stay on the line, where lengths are counted exactly
        const int last = p.w_kblocks - (chunks - 1) * kbc;
        const long long even = last == kbc ? w_units : w_units - p.w_tiles;
        const double mean = (1.0 * p.w_kblocks * p.w_tiles + 1.0 * kCostW * (w_units + P) + cD * p.d_tail) / P;
        long long hi = even / P;
        const long long below = static_cast<long long>((mean - cD) / (kbc + kCostW)) + 1;
        if (p.d_tail && below < hi) hi = below;
        if (hi > kLbMaxRounds - p.d_rounds) hi = kLbMaxRounds - p.d_rounds;
        if (hi < 0) hi = 0;
        for (long long aW = hi; aW >= 0 && aW >= hi - 2; --aW) {
            Form f;
            f.units = w_units - aW * P;
            f.line = {(even - aW * P) * kbc + (w_units - even) * last, (even - aW * P) * kbc, kbc, last};
            f.chunks = chunks;
            f.rounds = static_cast<int>(aW);
            if (f.line.total >= (1ll << 30)) break;
            const double pieces = static_cast<double>(f.units > P - p.d_tail ? f.units : P - p.d_tail);
            const double level = (static_cast<double>(f.line.total) + kCostW * pieces + cD * p.d_tail) / P;
            f.estimate = price(p.d_tail && cD > level ? cD : level, level * P, f.rounds, kbc) - (fresh && chunks == 1 ? kCostClear : 0);
            int at = n_forms < kLbTries ? n_forms++ : kLbTries;
            for (; at > 0 && forms[at - 1].estimate > f.estimate; --at)
                if (at < kLbTries) forms[at] = forms[at - 1];
            if (at < kLbTries) forms[at] = f;
        }
    }
    double best = -1.0;
    const Form *best_form = nullptr;
    // cuts, keeps what is cheaper; the cost of the last pair where that has more than its share, else 0
    auto take = [&](const Form &f, double limit, bool whole) {
        int begin[kMaxPairs + 1];
        const LbCut c = cut_line(f.line, P, p.d_tail, cD, limit, whole, begin);
        if (c.end >= c.most && c.end > limit + 1.0) return c.end;
        const double cost = price(c.most, c.sum, f.rounds, f.line.kbc) - (whole ? kCostClear : 0);
        if (best < 0.0 || cost < best) {
            best = cost;
            best_form = &f;
            for (int q = 0; q <= kMaxPairs; ++q) p.w_tail_begin[q] = begin[q < P ? q : P];
        }
        return 0.0;
    };
    for (int i = 0; i < n_forms; ++i) {
        const Form &f = forms[i];
        if (best >= 0.0 && f.estimate >= best) break;
        // the lowest limit: what is too much for the last pair is spread over all of them
        const double pieces = static_cast<double>(f.units > P - p.d_tail ? f.units : P - p.d_tail);
        double limit = (static_cast<double>(f.line.total) + kCostW * pieces + cD * p.d_tail) / P;
        for (double end; (end = take(f, limit, false)) > 0.0;) limit += (end - limit) / P > 0.5 ? (end - limit) / P : 0.5;
        // where the tail D tiles are the longest chain whatever the others do, a higher limit leaves more units whole
        if (p.d_tail && cD > limit)
            for (double at = limit + (cD - limit) / 3; at < cD; at += (cD - limit) / 3) (void)take(f, at, false);
        // a fresh dweight of whole tiles is not cleared: the lowest limit at which every unit has a place
        if (fresh && f.chunks == 1) {
            const double unit = f.line.kbc + kCostW;
            auto held = [&](double at) {
                return static_cast<double>(p.d_tail) * (at > cD ? floor((at - cD) / unit) : 0.0) +
                       static_cast<double>(P - p.d_tail) * floor(at / unit);
            };
            double with_d = cD + unit, without = unit, at = without < with_d || !p.d_tail ? without : with_d;
            while (held(at) < static_cast<double>(f.units)) {
                if (at >= without) without += unit;
                if (at >= with_d) with_d += unit;
                at = without < with_d || !p.d_tail ? without : with_d;
            }
            (void)take(f, at, true);
        }
    }
    if (best_form) {
        const Form &f = *best_form;
        p.w_kbc = f.line.kbc;
        p.w_units = f.chunks * p.w_tiles;
        p.w_rounds = f.rounds;
        p.w_last_len = f.line.last;
        p.w_tail_full = static_cast<int>(f.line.full);
    }
    // as few parts as leave dweight no less exact than the one-pass schedule
    p.w_chain = sums_of(p, p.w_kblocks).longest;
    for (int parts = 1, longest = p.w_chain; best_form; ++parts) {
        p.w_chain = (longest + parts - 1) / parts;
        if (p.w_chain <= 1 || sums_of(p, p.w_chain).no_worse_than(level)) break;
    }
    const int rounds = p.d_rounds + p.w_rounds;
    for (int r = 0; r < rounds; ++r)
        if (1ll * (r + 1) * p.w_rounds / rounds > 1ll * r * p.w_rounds / rounds) p.round_is_w |= 1ull << r;
    p.w_whole = p.w_kbc == p.w_kblocks;
    for (int q = 0; q < P; ++q) p.w_whole &= p.w_tail_begin[q] % p.w_kbc == 0;
    return NB_OK;
}

// The plan of a launch. Finding one takes 5 to 20 us, so those of the sizes used last are kept (they hold sizes only).
int cached_layer_bwd_plan(DeviceState &s, LayerBwdParams &p, int64_t BT, int64_t C, int64_t OC, int P, bool gelu_grad, bool fresh)
{
    // fresh and added-to gradients differ in their plans only where a tile's whole K may be one unit
    const int64_t tiles = ((OC + 255) / 256) * ((C + 255) / 256);
    const PlanKey key{BT, C, OC, P, gelu_grad, fresh && (BT <= kMaxChunk * kBlockK || tiles >= 2 * P)};
    PlanCache &c = s.plans;
    int at = 0;
    for (int i = 0; i < PlanCache::kSlots; ++i) {
        if (c.used[i] && c.keys[i] == key) {
            c.used[i] = ++c.clock;
            p = c.plans[i];
            return NB_OK;
        }
        if (c.used[i] < c.used[at]) at = i;
    }
    const int rc = plan_layer_bwd(p, BT, C, OC, P, gelu_grad, true, key.fresh);
    if (rc != NB_OK) return rc;
    c.keys[at] = key;
    c.used[at] = ++c.clock;
    c.plans[at] = p;
    return NB_OK;
}

// Whether the launch will add to a fresh dweight, which then has to be cleared before it: not where it stores whole tiles, and not
// where there is no such launch (the products by themselves start a fresh dweight their own way). (It decides for half the SMs as
// pairs; where the launch finds room for fewer this may be wrong, and the gradient is cleared once too often or by a launch of its own.)
bool layer_bwd_adds(DeviceState &s, int64_t BT, int64_t C, int64_t OC, bool gelu_grad)
{
    LayerBwdParams p;
    const int P = s.num_sms / 2 < kMaxPairs ? s.num_sms / 2 : kMaxPairs;
    return cached_layer_bwd_plan(s, p, BT, C, OC, P, gelu_grad, true) == NB_OK && !p.w_whole;
}

using LayerBwdPlain = LbCfg<false, false>;
using LayerBwdBias = LbCfg<false, true>;
using LayerBwdGelu = LbCfg<true, false>;
using LayerBwdGeluBias = LbCfg<true, true>;

template <class Cfg>
int launch_layer_bwd(DeviceState &s, const void *dz, const void *weight, const void *inp, void *dinp,
                     const void *inp_pre, void *dweight, float *dbias, int64_t BT, int64_t C, int64_t OC,
                     int accumulate, bool cleared, cudaStream_t stream)
{
    static bool attr_set[kMaxDevices] = {};
    static int max_pairs[kMaxDevices] = {};
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (!attr_set[dev]) {
        NB_CUDA(cudaFuncSetAttribute(layer_bwd_kernel<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(Cfg::SMEM_BYTES)));
        cudaLaunchConfig_t qc = {};
        qc.gridDim = dim3(static_cast<unsigned>(s.num_sms));
        qc.blockDim = dim3(kLbThreads);
        qc.dynamicSmemBytes = Cfg::SMEM_BYTES;
        cudaLaunchAttribute qa[1];
        qa[0].id = cudaLaunchAttributeClusterDimension;
        qa[0].val.clusterDim.x = 2;
        qa[0].val.clusterDim.y = 1;
        qa[0].val.clusterDim.z = 1;
        qc.attrs = qa;
        qc.numAttrs = 1;
        int n = 0;
        NB_CUDA(cudaOccupancyMaxActiveClusters(&n, layer_bwd_kernel<Cfg>, &qc));
        if (n < 1) return fail(NB_ERR_CUDA, "no CTA pair of the layer-backward kernel fits on the device");
        max_pairs[dev] = n < s.num_sms / 2 ? n : s.num_sms / 2;
        if (max_pairs[dev] > kMaxPairs) max_pairs[dev] = kMaxPairs;
        attr_set[dev] = true;
    }
    LayerBwdParams p;
    int rc = cached_layer_bwd_plan(s, p, BT, C, OC, max_pairs[dev], Cfg::GELU_GRAD, !accumulate);
    if (rc != NB_OK) return rc;
    p.dbias = Cfg::DBIAS ? dbias : nullptr;
    p.status = s.status;
    p.timeout_ns = kDefaultTimeoutNs;
    CUtensorMap tDz, tW, tInp, tDinp, tPre, tDw;
    if ((rc = get_tmap(s, &tDz, dz, BT, OC, 0, 64)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tW, weight, OC, C, 0, 64)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tInp, inp, BT, C, 0, 64)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tDinp, dinp, BT, C, 0, 32)) != NB_OK) return rc;
    if ((rc = get_tmap(s, &tDw, dweight, OC, C, 1, 32)) != NB_OK) return rc;
    tPre = tDinp;
    if (Cfg::GELU_GRAD && (rc = get_tmap(s, &tPre, inp_pre, BT, C, 0, 32)) != NB_OK) return rc;
    // partial sums of W units are reduce-added, so a fresh gradient starts from zero unless all of them are whole
    p.store_w = !accumulate && p.w_whole;
    p.after_clear = !accumulate && !p.store_w && !cleared;
    if (p.after_clear && (rc = launch_clear(s, dweight, OC * C, Cfg::DBIAS ? dbias : nullptr, OC, stream)) != NB_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(2 * p.num_pairs));
    cfg.blockDim = dim3(kLbThreads);
    cfg.dynamicSmemBytes = Cfg::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeClusterDimension;
    attrs[0].val.clusterDim.x = 2;
    attrs[0].val.clusterDim.y = 1;
    attrs[0].val.clusterDim.z = 1;
    attrs[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = dependent_launch_allowed(stream) ? 2 : 1;
    NB_CUDA(cudaLaunchKernelEx(&cfg, layer_bwd_kernel<Cfg>, tDz, tW, tInp, tDinp, tPre, tDw, p));
    ++g_launches;
    return NB_OK;
}

// dinp, fp32 dweight and (optionally) dbias of one layer from its dz in one launch. Returns
// NB_ERR_UNSUPPORTED (and launches nothing) for shapes the schedule does not cover; the caller
// then issues the products one by one.
int run_layer_bwd(DeviceState &s, const void *dz, const void *weight, const void *inp, void *dinp,
                  const void *inp_pre, void *dweight, float *dbias, int64_t BT, int64_t C, int64_t OC,
                  int accumulate, bool cleared, cudaStream_t stream)
{
    if (inp_pre) {
        if (dbias) return launch_layer_bwd<LayerBwdGeluBias>(s, dz, weight, inp, dinp, inp_pre, dweight, dbias, BT, C, OC, accumulate, cleared, stream);
        return launch_layer_bwd<LayerBwdGelu>(s, dz, weight, inp, dinp, inp_pre, dweight, dbias, BT, C, OC, accumulate, cleared, stream);
    }
    if (dbias) return launch_layer_bwd<LayerBwdBias>(s, dz, weight, inp, dinp, inp_pre, dweight, dbias, BT, C, OC, accumulate, cleared, stream);
    return launch_layer_bwd<LayerBwdPlain>(s, dz, weight, inp, dinp, inp_pre, dweight, dbias, BT, C, OC, accumulate, cleared, stream);
}

// Whether a forward product in CTA pairs runs in 192-column tiles: where it takes several waves of the pairs
// and as many with these as with 256-column ones, each wave is shorter (2021 rows, 768 -> 3072 with GELU,
// two waves: 17.4 -> 15.0 us; 8192 rows, 3072 -> 768: 35.3 -> 32.0 us; 4600 rows, 768 -> 2304, three
// waves: 18.0 -> 16.1 us; no upper limit on the waves). One more wave costs more than that (4096 rows, 768 -> 2304: 14.9 -> 15.7 us),
// and in a single wave the SMs' ports to L2 take back what the tensor cores save (4096 rows, 3072 -> 768:
// 18.6 us either way; 73 operand bytes per clock and SM against 64).
bool narrower_tiles(int sms, int M, int N)
{
    if (!use_pairs(M)) return false;
    auto waves = [&](int bn) {
        const long long tiles = 1ll * ((M + 2 * kBlockM - 1) / (2 * kBlockM)) * ((N + bn - 1) / bn);
        return (tiles + sms / 2 - 1) / (sms / 2);
    };
    return waves(256) > 1 && waves(192) == waves(256);
}

// Which kernel forms a product, and in which form.
struct Route {
    int kernel = NB_ROUTE_GEMM;
    SmallPlan pl;  // the tile kernels
};

// A forward product with its activation: on a few rows the row kernel (9 to 16 rows only up to 8 CTAs
// per SM: 16 rows, 768 -> 50304 takes 19.5 us there and 17.3 us in gemm_kernel), then the smaller of the
// tile and the persistent kernel's estimates.
Route route_forward(int sms, int M, int N, int K, int act, bool adapter)
{
    if (!adapter && (M <= 8 || (M <= kRowsMax && N <= 8 * sms * kRowsFeatures))) return {NB_ROUTE_ROWS, {}};
    const int kb = kblocks_of(K) + (adapter ? 1 : 0);
    const double other = persistent_us(sms, M, N, kb);
    // SwiGLU: 64 gate and 64 up columns per tile, so N counts both halves of the weight
    const SmallPlan pl = act == NB_ACT_SWIGLU ? plan_single(sms, M, N, kb, false, 1, 128, other)
                                              : plan_single(sms, M, N, kb, true, 0, 0, other);
    if (pl.bn) return {NB_ROUTE_TILE, pl};
    return {act != NB_ACT_SWIGLU && narrower_tiles(sms, M, N) ? NB_ROUTE_GEMM_192 : NB_ROUTE_GEMM, pl};
}

int run_forward(DeviceState &s, const GemmArgs &a, int act, cudaStream_t stream)
{
    const Route r = route_forward(s.num_sms, a.M, a.N, a.K, act, a.A2 != nullptr);
    if (r.kernel == NB_ROUTE_ROWS) {
        if (act == NB_ACT_NONE) return launch_rows_auto<kEpiStore>(s, a, stream);
        if (act == NB_ACT_GELU) return launch_rows_auto<kEpiGelu>(s, a, stream);
        return launch_rows_auto<kEpiSwiglu>(s, a, stream);
    }
    if (r.kernel == NB_ROUTE_TILE) {
        if (act == NB_ACT_SWIGLU) return launch_tile<128, false, kEpiSwiglu>(s, a, 1, stream);
        return act == NB_ACT_GELU ? launch_tile_plan<false, kEpiGelu>(s, a, r.pl, stream)
                                  : launch_tile_plan<false, kEpiStore>(s, a, r.pl, stream);
    }
    if (r.kernel == NB_ROUTE_GEMM_192)
        return act == NB_ACT_GELU ? launch_gemm<FwdGelu2N>(s, a, stream) : launch_gemm<FwdStore2N>(s, a, stream);
    if (act == NB_ACT_NONE) return launch_gemm_auto<FwdStore1, FwdStore2>(s, a, stream);
    if (act == NB_ACT_GELU) return launch_gemm_auto<FwdGelu1, FwdGelu2>(s, a, stream);
    return launch_gemm_auto<FwdSwiglu1, FwdSwiglu2>(s, a, stream);
}

// A layer's backward without the small-problem kernel: layer_bwd_kernel for both products, else a
// launch per product. An fp32 result that starts from zero costs the clearing besides. (sms / 2: the CTA pairs that
// the launch's occupancy query finds on B200.) The launch has become cheaper than this says where it stores a fresh dweight and
// where its ranges are level: from zero, 256 rows, 2048 -> 3072 takes 13.3 us with it and 17.8 in tiles, 768 rows, 3072 -> 768
// 11.1 and 12.7 (with gelu' 12.4 and 15.6), and these still go to the tiles; 1003 rows, 776 -> 1416 13.6 and 12.6.
double backward_us(int sms, int M, int BT, int N, int Mw, int kd, int kw, bool accumulate, bool apart, bool gelu)
{
    const int slots = sms / 2;
    const double d_tiles = static_cast<double>((M + 255) / 256) * ((N + 255) / 256);
    const double w_tiles = static_cast<double>((Mw + 255) / 256) * ((N + 255) / 256);
    // the fp32 result is cleared (unless it is added to) and reduce-added into
    const double clear = (accumulate ? 0.0 : 2.8) + 1e-6 * Mw * N;
    if (M > 0 && BT > kBlockM && !apart) {
        const bool narrow = !gelu && layer_bwd_narrow(static_cast<int>(d_tiles), kd, static_cast<int>(w_tiles), kw, slots);
        const double chain = narrow ? 0.7 * kd : kd;
        const double level = ((narrow ? 2.0 : 1.0) * d_tiles * (chain + 3) + w_tiles * (kw + 3)) / slots;
        return 6.0 + clear + 0.27 * (chain > level ? chain : level);
    }
    const double waves = w_tiles / slots;
    const double w_us = 5.0 + (waves < 1.0 ? 1.0 : waves) * (0.27 * (waves < 1.0 ? kw * waves : kw) + 0.8);
    return w_us + clear + (M > 0 ? persistent_us(sms, M, N, kd) : 0.0);
}

// D = A . B with B read MN-major (dinp and its like), plain or times gelu'(E).
Route route_dgrad(int sms, int M, int N, int kb)
{
    const int split = dinp_split(sms, M, N, kb);
    const SmallPlan pl = plan_single(sms, M, N, kb, false, split, 0, split > 1 ? 1e9 : persistent_us(sms, M, N, kb));
    return {pl.bn ? NB_ROUTE_TILE : NB_ROUTE_GEMM, pl};
}

int run_dgrad(DeviceState &s, const GemmArgs &a, cudaStream_t stream)
{
    const Route r = route_dgrad(s.num_sms, a.M, a.N, kblocks_of(a.K) + (a.A2 ? 1 : 0));
    if (a.E)
        return r.pl.bn ? launch_tile_plan<true, kEpiMulGeluGrad>(s, a, r.pl, stream)
                       : launch_gemm_auto<DgradMulGelu1, DgradMulGelu2>(s, a, stream);
    return r.pl.bn ? launch_tile_plan<true, kEpiStore>(s, a, r.pl, stream) : launch_gemm_auto<DgradStore1, DgradStore2>(s, a, stream);
}

// A layer's backward with an fp32 dweight: both products (dinp: with dinp) in tiles of one launch, both in the
// persistent launch, or each by itself (NB_ROUTE_GEMM; dinp then by route_dgrad).
Route route_backward(int sms, bool dinp, bool dbias, bool gelu, bool accumulate, int BT, int C, int OC)
{
    static const bool merge_allowed = env_int("NB_MERGED_BWD", 1) != 0;
    const int kd = kblocks_of(OC), kw = kblocks_of(BT);
    const int split = dinp ? dinp_split(sms, BT, C, kd) : 1;
    const SmallPlan pl = plan_pair(sms, dinp ? BT : 0, C, kd, split, OC, C, kw, dbias, gelu,
                                   backward_us(sms, dinp ? BT : 0, BT, C, OC, kd, kw, accumulate, split > 1, gelu), false);
    if (pl.bn) return {NB_ROUTE_TILE_PAIR, pl};
    return {merge_allowed && dinp && split == 1 && use_pairs(BT) ? NB_ROUTE_LAYER_BWD : NB_ROUTE_GEMM, pl};
}

// The rank-r products on 128 x 64 tiles, a CTA each (gemm_kernel's narrow forms).
double narrow_us(int sms, int tiles, int kblocks)
{
    return 4.3 + 0.2 * kblocks * static_cast<double>((tiles + sms - 1) / sms);
}

SmallPlan plan_lora_down(int sms, int M, int r, int kb)
{
    return plan_single(sms, M, r, kb, r <= 32, 0, 0, narrow_us(sms, (M + kBlockM - 1) / kBlockM, kb));
}

// u[:, r] by itself
SmallPlan plan_lora_u(int sms, int M, int r, int kb)
{
    return plan_single(sms, M, r, kb, false, 0, 0, narrow_us(sms, (M + kBlockM - 1) / kBlockM, kb));
}

// t[:, r] = scale * inp . A^T. late (or null): whether the next launch may start before this one is done.
int run_lora_down(DeviceState &s, void *t, const void *inp, const void *lora_a, float scale, int64_t BT, int64_t C,
                  int64_t r, cudaStream_t stream, bool *late = nullptr)
{
    GemmArgs a{};
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = lora_a; a.b_rows = r; a.b_cols = C;
    a.D = t; a.d_rows = BT; a.d_cols = r; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(r); a.K = static_cast<int>(C);
    a.splits = 1;
    a.alpha = scale;
    const SmallPlan pl = plan_lora_down(s.num_sms, a.M, a.N, kblocks_of(C));
    if (late) *late = a.trigger_late = pl.bn != 0;
    return pl.bn ? launch_tile_plan<false, kEpiStore>(s, a, pl, stream) : launch_gemm<FwdStoreNarrow>(s, a, stream);
}

struct LoraBwd {
    void *dinp, *dlora_a, *dlora_b, *u;
    const void *dout, *inp, *weight, *lora_a, *lora_b, *t;
    uint64_t u_ld, t_ld;  // row strides of u and t where they are column slices of stacks, else 0
    float scale;
    int64_t BT, C, OC, r;
    int accumulate;
};

// Backward of one adapted projection. Three ways, by estimate:
//   lora_udb_kernel (u, dB and dA from one pass over dout and inp, a CTA per 128 rows) and the dinp
//   product: the one to use when there are about as many 128-row panels as SMs;
//   two tile_pair_kernel launches (u and dB, then dinp and dA), which spread a short batch over the
//   chip: 519 rows are five panels, and five CTAs took 22 us;
//   the first of those and the other two products by themselves.
struct LoraRoute {
    SmallPlan ub, xa, a1;  // u with dB (bn == 0: lora_udb_kernel); dinp with dA, or (xa.bn == 0) dA alone
};
LoraRoute route_lora_backward(int sms, int BT, int C, int OC, int r, bool want_x, bool want_a, bool accumulate)
{
    const int kt = kblocks_of(BT), ko = kblocks_of(OC);
    const int panels = (BT + kBlockM - 1) / kBlockM;
    const int split = dinp_split(sms, BT, C, ko + 1);
    const double x_us = want_x ? plan_single(sms, BT, C, ko + 1, false, split, 0, persistent_us(sms, BT, C, ko + 1)).us : 0.0;
    const double clear = accumulate ? 0.0 : 2.8;
    const int udb_tiles = (OC + 127) / 128 + (want_a ? (C + 127) / 128 : 0);
    const double udb = 6.0 + clear + x_us + udb_tiles * static_cast<double>((panels + sms - 1) / sms) *
                       (0.37 + 0.25 * (panels < sms ? panels : sms) / sms);  // reading dout takes over towards one panel per SM
    const double far = 1e9;
    LoraRoute l;
    l.ub = plan_pair(sms, BT, r, ko, 0, OC, r, kt, false, false, far, true);
    if (want_x && want_a) l.xa = plan_pair(sms, BT, C, ko + 1, split, r, C, kt, false, false, far, false);
    if (want_a) l.a1 = plan_pair(sms, 0, 0, 0, 1, r, C, kt, false, false, far, false);
    const double apart = l.ub.us + x_us + l.a1.us, paired = l.xa.bn ? l.ub.us + l.xa.us : far;
    if (!l.ub.bn || (apart >= udb && paired >= udb)) return {};
    if (paired > apart) l.xa = {};
    return l;
}

int run_lora_backward(DeviceState &s, const LoraBwd &l, cudaStream_t stream)
{
    const int sms = s.num_sms, BT = static_cast<int>(l.BT), C = static_cast<int>(l.C), OC = static_cast<int>(l.OC), r = static_cast<int>(l.r);
    int rc;
    GemmArgs u{};  // u = scale * dout . B   (B [OC, r] read as an MN-major operand)
    u.A = l.dout; u.a_rows = BT; u.a_cols = OC;
    u.B = l.lora_b; u.b_rows = OC; u.b_cols = r;
    u.D = l.u; u.d_rows = BT; u.d_cols = r; u.d_ld = l.u_ld;
    u.M = BT; u.N = r; u.K = OC;
    u.splits = 1;
    u.alpha = l.scale;
    GemmArgs dB{};  // dB [OC, r] (+)= dout^T . t      (t already carries the scale)
    dB.A = l.dout; dB.a_rows = BT; dB.a_cols = OC;
    dB.B = l.t; dB.b_rows = BT; dB.b_cols = r; dB.b_ld = l.t_ld;
    dB.D = l.dlora_b; dB.d_rows = OC; dB.d_cols = r; dB.d_dtype = 1;
    dB.M = OC; dB.N = r; dB.K = BT;
    GemmArgs dx{};  // dinp = dout . W + u . A: r extra rows of K
    dx.A = l.dout; dx.a_rows = BT; dx.a_cols = OC;
    dx.B = l.weight; dx.b_rows = OC; dx.b_cols = C;
    dx.D = l.dinp; dx.d_rows = BT; dx.d_cols = C;
    dx.M = BT; dx.N = C; dx.K = OC;
    dx.splits = 1;
    dx.A2 = l.u; dx.a2_rows = BT; dx.a2_cols = r; dx.a2_ld = l.u_ld;
    dx.B2 = l.lora_a; dx.b2_rows = r; dx.b2_cols = C;
    dx.k2 = r;
    GemmArgs dA{};  // dA [r, C] (+)= u^T . inp        (u already carries the scale)
    dA.A = l.u; dA.a_rows = BT; dA.a_cols = r; dA.a_ld = l.u_ld;
    dA.B = l.inp; dA.b_rows = BT; dA.b_cols = C;
    dA.D = l.dlora_a; dA.d_rows = r; dA.d_cols = C; dA.d_dtype = 1;
    dA.M = r; dA.N = C; dA.K = BT;

    const bool want_x = l.dinp != nullptr, want_a = l.dlora_a != nullptr;
    if (l.dlora_b) {
        const LoraRoute w = route_lora_backward(sms, BT, C, OC, r, want_x, want_a, l.accumulate != 0);
        if (w.ub.bn) {
            dB.trigger_late = dx.wait_ext = want_x;
            if ((rc = launch_tile_pair_plan(s, &u, dB, false, l.accumulate, w.ub, stream)) != NB_OK) return rc;
            if (w.xa.bn) return launch_tile_pair_plan(s, &dx, dA, false, l.accumulate, w.xa, stream);
            if (want_x && (rc = run_dgrad(s, dx, stream)) != NB_OK) return rc;
            return want_a ? launch_tile_pair_plan(s, nullptr, dA, false, l.accumulate, w.a1, stream) : NB_OK;
        }
        if ((rc = launch_lora_udb(s, l.dout, l.lora_b, l.t, l.t_ld, l.dlora_b, l.u, l.u_ld ? l.u_ld : static_cast<uint64_t>(r),
                                  l.scale, BT, OC, r, l.accumulate, stream, want_a ? l.inp : nullptr, l.dlora_a, C)) != NB_OK)
            return rc;
        return want_x ? run_dgrad(s, dx, stream) : NB_OK;
    }
    const SmallPlan up = plan_lora_u(sms, BT, r, kblocks_of(OC));
    rc = up.bn ? launch_tile_plan<true, kEpiStore>(s, u, up, stream) : launch_gemm<DgradStoreNarrow>(s, u, stream);
    if (rc != NB_OK) return rc;
    if (want_x && (rc = run_dgrad(s, dx, stream)) != NB_OK) return rc;
    return want_a ? run_wgrad_f32(s, l.u, l.inp, l.dlora_a, nullptr, BT, r, C, l.accumulate, stream) : NB_OK;
}

}  // namespace

// ================================================================================ C ABI
extern "C" {

int nb_version(void) { return 100; }

const char *nb_last_error(void) { return g_err.c_str(); }

int nb_set_stream(void *stream)
{
    g_stream = static_cast<cudaStream_t>(stream);
    return NB_OK;
}
void *nb_get_stream(void) { return g_stream; }

int64_t nb_linear_out_elems(int64_t BT, int64_t OC, int act)
{
    if (BT < 0 || OC < 0) return -1;
    switch (act) {
        case NB_ACT_NONE: return BT * OC;
        case NB_ACT_GELU: return 2 * BT * OC;
        case NB_ACT_SWIGLU: return (OC % 2) ? -1 : BT * (OC / 2) + BT * OC;
        default: return -1;
    }
}

int nb_linear_forward_ex(void *out, void *pre_act, const void *inp, const void *weight,
                         const void *bias, int64_t BT, int64_t C, int64_t OC, int act, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (act != NB_ACT_NONE && act != NB_ACT_GELU && act != NB_ACT_SWIGLU)
        return fail(NB_ERR_INVALID_ARG, "unknown activation %d", act);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if (act == NB_ACT_SWIGLU && OC % 16 != 0)
        return fail(NB_ERR_UNSUPPORTED, "SwiGLU needs OC/2 to be a multiple of 8");
    if (!out || !inp || !weight) return fail(NB_ERR_INVALID_ARG, "out, inp and weight must not be NULL");
    if (!aligned16(out) || !aligned16(inp) || !aligned16(weight) || !aligned16(pre_act) ||
        (bias && (reinterpret_cast<uintptr_t>(bias) & 1u)))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;

    GemmArgs a{};
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = weight; a.b_rows = OC; a.b_cols = C;
    a.D = out; a.d_rows = BT; a.d_cols = (act == NB_ACT_SWIGLU) ? OC / 2 : OC; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(OC); a.K = static_cast<int>(C);
    a.bias = bias;
    a.splits = 1;
    if (act != NB_ACT_NONE && !pre_act) {
        // the activated result without its pre-activation: only NONE can skip the second plane
        return fail(NB_ERR_INVALID_ARG, "pre_act must be given when act != NONE");
    }
    if (act != NB_ACT_NONE) { a.E = pre_act; a.e_rows = BT; a.e_cols = OC; }
    if (act == NB_ACT_SWIGLU) a.swiglu_h = static_cast<int>(OC / 2);
    return run_forward(*s, a, act, stream);
}

int nb_linear_forward(void *out, const void *inp, const void *weight, const void *bias, int64_t BT,
                      int64_t C, int64_t OC, int act)
{
    void *pre = nullptr;
    if (out && BT >= 0 && OC >= 0) {
        if (act == NB_ACT_GELU) pre = static_cast<uint16_t *>(out) + BT * OC;
        if (act == NB_ACT_SWIGLU) pre = static_cast<uint16_t *>(out) + BT * (OC / 2);
    }
    return nb_linear_forward_ex(out, pre, inp, weight, bias, BT, C, OC, act, g_stream);
}

int nb_linear_backward_ex(void *dinp, void *dweight, void *dbias, const void *dout, const void *inp,
                          const void *weight, const void *pre_act, const void *inp_pre_act,
                          int64_t BT, int64_t C, int64_t OC, int act, int accumulate,
                          int dweight_dtype, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (act != NB_ACT_NONE && act != NB_ACT_GELU && act != NB_ACT_SWIGLU)
        return fail(NB_ERR_INVALID_ARG, "unknown activation %d", act);
    if (dweight_dtype != NB_DTYPE_F32 && dweight_dtype != NB_DTYPE_BF16)
        return fail(NB_ERR_INVALID_ARG, "unknown dweight dtype %d", dweight_dtype);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if (act == NB_ACT_SWIGLU && OC % 16 != 0)
        return fail(NB_ERR_UNSUPPORTED, "SwiGLU needs OC/2 to be a multiple of 8");
    if (!dout) return fail(NB_ERR_INVALID_ARG, "dout must not be NULL");
    if (act != NB_ACT_NONE && !pre_act)
        return fail(NB_ERR_INVALID_ARG, "pre_act is required when act != NONE");
    if (dinp && !weight) return fail(NB_ERR_INVALID_ARG, "weight is required to compute dinp");
    if (dweight && !inp) return fail(NB_ERR_INVALID_ARG, "inp is required to compute dweight");
    if (inp_pre_act && !dinp) return fail(NB_ERR_INVALID_ARG, "inp_pre_act given without dinp");
    if (dweight_dtype == NB_DTYPE_BF16 && accumulate && dweight)
        return fail(NB_ERR_UNSUPPORTED, "bf16 dweight cannot be accumulated across micro-steps");
    if (!aligned16(dinp) || !aligned16(dweight) || !aligned16(dbias) || !aligned16(dout) ||
        !aligned16(inp) || !aligned16(weight) || !aligned16(pre_act) || !aligned16(inp_pre_act))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");

    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;

    if (BT == 0) {
        if (!accumulate) {
            const size_t wsz = dweight_dtype == NB_DTYPE_F32 ? 4 : 2;
            if (dweight) NB_CUDA(cudaMemsetAsync(dweight, 0, static_cast<size_t>(OC * C) * wsz, stream));
            if (dbias) NB_CUDA(cudaMemsetAsync(dbias, 0, static_cast<size_t>(OC) * 4, stream));
        }
        return NB_OK;
    }

    // dz: either dout itself, or dout times this layer's activation derivative (workspace)
    const void *dz = dout;
    // The pass that forms dz also clears a dweight that layer_bwd_kernel adds to, which saves that launch (4096 rows, from zero,
    // with the schedule: 1024 -> 6144 SwiGLU 104 -> 98 us, 768 -> 3072 GELU 49.4 -> 45.7).
    Route r;
    if (dweight && dweight_dtype == NB_DTYPE_F32)
        r = route_backward(s->num_sms, dinp != nullptr, dbias != nullptr, inp_pre_act != nullptr, accumulate != 0,
                           static_cast<int>(BT), static_cast<int>(C), static_cast<int>(OC));
    float *clear_w = nullptr;
    if (act != NB_ACT_NONE) {
        if (dweight && dweight_dtype == NB_DTYPE_F32 && !accumulate && r.kernel == NB_ROUTE_LAYER_BWD &&
            layer_bwd_adds(*s, BT, C, OC, inp_pre_act != nullptr))
            clear_w = static_cast<float *>(dweight);
        float *const clear_b = clear_w ? static_cast<float *>(dbias) : nullptr;
        const long long nw = clear_w ? static_cast<long long>(OC * C) : 0, nb_ = clear_b ? static_cast<long long>(OC) : 0;
        if ((rc = ensure_workspace(*s, static_cast<size_t>(BT * OC) * 2, stream)) != NB_OK) return rc;
        if (act == NB_ACT_GELU) {
            const long long nvec = BT * OC / 8;
            rc = launch_chained(gelu_backward_kernel, dim3(elementwise_grid(*s, nvec)), 256, stream,
                                static_cast<uint4 *>(s->workspace), static_cast<const uint4 *>(dout),
                                static_cast<const uint4 *>(pre_act), nvec, clear_w, nw, clear_b, nb_);
        } else {
            const int hvec = static_cast<int>(OC / 16);
            rc = launch_chained(swiglu_backward_kernel, dim3(elementwise_grid(*s, BT * hvec)), 256, stream,
                                static_cast<uint4 *>(s->workspace), static_cast<const uint4 *>(dout),
                                static_cast<const uint4 *>(pre_act), BT, hvec, clear_w, nw, clear_b, nb_);
        }
        if (rc != NB_OK) return rc;
        ++g_launches;
        dz = s->workspace;
    }

    GemmArgs d{}, w{};
    // dinp[BT, C] = dz[BT, OC] . W[OC, C]
    d.A = dz; d.a_rows = BT; d.a_cols = OC;
    d.B = weight; d.b_rows = OC; d.b_cols = C;
    d.D = dinp; d.d_rows = BT; d.d_cols = C; d.d_dtype = 0;
    d.M = static_cast<int>(BT); d.N = static_cast<int>(C); d.K = static_cast<int>(OC);
    d.splits = 1;
    if (inp_pre_act) { d.E = inp_pre_act; d.e_rows = BT; d.e_cols = C; }
    if (dweight && dweight_dtype == NB_DTYPE_F32) {
        // dweight[OC, C] (+)= dz^T[OC, BT] . inp[BT, C]
        w.A = dz; w.a_rows = BT; w.a_cols = OC;
        w.B = inp; w.b_rows = BT; w.b_cols = C;
        w.D = dweight; w.d_rows = OC; w.d_cols = C; w.d_dtype = 1;
        w.M = static_cast<int>(OC); w.N = static_cast<int>(C); w.K = static_cast<int>(BT);
        w.splits = 1;
        w.dbias = static_cast<float *>(dbias);
        if (r.kernel == NB_ROUTE_TILE_PAIR)
            return launch_tile_pair_plan(*s, dinp ? &d : nullptr, w, inp_pre_act != nullptr, accumulate, r.pl, stream);
        // Both products of the layer in one launch (the usual case of a training step): the weight
        // gradient's k-blocks fill the waves the input gradient's tiles leave partly empty.
        if (r.kernel == NB_ROUTE_LAYER_BWD) {
            rc = run_layer_bwd(*s, dz, weight, inp, dinp, inp_pre_act, dweight, static_cast<float *>(dbias), BT, C,
                               OC, accumulate, clear_w != nullptr, stream);
            if (rc != NB_ERR_UNSUPPORTED) return rc;
        }
    }

    if (dinp && (rc = run_dgrad(*s, d, stream)) != NB_OK) return rc;

    if (dweight) {  // dweight[OC, C] (+)= dz^T[OC, BT] . inp[BT, C]
        GemmArgs a{};
        a.A = dz; a.a_rows = BT; a.a_cols = OC;
        a.B = inp; a.b_rows = BT; a.b_cols = C;
        a.D = dweight; a.d_rows = OC; a.d_cols = C;
        a.M = static_cast<int>(OC); a.N = static_cast<int>(C); a.K = static_cast<int>(BT);
        if (dweight_dtype == NB_DTYPE_F32) {
            rc = run_wgrad_f32(*s, dz, inp, dweight, static_cast<float *>(dbias), BT, OC, C, accumulate,
                               stream);
            dbias = nullptr;  // done inside the wgrad kernel
        } else {
            a.d_dtype = 0;
            a.splits = 1;
            rc = launch_gemm_auto<WgradBf16_1, WgradBf16_2>(*s, a, stream);
        }
        if (rc != NB_OK) return rc;
    }

    if (dbias) {
        if ((rc = launch_dbias(*s, static_cast<float *>(dbias), dz, BT, OC, accumulate, stream)) != NB_OK)
            return rc;
    }
    return NB_OK;
}

int nb_linear_backward(void *dinp, void *dweight, void *dbias, const void *dout, const void *inp,
                       const void *weight, const void *pre_act, int64_t BT, int64_t C, int64_t OC,
                       int accumulate)
{
    return nb_linear_backward_ex(dinp, dweight, dbias, dout, inp, weight, pre_act, nullptr, BT, C, OC,
                                 pre_act ? NB_ACT_GELU : NB_ACT_NONE, accumulate, NB_DTYPE_F32,
                                 g_stream);
}

int nb_reduce_dbias(void *dbias, const void *dout, int64_t BT, int64_t OC, int accumulate)
{
    if (!dbias || !dout) return fail(NB_ERR_INVALID_ARG, "dbias and dout must not be NULL");
    if (BT < 0 || OC <= 0) return fail(NB_ERR_INVALID_ARG, "negative or zero dimension");
    if (OC % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "OC must be a multiple of 8");
    if (!aligned16(dbias) || !aligned16(dout))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    return launch_dbias(*s, static_cast<float *>(dbias), dout, BT, OC, accumulate, g_stream);
}

int nb_lm_head_ce_forward(void *logits, void *loss, void *lse, const void *inp, const void *weight,
                          const void *targets, int64_t BT, int64_t C, int64_t Vp, int64_t V,
                          void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, Vp);
    if (rc != NB_OK) return rc;
    if (V <= 0 || V > Vp) return fail(NB_ERR_INVALID_ARG, "V must be within (0, Vp]");
    if (!logits || !loss || !lse || !inp || !weight || !targets)
        return fail(NB_ERR_INVALID_ARG, "all pointers must be given");
    if (!aligned16(logits) || !aligned16(inp) || !aligned16(weight) ||
        (reinterpret_cast<uintptr_t>(loss) & 3u) || (reinterpret_cast<uintptr_t>(lse) & 3u) ||
        (reinterpret_cast<uintptr_t>(targets) & 3u))
        return fail(NB_ERR_INVALID_ARG, "misaligned pointer");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    const int stats_ld = 2 * static_cast<int>((Vp + 255) / 256);
    if ((rc = ensure_workspace(*s, static_cast<size_t>(BT) * stats_ld * sizeof(float2), stream)) != NB_OK) return rc;
    GemmArgs a{};
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = weight; a.b_rows = Vp; a.b_cols = C;
    a.D = logits; a.d_rows = BT; a.d_cols = Vp; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(Vp); a.K = static_cast<int>(C);
    a.splits = 1;
    a.stats = static_cast<float2 *>(s->workspace);
    a.stats_ld = stats_ld;
    a.v_real = static_cast<int>(V);
    if ((rc = launch_gemm_auto<FwdStoreStats1, FwdStoreStats2>(*s, a, stream)) != NB_OK) return rc;
    rc = launch_chained(ce_reduce_kernel, dim3(static_cast<unsigned>((BT + 7) / 8)), 256, stream, static_cast<float *>(loss),
                        static_cast<float *>(lse), static_cast<const float2 *>(s->workspace), stats_ld,
                        static_cast<const __nv_bfloat16 *>(logits), Vp, static_cast<const int *>(targets), BT,
                        static_cast<int>(V));
    if (rc != NB_OK) return rc;
    ++g_launches;
    return NB_OK;
}

int nb_ce_backward(void *dlogits, const void *logits, const void *lse, const void *targets, float gscale,
                   int64_t BT, int64_t Vp, int64_t V, void *stream_)
{
    if (BT < 0 || Vp <= 0 || V <= 0 || V > Vp) return fail(NB_ERR_INVALID_ARG, "bad dimension");
    if (Vp % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "Vp must be a multiple of 8");
    if (BT >= (1ll << 31) || Vp >= (1ll << 31)) return fail(NB_ERR_UNSUPPORTED, "dimension too large");
    if (!dlogits || !logits || !lse || !targets) return fail(NB_ERR_INVALID_ARG, "all pointers must be given");
    if (!aligned16(dlogits) || !aligned16(logits)) return fail(NB_ERR_INVALID_ARG, "misaligned pointer");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    const int vec_per_row = static_cast<int>(Vp / 8);
    rc = launch_chained(ce_backward_kernel, dim3(elementwise_grid(*s, BT * vec_per_row)), 256,
                        static_cast<cudaStream_t>(stream_), static_cast<uint4 *>(dlogits), static_cast<const uint4 *>(logits),
                        static_cast<const float *>(lse), static_cast<const int *>(targets), gscale, BT, vec_per_row,
                        static_cast<int>(V));
    if (rc != NB_OK) return rc;
    ++g_launches;
    return NB_OK;
}

int nb_lora_linear_forward(void *out, void *t, const void *inp, const void *weight, const void *bias,
                           const void *lora_a, const void *lora_b, float scale, int64_t BT, int64_t C,
                           int64_t OC, int64_t r, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if (r < 8 || r > 64 || r % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "rank must be 8..64, a multiple of 8");
    if (!out || !t || !inp || !weight || !lora_a || !lora_b)
        return fail(NB_ERR_INVALID_ARG, "out, t, inp, weight, lora_a and lora_b must not be NULL");
    if (!aligned16(out) || !aligned16(t) || !aligned16(inp) || !aligned16(weight) || !aligned16(lora_a) ||
        !aligned16(lora_b))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    bool late = false;
    if ((rc = run_lora_down(*s, t, inp, lora_a, scale, BT, C, r, stream, &late)) != NB_OK) return rc;
    GemmArgs a{};  // out = inp . W^T (+ bias) + t . B^T: r extra columns of K
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = weight; a.b_rows = OC; a.b_cols = C;
    a.D = out; a.d_rows = BT; a.d_cols = OC; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(OC); a.K = static_cast<int>(C);
    a.bias = bias;
    a.splits = 1;
    a.A2 = t; a.a2_rows = BT; a.a2_cols = r;
    a.B2 = lora_b; a.b2_rows = OC; a.b2_cols = r;
    a.k2 = static_cast<int>(r);
    a.wait_ext = late;
    return run_forward(*s, a, NB_ACT_NONE, stream);
}

int nb_lora_linear_backward(void *dinp, void *dlora_a, void *dlora_b, void *u, const void *dout,
                            const void *inp, const void *weight, const void *lora_a, const void *lora_b,
                            const void *t, float scale, int64_t BT, int64_t C, int64_t OC, int64_t r,
                            int accumulate, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if (r < 8 || r > 64 || r % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "rank must be 8..64, a multiple of 8");
    if (!u || !dout || !inp || !lora_a || !lora_b)
        return fail(NB_ERR_INVALID_ARG, "u, dout, inp, lora_a and lora_b must not be NULL");
    if (dinp && !weight) return fail(NB_ERR_INVALID_ARG, "weight is required to compute dinp");
    if (dlora_b && !t) return fail(NB_ERR_INVALID_ARG, "t (from the forward call) is required for dlora_b");
    if (!aligned16(dinp) || !aligned16(dlora_a) || !aligned16(dlora_b) || !aligned16(u) || !aligned16(dout) ||
        !aligned16(inp) || !aligned16(weight) || !aligned16(lora_a) || !aligned16(lora_b) || !aligned16(t))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    if (BT == 0) {
        if (!accumulate) {
            if (dlora_a) NB_CUDA(cudaMemsetAsync(dlora_a, 0, static_cast<size_t>(r * C) * 4, stream));
            if (dlora_b) NB_CUDA(cudaMemsetAsync(dlora_b, 0, static_cast<size_t>(OC * r) * 4, stream));
        }
        return NB_OK;
    }
    const LoraBwd l{dinp, dlora_a, dlora_b, u, dout, inp, weight, lora_a, lora_b, t, 0, 0, scale, BT, C, OC, r, accumulate};
    return run_lora_backward(*s, l, stream);
}

// --- adapters that share an input, stacked (q, k, v; gate, up): one rank-R product for all of them
namespace {
int check_stack(int64_t r, int64_t R, int64_t off)
{
    if (r < 8 || r > 64 || r % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "rank must be 8..64, a multiple of 8");
    if (R < r || R > 64 || R % 8 != 0)
        return fail(NB_ERR_UNSUPPORTED, "stacked rank must be a multiple of 8, at least r and at most 64");
    if (off < 0 || off % 8 != 0 || off + r > R)
        return fail(NB_ERR_INVALID_ARG, "slice [%lld, %lld) does not lie in the %lld stacked columns",
                    static_cast<long long>(off), static_cast<long long>(off + r), static_cast<long long>(R));
    return NB_OK;
}
}  // namespace

int nb_lora_down_stacked(void *t_stack, const void *inp, const void *a_stack, float scale, int64_t BT,
                         int64_t C, int64_t R, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, R);
    if (rc != NB_OK) return rc;
    if (R > 64) return fail(NB_ERR_UNSUPPORTED, "stacked rank must be at most 64");
    if (!t_stack || !inp || !a_stack) return fail(NB_ERR_INVALID_ARG, "t_stack, inp and a_stack must not be NULL");
    if (!aligned16(t_stack) || !aligned16(inp) || !aligned16(a_stack))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    return run_lora_down(*s, t_stack, inp, a_stack, scale, BT, C, R, stream);
}

int nb_lora_linear_forward_stacked(void *out, const void *inp, const void *weight, const void *bias,
                                   const void *t_stack, const void *lora_b, int64_t BT, int64_t C,
                                   int64_t OC, int64_t r, int64_t R, int64_t off, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if ((rc = check_stack(r, R, off)) != NB_OK) return rc;
    if (!out || !inp || !weight || !t_stack || !lora_b)
        return fail(NB_ERR_INVALID_ARG, "out, inp, weight, t_stack and lora_b must not be NULL");
    if (!aligned16(out) || !aligned16(inp) || !aligned16(weight) || !aligned16(t_stack) || !aligned16(lora_b))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (BT == 0) return NB_OK;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    GemmArgs a{};  // out = inp . W^T (+ bias) + t_slice . B^T: r extra columns of K
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = weight; a.b_rows = OC; a.b_cols = C;
    a.D = out; a.d_rows = BT; a.d_cols = OC; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(OC); a.K = static_cast<int>(C);
    a.bias = bias;
    a.splits = 1;
    a.A2 = static_cast<const uint16_t *>(t_stack) + off; a.a2_rows = BT; a.a2_cols = r; a.a2_ld = R;
    a.B2 = lora_b; a.b2_rows = OC; a.b2_cols = r;
    a.k2 = static_cast<int>(r);
    return run_forward(*s, a, NB_ACT_NONE, stream);
}

int nb_lora_linear_backward_stacked(void *dinp, void *dlora_b, void *u_stack, const void *dout,
                                    const void *weight, const void *lora_a, const void *lora_b,
                                    const void *t_stack, float scale, int64_t BT, int64_t C, int64_t OC,
                                    int64_t r, int64_t R, int64_t off, int accumulate, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, OC);
    if (rc != NB_OK) return rc;
    if ((rc = check_stack(r, R, off)) != NB_OK) return rc;
    if (!u_stack || !dout || !lora_a || !lora_b)
        return fail(NB_ERR_INVALID_ARG, "u_stack, dout, lora_a and lora_b must not be NULL");
    if (dinp && !weight) return fail(NB_ERR_INVALID_ARG, "weight is required to compute dinp");
    if (dlora_b && !t_stack) return fail(NB_ERR_INVALID_ARG, "t_stack (from the forward calls) is required for dlora_b");
    if (!aligned16(dinp) || !aligned16(dlora_b) || !aligned16(u_stack) || !aligned16(dout) || !aligned16(weight) ||
        !aligned16(lora_a) || !aligned16(lora_b) || !aligned16(t_stack))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    if (BT == 0) {
        if (!accumulate && dlora_b) NB_CUDA(cudaMemsetAsync(dlora_b, 0, static_cast<size_t>(OC * r) * 4, stream));
        return NB_OK;
    }
    const LoraBwd l{dinp, nullptr, dlora_b, static_cast<uint16_t *>(u_stack) + off, dout, nullptr, weight, lora_a, lora_b,
                    static_cast<const uint16_t *>(t_stack) + off, static_cast<uint64_t>(R), static_cast<uint64_t>(R),
                    scale, BT, C, OC, r, accumulate};
    return run_lora_backward(*s, l, stream);
}

int nb_lora_da_stacked(void *da_stack, const void *u_stack, const void *inp, int64_t BT, int64_t C, int64_t R,
                       int accumulate, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    int rc = check_dims(BT, C, R);
    if (rc != NB_OK) return rc;
    if (R > 64) return fail(NB_ERR_UNSUPPORTED, "stacked rank must be at most 64");
    if (!da_stack || !u_stack || !inp) return fail(NB_ERR_INVALID_ARG, "da_stack, u_stack and inp must not be NULL");
    if (!aligned16(da_stack) || !aligned16(u_stack) || !aligned16(inp))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    if ((rc = get_state(&s)) != NB_OK) return rc;
    if (BT == 0) {
        if (!accumulate) NB_CUDA(cudaMemsetAsync(da_stack, 0, static_cast<size_t>(R * C) * 4, stream));
        return NB_OK;
    }
    GemmArgs w{};  // dA (+)= u^T . inp
    w.A = u_stack; w.a_rows = BT; w.a_cols = R;
    w.B = inp; w.b_rows = BT; w.b_cols = C;
    w.D = da_stack; w.d_rows = R; w.d_cols = C; w.d_dtype = 1;
    w.M = static_cast<int>(R); w.N = static_cast<int>(C); w.K = static_cast<int>(BT);
    const int kw = kblocks_of(BT);
    const SmallPlan pl = plan_pair(s->num_sms, 0, 0, 0, 1, w.M, w.N, kw, false, false,
                                   backward_us(s->num_sms, 0, w.K, w.N, w.M, 0, kw, accumulate != 0, true, false), false);
    if (pl.bn) return launch_tile_pair_plan(*s, nullptr, w, false, accumulate, pl, stream);
    return run_wgrad_f32(*s, u_stack, inp, da_stack, nullptr, BT, R, C, accumulate, stream);
}

int nb_cast_f32_to_bf16(void *dst, const void *src, int64_t n, void *stream_)
{
    if (n < 0) return fail(NB_ERR_INVALID_ARG, "negative size");
    if (n == 0) return NB_OK;
    if (!dst || !src) return fail(NB_ERR_INVALID_ARG, "dst and src must not be NULL");
    if (!aligned16(dst) || !aligned16(src))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    rc = launch_chained(cast_f32_bf16_kernel, dim3(elementwise_grid(*s, n / 8 + 1)), 256, static_cast<cudaStream_t>(stream_),
                        static_cast<__nv_bfloat16 *>(dst), static_cast<const float *>(src), n);
    if (rc != NB_OK) return rc;
    ++g_launches;
    return NB_OK;
}

int nb_workspace_reserve(int64_t bytes)
{
    if (bytes < 0) return fail(NB_ERR_INVALID_ARG, "negative size");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    return ensure_workspace(*s, static_cast<size_t>(bytes));
}

int nb_release(void)
{
    std::lock_guard<std::mutex> lock(g_mu);
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(NB_ERR_UNSUPPORTED, "device index %d", dev);
    DeviceState &s = g_dev[dev];
    if (!s.init) return NB_OK;
    NB_CUDA(cudaDeviceSynchronize());
    if (s.workspace) NB_CUDA(cudaFree(s.workspace));
    if (s.status) NB_CUDA(cudaFree(s.status));
    s = DeviceState();
    return NB_OK;
}

int nb_check_status(void)
{
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    NB_CUDA(cudaDeviceSynchronize());
    int host[4] = {0, 0, 0, 0};
    NB_CUDA(cudaMemcpy(host, s->status, sizeof(host), cudaMemcpyDeviceToHost));
    if (host[0] == 0) return NB_OK;
    NB_CUDA(cudaMemset(s->status, 0, 64));
    if (host[0] == kStatusTimeout)
        return fail(NB_ERR_TIMEOUT, "a bounded device wait expired (wait id %d, block %d)", host[1],
                    host[2]);
    return fail(NB_ERR_CUDA, "kernel reported internal error %d (block %d)", host[0], host[2]);
}

int64_t nb_kernel_launches(void) { return g_launches.load(); }

int nb_debug_split_plan(int64_t M, int64_t N, int64_t K, int slots, int tile_m, int *out)
{
    if (!out || M <= 0 || N <= 0 || K <= 0 || slots <= 0 || (tile_m != 128 && tile_m != 256))
        return fail(NB_ERR_INVALID_ARG, "bad argument");
    const int tiles_m = static_cast<int>((M + tile_m - 1) / tile_m);
    const int tiles_n = static_cast<int>((N + 255) / 256);
    const int kblocks = static_cast<int>((K + kBlockK - 1) / kBlockK);
    int splits = choose_splits(tiles_m * tiles_n, kblocks, slots);
    const int kps = (kblocks + splits - 1) / splits;  // as launch_gemm derives it
    splits = (kblocks + kps - 1) / kps;
    out[0] = tiles_m;
    out[1] = tiles_n;
    out[2] = splits;
    out[3] = kps;
    out[4] = kblocks;
    return NB_OK;
}

int nb_debug_layer_bwd_plan(int64_t BT, int64_t C, int64_t OC, int pairs, int flags, int *out,
                            int64_t cap)
{
    if (!out || cap < 8 || BT <= 0 || C <= 0 || OC <= 0) return -fail(NB_ERR_INVALID_ARG, "bad argument");
    LayerBwdParams p;
    const int rc = plan_layer_bwd(p, BT, C, OC, pairs, (flags & NB_PLAN_GELU_GRAD) != 0, (flags & NB_PLAN_LAUNCHED) != 0,
                                  (flags & NB_PLAN_FRESH) != 0);
    if (rc != NB_OK) return -rc;
    out[0] = p.d_tiles_m; out[1] = p.d_tiles_n; out[2] = p.d_kblocks;
    out[3] = p.w_tiles_m; out[4] = p.w_tiles_n; out[5] = p.w_kblocks;
    out[6] = p.w_kbc; out[7] = p.d_rounds + p.w_rounds;
    int64_t n = 8;
    int records = 0;
    for (int q = 0; q < pairs; ++q) {
        LbIter it(p, q);
        LbUnit u;
        while (it.next(p, u)) {
            const int part = flags & NB_PLAN_SUMS ? chain_len(u, p.w_chain) : u.kb1 - u.kb0;
            for (int kb = u.kb0; kb < u.kb1; kb += part) {
                if (n + 6 > cap) return -fail(NB_ERR_INVALID_ARG, "output buffer too small");
                out[n++] = q; out[n++] = u.is_w; out[n++] = u.m_blk; out[n++] = u.n_blk;
                out[n++] = kb; out[n++] = LbIter::imin(kb + part, u.kb1);
                ++records;
            }
        }
    }
    return records;
}

int nb_debug_route(int call, int64_t BT, int64_t C, int64_t OC, int64_t r, int act, int flags, int sms, int *out)
{
    if (!out || BT <= 0 || C <= 0 || OC <= 0 || sms < 2 || BT >= (1ll << 31) || C >= (1ll << 31) || OC >= (1ll << 31))
        return -fail(NB_ERR_INVALID_ARG, "bad argument");
    const int M = static_cast<int>(BT), K = static_cast<int>(C), N = static_cast<int>(OC), R = static_cast<int>(r);
    const bool adapter = call == NB_CALL_LORA_FORWARD || call == NB_CALL_LORA_BACKWARD;
    if (adapter && (r < 8 || r > 64 || r % 8 != 0)) return -fail(NB_ERR_UNSUPPORTED, "rank must be 8..64, a multiple of 8");
    const bool dinp = flags & NB_CALL_DINP, dweight = flags & NB_CALL_DWEIGHT, dbias = flags & NB_CALL_DBIAS;
    const bool gelu = flags & NB_CALL_GELU_GRAD, accumulate = flags & NB_CALL_ACCUMULATE;
    int n = 0;
    auto put = [&](int kernel, int width, int shared, int per_sm) {
        out[4 * n] = kernel; out[4 * n + 1] = width; out[4 * n + 2] = shared; out[4 * n + 3] = per_sm;
        ++n;
    };
    auto tiles = [&](int kernel, const SmallPlan &pl) { put(kernel, pl.bn, pl.cluster, pl.two ? 2 : 1); };
    auto product = [&](const Route &t) {
        if (t.kernel == NB_ROUTE_TILE) tiles(t.kernel, t.pl);
        else put(t.kernel, t.kernel == NB_ROUTE_GEMM_192 ? 192 : 256, 1, 1);
    };
    auto narrow = [&](const SmallPlan &pl) {
        if (pl.bn) tiles(NB_ROUTE_TILE, pl);
        else put(NB_ROUTE_GEMM, kNarrowN, 1, 1);
    };
    if (call == NB_CALL_FORWARD || call == NB_CALL_LORA_FORWARD) {
        if (adapter) narrow(plan_lora_down(sms, M, R, kblocks_of(K)));
        const Route t = route_forward(sms, M, N, K, adapter ? NB_ACT_NONE : act, adapter);
        const int span = act == NB_ACT_SWIGLU ? N / 2 : N;
        if (t.kernel == NB_ROUTE_ROWS)
            put(t.kernel, kRowsFeatures, rows_split(sms, (span + kRowsFeatures - 1) / kRowsFeatures, K),
                rows_many(sms, M, span, act == NB_ACT_SWIGLU) ? 4 : 2);
        else product(t);
    } else if (call == NB_CALL_BACKWARD) {
        const Route t = dweight ? route_backward(sms, dinp, dbias, gelu, accumulate, M, K, N) : Route{};
        if (t.kernel == NB_ROUTE_TILE_PAIR) {
            tiles(t.kernel, t.pl);
        } else if (t.kernel == NB_ROUTE_LAYER_BWD) {
            LayerBwdParams p;
            const int rc = plan_layer_bwd(p, BT, C, OC, sms / 2 < kMaxPairs ? sms / 2 : kMaxPairs, gelu, true, !accumulate);
            if (rc != NB_OK) return -rc;
            put(t.kernel, p.d_w, 1, 1);
        } else {
            if (dinp) product(route_dgrad(sms, M, K, kblocks_of(N)));
            if (dweight) put(NB_ROUTE_GEMM, 256, 1, 1);
        }
    } else if (call == NB_CALL_LORA_BACKWARD) {
        const LoraRoute t = dbias ? route_lora_backward(sms, M, K, N, R, dinp, dweight, accumulate) : LoraRoute{};
        if (t.ub.bn) tiles(NB_ROUTE_TILE_PAIR, t.ub);
        else if (dbias) put(NB_ROUTE_LORA_UDB, kNarrowN, 1, 1);
        else narrow(plan_lora_u(sms, M, R, kblocks_of(N)));
        if (t.xa.bn) {
            tiles(NB_ROUTE_TILE_PAIR, t.xa);
        } else {
            if (dinp) product(route_dgrad(sms, M, K, kblocks_of(N) + 1));
            if (dweight && t.ub.bn) tiles(NB_ROUTE_TILE_PAIR, t.a1);
            else if (dweight && !dbias) put(NB_ROUTE_GEMM, 256, 1, 1);
        }
    } else {
        return -fail(NB_ERR_INVALID_ARG, "unknown call %d", call);
    }
    return n;
}

int nb_debug_gemm_timeout(void *out, const void *inp, const void *weight, int64_t limit_us)
{
    if (!out || !inp || !weight) return fail(NB_ERR_INVALID_ARG, "out, inp and weight must not be NULL");
    if (!aligned16(out) || !aligned16(inp) || !aligned16(weight))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (limit_us < 100 || limit_us > 1000000)
        return fail(NB_ERR_INVALID_ARG, "limit_us must be within [100, 1000000]");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    const int64_t BT = 128, C = 256, OC = 256;  // one tile, one CTA, four k-blocks
    GemmArgs a{};
    a.A = inp; a.a_rows = BT; a.a_cols = C;
    a.B = weight; a.b_rows = OC; a.b_cols = C;
    a.D = out; a.d_rows = BT; a.d_cols = OC; a.d_dtype = 0;
    a.M = static_cast<int>(BT); a.N = static_cast<int>(OC); a.K = static_cast<int>(C);
    a.splits = 1;
    a.debug_stop_kb = 2;  // the first two k-blocks are loaded, the third never is
    a.debug_timeout_ns = static_cast<unsigned long long>(limit_us) * 1000ull;
    return launch_gemm<FwdStore1>(*s, a, g_stream);
}

int nb_debug_wait_timeout(int64_t limit_us)
{
    if (limit_us < 1 || limit_us > 1000000)
        return fail(NB_ERR_INVALID_ARG, "limit_us must be within [1, 1000000]");
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceState *s;
    int rc = get_state(&s);
    if (rc != NB_OK) return rc;
    wait_timeout_kernel<<<1, 32, 0, g_stream>>>(s->status, static_cast<unsigned long long>(limit_us) * 1000ull);
    NB_CUDA(cudaGetLastError());
    ++g_launches;
    return NB_OK;
}

// ----------------------------------------------------------------------------- no allocation
// Scratch for nb_gelu_dbias_noalloc: part of the library image, so it exists on every device that
// loads the library without anyone allocating it. In host code `nb_noalloc_scratch` is only a
// handle for the runtime, not a device address: the address a kernel can use comes from
// cudaGetSymbolAddress, once per device.
}  // extern "C" (the array and its bookkeeping have internal linkage)

namespace {
static __device__ __align__(256) unsigned char nb_noalloc_scratch[NB_NOALLOC_MAX_ELEMS * 2];
void *g_noalloc_ptr[kMaxDevices] = {};
int g_noalloc_sms[kMaxDevices] = {};
}  // namespace

extern "C" {

int nb_gelu_dbias_noalloc(void *dbias, const void *dout, const void *pre_act, int64_t BT, int64_t OC,
                          int accumulate, void *stream_)
{
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!dbias || !dout || !pre_act)
        return fail(NB_ERR_INVALID_ARG, "dbias, dout and pre_act must not be NULL");
    if (BT < 0 || OC <= 0) return fail(NB_ERR_INVALID_ARG, "negative or zero dimension");
    if (OC % 8 != 0) return fail(NB_ERR_UNSUPPORTED, "OC must be a multiple of 8");
    if (!aligned16(dbias) || !aligned16(dout) || !aligned16(pre_act))
        return fail(NB_ERR_INVALID_ARG, "tensor pointers must be 16-byte aligned");
    if (BT >= (1ll << 31) || OC >= (1ll << 31) || BT * OC > static_cast<int64_t>(NB_NOALLOC_MAX_ELEMS))
        return fail(NB_ERR_UNSUPPORTED,
                    "BT*OC = %lld exceeds the built-in scratch of %d elements (NB_NOALLOC_MAX_ELEMS); "
                    "use nb_linear_backward_ex, which allocates a workspace",
                    static_cast<long long>(BT * OC), NB_NOALLOC_MAX_ELEMS);

    std::lock_guard<std::mutex> lock(g_mu);
    int dev = 0;
    NB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(NB_ERR_UNSUPPORTED, "device index %d", dev);
    if (!g_noalloc_ptr[dev]) {  // set-up, once per device, with that device current
        void *ptr = nullptr;
        NB_CUDA(cudaGetSymbolAddress(&ptr, nb_noalloc_scratch));
        int sms = 0;
        NB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (!ptr || sms <= 0) return fail(NB_ERR_CUDA, "could not resolve the built-in scratch array");
        g_noalloc_sms[dev] = sms;
        g_noalloc_ptr[dev] = ptr;
    }
    DeviceState local;  // only the SM count is read by the launch helpers below
    local.num_sms = g_noalloc_sms[dev];
    void *dz = g_noalloc_ptr[dev];

    if (BT > 0) {
        // dz = dout * gelu'(pre_act) overwrites the first BT*OC elements of the scratch
        const long long nvec = BT * OC / 8;
        const int rc = launch_chained(gelu_backward_kernel, dim3(elementwise_grid(local, nvec)), 256, stream,
                                      static_cast<uint4 *>(dz), static_cast<const uint4 *>(dout),
                                      static_cast<const uint4 *>(pre_act), nvec, nullptr, 0, nullptr, 0);
        if (rc != NB_OK) return rc;
        ++g_launches;
    }
    return launch_dbias(local, static_cast<float *>(dbias), dz, BT, OC, accumulate, stream);
}

}  // extern "C"
