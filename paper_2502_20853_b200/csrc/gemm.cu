// Block-scaled MXFP4 GEMM for sm_100a:  D[M,N] = deq(A)[M,Kc] * deq(B)[N,Kc]^T  (Eq. 3-5).
//
// One persistent, warp-specialised CTA per SM (12 warps):
//   warp 0      TMA producer: packed E2M1 tiles (128B-swizzled, 256 K elements per stage) -> shared-memory ring
//   warp 1      MMA issuer: tcgen05.mma kind::mxf4.block_scale, FP32 accumulators in TMEM; owns the TMEM
//               allocation
//   warp 2      scale copier: tcgen05.cp (scales smem -> TMEM).  tcgen05 operations of ONE thread run in
//               order, so copies issued by the MMA thread would stall its MMAs; from a thread of their own
//               they overlap them completely.  Each ring stage has its own scale columns in TMEM.
//   warp 3      second producer: the scale chunks (issuing an asynchronous copy costs its thread ~100 ns, a stage needs five)
//   warps 4-11  epilogue: tcgen05.ld -> (+bias) -> cast -> swizzled staging in shared memory -> TMA store;
//               two warps share each quarter of the TMEM lanes and split the columns
// Every mbarrier wait is bounded; on expiry MXFP4_DEV_TIMEOUT is raised and all roles drain.
#include <algorithm>

#include "common.cuh"
#include "quant_tile.cuh"
#include "tma.cuh"

namespace mx {

constexpr int kBM = 128;           // rows of A per tile (one UMMA M)
constexpr int kBKBytes = 128;      // packed bytes of K per stage = 256 elements = one 128B swizzle atom
constexpr int kBKElems = 256;
constexpr int kMmaKBytes = 32;     // one tcgen05.mma kind::mxf4 consumes K = 64 elements = 32 bytes
constexpr int kSfChunk = 512;      // scales of 128 rows x 4 blocks (= 128 K elements)
constexpr int kEpiWarp0 = 4;       // first epilogue warp
constexpr int kEpiWarps = 8;
constexpr int kGemmThreads = 32 * (kEpiWarp0 + kEpiWarps);
constexpr int kStagingBytes = 2048;             // per epilogue warp: 32 rows x 64 bytes

template <int BN>
struct GemmCfg {
    static constexpr int kRB = (BN + 127) / 128;                        // 128-row scale blocks of B per tile
    static constexpr int kABytes = kBM * kBKBytes;                      // 16 KB
    static constexpr int kBBytes = BN * kBKBytes;
    static constexpr int kSfaBytes = 2 * kSfChunk;                      // two K chunks of 128 elements
    static constexpr int kSfbBytes = 2 * kSfChunk * kRB;
    static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;
    static constexpr int kStages = BN <= 128 ? 5 : 4;
    static constexpr int kStagingBufs = BN <= 192 ? BN / 64 : 1;        // up to 192: one buffer per 32-column chunk of a warp's share
    static constexpr int kAccStages = (BN <= 192) ? 2 : 1;              // tiles up to 192 wide leave room for two accumulators
    static constexpr int kSfCol = kAccStages * BN;                      // TMEM columns: accumulators, then per ring stage SFA (8) + SFB (8 kRB)
    static constexpr int kSfSlot = 8 + 8 * kRB;
    static constexpr int kTmemCols = 512;
    static constexpr int kStagingOff = kStages * kStageBytes;           // multiple of 1024
    static constexpr int kBarOff = kStagingOff + kEpiWarps * kStagingBufs * kStagingBytes;
    static constexpr int kBiasOff = kBarOff + 256;                      // a line of BN / 2 bf16 per epilogue warp
    static constexpr int kSmemBytes = kBiasOff + kEpiWarps * BN + 1024 /*align*/;
    static_assert(kSfCol + kStages * kSfSlot <= 512, "TMEM budget");
    static_assert(kStageBytes % 1024 == 0, "stage alignment");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

// Division by a number known at launch: the quotient of n < 2^31 by a multiplication (the roles of a kernel find their tile's
// coordinates once per tile in the middle of their chains; the compiler's division is a chain of about 150 cycles, and a role
// needed up to four).
struct FastDiv {
    uint32_t d, m, s;
    __device__ __forceinline__ int div(int n) const { return (int)((__umulhi((uint32_t)n, m) + (uint32_t)n) >> s); }
    __device__ __forceinline__ int mod(int n) const { return n - div(n) * (int)d; }
};
static FastDiv fast_div(int64_t d)
{
    FastDiv f = {(uint32_t)d, 0u, 0u};
    while ((1ll << f.s) < d) f.s++;
    f.m = (uint32_t)((((1ull << f.s) - (uint64_t)d) << 32) / (uint64_t)d + 1u);
    return f;
}

struct GemmParams {
    const uint8_t *sfa;   // scales of A, tiled order
    const uint8_t *sfb;
    int64_t M, N, Kc;
    int nblk4;            // ceil(Kc/32/4): 512-byte chunks per 128-row block
    int rbA, rbB;         // 128-row scale blocks present in A / B buffers
    int tiles_m, tiles_n, splits, kt_total, kt_per_split;
    FastDiv by_splits, by_tiles_n;
    // the walk of the B-stationary kernels, see Walk
    FastDiv by_rest_rows, by_rest_workers;
    int abreast, rounds, rows, rest_row0, share, extra;
    int head;             // second product of a launch of CTA pairs: see pair_item
    int out_fp32;         // element type of the stored tile (FP32 also for split-K partials)
    const __nv_bfloat16 *bias;   // applied only when splits == 1 (and by the cluster kernel, whose sum is complete)
    uint32_t *dev_status;
    void *d;              // the caller's output and its leading dimension (cluster kernel: plain stores)
    int64_t ldd;
    uint32_t spin_limit;  // polls after which a bounded wait gives up (kWaitSpinLimit in normal use)
    int withhold_loads;   // self-test of the drain path: the producers issue nothing, so every wait runs out
};

// One product of a launch, and the one or two products of a launch.
struct GemmJob {
    CUtensorMap a, b, d, dw;
    GemmParams p;
};
struct PairJob : GemmJob {
    CUtensorMap sfa, sfb;
};
struct NoJob {};

// How the workers (CTAs, or pairs of them) of the B-stationary kernels share the tiles.  A worker keeps the B block of its tile
// column for as long as it can, and all workers write the same stretch of the output at the same time: stores to many distant
// places are slow here (a kernel that does nothing but store, 384 bytes of a row at a time: 4.7-5.1 TB/s with a far-away
// stretch of rows for each SM, 5.5-5.8 TB/s when all SMs fill the same rows).  So `abreast` workers go down each column,
// taking its row tiles in turn, and at any moment all columns are near the same rows (the columns ask for an A tile at about
// the same time, too, and it comes from L2).  Workers that are left over because the columns do not divide
// their number take the last rows: contiguous ranges, of equal length, of those rows' tiles, numbered column by column.  With
// more columns than workers everything is shared that way.
// Against contiguous ranges of all tiles, in us: 401408 x 384 x 96 75.7 -> 64.9, 100352 x 1536 x 384 87 -> 58, 25216 x 1536 x 384
// 19.8 -> 18.1; on pairs 100352 x 1536 x 768 75.9 -> 66.4, 50432 x 4096 x 1024 106 -> 101, 50432 x 2304 x 768 52 -> 50.
struct Walk {
    int count;            // tiles of this worker
    int col, row, step;   // step > 0: rows row, row + step, .. of the column; 0: the tiles t0, t0 + 1, .. of the last rows
    int t0;
};
struct WalkItem {
    int col, row;
    bool first, last;   // of this worker's run in the column
};
__device__ __forceinline__ Walk walk_begin(const GemmParams &p, int w)
{
    Walk x;
    const int r = p.by_tiles_n.div(w);
    x.step = r < p.abreast ? p.abreast : 0;
    x.row = r;
    x.col = w - r * p.tiles_n;
    w -= p.abreast * p.tiles_n;
    // floor(tiles w / workers): the workers with one tile more are spread evenly (at a constant stride between the ranges their
    // stores meet in the same parts of the memory: 401408 x 384 x 96 took 82 us instead of 76)
    x.t0 = w * p.share + p.by_rest_workers.div(w * p.extra);
    x.count = x.step ? p.rounds - (r + (p.rounds - 1) * p.abreast >= p.rows) : (w + 1) * p.share + p.by_rest_workers.div((w + 1) * p.extra) - x.t0;
    return x;
}
__device__ __forceinline__ WalkItem walk_item(const GemmParams &p, const Walk &w, int i)
{
    WalkItem x;
    x.first = i == 0;
    x.last = i == w.count - 1;
    if (w.step) {
        x.col = w.col;
        x.row = w.row + i * w.step;
    } else {
        const int rows = (int)p.by_rest_rows.d;
        x.col = p.by_rest_rows.div(w.t0 + i);
        const int r = w.t0 + i - x.col * rows;
        x.first |= r == 0;
        x.last |= r == rows - 1;
        x.row = p.rest_row0 + r;
    }
    return x;
}

// ---- PTX wrappers of the tensor-core instructions (mbarrier, TMA and elect wrappers: tma.cuh) ----
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_cp_sf(uint32_t taddr, uint64_t sdesc)
{
    asm volatile("tcgen05.cp.cta_group::1.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void tc_mma_mxf4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t sfa_tmem,
                                            uint32_t sfb_tmem, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem) : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor (sm_100 format, version 1).
//   K-major operand tile, rows of 128 bytes, 128B swizzle: 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_operand_sw128(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
//   Scale chunk: 32 rows x 16 bytes, no swizzle: 8-row core matrices are 128 bytes apart.
__device__ __forceinline__ uint64_t desc_sf(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 32) | (1ull << 46);
}
// Instruction descriptor of kind::mxf4 (block scaled): E2M1 x E2M1, UE8M0 scales, K-major A and B, M = 128.
__device__ __forceinline__ uint32_t idesc_mxf4(int n, uint32_t a_sf_id, uint32_t b_sf_id)
{
    return (b_sf_id << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(kBM >> 4) << 24) |
           (a_sf_id << 29);
}

// The bias of a warp's share of a tile.  The lanes hold one accumulator row each, so every lane needs every column's value: they
// fetch it together, a bf16 pair per lane and turn, before the wait for the accumulator (bias_fetch; zero beyond N, where
// nothing is stored), put it into the warp's own line of shared memory (bias_stage), and read it back as broadcasts, 16 bytes
// at a time, for the mixed-precision add, which takes bf16 values as they are (add_bias_chunk).  50432 x 4096 x 1024, back to
// back: 99 us without a bias, 102 with it.  (When the kernel took 109 and 120 us, passing the pairs round with shuffles instead
// took 123 to 125, every lane fetching every value by itself behind the wait 160.)
template <int COLS>
__device__ __forceinline__ void bias_fetch(uint32_t (&w)[(COLS + 63) / 64], const __nv_bfloat16 *bias, int64_t col, int64_t N, int lane)
{
#pragma unroll
    for (int i = 0; i < (COLS + 63) / 64; i++) {
        const int64_t c = col + 64 * i + 2 * lane;
        w[i] = 0u;
        if (bias != nullptr && c < N) asm volatile("ld.global.u32 %0, [%1];" : "=r"(w[i]) : "l"(bias + c));
    }
}
template <int COLS>
__device__ __forceinline__ void bias_stage(const uint32_t (&w)[(COLS + 63) / 64], uint32_t line, int lane)
{
#pragma unroll
    for (int i = 0; i < (COLS + 63) / 64; i++)
        if (64 * i + 2 * lane < COLS) asm volatile("st.shared.u32 [%0], %1;" ::"r"(line + (uint32_t)(128 * i + 4 * lane)), "r"(w[i]) : "memory");
    __syncwarp();
}
__device__ __forceinline__ void add_bias_chunk(uint32_t (&r)[32], uint32_t line)
{
#pragma unroll
    for (int j = 0; j < 4; j++) {
        uint32_t b[4];
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(line + 16u * j));
#pragma unroll
        for (int t = 0; t < 4; t++)
            asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %4;\n\tadd.rn.f32.bf16 %0, l, %2;\n\tadd.rn.f32.bf16 %1, h, %3;\n\t}"
                : "=&r"(r[8 * j + 2 * t]), "=&r"(r[8 * j + 2 * t + 1]) : "r"(r[8 * j + 2 * t]), "r"(r[8 * j + 2 * t + 1]), "r"(b[t]));
    }
}
// The same without a line of shared memory (the streaming pair kernel has none to spare, and its long K loops hide it): each
// lane keeps columns 2 (l & 15) and 2 (l & 15) + 1 of a 32-column chunk, the warp passes the pairs round with shuffles.
__device__ __forceinline__ uint32_t load_bias_pair(const __nv_bfloat16 *bias, int64_t col, int64_t N, int lane)
{
    const int64_t c = col + 2 * (lane & 15);
    uint32_t v = 0u;
    if (bias != nullptr && c < N) asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(bias + c));
    return v;
}
__device__ __forceinline__ void add_bias_chunk_shfl(uint32_t (&r)[32], uint32_t pair)
{
#pragma unroll
    for (int j = 0; j < 16; j++) {
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, pair, j);
        asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %4;\n\tadd.rn.f32.bf16 %0, l, %2;\n\tadd.rn.f32.bf16 %1, h, %3;\n\t}"
            : "=&r"(r[2 * j]), "=&r"(r[2 * j + 1]) : "r"(r[2 * j]), "r"(r[2 * j + 1]), "r"(b));
    }
}

// 32 accumulator columns of one row -> 32 bf16 in 16 words
__device__ __forceinline__ void pack_row_bf16(const uint32_t (&r)[32], uint32_t (&w)[16])
{
#pragma unroll
    for (int j = 0; j < 16; j++) {
        __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
        w[j] = *reinterpret_cast<uint32_t *>(&h);
    }
}

// One row's 64 bytes into its staging line, in the 64B swizzle the TMA store expects: 16-byte chunk j of row r sits at
// chunk j ^ ((r >> 1) & 3).
__device__ __forceinline__ void stage_line(uint8_t *line, int row, const uint32_t *w /*16 words*/)
{
    const int sw = (row >> 1) & 3;
#pragma unroll
    for (int j = 0; j < 4; j++)
        *reinterpret_cast<uint4 *>(line + ((j ^ sw) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
}

// One row's 128 bytes (two 32-column chunks of bf16) into its line of a 128B-swizzled box: 16-byte piece j of row r sits
// at piece j ^ (r & 7).
__device__ __forceinline__ void stage_line_wide(uint8_t *line, int row, const uint32_t *w0 /*16 words*/, const uint32_t *w1)
{
    const int sw = row & 7;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        *reinterpret_cast<uint4 *>(line + ((j ^ sw) << 4)) = make_uint4(w0[4 * j], w0[4 * j + 1], w0[4 * j + 2], w0[4 * j + 3]);
        *reinterpret_cast<uint4 *>(line + (((j + 4) ^ sw) << 4)) = make_uint4(w1[4 * j], w1[4 * j + 1], w1[4 * j + 2], w1[4 * j + 3]);
    }
}

// ---- epilogue of one tile for one warp -----------------------------------------------------------------
// The warp owns TMEM lanes (= tile rows) row0 .. row0 + 31 and BN / 2 accumulator columns starting at `taddr`
// (global column `colbase`).  bf16: the whole share is read and packed first, the accumulator is handed back (an
// arrive on `acc_empty_bar`), then the rows go through 64B-swizzled staging buffers to TMA stores clipped at M, N.
// `map_w` (bf16 only): the same output with boxes of 64 columns and 128B swizzle; pairs of chunks then
// leave through one store instead of two (issuing a store costs its thread about 150 cycles).
// Arrive on a barrier of another CTA of the cluster (a shared::cluster address).  Used to hand an accumulator back: what
// the arrive has to order are this warp's accumulator reads, which tcgen05.wait::ld has already completed, so the default
// semantics (release at CTA scope) do; a release at cluster scope costs the arriving thread 2500-4000 cycles while the
// memory system is busy (measured), which made the epilogue the slowest role of the two-CTA kernels.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// `bias_line`: the share's bias in shared memory (bias_stage).
// REMOTE: `acc_empty_bar` is a shared::cluster address (the barrier lives in the leader of a CTA pair).
template <int BN, int BUFS, bool REMOTE = false>
__device__ __forceinline__ void epilogue_tile(const CUtensorMap *map_d, const CUtensorMap *map_w, const GemmParams &p, uint32_t taddr,
                                              int row0, int colbase, int split, uint8_t *staging, uint32_t &sbuf, int lane,
                                              uint32_t acc_empty_bar, uint32_t bias_line)
{
    constexpr int kHalfCols = BN / 2;
    constexpr int kChunks = kHalfCols / 32;
    const bool use_bias = p.bias != nullptr && p.splits == 1;
    // one staged 64-byte-wide box (32 rows) -> global
    auto store_box = [&](const uint32_t *w, int x) {
        // the store that last used this staging buffer must have finished reading it
        if (lane == 0) bulk_wait_read<BUFS - 1>();
        __syncwarp();
        uint8_t *buf = staging + sbuf * kStagingBytes;
        stage_line(buf + lane * 64, lane, w);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
            tma_store_3d(map_d, x, row0, split, smem_u32(buf));
            bulk_commit();
        }
        sbuf = (sbuf + 1) % BUFS;
    };
    auto release_acc = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            if (REMOTE) mbar_arrive_remote(acc_empty_bar);
            else mbar_arrive(acc_empty_bar);
        }
    };
    if (!p.out_fp32) {
        // bf16: read and pack the warp's whole share first, hand the accumulator back, then store
        uint32_t pk[kChunks][16];
#pragma unroll
        for (int cc = 0; cc < kChunks; cc++) {
            const int col = colbase + cc * 32;
            if (col < p.N && row0 < p.M) {     // uniform across the warp; nothing to store otherwise
                uint32_t r[32];
                tc_ld32(taddr + cc * 32, r);
                tc_wait_ld();
                if (use_bias) add_bias_chunk(r, bias_line + 64u * cc);
                pack_row_bf16(r, pk[cc]);
            }
        }
        release_acc();
        if (BUFS >= kChunks) {
            // a staging buffer per chunk: stage everything, each pair of chunks as one 128-byte-wide box (two staging buffers are
            // contiguous), make it visible once, then issue all the stores
            if (lane == 0) bulk_wait_read<0>();   // the stores of the previous tile have long been read
            __syncwarp();
#pragma unroll
            for (int cc = 0; cc < kChunks; cc += 2) {
                if (colbase + cc * 32 < p.N && row0 < p.M) {
                    if (cc + 1 < kChunks) stage_line_wide(staging + cc * kStagingBytes + lane * 128, lane, pk[cc], pk[cc + 1 < kChunks ? cc + 1 : cc]);
                    else stage_line(staging + cc * kStagingBytes + lane * 64, lane, pk[cc]);
                }
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int cc = 0; cc < kChunks; cc += 2)
                    if (colbase + cc * 32 < p.N && row0 < p.M)
                        tma_store_3d(cc + 1 < kChunks ? map_w : map_d, colbase + cc * 32, row0, split, smem_u32(staging + cc * kStagingBytes));
                bulk_commit();
            }
        } else {
#pragma unroll
            for (int cc = 0; cc < kChunks; cc++) {
                const int col = colbase + cc * 32;
                if (col < p.N && row0 < p.M) store_box(pk[cc], col);
            }
        }
    } else {
        // fp32 (dW and split-K partials: long K loops): chunk by chunk, 16 columns per box
#pragma unroll 1
        for (int cc = 0; cc < kChunks; cc++) {
            const int col = colbase + cc * 32;
            const bool live = col < p.N && row0 < p.M;
            uint32_t r[32];
            if (live) {
                tc_ld32(taddr + cc * 32, r);
                tc_wait_ld();
            }
            if (cc == kChunks - 1) release_acc();
            if (!live) continue;
            const int ncols = (int)min((int64_t)32, p.N - col);
            if (use_bias) add_bias_chunk(r, bias_line + 64u * cc);
            store_box(r, col);
            if (ncols > 16) store_box(r + 16, col + 16);
        }
    }
}

// ---- the roles that feed the tensor core (warps 0-3 of the single-CTA kernels) -------------------------------
// warp 0 / 3: TMA producers, warp 2: scale copier, warp 1: MMA issuer; C gives the shared-memory and TMEM layout.
template <class C, int BN>
__device__ __forceinline__ void gemm_feed_roles(int warp, uint32_t smem_base, uint32_t bar_full, uint32_t bar_sf_full, uint32_t bar_empty,
                                                uint32_t bar_acc_full, uint32_t bar_acc_empty, uint32_t tmem_base, volatile uint32_t *abort_flag,
                                                const CUtensorMap &map_a, const CUtensorMap &map_b, const GemmParams &p, int block,
                                                int blocks)
{
    const int items = p.tiles_m * p.tiles_n * p.splits;
    if (warp == 0 || warp == 3) {
        // ================= TMA producers =================
        // Issuing an asynchronous copy costs its thread on the order of 100 ns, and a stage needs five: warp 0 issues the
        // two operand tiles (and posts the byte count), warp 3 the scale chunks, both onto the stage's full barrier.
        {
            const bool leader = elect_one() && !p.withhold_loads;
            const bool operands = warp == 0;
            uint32_t stage = 0, phase = 0;
            bool alive = true;
            pdl_wait();
            for (int item = block; item < items && alive; item += blocks) {
                const int tile = p.by_splits.div(item), split = item - tile * p.splits;
                const int mb = p.by_tiles_n.div(tile), nb = tile - mb * p.tiles_n;
                const int kt0 = split * p.kt_per_split;
                const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
                // 128-row scale blocks of B that this tile touches (a 192-wide tile starts in the middle of one every other time)
                const int rb0 = (nb * BN) >> 7;
                int rbs = 0;
                for (int rb = 0; rb < C::kRB; rb++) rbs += (rb0 + rb) < p.rbB;
                for (int kt = kt0; kt < kt1; kt++) {
                    if (!mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                    const uint32_t sA = smem_base + stage * C::kStageBytes;
                    const uint32_t sB = sA + C::kABytes;
                    const uint32_t sSFA = sB + C::kBBytes;
                    const uint32_t sSFB = sSFA + C::kSfaBytes;
                    const uint32_t full = bar_full + 8 * stage;
                    // scale chunks present in this K tile (the last tile of an odd chunk count has one)
                    const int nch = min(2, p.nblk4 - 2 * kt);
                    if (leader && operands) {
                        mbar_expect_tx(full, (uint32_t)(C::kABytes + C::kBBytes + nch * kSfChunk * (1 + rbs)));
                        tma_load_2d(sA, &map_a, kt * kBKBytes, mb * kBM, full);
                        tma_load_2d(sB, &map_b, kt * kBKBytes, nb * BN, full);
                    }
                    if (leader && !operands) {
                        bulk_load(sSFA, p.sfa + ((size_t)mb * p.nblk4 + 2 * kt) * kSfChunk, (uint32_t)(nch * kSfChunk), full);
#pragma unroll
                        for (int rb = 0; rb < C::kRB; rb++)
                            if ((rb0 + rb) < p.rbB)
                                bulk_load(sSFB + rb * 2 * kSfChunk, p.sfb + ((size_t)(rb0 + rb) * p.nblk4 + 2 * kt) * kSfChunk,
                                          (uint32_t)(nch * kSfChunk), full);
                    }
                    __syncwarp();
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 2) {
        // ================= scale copier =================
        pdl_wait();
        // Stage s of the ring owns TMEM columns kSfCol + s * kSfSlot ..: they are free again exactly when the stage's
        // shared memory is (the producer refills it only after the MMAs that read both have completed).
        {
            const bool leader = elect_one();
            uint32_t stage = 0, phase = 0;
            bool alive = true;
            for (int item = block; item < items && alive; item += blocks) {
                const int split = p.by_splits.mod(item);
                const int kt0 = split * p.kt_per_split;
                const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
                for (int kt = kt0; kt < kt1; kt++) {
                    if (!mbar_wait_warp(bar_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sSFA = smem_base + stage * C::kStageBytes + C::kABytes + C::kBBytes;
                    const uint32_t sSFB = sSFA + C::kSfaBytes;
                    const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8;
                    const int64_t kleft = p.Kc - (int64_t)kt * kBKElems;
                    const int nch = kleft > 128 ? 2 : 1;
                    if (leader) {
#pragma unroll
                        for (int c = 0; c < 2; c++) {
                            if (c < nch) {
                                tc_cp_sf(t_sfa + 4 * c, desc_sf(sSFA + c * kSfChunk));
#pragma unroll
                                for (int rb = 0; rb < C::kRB; rb++)
                                    tc_cp_sf(t_sfb + 4 * C::kRB * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
                            }
                        }
                        tc_commit(bar_sf_full + 8 * stage);   // arrives once the copies have landed in TMEM
                    }
                    __syncwarp();
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        pdl_wait();
        // This warp's loop is the serial chain that bounds short and medium K loops (with every load, copy and store
        // taken out the kernel ran no faster), so it is kept short: one wait per stage (the scale copier has seen the
        // operands land before its copies, and its commit orders them before this warp's MMAs), and the barrier of the
        // NEXT stage is tested before this stage's MMAs are issued, so that the answer is there when it is needed.
        {
            const bool leader = elect_one();
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            const int nmma_last = (int)((p.Kc - (int64_t)(p.kt_total - 1) * kBKElems + 63) / 64);   // MMAs of the last K tile
            bool ready = false;   // the current stage's scales (hence operands) are known to be in place
            bool alive = true;
            for (int item = block; item < items && alive; item += blocks) {
                const int tile = p.by_splits.div(item), split = item - tile * p.splits;
                const int nb = p.by_tiles_n.mod(tile);
                const int kt0 = split * p.kt_per_split;
                const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
                // scale columns hold 32 rows each: a tile that starts 64 rows into a 128-row block starts 2 columns in
                const uint32_t sfb_shift = (uint32_t)(((nb * BN) & 127) >> 5);
                if (!mbar_wait_warp(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                const uint32_t d_tmem = tmem_base + acc * BN;
                for (int kt = kt0; kt < kt1; kt++) {
                    if (!ready && !mbar_wait_warp(bar_sf_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sA = smem_base + stage * C::kStageBytes;
                    const uint32_t sB = sA + C::kABytes;
                    const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8 + sfb_shift;
                    const int nmma = kt == p.kt_total - 1 ? nmma_last : 4;
                    const uint64_t adesc = desc_operand_sw128(sA), bdesc = desc_operand_sw128(sB);
                    const uint32_t cur = stage;
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                    ready = __all_sync(0xFFFFFFFFu, mbar_test_wait(bar_sf_full + 8 * stage, phase));
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < 4; k++) {
                            if (k < nmma) {
                                const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                                tc_mma_mxf4(d_tmem, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                            idesc_mxf4(BN, sf_id, sf_id), t_sfa + 4 * (k >> 1), t_sfb + 4 * C::kRB * (k >> 1),
                                            (kt > kt0 || k > 0) ? 1u : 0u);
                            }
                        }
                        tc_commit(bar_empty + 8 * cur);   // frees the stage (shared memory and scale columns) once these MMAs have read it
                    }
                }
                if (alive && leader) tc_commit(bar_acc_full + 8 * acc);  // accumulator complete
                __syncwarp();
                if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
            }
        }
    }
}

// ---- the kernel ------------------------------------------------------------------------------------
template <int BN, class Job2>   // Job2 = GemmJob: the blocks behind those of the first product's tiles make a second one; NoJob: there is none
__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4(const __grid_constant__ GemmJob one, const __grid_constant__ Job2 two)
{
    using C = GemmCfg<BN>;
    constexpr bool kTwo = sizeof(Job2) == sizeof(GemmJob);
    const int blocks1 = one.p.tiles_m * one.p.tiles_n;
    const bool second = kTwo && (int)blockIdx.x >= blocks1;
    const GemmJob &job = second ? reinterpret_cast<const GemmJob &>(two) : one;
    const GemmParams &p = job.p;
    const int block = (int)blockIdx.x - (second ? blocks1 : 0), blocks = !kTwo ? (int)gridDim.x : second ? (int)gridDim.x - blocks1 : blocks1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    // barrier slots: full[kStages], sf_full[kStages], empty[kStages], acc_full[kAccStages], acc_empty[kAccStages]
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_full + 8 * C::kStages;
    const uint32_t bar_empty = bar_sf_full + 8 * C::kStages;
    const uint32_t bar_acc_full = bar_empty + 8 * C::kStages;
    const uint32_t bar_acc_empty = bar_acc_full + 8 * C::kAccStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * C::kStages + 2 * C::kAccStages);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);

    if (threadIdx.x == 32 * 3) { prefetch_map(&job.a); prefetch_map(&job.b); prefetch_map(&job.d); prefetch_map(&job.dw); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; s++) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < C::kAccStages; a++) {
            mbar_init(bar_acc_full + 8 * a, 1);
            mbar_init(bar_acc_empty + 8 * a, kEpiWarps);
        }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const int items = p.tiles_m * p.tiles_n * p.splits;

    if (warp < kEpiWarp0) {
        gemm_feed_roles<C, BN>(warp, smem_base, bar_full, bar_sf_full, bar_empty, bar_acc_full, bar_acc_empty, tmem_base, abort_flag, job.a, job.b, p, block, blocks);
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue (warps 4..11) =================
        pdl_wait();
        const int ew = warp - kEpiWarp0;
        const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31 are the ones this warp may read
        const int chalf = ew >> 2;               // which half of the tile's columns this warp stores
        uint8_t *staging = smem + C::kStagingOff + ew * C::kStagingBufs * kStagingBytes;
        const uint32_t bias_line = smem_base + C::kBiasOff + ew * (BN / 2) * 2;
        uint32_t sbuf = 0;                       // staging buffer of the next box (round robin)
        constexpr int kHalfCols = BN / 2;
        constexpr int kChunks = kHalfCols / 32;
        uint32_t acc = 0, acc_phase = 0;
        bool alive = true;
        for (int item = block; item < items && alive; item += blocks) {
            const int tile = p.by_splits.div(item), split = item - tile * p.splits;
            const int mb = p.by_tiles_n.div(tile), nb = tile - mb * p.tiles_n;
            uint32_t bias[(kHalfCols + 63) / 64];
            bias_fetch<kHalfCols>(bias, p.bias, (int64_t)nb * BN + chalf * kHalfCols, p.N, lane);
            if (!mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
            tc_fence_after();
            const int row0 = mb * kBM + quarter * 32;
            const int colbase = nb * BN + chalf * kHalfCols;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + chalf * kHalfCols;
            if (p.bias != nullptr) bias_stage<kHalfCols>(bias, bias_line, lane);
            epilogue_tile<BN, C::kStagingBufs>(&job.d, &job.dw, p, taddr, row0, colbase, split, staging, sbuf, lane,
                                               bar_acc_empty + 8 * acc, bias_line);
            if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) bulk_wait_read<0>();   // the stores of this warp have read their staging buffers: the shared memory may go
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// ---- the quantizing kernel ------------------------------------------------------------------------------
// The product with the NEXT quantization fused into its epilogue (Sec. 3.3: every product's result is quantized again
// before the next product reads it).  Tiles are 128 x 128, exactly one tile of the two-axis quantizer: the epilogue
// warps cast their part of the accumulator (+ bias) to bf16 (Y), apply an elementwise hook (identity, GELU, or a
// multiplication by a caller's bf16 tensor: the derivative of an activation on the way back), round to bf16 again
// (Z) and lay Z down in shared memory in the layout the quantizer's passes read; Z can leave through TMA stores, Y
// through plain stores.  Then the same 256 threads run the row pass (codes of Z with groups along N, the forward /
// gradient operand of the next product) and the column pass (groups along M, stored transposed; with DQ it
// re-quantizes the dequantized result of the row pass: double quantization).  The results are bit for bit those of the
// stand-alone quantizers applied to Z.  Two accumulators: the next tile's K loop runs during this long epilogue, and a second group
// of epilogue warps may take every other tile (two_groups).
// GROUPS = 2: two groups of eight epilogue warps take the tiles in turn, each with an accumulator, tiles and staging of its own, on a
// ring of two stages.  TILES: 32 KB tiles per group: Z, and one each for the hook's second factor or the dequantized row codes beside
// a Z that is stored, and for a Y that is stored beside a Z that differs from it.
template <int GROUPS, int TILES>
struct GemmQCfg {
    static constexpr int BN = 128;
    static constexpr int kRB = 1;
    static constexpr int kABytes = kBM * kBKBytes;
    static constexpr int kBBytes = BN * kBKBytes;
    static constexpr int kSfaBytes = 2 * kSfChunk;
    static constexpr int kSfbBytes = 2 * kSfChunk;
    static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;   // 34 KB
    static constexpr int kStages = GROUPS == 2 ? 2 : TILES == 3 ? 3 : 4;
    static constexpr int kAccStages = 2;
    static constexpr int kSfCol = kAccStages * BN;
    static constexpr int kSfSlot = 16;
    static constexpr int kTmemCols = 512;
    static constexpr int kThreads = 32 * (kEpiWarp0 + GROUPS * kEpiWarps);
    static constexpr int kTileOff = kStages * kStageBytes;           // per group: TILES tiles
    static constexpr int kStagingOff = kTileOff + GROUPS * TILES * kTileBytes;   // transposed codes 8 KB + two scale chunks: two for one group, else one per group
    static constexpr int kStagingBytes = kTile * 64 + 1024;
    static constexpr int kBarOff = kStagingOff + 2 * kStagingBytes;
    static constexpr int kBiasOff = kBarOff + 256;                   // a line of 64 bf16 per epilogue warp
    static constexpr int kSmemBytes = kBiasOff + GROUPS * kEpiWarps * 128 + 1024 /*align*/;
    static_assert(kSfCol + kStages * kSfSlot <= 512, "TMEM budget");
    static_assert(kStageBytes % 1024 == 0 && kStagingBytes % 1024 == 0, "alignment");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

struct QuantEpilogue {
    QuantSide rw, tr;             // row-wise result [M, N] and transposed result [N, M]
    int emit_row, emit_t;
    int hook;                     // MXFP4_HOOK_*
    const __nv_bfloat16 *aux;     // hook = multiply: bf16 [M, N]
    int64_t ld_aux;
    int store_y;                  // the bf16 result before the hook leaves through map_y
    int store_z;                  // the bf16 tile that is quantized leaves through map_z
    int aux_tma;                  // the hook's second factor arrives through map_aux (otherwise per-thread loads)
};

// named barriers of the 256 threads of an epilogue group (barrier 0 belongs to __syncthreads)
__device__ __forceinline__ void epi_sync(int id) { asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory"); }
__device__ __forceinline__ bool epi_any(int id, bool x)
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, %2, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r) : "r"((uint32_t)x), "r"(id) : "memory");
    return r != 0;
}

template <bool SR_ROW, bool SR_T, bool DQ, bool WITH_Y, int GROUPS>
__global__ void __launch_bounds__(32 * (kEpiWarp0 + GROUPS * kEpiWarps), 1)
k_gemm_mxf4_q(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
              const __grid_constant__ CUtensorMap map_y, const __grid_constant__ CUtensorMap map_z, const __grid_constant__ CUtensorMap map_aux,
              const __grid_constant__ CUtensorMap map_t, const GemmParams p, const __grid_constant__ QuantEpilogue e)
{
    constexpr int kTiles = WITH_Y && GROUPS == 1 ? 3 : 2;
    using C = GemmQCfg<GROUPS, kTiles>;
    constexpr int BN = C::BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_full + 8 * C::kStages;
    const uint32_t bar_empty = bar_sf_full + 8 * C::kStages;
    const uint32_t bar_acc_full = bar_empty + 8 * C::kStages;
    const uint32_t bar_acc_empty = bar_acc_full + 8 * C::kAccStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * C::kStages + 2 * C::kAccStages);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const uint32_t bar_aux0 = smem_u32(bars + 3 * C::kStages + 2 * C::kAccStages + 1);   // per group: the hook's second factor has landed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);

    if (threadIdx.x == 32 * 3) { prefetch_map(&map_a); prefetch_map(&map_b); prefetch_map(&map_z); prefetch_map(&map_t); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; s++) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < C::kAccStages; a++) {
            mbar_init(bar_acc_full + 8 * a, 1);
            mbar_init(bar_acc_empty + 8 * a, kEpiWarps);
        }
        for (int g = 0; g < GROUPS; g++) mbar_init(bar_aux0 + 8 * g, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp < kEpiWarp0) {
        gemm_feed_roles<C, BN>(warp, smem_base, bar_full, bar_sf_full, bar_empty, bar_acc_full, bar_acc_empty, tmem_base, abort_flag, map_a, map_b, p, blockIdx.x,
                               gridDim.x);
    } else {
        // ================= quantizing epilogue (warps 4..11, and 12..19 of a second group: 256 threads each) =================
        pdl_wait();
        const int group = GROUPS == 1 ? 0 : (warp - kEpiWarp0) / kEpiWarps, sync_id = 1 + group;
        const int et = (int)threadIdx.x - 32 * (kEpiWarp0 + group * kEpiWarps);
        const int quarter = warp & 3, chalf = GROUPS == 1 ? (warp - kEpiWarp0) >> 2 : et >> 7;
        const uint32_t bar_aux = bar_aux0 + 8 * group;
        const int M = (int)p.M, N = (int)p.N;
        const QsGeom g = qs_geom(et, M, N, e.rw.packed);
        const uint32_t tfa_r2 = tf_add_of(e.rw.scale_mode) * 0x00010001u, tfa_t2 = tf_add_of(e.tr.scale_mode) * 0x00010001u;
        const uint32_t t_base = smem_base + C::kTileOff + group * kTiles * kTileBytes, t2_base = t_base + kTileBytes, ty_base = t_base + (kTiles - 1) * kTileBytes;
        const uint32_t dq_base = GROUPS == 1 || e.store_z ? t2_base : t_base;   // a Z that is stored keeps its tile until it has left
        const int trow = quarter * 32 + lane;                        // this thread's row of the tile
        const uint32_t row_off = (uint32_t)(chalf * (kTileBytes / 2) + trow * 128);
        const uint32_t t_row = t_base + row_off;
        // the hook's second factor travels by TMA into the second tile one tile ahead (that tile is free unless DQ uses it)
        const bool aux_tma = e.hook == MXFP4_HOOK_MULTIPLY && e.aux_tma && !DQ;
        auto issue_aux = [&](int item) {
            const int mb = p.by_tiles_n.div(item), nb = item - mb * p.tiles_n;
            mbar_expect_tx(bar_aux, kTileBytes);
            tma_load_2d(t2_base, &map_aux, nb * BN, mb * kBM, bar_aux);
            tma_load_2d(t2_base + kTileBytes / 2, &map_aux, nb * BN + 64, mb * kBM, bar_aux);
        };
        const int items = p.tiles_m * p.tiles_n, step = GROUPS * (int)gridDim.x, item0 = (int)blockIdx.x + group * (int)gridDim.x;
        if (aux_tma && et == 0 && !p.withhold_loads && item0 < items) issue_aux(item0);
        const bool use_bias = p.bias != nullptr;
        const uint32_t bias_line = smem_base + C::kBiasOff + (warp - kEpiWarp0) * 128;
        uint32_t nonfinite = 0;
        int it = 0;            // turn of the group; the block's tiles take the accumulators in turn
        for (int item = item0; item < items; item += step, it++) {
            const uint32_t acc = GROUPS == 1 ? it & 1 : group, acc_phase = GROUPS == 1 ? (it >> 1) & 1 : it & 1;
            const int mb = p.by_tiles_n.div(item), nb = item - mb * p.tiles_n;
            const int row0 = mb * kBM, col0 = nb * BN;
            uint32_t bias[1];
            bias_fetch<64>(bias, p.bias, col0 + chalf * 64, N, lane);
            bool ok = mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag, p.dev_status, p.spin_limit);
            if (aux_tma) ok = mbar_wait(bar_aux, (uint32_t)it & 1u, abort_flag, p.dev_status, p.spin_limit) && ok;
            if (GROUPS == 2 && et == 0) bulk_wait_read<0>();   // the codes of the group's last tile have left its staging tile
            if (epi_any(sync_id, !ok)) break;      // a wait ran out in one of the eight warps: all of them leave together
            tc_fence_after();
            if (use_bias) bias_stage<64>(bias, bias_line, lane);
            uint8_t *staging = smem + C::kStagingOff + (GROUPS == 1 ? it & 1 : group) * C::kStagingBytes;
            uint8_t *s_sc_row = staging + kTile * 64, *s_sc_t = s_sc_row + 512;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + chalf * 64;
            const int grow = row0 + trow;

            // ---- accumulator -> Y (bf16) -> hook -> Z (bf16) -> the tile in shared memory ----
            // One group has this code once per hook: beside the packed multiplication a common one took 1-4 % longer than before it where
            // there is no hook (25216 x 1536 x 1024, Q3 + Q5 48.1, 49.9 us, so 45.4); with the 96 registers of two groups that would spill.
            const auto fill = [&](auto hook) {
#pragma unroll
                for (int cc = 0; cc < 2; cc++) {
                    const int col = col0 + chalf * 64 + cc * 32;
                    const bool live = grow < M && col < N;     // N is a multiple of 32: a chunk is inside the matrix or outside it
                    uint32_t r[32];
                    tc_ld32(taddr + cc * 32, r);
                    tc_wait_ld();
                    if (cc == 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_acc_empty + 8 * acc);   // the accumulator goes back to the MMA issuer
                    }
                    if (use_bias) add_bias_chunk(r, bias_line + 64u * cc);
                    uint32_t yw[16];
                    pack_row_bf16(r, yw);
                    if (WITH_Y && e.store_y) {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            asm volatile("st.shared.v4.u32 [%4], {%0,%1,%2,%3};" ::"r"(yw[4 * j]), "r"(yw[4 * j + 1]), "r"(yw[4 * j + 2]), "r"(yw[4 * j + 3]),
                                         "r"(ty_base + row_off + (uint32_t)((((cc * 4 + j) ^ (trow & 7))) << 4)) : "memory");
                    }
                    if (hook != MXFP4_HOOK_IDENTITY) {
                        if (hook == MXFP4_HOOK_GELU) {
#pragma unroll
                            for (int j = 0; j < 16; j++) yw[j] = gelu_bf16x2(yw[j]);
                        } else {
                            uint4 aw[4] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
                            if (aux_tma) {
#pragma unroll
                                for (int j = 0; j < 4; j++)
                                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(aw[j].x), "=r"(aw[j].y), "=r"(aw[j].z), "=r"(aw[j].w)
                                                 : "r"(t2_base + row_off + (uint32_t)((((cc * 4 + j) ^ (trow & 7))) << 4)));
                            } else if (live) {
                                const uint4 *ap = reinterpret_cast<const uint4 *>(e.aux + (int64_t)grow * e.ld_aux + col);
#pragma unroll
                                for (int j = 0; j < 4; j++) aw[j] = ld_stream_16(ap + j);
                            }
                            const uint32_t *a32 = reinterpret_cast<const uint32_t *>(aw);
#pragma unroll
                            for (int j = 0; j < 16; j++) yw[j] = mul_bf16x2(yw[j], a32[j]);   // one rounding, as of the FP32 product, which is exact
                        }
                    }
                    if (!live) {
#pragma unroll
                        for (int j = 0; j < 16; j++) yw[j] = 0u;   // outside the matrix the tile holds zeros, as a TMA load would leave them
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        asm volatile("st.shared.v4.u32 [%4], {%0,%1,%2,%3};" ::"r"(yw[4 * j]), "r"(yw[4 * j + 1]), "r"(yw[4 * j + 2]), "r"(yw[4 * j + 3]),
                                     "r"(t_row + (uint32_t)((((cc * 4 + j) ^ (trow & 7))) << 4)) : "memory");
                }
            };
            if (GROUPS == 2) fill(e.hook);
            else if (e.hook == MXFP4_HOOK_IDENTITY) fill(std::integral_constant<int, MXFP4_HOOK_IDENTITY>());
            else if (e.hook == MXFP4_HOOK_GELU) fill(std::integral_constant<int, MXFP4_HOOK_GELU>());
            else fill(std::integral_constant<int, MXFP4_HOOK_MULTIPLY>());
            fence_async_smem();
            epi_sync(sync_id);                            // the tile is complete, the second factor has been read
            if (et == 0) {
                if (e.store_z) {
                    tma_store_2d(&map_z, col0, row0, t_base);
                    tma_store_2d(&map_z, col0 + 64, row0, t_base + kTileBytes / 2);
                }
                if (WITH_Y && e.store_y) {
                    tma_store_2d(&map_y, col0, row0, ty_base);
                    tma_store_2d(&map_y, col0 + 64, row0, ty_base + kTileBytes / 2);
                }
                bulk_commit();
                if (aux_tma && item + step < items) issue_aux(item + step);
            }
            qs_tile<SR_ROW, SR_T, DQ>(g, t_base, dq_base, row0, col0, M, N, e.emit_row, e.emit_t, e.rw, e.tr, tfa_r2, tfa_t2, staging, s_sc_row, s_sc_t,
                                      nonfinite);
            fence_async_smem();
            if (et == 0) bulk_wait_read<0>();             // Z has left the tile, the previous tile's codes their staging buffer
            epi_sync(sync_id);
            if (et == 0) {
                if (e.emit_t) {
                    tma_store_2d(&map_t, row0 >> 1, col0, smem_u32(staging));
                    bulk_store(e.tr.scales + ((size_t)(col0 >> 7) * e.tr.nblk4 + (row0 >> 7)) * 512, smem_u32(s_sc_t), 512);
                }
                if (e.emit_row) bulk_store(e.rw.scales + ((size_t)(row0 >> 7) * e.rw.nblk4 + (col0 >> 7)) * 512, smem_u32(s_sc_row), 512);
                bulk_commit();
            }
        }
        if (et == 0) bulk_wait_read<0>();
        if (nonfinite && p.dev_status) atomicOr(p.dev_status, MXFP4_DEV_NONFINITE);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// ---- the B-stationary kernel --------------------------------------------------------------------------
// For contraction lengths of a few K tiles (the forward and input-gradient products of the layers: Kc = 384 .. 1536)
// the ring of the kernel above carries, per stage, a B tile that the CTA has loaded many times before, and its rate
// is ring bytes in flight over load latency.  Here a CTA walks DOWN a column of tiles (see Walk): the whole B block of the
// column (BN rows x Kc, with its scales in TMEM) stays resident, and the ring carries A alone, so that the same
// shared memory holds two to three times as many tiles in flight.
template <int BN, int KT, int AS>   // KT: K tiles the resident B block can hold; AS: stages of the A ring
struct GemmBsCfg {
    static constexpr int kRB = (BN + 127) / 128;
    static constexpr int kABytes = kBM * kBKBytes;             // 16 KB
    static constexpr int kBBytes = BN * kBKBytes;              // one K tile of the B block
    static constexpr int kSfaBytes = 2 * kSfChunk;
    static constexpr int kSfbBytes = 2 * kSfChunk * kRB;       // per K tile
    static constexpr int kStagingBufs = BN / 64;
    static constexpr int kAOff = KT * kBBytes;
    static constexpr int kSfbOff = kAOff + AS * kABytes;
    static constexpr int kSfaOff = kSfbOff + KT * kSfbBytes;
    static constexpr int kStagingOff = kSfaOff + AS * kSfaBytes;
    static constexpr int kBarOff = kStagingOff + kEpiWarps * kStagingBufs * kStagingBytes;
    static constexpr int kBiasOff = kBarOff + 256;             // a line of BN / 2 bf16 per epilogue warp
    static constexpr int kSmemBytes = kBiasOff + kEpiWarps * BN + 1024 /*align*/;
    static constexpr int kSfbCol = 2 * BN;                     // TMEM columns: two accumulators, resident SFB (8 kRB per K tile), SFA ring (8 per stage)
    static constexpr int kSfaCol = kSfbCol + KT * 8 * kRB;
    static constexpr int kTmemCols = 512;
    static_assert(kSfaCol + AS * 8 <= 512, "TMEM budget");
    static_assert(kStagingOff % 1024 == 0, "staging alignment");
    static_assert(3 * AS + 7 <= 30, "barrier slots");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

template <int BN, int KT, int AS>
__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4_bs(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
               const __grid_constant__ CUtensorMap map_d, const __grid_constant__ CUtensorMap map_dw, const GemmParams p)
{
    using C = GemmBsCfg<BN, KT, AS>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    // barrier slots: a_full[AS], sf_full[AS], a_empty[AS], acc_full[2], acc_empty[2], b_full, b_sf_full, b_empty
    const uint32_t bar_a_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_a_full + 8 * AS;
    const uint32_t bar_a_empty = bar_sf_full + 8 * AS;
    const uint32_t bar_acc_full = bar_a_empty + 8 * AS;
    const uint32_t bar_acc_empty = bar_acc_full + 16;
    const uint32_t bar_b_full = bar_acc_empty + 16;
    const uint32_t bar_b_sf_full = bar_b_full + 8;
    const uint32_t bar_b_empty = bar_b_sf_full + 8;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * AS + 7);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);

    if (threadIdx.x == 32 * 3) { prefetch_map(&map_a); prefetch_map(&map_b); prefetch_map(&map_d); prefetch_map(&map_dw); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < AS; s++) {
            mbar_init(bar_a_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_a_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(bar_acc_full + 8 * a, 1);
            mbar_init(bar_acc_empty + 8 * a, kEpiWarps);
        }
        mbar_init(bar_b_full, 1);
        mbar_init(bar_b_sf_full, 1);
        mbar_init(bar_b_empty, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const Walk walk = walk_begin(p, blockIdx.x);
    const int ktn = p.kt_total;

    if (warp == 0) {
        // ================= A producer: one A tile and its scales per stage =================
        const bool leader = elect_one() && !p.withhold_loads;
        uint32_t stage = 0, phase = 0;
        bool alive = true;
        pdl_wait();
        for (int i = 0; i < walk.count && alive; i++) {
            const int mb = walk_item(p, walk, i).row;
            for (int kt = 0; kt < ktn; kt++) {
                if (!mbar_wait_warp(bar_a_empty + 8 * stage, phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                const int nch = min(2, p.nblk4 - 2 * kt);
                if (leader) {
                    const uint32_t full = bar_a_full + 8 * stage;
                    mbar_expect_tx(full, (uint32_t)(C::kABytes + nch * kSfChunk));
                    tma_load_2d(smem_base + C::kAOff + stage * C::kABytes, &map_a, kt * kBKBytes, mb * kBM, full);
                    bulk_load(smem_base + C::kSfaOff + stage * C::kSfaBytes, p.sfa + ((size_t)mb * p.nblk4 + 2 * kt) * kSfChunk,
                              (uint32_t)(nch * kSfChunk), full);
                }
                __syncwarp();
                if (++stage == AS) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 3) {
        // ================= B producer: the block of a column, once per run of tiles in that column =================
        const bool leader = elect_one() && !p.withhold_loads;
        uint32_t runs = 0;
        pdl_wait();
        for (int i = 0; i < walk.count; i++) {
            const WalkItem x = walk_item(p, walk, i);
            if (!x.first) continue;
            const int nb = x.col;
            // the MMAs of the previous column have finished reading the block
            if (runs > 0 && !mbar_wait_warp(bar_b_empty, (runs - 1u) & 1u, abort_flag, p.dev_status, p.spin_limit)) break;
            const int rb0 = (nb * BN) >> 7;
            int rbs = 0;
            for (int rb = 0; rb < C::kRB; rb++) rbs += (rb0 + rb) < p.rbB;
            if (leader) {
                mbar_expect_tx(bar_b_full, (uint32_t)(ktn * C::kBBytes + p.nblk4 * kSfChunk * rbs));
                for (int kt = 0; kt < ktn; kt++) {
                    const int nch = min(2, p.nblk4 - 2 * kt);
                    tma_load_2d(smem_base + kt * C::kBBytes, &map_b, kt * kBKBytes, nb * BN, bar_b_full);
#pragma unroll
                    for (int rb = 0; rb < C::kRB; rb++)
                        if ((rb0 + rb) < p.rbB)
                            bulk_load(smem_base + C::kSfbOff + kt * C::kSfbBytes + rb * 2 * kSfChunk,
                                      p.sfb + ((size_t)(rb0 + rb) * p.nblk4 + 2 * kt) * kSfChunk, (uint32_t)(nch * kSfChunk), bar_b_full);
                }
            }
            __syncwarp();
            runs++;
            if (walk.step) break;   // its only run
        }
    } else if (warp == 2) {
        // ================= scale copier: B scales once per column, A scales per stage =================
        pdl_wait();
        const bool leader = elect_one();
        uint32_t stage = 0, phase = 0, runs = 0;
        bool alive = true;
        for (int i = 0; i < walk.count && alive; i++) {
            if (walk_item(p, walk, i).first) {
                if (!mbar_wait_warp(bar_b_full, runs & 1u, abort_flag, p.dev_status, p.spin_limit)) break;
                tc_fence_after();
                if (leader) {
                    for (int kt = 0; kt < ktn; kt++) {
                        const int nch = min(2, p.nblk4 - 2 * kt);
                        const uint32_t sSFB = smem_base + C::kSfbOff + kt * C::kSfbBytes;
                        const uint32_t t_sfb = tmem_base + C::kSfbCol + kt * 8 * C::kRB;
                        for (int c = 0; c < nch; c++)
#pragma unroll
                            for (int rb = 0; rb < C::kRB; rb++)
                                tc_cp_sf(t_sfb + 4 * C::kRB * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
                    }
                    tc_commit(bar_b_sf_full);
                }
                __syncwarp();
                runs++;
            }
            for (int kt = 0; kt < ktn; kt++) {
                if (!mbar_wait_warp(bar_a_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                tc_fence_after();
                const uint32_t sSFA = smem_base + C::kSfaOff + stage * C::kSfaBytes;
                const uint32_t t_sfa = tmem_base + C::kSfaCol + stage * 8;
                const int nch = min(2, p.nblk4 - 2 * kt);
                if (leader) {
                    tc_cp_sf(t_sfa, desc_sf(sSFA));
                    if (nch > 1) tc_cp_sf(t_sfa + 4, desc_sf(sSFA + kSfChunk));
                    tc_commit(bar_sf_full + 8 * stage);   // arrives once the copies have landed in TMEM
                }
                __syncwarp();
                if (++stage == AS) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        pdl_wait();
        const bool leader = elect_one();
        uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0, runs = 0;
        const int nmma_last = (int)((p.Kc - (int64_t)(ktn - 1) * kBKElems + 63) / 64);   // MMAs of the last K tile
        bool ready = false;
        bool alive = true;
        for (int i = 0; i < walk.count && alive; i++) {
            const WalkItem x = walk_item(p, walk, i);
            const int nb = x.col;
            if (x.first) {
                // the block of this column and its scales are in place (the copier saw the block land before it copied)
                if (!mbar_wait_warp(bar_b_sf_full, runs & 1u, abort_flag, p.dev_status, p.spin_limit)) break;
                runs++;
            }
            const uint32_t sfb_shift = (uint32_t)(((nb * BN) & 127) >> 5);
            if (!mbar_wait_warp(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) break;
            const uint32_t d_tmem = tmem_base + acc * BN;
            for (int kt = 0; kt < ktn; kt++) {
                if (!ready && !mbar_wait_warp(bar_sf_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                tc_fence_after();
                const uint64_t adesc = desc_operand_sw128(smem_base + C::kAOff + stage * C::kABytes);
                const uint64_t bdesc = desc_operand_sw128(smem_base + kt * C::kBBytes);
                const uint32_t t_sfa = tmem_base + C::kSfaCol + stage * 8;
                const uint32_t t_sfb = tmem_base + C::kSfbCol + kt * 8 * C::kRB + sfb_shift;
                const int nmma = kt == ktn - 1 ? nmma_last : 4;
                const uint32_t cur = stage;
                if (++stage == AS) { stage = 0; phase ^= 1u; }
                ready = __all_sync(0xFFFFFFFFu, mbar_test_wait(bar_sf_full + 8 * stage, phase));
                if (leader) {
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        if (k < nmma) {
                            const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                            tc_mma_mxf4(d_tmem, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                        idesc_mxf4(BN, sf_id, sf_id), t_sfa + 4 * (k >> 1), t_sfb + 4 * C::kRB * (k >> 1),
                                        (kt > 0 || k > 0) ? 1u : 0u);
                        }
                    }
                    tc_commit(bar_a_empty + 8 * cur);   // frees the A stage and its scale columns once these MMAs have read them
                }
            }
            if (alive && leader) {
                tc_commit(bar_acc_full + 8 * acc);            // accumulator complete
                if (x.last) tc_commit(bar_b_empty);           // and the resident block may be replaced
            }
            __syncwarp();
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue (warps 4..11) =================
        pdl_wait();
        const int ew = warp - kEpiWarp0;
        const int quarter = warp & 3;
        const int chalf = ew >> 2;
        uint8_t *staging = smem + C::kStagingOff + ew * C::kStagingBufs * kStagingBytes;
        const uint32_t bias_line = smem_base + C::kBiasOff + ew * (BN / 2) * 2;
        uint32_t sbuf = 0;
        constexpr int kHalfCols = BN / 2;
        uint32_t acc = 0, acc_phase = 0;
        for (int i = 0; i < walk.count; i++) {
            const WalkItem x = walk_item(p, walk, i);
            const int nb = x.col, mb = x.row;
            uint32_t bias[(kHalfCols + 63) / 64];
            bias_fetch<kHalfCols>(bias, p.bias, (int64_t)nb * BN + chalf * kHalfCols, p.N, lane);
            if (!mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag, p.dev_status, p.spin_limit)) break;
            tc_fence_after();
            const int row0 = mb * kBM + quarter * 32;
            const int colbase = nb * BN + chalf * kHalfCols;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + chalf * kHalfCols;
            if (p.bias != nullptr) bias_stage<kHalfCols>(bias, bias_line, lane);
            epilogue_tile<BN, C::kStagingBufs>(&map_d, &map_dw, p, taddr, row0, colbase, 0, staging, sbuf, lane,
                                               bar_acc_empty + 8 * acc, bias_line);
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) bulk_wait_read<0>();   // the stores of this warp have read their staging buffers: the shared memory may go
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// ---- the cluster split-K kernel -----------------------------------------------------------------------
// Weight-gradient products have a small output and a very long contraction: too few tiles for the machine.  Here the
// S CTAs of a thread-block cluster share ONE 128 x 192 tile, each taking 1/S of the contraction into its own
// accumulator, and the partial sums meet in distributed shared memory instead of in global memory: every CTA owns the
// 32-column chunks c with c mod S = its rank, receives those chunks from all S CTAs (its own included) into the shared
// memory its operand ring occupied, adds them in rank order (a fixed order: the result does not depend on timing)
// and stores the finished chunk.  No workspace, no second kernel.
//   barrier 1: every CTA's ring is idle (its MMAs have completed), so peers may write into it
//   barrier 2: all partial sums have arrived (release / acquire over the cluster)
// The tensor core adds into its FP32 accumulator with truncation, so the error of a sum grows with the number of MMAs
// chained into one accumulator.  A CTA here has a long chain (half of a long contraction), so it keeps TWO accumulators,
// one for its even and one for its odd K tiles, and adds them when it reads them out: the chains are as short as with
// four partial sums.
struct GemmCkCfg {
    static constexpr int BN = 192;
    static constexpr int kRB = 2;
    static constexpr int kABytes = kBM * kBKBytes;
    static constexpr int kBBytes = BN * kBKBytes;
    static constexpr int kSfaBytes = 2 * kSfChunk;
    static constexpr int kSfbBytes = 2 * kSfChunk * kRB;
    static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;   // 43 KB
    static constexpr int kStages = 5;
    static constexpr int kSfCol = 2 * BN;                               // TMEM: two accumulators (even / odd K tiles), then SFA (8) + SFB (16) per stage
    static constexpr int kSfSlot = 8 + 8 * kRB;
    static constexpr int kTmemCols = 512;
    static constexpr int kChunks = BN / 32;                             // 6: the cluster size divides it
    static constexpr int kChunkBytes = kBM * 32 * 4;                    // one 128 x 32 FP32 chunk: 16 KB
    static constexpr int kBarOff = kStages * kStageBytes;
    static constexpr int kSmemBytes = kBarOff + 1024 /*align*/ + 256 /*barriers*/;
    static_assert(kSfCol + kStages * kSfSlot <= 512, "TMEM budget");
    static_assert(kChunks * kChunkBytes <= kStages * kStageBytes, "the received chunks fit where the ring was");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

__device__ __forceinline__ uint32_t ck_cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t ck_cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void ck_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of `local` (a shared::cta address) in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t ck_map(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void ck_store_remote(uint32_t addr, float a, float b, float c, float d)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4_ck(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, const GemmParams p)
{
    using C = GemmCkCfg;
    constexpr int BN = C::BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_full + 8 * C::kStages;
    const uint32_t bar_empty = bar_sf_full + 8 * C::kStages;
    const uint32_t bar_acc_full = bar_empty + 8 * C::kStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * C::kStages + 1);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t rank = ck_cluster_rank(), S = ck_cluster_size();

    if (threadIdx.x == 32 * 3) { prefetch_map(&map_a); prefetch_map(&map_b); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; s++) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        mbar_init(bar_acc_full, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();

    // the cluster's tile and this CTA's part of the contraction
    const int tile = (int)(blockIdx.x / S);
    const int mb = tile / p.tiles_n, nb = tile % p.tiles_n;
    const int kt0 = min((int)rank * p.kt_per_split, p.kt_total);
    const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
    const int rb0 = (nb * BN) >> 7;

    if (warp == 0 || warp == 3) {
        // ================= TMA producers (operands / scales) =================
        const bool leader = elect_one() && !p.withhold_loads;
        const bool operands = warp == 0;
        uint32_t stage = 0, phase = 0;
        int rbs = 0;
        for (int rb = 0; rb < C::kRB; rb++) rbs += (rb0 + rb) < p.rbB;
        for (int kt = kt0; kt < kt1; kt++) {
            if (!mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) break;
            const uint32_t sA = smem_base + stage * C::kStageBytes;
            const uint32_t sB = sA + C::kABytes;
            const uint32_t sSFA = sB + C::kBBytes;
            const uint32_t sSFB = sSFA + C::kSfaBytes;
            const uint32_t full = bar_full + 8 * stage;
            const int nch = min(2, p.nblk4 - 2 * kt);
            if (leader && operands) {
                mbar_expect_tx(full, (uint32_t)(C::kABytes + C::kBBytes + nch * kSfChunk * (1 + rbs)));
                tma_load_2d(sA, &map_a, kt * kBKBytes, mb * kBM, full);
                tma_load_2d(sB, &map_b, kt * kBKBytes, nb * BN, full);
            }
            if (leader && !operands) {
                bulk_load(sSFA, p.sfa + ((size_t)mb * p.nblk4 + 2 * kt) * kSfChunk, (uint32_t)(nch * kSfChunk), full);
#pragma unroll
                for (int rb = 0; rb < C::kRB; rb++)
                    if ((rb0 + rb) < p.rbB)
                        bulk_load(sSFB + rb * 2 * kSfChunk, p.sfb + ((size_t)(rb0 + rb) * p.nblk4 + 2 * kt) * kSfChunk,
                                  (uint32_t)(nch * kSfChunk), full);
            }
            __syncwarp();
            if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == 2) {
        // ================= scale copier =================
        const bool leader = elect_one();
        uint32_t stage = 0, phase = 0;
        for (int kt = kt0; kt < kt1; kt++) {
            if (!mbar_wait_warp(bar_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) break;
            tc_fence_after();
            const uint32_t sSFA = smem_base + stage * C::kStageBytes + C::kABytes + C::kBBytes;
            const uint32_t sSFB = sSFA + C::kSfaBytes;
            const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8;
            const int nch = min(2, p.nblk4 - 2 * kt);
            if (leader) {
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    if (c < nch) {
                        tc_cp_sf(t_sfa + 4 * c, desc_sf(sSFA + c * kSfChunk));
#pragma unroll
                        for (int rb = 0; rb < C::kRB; rb++)
                            tc_cp_sf(t_sfb + 4 * C::kRB * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
                    }
                }
                tc_commit(bar_sf_full + 8 * stage);
            }
            __syncwarp();
            if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        const bool leader = elect_one();
        uint32_t stage = 0, phase = 0;
        const int nmma_last = (int)((p.Kc - (int64_t)(p.kt_total - 1) * kBKElems + 63) / 64);
        const uint32_t sfb_shift = (uint32_t)(((nb * BN) & 127) >> 5);
        bool alive = true;
        for (int kt = kt0; kt < kt1; kt++) {
            if (!mbar_wait_warp(bar_sf_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
            tc_fence_after();
            const uint32_t sA = smem_base + stage * C::kStageBytes;
            const uint64_t adesc = desc_operand_sw128(sA), bdesc = desc_operand_sw128(sA + C::kABytes);
            const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8 + sfb_shift;
            const int nmma = kt == p.kt_total - 1 ? nmma_last : 4;
            if (leader) {
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (k < nmma) {
                        const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                        tc_mma_mxf4(tmem_base + (uint32_t)((kt - kt0) & 1) * BN, adesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                    bdesc + (uint64_t)(k * (kMmaKBytes >> 4)), idesc_mxf4(BN, sf_id, sf_id), t_sfa + 4 * (k >> 1),
                                    t_sfb + 4 * C::kRB * (k >> 1), (kt - kt0 >= 2 || k > 0) ? 1u : 0u);
                    }
                }
                tc_commit(bar_empty + 8 * stage);
            }
            __syncwarp();
            if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
        }
        if (alive && leader) tc_commit(bar_acc_full);   // also with no K tiles at all: nothing pending, arrives at once
        __syncwarp();
    }

    // ---- the epilogue warps wait for the accumulator; then the whole cluster meets: every ring is idle ----
    if (warp >= kEpiWarp0) {
        mbar_wait_warp(bar_acc_full, 0u, abort_flag, p.dev_status, p.spin_limit);
        tc_fence_after();
    }
    ck_cluster_sync();

    // ---- send: warp (quarter q, column half h) reads its 32 rows x 96 columns and hands each 32-column chunk to its owner ----
    const uint32_t slots = (uint32_t)((C::kChunks + S - 1) / S);    // chunks owned per CTA
    if (warp >= kEpiWarp0) {
        const int quarter = warp & 3, chalf = (warp - kEpiWarp0) >> 2;
        const int row = quarter * 32 + lane;
        const bool have = kt1 > kt0;          // a CTA without K tiles contributes zeros
        const bool have_odd = kt1 - kt0 >= 2; // the second accumulator has been written
#pragma unroll 1
        for (int cc = 0; cc < 3; cc++) {
            const uint32_t chunk = (uint32_t)(chalf * 3 + cc);
            uint32_t r[32];
            if (have) {
                tc_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + chunk * 32, r);
                tc_wait_ld();
                if (have_odd) {
                    uint32_t r2[32];
                    tc_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + BN + chunk * 32, r2);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; j++) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
                }
            } else {
#pragma unroll
                for (int j = 0; j < 32; j++) r[j] = 0u;
            }
            const uint32_t owner = chunk % S, slot = chunk / S;
            // receive area of the owner: [source rank][slot][row][32 floats], 16-byte pieces swizzled by the row
            const uint32_t local = smem_base + ((rank * slots + slot) * kBM + (uint32_t)row) * 128u;
            const uint32_t remote = ck_map(local, owner);
#pragma unroll
            for (int j = 0; j < 8; j++)
                ck_store_remote(remote + (uint32_t)((j ^ (row & 7)) << 4), __uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
        }
        tc_fence_before();
    }
    ck_cluster_sync();

    // ---- reduce and store the chunks this CTA owns: sources added in rank order ----
    {
        const bool use_bias = p.bias != nullptr;
        for (uint32_t slot = 0; slot < slots; slot++) {
            const uint32_t chunk = slot * S + rank;
            if (chunk >= (uint32_t)C::kChunks) break;
            const int col0 = nb * BN + (int)chunk * 32;
            if (col0 >= p.N) continue;
            for (int e = threadIdx.x; e < kBM * 8; e += kGemmThreads) {
                const int row = e >> 3, j = e & 7;
                const int grow = mb * kBM + row, gcol = col0 + j * 4;
                if (grow >= p.M || gcol >= p.N) continue;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                for (uint32_t src = 0; src < S; src++) {
                    const float4 v = *reinterpret_cast<const float4 *>(smem + ((src * slots + slot) * kBM + (uint32_t)row) * 128u +
                                                                        (uint32_t)((j ^ (row & 7)) << 4));
                    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
                }
                if (use_bias) {
                    acc.x += __bfloat162float(p.bias[gcol]); acc.y += __bfloat162float(p.bias[gcol + 1]);
                    acc.z += __bfloat162float(p.bias[gcol + 2]); acc.w += __bfloat162float(p.bias[gcol + 3]);
                }
                if (p.out_fp32) {
                    *reinterpret_cast<float4 *>(static_cast<float *>(p.d) + (int64_t)grow * p.ldd + gcol) = acc;
                } else {
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
                    uint2 o;
                    o.x = *reinterpret_cast<const uint32_t *>(&lo);
                    o.y = *reinterpret_cast<const uint32_t *>(&hi);
                    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p.d) + (int64_t)grow * p.ldd + gcol) = o;
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// ---- the kernel of a small forward pass -------------------------------------------------------------------
// Y = Q1(X) Q2(W)^T for a batch whose 128 x 128 tiles all fit on the SMs at once, X in bf16: one launch quantizes X and multiplies.
// Such a call is bound by the host and by the latency of its launches, so the quantizer as a launch of its own is a fifth of it.
// The CTAs of a cluster have the same 128 rows of X and share their quantization: each takes every cluster-size-th group of 32, rounds it
// as k_quantize_rows does, and writes codes and scale into the shared memory of all of them, in the layout the tensor core reads.  The B
// tile and its scales, the whole contraction of them, travel meanwhile.  The cluster that has the first columns also stores the
// codes and scales of X, padding included: the backward pass reads them.
constexpr int kXQuantThreads = kGemmThreads - 32;   // all warps but the one that loads B
constexpr int kXMaxKt = 2;
struct XSource {
    const __nv_bfloat16 *x;
    int64_t ldx;
    uint8_t *codes, *scales;
    int scale_mode, cluster;
};
constexpr int x_staging_off(int kt) { return kt * (2 * kBM * kBKBytes + 4 * kSfChunk); }
constexpr int x_smem_bytes(int kt) { return x_staging_off(kt) + kEpiWarps * 2 * kStagingBytes + 256 + kEpiWarps * 128 + 1024; }
constexpr int kXSmemBytes = 120 << 10;   // one CTA per SM: a CTA that waited for tensor memory would keep its cluster waiting
static_assert(x_smem_bytes(kXMaxKt) <= kXSmemBytes, "shared memory budget");

__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4_x(const __grid_constant__ CUtensorMap map_b, const __grid_constant__ CUtensorMap map_d, const __grid_constant__ CUtensorMap map_dw,
              const __grid_constant__ GemmParams p, const XSource x)
{
    constexpr int BN = 128, kTmemCols = 256, kSfaCol = BN, kSfbCol = BN + 8 * kXMaxKt;   // 8 columns of scales per K tile
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int ktn = p.kt_total;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t sA = smem_base, sB = sA + ktn * kBM * kBKBytes, sSFA = sB + ktn * kBM * kBKBytes, sSFB = sSFA + ktn * 2 * kSfChunk;
    uint8_t *staging0 = smem + x_staging_off(ktn);
    uint64_t *bars = reinterpret_cast<uint64_t *>(staging0 + kEpiWarps * 2 * kStagingBytes);
    const uint32_t bar_b = smem_u32(bars), bar_acc_full = bar_b + 8 * kXMaxKt, bar_acc_empty = bar_acc_full + 8;   // bar_b: one per K tile
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + kXMaxKt + 2);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mb = p.by_tiles_n.div(blockIdx.x), nb = (int)blockIdx.x - mb * p.tiles_n;
    const uint32_t rank = ck_cluster_rank();

    if (threadIdx.x == 0) {
        prefetch_map(&map_b);
        for (int k = 0; k < ktn; k++) mbar_init(bar_b + 8 * k, 1);
        mbar_init(bar_acc_full, 1);
        mbar_init(bar_acc_empty, kEpiWarps);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // this CTA is there: its shared memory may be written
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const int ew = warp - kEpiWarp0, quarter = warp & 3, chalf = ew >> 2;   // epilogue warps
    pdl_wait();
    uint32_t bias[1];
    if (warp >= kEpiWarp0) bias_fetch<BN / 2>(bias, p.bias, (int64_t)nb * BN + chalf * (BN / 2), p.N, lane);

    if (warp == 0) {
        if (elect_one() && !p.withhold_loads) {
            for (int kt = 0; kt < ktn; kt++) {
                const int nch = min(2, p.nblk4 - 2 * kt);
                mbar_expect_tx(bar_b + 8 * kt, (uint32_t)(kBM * kBKBytes + nch * kSfChunk));
                tma_load_2d(sB + kt * kBM * kBKBytes, &map_b, kt * kBKBytes, nb * BN, bar_b + 8 * kt);
                bulk_load(sSFB + kt * 2 * kSfChunk, p.sfb + ((size_t)nb * p.nblk4 + 2 * kt) * kSfChunk, (uint32_t)(nch * kSfChunk), bar_b + 8 * kt);
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        // ================= this CTA's share of Q1(X) =================
        const int nblk = (int)(p.Kc / 32), nb_pad = p.nblk4 * 4, total = kBM * nb_pad;
        const uint32_t tf_add = tf_add_of(x.scale_mode);
        bool nonfinite = false, there = false;
        // (the condition is that of the warp's first lane: the warp stays together for the barrier)
        for (int e = ((int)threadIdx.x - 32) * x.cluster + (int)rank; e - lane * x.cluster < total; e += kXQuantThreads * x.cluster) {
            const int row = e / nb_pad, blk = e - row * nb_pad;
            const int64_t grow = (int64_t)mb * kBM + row;
            const bool in = e < total && grow < p.M && blk < nblk;
            uint4 q[4] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
            if (in) {
                const uint4 *src = reinterpret_cast<const uint4 *>(x.x + grow * x.ldx + blk * 32);
#pragma unroll
                for (int j = 0; j < 4; j++) q[j] = ld_stream_16(src + j);
            }
            uint32_t byte;
            const uint4 codes = rne_group(q, tf_add, byte);
            if (!in) byte = 0x7Fu;
            nonfinite |= byte == 0xFFu;
            if (!there) {                                       // before the first store into another CTA; the whole warp, once
                __syncwarp();
                asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
                there = true;
            }
            if (e < total) {
                const uint32_t at = sA + (uint32_t)((blk >> 3) * kBM * kBKBytes + row * kBKBytes + (((blk & 7) ^ (row & 7)) << 4));
                const uint32_t sc = sSFA + (uint32_t)((blk >> 2) * kSfChunk + (row & 31) * 16 + (row >> 5) * 4 + (blk & 3));
                for (int t = 0; t < x.cluster; t++) {
                    if (blk < nblk)
                        asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(ck_map(at, t)), "r"(codes.x), "r"(codes.y), "r"(codes.z), "r"(codes.w) : "memory");
                    asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(ck_map(sc, t)), "r"(byte) : "memory");
                }
            }
        }
        __syncwarp();
        if (!there) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (nonfinite && p.dev_status) atomicOr(p.dev_status, MXFP4_DEV_NONFINITE);
        asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");   // the stores above, before the tensor core reads them
        __syncwarp();
    }
    ck_cluster_sync();                                          // all of Q1(X) is in place

    if (warp == 1) {
        // ================= scale copies and MMAs, from one thread: they run in order =================
        asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
        const bool leader = elect_one();
        bool alive = true;
        for (int kt = 0; kt < ktn; kt++) {
            if (!mbar_wait_warp(bar_b + 8 * kt, 0u, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
            tc_fence_after();
            const int64_t left = p.Kc - (int64_t)kt * kBKElems;
            const uint32_t t_sfa = tmem_base + kSfaCol + 8 * kt, t_sfb = tmem_base + kSfbCol + 8 * kt;
            const uint64_t adesc = desc_operand_sw128(sA + kt * kBM * kBKBytes), bdesc = desc_operand_sw128(sB + kt * kBM * kBKBytes);
            if (leader) {
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    if (left > 128 * c) {
                        tc_cp_sf(t_sfa + 4 * c, desc_sf(sSFA + (2 * kt + c) * kSfChunk));
                        tc_cp_sf(t_sfb + 4 * c, desc_sf(sSFB + (2 * kt + c) * kSfChunk));
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (left > 64 * k) {
                        const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                        tc_mma_mxf4(tmem_base, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)), idesc_mxf4(BN, sf_id, sf_id),
                                    t_sfa + 4 * (k >> 1), t_sfb + 4 * (k >> 1), (kt > 0 || k > 0) ? 1u : 0u);
                    }
                }
            }
            __syncwarp();
        }
        if (alive && leader) tc_commit(bar_acc_full);
        __syncwarp();
    } else if (warp < kEpiWarp0 && nb < x.cluster) {
        // ================= codes and scales of X, by the row block's first cluster =================
        // (behind the cluster's barrier: a barrier that releases stores to global memory waits for them)
        const int nblk = (int)(p.Kc / 32), nb_pad = p.nblk4 * 4, total = kBM * nb_pad, me = warp == 0 ? lane : 32 * (warp - 1) + lane;
        for (int e = me * x.cluster + (int)rank; e < total; e += 96 * x.cluster) {
            const int row = e / nb_pad, blk = e - row * nb_pad;
            const int64_t grow = (int64_t)mb * kBM + row;
            const uint32_t at = (uint32_t)((blk >> 3) * kBM * kBKBytes + row * kBKBytes + (((blk & 7) ^ (row & 7)) << 4));
            const uint32_t sc = (sSFA - smem_base) + (uint32_t)((blk >> 2) * kSfChunk + (row & 31) * 16 + (row >> 5) * 4 + (blk & 3));
            if (grow < p.M && blk < nblk) *reinterpret_cast<uint4 *>(x.codes + grow * (p.Kc / 2) + blk * 16) = *reinterpret_cast<const uint4 *>(smem + at);
            x.scales[scale_offset(grow, blk, p.nblk4)] = smem[sc];
        }
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue =================
        const uint32_t bias_line = smem_u32(staging0) + kEpiWarps * 2 * kStagingBytes + 256 + ew * 128;
        uint32_t sbuf = 0;
        if (mbar_wait(bar_acc_full, 0u, abort_flag, p.dev_status, p.spin_limit)) {
            tc_fence_after();
            if (p.bias != nullptr) bias_stage<BN / 2>(bias, bias_line, lane);
            epilogue_tile<BN, 2>(&map_d, &map_dw, p, tmem_base + ((uint32_t)(quarter * 32) << 16) + chalf * (BN / 2), mb * kBM + quarter * 32,
                                 nb * BN + chalf * (BN / 2), 0, staging0 + ew * 2 * kStagingBytes, sbuf, lane, bar_acc_empty, bias_line);
        }
        if (lane == 0) bulk_wait_read<0>();   // the stores of this warp have read their staging buffers: the shared memory may go
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

// ---- MMA issue ceiling -----------------------------------------------------------------------------------
// What the tensor pipe takes when nothing else is in the way: one CTA per SM, operands and scales resident in shared
// memory / TMEM, one warp issuing kind::mxf4 MMAs of 128 x BN x 64 back to back into one accumulator, no loads, no
// scale copies inside the loop, no epilogue.  The rate of this loop is the ceiling a GEMM kernel on this part can be
// held against (the roofline denominators of the benchmark are measured copies and bf16 GEMMs, not FP4).
template <int BN>
__global__ void __launch_bounds__(128, 1) k_mma_ceiling(int iters, uint32_t *dev_status)
{
    constexpr int kRB = (BN + 127) / 128;
    constexpr int kABytes = kBM * kBKBytes, kBBytes = BN * kBKBytes, kSfBytes = 2 * kSfChunk * (1 + kRB);
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kABytes + kBBytes + kSfBytes);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const uint32_t smem_base = smem_u32(smem), bar_sf = smem_u32(bars), bar_done = bar_sf + 8;
    const int warp = threadIdx.x >> 5;

    // operands: any bit pattern is a valid pair of E2M1 codes; scales: 2^0
    for (int i = threadIdx.x; i < (kABytes + kBBytes) / 4; i += 128)
        reinterpret_cast<uint32_t *>(smem)[i] = 0x9E3779B9u * (uint32_t)(i + 1) + blockIdx.x;
    for (int i = threadIdx.x; i < kSfBytes / 4; i += 128) reinterpret_cast<uint32_t *>(smem + kABytes + kBBytes)[i] = 0x7F7F7F7Fu;
    if (threadIdx.x == 0) {
        mbar_init(bar_sf, 1);
        mbar_init(bar_done, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_async_smem();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        const bool leader = elect_one();
        const uint32_t sSFA = smem_base + kABytes + kBBytes, sSFB = sSFA + 2 * kSfChunk;
        const uint32_t t_sfa = tmem_base + BN, t_sfb = t_sfa + 8;
        if (leader) {
#pragma unroll
            for (int c = 0; c < 2; c++) {
                tc_cp_sf(t_sfa + 4 * c, desc_sf(sSFA + c * kSfChunk));
#pragma unroll
                for (int rb = 0; rb < kRB; rb++) tc_cp_sf(t_sfb + 4 * kRB * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
            }
            tc_commit(bar_sf);
        }
        __syncwarp();
        bool ok = mbar_wait_warp(bar_sf, 0u, abort_flag, dev_status);
        tc_fence_after();
        const uint64_t adesc = desc_operand_sw128(smem_base), bdesc = desc_operand_sw128(smem_base + kABytes);
        for (int it = 0; it < iters && ok; it++) {
            if (leader) {
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                    tc_mma_mxf4(tmem_base, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                idesc_mxf4(BN, sf_id, sf_id), t_sfa + 4 * (k >> 1), t_sfb + 4 * kRB * (k >> 1), (it > 0 || k > 0) ? 1u : 0u);
                }
            }
            __syncwarp();
        }
        if (leader) tc_commit(bar_done);
        __syncwarp();
        mbar_wait_warp(bar_done, 0u, abort_flag, dev_status);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// ---- the two-CTA kernel ---------------------------------------------------------------------------------
// A pair of CTAs (a cluster of two SMs) computes a 256 x 256 tile with tcgen05.mma.cta_group::2: each CTA holds 128
// rows of A, HALF of the B tile, the scales of its own A rows and the scales of all 256 B rows, and ends up with the
// accumulator of its own 128 rows.  Per SM and stage that is 32 KB of operands instead of 48 KB for the same flops:
// the single-CTA kernel is limited by operand delivery from L2, not by the tensor pipe.
// Roles per CTA are those of the single-CTA kernel, except that only the leader (rank 0) issues scale copies and MMAs
// (both act on the shared memory and TMEM of both CTAs), and warp 2 of the peer relays "my stage has landed" to the
// leader.  Stage and accumulator releases reach both CTAs through multicast commits.
// BN = 192: 256 x 192 tiles for output widths that are multiples of 192 but not of 256.  Narrower stages (31 KB), two
// accumulators (the next tile's K loop runs under the epilogue), which leaves TMEM columns for the scales of five stages.
template <int BN>
struct Gemm2Cfg {
    static constexpr int kABytes = kBM * kBKBytes;                      // 16 KB: this CTA's 128 rows of A
    static constexpr int kBBytes = (BN / 2) * kBKBytes;                 // this CTA's half of the B rows
    static constexpr int kSfaBytes = 2 * kSfChunk;
    static constexpr int kSfbBytes = 2 * kSfChunk * 2;                  // all B rows: the two 128-row blocks a tile touches
    static constexpr int kStageBytes = kABytes + kBBytes + kSfaBytes + kSfbBytes;   // 35 KB / 31 KB
    // The loop is bound by operand bytes in flight over load latency, so every stage counts: six stages and a single
    // staging buffer per epilogue warp (8192^3 184 us, 198 with five and three, 187 with no slack to align the window: the kernel
    // declares its window 1024-byte aligned and checks that it is).  So do short K loops, whose epilogue is the larger part: with four
    // stages and four buffers 50432 x 1024 x 1536 took 52.6 us, 43.6 with five and three, and takes 38.8.
    static constexpr int kStages = BN == 192 ? 5 : 6;
    static constexpr int kStagingBufs = BN == 192 ? 3 : 1;
    static constexpr int kAccStages = BN == 192 ? 2 : 1;
    static constexpr int kSfCol = kAccStages * BN;                      // TMEM: accumulators, then per ring stage SFA (8) + SFB (16)
    static constexpr int kSfSlot = 24;
    static constexpr int kTmemCols = 512;
    static constexpr int kStagingOff = kStages * kStageBytes;
    static constexpr int kBarOff = kStagingOff + kEpiWarps * kStagingBufs * kStagingBytes;
    static constexpr int kBiasOff = kBarOff + 256;                      // BN = 192: a line of BN / 2 bf16 per epilogue warp
    static constexpr int kSmemBytes = kBiasOff + (BN == 192 ? kEpiWarps * BN : 0);
    static_assert(kSfCol + kStages * kSfSlot <= 512, "TMEM budget");
    static_assert(kStageBytes % 1024 == 0 && kStagingOff % 1024 == 0, "alignment");
    static_assert((3 * kStages + 2 * kAccStages + 1) * 8 <= 256, "barrier slots");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
// Non-blocking test: a suspended try_wait was seen to notice an arrival from the other CTA only after its time slice
// (about a microsecond), which stalls the pipeline every other stage.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait on a barrier that CTAs of the cluster arrive on; warp-uniform result.
__device__ __forceinline__ bool mbar_wait_cluster_warp(uint32_t bar, uint32_t parity, volatile uint32_t *abort_flag, uint32_t *dev_status,
                                                       uint32_t limit)
{
    bool ok = false;
    for (uint32_t spin = 0; spin < limit; spin++) {
        if (mbar_try_wait_cluster(bar, parity)) { ok = true; break; }
        if (spin > 4096) {
            if (*abort_flag) break;
            __nanosleep(64);
        }
    }
    if (!ok && !*abort_flag) {
        *abort_flag = 1u;
        if (dev_status) atomicOr(dev_status, MXFP4_DEV_TIMEOUT);
    }
    return __all_sync(0xFFFFFFFFu, ok);
}
// Tile load whose completion is counted on a barrier that may live in the other CTA of the pair.
__device__ __forceinline__ void tma2_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar_cluster_addr)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void tc2_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc2_commit_both(uint32_t bar)   // the same barrier in both CTAs of the pair
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tc2_cp_sf(uint32_t taddr, uint64_t sdesc)
{
    asm volatile("tcgen05.cp.cta_group::2.32x128b.warpx4 [%0], %1;" ::"r"(taddr), "l"(sdesc) : "memory");
}
__device__ __forceinline__ void tc2_mma_mxf4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t sfa_tmem,
                                             uint32_t sfb_tmem, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa_tmem), "r"(sfb_tmem) : "memory");
}
// Instruction descriptor of the pair MMA: M = 256 (128 rows per CTA), N = n (256 unless said otherwise).
__device__ __forceinline__ uint32_t idesc_mxf4_pair(uint32_t a_sf_id, uint32_t b_sf_id, int n = 256)
{
    return (b_sf_id << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(256 >> 4) << 24) | (a_sf_id << 29);
}

// The work items (tile, part of the contraction) of one CTA pair.  Two products in one launch (the weight gradient and the input
// gradient of a layer): the first has the longer items.  The pairs take its items in turn; those that this leaves with one
// item fewer start on the second product, `head` rounds ahead of the others.
struct PairItem {
    bool second, done;
    int mb2, nb, split;
};
struct PairWalk {
    int w, workers, items, items2;   // this pair, the pairs of the launch, the items of either product
    int mine, full, ahead;           // this pair's items of the first; pairs with one item more, and with one fewer (all, when none has more)
};
__device__ __forceinline__ int pair_items(const GemmParams &p) { return ((p.tiles_m + 1) >> 1) * p.tiles_n * p.splits; }
template <bool TWO> __device__ __forceinline__ PairWalk pair_walk(const GemmParams &p, const GemmParams &p2)
{
    PairWalk k;
    k.w = blockIdx.x >> 1, k.workers = gridDim.x >> 1;
    k.items = pair_items(p);
    if (TWO) {
        k.items2 = pair_items(p2);
        k.mine = (k.items - k.w + k.workers - 1) / k.workers;
        k.full = k.items % k.workers;
        k.ahead = k.workers - k.full;
    }
    return k;
}
template <bool TWO> __device__ __forceinline__ PairItem pair_item(const GemmParams &p, const GemmParams &p2, const PairWalk &k, int i)
{
    PairItem x;
    int item = k.w + i * k.workers;
    x.second = false;
    x.done = item >= k.items;
    const GemmParams *q = &p;
    if (TWO && x.done) {
        const int j = i - k.mine, head = p2.head;
        item = k.w >= k.full && j < head ? j * k.ahead + k.w - k.full : head * k.ahead + (k.w >= k.full ? j - head : j) * k.workers + k.w;
        x.second = true;
        x.done = item >= k.items2;
        q = &p2;
    }
    const int tile = q->by_splits.div(item), tm = q->by_tiles_n.div(tile);
    x.split = item - tile * q->splits;
    x.mb2 = ((q->tiles_m + 1) >> 1) - 1 - tm;
    x.nb = tile - tm * q->tiles_n;
    return x;
}

template <int BN, class Job2>   // Job2 = PairJob: a second product follows; NoJob: there is none
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4_pair(const __grid_constant__ PairJob one, const __grid_constant__ Job2 two)
{
    using C = Gemm2Cfg<BN>;
    constexpr bool kTwo = sizeof(Job2) == sizeof(PairJob);
    const PairJob *const job2 = kTwo ? reinterpret_cast<const PairJob *>(&two) : &one;
    const GemmParams &p0 = one.p;   // what both products share: limits, status
    extern __shared__ __align__(1024) uint8_t smem_aligned[];
    uint8_t *smem = smem_aligned;
    if (smem_u32(smem) & 1023u) {   // the swizzled operand tiles need it; nothing has been set up yet, so everybody just leaves
        pdl_wait();
        if (threadIdx.x == 0 && p0.dev_status) atomicOr(p0.dev_status, MXFP4_DEV_SMEM_LAYOUT);
        return;
    }
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    // barrier slots: full[S] (used in the leader only: the loads of BOTH CTAs complete on it), sf_full[S], empty[S],
    // acc_full, acc_empty
    const uint32_t bar_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_full + 8 * C::kStages;
    const uint32_t bar_empty = bar_sf_full + 8 * C::kStages;
    const uint32_t bar_acc_full = bar_empty + 8 * C::kStages;
    const uint32_t bar_acc_empty = bar_acc_full + 8 * C::kAccStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * C::kStages + 2 * C::kAccStages);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 32 * 3) { prefetch_map(&one.a); prefetch_map(&one.b); prefetch_map(&one.sfa); prefetch_map(&one.sfb); prefetch_map(&one.d); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; s++) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < C::kAccStages; a++) {
            mbar_init(bar_acc_full + 8 * a, 1);
            mbar_init(bar_acc_empty + 8 * a, 2 * kEpiWarps);   // the epilogue warps of both CTAs hand an accumulator back to the leader
        }
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();     // both CTAs have their barriers and TMEM before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const PairWalk walk = pair_walk<kTwo>(one.p, job2->p);

    if (warp == 0 || warp == 3) {
        // ===== TMA producers (both CTAs: own rows of A and own half of B by warp 0; own SFA and all of SFB by warp 3) =====
        // All loads of both CTAs complete on the LEADER's full barrier (the cta_group::2 form of the load allows the
        // barrier to live in the other CTA of the pair), so the leader learns that a stage has landed in both shared
        // memories without any message between the CTAs.  The leader's warp 0 posts the byte count of both.
        const bool leader = elect_one() && !p0.withhold_loads;
        const bool operands = warp == 0;
        uint32_t stage = 0, phase = 0;
        bool alive = true;
        pdl_wait();
        for (int i = 0; alive; i++) {
            const PairItem x = pair_item<kTwo>(one.p, job2->p, walk, i);
            if (x.done) break;
            const PairJob &job = x.second ? *job2 : one;
            const GemmParams &p = job.p;
            const int mb = x.mb2 * 2 + (int)rank, nb = x.nb;
            const int kt0 = x.split * p.kt_per_split;
            const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
            for (int kt = kt0; kt < kt1; kt++) {
                if (!mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1u, abort_flag, p0.dev_status, p0.spin_limit)) { alive = false; break; }
                const uint32_t sA = smem_base + stage * C::kStageBytes;
                const uint32_t sB = sA + C::kABytes;
                const uint32_t sSFA = sB + C::kBBytes;
                const uint32_t sSFB = sSFA + C::kSfaBytes;
                const uint32_t full = map_to_cta(bar_full + 8 * stage, 0);
                const int ktr = kt1 - 1 - (kt - kt0);   // the K tiles are taken from the last to the first
                if (leader && operands) {
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * stage, 2u * (uint32_t)C::kStageBytes);
                    tma2_load_2d(sA, &job.a, ktr * kBKBytes, mb * kBM, full);
                    tma2_load_2d(sB, &job.b, ktr * kBKBytes, nb * BN + (int)rank * (BN / 2), full);
                }
                if (leader && !operands) {
                    // scale rows are 128-row blocks, 256 words (two 512-byte chunks) per stage; blocks beyond the matrix read as zero
                    tma2_load_2d(sSFA, &job.sfa, ktr * 256, mb, full);
                    tma2_load_2d(sSFB, &job.sfb, ktr * 256, (nb * BN) >> 7, full);
                }
                __syncwarp();
                if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 2) {
        // ================= scale copier (leader CTA only; each copy acts on both CTAs) =================
        pdl_wait();
        if (rank == 0) {
            const bool leader = elect_one();
            uint32_t stage = 0, phase = 0;
            bool alive = true;
            for (int i = 0; alive; i++) {
                const PairItem x = pair_item<kTwo>(one.p, job2->p, walk, i);
                if (x.done) break;
                const GemmParams &p = x.second ? job2->p : one.p;
                const int kt0 = x.split * p.kt_per_split;
                const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
                for (int kt = kt0; kt < kt1; kt++) {
                    if (!mbar_wait_warp(bar_full + 8 * stage, phase, abort_flag, p0.dev_status, p0.spin_limit)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sSFA = smem_base + stage * C::kStageBytes + C::kABytes + C::kBBytes;
                    const uint32_t sSFB = sSFA + C::kSfaBytes;
                    const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8;
                    const int64_t kleft = p.Kc - (int64_t)(kt1 - 1 - (kt - kt0)) * kBKElems;
                    const int nch = kleft > 128 ? 2 : 1;
                    if (leader) {
#pragma unroll
                        for (int c = 0; c < 2; c++) {
                            if (c < nch) {
                                tc2_cp_sf(t_sfa + 4 * c, desc_sf(sSFA + c * kSfChunk));
#pragma unroll
                                for (int rb = 0; rb < 2; rb++) tc2_cp_sf(t_sfb + 8 * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
                            }
                        }
                        tc2_commit(bar_sf_full + 8 * stage);   // arrives once the copies have landed in both TMEMs
                    }
                    __syncwarp();
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer (leader CTA only) =================
        pdl_wait();
        if (rank == 0) {
            const bool leader = elect_one();
            uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
            bool alive = true;
            for (int i = 0; alive; i++) {
                const PairItem x = pair_item<kTwo>(one.p, job2->p, walk, i);
                if (x.done) break;
                const GemmParams &p = x.second ? job2->p : one.p;
                const int kt0 = x.split * p.kt_per_split;
                const int kt1 = min(kt0 + p.kt_per_split, p.kt_total);
                // scale columns hold 32 rows each: a tile that starts 64 rows into a 128-row block starts 2 columns in
                const uint32_t sfb_shift = BN == 192 ? (uint32_t)((x.nb * BN & 127) >> 5) : 0u;
                const uint32_t d_tmem = tmem_base + acc * BN;
                if (!mbar_wait_cluster_warp(bar_acc_empty + 8 * acc, acc_phase ^ 1u, abort_flag, p0.dev_status, p0.spin_limit)) { alive = false; break; }
                tc_fence_after();
                for (int kt = kt0; kt < kt1; kt++) {
                    if (!mbar_wait_warp(bar_sf_full + 8 * stage, phase, abort_flag, p0.dev_status, p0.spin_limit)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sA = smem_base + stage * C::kStageBytes;
                    const uint32_t sB = sA + C::kABytes;
                    const uint32_t t_sfa = tmem_base + C::kSfCol + stage * C::kSfSlot, t_sfb = t_sfa + 8 + sfb_shift;
                    const int64_t kleft = p.Kc - (int64_t)(kt1 - 1 - (kt - kt0)) * kBKElems;
                    const int krem = kleft < kBKElems ? (int)kleft : kBKElems;
                    const int nmma = (krem + 63) / 64;
                    const uint64_t adesc = desc_operand_sw128(sA), bdesc = desc_operand_sw128(sB);
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < 4; k++) {
                            if (k < nmma) {
                                const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                                tc2_mma_mxf4(d_tmem, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                             idesc_mxf4_pair(sf_id, sf_id, BN), t_sfa + 4 * (k >> 1), t_sfb + 8 * (k >> 1),
                                             (kt > kt0 || k > 0) ? 1u : 0u);
                            }
                        }
                        tc2_commit_both(bar_empty + 8 * stage);   // frees the stage in both CTAs once these MMAs have read it
                    }
                    __syncwarp();
                    if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
                }
                if (alive && leader) tc2_commit_both(bar_acc_full + 8 * acc);   // both CTAs' accumulators are complete
                __syncwarp();
                if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ================= epilogue (warps 4..11 of both CTAs: own 128 rows x BN columns) =================
        pdl_wait();
        const int ew = warp - kEpiWarp0;
        const int quarter = warp & 3;
        const int chalf = ew >> 2;
        uint8_t *staging = smem + C::kStagingOff + ew * C::kStagingBufs * kStagingBytes;
        constexpr int kHalfCols = BN / 2;
        constexpr int kChunks = kHalfCols / 32;
        if constexpr (BN == 192) {
            const uint32_t bias_line = smem_base + C::kBiasOff + ew * (BN / 2) * 2;
            uint32_t sbuf = 0, acc = 0, acc_phase = 0;
            for (int i = 0;; i++) {
                const PairItem x = pair_item<kTwo>(one.p, job2->p, walk, i);
                if (x.done) break;
                const PairJob &job = x.second ? *job2 : one;
                const GemmParams &p = job.p;
                const int mb = x.mb2 * 2 + (int)rank, nb = x.nb;
                uint32_t bias[(kHalfCols + 63) / 64];
                bias_fetch<kHalfCols>(bias, p.bias, (int64_t)nb * BN + chalf * kHalfCols, p.N, lane);
                if (!mbar_wait_warp(bar_acc_full + 8 * acc, acc_phase, abort_flag, p0.dev_status, p0.spin_limit)) break;
                tc_fence_after();
                if (p.bias != nullptr) bias_stage<kHalfCols>(bias, bias_line, lane);
                epilogue_tile<BN, C::kStagingBufs, true>(&job.d, &job.dw, p,
                                                         tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + chalf * kHalfCols, mb * kBM + quarter * 32,
                                                         nb * BN + chalf * kHalfCols, x.split, staging, sbuf, lane, map_to_cta(bar_acc_empty + 8 * acc, 0), bias_line);
                if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
            }
        } else {
        const uint32_t acc_empty_leader = map_to_cta(bar_acc_empty, 0);
        uint32_t acc_phase = 0;
        bool alive = true;
        for (int i = 0; alive; i++) {
            const PairItem x = pair_item<kTwo>(one.p, job2->p, walk, i);
            if (x.done) break;
            const PairJob &job = x.second ? *job2 : one;
            const GemmParams &p = job.p;
            const int mb = x.mb2 * 2 + (int)rank, nb = x.nb;
            uint32_t bias[kHalfCols / 32];
#pragma unroll
            for (int cc = 0; cc < kHalfCols / 32; cc++) bias[cc] = load_bias_pair(p.bias, (int64_t)nb * BN + chalf * kHalfCols + cc * 32, p.N, lane);
            if (!mbar_wait_warp(bar_acc_full, acc_phase, abort_flag, p0.dev_status, p0.spin_limit)) { alive = false; break; }
            tc_fence_after();
            const int row0 = mb * kBM + quarter * 32;
            const int colbase = nb * BN + chalf * kHalfCols;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + chalf * kHalfCols;
            const bool use_bias = p.bias != nullptr && p.splits == 1;
            auto store_box = [&](const uint32_t *w, int col0) {
                if (lane == 0) bulk_wait_read<0>();     // the one staging buffer has been read
                __syncwarp();
                stage_line(staging + lane * 64, lane, w);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_3d(&job.d, col0, row0, x.split, smem_u32(staging));
                    bulk_commit();
                }
            };
            auto release_acc = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(acc_empty_leader);
            };
            if (!p.out_fp32) {
                uint32_t pk[kChunks][16];
#pragma unroll
                for (int cc = 0; cc < kChunks; cc++) {
                    const int col = colbase + cc * 32;
                    if (col < p.N && row0 < p.M) {
                        uint32_t r[32];
                        tc_ld32(taddr + cc * 32, r);
                        tc_wait_ld();
                        if (use_bias) add_bias_chunk_shfl(r, bias[cc]);
                        pack_row_bf16(r, pk[cc]);
                    }
                }
                release_acc();
#pragma unroll
                for (int cc = 0; cc < kChunks; cc++) {
                    const int col = colbase + cc * 32;
                    if (col < p.N && row0 < p.M) store_box(pk[cc], col);
                }
            } else {
#pragma unroll 1
                for (int cc = 0; cc < kChunks; cc++) {
                    const int col = colbase + cc * 32;
                    const bool live = col < p.N && row0 < p.M;
                    uint32_t r[32];
                    if (live) {
                        tc_ld32(taddr + cc * 32, r);
                        tc_wait_ld();
                    }
                    if (cc == kChunks - 1) release_acc();
                    if (!live) continue;
                    const int ncols = (int)min((int64_t)32, p.N - col);
                    if (use_bias) add_bias_chunk_shfl(r, load_bias_pair(p.bias, col, p.N, lane));
                    store_box(r, col);
                    if (ncols > 16) store_box(r + 16, col + 16);
                }
            }
            acc_phase ^= 1u;
        }
        }
        if (lane == 0) bulk_wait_read<0>();
    }

    // neither CTA may leave (or free TMEM) while the other can still reach its shared memory, barriers or TMEM
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// ---- the two-CTA B-stationary kernel ----------------------------------------------------------------------
// Short contractions (Kc up to KT K tiles) with many rows: the forward and input-gradient products whose output write
// dominates.  The single-CTA kernels are bound there by shared-memory bandwidth (every operand byte is written once by
// TMA and read once by the tensor core through the same 128 B / cycle port) and the streaming pair kernel by its single
// accumulator.  Here a pair of CTAs walks DOWN a column of 256 x 192 tiles: each CTA keeps its half (96 rows) of the
// column's B block and the scales of all 192 B rows resident for the whole column, the ring carries this CTA's 128 rows
// of A alone (16 KB + 1 KB of scales per stage, eight stages), and two accumulators of 192 columns let the
// epilogue of one tile run under the K loop of the next.  Per stage and SM the port sees 16 KB written and 16 + 12 KB read for a 128 x 192 x 256
// block of the product, less than the tensor pipe needs for it.  Roles, barriers and the cross-CTA signalling are those
// of the two kernels this combines (k_gemm_mxf4_pair, k_gemm_mxf4_bs).
template <int KT, int AS>   // KT: K tiles the resident B block can hold; AS: stages of the A ring
struct GemmPbsCfg {
    static constexpr int BN = 192;
    static constexpr int kABytes = kBM * kBKBytes;              // 16 KB: this CTA's 128 rows of A
    static constexpr int kBBytes = (BN / 2) * kBKBytes;         // 12 KB: this CTA's 96 B rows of one K tile
    static constexpr int kSfaBytes = 2 * kSfChunk;
    static constexpr int kSfbBytes = 2 * kSfChunk * 2;          // per K tile: the two 128-row blocks a tile touches
    static constexpr int kStagingBufs = 2;                     // the ring is worth more than a third buffer: the loop is bound by operand bytes in flight
    static constexpr int kAOff = KT * kBBytes;
    static constexpr int kSfbOff = kAOff + AS * kABytes;
    static constexpr int kSfaOff = kSfbOff + KT * kSfbBytes;
    static constexpr int kStagingOff = kSfaOff + AS * kSfaBytes;
    static constexpr int kBarOff = kStagingOff + kEpiWarps * kStagingBufs * kStagingBytes;
    static constexpr int kBiasOff = kBarOff + 256;              // a line of BN / 2 bf16 per epilogue warp
    static constexpr int kSmemBytes = kBiasOff + kEpiWarps * BN + 1024 /*align*/;
    static constexpr int kSfbCol = 2 * BN;                      // TMEM columns: two accumulators, resident SFB (16 per K tile), SFA ring (8 per stage)
    static constexpr int kSfaCol = kSfbCol + KT * 16;
    static constexpr int kTmemCols = 512;
    static_assert(kSfaCol + AS * 8 <= 512, "TMEM budget");
    static_assert(kAOff % 1024 == 0 && kStagingOff % 1024 == 0, "alignment");
    static_assert((3 * AS + 7) * 8 + 8 <= 256, "barrier slots");
    static_assert(kSmemBytes <= 232448, "shared memory budget");
};

template <int KT, int AS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
k_gemm_mxf4_pbs(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                const __grid_constant__ CUtensorMap map_sfa, const __grid_constant__ CUtensorMap map_sfb,
                const __grid_constant__ CUtensorMap map_d, const __grid_constant__ CUtensorMap map_dw, const GemmParams p)
{
    using C = GemmPbsCfg<KT, AS>;
    constexpr int BN = C::BN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + C::kBarOff);
    // barrier slots: a_full[AS] and b_full (used in the leader only: the loads of BOTH CTAs complete on them), sf_full[AS],
    // b_sf_full (leader only), a_empty[AS], b_empty, acc_full[2] (both CTAs, through multicast commits), acc_empty[2] (leader)
    const uint32_t bar_a_full = smem_u32(bars);
    const uint32_t bar_sf_full = bar_a_full + 8 * AS;
    const uint32_t bar_a_empty = bar_sf_full + 8 * AS;
    const uint32_t bar_acc_full = bar_a_empty + 8 * AS;
    const uint32_t bar_acc_empty = bar_acc_full + 16;
    const uint32_t bar_b_full = bar_acc_empty + 16;
    const uint32_t bar_b_sf_full = bar_b_full + 8;
    const uint32_t bar_b_empty = bar_b_sf_full + 8;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 3 * AS + 7);
    volatile uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t rank = cluster_rank();

    if (threadIdx.x == 32 * 3) { prefetch_map(&map_a); prefetch_map(&map_b); prefetch_map(&map_sfa); prefetch_map(&map_sfb); prefetch_map(&map_d); }
    if (threadIdx.x == 0) {
        for (int s = 0; s < AS; s++) {
            mbar_init(bar_a_full + 8 * s, 1);
            mbar_init(bar_sf_full + 8 * s, 1);
            mbar_init(bar_a_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; a++) {
            mbar_init(bar_acc_full + 8 * a, 1);
            mbar_init(bar_acc_empty + 8 * a, 2 * kEpiWarps);   // the epilogue warps of both CTAs hand an accumulator back to the leader
        }
        mbar_init(bar_b_full, 1);
        mbar_init(bar_b_sf_full, 1);
        mbar_init(bar_b_empty, 2);    // both MMA issuers
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(C::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();     // both CTAs have their barriers and TMEM before anyone signals across
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    const Walk walk = walk_begin(p, blockIdx.x >> 1);   // pair tiles: 256 rows x 192 columns
    const int ktn = p.kt_total;

    if (warp == 0) {
        // ===== producer (both CTAs): own 128 rows of A and their scales per stage; own half of a column's B block and all
        // its scales once per run of tiles in that column.  Everything is counted on the LEADER's barriers. =====
        const bool leader = elect_one() && !p.withhold_loads;
        uint32_t stage = 0, phase = 0, runs = 0;
        int nb = 0;
        pdl_wait();
        bool alive = true;
        auto load_block = [&]() -> bool {
            // the MMAs of the previous column have finished reading the block (multicast commits reach both CTAs)
            if (runs > 0 && !mbar_wait_warp(bar_b_empty, (runs - 1u) & 1u, abort_flag, p.dev_status, p.spin_limit)) return false;
            if (leader) {
                const uint32_t full = map_to_cta(bar_b_full, 0);
                if (rank == 0) mbar_expect_tx(bar_b_full, 2u * (uint32_t)ktn * (uint32_t)(C::kBBytes + C::kSfbBytes));
                for (int kt = 0; kt < ktn; kt++) {
                    tma2_load_2d(smem_base + kt * C::kBBytes, &map_b, kt * kBKBytes, nb * BN + (int)rank * (BN / 2), full);
                    // scale rows are 128-row blocks, 256 words (two 512-byte chunks) per K tile; what lies beyond the matrix reads as zero
                    tma2_load_2d(smem_base + C::kSfbOff + kt * C::kSfbBytes, &map_sfb, kt * 256, (nb * BN) >> 7, full);
                }
            }
            __syncwarp();
            runs++;
            return true;
        };
        for (int i = 0; i < walk.count && alive; i++) {
            // the first block before anything else; later ones after the A stages of the column's first tile, which need
            // nothing from the new block and keep the ring full while the old column drains
            const WalkItem x = walk_item(p, walk, i);
            nb = x.col;
            if (i == 0 && !load_block()) break;
            const int mb = x.row * 2 + (int)rank;
            for (int kt = 0; kt < ktn; kt++) {
                if (!mbar_wait_warp(bar_a_empty + 8 * stage, phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                if (leader) {
                    const uint32_t full = map_to_cta(bar_a_full + 8 * stage, 0);
                    if (rank == 0) mbar_expect_tx(bar_a_full + 8 * stage, 2u * (uint32_t)(C::kABytes + C::kSfaBytes));
                    tma2_load_2d(smem_base + C::kAOff + stage * C::kABytes, &map_a, kt * kBKBytes, mb * kBM, full);
                    tma2_load_2d(smem_base + C::kSfaOff + stage * C::kSfaBytes, &map_sfa, kt * 256, mb, full);
                }
                __syncwarp();
                if (++stage == AS) { stage = 0; phase ^= 1u; }
            }
            if (alive && i > 0 && x.first && !load_block()) break;
        }
    } else if (warp == 2) {
        // ===== scale copier (leader only; each copy acts on both CTAs): B scales once per column, A scales per stage =====
        pdl_wait();
        if (rank == 0) {
            const bool leader = elect_one();
            uint32_t stage = 0, phase = 0, runs = 0;
            bool alive = true;
            for (int i = 0; i < walk.count && alive; i++) {
                if (walk_item(p, walk, i).first) {
                    if (!mbar_wait_warp(bar_b_full, runs & 1u, abort_flag, p.dev_status, p.spin_limit)) break;
                    tc_fence_after();
                    if (leader) {
                        for (int kt = 0; kt < ktn; kt++) {
                            const int nch = min(2, p.nblk4 - 2 * kt);
                            const uint32_t sSFB = smem_base + C::kSfbOff + kt * C::kSfbBytes;
                            const uint32_t t_sfb = tmem_base + C::kSfbCol + kt * 16;
                            for (int c = 0; c < nch; c++)
#pragma unroll
                                for (int rb = 0; rb < 2; rb++) tc2_cp_sf(t_sfb + 8 * c + 4 * rb, desc_sf(sSFB + rb * 2 * kSfChunk + c * kSfChunk));
                        }
                        tc2_commit(bar_b_sf_full);
                    }
                    __syncwarp();
                    runs++;
                }
                for (int kt = 0; kt < ktn; kt++) {
                    if (!mbar_wait_warp(bar_a_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sSFA = smem_base + C::kSfaOff + stage * C::kSfaBytes;
                    const uint32_t t_sfa = tmem_base + C::kSfaCol + stage * 8;
                    const int nch = min(2, p.nblk4 - 2 * kt);
                    if (leader) {
                        tc2_cp_sf(t_sfa, desc_sf(sSFA));
                        if (nch > 1) tc2_cp_sf(t_sfa + 4, desc_sf(sSFA + kSfChunk));
                        tc2_commit(bar_sf_full + 8 * stage);   // arrives once the copies have landed in both TMEMs
                    }
                    __syncwarp();
                    if (++stage == AS) { stage = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1 || warp == 3) {
        // ===== MMA issuers (leader only): warp 1 takes this pair's even tiles into accumulator 0, warp 3 the odd ones
        pdl_wait();
        // into accumulator 1.  One issuing thread needs about 350 cycles per stage (a barrier query, four MMAs, a commit)
        // and several hundred per tile, more than the tensor pipe needs for the stage; two of them leave it waiting for
        // nothing but operands.  Both walk over EVERY stage and every column in order and wait on each barrier phase
        // (a wait that skipped a phase could mistake the phase before for the one it wants); a warp issues and commits only
        // for its own tiles, so a stage's release tracks exactly the MMAs that read it (commits count the issuing thread's
        // operations), and the resident block is released by both (its barrier counts two arrivals). =====
        if (rank == 0) {
            const bool leader = elect_one();
            const uint32_t me = warp == 1 ? 0u : 1u;
            uint32_t stage = 0, phase = 0, acc_phase = 0, runs = 0;
            const int nmma_last = (int)((p.Kc - (int64_t)(ktn - 1) * kBKElems + 63) / 64);   // MMAs of the last K tile
            const uint32_t d_tmem = tmem_base + me * BN;
            bool alive = true;
            for (int i = 0; i < walk.count && alive; i++) {
                const bool mine = (uint32_t)(i & 1) == me;
                const WalkItem x = walk_item(p, walk, i);
                const int nb = x.col;
                if (x.first) {
                    // the block of this column and its scales are in place in both CTAs (the copier saw them land before it copied)
                    if (!mbar_wait_warp(bar_b_sf_full, runs & 1u, abort_flag, p.dev_status, p.spin_limit)) break;
                    runs++;
                }
                // scale columns hold 32 rows each: a tile that starts 64 rows into a 128-row block starts 2 columns in
                const uint32_t sfb_shift = (uint32_t)(((nb * BN) & 127) >> 5);
                if (mine) {
                    if (!mbar_wait_cluster_warp(bar_acc_empty + 8 * me, acc_phase ^ 1u, abort_flag, p.dev_status, p.spin_limit)) break;
                    acc_phase ^= 1u;
                }
                for (int kt = 0; kt < ktn; kt++) {
                    if (!mbar_wait_warp(bar_sf_full + 8 * stage, phase, abort_flag, p.dev_status, p.spin_limit)) { alive = false; break; }
                    if (mine) {
                        tc_fence_after();
                        const uint64_t adesc = desc_operand_sw128(smem_base + C::kAOff + stage * C::kABytes);
                        const uint64_t bdesc = desc_operand_sw128(smem_base + kt * C::kBBytes);
                        const uint32_t t_sfa = tmem_base + C::kSfaCol + stage * 8;
                        const uint32_t t_sfb = tmem_base + C::kSfbCol + kt * 16 + sfb_shift;
                        const int nmma = kt == ktn - 1 ? nmma_last : 4;
                        if (leader) {
#pragma unroll
                            for (int k = 0; k < 4; k++) {
                                if (k < nmma) {
                                    const uint32_t sf_id = (uint32_t)(k & 1) * 2u;
                                    tc2_mma_mxf4(d_tmem, adesc + (uint64_t)(k * (kMmaKBytes >> 4)), bdesc + (uint64_t)(k * (kMmaKBytes >> 4)),
                                                 idesc_mxf4_pair(sf_id, sf_id, BN), t_sfa + 4 * (k >> 1), t_sfb + 8 * (k >> 1),
                                                 (kt > 0 || k > 0) ? 1u : 0u);
                                }
                            }
                            tc2_commit_both(bar_a_empty + 8 * stage);   // frees the A stage in both CTAs once these MMAs have read it
                        }
                        __syncwarp();
                    }
                    if (++stage == AS) { stage = 0; phase ^= 1u; }
                }
                if (alive && leader) {
                    if (mine) tc2_commit_both(bar_acc_full + 8 * me);   // both CTAs' accumulators are complete
                    if (x.last) tc2_commit_both(bar_b_empty);      // this warp's MMAs on the resident blocks are complete
                }
                __syncwarp();
            }
        }
    } else if (warp >= kEpiWarp0) {
        // ===== epilogue (warps 4..11 of both CTAs: own 128 rows x 192 columns) =====
        pdl_wait();
        const int ew = warp - kEpiWarp0;
        const int quarter = warp & 3;
        const int chalf = ew >> 2;
        uint8_t *staging = smem + C::kStagingOff + ew * C::kStagingBufs * kStagingBytes;
        const uint32_t bias_line = smem_base + C::kBiasOff + ew * (BN / 2) * 2;
        uint32_t sbuf = 0;
        constexpr int kHalfCols = BN / 2;
        uint32_t acc = 0, acc_phase = 0;
        for (int i = 0; i < walk.count; i++) {
            const WalkItem x = walk_item(p, walk, i);
            const int mb = x.row * 2 + (int)rank, nb = x.col;
            uint32_t bias[(kHalfCols + 63) / 64];
            bias_fetch<kHalfCols>(bias, p.bias, (int64_t)nb * BN + chalf * kHalfCols, p.N, lane);
            if (!mbar_wait(bar_acc_full + 8 * acc, acc_phase, abort_flag, p.dev_status, p.spin_limit)) break;
            tc_fence_after();
            const int row0 = mb * kBM + quarter * 32;
            const int colbase = nb * BN + chalf * kHalfCols;
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + chalf * kHalfCols;
            if (p.bias != nullptr) bias_stage<kHalfCols>(bias, bias_line, lane);
            epilogue_tile<BN, C::kStagingBufs, true>(&map_d, &map_dw, p, taddr, row0, colbase, 0, staging, sbuf, lane,
                                                     map_to_cta(bar_acc_empty + 8 * acc, 0), bias_line);
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (lane == 0) bulk_wait_read<0>();   // the stores of this warp have read their staging buffers: the shared memory may go
    }

    // neither CTA may leave (or free TMEM) while the other can still reach its shared memory, barriers or TMEM
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols) : "memory");
    }
}

// Sum of the split-K partial tiles in a fixed order, + bias, cast.  GROUPS threads share four output columns: each adds every
// GROUPS-th partial, then the sums meet in shared memory in rising order: eight where one thread per output would leave most
// SMs without a block and each with a long chain of loads (products with their reductions, back to back: 96 x 288 x 401408
// 32.5 -> 24.9 us, 128 x 128 x 50432 9.0 -> 7.9, both with the higher limit on the splits), one where the output fills the
// machine (384 x 384 x 25216: 11.8 us, 12.9 with eight).
template <int GROUPS>
__global__ void __launch_bounds__(256) k_splitk_reduce(const float *part, int splits, int64_t M, int64_t N,
                                                       void *__restrict__ d, int64_t ldd, int out_fp32,
                                                       const __nv_bfloat16 *bias)
{
    constexpr int kCols = 256 / GROUPS;
    __shared__ float4 s_sum[GROUPS][kCols];
    pdl_launch_dependents();
    pdl_wait();
    const int64_t total4 = M * N / 4;
    const int c = threadIdx.x % kCols, g = threadIdx.x / kCols;
    for (int64_t i0 = blockIdx.x * (int64_t)kCols; i0 < total4; i0 += (int64_t)gridDim.x * kCols) {
        const int64_t i = i0 + c, e = i * 4, row = e / N, col = e - row * N;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < total4 && g < splits) {
            acc = *reinterpret_cast<const float4 *>(part + (size_t)g * M * N + e);
            for (int s = g + GROUPS; s < splits; s += 8 * GROUPS) {      // eight loads in flight
                float4 v[8];
#pragma unroll
                for (int j = 0; j < 8; j++)
                    if (s + j * GROUPS < splits) v[j] = *reinterpret_cast<const float4 *>(part + (size_t)(s + j * GROUPS) * M * N + e);
#pragma unroll
                for (int j = 0; j < 8; j++)
                    if (s + j * GROUPS < splits) acc.x += v[j].x, acc.y += v[j].y, acc.z += v[j].z, acc.w += v[j].w;
            }
        }
        if (GROUPS > 1) {
            s_sum[g][c] = acc;
            __syncthreads();
            if (g == 0) {
#pragma unroll
                for (int q = 1; q < GROUPS; q++) {
                    const float4 v = s_sum[q][c];
                    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
                }
            }
            __syncthreads();
        }
        if (g != 0 || i >= total4) continue;
        if (bias) {
            acc.x += __bfloat162float(bias[col]); acc.y += __bfloat162float(bias[col + 1]);
            acc.z += __bfloat162float(bias[col + 2]); acc.w += __bfloat162float(bias[col + 3]);
        }
        if (out_fp32) {
            *reinterpret_cast<float4 *>(static_cast<float *>(d) + row * ldd + col) = acc;
        } else {
            __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
            uint2 o;
            o.x = *reinterpret_cast<uint32_t *>(&lo);
            o.y = *reinterpret_cast<uint32_t *>(&hi);
            *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(d) + row * ldd + col) = o;
        }
    }
}

// ---- host side -------------------------------------------------------------------------------------
// Packed operand [rows, kc/2 bytes] viewed as a 2-D byte tensor; box = 128 bytes x box_rows, 128B swizzle.
static bool make_operand_map(CUtensorMap *map, const void *data, int64_t rows, int64_t kc, int box_rows)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)(kc / 2), (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)(kc / 2)};
    cuuint32_t box[2] = {(cuuint32_t)kBKBytes, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void *>(data), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Scales of a packed [rows, kc] matrix as a 2-D tensor of 32-bit words: one row per 128-row block, 128 words per
// 512-byte chunk; box = 256 words (the two chunks of a 256-K stage) x box_blocks, no swizzle, zero beyond the edges.
static bool make_scale_map(CUtensorMap *map, const void *scales, int64_t rows, int64_t kc, int box_blocks)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint64_t nblk4 = (cuuint64_t)ceil_div(kc / 32, 4);
    cuuint64_t gdim[2] = {nblk4 * 128, (cuuint64_t)ceil_div(rows, 128)};
    cuuint64_t gstride[1] = {nblk4 * 512};
    cuuint32_t box[2] = {256, (cuuint32_t)box_blocks};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void *>(scales), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output [splits][M][N] (splits = 1: the caller's matrix with leading dimension ld) as a 3-D tensor for the
// epilogue's stores; box = 64 bytes x 32 rows, 64B swizzle.  Stores are clipped at M and N.
static bool make_output_map(CUtensorMap *map, void *d, int64_t m, int64_t n, int64_t ld, int splits, bool fp32)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    const cuuint64_t esz = fp32 ? 4 : 2;
    cuuint64_t gdim[3] = {(cuuint64_t)n, (cuuint64_t)m, (cuuint64_t)splits};
    cuuint64_t gstride[2] = {(cuuint64_t)ld * esz, (cuuint64_t)m * (cuuint64_t)ld * esz};
    cuuint32_t box[3] = {(cuuint32_t)(64 / esz), 32, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, d, gdim, gstride, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The bf16 output once more with boxes of 64 columns x 32 rows and 128B swizzle (pairs of 32-column chunks in one store).
static bool make_output_map_wide(CUtensorMap *map, void *d, int64_t m, int64_t n, int64_t ld)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[3] = {(cuuint64_t)n, (cuuint64_t)m, 1};
    cuuint64_t gstride[2] = {(cuuint64_t)ld * 2, (cuuint64_t)m * (cuuint64_t)ld * 2};
    cuuint32_t box[3] = {64, 32, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, d, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct GemmPlan {
    bool pair;   // 256 x 256 tiles on pairs of CTAs (cta_group::2)
    int bs;      // B-stationary kernel: 0 = no, 1 = 192 wide, up to 2 K tiles
    int ck;      // cluster split-K kernel: 0 = no, else the cluster size (CTAs sharing one 128 x 192 tile)
    bool pbs;    // two-CTA B-stationary kernel: 256 x 192 tiles, up to 4 K tiles
    int bn, tiles_m, tiles_n, splits, kt_total, kt_per_split;
};

// Tile width, CTA pairing and split-K factor.
// An MMA takes the same time for any width up to 256, so wide tiles are cheaper per flop; but only tiles up to 192
// wide leave room in TMEM for a second accumulator, which hides the epilogue behind the next K loop.  For long K
// loops the product is limited by operand delivery from L2, and pairs of CTAs sharing the B tile cut that by a third.
// Split K when the output has too few tiles to fill the machine, beyond a least number of parts only as far as their sums fit into
// `scratch` bytes.
static GemmPlan plan_gemm(int64_t m, int64_t n, int64_t kc, int sms, bool allow_split = true, size_t scratch = SIZE_MAX)
{
    GemmPlan g;
    g.kt_total = (int)ceil_div(kc, kBKElems);
    g.bs = 0;
    g.ck = 0;
    g.pbs = false;
    const int64_t rows = ceil_div(m, kBM), tiles128 = rows * ceil_div(n, 128), tiles192 = rows * ceil_div(n, 192);
    if (g.kt_total >= 16) {
        // Few tiles, long contraction (weight-gradient products): pairs of CTAs share a 128 x 192 tile and add their
        // halves of the contraction through distributed shared memory, when that fills between half and all of the
        // machine.  Larger clusters lose: a cluster of six such CTAs (a whole SM each) finds room only 22 times on this
        // part (cudaOccupancyMaxActiveClusters; 33 times for four, 45 for three), and with fewer, longer K loops the
        // two-kernel path below (CTA pairs on 256 x 256 tiles, partial sums through L2) was measured faster.
        const int units = (int)(ceil_div(m, kBM) * ceil_div(n, 192));
        if (units * 2 <= sms && units * 4 >= sms) g.ck = 2;
    }
    if (g.ck) {
        g.bn = 192;
        g.pair = false;
        g.tiles_m = (int)ceil_div(m, kBM);
        g.tiles_n = (int)ceil_div(n, g.bn);
        g.splits = 1;                                   // nothing goes through a workspace
        g.kt_per_split = (int)ceil_div(g.kt_total, g.ck);
        return g;
    }
    if (tiles128 <= sms && (!allow_split || g.kt_total < 8)) {
        // One tile per SM at most: the time is one tile's, from the launch to its last store, and the narrowest tile has the shortest.
        // Back to back, against the wide kernels below, in us: 197 x 1536 x 384 5.7 -> 4.3, 1024 x 768 x 192 5.2 -> 4.2,
        // 1024 x 1024 x 1536 7.7 -> 5.5, 128 x 4096 x 2048 9.0 -> 5.9.  (768 x 768 x 2048 would take 6.3 us this way, 9.6 with K split;
        // but split sums are the more accurate ones, and the faster ones from about 768 x 768 x 8192 on: 12.8 us on either.)
        g.bn = 128;
        g.pair = false;
        g.tiles_m = (int)rows;
        g.tiles_n = (int)ceil_div(n, 128);
        g.splits = 1;
        g.kt_per_split = g.kt_total;
        return g;
    }
    if (g.kt_total >= 3 && g.kt_total <= 4 && n >= 192 && m >= 2048 && sms >= 2 &&
        ceil_div(ceil_div(m, kBM), 2) * ceil_div(n, 192) >= sms) {
        // short contraction, tall output: pairs of CTAs walk down columns of 256 x 192 tiles with the column's B block resident
        // (with one or two K tiles the single-CTA B-stationary kernel below is faster: 401408 x 384 x 96 65.1 against 67.4 us,
        // 25216 x 1152 x 384 14.6 against 16.1, and even at 100352 x 1536 x 384, 58; with fewer than two pair
        // tiles per CTA pair the set-up of a column costs more than the kernel saves: 12.3 against 10.2 us at 2048 x 768 x 768)
        g.pbs = true;
        g.bn = 192;
        g.pair = false;
        g.tiles_m = (int)ceil_div(m, kBM);
        g.tiles_n = (int)ceil_div(n, g.bn);
        g.splits = 1;
        g.kt_per_split = g.kt_total;
        return g;
    }
    if (g.kt_total <= 2 && n > 128) {
        // the whole B block of a tile column fits in shared memory next to a deep ring of A tiles.  (Instances for up to
        // four and six K tiles, whose rings hold barely more than one tile, measured no faster than the kernel above.)
        g.bs = 1;
        g.bn = 192;
        g.pair = false;
        g.tiles_m = (int)ceil_div(m, kBM);
        g.tiles_n = (int)ceil_div(n, g.bn);
        g.splits = 1;
        g.kt_per_split = g.kt_total;
        return g;
    }
    // One wave of 192-wide tiles on single CTAs, where K would not be split, up to 32 K tiles (6272 x 512 x 1536 8.9 -> 7.0 us,
    // 4096 x 768 x 2048 11.1 -> 8.9, x 8192 18.4 on either, x 16384 28.3 -> 31.0).
    const bool one_wave = tiles192 <= sms && g.kt_total <= 32 && (!allow_split || ceil_div(rows, 2) * ceil_div(n, 256) * 4 > sms);
    if (n <= 128) g.bn = 128;
    else if (kc <= 1024 || one_wave) g.bn = 192;
    else g.bn = 256;
    g.pair = g.bn == 256 && m > 128 && sms >= 2;
    // 256 x 192 tiles on pairs, for widths that 256-wide tiles waste a quarter of or more, when K is split (1536 x 384 x 25216
    // 16.7 -> 15.8 us, 384 x 384 x 25216 12.1 -> 11.0, 512 x 384 x 4096 9.5 -> 8.8).  K loops that are not split are faster on the 256-wide
    // pair with its sixth stage, even with the waste (25216 x 1152 x 1536 27.7 us on single CTAs, 25.1 on the pair; 50432 x 1152 x 2048
    // 64.6 with 192-wide pairs, 57.7; 50432 x 960 x 4096 96 and 82; 50432 x 224 x 1536 22.6 and 15.5).
    if (m > 128 && n % 192 == 0 && n % 256 != 0 && n <= 576 && kc > 1024 && sms >= 2 && allow_split && g.kt_total >= 8 &&
        ceil_div(ceil_div(m, kBM), 2) * ceil_div(n, 256) * 2 <= sms / 2)
        g.pair = true, g.bn = 192;
    g.tiles_m = (int)ceil_div(m, kBM);
    g.tiles_n = (int)ceil_div(n, g.bn);
    const int units = (g.pair ? (g.tiles_m + 1) / 2 : g.tiles_m) * g.tiles_n;   // work items before splitting K
    const int workers = g.pair ? sms / 2 : sms;
    int splits = 1;
    if (allow_split && units * 2 <= workers && g.kt_total >= 8) {
        splits = min(workers / units, g.kt_total / 4);
        splits = max(1, min(splits, 64));   // (at 32, three tiles of 384 x 96 x 401408 left 52 of 148 SMs idle: 26.2 us with the reduction, now 24.6)
        // what a caller has to bring room for: 32 parts, or what tiles of 192 on single CTAs would be split into where those are the
        // natural ones (widths that a 256-wide tile does not fill), or none where K is split only because of the narrower tiles
        int least = one_wave ? 1 : min(splits, 32);
        if ((n > 192 && n < 256) || (kc <= 2304 && n % 192 == 0 && n % 256 != 0))
            least = min(least, tiles192 * 2 <= sms ? max(1, min((int)(sms / tiles192), g.kt_total / 4)) : 1);
        const size_t part = (size_t)m * n * sizeof(float);
        if (splits > least && splits * part > scratch) splits = (int)max((size_t)least, scratch / part);
    }
    g.kt_per_split = (int)ceil_div(g.kt_total, splits);
    g.splits = (int)ceil_div(g.kt_total, g.kt_per_split);
    return g;
}

static bool ensure_device_ok()
{
    static int ok[kMaxDevices];   // 0 unknown, 1 yes, -1 no
    const int dev = current_device();
    if (dev < 0) return false;
    std::lock_guard<std::mutex> hold(g_dev_lock);
    if (!ok[dev]) {
        int major = 0;
        ok[dev] = (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess && major == 10) ? 1 : -1;
    }
    return ok[dev] == 1;
}

template <int BN, class Job2>
static mxfp4_status_t launch_gemm_pair(const PairJob &one, const Job2 &two, int grid, cudaStream_t st)
{
    using C = Gemm2Cfg<BN>;
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_pair<BN, Job2>, C::kSmemBytes));
    MX_CHECK_CUDA(launch_pdl(k_gemm_mxf4_pair<BN, Job2>, (unsigned)grid, 1, kGemmThreads, C::kSmemBytes, st, one, two));
    return MXFP4_OK;
}

template <int KT, int AS>
static mxfp4_status_t launch_gemm_pbs(const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &msa, const CUtensorMap &msb,
                                      const CUtensorMap &md, const CUtensorMap &mdw, const GemmParams &p, int grid, cudaStream_t st)
{
    using C = GemmPbsCfg<KT, AS>;
    if (p.kt_total > KT) return MXFP4_INVALID_ARG;   // the resident block holds KT K tiles
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_pbs<KT, AS>, C::kSmemBytes));
    MX_CHECK_CUDA(launch_pdl(k_gemm_mxf4_pbs<KT, AS>, (unsigned)grid, 1, kGemmThreads, C::kSmemBytes, st, ma, mb, msa, msb, md, mdw, p));
    return MXFP4_OK;
}

template <int BN, int KT, int AS>
static mxfp4_status_t launch_gemm_bs(const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &md, const CUtensorMap &mdw,
                                     const GemmParams &p, int grid, cudaStream_t st)
{
    using C = GemmBsCfg<BN, KT, AS>;
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_bs<BN, KT, AS>, C::kSmemBytes));
    MX_CHECK_CUDA(launch_pdl(k_gemm_mxf4_bs<BN, KT, AS>, (unsigned)grid, 1, kGemmThreads, C::kSmemBytes, st, ma, mb, md, mdw, p));
    return MXFP4_OK;
}

static mxfp4_status_t launch_gemm_ck(const CUtensorMap &ma, const CUtensorMap &mb, const GemmParams &p, int tiles, int cluster,
                                     cudaStream_t st)
{
    using C = GemmCkCfg;
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_ck, C::kSmemBytes));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * cluster));
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = C::kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    MX_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k_gemm_mxf4_ck, ma, mb, p));
    MX_LAUNCHED();
    return MXFP4_OK;
}

template <int BN, class Job2>
static mxfp4_status_t launch_gemm(const GemmJob &one, const Job2 &two, int grid, cudaStream_t st)
{
    using C = GemmCfg<BN>;
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4<BN, Job2>, C::kSmemBytes));
    MX_CHECK_CUDA(launch_pdl(k_gemm_mxf4<BN, Job2>, (unsigned)grid, 1, kGemmThreads, C::kSmemBytes, st, one, two));
    return MXFP4_OK;
}

// Everything gemm() checks before it enqueues anything, without enqueuing anything: callers that launch other kernels
// first (the linear layer) ask here so that an error leaves the stream untouched.  allow_split = false: plan without
// split-K (no workspace needed).
mxfp4_status_t gemm_check(mxfp4_mat_t a, mxfp4_mat_t b, const void *d, int64_t ldd, int out_dtype, const void *bias,
                          const void *workspace, size_t workspace_bytes, bool allow_split)
{
    if (!a.data || !a.scales || !b.data || !b.scales || !d) return MXFP4_INVALID_ARG;
    if (out_dtype != MXFP4_OUT_BF16 && out_dtype != MXFP4_OUT_FP32) return MXFP4_INVALID_ARG;
    if (a.rows < 0 || b.rows < 0 || a.cols < 0) return MXFP4_INVALID_ARG;
    if (a.cols != b.cols || a.cols % 32 != 0 || b.rows % 8 != 0 || ldd < b.rows) return MXFP4_BAD_SHAPE;
    const int esz = out_dtype == MXFP4_OUT_FP32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(a.data) | reinterpret_cast<uintptr_t>(b.data) | reinterpret_cast<uintptr_t>(a.scales) |
         reinterpret_cast<uintptr_t>(b.scales) | reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(bias)) & 15u)
        return MXFP4_MISALIGNED;
    if ((ldd * esz) % 16 != 0) return MXFP4_MISALIGNED;
    const int64_t M = a.rows, N = b.rows, Kc = a.cols;
    if (M == 0 || N == 0) return MXFP4_OK;
    if (!ensure_device_ok()) return MXFP4_UNSUPPORTED_DEVICE;
    if (Kc == 0) return MXFP4_BAD_SHAPE;
    const GemmPlan g = plan_gemm(M, N, Kc, sm_count(), allow_split, workspace ? workspace_bytes : 0);
    const size_t need = g.splits > 1 ? (size_t)g.splits * M * N * sizeof(float) : 0;
    if (need > 0 && (!workspace || workspace_bytes < need)) return MXFP4_WORKSPACE_TOO_SMALL;
    if (need > 0 && (reinterpret_cast<uintptr_t>(workspace) & 15u)) return MXFP4_MISALIGNED;
    return MXFP4_OK;
}

// The divisors of the tile numbering and, for the B-stationary kernels, how `rows` row tiles (of one CTA or of a pair) are shared by
// `workers`: the smallest number of rounds for which the rest, the rows behind those that the rounds reach, keeps the left-over
// workers no longer than that.  A change of column costs them about a tile (with that left out, 50432 x 2304 x 768 took
// 54 us, its two left-over pairs the last to finish; 49 with one round more and no rest).
static void set_walk(GemmParams &p, int workers = 1, int rows = 1)
{
    p.by_splits = fast_div(p.splits);
    p.by_tiles_n = fast_div(p.tiles_n);
    p.rows = rows;
    p.abreast = workers / p.tiles_n;
    const int rest_workers = workers - p.abreast * p.tiles_n;
    int64_t rest = (int64_t)rows * p.tiles_n;
    p.rounds = 0;
    p.rest_row0 = 0;
    if (p.abreast > 0) {
        for (p.rounds = (int)((rest - 1) / workers); p.rest_row0 < rows; p.rounds++) {
            p.rest_row0 = min(rows, (p.rounds + 1) * p.abreast);
            rest = (int64_t)(rows - p.rest_row0) * p.tiles_n;
            if (rest_workers > 0 && ceil_div(rest, rest_workers) + p.tiles_n / rest_workers - 1 <= p.rounds + 1) { p.rounds++; break; }
        }
    }
    p.by_rest_rows = fast_div(max(1, rows - p.rest_row0));
    p.by_rest_workers = fast_div(max(1, rest_workers));
    p.share = rest_workers ? (int)(rest / rest_workers) : 0;
    p.extra = rest_workers ? (int)(rest % rest_workers) : 0;
}

// The maps and parameters of one product with plan g.  spin_limit / withhold_loads: see GemmParams (normal use: kWaitSpinLimit, 0).
static bool make_job(PairJob &job, const GemmPlan &g, mxfp4_mat_t a, mxfp4_mat_t b, void *d, int64_t ldd, int out_dtype, const void *bias, void *workspace,
                     uint32_t *dev_status, uint32_t spin_limit, int withhold_loads)
{
    const int64_t M = a.rows, N = b.rows, Kc = a.cols;
    const bool store_fp32 = g.splits > 1 || out_dtype == MXFP4_OUT_FP32;
    GemmParams &p = job.p;
    p.sfa = a.scales; p.sfb = b.scales;
    p.M = M; p.N = N; p.Kc = Kc;
    p.nblk4 = (int)ceil_div(Kc / 32, 4);
    p.rbA = (int)ceil_div(M, 128); p.rbB = (int)ceil_div(N, 128);
    p.tiles_m = g.tiles_m; p.tiles_n = g.tiles_n; p.splits = g.splits;
    p.kt_total = g.kt_total; p.kt_per_split = g.kt_per_split;
    p.head = 0;
    p.out_fp32 = store_fp32;
    p.bias = static_cast<const __nv_bfloat16 *>(bias);
    p.dev_status = dev_status;
    p.d = d;
    p.ldd = ldd;
    p.spin_limit = spin_limit;
    p.withhold_loads = withhold_loads;
    set_walk(p);
    if (!make_operand_map(&job.a, a.data, M, Kc, kBM) || !make_operand_map(&job.b, b.data, N, Kc, g.pbs ? 96 : g.pair ? g.bn / 2 : g.bn) ||
        !make_output_map(&job.d, g.splits > 1 ? workspace : d, M, N, g.splits > 1 ? N : ldd, g.splits, store_fp32))
        return false;
    if ((g.pair || g.pbs) && (!make_scale_map(&job.sfa, a.scales, M, Kc, 1) || !make_scale_map(&job.sfb, b.scales, N, Kc, 2))) return false;
    job.dw = job.d;
    return store_fp32 || make_output_map_wide(&job.dw, d, M, N, ldd);
}

static mxfp4_status_t launch_splitk_reduce(const GemmPlan &g, const void *workspace, int64_t M, int64_t N, void *d, int64_t ldd, int out_dtype,
                                           const void *bias, int sms, cudaStream_t st)
{
    const int groups = g.splits >= 8 && M * N / 4 < 64 * 256 ? 8 : 1;   // fewer than 64 blocks otherwise
    const int64_t nb4 = ceil_div(M * N / 4, 256 / groups);
    const unsigned blocks = (unsigned)(nb4 < (int64_t)sms * 8 ? nb4 : (int64_t)sms * 8);
    MX_CHECK_CUDA(launch_pdl(groups == 8 ? k_splitk_reduce<8> : k_splitk_reduce<1>, blocks, 1, 256, 0, st, static_cast<const float *>(workspace),
                             g.splits, M, N, d, ldd, (int)(out_dtype == MXFP4_OUT_FP32), static_cast<const __nv_bfloat16 *>(bias)));
    return MXFP4_OK;
}

static mxfp4_status_t gemm_impl(mxfp4_mat_t a, mxfp4_mat_t b, void *d, int64_t ldd, int out_dtype, const void *bias, void *workspace,
                                size_t workspace_bytes, uint32_t *dev_status, cudaStream_t st, bool allow_split, uint32_t spin_limit,
                                int withhold_loads)
{
    const mxfp4_status_t chk = gemm_check(a, b, d, ldd, out_dtype, bias, workspace, workspace_bytes, allow_split);
    if (chk) return chk;
    const int64_t M = a.rows, N = b.rows;
    if (M == 0 || N == 0) return MXFP4_OK;
    const int sms = sm_count();
    const GemmPlan g = plan_gemm(M, N, a.cols, sms, allow_split, workspace ? workspace_bytes : 0);
    PairJob job;
    if (!make_job(job, g, a, b, d, ldd, out_dtype, bias, workspace, dev_status, spin_limit, withhold_loads)) return MXFP4_CUDA_ERROR;
    GemmParams &p = job.p;
    if (g.ck) {
        p.splits = g.ck;
        return launch_gemm_ck(job.a, job.b, p, g.tiles_m * g.tiles_n, g.ck, st);
    }
    const bool paired = g.pair || g.pbs;
    const int rows = paired ? (g.tiles_m + 1) / 2 : g.tiles_m, workers = paired ? sms / 2 : sms;
    const int items = min(workers, rows * g.tiles_n * g.splits), grid = paired ? 2 * items : items;
    set_walk(p, items, rows);
    const mxfp4_status_t s = g.pbs         ? launch_gemm_pbs<4, 8>(job.a, job.b, job.sfa, job.sfb, job.d, job.dw, p, grid, st)
                             : g.bs == 1   ? launch_gemm_bs<192, 2, 7>(job.a, job.b, job.d, job.dw, p, grid, st)
                             : g.pair      ? (g.bn == 192 ? launch_gemm_pair<192>(job, NoJob{}, grid, st) : launch_gemm_pair<256>(job, NoJob{}, grid, st))
                             : g.bn == 256 ? launch_gemm<256>(job, NoJob{}, grid, st)
                             : g.bn == 192 ? launch_gemm<192>(job, NoJob{}, grid, st)
                                           : launch_gemm<128>(job, NoJob{}, grid, st);
    if (s || g.splits == 1 || withhold_loads) return s;
    return launch_splitk_reduce(g, workspace, M, N, d, ldd, out_dtype, bias, sms, st);
}

// The CTAs that share the quantization of a row block, for a forward pass in one launch; 0: not in one launch.  What one launch saves is
// host time, so it is for eager calls: in a row 13.0-13.3 us with two launches, 10.4 with one, at all sizes here.  The kernel itself is
// slower than the two it replaces, and a graph takes those two.  Two launches / one, from the call to its synchronized result and (device
// time) of calls that queue behind other work, in us, clusters of c:
//   197 x 1536 x 384 22.6 / 23.0 (5.8 / 7.2) c = 3, 23.5 (7.6) c = 4, 23.5 (7.7) c = 2, 24.4 (8.5) c = 1
//   1 x 1536 x 384 22.1 / 21.6 (5.0 / 5.6) c = 3, 22.8 (6.9) c = 1;  128 x 1024 x 384 22.5 / 23.5 (5.8 / 7.6) c = 2
//   197 x 1152 x 256 22.2 / 21.8 (5.3 / 6.0) c = 3;  300 x 640 x 256 22.2 / 22.6 (5.4 / 6.8) c = 1, x 128 21.5 (5.3 / 5.6)
//   3136 x 384 x 96 22.7 / 21.4 (5.9 / 5.4) c = 3
// Beyond: 197 x 1536 x 448 22.7 / 23.6 (5.9 / 7.6), x 512 22.7 / 23.8 (5.8 / 7.8), both c = 3, 128 x 1024 x 512 22.6 / 24.3 (5.6 / 8.5) c = 2.  Taken while
// a synchronized call loses no more than a microsecond: contractions of at most 384 and three groups of X per thread (a chain of loads).
// Three CTAs share best.  Clusters of three fit on the GPU 45 at once (the SMs left over in its partitions make none): a second wave costs
// 27.8 (11.7) instead of 23.1 (7.0) at 2048 x 1152 x 256 (144 tiles), so they are taken up to six sevenths of the SMs (126 tiles: 784 x 2304 x 384 23.4,
// c = 2 23.9).  Pairs fit on all SMs.
static int x_cluster(int64_t m, int64_t n, int64_t kc, int sms)
{
    const int64_t tiles_n = ceil_div(n, 128), tiles = ceil_div(m, kBM) * tiles_n;
    if (m <= 0 || n <= 0 || kc <= 0 || kc > 384 || tiles > sms) return 0;
    const int c = tiles_n % 3 == 0 && 7 * tiles <= 6 * sms ? 3 : tiles_n % 2 == 0 ? 2 : 1;
    return kBM * ceil_div(kc, 128) * 4 <= 3 * kXQuantThreads * c ? c : 0;
}
bool gemm_from_x_fits(int64_t m, int64_t n, int64_t kc, cudaStream_t st)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    return x_cluster(m, n, kc, sm_count()) > 0 && cudaStreamIsCapturing(st, &capture) == cudaSuccess && capture == cudaStreamCaptureStatusNone;
}

// Y = Q1(X) b^T in one launch; xq receives Q1(X).  The caller has checked every argument, and that it fits.
mxfp4_status_t gemm_from_x(const void *x, int64_t ldx, const mxfp4_mat_t &xq, const mxfp4_mat_t &b, void *y, int64_t ldy, const void *bias, int scale_mode,
                           uint32_t *dev_status, cudaStream_t st, uint32_t spin_limit, int withhold_loads)
{
    const int64_t M = xq.rows, N = b.rows, Kc = xq.cols;
    GemmParams p;
    p.sfa = nullptr; p.sfb = b.scales;
    p.M = M; p.N = N; p.Kc = Kc;
    p.nblk4 = (int)ceil_div(Kc / 32, 4);
    p.rbA = (int)ceil_div(M, 128); p.rbB = (int)ceil_div(N, 128);
    p.tiles_m = p.rbA; p.tiles_n = p.rbB; p.splits = 1;
    p.kt_total = p.kt_per_split = (int)ceil_div(Kc, kBKElems);
    p.head = 0;
    p.out_fp32 = 0;
    p.bias = static_cast<const __nv_bfloat16 *>(bias);
    p.dev_status = dev_status;
    p.d = y;
    p.ldd = ldy;
    p.spin_limit = spin_limit;
    p.withhold_loads = withhold_loads;
    set_walk(p);
    CUtensorMap mb, md, mdw;
    if (!make_operand_map(&mb, b.data, N, Kc, 128) || !make_output_map(&md, y, M, N, ldy, 1, false) || !make_output_map_wide(&mdw, y, M, N, ldy)) return MXFP4_CUDA_ERROR;
    const XSource x_ = {static_cast<const __nv_bfloat16 *>(x), ldx, static_cast<uint8_t *>(xq.data), xq.scales, scale_mode, x_cluster(M, N, Kc, sm_count())};
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_x, kXSmemBytes));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.tiles_m * p.tiles_n));
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = kXSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)x_.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    MX_CHECK_CUDA(cudaLaunchKernelEx(&cfg, k_gemm_mxf4_x, mb, md, mdw, p, x_));
    MX_LAUNCHED();
    return MXFP4_OK;
}

enum class TwoKind { kSeparate, kOneWave, kPairs };

// The plans of two products (rows m1, m2, contractions kc1, kc2, n columns each) that may share a launch, if its partial sums fit into
// `scratch` bytes.
static TwoKind plan_two(int64_t m1, int64_t kc1, int64_t m2, int64_t kc2, int64_t n, int sms, size_t scratch, GemmPlan &g1, GemmPlan &g2)
{
    g1 = plan_gemm(m1, n, kc1, sms, true, scratch);
    g2 = plan_gemm(m2, n, kc2, sms, true, scratch);
    const auto single = [](const GemmPlan &g) { return !g.pair && !g.pbs && !g.bs && !g.ck; };
    if (single(g1) && single(g2) && g1.bn == 128 && g2.bn == 128 && g1.splits == 1 && g2.splits == 1 &&
        g1.tiles_m * g1.tiles_n + g2.tiles_m * g2.tiles_n <= sms)
        return TwoKind::kOneWave;
    const GemmPlan own = g1;
    if (g1.ck && g2.splits == 1 && (g2.pair || single(g2))) {
        // CTA pairs with four partial sums in place of the cluster kernel's two pairs of accumulators: chains of the same length, and in one
        // launch with the other product faster in spite of the sums' way through L2 (both products, in us: 25216, 768, 1536 46.7 -> 35.5;
        // 6272, 768, 2304 33.9 -> 30.4; 4096, 768, 1536 20.6 -> 16.7; 100352, 768, 2304 182 -> 171; 50432, 768, 2304 89 -> 87)
        g1.ck = 0;
        g1.pair = true;
        g1.bn = g2.pair ? g2.bn : 256;
        g1.tiles_n = (int)ceil_div(n, g1.bn);
        g1.kt_per_split = (int)ceil_div(g1.kt_total, 4);
        g1.splits = (int)ceil_div(g1.kt_total, g1.kt_per_split);
    }
    // A product on single CTAs joins the other one's pairs, and the second takes the width of the first (192 only where 256 gives as
    // many columns): its sums stay as they are.  Widths up to 128 and the B-stationary kernels keep their own launch.
    const int width = g1.pair ? g1.bn : g2.pair && g2.splits == 1 ? g2.bn : 0;
    const auto join = [&](GemmPlan &g) {
        if (!(single(g) || g.pair) || g.splits != 1 || n <= 128) return;
        g.pair = true;
        g.bn = width;
        g.tiles_n = (int)ceil_div(n, width);
    };
    if (width) {
        if (!g1.pair) join(g1);
        join(g2);
    }
    if (g1.pair && g2.pair && g1.bn == g2.bn && g2.splits == 1 && (g1.splits == 1 || (size_t)g1.splits * m1 * n * sizeof(float) <= scratch))
        return TwoKind::kPairs;
    g1 = own;
    return TwoKind::kSeparate;
}

// The two products of a backward pass, d1 = a1 b1^T and d2 = a2 b2^T: in one launch where all their 128-wide tiles fit on the SMs, or
// where one runs on CTA pairs and the other can (the second not split); else one after the other.  One launch pays once for filling and
// draining the machine and lets the second product's tiles fill the pairs that the first one leaves idle (64 items of 197 K tiles
// on 74 pairs).  Both together, back to back, in us (rows, columns of X and of dY): 1024, 192, 768 9.6 -> 5.3; 2048, 384, 768
// 12.7 -> 8.2; 4096, 768, 3072 26.9 -> 21.7; 25216, 384, 1536 41 -> 30; 8192, 2048, 2048 39 -> 33; 50432, 1024, 4096 189 -> 174.
// spin_limit / withhold_loads: see GemmParams; the self-test runs the joint launch alone.
static mxfp4_status_t gemm_two_impl(mxfp4_mat_t a1, mxfp4_mat_t b1, void *d1, int64_t ldd1, int dtype1, mxfp4_mat_t a2, mxfp4_mat_t b2, void *d2, int64_t ldd2,
                                    int dtype2, void *workspace, size_t workspace_bytes, uint32_t *dev_status, cudaStream_t st, uint32_t spin_limit,
                                    int withhold_loads)
{
    mxfp4_status_t s;
    if ((s = gemm_check(a1, b1, d1, ldd1, dtype1, nullptr, workspace, workspace_bytes, true)) ||
        (s = gemm_check(a2, b2, d2, ldd2, dtype2, nullptr, workspace, workspace_bytes, true)))
        return s;
    if (a1.rows > 0 && b1.rows > 0 && a2.rows > 0 && b2.rows > 0) {
        const int sms = sm_count();
        GemmPlan g1, g2;
        const TwoKind kind = plan_two(a1.rows, a1.cols, a2.rows, a2.cols, b1.rows, sms, workspace ? workspace_bytes : 0, g1, g2);
        if (kind != TwoKind::kSeparate) {
            PairJob j1, j2;
            if (!make_job(j1, g1, a1, b1, d1, ldd1, dtype1, nullptr, workspace, dev_status, spin_limit, withhold_loads) ||
                !make_job(j2, g2, a2, b2, d2, ldd2, dtype2, nullptr, nullptr, dev_status, spin_limit, withhold_loads))
                return MXFP4_CUDA_ERROR;
            if (kind == TwoKind::kOneWave) return launch_gemm<128, GemmJob>(j1, j2, g1.tiles_m * g1.tiles_n + g2.tiles_m * g2.tiles_n, st);
            const int items = (g1.tiles_m + 1) / 2 * g1.tiles_n * g1.splits + (g2.tiles_m + 1) / 2 * g2.tiles_n, workers = min(sms / 2, items);
            const bool first = g1.kt_per_split >= g2.kt_per_split;
            PairJob &a = first ? j1 : j2, &b = first ? j2 : j1;
            // an item costs its K tiles and, where the epilogue is not hidden, about three more (without the head start
            // 50432 x 1024 x 4096 takes 183 us)
            const int tile = g1.bn == 256 ? 3 : 1, ka = a.p.kt_per_split + tile, kb = b.p.kt_per_split + tile;
            b.p.head = (ka + kb / 2) / kb;
            if ((s = g1.bn == 256 ? launch_gemm_pair<256>(a, b, 2 * workers, st) : launch_gemm_pair<192>(a, b, 2 * workers, st))) return s;
            return g1.splits > 1 && !withhold_loads ? launch_splitk_reduce(g1, workspace, a1.rows, b1.rows, d1, ldd1, dtype1, nullptr, sms, st) : MXFP4_OK;
        }
    }
    if (withhold_loads) return MXFP4_OK;
    if ((s = gemm_impl(a1, b1, d1, ldd1, dtype1, nullptr, workspace, workspace_bytes, dev_status, st, true, kWaitSpinLimit, 0))) return s;
    return gemm_impl(a2, b2, d2, ldd2, dtype2, nullptr, workspace, workspace_bytes, dev_status, st, true, kWaitSpinLimit, 0);
}

mxfp4_status_t gemm_two(mxfp4_mat_t a1, mxfp4_mat_t b1, void *d1, int64_t ldd1, int dtype1, mxfp4_mat_t a2, mxfp4_mat_t b2, void *d2, int64_t ldd2, int dtype2,
                        void *workspace, size_t workspace_bytes, uint32_t *dev_status, cudaStream_t st)
{
    return gemm_two_impl(a1, b1, d1, ldd1, dtype1, a2, b2, d2, ldd2, dtype2, workspace, workspace_bytes, dev_status, st, kWaitSpinLimit, 0);
}

mxfp4_status_t gemm(mxfp4_mat_t a, mxfp4_mat_t b, void *d, int64_t ldd, int out_dtype, const void *bias, void *workspace,
                    size_t workspace_bytes, uint32_t *dev_status, cudaStream_t st, bool allow_split)
{
    return gemm_impl(a, b, d, ldd, out_dtype, bias, workspace, workspace_bytes, dev_status, st, allow_split, kWaitSpinLimit, 0);
}

// bf16 matrix [m, n] (leading dimension ld) as a 2-D tensor; box = 64 columns x 128 rows, 128B swizzle: one half of the
// quantizing kernel's tile.
static bool make_tile_map_bf16(CUtensorMap *map, void *d, int64_t m, int64_t n, int64_t ld)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)n, (cuuint64_t)m};
    cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, d, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// packed transposed codes [n, m / 2 bytes]; box = 64 bytes x 128 rows, 64B swizzle (the column pass's staging tile)
static bool make_codes_t_map(CUtensorMap *map, void *packed, int64_t m, int64_t n)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)(m / 2), (cuuint64_t)n};
    cuuint64_t gstride[1] = {(cuuint64_t)(m / 2)};
    cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, packed, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
              CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static QuantSide make_quant_side(const mxfp4_mat_t &m, const mxfp4_qparams_t &qp)
{
    QuantSide s;
    s.packed = static_cast<uint8_t *>(m.data);
    s.scales = m.scales;
    s.nblk4 = (int)ceil_div(m.cols / 32, 4);
    s.scale_mode = qp.scale_mode;
    s.sr = make_sr_stream(qp.seed, qp.stream_id, m.rows * m.cols);
    return s;
}

template <bool SR_ROW, bool SR_T, bool DQ, bool WITH_Y, int GROUPS>
static mxfp4_status_t launch_gemm_q(const CUtensorMap &ma, const CUtensorMap &mb, const CUtensorMap &my, const CUtensorMap &mz,
                                    const CUtensorMap &mx_, const CUtensorMap &mt, const GemmParams &p, const QuantEpilogue &e, int grid,
                                    cudaStream_t st)
{
    using C = GemmQCfg<GROUPS, WITH_Y && GROUPS == 1 ? 3 : 2>;
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_gemm_mxf4_q<SR_ROW, SR_T, DQ, WITH_Y, GROUPS>, C::kSmemBytes));
    MX_CHECK_CUDA(launch_pdl(k_gemm_mxf4_q<SR_ROW, SR_T, DQ, WITH_Y, GROUPS>, (unsigned)grid, 1, C::kThreads, C::kSmemBytes, st, ma, mb, my, mz, mx_, mt, p, e));
    return MXFP4_OK;
}

static bool valid_qp(const mxfp4_qparams_t &qp)
{
    return (qp.scale_mode == MXFP4_SCALE_TRUNCATION_FREE || qp.scale_mode == MXFP4_SCALE_FLOOR) &&
           (qp.rounding == MXFP4_ROUND_NEAREST || qp.rounding == MXFP4_ROUND_STOCHASTIC);
}

// Everything gemm_quant() checks, without enqueuing anything.
mxfp4_status_t gemm_quant_check(mxfp4_mat_t a, mxfp4_mat_t b, const void *bias, const mxfp4_epilogue_t *epi)
{
    if (!epi || !a.data || !a.scales || !b.data || !b.scales) return MXFP4_INVALID_ARG;
    if (a.rows < 0 || b.rows < 0 || a.cols < 0) return MXFP4_INVALID_ARG;
    if (epi->hook != MXFP4_HOOK_IDENTITY && epi->hook != MXFP4_HOOK_GELU && epi->hook != MXFP4_HOOK_MULTIPLY) return MXFP4_INVALID_ARG;
    const int64_t M = a.rows, N = b.rows, Kc = a.cols;
    const bool row = epi->zq.data != nullptr, tr = epi->zq_t.data != nullptr;
    if (!row && !tr && !epi->y_bf16 && !epi->z_bf16) return MXFP4_INVALID_ARG;
    if (epi->chain && !(row && tr)) return MXFP4_INVALID_ARG;
    if (epi->hook == MXFP4_HOOK_MULTIPLY && !epi->aux_bf16) return MXFP4_INVALID_ARG;
    if ((row && (!epi->zq.scales || !valid_qp(epi->qp_row))) || (tr && (!epi->zq_t.scales || !valid_qp(epi->qp_t)))) return MXFP4_INVALID_ARG;
    if (a.cols != b.cols || Kc % 32 != 0 || N % 32 != 0 || (tr && M % 32 != 0)) return MXFP4_BAD_SHAPE;
    if (M > 0x7FFFFF80 || N > 0x7FFFFF80) return MXFP4_BAD_SHAPE;
    if (row && (epi->zq.rows != M || epi->zq.cols != N)) return MXFP4_BAD_SHAPE;
    if (tr && (epi->zq_t.rows != N || epi->zq_t.cols != M)) return MXFP4_BAD_SHAPE;
    if ((epi->y_bf16 && epi->ldy < N) || (epi->z_bf16 && epi->ldz < N) || (epi->hook == MXFP4_HOOK_MULTIPLY && epi->ld_aux < N)) return MXFP4_BAD_SHAPE;
    uintptr_t bits = reinterpret_cast<uintptr_t>(a.data) | reinterpret_cast<uintptr_t>(b.data) | reinterpret_cast<uintptr_t>(a.scales) |
                     reinterpret_cast<uintptr_t>(b.scales) | reinterpret_cast<uintptr_t>(bias) | reinterpret_cast<uintptr_t>(epi->y_bf16) |
                     reinterpret_cast<uintptr_t>(epi->z_bf16);
    if (epi->hook == MXFP4_HOOK_MULTIPLY) bits |= reinterpret_cast<uintptr_t>(epi->aux_bf16);
    if (row) bits |= reinterpret_cast<uintptr_t>(epi->zq.data) | reinterpret_cast<uintptr_t>(epi->zq.scales);
    if (tr) bits |= reinterpret_cast<uintptr_t>(epi->zq_t.data) | reinterpret_cast<uintptr_t>(epi->zq_t.scales);
    if (bits & 15u) return MXFP4_MISALIGNED;
    if ((epi->y_bf16 && epi->ldy % 8) || (epi->z_bf16 && epi->ldz % 8) || (epi->hook == MXFP4_HOOK_MULTIPLY && epi->ld_aux % 8)) return MXFP4_MISALIGNED;
    if (M == 0 || N == 0) return MXFP4_OK;
    if (!ensure_device_ok()) return MXFP4_UNSUPPORTED_DEVICE;
    if (Kc == 0) return MXFP4_BAD_SHAPE;
    return MXFP4_OK;
}

mxfp4_status_t quantize_gelu_chain(const void *y_bf16, int64_t rows, int64_t cols, int64_t ldy, void *z_bf16, int64_t ldz, mxfp4_mat_t dst,
                                   const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t, const mxfp4_qparams_t *qp_t, uint32_t *dev_status, cudaStream_t st);

// Whether two groups of epilogue warps take the tiles in turn.  Where the epilogue is bound by the instructions it issues, eight warps
// with their waits for the accumulator and for one another do not fill the SM.  The second group's tiles and staging cost the ring two
// of its four stages, so the contraction has to be short, and the shorter the less the epilogue does; the groups have to fit (GemmQCfg),
// and a block needs a second tile.  K tiles of 256 up to which two groups are taken, with one group / two, back to back, in us:
//   GELU: 4.  Chain and Y 25216 x 1536 x 384 66.6 / 59.4, x 1024 69.5 / 64.4.  3 where Y and Z are stored, or one of them without a
//     stochastic column pass behind a row pass: Y and a row pass 25216 x 1536 x 768 48.6 / 45.9, x 1024 49.9 / 54.7, Z alone x 1024 45.7 / 50.5.
//   Multiply: 2, as the second factor is loaded too.  A nearest row pass 25216 x 1536 x 512 31.9 / 27.4, x 768 33.7 / 38.4; Z alone
//     48.7 / 36.1, x 1024 48.8 / 54.9.  With both passes stochastic 3: 25216 x 1536 x 768 50.6 / 47.4, x 1024 51.2 / 54.2; without Z, on wide
//     outputs (the SMs share more of the rows that they read) of very many tiles 4: 50432 x 4096 x 1024 271 / 259, 50432 x 3072 x 1024
//     196 / 192, but 12544 x 4096 x 896 (21 tiles per SM) 67.8 / 68.0, 50432 x 768 x 1024 51.2 / 55.0.  With the chain, the longest passes, 4:
//     25216 x 1536 x 1024 99.8 / 97.9.
//   Identity: 2.  Q3 + Q5 25216 x 1536 x 384 43.2 / 42.1, a nearest row pass 25.3 / 21.7, x 768 26.3 / 28.1.  None where Z is stored and at
//     most one pass is made, the stores being the bound: 25216 x 1536 x 384 28.2 / 31.8.
// The short epilogues of these two take one group between two and four tiles per SM, where one of the groups often has a tile more than
// the other: Q3 + Q5 4096 x 1536 x 384 (2.6) 11.7 / 11.9 and 10.9 / 11.1, the chain without a hook 10.8 / 11.2; but 2400 x 1024 x 256 (1.03)
// 8.5 / 8.1 and 7.9 / 7.7, multiply 6272 x 3072 x 768 (8.3) 26.7 / 25.0.
static bool two_groups(const mxfp4_epilogue_t *epi, int64_t M, int64_t N, int64_t Kc)
{
    const bool identity = epi->hook == MXFP4_HOOK_IDENTITY, y = epi->y_bf16 && !(identity && !epi->z_bf16), z = epi->z_bf16 || (identity && epi->y_bf16);
    const int smem_tiles = 1 + (epi->hook == MXFP4_HOOK_MULTIPLY && !epi->chain) + (epi->chain && z) + y;
    const int64_t tiles = ceil_div(M, kBM) * ceil_div(N, 128), sms = sm_count();
    if (smem_tiles > 2 || tiles <= sms) return false;
    const bool row = epi->zq.data != nullptr, tr = epi->zq_t.data != nullptr, both = row && tr;
    const bool sr_row = row && epi->qp_row.rounding == MXFP4_ROUND_STOCHASTIC, sr_t = tr && epi->qp_t.rounding == MXFP4_ROUND_STOCHASTIC;
    int kt;
    if (epi->hook == MXFP4_HOOK_GELU) kt = !(y || z) || (both && sr_t && !(y && z)) ? 4 : 3;
    else if (epi->hook == MXFP4_HOOK_MULTIPLY && epi->chain) kt = 4;
    else if (tiles > 2 * sms && tiles < 4 * sms) kt = 0;
    else if (identity) kt = both || !(y || z) ? 2 : 0;
    else kt = !(sr_row && sr_t) || tiles <= sms * 2 ? 2 : z || N < 3072 || tiles < 32 * sms ? 3 : 4;
    return Kc <= kt * kBKElems;
}

// Whether what the quantization writes lies in memory that the product reads.
static bool over_operands(const mxfp4_epilogue_t *epi, const mxfp4_mat_t &a, const mxfp4_mat_t &b, const void *bias)
{
    const auto codes = [](const mxfp4_mat_t &q) { return span_of(q.data, q.data ? q.rows * (q.cols / 2) : 0); };
    const auto scales = [](const mxfp4_mat_t &q) { return span_of(q.scales, q.data ? (int64_t)mxfp4_scale_bytes(q.rows, q.cols) : 0); };
    const Span in[] = {codes(a), scales(a), codes(b), scales(b), span_of_bf16(bias, 0, 1, b.rows)};
    const Span out[] = {codes(epi->zq), scales(epi->zq), codes(epi->zq_t), scales(epi->zq_t), span_of_bf16(epi->z_bf16, epi->ldz, a.rows, b.rows)};
    for (const Span &i : in)
        for (const Span &o : out)
            if (meet(i, o)) return true;
    return false;
}

// Whether the product and the quantization run as two kernels: when the epilogue is GELU with the double-quantization chain,
// Y is stored anyway, and there are many 128 x 128 tiles per SM.  The fused epilogue's passes are the bottleneck; the two kernels read
// Y back (2 of 5 bytes per element more) but run at the product's and the tile quantizer's own rates.  With one group of epilogue
// warps the line lies at four tiles per SM: fused / two kernels 84 / 64.2 us at 25216 x 1536 x 384, 396 / 307 at 50432 x 4096 x 1024,
// 33.6 / 31.7 at 8192 x 1536 x 384 (5.2 tiles per SM), but 20.6 / 22.5 at 4096 x 1536 x 384 (2.6) and 12.3 / 15.3 at 1024 x 768 x 192,
// where a second launch costs more.  With two groups the two ways are within 2 % of each other from eight to sixteen tiles per SM, at all
// contractions up to 1024, and the line is in the middle (back to back): 24.5 / 27.6 at 9472 x 1536 x 384 (6.0 tiles per SM), 35.3 / 35.3 at 12672
// (8.0), 45.9 / 47.2 at 18944 (12.0), 60.2 / 60.0 at 25216 (16), 91.8 / 88.9 at 38016 (24); x 1024 49.8 / 50.9 (12.0) and 94.5 / 94.2 (24).
// Outputs of the quantization in the operands' memory are in time behind a product of its own: from four tiles per SM on they get one.
static bool two_pass(const mxfp4_epilogue_t *epi, const mxfp4_mat_t &a, const mxfp4_mat_t &b, const void *bias)
{
    const int64_t tiles = ceil_div(a.rows, kBM) * ceil_div(b.rows, 128), sms = sm_count();
    return epi->hook == MXFP4_HOOK_GELU && epi->chain && epi->y_bf16 && epi->y_bf16 != epi->z_bf16 && tiles >= 4 * sms &&
           (tiles >= 12 * sms || !two_groups(epi, a.rows, b.rows, a.cols) || over_operands(epi, a, b, bias));
}

// spin_limit / withhold_loads: see GemmParams; the self-test runs the quantizing kernel alone.
mxfp4_status_t gemm_quant(mxfp4_mat_t a, mxfp4_mat_t b, const void *bias, const mxfp4_epilogue_t *epi, uint32_t *dev_status, cudaStream_t st,
                          uint32_t spin_limit, int withhold_loads)
{
    const mxfp4_status_t chk = gemm_quant_check(a, b, bias, epi);
    if (chk) return chk;
    const int64_t M = a.rows, N = b.rows, Kc = a.cols;
    if (M == 0 || N == 0) return MXFP4_OK;
    const bool row = epi->zq.data != nullptr, tr = epi->zq_t.data != nullptr;
    if (two_pass(epi, a, b, bias)) {
        if (withhold_loads) return MXFP4_BAD_SHAPE;
        // Y by the product's own kernels (the contraction is not split), then the tile quantizer reads it back
        mxfp4_status_t s = gemm(a, b, epi->y_bf16, epi->ldy, MXFP4_OUT_BF16, bias, nullptr, 0, dev_status, st, false);
        if (s) return s;
        return quantize_gelu_chain(epi->y_bf16, M, N, epi->ldy, epi->z_bf16, epi->ldz, epi->zq, &epi->qp_row, epi->zq_t, &epi->qp_t, dev_status, st);
    }
    CUtensorMap ma, mb, my, mz, mx_, mt;
    if (!make_operand_map(&ma, a.data, M, Kc, kBM) || !make_operand_map(&mb, b.data, N, Kc, 128)) return MXFP4_CUDA_ERROR;
    my = mz = mx_ = mt = ma;   // placeholders when the tensors they describe are not asked for
    if (epi->z_bf16 && !make_tile_map_bf16(&mz, epi->z_bf16, M, N, epi->ldz)) return MXFP4_CUDA_ERROR;
    if (tr && !make_codes_t_map(&mt, epi->zq_t.data, M, N)) return MXFP4_CUDA_ERROR;

    GemmParams p;
    p.sfa = a.scales; p.sfb = b.scales;
    p.M = M; p.N = N; p.Kc = Kc;
    p.nblk4 = (int)ceil_div(Kc / 32, 4);
    p.rbA = (int)ceil_div(M, 128); p.rbB = (int)ceil_div(N, 128);
    p.tiles_m = (int)ceil_div(M, kBM); p.tiles_n = (int)ceil_div(N, 128); p.splits = 1;
    p.kt_total = (int)ceil_div(Kc, kBKElems); p.kt_per_split = p.kt_total;
    p.out_fp32 = 0;
    p.bias = static_cast<const __nv_bfloat16 *>(bias);
    p.dev_status = dev_status;
    p.d = nullptr;
    p.ldd = 0;
    p.spin_limit = spin_limit;
    p.withhold_loads = withhold_loads;
    set_walk(p);

    QuantEpilogue e;
    const mxfp4_qparams_t none = {MXFP4_SCALE_TRUNCATION_FREE, MXFP4_ROUND_NEAREST, 0, 0, 0};
    const mxfp4_mat_t nomat = {nullptr, nullptr, 0, 32};
    e.rw = make_quant_side(row ? epi->zq : nomat, row ? epi->qp_row : none);
    e.tr = make_quant_side(tr ? epi->zq_t : nomat, tr ? epi->qp_t : none);
    e.emit_row = row; e.emit_t = tr;
    e.hook = epi->hook;
    e.aux = static_cast<const __nv_bfloat16 *>(epi->aux_bf16); e.ld_aux = epi->ld_aux;
    e.store_y = epi->y_bf16 != nullptr;
    e.store_z = epi->z_bf16 != nullptr;
    if (e.store_y && !make_tile_map_bf16(&my, epi->y_bf16, M, N, epi->ldy)) return MXFP4_CUDA_ERROR;
    if (e.hook == MXFP4_HOOK_IDENTITY && e.store_y && !e.store_z) {
        mz = my;         // Y = Z: one tile, one pair of stores
        e.store_y = 0;
        e.store_z = 1;
    }
    e.aux_tma = 0;
    if (e.hook == MXFP4_HOOK_MULTIPLY) {
        if (!make_tile_map_bf16(&mx_, const_cast<void *>(epi->aux_bf16), M, N, epi->ld_aux)) return MXFP4_CUDA_ERROR;
        e.aux_tma = 1;
    }
    const int items = p.tiles_m * p.tiles_n;
    const int sms = sm_count();
    const int grid = items < sms ? items : sms;
    const bool sr_r = row && epi->qp_row.rounding == MXFP4_ROUND_STOCHASTIC, sr_t = tr && epi->qp_t.rounding == MXFP4_ROUND_STOCHASTIC;
    const int sel = (e.store_y ? 8 : 0) | (epi->chain ? 4 : 0) | (sr_r ? 2 : 0) | (sr_t ? 1 : 0);
    const bool two = two_groups(epi, M, N, Kc);
#define MX_Q_CASE(i, a_, b_, c_, d_) \
    case i: return two ? launch_gemm_q<a_, b_, c_, d_, 2>(ma, mb, my, mz, mx_, mt, p, e, grid, st) : launch_gemm_q<a_, b_, c_, d_, 1>(ma, mb, my, mz, mx_, mt, p, e, grid, st)
    switch (sel) {
    MX_Q_CASE(0, false, false, false, false);
    MX_Q_CASE(1, false, true, false, false);
    MX_Q_CASE(2, true, false, false, false);
    MX_Q_CASE(3, true, true, false, false);
    MX_Q_CASE(4, false, false, true, false);
    MX_Q_CASE(5, false, true, true, false);
    MX_Q_CASE(6, true, false, true, false);
    MX_Q_CASE(7, true, true, true, false);
    MX_Q_CASE(8, false, false, false, true);
    MX_Q_CASE(9, false, true, false, true);
    MX_Q_CASE(10, true, false, false, true);
    MX_Q_CASE(11, true, true, false, true);
    MX_Q_CASE(12, false, false, true, true);
    MX_Q_CASE(13, false, true, true, true);
    MX_Q_CASE(14, true, false, true, true);
    MX_Q_CASE(15, true, true, true, true);
    default: return MXFP4_INVALID_ARG;
    }
#undef MX_Q_CASE
}

// scratch: what there is; the result may be more (then gemm() refuses it) or less.
size_t gemm_workspace_bytes(int64_t m, int64_t n, int64_t kc, size_t scratch)
{
    if (m <= 0 || n <= 0 || kc <= 0) return 0;
    // the same SM count gemm() plans with (148, the B200's, when no device is current)
    const GemmPlan g = plan_gemm(m, n, kc, sm_count(), true, scratch);
    return g.splits > 1 ? (size_t)g.splits * m * n * sizeof(float) : 0;
}

// Workspace for gemm_two()'s partial sums (scratch = 0: the least it takes).
size_t gemm_two_workspace_bytes(int64_t m1, int64_t kc1, int64_t m2, int64_t kc2, int64_t n, size_t scratch)
{
    if (m1 <= 0 || kc1 <= 0 || m2 <= 0 || kc2 <= 0 || n <= 0) return 0;
    GemmPlan g1, g2;
    const bool pairs = plan_two(m1, kc1, m2, kc2, n, sm_count(), scratch, g1, g2) == TwoKind::kPairs;
    const size_t two = pairs && g1.splits > 1 ? (size_t)g1.splits * m1 * n * sizeof(float) : 0;
    const size_t w1 = gemm_workspace_bytes(m1, n, kc1, scratch), w2 = gemm_workspace_bytes(m2, n, kc2, scratch);
    return std::max(two, std::max(w1, w2));
}

// The longest chain of MMAs (64 contraction elements each) that gemm() adds into one accumulator for this shape.
int64_t gemm_chain_mmas(int64_t m, int64_t n, int64_t kc)
{
    if (m <= 0 || n <= 0 || kc <= 0) return 0;
    const GemmPlan g = plan_gemm(m, n, kc, sm_count());
    const int64_t kt = g.ck ? (g.kt_per_split + 1) / 2 : g.kt_per_split;   // the cluster kernel alternates between two accumulators
    const int64_t elems = kt * kBKElems < kc ? kt * kBKElems : kc;
    return ceil_div(elems, 64);
}

}  // namespace mx

extern "C" {

int64_t mxfp4_gemm_chain_mmas(int64_t m, int64_t n, int64_t kc) { return mx::gemm_chain_mmas(m, n, kc); }

mxfp4_status_t mxfp4_mma_issue_ceiling(int32_t bn, int32_t iters, uint32_t *dev_status, void *stream)
{
    if (iters < 1 || iters > (1 << 24) || (bn != 128 && bn != 192 && bn != 256)) return MXFP4_INVALID_ARG;
    if (!mx::ensure_device_ok()) return MXFP4_UNSUPPORTED_DEVICE;
    const int smem = mx::kBM * mx::kBKBytes + bn * mx::kBKBytes + 2 * mx::kSfChunk * (1 + (bn + 127) / 128) + 1024 + 256;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int grid = mx::sm_count();
    if (bn == 128) {
        MX_CHECK_CUDA(cudaFuncSetAttribute(mx::k_mma_ceiling<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        mx::k_mma_ceiling<128><<<grid, 128, smem, st>>>(iters, dev_status);
    } else if (bn == 192) {
        MX_CHECK_CUDA(cudaFuncSetAttribute(mx::k_mma_ceiling<192>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        mx::k_mma_ceiling<192><<<grid, 128, smem, st>>>(iters, dev_status);
    } else {
        MX_CHECK_CUDA(cudaFuncSetAttribute(mx::k_mma_ceiling<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        mx::k_mma_ceiling<256><<<grid, 128, smem, st>>>(iters, dev_status);
    }
    MX_CHECK_LAUNCH();
    return MXFP4_OK;
}

size_t mxfp4_gemm_workspace_bytes(int64_t m, int64_t n, int64_t kc) { return mx::gemm_workspace_bytes(m, n, kc, SIZE_MAX); }

mxfp4_status_t mxfp4_gemm_quant(mxfp4_mat_t a, mxfp4_mat_t b, const void *bias_bf16, const mxfp4_epilogue_t *epi, uint32_t *dev_status,
                                void *stream)
{
    return mx::gemm_quant(a, b, bias_bf16, epi, dev_status, static_cast<cudaStream_t>(stream), mx::kWaitSpinLimit, 0);
}

mxfp4_status_t mxfp4_gemm_wait_selftest(mxfp4_mat_t a, mxfp4_mat_t b, void *d, int64_t ldd, int32_t out_dtype, void *workspace,
                                        size_t workspace_bytes, uint32_t spin_limit, uint32_t *dev_status, void *stream)
{
    if (!dev_status || spin_limit < 128u || spin_limit > (1u << 16)) return MXFP4_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const mxfp4_status_t s = mx::gemm_impl(a, b, d, ldd, out_dtype, nullptr, workspace, workspace_bytes, dev_status, st, true, spin_limit, 1);
    if (s) return s;
    mxfp4_mat_t a2 = a, b2 = b;
    a2.cols = b2.cols = std::min<int64_t>(a.cols, 1536);     // short enough not to be split
    return mx::gemm_two_impl(a, b, d, ldd, out_dtype, a2, b2, d, ldd, out_dtype, workspace, workspace_bytes, dev_status, st, spin_limit, 1);
}

mxfp4_status_t mxfp4_gemm(mxfp4_mat_t a, mxfp4_mat_t b, void *d, int64_t ldd, int32_t out_dtype, const void *bias_bf16,
                          void *workspace, size_t workspace_bytes, uint32_t *dev_status, void *stream)
{
    return mx::gemm(a, b, d, ldd, out_dtype, bias_bf16, workspace, workspace_bytes, dev_status, static_cast<cudaStream_t>(stream), true);
}

}  // extern "C"
