// MX quantizer kernels for sm_100a: row-wise, transposed / two-axis (a persistent TMA-fed tile kernel), double
// quantization of a packed source, Q-EMA, dequantize.  Element passes over HBM: scales are written straight into the
// 128x4 tiled order the GEMM consumes.
#include "common.cuh"
#include "quant_tile.cuh"
#include "tma.cuh"

namespace mx {

// ------------------------------------------------------------------------------------------------
// Row-wise quantizer: one thread per 32-element group (Eq. 1 with 1x32 groups).  The grid covers the scale buffer, rows up to
// a multiple of 128 and blocks up to a multiple of 4: a thread outside the matrix writes the padding entry 0x7F (= scale 1),
// so that ragged shapes take one launch (a launch of its own for the padding took 1.6 us at 197 rows and 3.1 us at 19700 x 768
// of the 12 and 15 us of the whole quantization with the gaps around it).
// ------------------------------------------------------------------------------------------------
template <int ROUNDING>
__global__ void __launch_bounds__(256) k_quantize_rows(const __nv_bfloat16 *src, int64_t rows, int nblk,
                                                       int64_t ld, uint8_t *__restrict__ packed,
                                                       uint8_t *__restrict__ scales, int nblk4, int scale_mode,
                                                       const SrStream sr, uint32_t *dev_status)
{
    pdl_launch_dependents();
    pdl_wait();
    const uint64_t gid = blockIdx.x * (uint64_t)256 + threadIdx.x;
    const uint32_t nb_pad = (uint32_t)nblk4 * 4u;
    const int64_t row = (gid >> 32) ? (int64_t)(gid / nb_pad) : (int64_t)((uint32_t)gid / nb_pad);
    const int blk = (int)(gid - (uint64_t)row * nb_pad);
    if (row >= rows || blk >= nblk) {
        scales[scale_offset(row, blk, nblk4)] = 0x7F;
        return;
    }
    const uint4 *p = reinterpret_cast<const uint4 *>(src + row * ld + blk * 32);
    uint4 q[4];
#pragma unroll
    for (int j = 0; j < 4; j++) q[j] = ld_stream_16(p + j);
    const uint32_t am = group_amax(q);
    uint4 out = make_uint4(0, 0, 0, 0);
    uint32_t byte;
    if (am >= 0x7F80u) {
        byte = 0xFFu;
        if (dev_status) atomicOr(dev_status, MXFP4_DEV_NONFINITE);
    } else {
        byte = scale_byte_from_amax(am, tf_add_of(scale_mode));
        const uint32_t inv = inv_scale_bf16x2(byte);
        if (ROUNDING == MXFP4_ROUND_NEAREST) {
            out = make_uint4(rne8(q[0], inv), rne8(q[1], inv), rne8(q[2], inv), rne8(q[3], inv));
        } else {
            const uint64_t q0 = ((uint64_t)row * ((uint64_t)nblk * 32) + (uint64_t)blk * 32) >> 4;
            uint4 ra, rb;
            sr_words_two(sr, q0, q0 + 1, ra, rb);
            out.x = sr8(q[0], inv, ra.x, ra.y);
            out.y = sr8(q[1], inv, ra.z, ra.w);
            out.z = sr8(q[2], inv, rb.x, rb.y);
            out.w = sr8(q[3], inv, rb.z, rb.w);
        }
    }
    *reinterpret_cast<uint4 *>(packed + row * ((int64_t)nblk * 16) + blk * 16) = out;
    scales[scale_offset(row, blk, nblk4)] = (uint8_t)byte;
}

// ------------------------------------------------------------------------------------------------
// Double quantization (Sec. 3.3) of an MXFP4 matrix along its other axis: Q4 and Q6 of Eq. 4-5.  A CTA owns a
// 128-row x 128-column tile of the packed source, which is exactly one 512-byte chunk of the tiled scale buffer of
// the source and of the output.  The tile is dequantized exactly into shared memory as bf16 on the way in, then the
// column pass re-quantizes it: a thread takes 16 consecutive rows of 4 columns, two lanes per group; the result is
// the transposed matrix, staged in shared memory and written out in 64-byte rows.  The random bits of 16
// consecutive elements of the output come from one Philox call.  The scale chunk is assembled in shared memory
// (padding entries 0x7F) and written whole.
// ------------------------------------------------------------------------------------------------
constexpr int kPitch = 2 * kTile + 16;   // bytes per staged row (16-byte skew against bank conflicts)

template <bool SR_T>
__global__ void __launch_bounds__(256, 3) k_requantize_tile(const void *src, const uint8_t *src_scales,
                                                            int src_nblk4, int rows, int cols, const __grid_constant__ QuantSide tr,
                                                            uint32_t *dev_status)
{
    __shared__ __align__(16) uint8_t s_in[kTile * kPitch];
    __shared__ __align__(16) uint2 s_out[kTile * 8];          // [output row = source column][8-byte slot], slots XOR-swizzled
    __shared__ __align__(16) uint8_t s_sc_t[512];

    pdl_launch_dependents();
    const int tid = threadIdx.x;
    const int row0 = blockIdx.y * kTile, col0 = blockIdx.x * kTile;
    uint32_t nonfinite = 0;

    if (tid < 32) reinterpret_cast<uint4 *>(s_sc_t)[tid] = make_uint4(0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu);

    // ---- stage the tile ----
    {
        // packed source: one thread per (row, 32-element group): 16 bytes of codes + 1 scale byte
        pdl_wait();
        const uint8_t *s = static_cast<const uint8_t *>(src);
        const uint8_t *sc_chunk = src_scales + ((size_t)(row0 >> 7) * src_nblk4 + (col0 >> 7)) * 512;
#pragma unroll
        for (int it = 0; it < 2; it++) {
            const int item = it * 256 + tid;
            const int r = item >> 2, g = item & 3;
            const int gr = row0 + r, gc = col0 + g * 32;
            uint32_t w[4] = {0, 0, 0, 0};
            uint32_t sc2 = 0u;
            if (gr < rows && gc < cols) {
                const uint4 q = ld_stream_16(s + (int64_t)gr * (cols >> 1) + (gc >> 1));
                w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
                const uint32_t sb = sc_chunk[(r & 31) * 16 + (r >> 5) * 4 + g];
                // a 0xFF scale marks a non-finite group of the first quantizer: propagate NaN
                sc2 = sb == 0xFFu ? 0x7FC07FC0u : (sb ? sb << 7 : 0x0040u) * 0x00010001u;   // byte 0: 2^-127
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                uint32_t o[4];
                dequant_x8(w[j], sc2, o);   // P * 2^s is exact in bf16
                *reinterpret_cast<uint4 *>(s_in + r * kPitch + g * 64 + j * 16) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }
    __syncthreads();

    // ---- column pass: warp = 32 rows x 64 columns; thread = 16 rows x 4 columns; lanes l, l^16 share the groups ----
    {
        const int warp = tid >> 5, lane = tid & 31;
        const int rg = warp >> 1, ch = warp & 1;
        const int h = lane >> 4, cl = lane & 15;
        const int c = ch * 64 + cl * 4;                 // first of this thread's 4 columns (tile-local)
        const int r = rg * 32 + h * 16;                 // first of its 16 rows
        uint2 v[16];
#pragma unroll
        for (int i = 0; i < 16; i++) v[i] = *reinterpret_cast<const uint2 *>(s_in + (r + i) * kPitch + c * 2);
        uint32_t am0 = 0, am1 = 0;
#pragma unroll
        for (int i = 0; i < 16; i++) {
            am0 = absmax2(am0, v[i].x);
            am1 = absmax2(am1, v[i].y);
        }
        am0 = __vmaxu2(am0, __shfl_xor_sync(0xFFFFFFFFu, am0, 16));
        am1 = __vmaxu2(am1, __shfl_xor_sync(0xFFFFFFFFu, am1, 16));
        // rows come in groups of 32 and columns in blocks of 32: a thread's 16 x 4 patch is inside the matrix or outside it
        if (row0 + r < rows && col0 + c < cols) {
            const uint32_t tfa2 = tf_add_of(tr.scale_mode) * 0x00010001u;
            // element index of (column, first row) in the transposed output, in units of 16
            const uint64_t qi = ((uint64_t)(col0 + c) * (uint64_t)rows + (uint64_t)(row0 + r)) >> 4;
#pragma unroll
            for (int jp = 0; jp < 2; jp++) {      // columns c + 2 jp and c + 2 jp + 1 share a word of every row
                const uint32_t am = jp ? am1 : am0;
                uint32_t m2, inv2;
                group_scales_x2(am, tfa2, m2, inv2);
                const uint32_t nfm = (am + 0x00800080u) & 0x80008000u;   // bit 15 of the half of a non-finite group
                nonfinite |= (uint32_t)(nfm != 0u);
                uint32_t out[2][2];            // codes of rows 0..7 / 8..15 of the two columns
                uint4 ra, rb;
                if (SR_T) {
                    const uint64_t qa = qi + (uint64_t)(2 * jp) * (uint64_t)(rows >> 4);
                    sr_words_two(tr.sr, qa, qa + (uint64_t)(rows >> 4), ra, rb);
                }
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    float a[8], b[8];
#pragma unroll
                    for (int i = 0; i < 8; i++) scale_pair(jp ? v[8 * k + i].y : v[8 * k + i].x, inv2, a[i], b[i]);
                    if (SR_T) {
                        out[0][k] = sr_x8(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], k ? ra.z : ra.x, k ? ra.w : ra.y);
                        out[1][k] = sr_x8(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7], k ? rb.z : rb.x, k ? rb.w : rb.y);
                    } else {
                        out[0][k] = rne_x8(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]);
                        out[1][k] = rne_x8(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7]);
                    }
                }
                if (nfm & 0x8000u) out[0][0] = out[0][1] = 0u;
                if (nfm >> 31) out[1][0] = out[1][1] = 0u;
                // output row c + j, bytes 16 rg + 8 h .. + 7: slot 2 rg + h, swizzled by the column quad
                const int j0 = 2 * jp;
                s_out[(c + j0) * 8 + ((2 * rg + h) ^ (cl & 7))] = make_uint2(out[0][0], out[0][1]);
                s_out[(c + j0 + 1) * 8 + ((2 * rg + h) ^ (cl & 7))] = make_uint2(out[1][0], out[1][1]);
                if (h == 0) {
                    s_sc_t[((c + j0) & 31) * 16 + ((c + j0) >> 5) * 4 + rg] = (uint8_t)((nfm & 0x8000u) ? 0xFFu : (am & 0xFFFFu) ? m2 - 2u : 98u);
                    s_sc_t[((c + j0 + 1) & 31) * 16 + ((c + j0 + 1) >> 5) * 4 + rg] = (uint8_t)((nfm >> 31) ? 0xFFu : am >= 0x10000u ? (m2 >> 16) - 2u : 98u);
                }
            }
        }
    }
    __syncthreads();

    // ---- copy the transposed tile out: 128 output rows x 64 bytes, 16 bytes per thread and step ----
    {
#pragma unroll
        for (int it = 0; it < 2; it++) {
            const int id = it * 256 + tid;
            const int oc = id >> 2, g = id & 3;        // output row (source column), 16-byte group = source row group
            const int gc = col0 + oc, gr = row0 + g * 32;
            if (gc < cols && gr < rows) {
                const int x = (oc >> 2) & 7;
                const uint2 a = s_out[oc * 8 + ((2 * g) ^ x)], b = s_out[oc * 8 + ((2 * g + 1) ^ x)];
                *reinterpret_cast<uint4 *>(tr.packed + (int64_t)gc * (rows >> 1) + (gr >> 1)) = make_uint4(a.x, a.y, b.x, b.y);
            }
        }
        // the scale chunk of this tile
        if (tid < 32)
            reinterpret_cast<uint4 *>(tr.scales + ((size_t)(col0 >> 7) * tr.nblk4 + (row0 >> 7)) * 512)[tid] =
                reinterpret_cast<const uint4 *>(s_sc_t)[tid];
    }
    if (nonfinite && dev_status) atomicOr(dev_status, MXFP4_DEV_NONFINITE);
}

// ------------------------------------------------------------------------------------------------
// Streaming two-axis quantizer for bf16 sources (Q3 + Q5 of Eq. 4-5, Q1 + Q6 by double quantization, or the
// transposed quantizer alone).  Persistent: two CTAs per SM walk over the 128 x 128 tiles; one thread feeds a ring of
// two tiles with TMA (each tile arrives as two 128B-swizzled boxes of 128 rows x 64 columns), so the next tile travels
// while this one is quantized, and nothing of the staging costs an instruction of the computing threads.
//   row pass   : a thread takes one whole 32-element group of a row (four 16-byte pieces) twice per tile and
//                stores its 16 bytes of codes straight to global memory;
//   column pass: a thread takes two adjacent columns x 32 rows (a bf16 pair per row), i.e. two whole groups of
//                the transposed output, scaled together by packed multiplies; the transposed codes are staged in a
//                64B-swizzled tile that leaves with one TMA store (clipped at the matrix edges).
// Both 512-byte scale chunks of a tile are assembled in shared memory (entries outside the matrix 0x7F) and leave
// as bulk copies.  The staging is double buffered: a tile's stores are read out while the next tile is computed.
// Random bits are drawn per 16 consecutive elements of each OUTPUT, as in every other quantizer here.
// ------------------------------------------------------------------------------------------------
constexpr int kQsThreads = 256;
constexpr int kQsStagingBytes = kTile * 64 + 1024;     // transposed codes (8 KB, 64B-swizzled) + the two scale chunks
constexpr int kQsBarOff = 2 * kTileBytes + 2 * kQsStagingBytes;
constexpr int kQsSmemBytes = kQsBarOff + 64 + 1024 /*align*/;
constexpr int kQsCtasPerSm = 2;

// One source matrix of a launch and its results.
struct QsJob {
    CUtensorMap map_src, map_t;
    QuantSide rw, tr;
    int rows, cols;
};
struct QsNone {};

// The walk of a CTA over the tiles of one matrix.  The tiles of a launch are numbered through: this matrix has the numbers
// [first, end), and `tile` and the ring's turn `it` run on from one matrix to the next.  load(tile, stage) starts the load of
// any tile of the launch.
template <bool EMIT_ROW, bool SR_ROW, bool SR_T, bool DQ, bool GELU, class Load>
__device__ __forceinline__ bool qs_walk(const QsJob &job, const QsGeom &g, int first, int end, int all, int &tile, int &it, uint8_t *smem, uint32_t smem_base,
                                        uint32_t bar_full, volatile uint32_t *abort_flag, uint32_t *dev_status, uint32_t spin_limit, uint32_t &nonfinite,
                                        __nv_bfloat16 *hook_out, int64_t hook_ld, const Load &load)
{
    const int rows = job.rows, cols = job.cols, ntx = (cols + kTile - 1) / kTile;
    const uint32_t tfa_r2 = tf_add_of(job.rw.scale_mode) * 0x00010001u, tfa_t2 = tf_add_of(job.tr.scale_mode) * 0x00010001u;
    // tile coordinates advance by the grid size without a division per tile
    const int step_y = (int)gridDim.x / ntx, step_x = (int)gridDim.x - step_y * ntx;
    int ty = (tile - first) / ntx, tx = (tile - first) - ty * ntx;
    for (; tile < end; tile += gridDim.x, it++) {
        const int stage = it & 1;
        const int row0 = ty * kTile, col0 = tx * kTile;
        const uint32_t st_base = smem_base + stage * kTileBytes;
        uint8_t *staging = smem + 2 * kTileBytes + stage * kQsStagingBytes;
        uint8_t *s_sc_row = staging + kTile * 64, *s_sc_t = s_sc_row + 512;

        const bool ok = mbar_wait_warp(bar_full + 8 * stage, (uint32_t)(it >> 1) & 1u, abort_flag, dev_status, spin_limit);
        if (ok)
            qs_tile<SR_ROW, SR_T, DQ, GELU>(g, st_base, st_base, row0, col0, rows, cols, EMIT_ROW, true, job.rw, job.tr, tfa_r2, tfa_t2, staging, s_sc_row, s_sc_t,
                                            nonfinite, hook_out, hook_ld);

        // ---- hand the tile's results to the copy engine, refill the ring ----
        fence_async_smem();                       // this thread's staging writes, before the asynchronous reads
        if (threadIdx.x == 0) bulk_wait_read<0>();   // the previous tile's stores have left the other staging buffer
        if (__syncthreads_or(!ok)) return false;   // a bounded wait ran out somewhere in the CTA: everybody leaves
        if (threadIdx.x == 0) {
            tma_store_2d(&job.map_t, row0 >> 1, col0, smem_u32(staging));
            bulk_store(job.tr.scales + ((size_t)(col0 >> 7) * job.tr.nblk4 + (row0 >> 7)) * 512, smem_u32(s_sc_t), 512);
            if (EMIT_ROW) bulk_store(job.rw.scales + ((size_t)(row0 >> 7) * job.rw.nblk4 + (col0 >> 7)) * 512, smem_u32(s_sc_row), 512);
            bulk_commit();
            const int next = tile + 2 * (int)gridDim.x;
            if (next < all) load(next, stage);
        }
        tx += step_x;
        ty += step_y;
        if (tx >= ntx) { tx -= ntx; ty++; }
    }
    return true;
}

// GELU: the source is a product's result Y, quantized behind the activation (see qs_row_pass).
// Job2 = QsJob: a second matrix with the same roundings follows in the same launch (its tiles fill the tail of the first:
// activations and weight of a forward pass); QsNone: there is none.
template <bool EMIT_ROW, bool SR_ROW, bool SR_T, bool DQ, bool GELU, class Job2>
__global__ void __launch_bounds__(kQsThreads, kQsCtasPerSm)
k_quantize_stream(const __grid_constant__ QsJob job, const __grid_constant__ Job2 job2, uint32_t *dev_status, uint32_t spin_limit, int withhold_loads,
                  __nv_bfloat16 *hook_out, int64_t hook_ld)
{
    constexpr bool kTwo = sizeof(Job2) == sizeof(QsJob);
    extern __shared__ uint8_t qs_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(qs_smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bar_full = smem_base + kQsBarOff;
    volatile uint32_t *abort_flag = reinterpret_cast<volatile uint32_t *>(smem + kQsBarOff + 32);

    pdl_launch_dependents();
    const int ntx = (job.cols + kTile - 1) / kTile, total = ntx * ((job.rows + kTile - 1) / kTile);
    int ntx2 = 1, all = total;
    if constexpr (kTwo) {
        ntx2 = (job2.cols + kTile - 1) / kTile;
        all += ntx2 * ((job2.rows + kTile - 1) / kTile);
    }
    auto load = [&](int tile, int stage) {
        const uint32_t bar = bar_full + 8 * stage, dst = smem_base + stage * kTileBytes;
        mbar_expect_tx(bar, kTileBytes);
        const CUtensorMap *map = &job.map_src;
        int n = ntx;
        if constexpr (kTwo) {
            if (tile >= total) map = &job2.map_src, n = ntx2, tile -= total;
        }
        const int ty = tile / n, tx = tile - ty * n;
        tma_load_2d(dst, map, tx * kTile, ty * kTile, bar);
        tma_load_2d(dst + kTileBytes / 2, map, tx * kTile + 64, ty * kTile, bar);
    };

    if (threadIdx.x == 0) {
        mbar_init(bar_full, 1);
        mbar_init(bar_full + 8, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_map(&job.map_src);
        prefetch_map(&job.map_t);
    }
    const QsGeom g = qs_geom(threadIdx.x, job.rows, job.cols, job.rw.packed);
    pdl_wait();
    if (threadIdx.x == 0) {
        // withhold_loads (self-test of the drain path): nothing is ever loaded, so the first bounded wait runs out
        for (int s = 0; s < 2; s++)
            if (!withhold_loads && (int)blockIdx.x + s * (int)gridDim.x < all) load(blockIdx.x + s * gridDim.x, s);
    }
    __syncthreads();

    uint32_t nonfinite = 0;
    int tile = blockIdx.x, it = 0;
    const bool alive = qs_walk<EMIT_ROW, SR_ROW, SR_T, DQ, GELU>(job, g, 0, total, all, tile, it, smem, smem_base, bar_full, abort_flag, dev_status, spin_limit,
                                                                 nonfinite, hook_out, hook_ld, load);
    if constexpr (kTwo) {
        if (alive && tile < all) {
            const QsGeom g2 = qs_geom(threadIdx.x, job2.rows, job2.cols, job2.rw.packed);
            qs_walk<EMIT_ROW, SR_ROW, SR_T, DQ, GELU>(job2, g2, total, all, all, tile, it, smem, smem_base, bar_full, abort_flag, dev_status, spin_limit, nonfinite,
                                                      hook_out, hook_ld, load);
        }
    }
    if (threadIdx.x == 0) bulk_wait_read<0>();    // every store has read its staging buffer: the shared memory may go
    if (nonfinite && dev_status) atomicOr(dev_status, MXFP4_DEV_NONFINITE);
}

// ------------------------------------------------------------------------------------------------
// Q-EMA (Algorithm 1) fused with the EMA update (Eq. 10) and the oscillation counters (Sec. 6.1).

// ------------------------------------------------------------------------------------------------
struct OscPtrs {
    __nv_bfloat16 *w_prev;
    uint8_t *q_prev;
    uint8_t *s_prev;
    float *dist_w;
    float *dist_q;
};

// value of an E2M1 code as float
__device__ __forceinline__ float e2m1_value(uint32_t code)
{
    const uint32_t m = code & 7u;
    const uint32_t bits = m >= 2u ? (0x3F000000u + (m << 22)) : (m ? 0x3F000000u : 0u);
    return __uint_as_float(bits | ((code & 8u) << 28));
}

// The element step of Algorithm 1: propose the two neighbouring grid values q1 <= |w / S| <= q2, keep the one nearer
// to the EMA.  "The nearer of q1, q2 to e" is the round-to-nearest (ties to the even code, as everywhere) of e clamped
// to [q1, q2], because no grid value lies strictly between the two; a latent value on the grid has q1 = q2 and is
// kept.  Returns that clamped value with the sign of w, ready for the hardware convert.  v = w / S, ve = ema / S.
__device__ __forceinline__ float qema_target(float v, float ve)
{
    const uint32_t vb = __float_as_uint(v);
    const uint32_t ab = vb & 0x7FFFFFFFu;
    uint32_t lo, hi;
    if (ab >= 0x40C00000u) {            // 6 and beyond (floor scaling): saturates
        lo = hi = 0x40C00000u;
    } else if (ab >= 0x3F000000u) {     // [0.5, 6): one mantissa bit from 1 upwards, none below
        const uint32_t mask = ab >= 0x3F800000u ? 0x003FFFFFu : 0x007FFFFFu;
        lo = ab & ~mask;
        hi = ab == lo ? lo : lo + mask + 1u;
    } else {                            // [0, 0.5)
        lo = 0u;
        hi = ab == 0u ? 0u : 0x3F000000u;
    }
    const float es = (vb >> 31) ? -ve : ve;   // EMA mirrored to the side of w
    const float t = fminf(fmaxf(es, __uint_as_float(lo)), __uint_as_float(hi));
    return __uint_as_float(__float_as_uint(t) | (vb & 0x80000000u));
}

// Four consecutive lanes share a 32-element group: a thread owns 8 consecutive elements (the weight is contiguous).  The grid
// covers the scale buffer with its padding entries, as in the row-wise quantizer.
template <bool OSC>
__global__ void __launch_bounds__(256) k_qema(const __nv_bfloat16 *w, float *__restrict__ ema, float beta,
                                              int update_ema, int64_t n, int nblk, uint8_t *__restrict__ packed,
                                              uint8_t *__restrict__ scales, int nblk4, int scale_mode, OscPtrs osc,
                                              uint32_t *dev_status)
{
    pdl_launch_dependents();
    pdl_wait();
    const uint64_t gid = blockIdx.x * (uint64_t)256 + threadIdx.x, grp_pad = gid >> 2;
    const uint32_t nb_pad = (uint32_t)nblk4 * 4u;
    const int64_t row_pad = (grp_pad >> 32) ? (int64_t)(grp_pad / nb_pad) : (int64_t)((uint32_t)grp_pad / nb_pad);
    const int blk_pad = (int)(grp_pad - (uint64_t)row_pad * nb_pad);
    // the lanes of a padding entry shadow group 0 and store that entry only; without padding blocks the weight is addressed
    // without waiting for the division
    const bool active = (int)nb_pad == nblk ? gid < (uint64_t)n * nblk * 4 : row_pad < n && blk_pad < nblk;
    const int64_t row = row_pad;
    const int blk = blk_pad;
    const int64_t cid = !active ? (int64_t)(gid & 3) : (int)nb_pad == nblk ? (int64_t)gid : (row * nblk + blk) * 4 + (int64_t)(gid & 3), e0 = cid * 8;
    const float omb = __fsub_rn(1.0f, beta);

    const uint4 q = *reinterpret_cast<const uint4 *>(w + e0);
    float4 ea = *reinterpret_cast<const float4 *>(ema + e0), eb = *reinterpret_cast<const float4 *>(ema + e0 + 4);
    const uint32_t ww[4] = {q.x, q.y, q.z, q.w};
    float wv[8];
#pragma unroll
    for (int t = 0; t < 4; t++) {
        wv[2 * t] = bf16lo(ww[t]);
        wv[2 * t + 1] = bf16hi(ww[t]);
    }
    if (update_ema) {
        ea.x = __fmaf_rn(beta, ea.x, __fmul_rn(omb, wv[0]));
        ea.y = __fmaf_rn(beta, ea.y, __fmul_rn(omb, wv[1]));
        ea.z = __fmaf_rn(beta, ea.z, __fmul_rn(omb, wv[2]));
        ea.w = __fmaf_rn(beta, ea.w, __fmul_rn(omb, wv[3]));
        eb.x = __fmaf_rn(beta, eb.x, __fmul_rn(omb, wv[4]));
        eb.y = __fmaf_rn(beta, eb.y, __fmul_rn(omb, wv[5]));
        eb.z = __fmaf_rn(beta, eb.z, __fmul_rn(omb, wv[6]));
        eb.w = __fmaf_rn(beta, eb.w, __fmul_rn(omb, wv[7]));
        if (active) {
            *reinterpret_cast<float4 *>(ema + e0) = ea;
            *reinterpret_cast<float4 *>(ema + e0 + 4) = eb;
        }
    }
    const float ev[8] = {ea.x, ea.y, ea.z, ea.w, eb.x, eb.y, eb.z, eb.w};
    uint32_t am = hmax_halves(absmax_u4(0, q));
    uint32_t badm = !(isfinite(ea.x) && isfinite(ea.y) && isfinite(ea.z) && isfinite(ea.w) && isfinite(eb.x) && isfinite(eb.y) &&
                      isfinite(eb.z) && isfinite(eb.w));
    am = max(am, __shfl_xor_sync(0xFFFFFFFFu, am, 1));
    am = max(am, __shfl_xor_sync(0xFFFFFFFFu, am, 2));
    badm |= __shfl_xor_sync(0xFFFFFFFFu, badm, 1);
    badm |= __shfl_xor_sync(0xFFFFFFFFu, badm, 2);
    const bool bad = badm != 0u || am >= 0x7F80u;

    uint32_t byte, out = 0;
    if (bad) {
        byte = 0xFFu;
        if (dev_status && active) atomicOr(dev_status, MXFP4_DEV_NONFINITE);
    } else {
        byte = scale_byte_from_amax(am, tf_add_of(scale_mode));
        const float inv = inv_scale_from_byte(byte);
        float z[8];
#pragma unroll
        for (int i = 0; i < 8; i++) z[i] = qema_target(wv[i] * inv, ev[i] * inv);
        out = rne_x8(z[0], z[1], z[2], z[3], z[4], z[5], z[6], z[7]);
    }
    if (!active) {
        if ((gid & 3) == 0) {
            scales[scale_offset(row_pad, blk_pad, nblk4)] = 0x7F;
            if (OSC) osc.s_prev[scale_offset(row_pad, blk_pad, nblk4)] = 0x7F;
        }
        return;
    }

    const int64_t pk = row * ((int64_t)nblk * 16) + blk * 16 + (cid & 3) * 4;   // this thread's 4 bytes of codes
    if (OSC) {
        const uint32_t prev = *reinterpret_cast<const uint32_t *>(osc.q_prev + pk);
        const uint32_t sbp = osc.s_prev[scale_offset(row, blk, nblk4)];
        const float sc = byte == 0xFFu ? __uint_as_float(0x7FC00000u) : scale_from_byte(byte);
        const float scp = sbp == 0xFFu ? __uint_as_float(0x7FC00000u) : scale_from_byte(sbp);
        const uint4 wp = *reinterpret_cast<const uint4 *>(osc.w_prev + e0);
        const uint32_t wpw[4] = {wp.x, wp.y, wp.z, wp.w};
#pragma unroll
        for (int j = 0; j < 2; j++) {
            float4 dw = *reinterpret_cast<const float4 *>(osc.dist_w + e0 + 4 * j);
            float4 dq = *reinterpret_cast<const float4 *>(osc.dist_q + e0 + 4 * j);
            float *dwp = &dw.x, *dqp = &dq.x;
#pragma unroll
            for (int t = 0; t < 4; t++) {
                const int i = 4 * j + t;
                const float wpv = (i & 1) ? bf16hi(wpw[i >> 1]) : bf16lo(wpw[i >> 1]);
                const float qc = e2m1_value((out >> (4 * i)) & 15u) * sc;
                const float qo = e2m1_value((prev >> (4 * i)) & 15u) * scp;
                dwp[t] = __fadd_rn(dwp[t], fabsf(__fsub_rn(wv[i], wpv)));
                dqp[t] = __fadd_rn(dqp[t], fabsf(__fsub_rn(qc, qo)));
            }
            *reinterpret_cast<float4 *>(osc.dist_w + e0 + 4 * j) = dw;
            *reinterpret_cast<float4 *>(osc.dist_q + e0 + 4 * j) = dq;
        }
        __syncwarp();   // every lane of the group has read the previous scale before one of them replaces it
        *reinterpret_cast<uint4 *>(osc.w_prev + e0) = q;
        *reinterpret_cast<uint32_t *>(osc.q_prev + pk) = out;
        if ((cid & 3) == 0) osc.s_prev[scale_offset(row, blk, nblk4)] = (uint8_t)byte;
    }
    *reinterpret_cast<uint32_t *>(packed + pk) = out;
    if ((cid & 3) == 0) scales[scale_offset(row, blk, nblk4)] = (uint8_t)byte;
}

// ------------------------------------------------------------------------------------------------
// Exact dequantization, one thread per group.
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_dequantize(const uint8_t *packed, const uint8_t *scales,
                                                    int64_t rows, int nblk, int nblk4, float *__restrict__ dst, int64_t ld)
{
    pdl_launch_dependents();
    pdl_wait();
    const int64_t gid = blockIdx.x * (int64_t)256 + threadIdx.x;
    if (gid >= rows * nblk) return;
    const int64_t row = gid / nblk;
    const int blk = (int)(gid - row * nblk);
    const uint4 q = *reinterpret_cast<const uint4 *>(packed + row * ((int64_t)nblk * 16) + blk * 16);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    const uint32_t sb = scales[scale_offset(row, blk, nblk4)];
    const float sc = sb == 0xFFu ? __uint_as_float(0x7FC00000u) : scale_from_byte(sb);
    float *o = dst + row * ld + blk * 32;
#pragma unroll
    for (int i = 0; i < 32; i += 4) {
        float4 f;
        f.x = e2m1_value((w[i >> 3] >> (4 * (i & 7))) & 15u) * sc;
        f.y = e2m1_value((w[i >> 3] >> (4 * ((i + 1) & 7))) & 15u) * sc;
        f.z = e2m1_value((w[i >> 3] >> (4 * ((i + 2) & 7))) & 15u) * sc;
        f.w = e2m1_value((w[i >> 3] >> (4 * ((i + 3) & 7))) & 15u) * sc;
        *reinterpret_cast<float4 *>(o + i) = f;
    }
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static mxfp4_status_t check_mat(const mxfp4_mat_t &m, int64_t rows, int64_t cols)
{
    if (!m.data || !m.scales) return MXFP4_INVALID_ARG;
    if (m.rows != rows || m.cols != cols) return MXFP4_BAD_SHAPE;
    if (!aligned16(m.data) || !aligned16(m.scales)) return MXFP4_MISALIGNED;
    return MXFP4_OK;
}

static mxfp4_status_t check_qp(const mxfp4_qparams_t *qp)
{
    if (!qp) return MXFP4_INVALID_ARG;
    if (qp->scale_mode != MXFP4_SCALE_TRUNCATION_FREE && qp->scale_mode != MXFP4_SCALE_FLOOR) return MXFP4_INVALID_ARG;
    if (qp->rounding != MXFP4_ROUND_NEAREST && qp->rounding != MXFP4_ROUND_STOCHASTIC) return MXFP4_INVALID_ARG;
    return MXFP4_OK;
}

mxfp4_status_t quantize_rows(const void *src, int64_t rows, int64_t cols, int64_t ld, mxfp4_mat_t dst,
                             const mxfp4_qparams_t *qp, uint32_t *dev_status, cudaStream_t st)
{
    if (rows < 0 || cols < 0) return MXFP4_INVALID_ARG;
    mxfp4_status_t s = check_qp(qp);
    if (s) return s;
    if (cols % 32 != 0 || ld < cols) return MXFP4_BAD_SHAPE;
    if (rows == 0 || cols == 0) return MXFP4_OK;  // nothing to do; pointers may be null
    if (!src) return MXFP4_INVALID_ARG;
    if ((s = check_mat(dst, rows, cols))) return s;
    if (!aligned16(src) || ld % 8 != 0) return MXFP4_MISALIGNED;
    if (rows == 0 || cols == 0) return MXFP4_OK;
    const int nblk = (int)(cols / 32), nblk4 = (nblk + 3) / 4;
    const unsigned blocks = (unsigned)(ceil_div(rows, 128) * nblk4 * 2);   // a thread per scale entry, padding included: 512 per chunk
    MX_CHECK_CUDA(launch_pdl(qp->rounding == MXFP4_ROUND_STOCHASTIC ? k_quantize_rows<MXFP4_ROUND_STOCHASTIC> : k_quantize_rows<MXFP4_ROUND_NEAREST>,
                             blocks, 1, 256, 0, st, static_cast<const __nv_bfloat16 *>(src), rows, nblk, ld, static_cast<uint8_t *>(dst.data),
                             dst.scales, nblk4, qp->scale_mode, make_sr_stream(qp->seed, qp->stream_id, rows * cols), dev_status));
    return MXFP4_OK;
}

static QuantSide make_side(const mxfp4_mat_t &m, const mxfp4_qparams_t *qp)
{
    QuantSide s;
    s.packed = static_cast<uint8_t *>(m.data);
    s.scales = m.scales;
    s.nblk4 = (int)ceil_div(m.cols / 32, 4);
    s.scale_mode = qp->scale_mode;
    s.sr = make_sr_stream(qp->seed, qp->stream_id, m.rows * m.cols);
    return s;
}

// bf16 source [rows, cols] (leading dimension ld) as a 2-D tensor of bf16; box = 64 columns x 128 rows, 128B swizzle.
static bool make_src_map(CUtensorMap *map, const void *src, int64_t rows, int64_t cols, int64_t ld)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t gstride[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(src), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Packed transposed output [cols, rows / 2 bytes] as a 2-D byte tensor; box = 64 bytes x 128 rows, 64B swizzle.
static bool make_packed_t_map(CUtensorMap *map, void *packed, int64_t rows, int64_t cols)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t gdim[2] = {(cuuint64_t)(rows / 2), (cuuint64_t)cols};
    cuuint64_t gstride[1] = {(cuuint64_t)(rows / 2)};
    cuuint32_t box[2] = {64, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, packed, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static int64_t qs_tiles(int64_t rows, int64_t cols) { return ceil_div(rows, kTile) * ceil_div(cols, kTile); }

static bool make_job(QsJob *job, const void *src_bf16, int64_t rows, int64_t cols, int64_t ld, const mxfp4_mat_t *dst, const mxfp4_qparams_t *qp_row,
                     const mxfp4_mat_t &dst_t, const mxfp4_qparams_t *qp_t)
{
    job->tr = make_side(dst_t, qp_t);
    job->rw = dst ? make_side(*dst, qp_row) : job->tr;
    job->rows = (int)rows;
    job->cols = (int)cols;
    return make_src_map(&job->map_src, src_bf16, rows, cols, ld) && make_packed_t_map(&job->map_t, dst_t.data, rows, cols);
}

template <bool EMIT_ROW, bool SR_ROW, bool SR_T, bool DQ, bool GELU = false, class Job2 = QsNone>
static mxfp4_status_t launch_stream(cudaStream_t st, const QsJob &job, uint32_t *dev_status, uint32_t spin_limit = kWaitSpinLimit, int withhold_loads = 0,
                                    __nv_bfloat16 *hook_out = nullptr, int64_t hook_ld = 0, const Job2 &job2 = Job2(), int64_t tiles2 = 0)
{
    static bool attr_set[kMaxDevices];
    MX_CHECK_CUDA(set_smem_once(attr_set, k_quantize_stream<EMIT_ROW, SR_ROW, SR_T, DQ, GELU, Job2>, kQsSmemBytes));
    const int64_t tiles = qs_tiles(job.rows, job.cols) + tiles2;
    const int64_t cap = kQsCtasPerSm * (int64_t)sm_count();
    const unsigned grid = (unsigned)(tiles < cap ? tiles : cap);
    MX_CHECK_CUDA(launch_pdl(k_quantize_stream<EMIT_ROW, SR_ROW, SR_T, DQ, GELU, Job2>, grid, 1, kQsThreads, kQsSmemBytes, st, job, job2, dev_status, spin_limit,
                             withhold_loads, hook_out, hook_ld));
    return MXFP4_OK;
}

// src_bf16 xor src_q; dst (row-wise) optional; dst_t required.  chain: dst_t is quantized from the dequantized dst
// (double quantization) instead of from the source; needs a bf16 source and dst.
// spin_limit / withhold_loads: normal use kWaitSpinLimit / 0; the self-test of the drain path withholds the loads of the
// streaming kernel so that its bounded waits run out after spin_limit polls.
static mxfp4_status_t quantize_tile_ex(const void *src_bf16, const mxfp4_mat_t *src_q, int64_t rows, int64_t cols, int64_t ld,
                                       const mxfp4_mat_t *dst, const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t,
                                       const mxfp4_qparams_t *qp_t, uint32_t *dev_status, cudaStream_t st, bool chain, uint32_t spin_limit,
                                       int withhold_loads)
{
    if (chain && (!dst || !src_bf16)) return MXFP4_INVALID_ARG;
    if ((src_bf16 == nullptr) == (src_q == nullptr) || rows < 0 || cols < 0) return MXFP4_INVALID_ARG;
    if (dst && src_q) return MXFP4_INVALID_ARG;
    mxfp4_status_t s = check_qp(qp_t);
    if (s) return s;
    if (dst && (s = check_qp(qp_row))) return s;
    if (rows % 32 != 0 || cols % 32 != 0) return MXFP4_BAD_SHAPE;
    if (rows > 0x7FFFFF80 || cols > 0x7FFFFF80) return MXFP4_BAD_SHAPE;
    if ((s = check_mat(dst_t, cols, rows))) return s;
    if (dst && (s = check_mat(*dst, rows, cols))) return s;
    if (src_bf16) {
        if (ld < cols) return MXFP4_BAD_SHAPE;
        if (!aligned16(src_bf16) || ld % 8 != 0) return MXFP4_MISALIGNED;
    } else {
        if ((s = check_mat(*src_q, rows, cols))) return s;
    }
    if (rows == 0 || cols == 0) return MXFP4_OK;
    // every tile writes its whole 512-byte scale chunk(s), padding entries included
    const dim3 grid((unsigned)ceil_div(cols, kTile), (unsigned)ceil_div(rows, kTile));
    if (src_q && grid.y > 65535u) return MXFP4_BAD_SHAPE;
    const bool sr_t = qp_t->rounding == MXFP4_ROUND_STOCHASTIC;
    const bool sr_r = dst && qp_row->rounding == MXFP4_ROUND_STOCHASTIC;
    if (src_q) {
        const int nb4 = (int)ceil_div(cols / 32, 4);
        MX_CHECK_CUDA(launch_pdl(sr_t ? k_requantize_tile<true> : k_requantize_tile<false>, grid.x, grid.y, 256, 0, st, src_q->data, src_q->scales, nb4, (int)rows,
                                 (int)cols, make_side(dst_t, qp_t), dev_status));
    } else {
        // bf16 source: the streaming kernel
        if (qs_tiles(rows, cols) > 0x7FFFFFFF) return MXFP4_BAD_SHAPE;
        QsJob job;
        if (!make_job(&job, src_bf16, rows, cols, ld, dst, qp_row, dst_t, qp_t)) return MXFP4_CUDA_ERROR;
        if (!dst) {
            return sr_t ? launch_stream<false, false, true, false>(st, job, dev_status, spin_limit, withhold_loads)
                        : launch_stream<false, false, false, false>(st, job, dev_status, spin_limit, withhold_loads);
        }
        const int sel = (chain ? 4 : 0) | (sr_r ? 2 : 0) | (sr_t ? 1 : 0);
        switch (sel) {
        case 0: return launch_stream<true, false, false, false>(st, job, dev_status, spin_limit, withhold_loads);
        case 1: return launch_stream<true, false, true, false>(st, job, dev_status, spin_limit, withhold_loads);
        case 2: return launch_stream<true, true, false, false>(st, job, dev_status, spin_limit, withhold_loads);
        case 3: return launch_stream<true, true, true, false>(st, job, dev_status, spin_limit, withhold_loads);
        case 4: return launch_stream<true, false, false, true>(st, job, dev_status, spin_limit, withhold_loads);
        case 5: return launch_stream<true, false, true, true>(st, job, dev_status, spin_limit, withhold_loads);
        case 6: return launch_stream<true, true, false, true>(st, job, dev_status, spin_limit, withhold_loads);
        default: return launch_stream<true, true, true, true>(st, job, dev_status, spin_limit, withhold_loads);
        }
    }
    return MXFP4_OK;
}

mxfp4_status_t quantize_tile(const void *src_bf16, const mxfp4_mat_t *src_q, int64_t rows, int64_t cols, int64_t ld,
                             const mxfp4_mat_t *dst, const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t,
                             const mxfp4_qparams_t *qp_t, uint32_t *dev_status, cudaStream_t st, bool chain)
{
    return quantize_tile_ex(src_bf16, src_q, rows, cols, ld, dst, qp_row, dst_t, qp_t, dev_status, st, chain, kWaitSpinLimit, 0);
}

// The second half of mxfp4_gemm_quant with GELU and the double-quantization chain: Z = bf16(GELU(Y)) and its quantizations from
// one read of Y.  The caller has checked every argument.
mxfp4_status_t quantize_gelu_chain(const void *y_bf16, int64_t rows, int64_t cols, int64_t ldy, void *z_bf16, int64_t ldz, mxfp4_mat_t dst,
                                   const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t, const mxfp4_qparams_t *qp_t, uint32_t *dev_status, cudaStream_t st)
{
    QsJob job;
    if (!make_job(&job, y_bf16, rows, cols, ldy, &dst, qp_row, dst_t, qp_t)) return MXFP4_CUDA_ERROR;
    __nv_bfloat16 *z = static_cast<__nv_bfloat16 *>(z_bf16);
    const bool sr_r = qp_row->rounding == MXFP4_ROUND_STOCHASTIC, sr_t = qp_t->rounding == MXFP4_ROUND_STOCHASTIC;
    if (sr_r)
        return sr_t ? launch_stream<true, true, true, true, true>(st, job, dev_status, kWaitSpinLimit, 0, z, ldz)
                    : launch_stream<true, true, false, true, true>(st, job, dev_status, kWaitSpinLimit, 0, z, ldz);
    return sr_t ? launch_stream<true, false, true, true, true>(st, job, dev_status, kWaitSpinLimit, 0, z, ldz)
                : launch_stream<true, false, false, true, true>(st, job, dev_status, kWaitSpinLimit, 0, z, ldz);
}

// The forward pass's two chains in one launch: Q1 + Q6 of x [m, k] and Q2 + Q4 of w [n, k] (round to nearest along the rows,
// then stochastic double quantization).  The caller has checked every argument; m, n and k are multiples of 32.
mxfp4_status_t quantize_chain_two(const void *x_bf16, int64_t m, int64_t k, int64_t ldx, const mxfp4_mat_t &xq, const mxfp4_mat_t &xq_t, const mxfp4_qparams_t *q6,
                                  const void *w_bf16, int64_t n, const mxfp4_mat_t &wq, const mxfp4_mat_t &wq_t, const mxfp4_qparams_t *q4,
                                  const mxfp4_qparams_t *rne, uint32_t *dev_status, cudaStream_t st, uint32_t spin_limit, int withhold_loads)
{
    if (m == 0 || n == 0 || k == 0) return MXFP4_BAD_SHAPE;
    if (qs_tiles(m, k) + qs_tiles(n, k) > 0x7FFFFFFF || m > 0x7FFFFF80 || n > 0x7FFFFF80 || k > 0x7FFFFF80) return MXFP4_BAD_SHAPE;
    QsJob x, w;
    if (!make_job(&x, x_bf16, m, k, ldx, &xq, rne, xq_t, q6) || !make_job(&w, w_bf16, n, k, k, &wq, rne, wq_t, q4)) return MXFP4_CUDA_ERROR;
    return launch_stream<true, false, true, true, false, QsJob>(st, x, dev_status, spin_limit, withhold_loads, nullptr, 0, w, qs_tiles(n, k));
}

std::atomic<unsigned long long> g_launches{0};

}  // namespace mx

using namespace mx;

extern "C" {

uint64_t mxfp4_launch_count(void) { return (uint64_t)mx::g_launches.load(std::memory_order_relaxed); }

mxfp4_status_t mxfp4_quantize_wait_selftest(const void *src_bf16, int64_t rows, int64_t cols, int64_t ld, mxfp4_mat_t dst,
                                            mxfp4_mat_t dst_t, uint32_t spin_limit, uint32_t *dev_status, void *stream)
{
    if (!src_bf16 || !dev_status || spin_limit < 128u || spin_limit > (1u << 16)) return MXFP4_INVALID_ARG;
    const mxfp4_qparams_t qp = {MXFP4_SCALE_TRUNCATION_FREE, MXFP4_ROUND_NEAREST, 0, 0, 0};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const mxfp4_status_t s = quantize_tile_ex(src_bf16, nullptr, rows, cols, ld, &dst, &qp, dst_t, &qp, dev_status, st, false, spin_limit, 1);
    if (s || rows == 0 || cols == 0) return s;
    return quantize_chain_two(src_bf16, rows, cols, ld, dst, dst_t, &qp, src_bf16, rows, dst, dst_t, &qp, &qp, dev_status, st, spin_limit, 1);
}

size_t mxfp4_scale_bytes(int64_t rows, int64_t cols)
{
    if (rows <= 0 || cols <= 0) return 0;
    return (size_t)(ceil_div(rows, 128) * ceil_div(ceil_div(cols, 32), 4) * 512);
}

size_t mxfp4_scale_offset(int64_t row, int64_t block, int64_t cols)
{
    return scale_offset(row, block, ceil_div(ceil_div(cols, 32), 4));
}

mxfp4_status_t mxfp4_quantize(const void *src_bf16, int64_t rows, int64_t cols, int64_t ld, mxfp4_mat_t dst,
                              const mxfp4_qparams_t *qp, uint32_t *dev_status, void *stream)
{
    return quantize_rows(src_bf16, rows, cols, ld, dst, qp, dev_status, static_cast<cudaStream_t>(stream));
}

mxfp4_status_t mxfp4_quantize_t(const void *src_bf16, const mxfp4_mat_t *src_q, int64_t rows, int64_t cols, int64_t ld,
                                mxfp4_mat_t dst_t, const mxfp4_qparams_t *qp, uint32_t *dev_status, void *stream)
{
    return quantize_tile(src_bf16, src_q, rows, cols, ld, nullptr, nullptr, dst_t, qp, dev_status,
                         static_cast<cudaStream_t>(stream), false);
}

mxfp4_status_t mxfp4_quantize_2axis(const void *src_bf16, int64_t rows, int64_t cols, int64_t ld, mxfp4_mat_t dst,
                                    const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t, const mxfp4_qparams_t *qp_t,
                                    uint32_t *dev_status, void *stream)
{
    if (!src_bf16) return MXFP4_INVALID_ARG;
    return quantize_tile(src_bf16, nullptr, rows, cols, ld, &dst, qp_row, dst_t, qp_t, dev_status,
                         static_cast<cudaStream_t>(stream), false);
}

mxfp4_status_t mxfp4_quantize_chain(const void *src_bf16, int64_t rows, int64_t cols, int64_t ld, mxfp4_mat_t dst,
                                    const mxfp4_qparams_t *qp_row, mxfp4_mat_t dst_t, const mxfp4_qparams_t *qp_t,
                                    uint32_t *dev_status, void *stream)
{
    if (!src_bf16) return MXFP4_INVALID_ARG;
    return quantize_tile(src_bf16, nullptr, rows, cols, ld, &dst, qp_row, dst_t, qp_t, dev_status,
                         static_cast<cudaStream_t>(stream), true);
}

mxfp4_status_t mxfp4_qema_quantize(const void *w_bf16, float *ema, float beta, int32_t update_ema, int64_t n, int64_t k,
                                   mxfp4_mat_t dst, int32_t scale_mode, const mxfp4_osc_state_t *osc,
                                   uint32_t *dev_status, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!w_bf16 || !ema || n < 0 || k < 0) return MXFP4_INVALID_ARG;
    if (scale_mode != MXFP4_SCALE_TRUNCATION_FREE && scale_mode != MXFP4_SCALE_FLOOR) return MXFP4_INVALID_ARG;
    if (!(beta >= 0.f && beta <= 1.f)) return MXFP4_INVALID_ARG;
    if (k % 32 != 0) return MXFP4_BAD_SHAPE;
    mxfp4_status_t s = check_mat(dst, n, k);
    if (s) return s;
    if (!aligned16(w_bf16) || !aligned16(ema)) return MXFP4_MISALIGNED;
    OscPtrs op = {nullptr, nullptr, nullptr, nullptr, nullptr};
    if (osc) {
        if (!osc->w_prev || !osc->dist_w || !osc->dist_q) return MXFP4_INVALID_ARG;
        if ((s = check_mat(osc->wq_prev, n, k))) return s;
        if (!aligned16(osc->w_prev) || !aligned16(osc->dist_w) || !aligned16(osc->dist_q)) return MXFP4_MISALIGNED;
        op.w_prev = static_cast<__nv_bfloat16 *>(osc->w_prev);
        op.q_prev = static_cast<uint8_t *>(osc->wq_prev.data);
        op.s_prev = osc->wq_prev.scales;
        op.dist_w = osc->dist_w;
        op.dist_q = osc->dist_q;
    }
    if (n == 0 || k == 0) return MXFP4_OK;
    const int nblk = (int)(k / 32), nblk4 = (nblk + 3) / 4;
    const unsigned blocks = (unsigned)(ceil_div(n, 128) * nblk4 * 8);   // four threads per scale entry
    MX_CHECK_CUDA(launch_pdl(osc ? k_qema<true> : k_qema<false>, blocks, 1, 256, 0, st, static_cast<const __nv_bfloat16 *>(w_bf16), ema, beta, update_ema, n, nblk,
                             static_cast<uint8_t *>(dst.data), dst.scales, nblk4, scale_mode, op, dev_status));
    return MXFP4_OK;
}

mxfp4_status_t mxfp4_dequantize(mxfp4_mat_t src, float *dst, int64_t ld, void *stream)
{
    if (!dst || src.rows < 0 || src.cols < 0) return MXFP4_INVALID_ARG;
    if (src.cols % 32 != 0 || ld < src.cols) return MXFP4_BAD_SHAPE;
    mxfp4_status_t s = check_mat(src, src.rows, src.cols);
    if (s) return s;
    if (!aligned16(dst) || ld % 4 != 0) return MXFP4_MISALIGNED;
    if (src.rows == 0 || src.cols == 0) return MXFP4_OK;
    const int nblk = (int)(src.cols / 32), nblk4 = (nblk + 3) / 4;
    const unsigned blocks = (unsigned)ceil_div(src.rows * nblk, 256);
    MX_CHECK_CUDA(launch_pdl(k_dequantize, blocks, 1, 256, 0, static_cast<cudaStream_t>(stream), static_cast<const uint8_t *>(src.data), src.scales, src.rows, nblk,
                             nblk4, dst, ld));
    return MXFP4_OK;
}

}  // extern "C"
