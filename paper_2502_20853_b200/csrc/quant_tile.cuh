// The two passes of the tile quantizer over a 128 x 128 bf16 tile held in shared memory, shared by the streaming
// two-axis quantizer (tiles loaded by TMA) and the quantizing epilogue of the GEMM (tiles written by the epilogue warps).
// Tile layout: two boxes of 128 rows x 64 columns, one after the other, each with the 128B swizzle of a TMA tile
// (the 16-byte piece j of row r sits at piece j ^ (r & 7)).  256 threads take part.
#pragma once
#include "common.cuh"

namespace mx {

constexpr int kTile = 128;
constexpr int kTileBytes = kTile * kTile * 2;   // 32 KB


struct QuantSide {
    uint8_t *packed;
    uint8_t *scales;
    int nblk4;
    int scale_mode;
    SrStream sr;
};

__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// Scales of two groups at once, from the packed pair `am` of their 15-bit maxima: m2 = the packed pair of scale bytes plus 2,
// inv2 = the packed pair of 2^-s as bf16.  Valid for finite groups; all-zero groups get a byte of their own (98) where it is
// stored, their codes are zero with any scale.
__device__ __forceinline__ void group_scales_x2(uint32_t am, uint32_t tf_add2, uint32_t &m2, uint32_t &inv2)
{
    m2 = max_u16x2(((am + tf_add2) >> 7) & 0x01FF01FFu, 0x00020002u);   // the carry out of a mantissa is the increment
    inv2 = 0x80008000u - m2 * 128u;                                      // (254 - byte) << 7 in each half, no borrow across
}
// the maximum of both halves in both halves
__device__ __forceinline__ uint32_t max_both_halves(uint32_t am) { return max_u16x2(am, __byte_perm(am, am, 0x1032)); }

// 8 bf16 values held in one uint4, times the bf16 pair inv2 (2^-s in both halves) -> 8 FP32 latent values.
__device__ __forceinline__ void latents8(const uint4 &q, uint32_t inv2, float (&v)[8])
{
    scale_pair(q.x, inv2, v[0], v[1]);
    scale_pair(q.y, inv2, v[2], v[3]);
    scale_pair(q.z, inv2, v[4], v[5]);
    scale_pair(q.w, inv2, v[6], v[7]);
}

// The 8 codes (one u32, element 0 in the low nibble), round to nearest even.
__device__ __forceinline__ uint32_t rne8(const uint4 &q, uint32_t inv2)
{
    float v[8];
    latents8(q, inv2, v);
    return rne_x8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]);
}

// The same, and the codes' values times the bf16 pair sc2 (2^s in both halves) as bf16.  The converted bytes go on to the
// dequantization directly: taking them out of the packed word again is slower (137 against 131 us for the Q1 + Q6 pass at
// 50432 x 4096; 147 before).
__device__ __forceinline__ uint32_t rne8_dequant(const uint4 &q, uint32_t inv2, uint32_t sc2, uint32_t (&o)[4])
{
    float v[8];
    latents8(q, inv2, v);
    uint32_t r, h[4];
    asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b0, %6, %5;\n\tcvt.rn.satfinite.e2m1x2.f32 b1, %8, %7;\n\t"
        "cvt.rn.satfinite.e2m1x2.f32 b2, %10, %9;\n\tcvt.rn.satfinite.e2m1x2.f32 b3, %12, %11;\n\t"
        "mov.b32 %0, {b0, b1, b2, b3};\n\t"
        "cvt.rn.f16x2.e2m1x2 %1, b0;\n\tcvt.rn.f16x2.e2m1x2 %2, b1;\n\tcvt.rn.f16x2.e2m1x2 %3, b2;\n\tcvt.rn.f16x2.e2m1x2 %4, b3;\n\t}"
        : "=&r"(r), "=&r"(h[0]), "=&r"(h[1]), "=&r"(h[2]), "=&r"(h[3])
        : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]));
    scale_f16_pairs(h, sc2, o);
    return r;
}

// The same with stochastic rounding; r0 / r1 are the random words of elements 0..3 / 4..7.
__device__ __forceinline__ uint32_t sr8(const uint4 &q, uint32_t inv2, uint32_t r0, uint32_t r1)
{
    float v[8];
    latents8(q, inv2, v);
    return sr_x8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], r0, r1);
}

// max of the 15-bit magnitudes of the 8 bf16 values in q (NaN/Inf patterns compare as large magnitudes)
__device__ __forceinline__ uint32_t absmax_u4(uint32_t acc, const uint4 &q)
{
    acc = absmax2(acc, q.x);
    acc = absmax2(acc, q.y);
    acc = absmax2(acc, q.z);
    return absmax2(acc, q.w);
}

// The largest magnitude of a 32-element group, as bf16 bits (0x7F80 and above: it holds Inf / NaN).
__device__ __forceinline__ uint32_t group_amax(const uint4 (&q)[4])
{
    uint32_t am = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) am = absmax_u4(am, q[j]);
    return hmax_halves(am);
}

// The 16 bytes of codes of one 32-element group, round to nearest, and its scale byte (0xFF for a group with Inf / NaN, codes 0).
__device__ __forceinline__ uint4 rne_group(const uint4 (&q)[4], uint32_t tf_add, uint32_t &byte)
{
    const uint32_t am = group_amax(q);
    byte = 0xFFu;
    if (am >= 0x7F80u) return make_uint4(0, 0, 0, 0);
    byte = scale_byte_from_amax(am, tf_add);
    const uint32_t inv = inv_scale_bf16x2(byte);
    return make_uint4(rne8(q[0], inv), rne8(q[1], inv), rne8(q[2], inv), rne8(q[3], inv));
}

// Two FP32 values in one 64-bit register: an FMA of such pairs takes one issue slot (the passes are bound by issue).
__device__ __forceinline__ uint64_t f32x2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, float c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(f32x2(c, c)));
    return r;
}

// GELU (0.5 y (1 + erf(y / sqrt 2))) of a bf16 pair in FP32, rounded to bf16: max(y, 0) - |y| e with e = erfc(|y| / sqrt 2) / 2 =
// 2^(P(|y|) - 1), a form without cancellation: the small results of large negative y keep their digits.  P is a minimax fit (linear
// programming over [0, 13.2], where the result leaves the normal numbers) of log2 erfc(|y| / sqrt 2) without a constant term,
// degree 10, weighted so that the error of e stays within 1e-7 and within 1 % of e; its leading coefficient makes it fall for ever
// beyond.  Evaluated in |y| / 8 and with 8 e for |y| e, which keeps e a normal number for as long as the result.  Over all bf16 y the
// error is below 1.1e-7 |y| and 1.1 % of the result (down to 2^-125), and 113 results round to another bf16 than the exact value.
// The rational form of Abramowitz & Stegun 7.1.26 has 2.2e-7 |y|, 4 % and 169; degree 8 over [0, 6.2] behind 1 - e 6.9e-8 |y| and 197,
// and gives zero from y = -5.6 on.  Product and quantizer at 25216 x 1536 x 384: 58.5 us with that, 60.0 with this, 61.6 with
// degree 12 (6.6e-8 |y|, 17 results).
// +Inf gives +Inf (its magnitude is cut to the largest finite one: e = 0), -Inf and NaN give NaN.
__device__ __forceinline__ uint32_t gelu_bf16x2(uint32_t w)
{
    uint32_t cut, pos;
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(cut) : "r"(w), "r"(0x7F7F7F7Fu));
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(pos) : "r"(w), "r"(0x80008000u));   // -0 for y <= -0: a zero keeps its sign
    float a0, a1, p0, p1, e0, e1, t0, t1;
    scale_pair(cut & 0x7FFF7FFFu, 0x3E003E00u, a0, a1);
    const uint64_t a = f32x2(a0, a1);
    uint64_t p = fma_f32x2(f32x2(-2.7756042e+00f, -2.7756042e+00f), a, 1.7597485e+01f);
    p = fma_f32x2(p, a, -4.435496e+01f);
    p = fma_f32x2(p, a, 5.4649006e+01f);
    p = fma_f32x2(p, a, -2.7761135e+01f);
    p = fma_f32x2(p, a, -1.1350378e+01f);
    p = fma_f32x2(p, a, 3.0054832e+01f);
    p = fma_f32x2(p, a, -2.696964e+01f);
    p = fma_f32x2(p, a, -2.9386005e+01f);
    p = fma_f32x2(p, a, -9.208879e+00f);
    p = fma_f32x2(p, a, 2.0f);
    asm("mov.b64 {%0, %1}, %2;" : "=f"(p0), "=f"(p1) : "l"(p));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(p0));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(p1));
    uint64_t t;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(t) : "l"(a), "l"(f32x2(e0, e1)));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(t0), "=f"(t1) : "l"(t));
    uint32_t r;
    asm("{\n\t.reg .b16 l, h;\n\t.reg .f32 u, v;\n\tmov.b32 {l, h}, %1;\n\tsub.rn.f32.bf16 u, l, %2;\n\tsub.rn.f32.bf16 v, h, %3;\n\t"
        "cvt.rn.bf16x2.f32 %0, v, u;\n\t}" : "=r"(r) : "r"(pos), "f"(t0), "f"(t1));
    return r;
}

// Per-thread geometry of the two passes (the same for every tile of a launch).
//   row pass   : warps 0-3 take the left 64 columns, warps 4-7 the right; a lane pair shares a row (its two groups);
//                a thread handles rows r_row0 and r_row0 + 16
//   column pass: a warp takes the 32 rows x 64 columns it had in the row pass, a lane a pair of columns
// What depends on the thread alone is worked out here once; per tile the passes add what depends on the tile alone.
struct QsGeom {
    int r_row0, r_col;       // row pass: first row, first column
    uint32_t r_off[4];       // the thread's four 16-byte pieces inside its swizzled row
    uint32_t r_sc;           // its scale byte in the 512-byte chunk
    uint64_t r_q;            // its random counter (units of 16 elements)
    uint8_t *r_out;          // its codes
    int c_row, c_col;        // column pass: first row, first column
    uint32_t c_off[8];       // the column pair's word inside rows with (row & 7) = k
    uint32_t c_stage, c_sc;  // its codes in the staging tile, its first scale byte in the chunk
    uint64_t c_q;
};

__device__ __forceinline__ QsGeom qs_geom(int tid, int rows, int cols, uint8_t *row_codes)
{
    QsGeom g;
    const int warp = tid >> 5, lane = tid & 31, half = warp >> 2, rg = warp & 3;
    const int gg = lane & 1;
    g.r_row0 = rg * 32 + (lane >> 1);
    g.r_col = half * 64 + gg * 32;
#pragma unroll
    for (int j = 0; j < 4; j++) g.r_off[j] = (uint32_t)(half * (kTileBytes / 2) + g.r_row0 * 128 + (((gg * 4 + j) ^ (g.r_row0 & 7)) << 4));
    g.r_sc = (uint32_t)((lane >> 1) * 16 + rg * 4 + half * 2 + gg);
    g.r_q = (uint64_t)g.r_row0 * (uint64_t)(cols >> 4) + (uint64_t)(g.r_col >> 4);
    g.r_out = row_codes + ((int64_t)g.r_row0 * (cols >> 1) + (g.r_col >> 1));
    g.c_row = rg * 32;                // the same 32 rows x 64 columns this warp handled in the row pass: with DQ the column pass
    g.c_col = half * 64 + 2 * lane;   // reads only what its own warp wrote back, and a __syncwarp orders the two
#pragma unroll
    for (int k = 0; k < 8; k++)
        g.c_off[k] = (uint32_t)(half * (kTileBytes / 2) + rg * 32 * 128 + ((((lane >> 2) ^ k) << 4) | ((lane & 3) << 2)));
    // output rows c_col, c_col + 1 of the transposed tile: 16 bytes at piece rg, 64B swizzle (piece ^ ((row >> 1) & 3))
    g.c_stage = (uint32_t)(g.c_col * 64 + ((rg ^ (lane & 3)) << 4));
    g.c_sc = (uint32_t)((g.c_col & 31) * 16 + (g.c_col >> 5) * 4 + rg);
    g.c_q = (uint64_t)g.c_col * (uint64_t)(rows >> 4) + (uint64_t)(g.c_row >> 4);
    return g;
}

// Row pass: each thread quantizes two whole 32-element groups (Eq. 1, groups along the columns), stores their 16 bytes
// of codes straight to global memory and their scale bytes into the tile's 512-byte chunk `s_sc_row` (entries outside
// the matrix 0x7F).  st_base: shared-memory address of the tile; DQ: the exact dequantization P * 2^s of every group
// is written to the same position of the tile at dq_base (which may be st_base): double quantization, Sec. 3.3.
// The passes are bound by the instructions they issue (about 1.6 cycles each), so groups that hold Inf / NaN are quantized
// like any others and put right afterwards, behind one vote per pass (handling them in line cost 24 instructions per group,
// a tenth of the kernel's time).
// GELU: the tile holds Y and what is quantized is Z = bf16(GELU(Y)) (needs DQ: the column pass must not read the tile as it
// was); Z is stored too if hook_out is not null (bf16, leading dimension hook_ld).
template <bool SR_ROW, bool DQ, bool WIDE, bool GELU>
__device__ __forceinline__ void qs_row_pass(const QsGeom &g, uint32_t st_base, uint32_t dq_base, int row0, int col0, int rows, int cols,
                                            const QuantSide &rw, uint32_t tfa_r2, uint8_t *s_sc_row, uint32_t &nonfinite, __nv_bfloat16 *hook_out, int64_t hook_ld)
{
    uint8_t *out = g.r_out + ((int64_t)row0 * (cols >> 1) + (col0 >> 1));
    const uint64_t tile_q = (uint64_t)row0 * (uint64_t)(cols >> 4) + (uint64_t)(col0 >> 4);
    const int rows_left = col0 + g.r_col < cols ? rows - row0 - g.r_row0 : 0;
    uint32_t ams[2];
#pragma unroll
    for (int item = 0; item < 2; item++) {
        uint4 q[4];
#pragma unroll
        for (int j = 0; j < 4; j++)
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(q[j].x), "=r"(q[j].y), "=r"(q[j].z), "=r"(q[j].w)
                         : "r"(st_base + g.r_off[j] + (uint32_t)(item * 16 * 128)));
        if (GELU) {
#pragma unroll
            for (int j = 0; j < 4; j++) q[j] = make_uint4(gelu_bf16x2(q[j].x), gelu_bf16x2(q[j].y), gelu_bf16x2(q[j].z), gelu_bf16x2(q[j].w));
            if (hook_out != nullptr && rows_left > item * 16) {
                uint4 *z = reinterpret_cast<uint4 *>(hook_out + (int64_t)(row0 + g.r_row0 + item * 16) * hook_ld + col0 + g.r_col);
#pragma unroll
                for (int j = 0; j < 4; j++) z[j] = q[j];
            }
        }
        uint32_t am4[4];
#pragma unroll
        for (int j = 0; j < 4; j++) am4[j] = absmax_fold(absmax_fold(q[j].x, q[j].y), absmax_fold(q[j].z, q[j].w));
        const uint32_t am = max_both_halves(absmax_fold_end(absmax_fold(absmax_fold(am4[0], am4[1]), absmax_fold(am4[2], am4[3]))));
        ams[item] = am;
        uint32_t m2, inv;
        group_scales_x2(am, tfa_r2, m2, inv);                    // both halves alike
        // with DQ P * 2^s goes back into the staged tile (exact in bf16)
        const uint32_t sc2 = am ? max_u16x2((m2 - 0x00020002u) << 7, 0x00400040u) : 98u * 0x00800080u;   // byte 0: 2^-127
        uint32_t c[4], o[4][4];
        if (SR_ROW) {
            const uint64_t q0 = tile_q + g.r_q + (uint64_t)((int64_t)item * cols);    // 16 rows of cols / 16 counters further
            const uint4 ra = sr_words<WIDE>(rw.sr, q0), rb = sr_words<WIDE>(rw.sr, q0 + 1);
            c[0] = sr8(q[0], inv, ra.x, ra.y), c[1] = sr8(q[1], inv, ra.z, ra.w), c[2] = sr8(q[2], inv, rb.x, rb.y), c[3] = sr8(q[3], inv, rb.z, rb.w);
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (DQ) dequant_x8(c[j], sc2, o[j]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) c[j] = DQ ? rne8_dequant(q[j], inv, sc2, o[j]) : rne8(q[j], inv);
        }
        if (DQ) {
#pragma unroll
            for (int j = 0; j < 4; j++)
                asm volatile("st.shared.v4.u32 [%4], {%0,%1,%2,%3};" ::"r"(o[j][0]), "r"(o[j][1]), "r"(o[j][2]), "r"(o[j][3]),
                             "r"(dq_base + g.r_off[j] + (uint32_t)(item * 16 * 128)) : "memory");
        }
        const uint4 codes = make_uint4(c[0], c[1], c[2], c[3]);
        const bool in = rows_left > item * 16;
        if (in) *reinterpret_cast<uint4 *>(out + (int64_t)(item * 8) * cols) = codes;
        s_sc_row[g.r_sc + item * 256] = (uint8_t)(!in ? 0x7Fu : am ? m2 - 2u : 98u);
    }
    if (__any_sync(0xFFFFFFFFu, max(ams[0], ams[1]) >= 0x7F800000u)) {
        // Inf / NaN: scale byte 0xFF, codes 0, NaN for the pass that reads the dequantized group
#pragma unroll 1
        for (int item = 0; item < 2; item++) {
            if ((item ? ams[1] : ams[0]) < 0x7F800000u || rows_left <= item * 16) continue;
            *reinterpret_cast<uint4 *>(out + (int64_t)(item * 8) * cols) = make_uint4(0u, 0u, 0u, 0u);
            s_sc_row[g.r_sc + item * 256] = 0xFF;
            nonfinite = 1u;
            if (DQ) {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    asm volatile("st.shared.v4.u32 [%1], {%0,%0,%0,%0};" ::"r"(0x7FC07FC0u), "r"(dq_base + g.r_off[j] + (uint32_t)(item * 16 * 128)) : "memory");
            }
        }
    }
}

// Column pass: each thread quantizes two adjacent columns x 32 rows, i.e. two whole groups of the transposed output
// (groups of 32 source rows, Sec. 3.3 "Block Format"), writes their codes into the 64B-swizzled staging tile
// `staging` (128 output rows x 64 bytes, for one TMA store) and their scale bytes into the chunk `s_sc_t`.
template <bool SR_T, bool WIDE>
__device__ __forceinline__ void qs_col_pass(const QsGeom &g, uint32_t st_base, int row0, int col0, int rows, int cols, const QuantSide &tr,
                                            uint32_t tfa_t2, uint8_t *staging, uint8_t *s_sc_t, uint32_t &nonfinite)
{
    uint32_t v[32];
#pragma unroll
    for (int i = 0; i < 32; i++) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v[i]) : "r"(st_base + g.c_off[i & 7] + (uint32_t)i * 128u));
    uint32_t am8[8];
#pragma unroll
    for (int k = 0; k < 8; k++) am8[k] = absmax_fold(absmax_fold(v[4 * k], v[4 * k + 1]), absmax_fold(v[4 * k + 2], v[4 * k + 3]));
    const uint32_t am = absmax_fold_end(absmax_fold(absmax_fold(absmax_fold(am8[0], am8[1]), absmax_fold(am8[2], am8[3])),
                                                    absmax_fold(absmax_fold(am8[4], am8[5]), absmax_fold(am8[6], am8[7]))));   // maxima of the two columns, one per half
    uint32_t m2, inv2;
    group_scales_x2(am, tfa_t2, m2, inv2);
    uint32_t lo[4], hi[4];                                     // 32 codes of the first / second column
    uint4 ra[2], rb[2];
    if (SR_T) {
        const uint64_t qa = (uint64_t)col0 * (uint64_t)(rows >> 4) + (uint64_t)(row0 >> 4) + g.c_q;
        const uint64_t qb = qa + (uint64_t)(rows >> 4);
        ra[0] = sr_words<WIDE>(tr.sr, qa), ra[1] = sr_words<WIDE>(tr.sr, qa + 1);
        rb[0] = sr_words<WIDE>(tr.sr, qb), rb[1] = sr_words<WIDE>(tr.sr, qb + 1);
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        float a[8], b[8];                                      // eight rows of the first / second column
#pragma unroll
        for (int i = 0; i < 8; i++) scale_pair(v[8 * k + i], inv2, a[i], b[i]);
        if (SR_T) {
            const uint4 &wa = ra[k >> 1], &wb = rb[k >> 1];
            lo[k] = sr_x8(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], (k & 1) ? wa.z : wa.x, (k & 1) ? wa.w : wa.y);
            hi[k] = sr_x8(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7], (k & 1) ? wb.z : wb.x, (k & 1) ? wb.w : wb.y);
        } else {
            lo[k] = rne_x8(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7]);
            hi[k] = rne_x8(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7]);
        }
    }
    *reinterpret_cast<uint4 *>(staging + g.c_stage) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<uint4 *>(staging + g.c_stage + 64) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    const bool in = col0 + g.c_col < cols && row0 + g.c_row < rows;     // columns come in blocks of 32: both or neither
    uint32_t byte0 = (am & 0xFFFFu) ? m2 - 2u : 98u, byte1 = am >= 0x10000u ? (m2 >> 16) - 2u : 98u;   // in the low eight bits
    if (!in) byte0 = byte1 = 0x7Fu;
    s_sc_t[g.c_sc] = (uint8_t)byte0;
    s_sc_t[g.c_sc + 16] = (uint8_t)byte1;
    const uint32_t nfm = (am + 0x00800080u) & 0x80008000u;              // bit 15 of the half of a non-finite group
    if (__any_sync(0xFFFFFFFFu, nfm != 0u)) {
        if ((nfm & 0x8000u) && in) {
            *reinterpret_cast<uint4 *>(staging + g.c_stage) = make_uint4(0u, 0u, 0u, 0u);
            s_sc_t[g.c_sc] = 0xFF;
        }
        if ((nfm >> 31) && in) {
            *reinterpret_cast<uint4 *>(staging + g.c_stage + 64) = make_uint4(0u, 0u, 0u, 0u);
            s_sc_t[g.c_sc + 16] = 0xFF;
        }
        nonfinite |= (uint32_t)(nfm != 0u && in);
    }
}

// Both passes over a tile, by the width of the random streams' counters (a launch-uniform branch around the whole tile).
// With DQ the column pass reads what the row pass of the SAME warp wrote to dq_base.
template <bool SR_ROW, bool SR_T, bool DQ, bool WIDE, bool GELU>
__device__ __forceinline__ void qs_tile_w(const QsGeom &g, uint32_t st_base, uint32_t dq_base, int row0, int col0, int rows, int cols, bool emit_row,
                                          bool emit_t, const QuantSide &rw, const QuantSide &tr, uint32_t tfa_r2, uint32_t tfa_t2, uint8_t *staging,
                                          uint8_t *s_sc_row, uint8_t *s_sc_t, uint32_t &nonfinite, __nv_bfloat16 *hook_out, int64_t hook_ld)
{
    if (emit_row)
        qs_row_pass<SR_ROW, DQ, WIDE, GELU>(g, st_base, dq_base, row0, col0, rows, cols, rw, tfa_r2, s_sc_row, nonfinite, hook_out, hook_ld);
    if (DQ) __syncwarp();
    if (emit_t) qs_col_pass<SR_T, WIDE>(g, DQ ? dq_base : st_base, row0, col0, rows, cols, tr, tfa_t2, staging, s_sc_t, nonfinite);
}
template <bool SR_ROW, bool SR_T, bool DQ, bool GELU = false>
__device__ __forceinline__ void qs_tile(const QsGeom &g, uint32_t st_base, uint32_t dq_base, int row0, int col0, int rows, int cols, bool emit_row,
                                        bool emit_t, const QuantSide &rw, const QuantSide &tr, uint32_t tfa_r2, uint32_t tfa_t2, uint8_t *staging,
                                        uint8_t *s_sc_row, uint8_t *s_sc_t, uint32_t &nonfinite, __nv_bfloat16 *hook_out = nullptr, int64_t hook_ld = 0)
{
    if ((SR_ROW || SR_T) && (rw.sr.wide | tr.sr.wide))
        qs_tile_w<SR_ROW, SR_T, DQ, true, GELU>(g, st_base, dq_base, row0, col0, rows, cols, emit_row, emit_t, rw, tr, tfa_r2, tfa_t2, staging, s_sc_row, s_sc_t,
                                                nonfinite, hook_out, hook_ld);
    else
        qs_tile_w<SR_ROW, SR_T, DQ, false, GELU>(g, st_base, dq_base, row0, col0, rows, cols, emit_row, emit_t, rw, tr, tfa_r2, tfa_t2, staging, s_sc_row, s_sc_t,
                                                 nonfinite, hook_out, hook_ld);
}

}  // namespace mx
