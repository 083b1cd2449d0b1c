// Arithmetic of the batch decode kernel: stored words -> fp16 operands of mma.m16n8k16 (fp16 x fp16 -> fp32).
//
// The weights enter as the exact integers q - z (fp16 holds every integer up to 2048), the activations as the fp16 numbers
// they are; products and sums of a group of 128 columns are formed in fp32 and scaled once per group.  One MMA serves 16
// columns of 16 rows for up to eight batch entries, so the fields of a code are merged first (one shift and one AND-OR per
// field and four codes) instead of being multiplied one by one.
//
//   codes -> fp16: a byte q in the low mantissa bits under the exponent of 1024 is the fp16 number 1024 + q; codes that sit at
//   bit p of their byte give 1024 + q * 2^p, and fma(., 2^-p, -(1024 * 2^-p + z)) is q - z exactly.  Which p costs the fewest
//   shifts is chosen at compile time per k32 step.
//
//   The constant is exact for z below 1024, which covers every quantiser of up to eight bits; stored zero points have 16 bits.  Where a
//   context holds higher ones, their upper bits are taken out of a blob before it is computed (blob_take_high_zeros), in a kernel of
//   its own: a test, a mask or one more register in the usual one costs 2 - 7 % of the 13B stack at batch 8.
#pragma once
#include <cuda_fp16.h>

#include <cstdint>

#include "fq_layout.cuh"
#include "fq_merge.cuh"
#include "fq_ptx.cuh"

namespace fq {

// Batch entries are padded to 4 or 8: the width of the activation image and of the published sums.
FQ_HDC int batch_pad(int batch) { return batch <= 4 ? 4 : 8; }
// Activations in shared memory: the rows as they are in global memory, kXRowPad bytes more than a chunk of `kXCols` columns
// apart: the 8-byte loads of half a warp (four rows, four column runs) then hit every bank once.
constexpr int kXCols = kBlobSteps * kStepCols;
constexpr int kXRowPad = 32;
constexpr int kXRowBytes = kXCols * 2 + kXRowPad;

// D (+)= A(16 x 16 fp16, row) * B(16 x 8 fp16, col), fp32.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Where the code lies inside its byte in k32 step j of a superstep (bit p): the place that leaves the most fields where they
// are.  The nested formats keep p = 0: their codes are the top bits of the parent's byte.
FQ_HDC int field_bit(const FieldList& fl, int i, int j) { return (j % (8 / fl.width[i])) * fl.width[i]; }
FQ_HDC int code_place(int variant, int j)
{
    if (variant >= 7) return 0;
    const FieldList fl = variant_fields(variant);
    const int bits = variant + 2;
    int best = 0, best_moves = 99;
    for (int p = 0; p + bits <= 8; p++) {
        int moves = 0;
        for (int i = 0; i < fl.n; i++) moves += field_bit(fl, i, j) != fl.shift[i] + p ? 1 : 0;
        if (moves < best_moves) { best = p; best_moves = moves; }
    }
    return best;
}

template <int VARIANT, int J>
__device__ __forceinline__ uint32_t half2_of(uint32_t biased, __half2 neg_zero)
{
    constexpr int p = code_place(VARIANT, J);
    const __half2 v = *reinterpret_cast<const __half2*>(&biased);
    // neg_zero = -z;  -(1024 * 2^-p) - z is exact for z < 1024
    const __half2 c = __hadd2(__float2half2_rn(-1024.f / (float)(1 << p)), neg_zero);
    const __half2 d = p == 0 ? __hadd2(v, c) : __hfma2(v, __float2half2_rn(1.f / (float)(1 << p)), c);
    return *reinterpret_cast<const uint32_t*>(&d);
}

// One group of 128 columns (k32 steps 4 * GRP .. + 3 of a superstep) of one 16-row tile: acc[0] + acc[1] = sum_k (q_k - z) * x_k.
//   fa[i] : shared address of this lane's 16-byte chunk 0 of field i of the tile        xa : this lane's activations of the superstep
//   nz[r] : -(zero point) of rows g, g + 8, twice
template <int VARIANT, int GRP>
__device__ __forceinline__ void group_mma(const uint32_t (&fa)[kMaxFields], uint32_t xa, const __half2 (&nz)[2], float (&acc)[2][4])
{
    constexpr FieldList FL = variant_fields(VARIANT);
    // a nested child's dropped bits are filled with their mid-point
    constexpr uint32_t kFill = (VARIANT >= 7 && VARIANT < 13) ? (1u << (7 - (VARIANT - 5))) * 0x01010101u : 0u;
    uint4 raw[FL.n];                                                            // the chunk of every field that holds step j
    uint2 x[8];                                                                 // [k16 step]: columns 4c .. 4c + 3 of it
    static_for<0, 8>([&](auto H) { x[decltype(H)::value] = lds64<(8 * GRP + decltype(H)::value) * 32>(xa); });
    // a nested child of three or more bits: the words of all four steps are merged at once (fq_merge.cuh).  Four 7B blocks, 4 / 8
    // entries, without dependencies: 4 bits 134 / 135 -> 132 / 133 us, 6 bits 154.5 / 157 -> 152.4 / 157
    constexpr bool kMerged = VARIANT >= 7 && FL.n >= 2;
    uint32_t merged[4][4];                                                      // [A register][step]
    if constexpr (kMerged) {
        static_for<0, FL.n>([&](auto FI) { raw[decltype(FI)::value] = lds128<GRP * 512>(fa[decltype(FI)::value]); });
#pragma unroll
        for (int r = 0; r < 4; r++) {
            uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int i = 0; i < FL.n; i++) w[i] = r == 0 ? raw[i].x : r == 1 ? raw[i].y : r == 2 ? raw[i].z : raw[i].w;
            merge_bytes<FL.n, FL.keep[FL.n - 1]>(w, merged[r]);
        }
    }
    static_for<0, 4>([&](auto JJ) {
        constexpr int j = 4 * GRP + decltype(JJ)::value, place = code_place(VARIANT, j);
        uint32_t lo[4], hi[4];                                                  // columns 4c, 4c + 1 and 4c + 2, 4c + 3
        {
            uint32_t code[4] = {kFill, kFill, kFill, kFill};
            if constexpr (kMerged) {
#pragma unroll
                for (int r = 0; r < 4; r++) code[r] |= merged[r][j & 3];
            } else static_for<0, FL.n>([&](auto FI) {
                constexpr int fi = decltype(FI)::value, F = FL.width[fi], P = 8 / F;
                constexpr int at = (j % P) * F, to = FL.shift[fi] + place;
                constexpr uint32_t m = (field_keep_mask(F, FL.keep[fi]) * 0x01010101u) << to;
                if constexpr (j % P == 0 || j % 4 == 0) raw[fi] = lds128<(j / P) * 512>(fa[fi]);
                const uint32_t ww[4] = {raw[fi].x, raw[fi].y, raw[fi].z, raw[fi].w};
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    const uint32_t moved = at >= to ? ww[r] >> (at - to) : ww[r] << (to - at);
                    code[r] = F == 8 ? ww[r] : ((moved & m) | code[r]);
                }
            });
#pragma unroll
            for (int r = 0; r < 4; r++) {
                lo[r] = __byte_perm(code[r], 0x64646464u, 0x4140);
                hi[r] = __byte_perm(code[r], 0x64646464u, 0x4342);
            }
        }
        static_for<0, 2>([&](auto H) {                                          // register 2 * half + row half
            constexpr int h = decltype(H)::value;
            const uint2 xj = x[2 * (j & 3) + h];
            mma_f16(acc[h], half2_of<VARIANT, j>(lo[2 * h], nz[0]), half2_of<VARIANT, j>(lo[2 * h + 1], nz[1]),
                    half2_of<VARIANT, j>(hi[2 * h], nz[0]), half2_of<VARIANT, j>(hi[2 * h + 1], nz[1]), xj.x, xj.y);
        });
    });
}

// A blob, one 16-row tile: tot[0..1] row g, tot[2..3] row g + 8, batch entries 2c, 2c + 1.
//   blob : its shared address        xs : of the activation slot
template <int VARIANT, int BP>
__device__ __forceinline__ void blob_compute(uint32_t blob, uint32_t xs, int lane, int tile, float (&tot)[4])
{
    constexpr FieldList FL = variant_fields(VARIANT);
    const int g = lane >> 2, c = lane & 3;
    // batch entries beyond the padding read a valid entry's activations; nobody uses what they add up to
    uint32_t xa = xs + (uint32_t)((g & (BP - 1)) * kXRowBytes + c * 8);
#pragma unroll 1                                                     // (keeps the specialised loops small)
    for (int ss = 0; ss < kBlobSteps; ss++, xa += kStepCols * 2) {
        const int st_tile = ss * kBlobTiles + tile;
        uint32_t fa[kMaxFields];
        static_for<0, FL.n>([&](auto FI) {
            constexpr int fi = decltype(FI)::value;
            constexpr int prefix = [] { int p = 0; for (int i = 0; i < fi; i++) p += variant_fields(VARIANT).width[i]; return p; }();
            fa[fi] = blob + kBlobMetaBytes + kBlobSteps * kBlobTiles * 512 * prefix + st_tile * (FL.width[fi] * 512) + lane * 16;
        });
        const uint4 m4 = lds128(blob + st_tile * 128 + g * 16);   // scale/zero words: group 0 rows g, g + 8, group 1 rows g, g + 8
        static_for<0, 2>([&](auto G) {
            constexpr int grp = decltype(G)::value;
            const uint32_t m[2] = {grp ? m4.z : m4.x, grp ? m4.w : m4.y};
            __half2 nz[2];
            float sc[2];
#pragma unroll
            for (int r = 0; r < 2; r++) {
                sc[r] = __half2float(__ushort_as_half((unsigned short)(m[r] & 0xffffu)));
                nz[r] = __half2half2(__hneg(__ushort2half_rn((unsigned short)(m[r] >> 16))));
            }
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};      // two chains: an MMA waits long for its sums
            group_mma<VARIANT, grp>(fa, xa, nz, acc);
#pragma unroll
            for (int i = 0; i < 4; i++) tot[i] = fmaf(sc[i >> 1], acc[0][i] + acc[1][i], tot[i]);
        });
    }
}

// Takes the zero points of a blob's row tile (nobody else reads those words) down to their low ten bits; tot gets what
// that leaves out, -s * (upper bits of z) * (sum of the activations) over the groups.  The sums come from MMAs whose weights are all
// one, in the layout of tot.
template <int BP>
__device__ __forceinline__ void blob_take_high_zeros(uint32_t blob, uint32_t xs, int lane, int tile, float (&tot)[4])
{
    constexpr uint32_t kOnes = 0x3c003c00u;                           // 1.0 twice
    const int g = lane >> 2, c = lane & 3;
    uint32_t xa = xs + (uint32_t)((g & (BP - 1)) * kXRowBytes + c * 8);
#pragma unroll 1
    for (int i = 0; i < 2 * kBlobSteps; i++, xa += kGroup * 2) {      // one group at a time
        const uint32_t words = blob + (uint32_t)((i / 2 * kBlobTiles + tile) * 128 + g * 16 + (i & 1) * 8);
        const uint2 m = lds64(words);                                 // rows g, g + 8
        if (!__any_sync(0xffffffffu, ((m.x | m.y) >> 26) != 0u)) continue;
        float sums[4] = {0.f, 0.f, 0.f, 0.f};
        static_for<0, kGroup / 16>([&](auto H) {
            const uint2 x = lds64<decltype(H)::value * 32>(xa);
            mma_f16(sums, kOnes, kOnes, kOnes, kOnes, x.x, x.y);
        });
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const uint32_t w = e < 2 ? m.x : m.y;
            const float share = __half2float(__ushort_as_half((unsigned short)(w & 0xffffu))) * (float)((w >> 16) & ~1023u);   // exact: 11 x 6 bits
            tot[e] = fmaf(-share, sums[e], tot[e]);
        }
        if (c == 0) sts64(words, make_uint2(m.x & 0x03ffffffu, m.y & 0x03ffffffu));           // (all lanes have read them: the vote)
    }
    __syncwarp();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the next copy into this place comes after these stores
}

template <int BP>
__device__ __forceinline__ void blob_dispatch(int variant, uint32_t blob, uint32_t xs, int lane, int tile, float (&tot)[4])
{
#define FQ_VARIANT_CASE(V) case V: blob_compute<V, BP>(blob, xs, lane, tile, tot); break;
    switch (variant) {
        FQ_VARIANT_CASE(0) FQ_VARIANT_CASE(1) FQ_VARIANT_CASE(2) FQ_VARIANT_CASE(3) FQ_VARIANT_CASE(4)
        FQ_VARIANT_CASE(5) FQ_VARIANT_CASE(6) FQ_VARIANT_CASE(7) FQ_VARIANT_CASE(8) FQ_VARIANT_CASE(9)
        FQ_VARIANT_CASE(10) FQ_VARIANT_CASE(11) FQ_VARIANT_CASE(12) FQ_VARIANT_CASE(13)
        default: break;
    }
#undef FQ_VARIANT_CASE
    static_assert(kVariants == 14, "one case per variant");
}

}  // namespace fq
