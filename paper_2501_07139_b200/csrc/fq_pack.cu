// Quantiser, packer (canonical codes -> tiled field arrays) and exporters (back to canonical).
#include <cuda_fp16.h>

#include "fq_internal.cuh"

namespace fq {

#define FQ_CUDA_OK(expr) do { if ((expr) != cudaSuccess) return FQ_ERR_CUDA; } while (0)

// ---------------------------------------------------------------------------------------
// Quantiser: a code is decided by arithmetic in double, or by single precision where that cannot differ.
// ---------------------------------------------------------------------------------------

// Nearest-even conversion of a non-negative finite double to fp16 bits, done on the
// integer image of the double so that there is exactly one rounding.
__device__ __forceinline__ unsigned f64_to_f16_bits_nonneg(double v)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(u >> 52) & 0x7ff;
    if (e == 0) return 0u;
    if (e == 0x7ff) return 0x7c00u;
    const int E = e - 1023;
    const unsigned long long sig = (u & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    int drop = 42;                        // 53-bit significand -> 11 bits
    if (E < -14) drop += -14 - E;         // subnormal result keeps fewer bits
    if (drop > 63) return 0u;
    unsigned long long kept = sig >> drop;
    const unsigned long long lost = sig & ((1ull << drop) - 1ull);
    const unsigned long long tie = 1ull << (drop - 1);
    kept += (lost > tie) || (lost == tie && (kept & 1ull));
    if (E < -14) return (unsigned)kept;
    const unsigned long long r = ((unsigned long long)(E + 15) << 10) + kept - 1024ull;
    return r >= 0x7c00ull ? 0x7c00u : (unsigned)r;
}

// Bound by HBM: 4 bytes in, 1 out per weight.  A warp takes kQuantGroups groups at once, so that a lane has that many
// 16-byte loads in flight, and scale and zero point of a group are formed once, by one lane, instead of by all 32.  A code
// is rint(w / s) + z with the quotient in double; it is first formed as w * (1 / s), whose error for |w / s| < 1024 is below
// 1024 * 2^-24 < 2^-12 (s is an fp16 number, so exact; 1 / s is rounded once).  Only where the quotient is that close to a
// rounding boundary, or not finite, it is formed in double: the codes are the same integers.  11008 x 4096: 126 us with every division in double,
// about 40 us like this (225 MB, 34 us at the copy bandwidth).
constexpr int kQuantGroups = 8;                // groups per warp
constexpr int kQuantWarps = 8;
constexpr float kRint = 12582912.f;            // 1.5 * 2^23: adding it rounds to an integer, ties to even

__global__ void __launch_bounds__(kQuantWarps * 32, 4)
quantize_kernel(const float* __restrict__ w, long long n_groups_total, int bits,
                uint8_t* __restrict__ codes, uint16_t* __restrict__ scales, uint16_t* __restrict__ zeros)
{
    const int lane = threadIdx.x & 31;
    const long long g0 = ((long long)blockIdx.x * kQuantWarps + (threadIdx.x >> 5)) * kQuantGroups;
    if (g0 >= n_groups_total) return;
    const int n = (int)min((long long)kQuantGroups, n_groups_total - g0);
    const float top = (float)((1 << bits) - 1);
    const double qmax = top;
    float4 v[kQuantGroups];
#pragma unroll
    for (int i = 0; i < kQuantGroups; i++)
        v[i] = i < n ? __ldcs(reinterpret_cast<const float4*>(w + (g0 + i) * kGroup) + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
    // minimum and (negated) maximum of the eight groups: every step of the reduction halves the number of values a lane holds,
    // 17 shuffles in all instead of 80; lane l ends up with group (l >> 1) & 7
    float r[2 * kQuantGroups];
#pragma unroll
    for (int i = 0; i < kQuantGroups; i++) {
        r[i] = fminf(fminf(v[i].x, v[i].y), fminf(v[i].z, v[i].w));
        r[kQuantGroups + i] = -fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w));
    }
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) {
        const bool upper = lane & o;
#pragma unroll
        for (int i = 0; i < o / 2; i++) {
            const float keep = upper ? r[i + o / 2] : r[i], send = upper ? r[i] : r[i + o / 2];
            r[i] = fminf(keep, __shfl_xor_sync(0xffffffffu, send, o));
        }
    }
    r[0] = fminf(r[0], __shfl_xor_sync(0xffffffffu, r[0], 1));
    const float other = __shfl_xor_sync(0xffffffffu, r[0], 16);
    const float mn = lane & 16 ? other : r[0], mx = -(lane & 16 ? r[0] : other);
    const int mine = (lane >> 1) & (kQuantGroups - 1);
    static_assert(kQuantGroups == 8, "lanes of the reduction");
    float scale = 1.f, zero = 0.f;
    if (mine < n) {
        // scale = fp16((max - min) / qmax): in single precision the quotient is off by at most three units in the last
        // place, so its rounding to fp16 is the right one unless it lies within eight of them from a tie
        unsigned sb;
        const float f = (mx - mn) * (1.f / top);
        if (f >= 0x1p-14f && f < 60000.f && abs((int)(__float_as_uint(f) & 0x1fffu) - 0x1000) > 8) {
            sb = __half_as_ushort(__float2half_rn(f));
        } else {
            sb = f64_to_f16_bits_nonneg(((double)mx - (double)mn) / qmax);
            if (sb == 0u) sb = 0x0400u;
            if (sb >= 0x7c00u) sb = 0x7bffu;
        }
        scale = __half2float(__ushort_as_half((unsigned short)sb));  // exact
        // zero = clamp(rint(-min / scale)): as for the codes below
        const float ratio = -mn * (1.f / scale);
        zero = __fadd_rn(__fadd_rn(ratio, kRint), -kRint);
        if (!(fabsf(ratio) < 1024.f && fabsf(ratio - zero) < 0.5f - 0x1p-12f)) {
            const double z = rint(-(double)mn / (double)scale);
            zero = z > qmax ? top : (float)z;
        }
        if (!(zero > 0.f)) zero = 0.f;                               // (also -0 and NaN)
        if (zero > top) zero = top;
        if (lane == 2 * mine) {
            scales[g0 + mine] = (uint16_t)sb;
            zeros[g0 + mine] = __half_as_ushort(__float2half_rn(zero));   // an integer <= 255: exact
        }
    }
    const float inverse = 1.f / scale, shifted = kRint + zero;       // exact: a small integer
#pragma unroll
    for (int i = 0; i < kQuantGroups; i++) {
        const float inv = __shfl_sync(0xffffffffu, inverse, 2 * i), base = __shfl_sync(0xffffffffu, shifted, 2 * i);
        if (i >= n) break;
        const float vals[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        float u[4];
        bool sure = true;
#pragma unroll
        for (int e = 0; e < 4; e++) {
            u[e] = fmaf(vals[e], inv, base);                         // kRint + z + rint(w / s), one rounding
            const float off = fmaf(vals[e], inv, -(u[e] - base));    // how far w / s is from that integer
            sure = sure && fabsf(off) < 0.5f - 0x1p-12f;             // (false for NaN; beyond 1024 the code is clamped anyway)
            u[e] = fminf(fmaxf(u[e], kRint), kRint + top);           // the code is the low byte
        }
        if (!sure) {
            const double s = __half2float(__float2half_rn(1.f / inv)), z = base - kRint;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                double qd = rint((double)vals[e] / s) + z;
                qd = qd < 0.0 ? 0.0 : (qd > qmax ? qmax : qd);
                u[e] = kRint + (float)(unsigned)qd;                  // (NaN becomes 0)
            }
        }
        const unsigned packed = __byte_perm(__byte_perm(__float_as_uint(u[0]), __float_as_uint(u[1]), 0x0040),
                                            __byte_perm(__float_as_uint(u[2]), __float_as_uint(u[3]), 0x0040), 0x5410);
        reinterpret_cast<unsigned*>(codes + (g0 + i) * kGroup)[lane] = packed;
    }
}

int current_sm_count()
{
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 132;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 132;
        cached[dev] = n;
    }
    return cached[dev];
}

int launch_quantize(const float* w, int n_out, int k_in, int bits, uint8_t* codes, uint16_t* scales,
                    uint16_t* zeros, cudaStream_t st)
{
    const long long groups = (long long)n_out * (k_in / kGroup);
    if (groups < 1) return FQ_OK;
    const long long per_block = kQuantWarps * kQuantGroups;
    const long long blocks = (groups + per_block - 1) / per_block;
    if (blocks > 0x7fffffffll) return FQ_ERR_SHAPE;
    quantize_kernel<<<(unsigned)blocks, kQuantWarps * 32, 0, st>>>(w, groups, bits, codes, scales, zeros);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

// ---------------------------------------------------------------------------------------
// Packer (blob layout, see fq_layout.cuh): one block per blob, one warp per (superstep, row tile) of it.
//
// Bound by HBM (1 byte in, bits / 8 out per weight; the codes are usually still in L2 after the quantiser).  The 32 x 512
// codes of the blob go through shared memory with 16-byte loads; a lane then holds, as 32 words of four codes, exactly the A
// registers it owns in the decode kernel (rows g and g + 8, columns 4c .. 4c + 3 of every half k32 step), and a field is
// cut out of four codes at once with one shift and one AND, because a field never crosses a byte.  Every store is 16 bytes
// a lane, 512 contiguous bytes a warp.  11008 x 4096, 8 / 5 / 3 bits: 160 / 230 / 197 us with one thread per stored
// word gathering its codes byte by byte, about 13 us like this (whatever the width).
// ---------------------------------------------------------------------------------------
struct StoreArgs {
    const uint8_t* codes;          // canonical codes, one per byte
    const uint16_t* scales;
    const uint16_t* zeros;
    uint8_t* store;                // the stored variant
    int n_out, k_in, n_kb, groups;
    int stored_bits;               // bits of the stored variant (size of its blobs)
    FieldList fl;                  // fields that are written
    bool wide;                     // codes are 16-byte aligned (rows are multiples of 128 bytes)
    unsigned* high_zeros;          // set where a zero point is above 1023
};

constexpr int kPackThreads = kBlobSteps * kBlobTiles * 32;
constexpr int kPackCols = kBlobSteps * kStepCols;                // columns of a blob
constexpr int kPackRow = kPackCols + 16;                         // bytes between rows: lanes (g, c) hit banks 4g + c

// Field of width F at bit `shift`: registers of P = 8 / F consecutive k32 steps on top of each other.
template <int F>
__device__ __forceinline__ void pack_field(const uint32_t (&code)[8][4], int shift, uint8_t* dst)
{
    constexpr int P = 8 / F;
    constexpr uint32_t kMask = ((1u << F) - 1u) * 0x01010101u;
#pragma unroll
    for (int chunk = 0; chunk < F; chunk++) {
        uint32_t word[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int t = 0; t < P; t++)
#pragma unroll
            for (int a = 0; a < 4; a++) word[a] |= ((code[chunk * P + t][a] >> shift) & kMask) << (t * F);
        *reinterpret_cast<uint4*>(dst + chunk * 512) = make_uint4(word[0], word[1], word[2], word[3]);
    }
}

__global__ void __launch_bounds__(kPackThreads) pack_kernel(const __grid_constant__ StoreArgs a)
{
    __shared__ __align__(16) uint8_t tile_codes[kBlobTiles * kTileRows * kPackRow];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rp = (int)(blockIdx.x / (unsigned)a.n_kb), kb = (int)(blockIdx.x % (unsigned)a.n_kb);
    const long long n0 = (long long)rp * kBlobTiles * kTileRows;
    const int k0 = kb * kPackCols;
    uint8_t* blob = a.store + (long long)blockIdx.x * blob_bytes(a.stored_bits);

    uint4 raw[kBlobTiles * kTileRows / (kPackThreads / 32)];         // a warp reads a row of the blob, 16 bytes a lane
#pragma unroll
    for (int i = 0; i < (int)(sizeof raw / sizeof raw[0]); i++) {
        const int r = i * (kPackThreads / 32) + warp, k = k0 + lane * 16;
        raw[i] = make_uint4(0u, 0u, 0u, 0u);
        if (n0 + r < a.n_out && k < a.k_in) {                        // (k_in is a multiple of 128)
            const uint8_t* src = a.codes + (n0 + r) * a.k_in + k;
            if (a.wide) {
                raw[i] = *reinterpret_cast<const uint4*>(src);
            } else {
                uint32_t* w = reinterpret_cast<uint32_t*>(&raw[i]);
#pragma unroll
                for (int b = 0; b < 16; b++) w[b >> 2] |= (uint32_t)src[b] << (8 * (b & 3));
            }
        }
    }
    {   // scale/zero word: [superstep][tile][row & 7][group][row >> 3]
        const int off = t * 4;
        const int r = ((off >> 4) & 7) + 8 * ((off >> 2) & 1), grp = (off >> 3) & 1, tile = (off >> 7) & 1, ssl = off >> 8;
        const long long n = n0 + tile * kTileRows + r;
        const int g = (kb * kBlobSteps + ssl) * 2 + grp;
        unsigned v = 0;
        if (n < a.n_out && g < a.groups) {
            const float z = __half2float(__ushort_as_half(a.zeros[n * a.groups + g]));
            const unsigned zi = (unsigned)fminf(fmaxf(rintf(z), 0.f), 65535.f);
            v = (unsigned)a.scales[n * a.groups + g] | (zi << 16);
            if (zi > 1023u) *a.high_zeros = 1u;
        }
        reinterpret_cast<uint32_t*>(blob)[t] = v;
        static_assert(kBlobMetaBytes == 4 * kPackThreads, "one scale/zero word per thread");
    }
#pragma unroll
    for (int i = 0; i < (int)(sizeof raw / sizeof raw[0]); i++)
        *reinterpret_cast<uint4*>(tile_codes + (i * (kPackThreads / 32) + warp) * kPackRow + lane * 16) = raw[i];
    __syncthreads();

    const int ssl = warp / kBlobTiles, tile = warp % kBlobTiles, g = lane >> 2, c = lane & 3;
    uint32_t code[8][4];                                             // [k32 step][A register]
#pragma unroll
    for (int j = 0; j < 8; j++)
#pragma unroll
        for (int r = 0; r < 4; r++)
            code[j][r] = *reinterpret_cast<const uint32_t*>(tile_codes + (tile * kTileRows + g + 8 * (r & 1)) * kPackRow +
                                                            ssl * kStepCols + j * 32 + (r >> 1) * 16 + c * 4);
    int prefix = 0;
    for (int fi = 0; fi < a.fl.n; fi++) {
        const int f = a.fl.width[fi], shift = a.fl.shift[fi];
        uint8_t* dst = blob + blob_field_off(prefix, f, ssl, tile) + lane * 16;
        switch (f) {
            case 8: pack_field<8>(code, shift, dst); break;
            case 4: pack_field<4>(code, shift, dst); break;
            case 2: pack_field<2>(code, shift, dst); break;
            default: pack_field<1>(code, shift, dst); break;
        }
        prefix += f;
    }
}

static unsigned grid_for(long long total)
{
    long long b = (total + 255) / 256;
    if (b > (long long)current_sm_count() * 32) b = (long long)current_sm_count() * 32;
    return (unsigned)(b < 1 ? 1 : b);
}

int launch_pack(const uint8_t* codes, const uint16_t* scales, const uint16_t* zeros, int n_out, int k_in,
                int stored_bits, const FieldList& fl, void* store, unsigned* high_zeros, cudaStream_t st)
{
    StoreArgs a{};
    a.high_zeros = high_zeros;
    a.codes = codes; a.scales = scales; a.zeros = zeros; a.store = (uint8_t*)store;
    a.n_out = n_out; a.k_in = k_in; a.n_kb = k_blobs(k_in); a.groups = k_in / kGroup;
    a.stored_bits = stored_bits; a.fl = fl;
    a.wide = (reinterpret_cast<uintptr_t>(codes) & 15) == 0;
    const long long blobs = (long long)row_pairs(n_out) * a.n_kb;
    if (blobs > 0x7fffffffll) return FQ_ERR_SHAPE;
    pack_kernel<<<(unsigned)blobs, kPackThreads, 0, st>>>(a);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

// Scale/zero words are the first kBlobMetaBytes of every blob.
__global__ void __launch_bounds__(256) find_high_zeros_kernel(const uint8_t* store, long long blobs, int blob_stride, unsigned* high_zeros)
{
    constexpr int kWords = kBlobMetaBytes / 16;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < blobs * kWords; i += (long long)gridDim.x * blockDim.x) {
        const uint4 m = *reinterpret_cast<const uint4*>(store + i / kWords * blob_stride + i % kWords * 16);
        if (((m.x | m.y | m.z | m.w) >> 26) != 0u) *high_zeros = 1u;
    }
}

int launch_find_high_zeros(const void* store, int n_out, int k_in, int stored_bits, unsigned* high_zeros, cudaStream_t st)
{
    const long long blobs = (long long)row_pairs(n_out) * k_blobs(k_in);
    find_high_zeros_kernel<<<grid_for(blobs * (kBlobMetaBytes / 16)), 256, 0, st>>>((const uint8_t*)store, blobs, blob_bytes(stored_bits), high_zeros);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

// ---------------------------------------------------------------------------------------
// Exporters: rebuild canonical bytes from the stored variant (test / reporting support).
// ---------------------------------------------------------------------------------------
struct ExportArgs {
    const uint8_t* store;
    FieldList fl;                  // fields to read (a prefix of the stored ones for a nested child)
    int n_out, k_in, n_kb, groups, stored_bits, bits;
    uint32_t* out;
    uint16_t* scales;
    uint16_t* zeros;
    long long total_words;
};

__device__ __forceinline__ const uint8_t* blob_of(const ExportArgs& a, long long n, long long k, int& tile, int& ssl)
{
    const int rt = (int)(n / kTileRows), ss = (int)(k / kStepCols);
    tile = rt % kBlobTiles;
    ssl = ss % kBlobSteps;
    return a.store + ((long long)(rt / kBlobTiles) * a.n_kb + ss / kBlobSteps) * blob_bytes(a.stored_bits);
}

// The stored code of element (n, k), assembled from the fields in a.fl (shifts as stored).
__device__ __forceinline__ unsigned stored_code(const ExportArgs& a, long long n, long long k)
{
    int tile, ssl;
    const uint8_t* blob = blob_of(a, n, k, tile, ssl);
    const int r = (int)(n % kTileRows), kk = (int)(k % kStepCols);
    unsigned code = 0;
    int prefix = 0;
    for (int fi = 0; fi < a.fl.n; fi++) {
        const int f = a.fl.width[fi];
        const FieldPos p = field_pos(f, r, kk);
        const uint32_t wv = *reinterpret_cast<const uint32_t*>(blob + blob_field_off(prefix, f, ssl, tile) + p.word_byte);
        code |= ((wv >> p.bit) & ((1u << f) - 1u)) << a.fl.shift[fi];
        prefix += f;
    }
    return code;
}

__global__ void __launch_bounds__(256) export_packed_kernel(const ExportArgs a)
{
    const long long words_per_row = (long long)a.k_in * a.bits / 32;
    for (long long wi = (long long)blockIdx.x * blockDim.x + threadIdx.x; wi < a.total_words;
         wi += (long long)gridDim.x * blockDim.x) {
        const long long n = wi / words_per_row, w = wi % words_per_row;
        unsigned v = 0;
        for (int bit = 0; bit < 32; bit++) {
            const long long pos = w * 32 + bit;
            const long long k = pos / a.bits;
            const int j = (int)(pos % a.bits);
            v |= ((stored_code(a, n, k) >> j) & 1u) << bit;
        }
        a.out[wi] = v;
    }
}

// Canonical planes of the first `bits` stored planes: out[t][n][k/32], plane t = parent bit 7-t.
__global__ void __launch_bounds__(256) export_planes_kernel(const ExportArgs a)
{
    const long long words_per_row = a.k_in / 32;
    const long long words_per_plane = words_per_row * a.n_out;
    for (long long wi = (long long)blockIdx.x * blockDim.x + threadIdx.x; wi < a.total_words;
         wi += (long long)gridDim.x * blockDim.x) {
        const int t = (int)(wi / words_per_plane);
        const long long rem = wi % words_per_plane;
        const long long n = rem / words_per_row, w = rem % words_per_row;
        unsigned v = 0;
        for (int bit = 0; bit < 32; bit++)
            v |= ((stored_code(a, n, w * 32 + bit) >> (7 - t)) & 1u) << bit;
        a.out[wi] = v;
    }
}

__global__ void __launch_bounds__(256) export_meta_kernel(const ExportArgs a)
{
    const long long total = (long long)a.n_out * a.groups;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const long long n = i / a.groups;
        const int g = (int)(i % a.groups);
        int tile, ssl;
        const uint8_t* blob = blob_of(a, n, (long long)g * kGroup, tile, ssl);
        const uint32_t v = *reinterpret_cast<const uint32_t*>(blob + blob_meta_off(ssl, tile) +
                                                              blob_meta_word(g & 1, (int)(n % kTileRows)));
        a.scales[i] = (uint16_t)(v & 0xffffu);
        a.zeros[i] = __half_as_ushort(__float2half_rn((float)(v >> 16)));
    }
}

static void fill_export(ExportArgs& a, const void* store, int n_out, int k_in, int stored_bits, int bits,
                        const FieldList& fl)
{
    a.store = (const uint8_t*)store; a.fl = fl; a.n_out = n_out; a.k_in = k_in; a.n_kb = k_blobs(k_in);
    a.groups = k_in / kGroup; a.stored_bits = stored_bits; a.bits = bits;
    a.total_words = (long long)n_out * k_in * bits / 32;
}

int launch_export_packed(const void* store, int n_out, int k_in, int bits, const FieldList& fl, uint32_t* out,
                         cudaStream_t st)
{
    ExportArgs a{};
    fill_export(a, store, n_out, k_in, bits, bits, fl);
    a.out = out;
    export_packed_kernel<<<grid_for(a.total_words), 256, 0, st>>>(a);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

int launch_export_planes(const void* store, int n_out, int k_in, int bits, const FieldList& fl, uint32_t* out,
                         cudaStream_t st)
{
    ExportArgs a{};
    fill_export(a, store, n_out, k_in, 8, bits, fl);
    a.out = out;
    export_planes_kernel<<<grid_for(a.total_words), 256, 0, st>>>(a);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

int launch_export_meta(const void* store, int n_out, int k_in, int stored_bits, uint16_t* scales, uint16_t* zeros,
                       cudaStream_t st)
{
    ExportArgs a{};
    fill_export(a, store, n_out, k_in, stored_bits, stored_bits, FieldList{});
    a.scales = scales; a.zeros = zeros;
    export_meta_kernel<<<grid_for((long long)n_out * a.groups), 256, 0, st>>>(a);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

// ------------------------------------------------------------------------------- streaming read (measurement)
// Reads a buffer once with 16-byte loads, four in flight per thread, and folds the words into one value per
// thread block: what a kernel that only READS memory (as the decode path does) can reach on this part.
__global__ void __launch_bounds__(512) stream_read_kernel(const uint4* __restrict__ src, long long n16, unsigned* sink)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned acc = 0u;
    for (; i + 3 * stride < n16; i += 4 * stride) {
        const uint4 a = __ldcs(src + i), b = __ldcs(src + i + stride), c = __ldcs(src + i + 2 * stride), d = __ldcs(src + i + 3 * stride);
        acc ^= a.x ^ a.y ^ a.z ^ a.w ^ b.x ^ b.y ^ b.z ^ b.w ^ c.x ^ c.y ^ c.z ^ c.w ^ d.x ^ d.y ^ d.z ^ d.w;
    }
    for (; i < n16; i += stride) {
        const uint4 a = __ldcs(src + i);
        acc ^= a.x ^ a.y ^ a.z ^ a.w;
    }
    for (int o = 16; o > 0; o >>= 1) acc ^= __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && acc == 0x9e3779b9u) atomicXor(sink, acc);      // (keeps the loads alive; practically never taken)
}

int launch_stream_read(const void* src, size_t bytes, unsigned* sink, int sm_count, cudaStream_t st)
{
    stream_read_kernel<<<sm_count * 4, 512, 0, st>>>(static_cast<const uint4*>(src), (long long)(bytes / 16), sink);
    return cudaGetLastError() == cudaSuccess ? FQ_OK : FQ_ERR_CUDA;
}

}  // namespace fq
