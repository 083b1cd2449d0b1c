// Prefill path:  Y[m][n] = sum_k X[m][k] * w^[n][k],  X and Y bf16, fp32 accumulation in TMEM.
//
// Two kernels per call:
//   1. dequant_kernel    stored blobs -> w^ as bf16 [n_out][k_in] in the context workspace
//                        (w^ = (q - z) * s computed exactly in fp32, rounded once to bf16);
//   2. gemm_pair_kernel  a persistent, warp-specialised tcgen05 GEMM over pairs of SMs (cta_group::2): a tile is 256 tokens x up
//                        to 256 outputs, each CTA of the pair keeps 128 of the tokens and half of the outputs' weights in its
//                        shared memory (six stages of 64 columns) and its 128 tokens' sums in its TMEM (two accumulators, so
//                        that four warps drain one while the MMAs fill the other).
// Every mbarrier wait is bounded by a timer; when one runs out the kernel records FQ_ERR_TIMEOUT,
// all roles leave their loops, and the TMEM allocation is released before the CTA exits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fq_dequant.cuh"
#include "fq_internal.cuh"
#include "fq_ptx.cuh"
#include "fq_umma.cuh"

namespace fq {

#define FQ_CUDA_OK(expr) do { if ((expr) != cudaSuccess) return FQ_ERR_CUDA; } while (0)

// ------------------------------------------------------------------------------- dequantise to bf16
struct DequantArgs {
    const uint8_t* store;
    int n_out, k_in, n_kb, blob_stride;
    int zero_adjust;
    __nv_bfloat16* out;              // [n_out][k_in]
};

// One warp per (row strip of 32, 64 columns): the lanes read the stored words of the two k32 steps exactly as
// the decode kernel does (16 bytes per lane and field chunk), merge the fields into four codes per register,
// convert (w^ = (q - z) * s exactly, one rounding to bf16) and write 8-byte runs; the four lanes of a quad
// cover 32 contiguous bytes of a row.  Specialised per field list like fq_gemm_split.cu, whose helpers it shares.
template <int VARIANT>
__global__ void __launch_bounds__(256) dequant_kernel(const DequantArgs a)
{
    constexpr FieldList FL = variant_fields(VARIANT);
    constexpr int kLoads = fields_loads(FL, FL.n);
    constexpr bool kSmallCodes = VARIANT < 6;            // PACKED 2..7 bits: codes below 128, no zero adjustment
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, c = lane & 3;
    const int n_rp = row_pairs(a.n_out), n_st = a.k_in / 64;
    const long long total = (long long)n_rp * n_st;
    const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long ti = warp0; ti < total; ti += n_warps) {
        const int rp = (int)(ti / n_st), ks = (int)(ti % n_st);       // consecutive warps: consecutive columns of a strip
        const int kb = ks >> 3, ssl = (ks >> 2) & 1, j0 = (ks & 3) * 2, grp = (ks >> 1) & 1;
        const uint8_t* blob_lane = a.store + ((long long)rp * a.n_kb + kb) * a.blob_stride + lane * 16;
        uint4 raw[kBlobTiles][kLoads];
        uint2 meta[kBlobTiles];
        load_stage_words<VARIANT, 0>(blob_lane, ssl, j0, raw[0]);
        load_stage_words<VARIANT, 1>(blob_lane, ssl, j0, raw[1]);
#pragma unroll
        for (int tl = 0; tl < kBlobTiles; tl++)
            meta[tl] = __ldg(reinterpret_cast<const uint2*>(blob_lane - lane * 16 + blob_meta_off(ssl, tl) + blob_meta_word(grp, g)));
#pragma unroll
        for (int tl = 0; tl < kBlobTiles; tl++) {
            uint32_t code[2][4];
            merge_codes<VARIANT>(raw[tl], j0, code);
            const uint32_t mm[2] = {meta[tl].x, meta[tl].y};
#pragma unroll
            for (int hr = 0; hr < 2; hr++) {
                const long long n = (long long)rp * 32 + tl * kTileRows + g + 8 * hr;
                if (n >= a.n_out) continue;
                const float s = __half2float(__ushort_as_half((unsigned short)(mm[hr] & 0xffffu)));
                const WideZero zz(mm[hr], a.zero_adjust, s);
                const float cc = -(float)(128 + (int)(mm[hr] >> 16)) * s;
                __nv_bfloat16* row = a.out + n * a.k_in + ks * 64 + 4 * c;
#pragma unroll
                for (int jj = 0; jj < 2; jj++)
#pragma unroll
                    for (int half = 0; half < 2; half++) {
                        const uint32_t q4 = code[jj][2 * half + hr];          // A register r = 2 * half + row half
                        const uint2 o = kSmallCodes ? small_codes_to_bf16(q4, cc, s) : codes_to_bf16(q4, zz, s);
                        *reinterpret_cast<uint2*>(row + 32 * jj + 16 * half) = o;
                    }
            }
        }
    }
}

template <int VARIANT>
static int launch_dequant(const DequantArgs& da, int sm_count, cudaStream_t st)
{
    const long long items = (long long)row_pairs(da.n_out) * (da.k_in / 64);     // one warp each
    long long blocks = (items + 7) / 8;
    if (blocks > (long long)sm_count * 8) blocks = (long long)sm_count * 8;
    dequant_kernel<VARIANT><<<(unsigned)blocks, 256, 0, st>>>(da);
    FQ_CUDA_OK(cudaGetLastError());
    return FQ_OK;
}

// ------------------------------------------------------------------------------- tcgen05 GEMM over SM pairs
// At thousands of tokens this kernel runs into the power limit, not into the tensor pipe: what counts is energy per product.
// A pair shares the weight tile (each SM loads and holds half of it), which halves the shared-memory writes and L2 reads of
// the weights against 128 x 256 tiles on single SMs.  4096 x 4096, 8192 tokens, both passes:
// 235-267 us with such tiles, 195 us like this.
constexpr int kBM = 128;                 // tokens per CTA (UMMA M = 256 over the pair)
constexpr int kBN = 256;                 // outputs per tile, at most (UMMA N)
constexpr int kBK = 64;                  // K per stage: 64 bf16 = one 128-byte swizzle span
constexpr int kGemmStages = 6;
constexpr int kGemmThreads = 192;        // warp 0: TMA, warp 1: TMEM owner, of the leading CTA also MMA; warps 2..5: epilogue
constexpr int kTmemCols = 512;           // two accumulators of up to kBN columns

struct GemmSmem {
    static constexpr int kABytes = kBM * kBK * 2;                  // 16 KB
    static constexpr int kBBytes = kBN / 2 * kBK * 2;              // 16 KB
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int oBars = kGemmStages * kStageBytes;        // full[S], empty[S], tmem_full[2], tmem_empty[2]
    static constexpr int oTmemPtr = oBars + (2 * kGemmStages + 4) * 8;
    static constexpr int oFlag = oTmemPtr + 8;
    static constexpr int kTotal = oFlag + 8 + 1024;                // + slack for the 1024-byte alignment of the tiles
};
static_assert(GemmSmem::kTotal <= 232448, "GEMM: shared memory over the per-CTA limit");

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The same shared-memory location in the leading CTA of the pair.
__device__ __forceinline__ uint32_t in_leader(uint32_t addr)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrives at `bar` of both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                 __nv_bfloat16* __restrict__ Y, int M, int N, int K, int ldy, int tile_n, int* status)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank(), pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
    const uint32_t bars = g_smem_u32(smem + GemmSmem::oBars);
    // a stage's "full" and an accumulator's "empty" barriers are those of the leading CTA, the others exist in both
    const uint32_t full0 = bars, empty0 = bars + 8 * kGemmStages;
    const uint32_t tfull0 = bars + 16 * kGemmStages, tempty0 = tfull0 + 16;
    volatile uint32_t* tmem_ptr = reinterpret_cast<volatile uint32_t*>(smem + GemmSmem::oTmemPtr);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + GemmSmem::oFlag);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGemmStages; s++) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; b++) {
            mbar_init(tfull0 + 8 * b, 1);
            mbar_init(tempty0 + 8 * b, 8);                              // one arrival per epilogue warp of both CTAs
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {                     // this warp owns the TMEM allocation
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(g_smem_u32(const_cast<uint32_t*>(tmem_ptr))), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();                      // the peer's barriers exist, its TMEM is allocated
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_ptr;
    asm volatile("griddepcontrol.wait;" ::: "memory");                  // w^ is the previous kernel's output

    const int m_blocks = (M + 2 * kBM - 1) / (2 * kBM), n_blocks = (N + tile_n - 1) / tile_n;
    const int n_tiles = m_blocks * n_blocks;
    const int k_steps = K / kBK;

    if (warp == 0) {
        // ================================================================== TMA producer
        if (lane == 0) {
            const uint32_t bytes = 2u * (uint32_t)(GemmSmem::kABytes + tile_n / 2 * kBK * 2);    // of both CTAs
            int stage = 0;
            uint32_t wraps = 0;
            bool ok = true;
            for (int t = pair; t < n_tiles && ok; t += n_pairs) {
                const int mb = t % m_blocks, nb = t / m_blocks;        // m fastest: the w^ tile stays in L2
                for (int ks = 0; ks < k_steps; ks++) {
                    if (wraps > 0 && !g_wait(empty0 + 8 * stage, (wraps - 1u) & 1u, abort_flag)) { ok = false; break; }
                    const uint32_t full = in_leader(full0 + 8 * stage);
                    const uint32_t a_dst = g_smem_u32(smem + stage * GemmSmem::kStageBytes);
                    if (rank == 0) mbar_expect_tx(full0 + 8 * stage, bytes);
                    tma_load_pair(a_dst, &map_x, ks * kBK, mb * (2 * kBM) + rank * kBM, full);
                    tma_load_pair(a_dst + GemmSmem::kABytes, &map_w, ks * kBK, nb * tile_n + rank * (tile_n / 2), full);
                    if (++stage == kGemmStages) { stage = 0; wraps++; }
                }
            }
            if (!ok) { atomicCAS(status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
        }
    } else if (warp == 1) {
        if (rank == 0) {
            // ============================================================== MMA issuer (for both CTAs)
            const uint32_t idesc = umma_idesc_bf16(2 * kBM, tile_n);
            const uint64_t adesc0 = umma_desc_sw128(g_smem_u32(smem)), bdesc0 = umma_desc_sw128(g_smem_u32(smem) + GemmSmem::kABytes);
            int stage = 0;
            uint32_t wraps = 0;
            int local = 0;
            bool ok = true;
            for (int t = pair; t < n_tiles && ok; t += n_pairs, local++) {
                const int buf = local & 1;
                const uint32_t use = (uint32_t)(local >> 1);           // how often this accumulator was used before
                if (use > 0) ok = __all_sync(0xffffffffu, g_wait(tempty0 + 8 * buf, (use - 1u) & 1u, abort_flag));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + (uint32_t)(buf * kBN);
                for (int ks = 0; ks < k_steps; ks++) {
                    ok = __all_sync(0xffffffffu, g_wait(full0 + 8 * stage, wraps & 1u, abort_flag));
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t step = (uint64_t)(stage * (GemmSmem::kStageBytes >> 4));
                    const uint32_t more = ks > 0 ? 1u : 0u;
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; kk++)
                            asm volatile(
                                "{\n\t.reg .pred p;\n\t"
                                "setp.ne.b32 p, %4, 0;\n\t"
                                "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                                ::"r"(d_tmem), "l"(adesc0 + step + (uint64_t)(kk * 2)), "l"(bdesc0 + step + (uint64_t)(kk * 2)), "r"(idesc),
                                  "r"(kk > 0 ? 1u : more) : "memory");
                        commit_pair(empty0 + 8 * stage);               // the stage may be refilled once these MMAs have read it
                    }
                    __syncwarp();
                    if (++stage == kGemmStages) { stage = 0; wraps++; }
                }
                if (!ok) break;
                if (elect_one()) commit_pair(tfull0 + 8 * buf);
                __syncwarp();
            }
            if (!ok && lane == 0) { atomicCAS(status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
        }
    } else {
        // ================================================================== epilogue (warps 2..5)
        const int quarter = warp & 3;                                   // TMEM lanes 32*quarter .. +31 belong to this warp
        int local = 0;
        bool ok = true;
        for (int t = pair; t < n_tiles && ok; t += n_pairs, local++) {
            const int mb = t % m_blocks, nb = t / m_blocks;
            const int buf = local & 1;
            const uint32_t use = (uint32_t)(local >> 1);
            ok = __all_sync(0xffffffffu, g_wait<64>(tfull0 + 8 * buf, use & 1u, abort_flag));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int row = mb * (2 * kBM) + rank * kBM + quarter * 32 + lane;      // token
            const uint32_t taddr0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * kBN);
#pragma unroll 1
            for (int cb = 0; cb < tile_n / 32; cb++) {
                uint32_t v[32];
                asm volatile(
                    "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                    "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                    "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                      "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                      "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(taddr0 + (uint32_t)(cb * 32)) : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                const int col0 = nb * tile_n + cb * 32;
                if (row < M && col0 < N) {
                    __nv_bfloat16* dst = Y + (long long)row * ldy + col0;
                    if (col0 + 32 <= N) {
#pragma unroll
                        for (int q = 0; q < 4; q++) {
                            uint4 o;
                            uint32_t* ow = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
                            for (int e = 0; e < 4; e++) {
                                const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[8 * q + 2 * e]),
                                                                               __uint_as_float(v[8 * q + 2 * e + 1]));
                                ow[e] = *reinterpret_cast<const uint32_t*>(&h);
                            }
                            *reinterpret_cast<uint4*>(dst + 8 * q) = o;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; e++)
                            if (col0 + e < N) dst[e] = __float2bfloat16_rn(__uint_as_float(v[e]));
                    }
                }
            }
            // the accumulator may be overwritten
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(in_leader(tempty0 + 8 * buf)) : "memory");
        }
        if (!ok && lane == 0) { atomicCAS(status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
    }

    // every path ends here.  After a wait that ran out, copies may still be on their way into shared memory: they land within
    // microseconds, the CTAs leave much later.
    __syncthreads();
    if (*abort_flag)
        for (const unsigned long long t0 = g_ns(); g_ns() - t0 < 200000ull;) __nanosleep(1000);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    cluster_sync();                      // nobody reads this CTA's shared memory or arrives at its barriers any more
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols) : "memory");
    }
}

// ------------------------------------------------------------------------------- host side
// Outputs per tile: the width for which the last wave leaves the least idle (the time of a wave goes with the width, plus
// something for a tile's ends); 5120 outputs and 2048 tokens are 160 tiles of 256 on 74 pairs, three waves where 2.2 are
// needed, but 216 tiles of 192, 2.9 waves.
struct PairTiles { int width; long long waves; };
static PairTiles pair_tile_n(int M, int n_out, int pairs)
{
    const long long m_blocks = (M + 2 * kBM - 1) / (2 * kBM);
    PairTiles best{256, -1};
    for (int w = 256; w >= 128; w -= 32) {
        const long long waves = (m_blocks * ((n_out + w - 1) / w) + pairs - 1) / pairs;
        if (best.waves < 0 || waves * (w + 16) < best.waves * (best.width + 16)) best = PairTiles{w, waves};
    }
    return best;
}

// Measured (4096 x 4096, 11008 x 4096 and 4096 x 11008, 16 to 8192 tokens): the conversion takes 0.33 us per million weights, a
// stage of 64 columns 0.4 us at 256 outputs and not much less at fewer, everything else 6 us.
double gemm_two_pass_us(const Ctx* ctx, int M, int n_out, int k_in)
{
    const PairTiles t = pair_tile_n(M, n_out, ctx->sm_count / 2);
    return 6.0 + 0.33e-6 * (double)n_out * (double)k_in + (double)t.waves * (k_in / kBK) * (0.2 + 0.2 * (t.width + 16) / 272.0);
}

int launch_gemm(Ctx* ctx, const void* store, int blob_stride, const FieldList& fl, int zero_adjust, int n_out, int k_in,
                const uint16_t* X, int M, int ldx, uint16_t* Y, int ldy, void* w_scratch, cudaStream_t st)
{
    // 1. w^ as bf16 [n_out][k_in]
    DequantArgs da{};
    da.store = static_cast<const uint8_t*>(store); da.n_out = n_out; da.k_in = k_in;
    da.n_kb = k_blobs(k_in); da.blob_stride = blob_stride; da.zero_adjust = zero_adjust;
    da.out = static_cast<__nv_bfloat16*>(w_scratch);
    int rc = FQ_ERR_ARG;
    switch (variant_of_fields(fl)) {
#define FQ_CASE(V) case V: rc = launch_dequant<V>(da, ctx->sm_count, st); break;
        FQ_CASE(0) FQ_CASE(1) FQ_CASE(2) FQ_CASE(3) FQ_CASE(4) FQ_CASE(5) FQ_CASE(6)
        FQ_CASE(7) FQ_CASE(8) FQ_CASE(9) FQ_CASE(10) FQ_CASE(11) FQ_CASE(12) FQ_CASE(13)
#undef FQ_CASE
        default: break;
    }
    if (rc != FQ_OK) return rc;

    // 2. tcgen05 GEMM
    static int pairs_on[64] = {};                        // pairs of SMs that can be resident together
    if (ctx->device >= 64) return FQ_ERR_ARG;
    if (!pairs_on[ctx->device]) {
        FQ_CUDA_OK(cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GemmSmem::kTotal));
        cudaLaunchConfig_t probe{};
        probe.gridDim = dim3((unsigned)(ctx->sm_count / 2 * 2)); probe.blockDim = dim3(kGemmThreads);
        probe.dynamicSmemBytes = GemmSmem::kTotal;
        int n = 0;
        FQ_CUDA_OK(cudaOccupancyMaxActiveClusters(&n, gemm_pair_kernel, &probe));
        if (n < 1) return FQ_ERR_CUDA;
        pairs_on[ctx->device] = n < ctx->sm_count / 2 ? n : ctx->sm_count / 2;
    }
    const int pairs = pairs_on[ctx->device];
    const int tile_n = pair_tile_n(M, n_out, pairs).width;
    const int m_blocks = (M + 2 * kBM - 1) / (2 * kBM);
    CUtensorMap map_x, map_w;
    rc = make_map(&map_x, X, M, k_in, ldx, kBM);
    if (rc != FQ_OK) return rc;
    rc = make_map(&map_w, w_scratch, n_out, k_in, k_in, tile_n / 2);
    if (rc != FQ_OK) return rc;
    const long long tiles = (long long)m_blocks * ((n_out + tile_n - 1) / tile_n);
    if (tiles > 0x3fffffffll) return FQ_ERR_SHAPE;
    const int grid = 2 * (int)(tiles < pairs ? tiles : pairs);
    cudaLaunchAttribute overlap{};                       // set up while the dequantisation pass drains
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kGemmThreads); cfg.dynamicSmemBytes = GemmSmem::kTotal;
    cfg.stream = st; cfg.attrs = &overlap; cfg.numAttrs = 1;
    FQ_CUDA_OK(cudaLaunchKernelEx(&cfg, gemm_pair_kernel, map_x, map_w, reinterpret_cast<__nv_bfloat16*>(Y), M, n_out, k_in, ldy, tile_n,
                                  ctx->status_dev));
    return FQ_OK;
}

}  // namespace fq
