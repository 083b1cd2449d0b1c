// Prefill path, fused:  Y[m][n] = sum_k X[m][k] * w^[n][k]  straight from the stored blobs.
//
// The WEIGHTS are the left operand: a tile is 128 outputs (TMEM lanes) x up to 160 tokens (TMEM columns), so that the tensor
// work follows the token count in steps of 16, and the converted weights go from registers straight into TMEM (tcgen05.st),
// from where the MMA reads its left operand: they never pass through shared memory.
//   warp 0        lane 0: TMA, two tile_n x 64 bf16 tiles of X per stage (128-byte swizzle)
//   warp 1        one lane issues tcgen05.mma (M = 128, N = tile_n, K = 16; A in TMEM, B in shared memory)
//   warps 2..5    first ask for the blobs of this CTA's first work items to be brought into the L2; then the epilogue: TMEM ->
//                 bf16 -> global, or partial sums -> workspace
//   warps 6..21   dequantisation, four groups of four that take the stages in turn; warp w owns the 32 output rows (one stored
//                 row pair) that are TMEM lanes 32 (w & 3) .. + 31.  The stored words of a stage are loaded as the decode
//                 kernel reads them; a lane then holds the runs of four columns 16 q + 4c .. + 3 of rows g and g + 8, which
//                 is the register layout of tcgen05.st.16x256b with two bf16 columns to a 32-bit TMEM column.
//
// Work.  (tile, K stage) pairs, tile-major, are cut into gridDim.x equal contiguous runs, one per CTA, so that a matrix with
// few tiles keeps every SM busy.  Each of the CTAs that share a tile leaves its fp32 sums in a workspace slot and counts itself;
// the last one to do so adds the slots up, in K order, and writes the tile: nobody waits for a CTA that may not be running
// yet, and the counter is back at zero for the next launch.  A CTA shares at most the first and the last tile of its run.
// Without a workspace, and where sharing would not pay, the tiles stay whole.
// Every wait is bounded by a timer; when one runs out the kernel records FQ_ERR_TIMEOUT, all roles leave their loops, and the
// TMEM allocation is released before the CTA exits.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "fq_dequant.cuh"
#include "fq_internal.cuh"
#include "fq_ptx.cuh"
#include "fq_umma.cuh"

namespace fq {

#define FQ_CUDA_OK(expr) do { if ((expr) != cudaSuccess) return FQ_ERR_CUDA; } while (0)

namespace {

constexpr int kRows = 128;               // outputs per tile (UMMA M)
constexpr int kTokens = 160;             // tokens per tile, at most (UMMA N): four stages of X and a tile of Y in shared memory, four
                                         // stages of weights beside the accumulator in TMEM
constexpr int kK = kGroup;               // K per stage: a group of 128 columns.  One pass of the issuing warp's loop (wait, issue,
                                         // commit) costs about 300 cycles whether it issues four MMAs or eight
constexpr int kStages = 4;
constexpr int kDqWarps = kRows / 32;     // one per stored row pair of the tile ...
constexpr int kDqGroups = 4;             // ... in each of four groups
constexpr int kThreads = (6 + kDqGroups * kDqWarps) * 32;
constexpr int kTmemCols = 512;
constexpr int kTmemA = 256;              // columns 0 .. 255: accumulator, then kStages x 64 columns of weights
constexpr int kMinRun = 2;               // stages per CTA, at least: a run has fixed costs of about that much
static_assert(kTokens <= kTmemA && kTmemA + kStages * (kK / 2) <= kTmemCols, "TMEM columns");

struct SplitSmem {
    static constexpr int kHalfBytes = kTokens * kUmmaBK * 2;       // 64 columns: one 128-byte swizzle span a token
    static constexpr int kStageBytes = 2 * kHalfBytes;             // 40 KB
    static constexpr int kOutRow = kRows * 2 + 16;                 // a token's outputs (bf16), and room that spreads tokens over the banks
    static constexpr int oOut = kStages * kStageBytes;
    static constexpr int oBars = oOut + kTokens * kOutRow;         // full[S], empty[S], tmem_full, tmem_empty
    static constexpr int oTmemPtr = oBars + (2 * kStages + 3) * 8; // (and sums_due)
    static constexpr int oFlag = oTmemPtr + 8;
    static constexpr int oDue = oFlag + 8;                         // int[2]: this CTA completes its first / last tile; int[2]: warps done
    static constexpr int kTotal = oDue + 16 + 1024;                // + slack for the 1024-byte alignment of the tiles
};
static_assert(SplitSmem::kTotal <= 232448, "prefill: shared memory over the per-CTA limit");

struct SplitArgs {
    const uint8_t* store;
    int n_kb, blob_stride, blob_read, zero_adjust;
    int M, N, K, ldy;
    int tile_n, m_blocks, n_tiles;
    unsigned run_base, run_extra;    // (tile, K stage) pairs of a CTA
    __nv_bfloat16* Y;
    int* status;
    float* parts;            // two slots of kRows x tile_n fp32 per CTA, or null: tiles stay whole
    unsigned* arrived;       // [CTA]: sharers that have left their sums of the tile whose first sharer the CTA is
};

// [tile][ks0, ks1) pieces of one CTA's run.
struct Item { int tile, ks0, ks1; };
struct Run {
    unsigned u, u_hi, k_steps;
    int n_tiles, next_tile;
    unsigned base, extra;                // run length, and how many runs are one longer
    bool split;
    __device__ Run(const SplitArgs& a)
        : k_steps((unsigned)a.K / kK), n_tiles(a.n_tiles), next_tile(blockIdx.x), base(a.run_base), extra(a.run_extra), split(a.parts != nullptr)
    {
        u = lo(blockIdx.x);
        u_hi = lo(blockIdx.x + 1);
    }
    __device__ unsigned lo(unsigned cta) const { return cta * base + min(cta, extra); }
    // the CTA whose run holds pair v
    __device__ int owner(unsigned v) const
    {
        const unsigned longer = extra * (base + 1);
        return (int)(v < longer ? v / (base + 1) : extra + (v - longer) / base);
    }
    __device__ bool next(Item& it)
    {
        if (!split) {
            if (next_tile >= n_tiles) return false;
            it.tile = next_tile; it.ks0 = 0; it.ks1 = (int)k_steps;
            next_tile += gridDim.x;
            return true;
        }
        if (u >= u_hi) return false;
        it.tile = (int)(u / k_steps);
        it.ks0 = (int)(u - (unsigned)it.tile * k_steps);
        it.ks1 = (int)min(k_steps, (unsigned)it.ks0 + (u_hi - u));
        u += (unsigned)(it.ks1 - it.ks0);
        return true;
    }
    __device__ bool whole(const Item& it) const { return it.ks0 == 0 && it.ks1 == (int)k_steps; }
};

// 16 TMEM lanes x 32 columns from this warp's registers: chunk q of eight columns is v[4 q .. 4 q + 3]; lane 4g + c of the warp
// holds columns 2c, 2c + 1 of TMEM lane g in the first two and of lane g + 8 in the last two.
__device__ __forceinline__ void tmem_st_16x256b_x4(uint32_t addr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_ld_x16(uint32_t addr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(addr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// D (+)= A * B, A in TMEM.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}

// Two tokens of this lane's output: lanes 2i and 2i + 1 swap, so that each stores both outputs of one token in one word.
//   y : row of the first token        n : this lane's output
__device__ __forceinline__ void store_pair(__nv_bfloat16* y, int ldy, int n, int N, float v0, float v1, bool has0, bool has1, int lane)
{
    const bool upper = lane & 1;
    const float other = __shfl_xor_sync(0xffffffffu, upper ? v0 : v1, 1);
    const __nv_bfloat162 o = upper ? __floats2bfloat162_rn(other, v1) : __floats2bfloat162_rn(v0, other);
    if (!(upper ? has1 : has0)) return;
    __nv_bfloat16* dst = y + (upper ? (long long)ldy : 0ll) + (n & ~1);
    if ((n | 1) < N) *reinterpret_cast<__nv_bfloat162*>(dst) = o;
    else if ((n & ~1) < N) *dst = o.x;
}

// The CTAs c0 .. c1 that share the tile of a piece, and the slot of the first one: its first if its run begins in this tile,
// else its second (the others' runs begin in the tile).
struct Sharers {
    int c0, c1, slot0;
    __device__ Sharers(const Run& run, int tile)
    {
        const unsigned first = (unsigned)tile * run.k_steps;
        c0 = run.owner(first);
        c1 = run.owner(first + run.k_steps - 1);
        slot0 = c0 * 2 + (run.lo(c0) < first ? 1 : 0);
    }
};

// Adds up and writes the shared tiles that this CTA was the last to contribute to.  Run by all warps that are done with their
// own work, in kSumSets sets of four (one per TMEM quarter): the slots come from the L2, so as many loads as possible
// have to be on their way at once.
//   set : this warp takes the float4 numbers congruent to it
constexpr int kSumSets = 1 + kDqGroups;
__device__ __forceinline__ void add_shared_tiles(const SplitArgs& a, const volatile int* due, int quarter, int set, int lane)
{
    const int trow = quarter * 32 + lane;                                // output of the tile
    Run run(a);
    Item it;
    for (int local = 0; run.next(it); local++) {
        if (run.whole(it) || !due[local > 0]) continue;
        const int mb = it.tile % a.m_blocks, n = it.tile / a.m_blocks * kRows + trow;
        const int tokens = min(a.tile_n, a.M - mb * a.tile_n), quads = (tokens + 3) / 4;
        const Sharers sh(run, it.tile);
        const int others = sh.c1 - sh.c0, slot = kRows * a.tile_n / 4;
        const float4* in0 = reinterpret_cast<const float4*>(a.parts) + (long long)sh.slot0 * slot + trow;
        const float4* in1 = reinterpret_cast<const float4*>(a.parts) + (long long)(sh.c0 + 1) * 2 * slot + trow;
        __nv_bfloat16* y = a.Y + (long long)mb * a.tile_n * a.ldy;
        for (int qa = set; qa < quads; qa += 2 * kSumSets) {             // two at a time: ten loads on their way with four others
            const int qb = qa + kSumSets < quads ? qa + kSumSets : qa;
            float4 sa = __ldcg(in0 + qa * kRows), sb = __ldcg(in0 + qb * kRows);
            for (int i0 = 0; i0 < others; i0 += 4) {
                float4 pa[4], pb[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    pa[i] = pb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i0 + i < others) {
                        const float4* in = in1 + (long long)(i0 + i) * 2 * slot;
                        pa[i] = __ldcg(in + qa * kRows);
                        pb[i] = __ldcg(in + qb * kRows);
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    sa.x += pa[i].x; sa.y += pa[i].y; sa.z += pa[i].z; sa.w += pa[i].w;
                    sb.x += pb[i].x; sb.y += pb[i].y; sb.z += pb[i].z; sb.w += pb[i].w;
                }
            }
            const int ta = 4 * qa, tb = 4 * qb;
            store_pair(y + (long long)ta * a.ldy, a.ldy, n, a.N, sa.x, sa.y, ta < tokens, ta + 1 < tokens, lane);
            store_pair(y + (long long)(ta + 2) * a.ldy, a.ldy, n, a.N, sa.z, sa.w, ta + 2 < tokens, ta + 3 < tokens, lane);
            if (qb == qa) break;
            store_pair(y + (long long)tb * a.ldy, a.ldy, n, a.N, sb.x, sb.y, tb < tokens, tb + 1 < tokens, lane);
            store_pair(y + (long long)(tb + 2) * a.ldy, a.ldy, n, a.N, sb.z, sb.w, tb + 2 < tokens, tb + 3 < tokens, lane);
        }
    }
}

template <int VARIANT>
__global__ void __launch_bounds__(kThreads, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap map_x, const SplitArgs a)
{
    constexpr FieldList FL = variant_fields(VARIANT);
    constexpr int kLoads = group_loads(FL, FL.n);
    constexpr bool kHalved = VARIANT >= 7 && VARIANT < 13;         // a nested child of 2..7 bits: half its codes are below 128
    constexpr bool kSmallCodes = VARIANT < 6 || kHalved;           // PACKED 2..7 bits: codes below 128, no zero adjustment
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bars = g_smem_u32(smem + SplitSmem::oBars);
    const uint32_t full0 = bars, empty0 = bars + 8 * kStages;
    const uint32_t tfull = bars + 16 * kStages, tempty = tfull + 8, sums_due = tfull + 16;
    volatile uint32_t* tmem_ptr = reinterpret_cast<volatile uint32_t*>(smem + SplitSmem::oTmemPtr);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + SplitSmem::oFlag);
    volatile int* due = reinterpret_cast<volatile int*>(smem + SplitSmem::oDue);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; s++) {
            mbar_init(full0 + 8 * s, 1 + kDqWarps);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tempty, 4);                                            // one arrival per epilogue warp
        mbar_init(sums_due, 4);
        *abort_flag = 0;
        due[0] = due[1] = due[2] = due[3] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {                     // this warp owns the TMEM allocation
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(g_smem_u32(const_cast<uint32_t*>(tmem_ptr))), "n"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const int n_rp = row_pairs(a.N);
    if (warp >= 2 && warp < 6) {
        // the blobs of the first two items: all of them on their way from HBM at once, while the pipeline starts (one warp per
        // stored row pair)
        Run run(a);
        Item it;
        for (int n = 0; n < 2 && run.next(it); n++) {
            const int rp = it.tile / a.m_blocks * kDqWarps + warp - 2, kb1 = (it.ks1 + 3) >> 2;
            for (int kb = (it.ks0 >> 2) + lane; kb < kb1; kb += 32)
                if (rp < n_rp && FQ_IN_BOUNDS(kb < a.n_kb, a.status))
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                                 ::"l"(a.store + ((long long)rp * a.n_kb + kb) * a.blob_stride), "r"(a.blob_read) : "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_ptr;
    // Everything above may run while the previous kernel of the stream finishes, and so may the dequantisation of the first four
    // stages: whatever wrote the stored blobs has come before an earlier launch of this kernel, or this launch does not overlap at all
    // (launch_gemm_split), so that weights are in TMEM when X may be read.  X, Y and the workspace may be the previous kernel's: the other
    // warps wait here, the dequantisation warps after their first stage.  A call, us, all warps waiting here -> these not:
    // 4096 x 4096 at 77 tokens 16.2 -> 15.0, at 160 20.3 -> 18.9; 11008 x 4096 at 77 18.7 -> 17.7, at 300 36.6 -> 35.1.
    if (warp < 6) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    if (warp == 0) {
        // ================================================================== TMA producer (X)
        if (lane == 0) {
            int stage = 0;
            uint32_t wraps = 0;
            bool ok = true;
            Run run(a);
            Item it;
            while (ok && run.next(it)) {
                const int mb = it.tile % a.m_blocks;                       // m fastest: the blobs of a row block stay in L2
                for (int ks = it.ks0; ks < it.ks1; ks++) {
                    if (wraps > 0 && !g_wait(empty0 + 8 * stage, (wraps - 1u) & 1u, abort_flag)) { ok = false; break; }
                    const uint32_t full = full0 + 8 * stage;
                    mbar_expect_tx(full, (uint32_t)a.tile_n * kK * 2);
#pragma unroll
                    for (int h = 0; h < 2; h++)
                        asm volatile(
                            "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                            ::"r"(g_smem_u32(smem + stage * SplitSmem::kStageBytes + h * SplitSmem::kHalfBytes)), "l"(&map_x),
                              "r"(ks * kK + h * kUmmaBK), "r"(mb * a.tile_n), "r"(full) : "memory");
                    if (++stage == kStages) { stage = 0; wraps++; }
                }
            }
            if (!ok) { atomicCAS(a.status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
        }
    } else if (warp == 1) {
        // ================================================================== MMA issuer
        const uint32_t idesc = umma_idesc_bf16(kRows, a.tile_n);
        const uint64_t bdesc0 = umma_desc_sw128(g_smem_u32(smem));
        int stage = 0;
        uint32_t wraps = 0;
        int local = 0;
        bool ok = true;
        Run run(a);
        Item it;
        for (; ok && run.next(it); local++) {
            // the accumulator belongs to this item: wait until the epilogue has drained the previous one
            if (local > 0) ok = __all_sync(0xffffffffu, g_wait(tempty, (uint32_t)(local - 1) & 1u, abort_flag));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int ks = it.ks0; ks < it.ks1; ks++) {
                ok = __all_sync(0xffffffffu, g_wait(full0 + 8 * stage, wraps & 1u, abort_flag));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t bdesc = bdesc0 + (uint64_t)(stage * (SplitSmem::kStageBytes >> 4));
                const uint32_t a_tmem = tmem_base + (uint32_t)(kTmemA + stage * (kK / 2));
                const bool more = ks > it.ks0;
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kK / 16; kk++)
                        umma_ts(tmem_base, a_tmem + kk * 8, bdesc + (uint64_t)((kk >> 2) * (SplitSmem::kHalfBytes >> 4) + (kk & 3) * 2), idesc,
                                kk > 0 || more);
                    umma_commit(empty0 + 8 * stage);                       // the stage may be refilled once these MMAs have read it
                }
                __syncwarp();
                if (++stage == kStages) { stage = 0; wraps++; }
            }
            if (!ok) break;
            if (elect_one()) umma_commit(tfull);
            __syncwarp();
        }
        if (!ok && lane == 0) { atomicCAS(a.status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
    } else if (warp < 6) {
        // ================================================================== epilogue (warps 2..5)
        const int quarter = warp & 3;                                   // TMEM lanes 32*quarter .. +31 belong to this warp
        const int trow = quarter * 32 + lane;                           // output of the tile
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
        int local = 0;
        bool ok = true;
        Run run(a);
        Item it;
        for (; ok && run.next(it); local++) {
            const int mb = it.tile % a.m_blocks;
            const int tokens = min(a.tile_n, a.M - mb * a.tile_n);      // of the tile
            ok = __all_sync(0xffffffffu, g_wait<128>(tfull, (uint32_t)local & 1u, abort_flag));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (run.whole(it)) {
                // through shared memory: the accumulator is free for the next tile as soon as it has been read, and the stores to
                // Y are 16 bytes a lane (straight from TMEM a lane has one output of every token: 9000 cycles for 160 tokens)
                uint8_t* mine = smem + SplitSmem::oOut + trow * 2;
#pragma unroll 1
                for (int t0 = 0; t0 < tokens; t0 += 16) {
                    uint32_t v[16];
                    tmem_ld_x16(taddr + (uint32_t)t0, v);
#pragma unroll
                    for (int e = 0; e < 16; e++)
                        *reinterpret_cast<__nv_bfloat16*>(mine + (t0 + e) * SplitSmem::kOutRow) = __float2bfloat16_rn(__uint_as_float(v[e]));
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty);                     // the accumulator may be overwritten
                // this warp's 32 outputs of every token: 64 bytes, four lanes; eight tokens at a time
                const int n4 = it.tile / a.m_blocks * kRows + quarter * 32 + (lane & 3) * 8;
                __nv_bfloat16* y = a.Y + (long long)mb * a.tile_n * a.ldy + n4;
                const uint8_t* from = smem + SplitSmem::oOut + (quarter * 32 + (lane & 3) * 8) * 2;
#pragma unroll 2
                for (int t = lane >> 2; t < tokens; t += 8) {
                    const uint4 o = *reinterpret_cast<const uint4*>(from + t * SplitSmem::kOutRow);
                    __nv_bfloat16* dst = y + (long long)t * a.ldy;
                    if (n4 + 8 <= a.N) {
                        *reinterpret_cast<uint4*>(dst) = o;
                    } else {
                        const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&o);
#pragma unroll
                        for (int e = 0; e < 8; e++)
                            if (n4 + e < a.N) dst[e] = h[e];
                    }
                }
                __syncwarp();
                continue;
            } else {
                // partial sums: float4 number q (tokens 4q .. 4q + 3) of the slot is [q][output of the tile]
                const int slot = blockIdx.x * 2 + (local > 0 ? 1 : 0);
                float4* out = reinterpret_cast<float4*>(a.parts) + (long long)slot * (kRows * a.tile_n / 4) + trow;
#pragma unroll 1
                for (int t0 = 0; t0 < tokens; t0 += 16) {
                    uint32_t v[16];
                    tmem_ld_x16(taddr + (uint32_t)t0, v);
#pragma unroll
                    for (int e = 0; e < 4; e++)
                        out[(t0 / 4 + e) * kRows] = make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]),
                                                                __uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3]));
                }
                fence_gpu();
                __syncwarp();
                if (lane == 0 && atomicAdd(const_cast<int*>(&due[2 + (local > 0)]), 1) == 3) {    // the fourth epilogue warp
                    fence_cta();                                        // (the other three warps' sums, too)
                    const Sharers sh(run, it.tile);
                    if (atom_add_acq_rel(a.arrived + sh.c0, 1u) == (unsigned)(sh.c1 - sh.c0)) {
                        a.arrived[sh.c0] = 0u;
                        due[local > 0] = 1;
                    }
                }
            }
            // the accumulator may be overwritten
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty);
        }
        if (a.parts) {
            if (lane == 0) mbar_arrive(sums_due);
            if (ok) ok = __all_sync(0xffffffffu, g_wait(sums_due, 0u, abort_flag));
            if (ok) add_shared_tiles(a, due, quarter, 0, lane);
        }
        if (!ok && lane == 0) { atomicCAS(a.status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
    } else {
        // ================================================================== dequantisation (warps 6..21)
        const int dw = warp & 3;                                        // row pair of the tile = TMEM quarter of this warp
        const int grp_id = (warp - 6) / kDqWarps;                       // this group takes the stages seq % kDqGroups == grp_id
        const int g = lane >> 2;
        const uint32_t ta = tmem_base + ((uint32_t)(dw * 32) << 16) + (uint32_t)kTmemA;
        int seq = 0;                                                    // stages of this CTA so far, over all its items
        static_assert(kDqGroups == kStages, "a group always fills the same stage");
        const int stage = grp_id;
        uint32_t wraps = 0;
        bool ok = true;
        Run run(a);
        Item it;
        while (ok && run.next(it)) {
            const int rp = it.tile / a.m_blocks * kDqWarps + dw;
            const bool have = rp < n_rp;
            const uint8_t* row_blobs = a.store + (long long)(have ? rp : 0) * a.n_kb * a.blob_stride;
            const int skip = (grp_id - seq % kDqGroups + kDqGroups) % kDqGroups;      // to this group's first stage of the item
            seq += it.ks1 - it.ks0;
            for (int ks = it.ks0 + skip; ks < it.ks1; ks += kDqGroups, wraps++) {
                // ---- the stored words of this stage: one group of one superstep of one blob
                const int kb = ks >> 2, ssl = (ks >> 1) & 1, grp = ks & 1;
                const uint8_t* blob = row_blobs + (long long)kb * a.blob_stride;
                if (!FQ_IN_BOUNDS(kb < a.n_kb && (have ? rp : 0) < n_rp, a.status)) {                      // (checked build)
                    if (lane == 0) *abort_flag = 1;
                    ok = false;
                    break;
                }
                uint4 raw[kBlobTiles][kLoads];
                uint2 meta[kBlobTiles];                                    // scale / zero words of rows g and g + 8: adjacent
                load_group_words<VARIANT, 0>(blob + lane * 16, ssl, grp, raw[0]);
                load_group_words<VARIANT, 1>(blob + lane * 16, ssl, grp, raw[1]);
#pragma unroll
                for (int tl = 0; tl < kBlobTiles; tl++)
                    meta[tl] = __ldg(reinterpret_cast<const uint2*>(blob + blob_meta_off(ssl, tl) + blob_meta_word(grp, g)));
                // ---- the stage's columns of TMEM must be free (the MMAs that read their previous contents are done).  The MMAs begin
                // when the previous kernel has ended, however long that takes: only then does a wait for them have a limit
                if (wraps == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
                const bool is_free = wraps == 0 || g_wait(empty0 + 8 * stage, (wraps - 1u) & 1u, abort_flag);
                if (!__all_sync(0xffffffffu, is_free)) { ok = false; break; }      // (the lanes must leave together)
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int tl = 0; tl < kBlobTiles; tl++) {
                    align_group_words<VARIANT>(raw[tl], grp);
                    const uint32_t mm[2] = {meta[tl].x, meta[tl].y};
                    float sc[2], cc[2];
#pragma unroll
                    for (int hr = 0; hr < 2; hr++) {
                        sc[hr] = have ? __half2float(__ushort_as_half((unsigned short)(mm[hr] & 0xffffu))) : 0.f;   // rows past N: zeros
                        cc[hr] = -(float)((kHalved ? 256 - a.zero_adjust : 128) + (int)(mm[hr] >> 16)) * sc[hr];
                        if (kHalved) sc[hr] *= 2.f;
                    }
                    const WideZero zz[2] = {{mm[0], a.zero_adjust, sc[0]}, {mm[1], a.zero_adjust, sc[1]}};
                    unrolled<0, 2>([&](auto H) {                               // 64 columns at a time
                        constexpr int h = decltype(H)::value;
                        uint32_t w[16];
                        unrolled<0, 2>([&](auto JJ) {
                            constexpr int jj = decltype(JJ)::value;
                            uint32_t code[4];
                            merge_group_codes<VARIANT, 2 * h + jj, kHalved ? 1 : 0>(raw[tl], code);
#pragma unroll
                            for (int r = 0; r < 4; r++) {
                                const int hr = r & 1, half = r >> 1;           // A register r = 2 * half + row half
                                const uint2 o = kSmallCodes ? small_codes_to_bf16(code[r], cc[hr], sc[hr]) : codes_to_bf16(code[r], zz[hr], sc[hr]);
                                w[4 * (2 * jj + half) + 2 * hr] = o.x;
                                w[4 * (2 * jj + half) + 2 * hr + 1] = o.y;
                            }
                        });
                        tmem_st_16x256b_x4(ta + ((uint32_t)(tl * 16) << 16) + (uint32_t)(stage * (kK / 2) + h * 32), w);
                    });
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8 * stage);
            }
        }
        if (wraps <= 1) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (a.parts) {
            if (ok) ok = __all_sync(0xffffffffu, g_wait<64>(sums_due, 0u, abort_flag));
            if (ok) add_shared_tiles(a, due, dw, 1 + grp_id, lane);
        }
        if (!ok && lane == 0) { atomicCAS(a.status, 0, FQ_ERR_TIMEOUT); *abort_flag = 1; }
    }

    // every path ends here: release TMEM before the CTA exits.  After a wait that ran out, copies may still be on their way into
    // shared memory: they land within microseconds, the CTA leaves much later.
    __syncthreads();
    if (*abort_flag)
        for (const unsigned long long t0 = g_ns(); g_ns() - t0 < 200000ull;) __nanosleep(1000);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(kTmemCols) : "memory");
    }
}

//   overlap : start while the previous kernel of the stream drains
template <int VARIANT>
int launch_variant(Ctx* ctx, const CUtensorMap& map_x, const SplitArgs& a, int grid, bool overlap, cudaStream_t st)
{
    static bool configured[64] = {};
    if (ctx->device < 64 && !configured[ctx->device]) {
        FQ_CUDA_OK(cudaFuncSetAttribute(gemm_split_kernel<VARIANT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SplitSmem::kTotal));
        configured[ctx->device] = true;
    }
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = SplitSmem::kTotal;
    cfg.stream = st; cfg.attrs = &early; cfg.numAttrs = overlap ? 1u : 0u;
    FQ_CUDA_OK(cudaLaunchKernelEx(&cfg, gemm_split_kernel<VARIANT>, map_x, a));
    return FQ_OK;
}

// Tokens per tile: as many equal tiles of at most kTokens as the token count needs, in steps of 16.
int split_tile_n(int M)
{
    const int tiles = (M + kTokens - 1) / kTokens;
    return (int)round_up((M + tiles - 1) / tiles, 16);
}

// Sharing tiles evens the CTAs out and costs an exchange of partial sums through the L2.  Measured (4096 x 4096, 11008 x 4096 and
// 4096 x 11008, 16 to 600 tokens): a stage takes about 0.33 us + 1 ns a token, the exchange 4.5 us + 60 ns a token, everything
// else 5 us.
struct Plan {
    long long tiles, pairs, runs;        // pairs: (tile, K stage); runs: CTAs when tiles are shared
    bool share;
    double us;                           // estimate of the kernel's time
    Plan(int sm_count, int M, int n_out, int k_in)
    {
        const int tile_n = split_tile_n(M), k_steps = k_in / kK;
        tiles = (long long)((M + tile_n - 1) / tile_n) * ((n_out + kRows - 1) / kRows);
        pairs = tiles * k_steps;
        const long long grid = tiles < sm_count ? tiles : sm_count;
        runs = pairs / kMinRun < sm_count ? pairs / kMinRun : sm_count;
        if (runs < grid) runs = grid;
        const double stage_us = 0.33 + 0.001 * tile_n, exchange_us = 4.5 + 0.06 * tile_n;
        const double whole = (double)((tiles + grid - 1) / grid * k_steps) * stage_us;
        const double shared = (double)((pairs + runs - 1) / runs) * stage_us + exchange_us;
        share = pairs < (1ll << 31) && shared < whole;
        us = 5.0 + (share ? shared : whole);
    }
};

}  // namespace

// Long prompts run into the power limit, and converting the weights once per token tile costs energy: chosen by the estimate of
// a cool chip alone, one 7B block at 8192 tokens took 3338 us in this kernel and 2692 us in the two-pass way, a 13B block at
// 2048 tokens 1334 and 1187 us.
double gemm_split_us(const Ctx* ctx, int M, int n_out, int k_in)
{
    return Plan(ctx->sm_count, M, n_out, k_in).us * (1.0 + 0.3 * (M < 2048 ? M : 2048) / 2048.0);
}

void gemm_split_plan(const Ctx* ctx, int M, int n_out, int k_in, fq_gemm_plan_report* out)
{
    const Plan plan(ctx->sm_count, M, n_out, k_in);
    out->shared = ctx->fused_ws && plan.share;
    out->tile_tokens = split_tile_n(M);
    out->tiles = plan.tiles;
    out->blocks = (int)(out->shared ? plan.runs : (plan.tiles < ctx->sm_count ? plan.tiles : ctx->sm_count));
}

size_t gemm_split_flag_bytes(int sm_count) { return (size_t)round_up((int64_t)sm_count * sizeof(unsigned), 256); }
size_t gemm_split_part_bytes(int sm_count) { return (size_t)sm_count * 2 * kRows * kTokens * sizeof(float); }

int launch_gemm_split(Ctx* ctx, const void* store, int blob_stride, int blob_read, const FieldList& fl, int zero_adjust, int n_out,
                      int k_in, const uint16_t* X, int M, int ldx, uint16_t* Y, int ldy, float* parts, unsigned* arrived,
                      cudaStream_t st)
{
    const int variant = variant_of_fields(fl);          // the kernel is specialised per field list
    if (variant < 0) return FQ_ERR_ARG;
    SplitArgs a{};
    a.store = static_cast<const uint8_t*>(store); a.n_kb = k_blobs(k_in); a.blob_stride = blob_stride; a.blob_read = blob_read;
    a.zero_adjust = zero_adjust; a.M = M; a.N = n_out; a.K = k_in; a.ldy = ldy;
    a.Y = reinterpret_cast<__nv_bfloat16*>(Y); a.status = ctx->status_dev;
    a.tile_n = split_tile_n(M);
    a.m_blocks = (M + a.tile_n - 1) / a.tile_n;
    CUtensorMap map_x;
    const int rc = make_map(&map_x, X, M, k_in, ldx, a.tile_n);                 // box: tile_n tokens x 64 columns
    if (rc != FQ_OK) return rc;
    const Plan plan(ctx->sm_count, M, n_out, k_in);
    if (plan.tiles > 0x7fffffffll) return FQ_ERR_SHAPE;
    a.n_tiles = (int)plan.tiles;
    long long grid = plan.tiles < ctx->sm_count ? plan.tiles : ctx->sm_count;
    if (parts && plan.share) {
        grid = plan.runs;
        a.parts = parts; a.arrived = arrived;
        a.run_base = (unsigned)(plan.pairs / grid); a.run_extra = (unsigned)(plan.pairs % grid);
    }
    // An overlapping launch reads stored weights while the stream's previous kernel may still be running, and where that one wrote
    // them (fq_pack_layer) nothing makes them visible before griddepcontrol.wait.  So the first launch on a stream after anything that
    // stores weights or changes the configuration comes after all of the stream's work, without overlap: what was stored before it is
    // in place for every later launch there.  A launch that is only captured orders nothing, and a captured call that stores weights
    // runs whenever its graph does: contexts with such calls do without overlap.
    const bool overlap = !ctx->stores_in_graphs && ctx->gemm_after_stores_at == ctx->config_epoch && ctx->gemm_after_stores_on == st;
    int launched = FQ_ERR_ARG;
    switch (variant) {
#define FQ_CASE(V) case V: launched = launch_variant<V>(ctx, map_x, a, (int)grid, overlap, st); break;
        FQ_CASE(0) FQ_CASE(1) FQ_CASE(2) FQ_CASE(3) FQ_CASE(4) FQ_CASE(5) FQ_CASE(6)
        FQ_CASE(7) FQ_CASE(8) FQ_CASE(9) FQ_CASE(10) FQ_CASE(11) FQ_CASE(12) FQ_CASE(13)
#undef FQ_CASE
        default: break;
    }
    if (launched == FQ_OK && !overlap && !is_capturing(st)) {
        ctx->gemm_after_stores_at = ctx->config_epoch;
        ctx->gemm_after_stores_on = st;
    }
    return launched;
}

}  // namespace fq
