// Decode path for a batch of 2..8 activation rows: fused dequantize-GEMV over tiled field arrays.
// (Batch 1 has its own kernel in fq_gemv1.cu.)
//
// One persistent CTA per SM with four roles:
//   producer warp   : streams "units" (32 output rows x one K chunk: every field array of the
//                     active variant plus the scale/zero words) from HBM into a shared-memory
//                     ring with bulk asynchronous copies (cp.async.bulk + mbarrier tx counts)
//                     and writes a small descriptor next to each stage;
//   activation warp : once per (op, K chunk) that this CTA touches, waits -- bounded -- for the
//                     previous dependency phase and fetches the activations of that chunk, one bulk copy per batch row;
//   consumer warps  : two or four warps share a unit, one 16-row tile, or a half of its columns, each.  Stored words become fp16 integers q - z, the fp16
//                     activations are the other operand of mma.m16n8k16, sums are fp32 and scaled once per group of 128
//                     columns (fq_batch_core.cuh).  The loops are compiled once per field list (14 variants) and chosen
//                     per unit.  13B nested at 4 bits, four blocks in
//                     dependency order: 4 / 8 entries 333 / 375 us, against 534 / 593 us with one 8-bit integer MMA per field and
//                     digit of fixed-point activations.
//   output warps    : finish row pairs (see below) and are the only warps that write y.
// The K chunks of one row pair are computed by different CTAs.  Each unit publishes its row sums
// as 64-bit words (fp32 value, launch tag) with plain stores; the unit whose chunk index is
// (row pair mod chunks) hands its own sums to an output warp, which polls the other chunks'
// words until they carry this launch's tag and adds them in chunk order, so results do not
// depend on scheduling and no fence or atomic sits on the consumers' path.
//
// A whole stack of layers runs as one launch.  Every op's units are dealt to the CTAs in
// contiguous, K-chunk-major blocks (a CTA needs the activations of one or two chunks only);
// the producer runs ahead across op boundaries because weights do not depend on activations.
// Every wait has a time limit (fq_set_wait_limit_ns); when one runs out the kernel records FQ_ERR_TIMEOUT, stops
// computing, stays until its copies have landed and returns.
#include <cuda_fp16.h>

#include "fq_batch_core.cuh"
#include "fq_internal.cuh"
#include "fq_ptx.cuh"

namespace fq {

#define FQ_CUDA_OK(expr) do { if ((expr) != cudaSuccess) return FQ_ERR_CUDA; } while (0)

constexpr int kConsumerWarps = 20;
constexpr int kProducerWarp = kConsumerWarps;          // warp index of the producer
constexpr int kActWarp = kConsumerWarps + 1;           // the warp that fetches activations
constexpr int kOutputWarp = kActWarp + 1;              // the warps that own every global store of results
constexpr int kOutputWarps = 2;                        // each takes every other place of the output queue
constexpr int kGemvThreads = (kConsumerWarps + 2 + kOutputWarps) * 32;     // 24 warps: 80 registers each
constexpr int kUnitBytes = 17408;                      // bytes of one unit (whole blobs), at most: 2 x 4-bit or 1 x 8-bit blob
constexpr int kBlobsMax = kXCols / 512;                // k blobs (512 columns) per chunk, at most
constexpr int kOutSlots = 16;                          // finished units waiting for an output warp (it scans one slot per lane)
constexpr int kXSlots = 3;                             // activation chunks kept in shared memory (a fourth costs a stage of the ring: 1 % slower)

// What the producer tells the consumers: once per op a copy of the op descriptor in a ring ...
constexpr int kOpRing = 16;                            // > stages + 1: an op slot outlives the start of its last unit
// ... and once per unit (next to the stage that holds the unit's weights)
struct UnitDesc {
    int ch, rp, nb, seg;                        // K chunk, row pair, blobs in the unit, activation segment
    int op_slot;                                // op ring slot
    int oseq;                                   // >= 0: this unit finishes its row pair, and is the oseq-th such unit of the CTA
    int pad[2];
};
static_assert(sizeof(UnitDesc) == 32, "descriptor layout");

// What a consumer hands to the output warp together with the unit's 32 x batch row sums.
struct OutDesc {
    int rp, ch, n_chunks, n_out, phase, batch;
    uint16_t* y;
    const unsigned long long* partial;
    int pad[2];
};
static_assert(sizeof(OutDesc) == 48, "descriptor layout");

template <int BP> struct GemvSmem {
    // Warps that share a unit: one 16-row tile each, and for up to eight entries also one half of the columns each.  Their stage
    // ring is the shorter one (more shared memory goes to activations), so a unit has to leave it sooner: 13B nested at
    // 4 bits, four blocks in dependency order: 399 -> 375 us; up to four entries lose by it (333 -> 362 us).
    static constexpr int kWarpsPerUnit = BP == 8 ? 2 * kUnitRowTiles : kUnitRowTiles;
    static constexpr bool kHalves = kWarpsPerUnit > kUnitRowTiles;
    static constexpr int kUnitsInFlight = kConsumerWarps / kWarpsPerUnit;
    static_assert(kConsumerWarps % kWarpsPerUnit == 0, "consumer warps come in groups of one unit");
    static constexpr int kStageBytes = kUnitBytes;
    static constexpr int kXSlotBytes = BP * kXRowBytes;              // one chunk's activations
    static constexpr int kOpBytes = (int)((sizeof(GemvOp) + 15) / 16 * 16);
    static constexpr int kOutFloats = 32 * BP;                               // row sums of one unit
    static constexpr int kHalfBytes = kHalves ? kUnitsInFlight * 2 * kOutFloats * 4 : 0;    // [unit in flight][half][row][batch entry]
    static constexpr int kOutBytes = kOutSlots * (kOutFloats * 4 + (int)sizeof(OutDesc));
    static constexpr int kFixed = kXSlots * kXSlotBytes + kOpRing * kOpBytes + 4 * kOpBytes +
                                  kOutBytes + kHalfBytes + 640;
    static constexpr int kPerStage = kStageBytes + (int)sizeof(UnitDesc) + 16 + 4;
    static constexpr int kAuto = (232448 - kFixed) / kPerStage;
    static constexpr int kStages = kAuto > 16 ? 16 : kAuto;
    static constexpr int oStages = 0;
    static constexpr int oDesc = oStages + kStages * kStageBytes;
    static constexpr int oX = oDesc + kStages * (int)sizeof(UnitDesc);
    static constexpr int oOpRing = oX + kXSlots * kXSlotBytes;       // GemvOp[kOpRing]
    static constexpr int oOpBuf = oOpRing + kOpRing * kOpBytes;   // GemvOp[2] producer, GemvOp[2] activation warp
    static constexpr int oOutData = oOpBuf + 4 * kOpBytes;   // float[kOutSlots][kOutFloats]
    static constexpr int oOutDesc = oOutData + kOutSlots * kOutFloats * 4;     // OutDesc[kOutSlots]
    static constexpr int oHalf = oOutDesc + kOutSlots * (int)sizeof(OutDesc);   // float[kUnitsInFlight][2][kOutFloats]
    static constexpr int oBars = oHalf + kHalfBytes;  // full[S], empty[S]
    static constexpr int oReleased = oBars + 2 * kStages * 8;        // u32[S]: consumer warps that released a stage, ever
    static constexpr int oCtl = oReleased + kStages * 4;             // x_ready[XS], x_pending[XS], flags[2], prep_cmd, pad
    static constexpr int oOutCtl = oCtl + 64;                        // out_fill[kOutSlots], out_gen[kOutSlots]
    static constexpr int oHalfCtl = oOutCtl + 2 * kOutSlots * 4 + 16;          // u32 [unit in flight][tile]: halves delivered, units done
    static constexpr int oXBars = (oHalfCtl + kUnitsInFlight * kUnitRowTiles * 8 + 7) / 8 * 8;   // (+ out_total) one mbarrier per activation slot
    static constexpr int kTotal = oXBars + 8 * kXSlots + 8;
    static_assert(kStages >= 4, "decode kernel: no room for a ring");
    static_assert(kOpRing >= kStages + 2, "an op's ring slot must outlive the units that refer to it");
    static_assert(kTotal <= 232448, "decode kernel: shared memory over the 227 KB per-CTA limit");
    static_assert(oBars % 8 == 0 && oXBars % 8 == 0, "mbarriers are 8-byte objects");
};

// K blobs (512 columns) per K chunk for a variant of which `bits` bits are read.
int gemv_chunk_blobs(int bits)
{
    int c = kUnitBytes / blob_bytes(bits);
    if (c > kBlobsMax) c = kBlobsMax;
    if (c < 1) c = 1;
    return c;
}
static_assert(kUnitBytes >= kBlobMetaBytes + kBlobSteps * kBlobTiles * 512 * 8, "a unit must hold an 8-bit blob");

// A split-K partial is one 64-bit word per (row, batch entry): fp32 sum in the low half, launch tag in the high half.
size_t gemv_partial_bytes_per_unit(int batch) { return (size_t)(32 * batch_pad(batch)) * sizeof(unsigned long long); }

// ------------------------------------------------------------------------------- per-CTA work split
// (this kernel numbers the units of an op chunk-major, u = ch * n_rp + rp, and deals them with cta_range)
void gemv_cta_range(int n_units, int rot, int cta, int grid, int& lo, int& hi) { cta_range(n_units, rot, cta, grid, lo, hi); }

struct StackArgs {
    const GemvOp* table;                   // device op table (nullptr: use the by-value op)
    const long long* phase_total;          // units per phase
    unsigned long long* phase_done;        // finished units per phase
    unsigned* exit_count;
    const int* cta_units;                  // units of every CTA (nullptr: single op, computed on the device)
    int* status;
    int n_ops, n_phases;
    unsigned epoch;                        // tag of this launch's split-K partials (never 0)
    const unsigned* high_zeros;            // not 0: some stored zero point is above 1023
    unsigned* note;                        // host memory (or null): the first CTA notes there what it found ...
    unsigned stored;                       // ... and as of which state of the context
    unsigned long long wait_ns;            // limit of every wait
};

// A wait ran out: stops every role of the CTA.
__device__ __forceinline__ void give_up(int* status, volatile int* flags)
{
    atomicCAS(status, 0, FQ_ERR_TIMEOUT);
    flags[0] = 1; flags[1] = 1;
}

// Warp-cooperative fetch of op descriptors with one op of look-ahead: the words of op i+1 travel
// while op i is processed.
struct OpFetch {
    uint32_t w0, w1;
    __device__ __forceinline__ void issue(const GemvOp* ops, int oi, int n_ops, int lane)
    {
        w0 = w1 = 0u;
        if (oi < n_ops) {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(ops + oi);
            if (lane < (int)(sizeof(GemvOp) / 4)) w0 = src[lane];
            if (lane + 32 < (int)(sizeof(GemvOp) / 4)) w1 = src[lane + 32];
        }
    }
    __device__ __forceinline__ void store(GemvOp* dst, int lane) const
    {
        uint32_t* d = reinterpret_cast<uint32_t*>(dst);
        if (lane < (int)(sizeof(GemvOp) / 4)) d[lane] = w0;
        if (lane + 32 < (int)(sizeof(GemvOp) / 4)) d[lane + 32] = w1;
    }
};
static_assert(sizeof(GemvOp) <= 256, "op descriptor too large for the two-word fetch");

//   HIGH : zero points above 1023 are possible (see zeros_are_low)
template <int BP, bool HIGH>
__global__ void __launch_bounds__(kGemvThreads, 1)
gemv_kernel(const __grid_constant__ GemvOp single, const StackArgs sa)
{
    using S = GemvSmem<BP>;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bars = smem_u32(smem + S::oBars);                          // full[0..S), empty[0..S)
    volatile unsigned* released = reinterpret_cast<volatile unsigned*>(smem + S::oReleased);
    volatile int* x_ready = reinterpret_cast<volatile int*>(smem + S::oCtl);   // segment number + 1 held by a slot
    const uint32_t xbars = smem_u32(smem + S::oXBars);                         // completes a phase per publication of a slot
    volatile int* x_pending = x_ready + kXSlots;                               // units that still need the slot
    volatile int* flags = x_pending + kXSlots;                                 // [0]: stop computing, [1]: stop everything
    volatile unsigned* out_fill = reinterpret_cast<volatile unsigned*>(smem + S::oOutCtl);   // consumer warps that filled a slot
    volatile unsigned* out_gen = out_fill + kOutSlots;                         // times the output warp drained a slot
    volatile unsigned* half_ctl = reinterpret_cast<volatile unsigned*>(smem + S::oHalfCtl);
    volatile int* out_total = reinterpret_cast<volatile int*>(out_gen + kOutSlots);   // finishing units of this CTA (-1: not known yet)

    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; s++) {
            mbar_init(bars + 8 * s, 1);
            mbar_init(bars + 8 * (S::kStages + s), S::kWarpsPerUnit);
            released[s] = 0u;
        }
        for (int i = 0; i < kXSlots; i++) { x_ready[i] = 0; x_pending[i] = 0; mbar_init(xbars + 8 * i, 1); }
        for (int i = 0; i < kOutSlots; i++) { out_fill[i] = 0u; out_gen[i] = 0u; }
        for (int i = 0; i < S::kUnitsInFlight * kUnitRowTiles * 2; i++) half_ctl[i] = 0u;
        out_total[0] = -1;
        flags[0] = 0; flags[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    const int grid = gridDim.x, cta = blockIdx.x;
    const GemvOp* ops = sa.table ? sa.table : &single;
    if constexpr (HIGH)
        if (sa.note && cta == 0 && threadIdx.x == 0)
            *reinterpret_cast<volatile unsigned*>(sa.note) = sa.stored * 2u + (*sa.high_zeros != 0u ? 1u : 0u);

    if (warp == kProducerWarp) {
        // ================================================================== producer (one warp)
        // Lane 0 owns the barriers and issues a unit's copy; of a nested child a lane per blob issues that blob's.
        GemvOp* opbuf = reinterpret_cast<GemvOp*>(smem + S::oOpBuf);
        uint8_t* opring = smem + S::oOpRing;
        OpFetch fetch;
        fetch.issue(ops, 0, sa.n_ops, lane);
        fetch.store(&opbuf[0], lane);
        __syncwarp();
        int stage = 0;                               // ring position and how often the ring wrapped (32-bit state only:
        unsigned wraps = 0;                          // this loop is the serial bottleneck of the CTA)
        int seg = -1, op_seq = -1;
        int oseq = 0;                                // finishing units issued so far
        bool stop = false;
        for (int oi = 0; oi < sa.n_ops && !stop; oi++) {
            const OpFetch cur = fetch;                                // the words of this op, still in registers
            fetch.issue(ops, oi + 1, sa.n_ops, lane);                 // travels while this op is issued
            const GemvOp& op = opbuf[oi & 1];
            int lo, hi;
            cta_range(op.n_units, op.rot, cta, grid, lo, hi);
            if (lo < hi) {
                op_seq++;
                const int op_slot = op_seq % kOpRing;
                cur.store(reinterpret_cast<GemvOp*>(opring + op_slot * S::kOpBytes), lane);   // for the consumers
                __threadfence_block();
                __syncwarp();          // all 32 lanes' words are in place before lane 0 announces the first unit
                // a PACKED variant's blobs are contiguous: one copy per unit (lane 0); a nested child reads a
                // prefix of every blob: one copy per blob (lanes 0 .. nb-1).
                // Everything the unit loop needs sits in registers and is advanced by additions: this loop
                // is the serial path that feeds the whole CTA.
                const int n_rp = op.n_rp, n_kb = op.n_kb, chunk_blobs = op.chunk_blobs, n_chunks = op.n_chunks;
                const uint32_t blob_read = (uint32_t)op.blob_read;
                const long long blob_stride = op.blob_stride;
                const uint8_t* store = op.store;
                const bool contiguous = op.blob_read == op.blob_stride;
                const long long rp_stride = (long long)n_kb * blob_stride;
                int ch = lo / n_rp, rp = lo - ch * n_rp;
                int rpm = rp % n_chunks;                             // rp mod n_chunks, kept up by counting
                int n_left = hi - lo;
                while (n_left > 0 && !stop) {
                    // ---- the units of one K chunk
                    seg++;
                    const int kb0 = ch * chunk_blobs;
                    const int nb = min(chunk_blobs, n_kb - kb0);
                    const uint32_t bytes = (uint32_t)nb * blob_read;
                    const uint8_t* src = store + ((long long)rp * n_kb + kb0) * blob_stride;
                    const int in_chunk = min(n_left, n_rp - rp);
                    for (int i = 0; i < in_chunk; i++) {
                        const uint32_t full = bars + 8 * stage, empty = bars + 8 * (S::kStages + stage);
                        int ok = 1;
                        if (lane == 0) {
                            if (wraps > 0 && !mbar_try_wait(empty, (wraps - 1u) & 1u)) {
                                // the ring is full: the usual case when the consumers wait for activations
                                if (flags[1]) ok = 0;
                                else if (!mbar_wait(empty, (wraps - 1u) & 1u, sa.wait_ns)) {
                                    give_up(sa.status, flags);
                                    ok = 0;
                                }
                            }
                            if (ok) {
                                // the chunk that adds up a row pair rotates with the row pair, so that this work
                                // (and the place in the output queue it needs) is spread evenly over the CTAs
                                int4* d = reinterpret_cast<int4*>(smem + S::oDesc + stage * (int)sizeof(UnitDesc));
                                d[0] = make_int4(ch, rp, nb, seg);
                                d[1] = make_int4(op_slot, ch == rpm ? oseq : -1, 0, 0);
                                mbar_expect_tx(full, bytes);
                            }
                        }
                        ok = __shfl_sync(0xffffffffu, ok, 0);
                        if (!ok) { stop = true; break; }
                        const uint32_t stage_base = smem_u32(smem + S::oStages) + (uint32_t)stage * S::kStageBytes;
                        // (checked build) the blobs of this copy lie inside the stored variant and fit the stage; the
                        // transaction stays pending, the status word ends every wait
                        if (!FQ_IN_BOUNDS(rp >= 0 && rp < n_rp && kb0 >= 0 && kb0 + nb <= n_kb && bytes <= (uint32_t)S::kStageBytes,
                                          sa.status)) {
                            if (lane == 0) give_up(sa.status, flags);
                            stop = true;
                            break;
                        }
                        if (contiguous) {
                            if (lane == 0) bulk_g2s(stage_base, src, bytes, full);
                        } else if (lane < nb) {
                            bulk_g2s(stage_base + lane * blob_read, src + lane * blob_stride, blob_read, full);
                        }
                        if (ch == rpm) oseq++;
                        if (++rpm == n_chunks) rpm = 0;
                        if (++stage == S::kStages) { stage = 0; wraps++; }
                        rp++;
                        src += rp_stride;
                    }
                    n_left -= in_chunk;
                    rp = 0; rpm = 0; ch++;
                }
                if (lane == 0 && flags[1]) stop = true;
                stop = __shfl_sync(0xffffffffu, stop ? 1 : 0, 0) != 0;
            }
            __syncwarp();
            fetch.store(&opbuf[(oi + 1) & 1], lane);
            __syncwarp();
        }
        if (stop) let_copies_land();
        if (lane == 0 && !stop) out_total[0] = oseq;                // the output warps may leave after this many
    } else if (warp == kActWarp) {
        // ================================================================== activations
        // One (op, K chunk) segment after the other: wait until a slot is free and the phase that produces the activations is
        // complete, then one bulk copy per batch row; the consumers sleep on the slot's barrier.
        GemvOp* opbuf = reinterpret_cast<GemvOp*>(smem + S::oOpBuf) + 2;
        OpFetch fetch;
        fetch.issue(ops, 0, sa.n_ops, lane);
        fetch.store(&opbuf[0], lane);
        __syncwarp();
        int seg = -1;
        int phase_known = -1;                       // every phase <= phase_known is complete
        bool stop = false;
        for (int oi = 0; oi < sa.n_ops && !stop; oi++) {
            if (oi > 0) {
                __syncwarp();
                fetch.store(&opbuf[oi & 1], lane);
                __syncwarp();
            }
            fetch.issue(ops, oi + 1, sa.n_ops, lane);                 // travels while this op is processed
            const GemvOp& op = opbuf[oi & 1];
            int lo, hi;
            cta_range(op.n_units, op.rot, cta, grid, lo, hi);
            if (lo >= hi) continue;
            const int ch_lo = lo / op.n_rp, ch_hi = (hi - 1) / op.n_rp;
            for (int ch = ch_lo; ch <= ch_hi && !stop; ch++) {
                seg++;
                const int units = min(hi, (ch + 1) * op.n_rp) - max(lo, ch * op.n_rp);
                const int slot = seg % kXSlots;
                const uint32_t xs = smem_u32(smem + S::oX) + (uint32_t)slot * S::kXSlotBytes, bar = xbars + 8 * slot;
                int go = 1;                                            // 0: stop, 1: fetch, 2: publish without fetching
                if (lane == 0) {
                    // the slot is free when every unit of the segment that used it before is done
                    if (!smem_wait([&] { return x_pending[slot] == 0 || flags[1]; }, sa.wait_ns)) give_up(sa.status, flags);
                    // the activations are the previous phase's outputs
                    if (!flags[0] && op.phase > 0 && phase_known < op.phase - 1) {
                        const unsigned long long need = (unsigned long long)sa.phase_total[op.phase - 1];
                        const unsigned long long t0 = global_ns();
                        unsigned it = 0;
                        while (ld_acquire_u64(sa.phase_done + (op.phase - 1)) < need) {
                            if ((++it & 63u) == 0u &&
                                (global_ns() - t0 > sa.wait_ns || *reinterpret_cast<volatile int*>(sa.status) != 0 ||
                                 flags[0])) { atomicCAS(sa.status, 0, FQ_ERR_TIMEOUT); flags[0] = 1; break; }
                        }
                    }
                    // other SMs' plain stores (y of the previous phase) and this SM's reads of the slot before the copies below
                    __threadfence_block();
                    asm volatile("fence.proxy.async;" ::: "memory");
                    go = flags[1] ? 0 : (flags[0] ? 2 : 1);
                }
                go = __shfl_sync(0xffffffffu, go, 0);
                if (op.phase > 0) phase_known = op.phase - 1;          // (meaningless after an abort; unused then)
                if (go == 0) { stop = true; break; }
                const int k0 = ch * op.chunk_blobs * (kBlobSteps * kStepCols);
                const int cols = min(op.chunk_blobs * (kBlobSteps * kStepCols), op.n_kb * (kBlobSteps * kStepCols) - k0);
                const int have = min(cols, op.k_in - k0);              // (a multiple of 128, at least 128)
                // columns beyond k_in have weights of zero: their activations must be numbers
                if (have < cols)
                    for (int i = lane; i < op.batch * ((cols - have) / 8); i += 32) {
                        const int b = i / ((cols - have) / 8), k = have + i % ((cols - have) / 8) * 8;
                        sts128(xs + (uint32_t)(b * kXRowBytes + k * 2), make_uint4(0u, 0u, 0u, 0u));
                    }
                __threadfence_block();
                __syncwarp();
                if (lane == 0) {
                    x_pending[slot] = units * S::kWarpsPerUnit;
                    __threadfence_block();
                    x_ready[slot] = seg + 1;
                    __threadfence_block();
                    if (go == 1) mbar_expect_tx(bar, (uint32_t)(op.batch * have * 2));
                    else mbar_arrive(bar);
                }
                __syncwarp();
                if (go == 1 && lane < op.batch && FQ_IN_BOUNDS(k0 + have <= op.k_in && have <= kXCols, sa.status))
                    bulk_g2s(xs + (uint32_t)(lane * kXRowBytes), reinterpret_cast<const __half*>(op.x) + (long long)lane * op.k_in + k0,
                             (uint32_t)have * 2u, bar);
            }
        }
        if (stop) let_copies_land();
    } else if (warp >= kOutputWarp) {
        // ================================================================== output warps
        // Finishes row pairs.  The unit whose K chunk is (row pair mod chunks) adds up its row pair: its own
        // sums arrive through the queue in shared memory, the other chunks' sums are tagged 64-bit words in
        // global memory (value, launch tag) that their consumers stored without any fence -- a word counts
        // once its tag is this launch's.  The sums are added in chunk order, so results do not depend on
        // timing.  One fence per batch of finished row pairs orders y before the phase counter.
        const int ow = warp - kOutputWarp;                               // takes the places congruent to ow
        const float* odata = reinterpret_cast<const float*>(smem + S::oOutData);
        const OutDesc* odesc = reinterpret_cast<const OutDesc*>(smem + S::oOutDesc);
        int processed = 0;
        unsigned long long last_progress = 0ull;
        unsigned idle_it = 0u;
        for (;;) {
            // every decision that ends the loop is taken by lane 0 and broadcast: the lanes must leave together
            const bool filled = lane < kOutSlots && lane % kOutputWarps == ow && out_fill[lane] == (unsigned)kUnitRowTiles;
            const unsigned m = __ballot_sync(0xffffffffu, filled);
            unsigned done = 0u;
            if (m) {
                __threadfence_block();                                   // the slots' contents after their fill counts
                for (unsigned mm = m; mm; mm &= mm - 1u) {
                    const int s = __ffs(mm) - 1;
                    const OutDesc& d = odesc[s];
                    const float* o = odata + s * S::kOutFloats;
                    // lane = row; a few chunks per round trip, every batch entry of them in flight at once; a round
                    // whose words are not all there ends the attempt
                    constexpr int QS = 16 / BP;
                    float sum[BP];
#pragma unroll
                    for (int i = 0; i < BP; i++) sum[i] = 0.f;
                    bool ok = true;
                    const unsigned long long* pt = d.partial + (long long)d.rp * d.n_chunks * (32 * BP) + lane * BP;
                    for (int q0 = 0; q0 < d.n_chunks; q0 += QS) {
                        ulonglong2 w[QS][BP / 2];
#pragma unroll
                        for (int j = 0; j < QS; j++) {
                            const int q = q0 + j;
#pragma unroll
                            for (int i = 0; i < BP / 2; i++) {
                                w[j][i] = make_ulonglong2(0ull, 0ull);
                                if (q < d.n_chunks && q != d.ch) w[j][i] = ld_relaxed_u64x2(pt + (long long)q * (32 * BP) + 2 * i);
                            }
                        }
#pragma unroll
                        for (int j = 0; j < QS; j++) {
                            const int q = q0 + j;
                            if (q >= d.n_chunks) break;
                            if (q == d.ch) {
#pragma unroll
                                for (int i = 0; i < BP; i++) sum[i] += o[lane * BP + i];
                            } else {
#pragma unroll
                                for (int i = 0; i < BP / 2; i++) {
                                    ok = ok && (unsigned)(w[j][i].x >> 32) == sa.epoch && (unsigned)(w[j][i].y >> 32) == sa.epoch;
                                    sum[2 * i] += __uint_as_float((unsigned)w[j][i].x);
                                    sum[2 * i + 1] += __uint_as_float((unsigned)w[j][i].y);
                                }
                            }
                        }
                        if (!__all_sync(0xffffffffu, ok)) break;
                    }
                    if (!__all_sync(0xffffffffu, ok)) continue;          // some chunk has not arrived yet: look again later
                    const int row = d.rp * (kUnitRowTiles * kTileRows) + lane;
                    __half* y = reinterpret_cast<__half*>(d.y);
                    if (row < d.n_out) {
                        // sums of numbers stay finite: an infinite one comes from an activation that is none, and such a one makes
                        // every output of its batch entry NaN (as the batch-1 kernel does, and fq_gemv promises)
#pragma unroll
                        for (int b = 0; b < BP; b++)
                            if (b < d.batch) y[(long long)b * d.n_out + row] = __float2half_rn(fmaf(sum[b], 0.f, sum[b]));
                    }
                    done |= 1u << s;
                }
            }
            if (done) {
                __syncwarp();
                __threadfence();                                         // y before the phase counter
                if ((done >> lane) & 1u) {
                    const int phase = odesc[lane].phase;
                    if (phase >= 0) red_add_relaxed_u64(sa.phase_done + phase, 1ull);
                    out_fill[lane] = 0u;                                 // hand the slot back
                    __threadfence_block();
                    out_gen[lane] = out_gen[lane] + 1u;
                }
                processed += __popc(done);
                last_progress = 0ull; idle_it = 0u;
                continue;
            }
            int leave = 0;
            if (lane == 0) {
                const int want = out_total[0];
                if (flags[0] || (want >= 0 && processed >= (want + kOutputWarps - 1 - ow) / kOutputWarps)) leave = 1;
                else if ((++idle_it & 127u) == 0u) {
                    const unsigned long long now = global_ns();
                    if (last_progress == 0ull) last_progress = now;
                    else if (now - last_progress > sa.wait_ns) {
                        give_up(sa.status, flags);
                        leave = 1;
                    }
                }
            }
            if (__shfl_sync(0xffffffffu, leave, 0)) break;
            __nanosleep(20);
        }
    } else {
        // ================================================================== consumers
        // Two or four warps share a unit (see GemvSmem), each computes one of its two 16-row tiles, over all or half of the columns.
        const int g = lane >> 2, c = lane & 3;
        const int uidx = warp / S::kWarpsPerUnit;                       // which of the units in flight
        const int tile = warp % kUnitRowTiles, half = S::kHalves ? warp / kUnitRowTiles % 2 : 0;   // this warp's row tile and columns
        volatile unsigned* delivered = half_ctl + (uidx * kUnitRowTiles + tile) * 2;   // halves of the unit at hand; [1]: units done
        float* halves = reinterpret_cast<float*>(smem + S::oHalf) + uidx * 2 * S::kOutFloats;
        unsigned turn = 0;                                           // units of this group so far
        int total = 0;                               // units of this CTA over the whole launch
        if (sa.cta_units) total = sa.cta_units[cta];
        else {
            int lo, hi;
            cta_range(single.n_units, single.rot, cta, grid, lo, hi);
            total = hi - lo;
        }
        const uint8_t* opring = smem + S::oOpRing;
        float* odata = reinterpret_cast<float*>(smem + S::oOutData);
        OutDesc* odesc = reinterpret_cast<OutDesc*>(smem + S::oOutDesc);
        bool stop = false;
        // ring position of this warp's next unit, advanced by additions
        int stage = uidx % S::kStages;
        unsigned use = (unsigned)(uidx / S::kStages);
        const uint32_t opring_a = smem_u32(smem + S::oOpRing), desc_a = smem_u32(smem + S::oDesc);
        for (int seq = uidx; seq < total && !stop; seq += S::kUnitsInFlight) {
            const uint32_t full = bars + 8 * stage, empty = bars + 8 * (S::kStages + stage);
            // a stage's uses are consumed strictly in order: wait for the release of the previous
            // use before trusting the parity of the full barrier
            bool ok = true;
            if (use > 0) ok = smem_wait([&] { return released[stage] >= use * S::kWarpsPerUnit || flags[1]; }, sa.wait_ns);
            if (ok) ok = mbar_wait(full, use & 1u, sa.wait_ns);
            if (!ok) give_up(sa.status, flags);
            if (!__all_sync(0xffffffffu, flags[1] == 0)) { stop = true; break; }      // (the lanes leave together, whatever the clocks of their waits said)
            struct { int ch, rp, cnt, seg, blob_read, variant, batch, op_slot, oseq, n_chunks;
                     unsigned long long* partial; } d;
            {
                const uint4 u0 = lds128(desc_a + stage * (int)sizeof(UnitDesc));            // ch, rp, nb, seg
                const uint2 u1 = lds64(desc_a + stage * (int)sizeof(UnitDesc) + 16);        // op_slot, oseq
                const uint32_t od = opring_a + u1.x * S::kOpBytes;
                const uint4 o1 = lds128(od + 16);                                           // blob_read, variant, batch, n_chunks
                const uint2 o0 = lds64(od + 8);                                             // partial
                d.ch = (int)u0.x; d.rp = (int)u0.y; d.cnt = (int)u0.z * kBlobSteps / (S::kHalves ? 2 : 1); d.seg = (int)u0.w;
                d.op_slot = (int)u1.x; d.oseq = (int)u1.y;
                d.blob_read = (int)o1.x; d.variant = (int)o1.y; d.batch = (int)o1.z; d.n_chunks = (int)o1.w;
                d.partial = reinterpret_cast<unsigned long long*>(((unsigned long long)o0.y << 32) | o0.x);
            }
            // a unit that finishes its row pair needs a place in the output queue: that place must be free
            // again; the descriptor goes there now, while the op's slot in the op ring is certainly still valid
            const int oslot = d.oseq % kOutSlots;
            if (d.oseq >= 0) {
                const unsigned ogen = (unsigned)(d.oseq / kOutSlots);
                if (!smem_wait([&] { return out_gen[oslot] == ogen || flags[1]; }, sa.wait_ns)) give_up(sa.status, flags);
                if (!__all_sync(0xffffffffu, flags[1] == 0)) { stop = true; break; }
                if (tile == 0 && half == 0 && lane == 0) {
                    const GemvOp& od = *reinterpret_cast<const GemvOp*>(opring + d.op_slot * S::kOpBytes);
                    OutDesc& q = odesc[oslot];
                    q.rp = d.rp; q.ch = d.ch; q.n_chunks = od.n_chunks; q.n_out = od.n_out; q.phase = od.phase; q.batch = od.batch;
                    q.y = od.y; q.partial = od.partial;
                }
            }
            const int slot = d.seg % kXSlots;
            // sleep on the slot's barrier (a hardware wake-up: this wait is on the critical path of every
            // dependency phase); a warp that is several publications ahead would read a stale parity, so only a barrier that
            // belongs to this segment counts
            const unsigned xpar = (unsigned)(d.seg / kXSlots) & 1u;
            if (x_ready[slot] != d.seg + 1 && !flags[1]) mbar_wait(xbars + 8 * slot, xpar, sa.wait_ns);
            if (!smem_wait([&] { return x_ready[slot] == d.seg + 1 || flags[1]; }, sa.wait_ns) || (!flags[1] && !mbar_wait(xbars + 8 * slot, xpar, sa.wait_ns)))
                give_up(sa.status, flags);
            __threadfence_block();
            const bool live = __all_sync(0xffffffffu, flags[0] == 0);

            float tot[4] = {0.f, 0.f, 0.f, 0.f};
            if constexpr (HIGH)
                if (live && *sa.high_zeros != 0u)
                    unit_take_high_zeros<BP>(smem_u32(smem + S::oStages) + (uint32_t)stage * S::kStageBytes, half * d.cnt, d.cnt, (uint32_t)d.blob_read,
                                             smem_u32(smem + S::oX) + (uint32_t)slot * S::kXSlotBytes, lane, tile, tot);
            if (live)
                unit_dispatch<BP>(d.variant, smem_u32(smem + S::oStages) + (uint32_t)stage * S::kStageBytes, half * d.cnt, d.cnt, (uint32_t)d.blob_read,
                                  smem_u32(smem + S::oX) + (uint32_t)slot * S::kXSlotBytes, lane, tile, tot);
            __syncwarp();
            if (lane == 0) {
                atomicAdd(const_cast<unsigned*>(&released[stage]), 1u);
                __threadfence_block();
                mbar_arrive(empty);                              // the stage may be refilled
                atomicSub(const_cast<int*>(&x_pending[slot]), 1);   // one warp fewer needs the activation slot
            }
            stage += S::kUnitsInFlight;
            while (stage >= S::kStages) { stage -= S::kStages; use++; }
            if (!live) continue;

            // ---- the row sums: tot[2 r + i] of lane (g, c) belongs to local row tile * 16 + g + 8 r, batch entry 2 c + i
            const int lr = tile * kTileRows + g;
            // the two halves of the columns: whoever delivers the second one adds the first (the order does not change the sum)
            if constexpr (S::kHalves) {
                if (!smem_wait([&] { return delivered[1] >= turn || flags[1]; }, sa.wait_ns)) give_up(sa.status, flags);        // the previous unit's have been taken
                if (__any_sync(0xffffffffu, flags[1] != 0)) { stop = true; break; }
                turn++;
                float* mine = halves + half * S::kOutFloats;
                if (2 * c < BP) {
                    *reinterpret_cast<float2*>(mine + lr * BP + 2 * c) = make_float2(tot[0], tot[1]);
                    *reinterpret_cast<float2*>(mine + (lr + 8) * BP + 2 * c) = make_float2(tot[2], tot[3]);
                }
                __threadfence_block();
                __syncwarp();
                unsigned before = 0;
                if (lane == 0) before = atomicAdd(const_cast<unsigned*>(&delivered[0]), 1u);
                if (__shfl_sync(0xffffffffu, before, 0) == 0u) continue;
                __threadfence_block();
                const float* other = halves + (half ^ 1) * S::kOutFloats;
                if (2 * c < BP) {
                    const float2 o0 = *reinterpret_cast<const float2*>(other + lr * BP + 2 * c);
                    const float2 o1 = *reinterpret_cast<const float2*>(other + (lr + 8) * BP + 2 * c);
                    tot[0] += o0.x; tot[1] += o0.y; tot[2] += o1.x; tot[3] += o1.y;
                }
                __syncwarp();
                if (lane == 0) {
                    delivered[0] = 0u;
                    __threadfence_block();
                    delivered[1] = turn;
                }
            }
            if (d.oseq >= 0) {
                // this unit finishes its row pair: hand the sums to the output warps
                float* o = odata + oslot * S::kOutFloats;
                if (2 * c < BP) {
                    *reinterpret_cast<float2*>(o + lr * BP + 2 * c) = make_float2(tot[0], tot[1]);
                    *reinterpret_cast<float2*>(o + (lr + 8) * BP + 2 * c) = make_float2(tot[2], tot[3]);
                }
                __threadfence_block();
                __syncwarp();
                if (lane == 0) atomicAdd(const_cast<unsigned*>(&out_fill[oslot]), 1u);
            } else if (2 * c < BP) {
                // another unit finishes it: publish tagged words (value, launch tag), fire and forget
                unsigned long long* pu = d.partial + ((long long)d.rp * d.n_chunks + d.ch) * (32 * BP) + lr * BP + 2 * c;
                const unsigned long long tag = (unsigned long long)sa.epoch << 32;
                st_relaxed_u64x2(pu, tag | __float_as_uint(tot[0]), tag | __float_as_uint(tot[1]));
                st_relaxed_u64x2(pu + 8 * BP, tag | __float_as_uint(tot[2]), tag | __float_as_uint(tot[3]));
            }
        }
        if (stop) let_copies_land();
    }

    __syncthreads();
    if (threadIdx.x == 0 && sa.n_phases > 0) {
        __threadfence();
        const unsigned old = atomicAdd(sa.exit_count, 1u);
        if (old == gridDim.x - 1) {                    // last CTA out: counters back to zero
            for (int p = 0; p < sa.n_phases; p++) sa.phase_done[p] = 0ull;
            *sa.exit_count = 0u;
            __threadfence();
        }
    }
}

// ------------------------------------------------------------------------------- launchers
// The launch is always cooperative: a CTA that finishes a row pair waits (bounded) for sums that other
// CTAs produce, so all CTAs of the grid have to be resident together.
template <int BP, bool HIGH>
static int launch_impl(Ctx* ctx, const GemvOp& single, const StackArgs& sa, long long total_units, cudaStream_t st)
{
    using S = GemvSmem<BP>;
    static bool configured[64] = {};
    if (ctx->device < 64 && !configured[ctx->device]) {
        FQ_CUDA_OK(cudaFuncSetAttribute(gemv_kernel<BP, HIGH>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kTotal));
        configured[ctx->device] = true;
    }
    long long blocks = ctx->sm_count;
    if (total_units < blocks) blocks = total_units;
    if (blocks < 1) return FQ_OK;
    void* args[] = {(void*)&single, (void*)&sa};
    FQ_CUDA_OK(cudaLaunchCooperativeKernel((const void*)gemv_kernel<BP, HIGH>, dim3((unsigned)blocks), dim3(kGemvThreads),
                                           args, S::kTotal, st));
    return FQ_OK;
}

// Are all zero points stored so far below 1024?  The kernel that need not ask is 2 % faster at batch 8, one that asks (HIGH) has the
// same results where they are.  The answer is on the device: a launch of the asking kernel leaves it in a word of host memory, with
// the state of the context that it holds for, and until that arrives every launch is of the asking one.  Nobody waits.
static bool zeros_are_low(const Ctx* ctx)
{
    return ctx->note && *const_cast<const volatile unsigned*>(ctx->note) == (ctx->stored & 0x7fffffffu) * 2u;
}

static int launch_batch(Ctx* ctx, const GemvOp& single, StackArgs& sa, int batch, long long total_units, cudaStream_t st)
{
    sa.high_zeros = high_zeros_word(ctx);
    sa.note = ctx->note;
    sa.stored = ctx->stored;
    sa.wait_ns = ctx->wait_limit_ns;
    if (zeros_are_low(ctx))
        return batch_pad(batch) == 4 ? launch_impl<4, false>(ctx, single, sa, total_units, st) : launch_impl<8, false>(ctx, single, sa, total_units, st);
    return batch_pad(batch) == 4 ? launch_impl<4, true>(ctx, single, sa, total_units, st) : launch_impl<8, true>(ctx, single, sa, total_units, st);
}

// Tag for the split-K partials of the next launch that uses the context's workspace.
static unsigned next_epoch(unsigned& e)
{
    if (++e == 0u) ++e;                        // 0 marks words that no launch has written
    return e;
}

int launch_gemv_single(Ctx* ctx, const GemvOp& op, cudaStream_t st)
{
    StackArgs sa{};
    sa.table = nullptr;
    sa.status = ctx->status_dev;
    sa.n_ops = 1;
    sa.n_phases = 0;
    sa.epoch = next_epoch(ctx->launch_epoch);
    const long long units = (long long)op.n_rp * op.n_chunks;
    return launch_batch(ctx, op, sa, op.batch, units, st);
}

int launch_gemv_stack(Ctx* ctx, const StackHeader& hdr, const char* table_dev, int max_batch, cudaStream_t st)
{
    // counters live in the workspace head
    StackArgs sa{};
    sa.table = reinterpret_cast<const GemvOp*>(table_dev);
    sa.phase_total = reinterpret_cast<const long long*>(table_dev + (size_t)hdr.n_ops * sizeof(GemvOp));
    sa.cta_units = reinterpret_cast<const int*>(sa.phase_total + (hdr.n_phases > 0 ? hdr.n_phases : 1));
    sa.phase_done = reinterpret_cast<unsigned long long*>(ctx->ws);
    sa.exit_count = reinterpret_cast<unsigned*>(ctx->ws + 8 * 4096);
    sa.status = ctx->status_dev;
    sa.n_ops = hdr.n_ops;
    sa.n_phases = hdr.n_phases;
    sa.epoch = next_epoch(ctx->launch_epoch);
    GemvOp dummy{};
    return launch_batch(ctx, dummy, sa, max_batch, hdr.total_units, st);
}

}  // namespace fq
