// Decode path for a batch of 2..8 activation rows: fused dequantize-GEMV over tiled field arrays.
// (Batch 1 has its own kernel in fq_gemv1.cu.)
//
// One persistent CTA per SM with four roles:
//   producer warp   : streams "units" (a blob: 32 output rows x one K chunk of 512 columns, every field array of the
//                     active variant plus the scale/zero words) from HBM into a shared-memory ring of bytes with bulk
//                     asynchronous copies (cp.async.bulk + mbarrier tx counts) and writes a small descriptor for each;
//   activation warp : once per (op, K chunk) that this CTA touches, waits -- bounded -- for the
//                     previous dependency phase and fetches the activations of that chunk, one bulk copy per batch row;
//   consumer warps  : two warps share a unit, one 16-row tile each.  Stored words become fp16 integers q - z, the fp16
//                     activations are the other operand of mma.m16n8k16, sums are fp32 and scaled once per group of 128
//                     columns (fq_batch_core.cuh).  The loops are compiled once per field list (14 variants) and chosen
//                     per unit;
//   output warps    : finish row pairs (see below) and are the only warps that write y.
// The K chunks of one row pair are computed by different CTAs.  Each unit publishes its row sums
// as 64-bit words (fp32 value, launch tag) with plain stores; the output warps of the CTA that has the unit whose chunk index is
// (row pair mod chunks) poll the words of all chunks until they carry this launch's tag and add them in chunk order, so results
// do not depend on scheduling and no fence or atomic sits on the consumers' path.
//
// What bounds it: a mma.sync holds its scheduler for 8 cycles, so the loops cost (instructions + 8 x MMAs) / 4 cycles of an SM, 45
// weights a cycle for one field, about what HBM delivers at 4 bits; beside that the latencies of a phase.  A ring of whole stages had as
// many of them (8 - 11 of 17 KB) as units in work, so that nothing was fetched ahead; units of one blob in a ring of bytes leave
// two thirds of it for that, whatever the width.  Four 7B blocks without / with dependencies, us, stages -> bytes: 8 entries, mixed
// widths 180 / 323 -> 143 / 250, nested 6 bits 223 / 376 -> 157 / 266; 4 entries 167 / 264 -> 134 / 230 and 220 / 317 -> 154 / 251.  (Of
// the ordered gain a third is the output warps': four instead of two, all loads of a row pair on their way at once, one count
// per CTA and phase instead of one per row pair.)
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

constexpr int kConsumerWarps = 16;                     // (20 are no faster: the loops are bound by issue slots, and then 80 registers are all there is)
constexpr int kProducerWarp = kConsumerWarps;          // warp index of the producer
constexpr int kActWarp = kConsumerWarps + 1;           // the warp that fetches activations
constexpr int kOutputWarp = kActWarp + 1;              // the warps that own every global store of results
constexpr int kOutputWarps = 4;                        // each writes a quarter of the rows of every row pair
constexpr int kGemvThreads = (kConsumerWarps + 2 + kOutputWarps) * 32;     // 22 warps: 88 registers each
constexpr int kWarpsPerUnit = kUnitRowTiles;           // one 16-row tile each
constexpr int kUnitsInFlight = kConsumerWarps / kWarpsPerUnit;
// Units that are on their way or in work, at most.  A multiple of the units in flight: a place then always belongs to the same warps,
// which have seen every use of it, so that the parity of its barrier says which use it is.
constexpr int kPlaces = 32;
static_assert(kPlaces % kUnitsInFlight == 0 && kPlaces <= 32, "a lane of the producer per place");
constexpr int kMarks = 64;                             // marks of units that finish a row pair (they are used again, see the output warps)
constexpr int kXSlots = 5;                             // activation chunks kept in shared memory

// What the producer tells the consumers of a unit.
struct UnitDesc {
    int ch, rp, off, seg;                       // K chunk, row pair, place of the weights in the ring, activation segment
    int variant, n_chunks;
    unsigned long long* partial;
    int oseq;                                   // >= 0: this CTA finishes the unit's row pair, the oseq-th one that it finishes
    unsigned start;                             // position in the ring, never wrapped
    int pad[2];
};
static_assert(sizeof(UnitDesc) == 48, "descriptor layout");

template <int BP> struct GemvSmem {
    static constexpr int kXSlotBytes = BP * kXRowBytes;              // one chunk's activations
    static constexpr int kOpBytes = (int)((sizeof(GemvOp) + 15) / 16 * 16);
    static constexpr int kFixed = kPlaces * ((int)sizeof(UnitDesc) + 16) + kXSlots * kXSlotBytes + (4 + 2 * kOutputWarps) * kOpBytes + kMarks * 4 + 256;
    static constexpr int kRing = (232448 - kFixed) / 512 * 512;      // (blobs are multiples of 512 bytes)
    static constexpr int oRing = 0;
    static constexpr int oDesc = oRing + kRing;                      // UnitDesc[kPlaces]
    static constexpr int oX = oDesc + kPlaces * (int)sizeof(UnitDesc);
    static constexpr int oOpBuf = oX + kXSlots * kXSlotBytes;        // GemvOp[2] of the producer, the activation warp and every output warp
    static constexpr int oBars = oOpBuf + (4 + 2 * kOutputWarps) * kOpBytes;   // full[kPlaces], empty[kPlaces]
    static constexpr int oXBars = oBars + 2 * kPlaces * 8;           // one mbarrier per activation slot
    static constexpr int oCtl = oXBars + 8 * kXSlots;                // x_ready[XS], x_pending[XS], flags[2]
    static constexpr int oMarks = oCtl + (2 * kXSlots + 2) * 4;      // u32[kMarks]
    static constexpr int oFinished = oMarks + kMarks * 4;            // u32[4]: output warps that are done with a phase
    static constexpr int kTotal = oFinished + 16;
    static_assert(kRing >= 6 * (kBlobMetaBytes + kBlobSteps * kBlobTiles * 512 * 8), "decode kernel: no room for a ring");
    static_assert(kTotal <= 232448, "decode kernel: shared memory over the 227 KB per-CTA limit");
    static_assert(oBars % 8 == 0 && oXBars % 8 == 0 && oX % 16 == 0 && kOpBytes % 16 == 0, "alignment");
};

// A split-K partial is one 64-bit word per (row, batch entry): fp32 sum in the low half, launch tag in the high half.
size_t gemv_partial_bytes_per_unit(int batch) { return (size_t)(32 * batch_pad(batch)) * sizeof(unsigned long long); }

// ------------------------------------------------------------------------------- per-CTA work split
// (this kernel numbers the units of an op chunk-major, u = ch * n_rp + rp, and deals them with cta_range)
void gemv_cta_range(int n_units, int rot, int cta, int grid, int& lo, int& hi) { cta_range(n_units, rot, cta, grid, lo, hi); }

struct StackArgs {
    const GemvOp* table;                   // device op table (nullptr: use the by-value op)
    const long long* phase_total;          // row pairs per phase
    unsigned long long* phase_done;        // finished row pairs per phase
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
    const uint32_t bars = smem_u32(smem + S::oBars);                          // full, empty
    volatile int* x_ready = reinterpret_cast<volatile int*>(smem + S::oCtl);   // segment number + 1 held by a slot
    const uint32_t xbars = smem_u32(smem + S::oXBars);                         // completes a phase per publication of a slot
    volatile int* x_pending = x_ready + kXSlots;                               // warps' units that still need the slot
    volatile int* flags = x_pending + kXSlots;                                 // [0]: stop computing, [1]: stop everything
    volatile unsigned* marks = reinterpret_cast<volatile unsigned*>(smem + S::oMarks);       // row tiles of finishing units that are done, ever
    volatile unsigned* finished = marks + kMarks;                              // [phase & 3]: output warps that are done with the phase

    if (threadIdx.x == 0) {
        for (int s = 0; s < kPlaces; s++) {
            mbar_init(bars + 8 * s, 1);
            mbar_init(bars + 8 * (kPlaces + s), kWarpsPerUnit);
        }
        for (int i = 0; i < kXSlots; i++) { x_ready[i] = 0; x_pending[i] = 0; mbar_init(xbars + 8 * i, 1); }
        for (int i = 0; i < kMarks + 4; i++) marks[i] = 0u;                   // (and finished)
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
        // Streams units into a ring of bytes, so that small ones are fetched as far ahead as large ones; space comes free in order.  This is
        // the serial path that feeds the whole CTA, so a lane takes a unit.
        GemvOp* opbuf = reinterpret_cast<GemvOp*>(smem + S::oOpBuf);
        OpFetch fetch;
        fetch.issue(ops, 0, sa.n_ops, lane);
        fetch.store(&opbuf[0], lane);
        __syncwarp();
        unsigned issued = 0, tail = 0;               // units asked for; units before `tail` are done
        unsigned head = 0, vhead = 0;                // where the next unit goes: in the ring, and without wrapping
        int seg = -1;
        int oseq = 0;                                // finishing units issued so far
        bool stop = false;
        for (int oi = 0; oi < sa.n_ops && !stop; oi++) {
            fetch.issue(ops, oi + 1, sa.n_ops, lane);                 // travels while this op is issued
            const GemvOp& op = opbuf[oi & 1];
            int lo, hi;
            cta_range(op.n_units, op.rot, cta, grid, lo, hi);
            if (lo < hi) {
                const int n_rp = op.n_rp, n_kb = op.n_kb, variant = op.variant;
                const uint32_t bytes = (uint32_t)op.blob_read;
                const long long blob_stride = op.blob_stride;
                const uint8_t* const store = op.store;
                unsigned long long* const partial = op.partial;
                const unsigned fit = (unsigned)S::kRing / bytes;
                int ch = lo / n_rp, rp = lo - ch * n_rp;
                int n_left = hi - lo;
                while (n_left > 0 && !stop) {
                    // ---- the units of one K chunk, up to a lane's worth at a time
                    seg++;
                    const int in_chunk = min(n_left, n_rp - rp);
                    for (int i0 = 0; i0 < in_chunk && !stop;) {
                        const unsigned before_wrap = ((unsigned)S::kRing - head) / bytes;
                        const int n = min(min(kPlaces, in_chunk - i0), (int)(before_wrap + fit)), my_rp = rp + i0 + lane;
                        const bool wrapped = (unsigned)lane >= before_wrap;
                        const unsigned off = wrapped ? ((unsigned)lane - before_wrap) * bytes : head + (unsigned)lane * bytes;
                        const unsigned start = wrapped ? vhead + ((unsigned)S::kRing - head) + off : vhead + (unsigned)lane * bytes;
                        // the chunk whose CTA adds up a row pair rotates with the row pair, so that this work is spread evenly over the CTAs
                        const bool finishes = lane < n && ch == my_rp % n_kb;
                        const unsigned fin = __ballot_sync(0xffffffffu, finishes);
                        const unsigned unit = issued + (unsigned)lane, place = unit % kPlaces, first = issued;
                        const uint32_t full = bars + 8 * place;
                        bool todo = lane < n;
                        // (checked build) the blobs of these copies lie inside the stored variant and the ring
                        if (!__all_sync(0xffffffffu, !todo || FQ_IN_BOUNDS(my_rp >= 0 && my_rp < n_rp && ch >= 0 && ch < n_kb && off + bytes <= (unsigned)S::kRing,
                                                                           sa.status))) {
                            if (lane == 0) give_up(sa.status, flags);
                            stop = true;
                            break;
                        }
                        unsigned long long t0 = 0ull;
                        unsigned moved = tail + issued;              // (both only grow)
                        for (unsigned it = 0;; it++) {
                            // units that have been consumed since, in order
                            const unsigned old = tail + (unsigned)lane;
                            const unsigned gone = __ballot_sync(0xffffffffu, (int)(issued - old) > 0 &&
                                                                                 mbar_test_wait(bars + 8 * (kPlaces + old % kPlaces), (old / kPlaces) & 1u));
                            __syncwarp();                            // (the descriptors that other lanes wrote)
                            tail += ~gone ? (unsigned)(__ffs(~gone) - 1) : 32u;
                            const unsigned next = __shfl_sync(0xffffffffu, start, (int)(issued - first));
                            const unsigned low = tail == issued ? next : reinterpret_cast<const volatile UnitDesc*>(smem + S::oDesc)[tail % kPlaces].start;
                            if (todo && start + bytes - low <= (unsigned)S::kRing && unit - tail < (unsigned)kPlaces) {
                                int4* d = reinterpret_cast<int4*>(smem + S::oDesc + place * (int)sizeof(UnitDesc));
                                d[0] = make_int4(ch, my_rp, (int)off, seg);
                                d[1] = make_int4(variant, n_kb, (int)(uint32_t)(uintptr_t)partial, (int)(uint32_t)((uintptr_t)partial >> 32));
                                *reinterpret_cast<int2*>(d + 2) = make_int2(finishes ? oseq + __popc(fin & ((1u << lane) - 1u)) : -1, (int)start);
                                mbar_expect_tx(full, bytes);
                                bulk_g2s(smem_u32(smem + S::oRing) + off, store + ((long long)my_rp * n_kb + ch) * blob_stride, bytes, full);
                                todo = false;
                            }
                            const unsigned left = __ballot_sync(0xffffffffu, todo);
                            issued = first + (unsigned)(n - __popc(left));
                            if (!left) break;
                            // the ring is full, the usual case when the consumers wait for activations: sleep on the oldest unit's barrier.
                            // What has a limit is the time without any progress
                            if (tail + issued != moved) { moved = tail + issued; t0 = 0ull; }
                            int leave = 0;
                            if (lane == 0 && !mbar_try_wait(bars + 8 * (kPlaces + tail % kPlaces), (tail / kPlaces) & 1u) && (it & 15u) == 15u) {
                                const unsigned long long now = global_ns();
                                if (flags[1]) leave = 1;
                                else if (t0 == 0ull) t0 = now;
                                else if (now - t0 > sa.wait_ns) { give_up(sa.status, flags); leave = 1; }
                            }
                            if (__shfl_sync(0xffffffffu, leave, 0)) { stop = true; break; }
                        }
                        oseq += __popc(fin);
                        head = __shfl_sync(0xffffffffu, off, n - 1) + bytes;
                        vhead = __shfl_sync(0xffffffffu, start, n - 1) + bytes;
                        i0 += n;
                    }
                    n_left -= in_chunk;
                    rp = 0; ch++;
                }
                if (lane == 0 && flags[1]) stop = true;
                stop = __shfl_sync(0xffffffffu, stop ? 1 : 0, 0) != 0;
            }
            __syncwarp();
            fetch.store(&opbuf[(oi + 1) & 1], lane);
            __syncwarp();
        }
        if (stop) let_copies_land();
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
                const int k0 = ch * kXCols;
                const int cols = kXCols, have = min(cols, op.k_in - k0);              // (a multiple of 128, at least 128)
                // the slot is free when every unit of the segment that used it before is done
                int go = 1;                                            // 0: stop, 1: fetch, 2: publish without fetching
                if (lane == 0 && !smem_wait([&] { return x_pending[slot] == 0 || flags[1]; }, sa.wait_ns)) give_up(sa.status, flags);
                __syncwarp();
                // columns beyond k_in have weights of zero: their activations must be numbers
                if (have < cols)
                    for (int i = lane; i < op.batch * ((cols - have) / 8); i += 32) {
                        const int b = i / ((cols - have) / 8), k = have + i % ((cols - have) / 8) * 8;
                        sts128(xs + (uint32_t)(b * kXRowBytes + k * 2), make_uint4(0u, 0u, 0u, 0u));
                    }
                fence_cta();
                __syncwarp();
                if (lane == 0) {
                    // all that can be done before the phase opens; from here on the consumers sleep on the slot's barrier
                    x_pending[slot] = units * kWarpsPerUnit;
                    fence_cta();
                    x_ready[slot] = seg + 1;
                    // the activations are the previous phase's outputs
                    if (!flags[0] && op.phase > 0 && phase_known < op.phase - 1) {
                        const unsigned long long need = (unsigned long long)sa.phase_total[op.phase - 1];
                        const unsigned long long t0 = global_ns();
                        unsigned it = 0;
                        while (ld_acquire_u64(sa.phase_done + (op.phase - 1)) < need) {
                            if ((++it & 3u) == 0u &&
                                (global_ns() - t0 > sa.wait_ns || *reinterpret_cast<volatile int*>(sa.status) != 0 ||
                                 flags[0])) { atomicCAS(sa.status, 0, FQ_ERR_TIMEOUT); flags[0] = 1; break; }
                        }
                    }
                    // other SMs' plain stores (y of the previous phase) and this SM's reads of the slot before the copies below
                    fence_cta();
                    asm volatile("fence.proxy.async;" ::: "memory");
                    go = flags[1] ? 0 : (flags[0] ? 2 : 1);
                    if (go == 1) mbar_expect_tx(bar, (uint32_t)(op.batch * have * 2));
                    else mbar_arrive(bar);
                }
                go = __shfl_sync(0xffffffffu, go, 0);
                __syncwarp();                                          // what lane 0 has seen comes before the other lanes' copies (a shuffle orders nothing)
                if (op.phase > 0) phase_known = op.phase - 1;          // (meaningless after an abort; unused then)
                if (go == 0) { stop = true; break; }
                if (go == 1 && lane < op.batch && FQ_IN_BOUNDS(k0 + have <= op.k_in && have <= kXCols, sa.status))
                    bulk_g2s(xs + (uint32_t)(lane * kXRowBytes), reinterpret_cast<const __half*>(op.x) + (long long)lane * op.k_in + k0,
                             (uint32_t)have * 2u, bar);
            }
        }
        if (stop) let_copies_land();
    } else if (warp >= kOutputWarp) {
        // ================================================================== output warps
        // Finish row pairs: the CTA that has the unit whose K chunk is (row pair mod chunks) adds up the sums of all chunks, tagged
        // 64-bit words in global memory (value, launch tag) that the consumers stored without any fence -- a word counts once its
        // tag is this launch's.  They are added in chunk order, so results do not depend on timing.  The warps walk the op list
        // by themselves: consumers never wait for them, so no order of units on different CTAs can lock up.  Each warp takes eight
        // rows of every row pair, four lanes a row, with the words of up to twelve chunks on their way at once: at the end of
        // a phase there are one or two row pairs for a CTA to finish, and everybody waits for them.
        const int ow = warp - kOutputWarp;                               // rows 8 ow .. 8 ow + 7
        constexpr int kEntries = BP / 4;                                 // batch entries of a lane
        constexpr int QS = 12;
        const int row_in = ow * (32 / kOutputWarps) + (lane >> 2), entry = (lane & 3) * kEntries;
        GemvOp* opbuf = reinterpret_cast<GemvOp*>(smem + S::oOpBuf) + 4 + 2 * ow;
        OpFetch fetch;
        fetch.issue(ops, 0, sa.n_ops, lane);
        unsigned oseq = 0;                                               // finishing units so far
        int uncounted = 0, phase = -1;                                   // row pairs of this phase that are written
        auto count = [&] {                                               // all of them are: the last of the warps to say so counts them
            if (uncounted > 0 && phase >= 0) {
                __syncwarp();
                if (lane == 0) {
                    fence_cta();                                     // this warp's y before its count
                    if (atomicAdd(const_cast<unsigned*>(&finished[phase & 3]), 1u) == kOutputWarps - 1u) {
                        finished[phase & 3] = 0u;
                        fence_gpu();                                 // all four warps' y before the phase counter
                        red_add_relaxed_u64(sa.phase_done + phase, (unsigned long long)uncounted);
                    }
                }
            }
            uncounted = 0;
        };
        bool stop = false;
        for (int oi = 0; oi < sa.n_ops && !stop; oi++) {
            __syncwarp();
            fetch.store(&opbuf[oi & 1], lane);
            __syncwarp();
            fetch.issue(ops, oi + 1, sa.n_ops, lane);                    // travels while this op is processed
            const GemvOp& op = opbuf[oi & 1];
            int lo, hi;
            cta_range(op.n_units, op.rot, cta, grid, lo, hi);
            if (lo >= hi) continue;
            const int n_rp = op.n_rp, n_chunks = op.n_kb;
            if (op.phase != phase) { count(); phase = op.phase; }
            for (int ch = lo / n_rp; ch <= (hi - 1) / n_rp && !stop; ch++) {
                const int rp_lo = max(lo - ch * n_rp, 0), rp_hi = min(hi - ch * n_rp, n_rp);
                for (int rp = rp_lo + (ch + n_chunks - rp_lo % n_chunks) % n_chunks; rp < rp_hi && !stop; rp += n_chunks, oseq++) {
                    const unsigned long long* pt = op.partial + (long long)rp * n_chunks * (32 * BP) + row_in * BP + entry;
                    const unsigned want = (oseq / kMarks + 1u) * kUnitRowTiles;
                    float sum[kEntries];
                    unsigned long long t0 = 0ull;
                    for (unsigned it = 0;; it++) {
                        // this CTA's own unit first (a mark is only a hint when to look: later units use it again)
                        bool ok = marks[oseq % kMarks] >= want;
                        if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
                            for (int i = 0; i < kEntries; i++) sum[i] = 0.f;
                            for (int q0 = 0; q0 < n_chunks; q0 += QS) {
                                unsigned long long w[QS][kEntries];
#pragma unroll
                                for (int j = 0; j < QS; j++) {
#pragma unroll
                                    for (int i = 0; i < kEntries; i++) w[j][i] = (unsigned long long)sa.epoch << 32;       // (+ 0.0)
                                    if (q0 + j < n_chunks) {
                                        if constexpr (kEntries == 2) {
                                            const ulonglong2 t = ld_relaxed_u64x2(pt + (long long)(q0 + j) * (32 * BP));
                                            w[j][0] = t.x; w[j][1] = t.y;
                                        } else w[j][0] = ld_relaxed_u64(pt + (long long)(q0 + j) * (32 * BP));
                                    }
                                }
#pragma unroll
                                for (int j = 0; j < QS; j++)
#pragma unroll
                                    for (int i = 0; i < kEntries; i++) {
                                        ok = ok && (unsigned)(w[j][i] >> 32) == sa.epoch;
                                        sum[i] += __uint_as_float((unsigned)w[j][i]);
                                    }
                                if (!__all_sync(0xffffffffu, ok)) break;
                            }
                            if (__all_sync(0xffffffffu, ok)) break;
                        }
                        // not yet.  Lane 0 decides to leave: the lanes leave together
                        int leave = 0;
                        if (lane == 0) {
                            if (flags[0]) leave = 1;
                            else if ((it & 15u) == 0u) {
                                const unsigned long long now = global_ns();
                                if (it == 0u) t0 = now;
                                else if (now - t0 > sa.wait_ns) { give_up(sa.status, flags); leave = 1; }
                            }
                        }
                        if (__shfl_sync(0xffffffffu, leave, 0)) { stop = true; break; }
                        __nanosleep(20);
                    }
                    if (stop) break;
                    const int row = rp * (kUnitRowTiles * kTileRows) + row_in;
                    __half* y = reinterpret_cast<__half*>(op.y);
                    if (row < op.n_out) {
                        // sums of numbers stay finite: an infinite one comes from an activation that is none, and such a one makes
                        // every output of its batch entry NaN (as the batch-1 kernel does, and fq_gemv promises)
#pragma unroll
                        for (int i = 0; i < kEntries; i++)
                            if (entry + i < op.batch) y[(long long)(entry + i) * op.n_out + row] = __float2half_rn(fmaf(sum[i], 0.f, sum[i]));
                    }
                    uncounted++;
                }
            }
        }
        if (!stop) count();
    } else {
        // ================================================================== consumers
        // Two warps share a unit, each computes one of its two 16-row tiles.
        const int g = lane >> 2, c = lane & 3;
        const int uidx = warp / kWarpsPerUnit;                          // which of the units in flight
        const int tile = warp % kUnitRowTiles;                          // this warp's row tile
        int total = 0;                               // units of this CTA over the whole launch
        if (sa.cta_units) total = sa.cta_units[cta];
        else {
            int lo, hi;
            cta_range(single.n_units, single.rot, cta, grid, lo, hi);
            total = hi - lo;
        }
        bool stop = false;
        int seg_seen = -1;                           // the segment whose activations this warp has seen in place
        const uint32_t desc_a = smem_u32(smem + S::oDesc);
        for (int seq = uidx; seq < total && !stop; seq += kUnitsInFlight) {
            const int place = seq % kPlaces;
            const uint32_t full = bars + 8 * place, empty = bars + 8 * (kPlaces + place);
            if (!mbar_wait(full, (unsigned)(seq / kPlaces) & 1u, sa.wait_ns)) give_up(sa.status, flags);
            if (!__all_sync(0xffffffffu, flags[1] == 0)) { stop = true; break; }      // (the lanes leave together, whatever the clocks of their waits said)
            struct { int ch, rp, seg, variant, oseq, n_chunks;
                     uint32_t blob;
                     unsigned long long* partial; } d;
            {
                const uint32_t ud = desc_a + (uint32_t)(place * (int)sizeof(UnitDesc));
                const uint4 u0 = lds128(ud), u1 = lds128<16>(ud);
                d.ch = (int)u0.x; d.rp = (int)u0.y; d.blob = smem_u32(smem + S::oRing) + u0.z; d.seg = (int)u0.w;
                d.variant = (int)u1.x; d.n_chunks = (int)u1.y;
                d.partial = reinterpret_cast<unsigned long long*>(((unsigned long long)u1.w << 32) | u1.z);
                d.oseq = (int)lds32<32>(ud);
            }
            const int slot = d.seg % kXSlots;
            // sleep on the slot's barrier (a hardware wake-up: this wait is on the critical path of every
            // dependency phase); a warp that is several publications ahead would read a stale parity, so only a barrier that
            // belongs to this segment counts
            if (d.seg != seg_seen) {
                const unsigned xpar = (unsigned)(d.seg / kXSlots) & 1u;
                if (x_ready[slot] != d.seg + 1 && !flags[1]) mbar_wait(xbars + 8 * slot, xpar, sa.wait_ns);
                if (!smem_wait([&] { return x_ready[slot] == d.seg + 1 || flags[1]; }, sa.wait_ns) || (!flags[1] && !mbar_wait(xbars + 8 * slot, xpar, sa.wait_ns)))
                    give_up(sa.status, flags);
                fence_cta();
                seg_seen = d.seg;
            }
            const bool live = __all_sync(0xffffffffu, flags[0] == 0);

            float tot[4] = {0.f, 0.f, 0.f, 0.f};
            const uint32_t xs = smem_u32(smem + S::oX) + (uint32_t)slot * S::kXSlotBytes;
            if constexpr (HIGH)
                if (live && *sa.high_zeros != 0u) blob_take_high_zeros<BP>(d.blob, xs, lane, tile, tot);
            if (live) blob_dispatch<BP>(d.variant, d.blob, xs, lane, tile, tot);
            __syncwarp();
            if (lane == 0) {
                fence_cta();                                     // all lanes' reads of the activations before the count below
                mbar_arrive(empty);                              // the place may be filled again
                atomicSub(const_cast<int*>(&x_pending[slot]), 1);   // one warp fewer needs the activation slot
            }
            if (!live) continue;

            // ---- the row sums: tot[2 r + i] of lane (g, c) belongs to local row tile * 16 + g + 8 r, batch entry 2 c + i.  They are
            // published as tagged words (value, launch tag), fire and forget
            if (2 * c < BP) {
                unsigned long long* pu = d.partial + ((long long)d.rp * d.n_chunks + d.ch) * (32 * BP) + (tile * kTileRows + g) * BP + 2 * c;
                const unsigned long long tag = (unsigned long long)sa.epoch << 32;
                st_relaxed_u64x2(pu, tag | __float_as_uint(tot[0]), tag | __float_as_uint(tot[1]));
                st_relaxed_u64x2(pu + 8 * BP, tag | __float_as_uint(tot[2]), tag | __float_as_uint(tot[3]));
            }
            if (d.oseq >= 0 && lane == 0) atomicAdd(const_cast<unsigned*>(&marks[d.oseq % kMarks]), 1u);
        }
        if (stop) let_copies_land();
    }

    __syncthreads();
    if (threadIdx.x == 0 && sa.n_phases > 0) {
        fence_gpu();
        const unsigned old = atomicAdd(sa.exit_count, 1u);
        if (old == gridDim.x - 1) {                    // last CTA out: counters back to zero
            fence_gpu();
            for (int p = 0; p < sa.n_phases; p++) sa.phase_done[p] = 0ull;
            *sa.exit_count = 0u;
            fence_gpu();
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
    // (a captured launch runs whenever its graph does, and so does a captured call that stores weights: no answer holds for them)
    if (zeros_are_low(ctx) && !ctx->stores_in_graphs && !is_capturing(st))
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
    const long long units = (long long)op.n_rp * op.n_kb;
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
