// Host-side context and the descriptors passed to the kernels.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "../../include/flexq.h"
#include "fq_layout.cuh"

namespace fq {

// One stored variant of a layer.
struct Variant {
    bool present = false;        // resident on the device: kernels may read `store`
    void* store = nullptr;       // blobs: scale/zero words + field arrays (fq_layout.cuh)
    const void* host = nullptr;  // the same bytes in host memory (swap model, fq_host_variant), or null
    bool swap_owned = false;     // `store` was allocated by fq_transition_swap: released when the variant is dropped
};

struct Layer {
    bool registered = false;
    int n_out = 0, k_in = 0, fmt = FQ_FMT_PACKED;
    int active_bits = 0;
    Variant var[9];              // PACKED: index = bits; PLANES: only [8]
};

constexpr int kUnitRowTiles = 2;   // a decode unit covers two 16-row tiles (32 output rows)

// What one decode op needs on the device.
struct GemvOp {
    const uint8_t* store;        // blobs [row_pair][k_blob]
    unsigned long long* partial; // split-K partial sums, one tagged word per (row pair, chunk, row, batch entry)
    int blob_read;               // bytes of every blob that this op reads (all of it, or a nested child's prefix)
    int variant;                 // variant_index(format, bits): selects the specialised inner loop
    int batch;
    const uint16_t* x;           // fp16 [batch][k_in]
    uint16_t* y;                 // fp16 [batch][n_out]
    int blob_stride;             // bytes from one blob to the next (size of the stored variant's blobs)
    int n_fields;
    int n_out, k_in;
    int n_kb;                    // k blobs; batch 2..8: K chunks, of a blob each
    int n_rp;                    // row pairs = units per K chunk
    int chunk_blobs;             // batch 1: k blobs that one stage of the ring holds, at most
    int phase;                   // -1: no ordering
    int n_units;                 // n_kb * n_rp
    int rot;                     // rotation of the CTA blocks for this op (evens out remainders); inline ops: its first strip counter
    int split;                   // batch 1: consumer items per blob: 1 (both 16-row tiles) or 2 (one tile each)
    unsigned blob_cost;          // batch 1: cost of a blob (512 bytes x cost of a byte of the variant)
};

struct StackHeader {
    int n_ops;
    int n_phases;
    long long total_units;
};

struct Ctx {
    int device = 0;
    int sm_count = 0;
    std::vector<Layer> layers;
    // workspace shared by all calls on this context
    char* ws = nullptr;          // device
    size_t ws_bytes = 0;
    bool ws_used = false;        // a launch has used a workspace: a graph may hold its address (asking costs 0.1 us a call)
    std::vector<char*> ws_kept;  // replaced workspaces that graphs may hold (freed with `owned`)
    int* status_dev = nullptr;   // device status word, and behind it the word of high_zeros_word()
    // stack-call staging
    char* stack_dev = nullptr;   // device copy of the op table
    size_t stack_dev_bytes = 0;
    // prefill: dequantised bf16 copy of the layer being multiplied
    char* gemm_ws = nullptr;
    size_t gemm_ws_bytes = 0;
    bool gemm_ws_captured = false;       // a captured graph holds the address of gemm_ws
    size_t gemm_ws_refused = 0;          // size that could not be had, under this configuration
    uint64_t gemm_ws_refused_at = ~0ull;
    int gemm_sliced = 0;                 // calls that did without a larger gemm_ws
    // prefill: everything that wrote stored weights came before a launch on this stream, as of this configuration (see launch_gemm_split)
    cudaStream_t gemm_after_stores_on = nullptr;
    uint64_t gemm_after_stores_at = ~0ull;
    bool stores_in_graphs = false;       // a captured call stores weights: nobody here sees when its graph runs
    char* fused_ws = nullptr;            // prefill: counters, then two fp32 tile slots per SM (part of the allocation of status_dev)
    std::vector<void*> owned;    // device buffers freed by fq_destroy: those of fq_load, workspaces that graphs may hold
    uint64_t config_epoch = 0;
    unsigned stored = 1;         // counts the calls that store weights
    unsigned* note = nullptr;    // host word that the device can write (or null): see zeros_are_low in fq_gemv.cu
    unsigned launch_epoch = 0;   // tag of the split-K partials of the latest decode launch (never 0)
    // the op list that is currently uploaded: every argument word of the call that built it
    std::vector<uint64_t> stack_sig;
    bool stack_valid = false;
    StackHeader stack_hdr{};
    // pinned staging buffers of the op table take turns; an event per buffer marks the end of its last upload
    char* stage_host[2] = {nullptr, nullptr};
    size_t stage_host_bytes[2] = {0, 0};
    cudaEvent_t stage_done[2] = {nullptr, nullptr};
    int stage_next = 0;
    size_t ws_reserved = 0;      // split-K bytes that the registered layers need (each used once per launch)
    unsigned long long wait_limit_ns = 2000000000ull;   // limit of every device-side wait
};

// Device word that is not 0 once a zero point above 1023 has been stored by any call on the context (it is never cleared).
inline unsigned* high_zeros_word(const Ctx* ctx) { return reinterpret_cast<unsigned*>(ctx->status_dev) + 1; }

// Is the work that is enqueued on `st` recorded into a graph?
bool is_capturing(cudaStream_t st);
// Bytes of device workspace for `n_ops` ops whose split-K needs are summed by the caller.
int ensure_workspace(Ctx* ctx, size_t bytes);

// kernels / launchers implemented in the .cu files
int launch_quantize(const float* w, int n_out, int k_in, int bits, uint8_t* codes, uint16_t* scales,
                    uint16_t* zeros, cudaStream_t st);
int launch_pack(const uint8_t* codes, const uint16_t* scales, const uint16_t* zeros, int n_out, int k_in,
                int stored_bits, const FieldList& fl, void* store, unsigned* high_zeros, cudaStream_t st);
// Looks through a stored variant that came from elsewhere (a file, host memory) for what launch_pack notes in high_zeros.
int launch_find_high_zeros(const void* store, int n_out, int k_in, int stored_bits, unsigned* high_zeros, cudaStream_t st);
int launch_export_packed(const void* store, int n_out, int k_in, int bits, const FieldList& fl,
                         uint32_t* out, cudaStream_t st);
int launch_export_planes(const void* store, int n_out, int k_in, int bits, const FieldList& fl,
                         uint32_t* out, cudaStream_t st);
int launch_export_meta(const void* store, int n_out, int k_in, int stored_bits, uint16_t* scales, uint16_t* zeros,
                       cudaStream_t st);

// Checked build (-DFQ_CHECKED): `inside` states that an index a kernel computed lies inside the buffer it is about to
// touch.  When it does not hold, the status word gets FQ_ERR_BOUNDS (the first error wins) and the result is false:
// the caller skips the access and winds the kernel down the way it does after a timeout.  Every lane of the
// warp evaluates the same condition wherever the result steers control flow.  In the normal build the condition
// is not evaluated.
#ifdef FQ_CHECKED
#define FQ_IN_BOUNDS(inside, status_ptr) ((inside) ? true : (atomicCAS((status_ptr), 0, FQ_ERR_BOUNDS), false))
#else
#define FQ_IN_BOUNDS(inside, status_ptr) true
#endif

// SM count of the current device (cached); sizes the grids of the grid-stride kernels that have no context at hand.
int current_sm_count();

int launch_stream_read(const void* src, size_t bytes, unsigned* sink, int sm_count, cudaStream_t st);

size_t gemv_partial_bytes_per_unit(int batch);
int launch_gemv_single(Ctx* ctx, const GemvOp& op, cudaStream_t st);                 // batch 2..8
// parts == nullptr: whole tiles only; else tiles may be shared between CTAs through these slots
int launch_gemm_split(Ctx* ctx, const void* store, int blob_stride, int blob_read, const FieldList& fl, int zero_adjust, int n_out,
                      int k_in, const uint16_t* X, int M, int ldx, uint16_t* Y, int ldy, float* parts, unsigned* arrived,
                      cudaStream_t st);
size_t gemm_split_flag_bytes(int sm_count);
size_t gemm_split_part_bytes(int sm_count);
void gemm_split_plan(const Ctx* ctx, int M, int n_out, int k_in, fq_gemm_plan_report* out);
double gemm_split_us(const Ctx* ctx, int M, int n_out, int k_in);       // estimates of the time of a call
double gemm_two_pass_us(const Ctx* ctx, int M, int n_out, int k_in);
struct CtaWork;
// batch 1, up to kInlineOps ops that depend on nothing in the same call: they travel as kernel parameters
constexpr int kInlineOps = 8;
struct InlineOps { GemvOp op[kInlineOps]; };
int launch_gemv1_inline(Ctx* ctx, const InlineOps& ops, int n_ops, cudaStream_t st);
// table_dev: [GemvOp x n_ops][int phase_total x max(n_phases,1)][uint2 strips x sm_count x n_ops]
int launch_gemv1_stack(Ctx* ctx, const StackHeader& hdr, const char* table_dev, cudaStream_t st);
int gemv1_max_phases();
int gemv1_max_phase_strips();       // strips of a phase that one CTA finishes
int gemv1_max_ops();
int gemv1_max_k();
int gemv1_chunk_blobs(int blob_read_bytes);
uint2 gemv1_pack_range(const CtaWork& w, int n_chunks);
int launch_gemv_static(Ctx* ctx, GemvOp op, size_t partial_bytes, cudaStream_t st);
// table_dev: [GemvOp x n_ops][long long phase_total x max(n_phases,1)][int cta_units x sm_count]
int launch_gemv_stack(Ctx* ctx, const StackHeader& hdr, const char* table_dev, int max_batch, cudaStream_t st);
// Units of an op (n_units units, block rotation rot) that CTA `cta` of `grid` processes: [lo, hi).
void gemv_cta_range(int n_units, int rot, int cta, int grid, int& lo, int& hi);

// ---- how a decode op is dealt to the CTAs of the persistent grid
// The pieces of an op (batch 1: the blobs of its 32-row strips; batch 2..8: K chunks of row pairs) are numbered
// strip-major, u = rp * pieces_per_strip + i, and dealt in contiguous blocks; the block boundaries rotate from
// op to op so that the remainders even out.
FQ_HD void cta_range(int n_units, int rot, int cta, int grid, int& lo, int& hi)
{
    const unsigned c = (unsigned)((cta + grid - rot) % grid);
    lo = (int)((unsigned)n_units * c / (unsigned)grid);              // n_units * grid < 2^31 (checked on the host)
    hi = (int)((unsigned)n_units * (c + 1u) / (unsigned)grid);
}
// The strips a CTA touches: rp_first .. rp_last; only the first may start and only the last may end inside a strip.
struct CtaWork {
    int lo, hi, rp_first, rp_last;
    FQ_HD bool any() const { return hi > lo; }
    // pieces [c0, c1) of strip rp that belong to this CTA
    FQ_HD void chunks(int n_chunks, int rp, int& c0, int& c1) const
    {
        c0 = rp == rp_first ? lo - rp * n_chunks : 0;
        c1 = rp == rp_last ? hi - rp * n_chunks : n_chunks;
    }
    // strips that this CTA finishes (it owns their first piece) and therefore writes to y
    FQ_HD int finishing(int n_chunks) const
    {
        if (!any()) return 0;
        return rp_last - rp_first + 1 - (lo - rp_first * n_chunks > 0 ? 1 : 0);
    }
};

int launch_gemm(Ctx* ctx, const void* store, int blob_stride, const FieldList& fl, int zero_adjust, int n_out, int k_in,
                const uint16_t* X, int M, int ldx, uint16_t* Y, int ldy, void* w_scratch, cudaStream_t st);

}  // namespace fq

struct fq_ctx : fq::Ctx {};
