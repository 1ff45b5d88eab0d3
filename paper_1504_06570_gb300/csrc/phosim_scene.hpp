// Host-side scene object behind the phosim C ABI.
#pragma once

#include <array>
#include <vector>

#include "phosim_device.cuh"
#include "photon_ds.cuh"

// One trace call's launch sequence as a CUDA graph: kernels ([chief rays, trace], or chief rays, then per chunk of
// the two-kernel path the entry, optics and bundle stages, then the moment-stripe sum) and the counter resets
// between chunks, one node each in launch order.  Built once for a sequence's shape and replayed with each
// call's kernel parameters and launch shapes.
struct TraceGraph {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    std::vector<const void*> func;              // per node: the kernel, or null for a memset
    std::vector<void*> memset_dst;              // per node: the memset's destination (null for a kernel)
    std::vector<size_t> memset_bytes;
    std::vector<std::array<int, 2>> after;      // per node: the nodes it follows (-1: none)
    std::vector<cudaGraphNode_t> node;
};

struct phosim_scene {
    phosim::TraceParams base;       // scalars and device table pointers; per-call fields filled by a trace
    int precision = PHOSIM_PLAIN_FP64;
    int device = 0;                 // the CUDA device current at creation; every call must run with it current
    bool optics_loaded = false, seds_loaded = false;
    int sm_count = 0;
    int host_atomics = 0;           // whether the GPU's atomics on host memory are native
    int threads = 256;
    int tile_photons = 0;           // 0 = chosen per call from the workload
    int n_sed = 0;
    int sersic_tables = 0;
    // host copy of the loaded optics (for the adjoint)
    std::vector<phosim_surface> surfaces;
    // device memory owned by the scene
    std::vector<void*> table_mem;   // sensor tables
    std::vector<void*> optics_mem;  // coating tables
    std::vector<void*> screen_mem;  // gradient screens
    std::vector<void*> sed_mem;
    std::vector<void*> sersic_mem;
    std::vector<void*> hf_mem;      // high-frequency kick quantiles
    // per-call scratch, grown on demand
    phosim::DSource* d_src = nullptr;           // the sources, with the tile prefix behind them
    size_t cap_src = 0;
    void* d_src_s = nullptr;                    // the sources' double-single constants (phosim::SourceS, n_src)
    unsigned long long* d_prefix = nullptr;     // in d_src's memory, behind cap_src sources
    unsigned long long* d_counters = nullptr;   // [0] tile counter, [1..9] counters
    uint32_t* d_stage = nullptr;                // staging image for host image pointers
    uint32_t* d_delta = nullptr;                // a short exposure's counts before they are added to a pinned image
    size_t cap_delta = 0;
    bool delta_clean = false;                   // all zeroes (no call has left counts behind)
    phosim::DSState* d_state = nullptr;         // entrance-plane states of the two-kernel double-single path
    size_t cap_state = 0;
    phosim::DSHit* d_hits = nullptr;            // detector hits of its bundle rays
    size_t cap_hits = 0;
    void* d_ghost = nullptr;                    // rays turned round by coatings: two rounds, their bins and their order
    size_t cap_ghost = 0;
    phosim::GhostRound* d_rounds = nullptr;     // the rounds' counts
    double* d_mom_stripes = nullptr;            // its striped per-source moment accumulators
    size_t cap_mom_stripes = 0;
    size_t cap_stage = 0;
    cudaStream_t last_stream = nullptr;
    // adjoint: Zernike monomial table (owned with the optics) and per-call scratch
    double* d_zmono = nullptr;
    double* d_grad_scratch = nullptr;           // seeds + gradient accumulators
    size_t cap_grad = 0;
    double* d_mom_scratch = nullptr;
    size_t cap_mom = 0;
    // CUDA graphs of the trace launch (PHOSIM_GRAPH), one per precision, captured on a private stream
    TraceGraph graphs[3];
    cudaStream_t capture_stream = nullptr;
    // resident blocks an SM of the trace's kernels for a block size (asked of the driver once)
    struct { int mode = -1, threads = 0, walk = 0, trace = 0, optics = 0, members = 0, listed = 0; } occupancy;
    // the last FP64 call's photon batches: whether they are all there (one chunk), for the adjoint that follows it
    phosim::PhotonBatch* d_batches = nullptr;
    size_t cap_batches = 0;
    bool batches_whole = false;
    // the adjoint's tape (BatchList): asked for while phosim_grad runs its forward pass, and whether that pass wrote it
    double* d_tape = nullptr;
    size_t cap_tape = 0;
    unsigned long long tape_batches = 0, tape_stride = 0;
    int tape_first = 0;
    bool tape_wanted = false, tape_written = false;
    uint32_t last_tile = 0;                     // the last call's photons per tile
    uint64_t last_tiles = 0;                    // and its tiles
    // per-kernel timing (phosim_set_stage_timing): an event pair per launch of the last call, with the
    // kernel kind (0 call preparation and chief, 1 one-kernel trace, 2 entry stage, 3 optics stage)
    bool stage_timing = false;
    std::vector<cudaEvent_t> timing_events;
    std::vector<int> timing_kind;
    int timing_used = 0;
};

namespace phosim {
// mode: the scene's precision (PHOSIM_PLAIN_FP64, PHOSIM_MIXED, PHOSIM_MIXED_DS)
// beside: start beside the chief rays, the kernel before on the stream
cudaError_t launch_trace(const TraceParams& P, int mode, int blocks, int threads, cudaStream_t st, bool beside = false);
// the FP64 paths with the dynamic transmission test: batches of photons that go on, then a warp a batch
cudaError_t launch_batches(const TraceParams& P, const BatchList& L, int mode, int blocks, int threads, cudaStream_t st);
cudaError_t launch_trace_batches(const TraceParams& P, const BatchList& L, int mode, int blocks, cudaStream_t st, bool beside);
const void* batch_kernel_ptr(int mode);
const void* trace_batch_kernel_ptr(int mode);
cudaError_t batch_occupancy(int mode, int threads, int* batch_per_sm, int* trace_per_sm);
cudaError_t launch_call_prep(const CallPrep& C, cudaStream_t st);
unsigned call_prep_blocks(const CallPrep& C);
const void* call_prep_kernel_ptr();
constexpr int kPrepThreads = 128;
cudaError_t launch_chief_rays(const TraceParams& P, DSource* sources, int n_src, double* moments, cudaStream_t st);
cudaError_t trace_occupancy(int mode, int threads, int* blocks_per_sm);
const void* trace_kernel_ptr(int mode);
const void* chief_kernel_ptr();
// threads per block of the chief rays: one warp, so that few sources spread over many SMs (a warp alone on an SM
// is bound by its FP64 latencies, four share the SM's FP64 pipe: 300 sources 53 us with 128 threads a block)
constexpr int kChiefThreads = 32;
size_t source_s_bytes();                       // sizeof(SourceS), which the host code does not see
// the two-kernel double-single path (PHOSIM_MIXED_DS in phosim_trace)
cudaError_t launch_ds_entry(const TraceParams& P, const DSStage& S, int blocks, int threads, cudaStream_t st, bool beside);
cudaError_t launch_ds_optics(const TraceParams& P, const DSStage& S, int kind, int blocks, int threads, cudaStream_t st, bool beside);
// a launch that starts beside the kernel before it on the stream as soon as that one lets it or ends; what the kernel
// reads of the one before must follow its own wait_for_previous
template <class... Params, class... Args>
cudaError_t launch_beside(void (*kernel)(Params...), int blocks, int threads, cudaStream_t st, const Args&... args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config = {};
    config.gridDim = dim3((unsigned)blocks);
    config.blockDim = dim3((unsigned)threads);
    config.stream = st;
    config.attrs = &attr;
    config.numAttrs = 1;
    return cudaLaunchKernelEx(&config, kernel, args...);
}
cudaError_t launch_ds_members(const TraceParams& P, const DSStage& S, int blocks, int threads, cudaStream_t st);
const void* ds_members_kernel_ptr();
cudaError_t ds_stage_occupancy(int kind, int threads, int* entry_per_sm, int* optics_per_sm, int* members_per_sm);
const void* ds_entry_kernel_ptr();
// kind of walk (WalkKind): 0 no reflecting coating, 1 forward with ghosts leaving, 2 a round of ghosts, 3 as 0 for simple surfaces
const void* ds_optics_kernel_ptr(int kind);
const void* ghost_order_kernel_ptr();
cudaError_t launch_ghost_order(const DSStage& S, int blocks, cudaStream_t st);
const void* moment_stripes_kernel_ptr();
cudaError_t launch_moment_stripes(const TraceParams& P, cudaStream_t st);
int ds_optics_threads(int threads);      // the optics stage's block size for a schedule's block size
void free_all(std::vector<void*>& v);
// PHOSIM_OK when the current device is the scene's, INVALID_ARGUMENT otherwise (CUDA on a failed query)
phosim_status check_scene_device(const phosim_scene* sc);
// PHOSIM_OK when p is null or device / managed memory usable on `device`; INVALID_ARGUMENT for host memory,
// unregistered pointers and another device's memory
phosim_status check_device_buffer(const void* p, int device);
// count, centroid and central second moments of n_src sources from their PHOSIM_MOMENT_WORDS additive sums
void derive_moments(const double* sums, int n_src, double* out6);
}  // namespace phosim
