// darkattn_forward_static: the forward pass for callers that cannot provide (or allocate) a workspace.
//
// Its scratch is a fixed array in the library's own device image. The array is shared by every call
// on a device and keeps whatever the previous call left in it.
#include "common.cuh"

#include <mutex>

namespace darkattn {
namespace {

// Scratch of the static entry point: DARKATTN_STATIC_SCRATCH_BYTES of device memory per GPU context
// that loads the library, resident until the process exits.
static __device__ __align__(256) unsigned char g_static_scratch[DARKATTN_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_setup_lock;
char *g_scratch_addr[kMaxDevices] = {};   // device address of g_static_scratch, per device ordinal

// In host code `g_static_scratch` names a host-side shadow of the symbol, not device memory, so the
// address kernels may use has to be asked for, with the target device current.
darkattn_status_t scratch_for_current_device(char **out)
{
    int dev = -1;
    DARKATTN_CUDA_TRY(cudaGetDevice(&dev), "forward_static: cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) return DARKATTN_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> guard(g_setup_lock);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        DARKATTN_CUDA_TRY(cudaGetSymbolAddress(&p, g_static_scratch), "forward_static: cudaGetSymbolAddress");
        if (!p) return DARKATTN_ERR_CUDA;
        g_scratch_addr[dev] = static_cast<char *>(p);
    }
    *out = g_scratch_addr[dev];
    return DARKATTN_OK;
}

// The plan of one (batch, head) pair of `plan`: what the array has to hold when all pairs at once are too much for it.
void single_pair(const darkattn_plan_s *plan, darkattn_plan_s &one)
{
    one.desc = plan->desc;
    one.path = plan->path;
    one.dims = plan->dims;
    Dims &D = one.dims;
    D.B = D.H = D.BH = D.Hkv = D.G = 1;
    simt_make_layout(&one);
}

// How a plan is run: all pairs at once where their intermediates fit the array, else one pair after the other, else by the FFMA
// kernels, whose intermediates take 4 bytes an element instead of 6 and which read fp32 inputs as they are (long sequences of wide
// queries: 5090 tokens of width 429 take 34 MB for one pair, 8 MB here).
enum Mode { ALL_PAIRS, PAIR_BY_PAIR, FFMA, REFUSED };
Mode choose(const darkattn_plan_s *plan, size_t &bytes)
{
    constexpr size_t room = DARKATTN_STATIC_SCRATCH_BYTES;
    bytes = plan->ffma.fwd_bytes;
    if (plan->ffma_fwd && bytes <= room) return FFMA;
    bytes = plan->simt_fwd.bytes;
    if (bytes <= room) return ALL_PAIRS;
    darkattn_plan_s one;
    single_pair(plan, one);
    bytes = one.simt_fwd.bytes;
    if (bytes <= room) return PAIR_BY_PAIR;
    if (plan->ffma.fwd_bytes > room) return REFUSED;
    bytes = plan->ffma.fwd_bytes;
    return FFMA;
}

}  // namespace
}  // namespace darkattn

using namespace darkattn;

extern "C" size_t darkattn_static_scratch_needed(darkattn_plan_t plan)
{
    if (!plan) return 0;
    size_t bytes = 0;
    choose(plan, bytes);
    return bytes;
}

extern "C" darkattn_status_t darkattn_forward_static(darkattn_plan_t plan, const void *Q, const void *K,
                                                     const void *V, const void *M, const void *W, void *O,
                                                     void *cuda_stream)
{
    if (!plan || !Q || !K || !V || !M || !W || !O) return DARKATTN_ERR_INVALID_ARG;
    const void *ptrs[6] = {Q, K, V, M, W, O};
    for (const void *p : ptrs)
        if (reinterpret_cast<uintptr_t>(p) & 15u) return DARKATTN_ERR_INVALID_ARG;
    // size check first: it needs no GPU, so a refusal never touches the device
    size_t bytes = 0;
    const Mode mode = choose(plan, bytes);
    if (mode == REFUSED) return DARKATTN_ERR_WORKSPACE;
    char *scratch = nullptr;
    darkattn_status_t s = scratch_for_current_device(&scratch);
    if (s != DARKATTN_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // the array still holds the previous call's data: the first kernel clears the status word and the per-feature maxima,
    // every other region is written by this call before it is read
    if (mode == ALL_PAIRS) return simt_forward(plan, Q, K, V, M, W, O, nullptr, scratch, st);
    if (mode == FFMA) return ffma_forward(plan, Q, K, V, M, W, O, scratch, st);
    // pair by pair (heads are independent of one another)
    darkattn_plan_s one;
    single_pair(plan, one);
    const Dims &D = plan->dims;
    const size_t es = D.bf16 ? 2 : 4;
    auto at = [&](const void *p, size_t elements) { return static_cast<const void *>(static_cast<const char *>(p) + elements * es); };
    for (int bh = 0; bh < D.BH && s == DARKATTN_OK; ++bh) {
        const size_t h = bh % D.H, kv = (size_t)(bh / D.H) * D.Hkv + h / D.G, N = D.N;
        s = simt_forward(&one, at(Q, bh * N * D.d), at(K, kv * N * D.d), at(V, kv * N * D.dv), at(M, h * D.r * D.d),
                         at(W, D.w_per_head ? h * D.m * D.r : 0), const_cast<void *>(at(O, bh * N * D.dv)), nullptr, scratch, st);
    }
    return s;
}
