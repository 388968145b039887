// noalloc.cu -- sl_step_noalloc: one step of the fast double-float kernel
// that performs no device allocation at all.
//
// Why: sl_step builds field tables and allocates its per-step constant
// buffers the first time it needs them (cudaMalloc), which synchronises the
// device and can fail when a host framework's caching allocator already owns
// the memory.  Code that steps a mesh from inside such an application's loop,
// from a callback that must not synchronise, or under a fixed device-memory
// budget reserved up front cannot allocate per step.
//
// The step reads the caller's doubles and writes doubles itself, so it needs
// no value scratch, and a single problem's constants are kernel parameters.
// Only a batch's constants have a home here: kNoAllocMaxProblems records (18
// KiB) in a static device array, held by every GPU that loads this library
// until the process exits, written from the parameters of a small kernel.
// Calls with several problems share it, so such calls that overlap on the GPU
// -- two streams, or two meshes stepped concurrently -- race on it and must be
// serialised by the caller.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "sl_internal.h"
#include "step_fast.cuh"
#include "step_common.cuh"

namespace sl {
namespace {

constexpr int64_t kNoAllocMaxNodes = SL_NOALLOC_MAX_NODES;
constexpr int32_t kNoAllocMaxProblems = SL_NOALLOC_MAX_PROBLEMS;
constexpr int kMaxDevices = 64;

// File-scope scratch.  In host code the name is only a stand-in for the device
// symbol; its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) FastProb g_noalloc_probs[kNoAllocMaxProblems];

FastProb *g_scratch[kMaxDevices];
std::mutex g_scratch_mutex;

// Device address of the records on the current device, looked up once per
// device (the first call on a device does it).
sl_status scratch_for(int dev, FastProb *&out)
{
    if (dev < 0 || dev >= kMaxDevices) return fail(SL_E_STATE, "sl_step_noalloc: device ordinal out of range");
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch[dev]) {
        void *pp = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&pp, g_noalloc_probs);
        if (e != cudaSuccess)
            return fail(SL_E_CUDA, std::string("sl_step_noalloc: cudaGetSymbolAddress(constants): ") + cudaGetErrorString(e));
        g_scratch[dev] = (FastProb *)pp;
    }
    out = g_scratch[dev];
    return SL_OK;
}

// Node tables of trigonometric fields must already match these problems
// (building them would allocate).
bool tables_ready(const sl_mesh *m, const sl_problem *probs)
{
    bool need1 = false, need2 = false;
    const std::vector<double> key = field_table_key(m->n_problems, probs, need1, need2);
    if (!need1) return true;
    if (!m->d.g1 || (need2 && !m->d.g2)) return false;
    return key == m->table_key;
}

}  // namespace
}  // namespace sl

using namespace sl;

extern "C" sl_status sl_step_noalloc(sl_mesh *m, const sl_problem *probs, int64_t n, const double *v_in,
                                     double *v_out, void *stream)
{
    if (!m || !probs || !v_in || !v_out) return fail(SL_E_ARG, "sl_step_noalloc: NULL argument");
    if ((const void *)v_in == (const void *)v_out) return fail(SL_E_ARG, "sl_step_noalloc: v_in and v_out must not alias");
    if (n < 0) return fail(SL_E_ARG, "sl_step_noalloc: n must be >= 0");
    if (m->precision != SL_FP64) return fail(SL_E_ARG, "sl_step_noalloc: FP64 meshes only");
    if (m->opt_strategy == 3)
        return fail(SL_E_STATE, "sl_step_noalloc: strategy (c) needs one launch per tree level (use sl_step)");
    if (m->N > kNoAllocMaxNodes)
        return fail(SL_E_ARG, "sl_step_noalloc: the mesh has " + std::to_string(m->N) + " nodes; sl_step_noalloc takes at most " +
                                  std::to_string(kNoAllocMaxNodes) + " (use sl_step)");
    if (m->n_problems > kNoAllocMaxProblems)
        return fail(SL_E_ARG, "sl_step_noalloc: at most " + std::to_string(kNoAllocMaxProblems) + " problems");
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(SL_E_CUDA, std::string("sl_step_noalloc: cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev != m->device) return fail(SL_E_STATE, "sl_step_noalloc: the current device is not the mesh's device");
    if (!tables_ready(m, probs))
        return fail(SL_E_STATE, "sl_step_noalloc: the node tables of these fields are not built; call sl_step or sl_run "
                                "once with the same problems first (that call allocates them)");
    FastProb *records = nullptr;
    sl_status st = scratch_for(dev, records);
    if (st != SL_OK) return st;

    FastProb host[kNoAllocMaxProblems];
    for (int32_t p = 0; p < m->n_problems; ++p) {
        st = fast_constants_one(m, probs[p], n, p, host[p]);
        if (st != SL_OK) return st;
    }
    cudaStream_t s = (cudaStream_t)stream;
    if (m->n_problems > 1) launch_put_constants(host, m->n_problems, records, s);

    // The fused kernel in the launch configuration sl_step would take for this
    // step (SL_OPT_KERNEL = 1 and SL_OPT_SPLIT do not apply here).
    FastArgs a;
    fast_args_for(m, records, v_in, v_out, nullptr, host, a);
    a.io = kIoIn | kIoOut;
    launch_fast_df(a, m->opt_stats != 0, false, m->t0_initial ? first_config(m) : later_config(m), s);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(SL_E_CUDA, std::string("sl_step_noalloc: launch: ") + cudaGetErrorString(e));
    m->stepped = true;
    m->t0_initial = false;
    return SL_OK;
}
