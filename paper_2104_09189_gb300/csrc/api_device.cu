// api_device.cu -- entry points of sl.h that touch the device: upload,
// sl_step, sl_run (CUDA graph of the time loop), sl_run_host, T^0 import /
// export, deferred status, counters, renumbering and destruction.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "sl_internal.h"
#include "step_fast.cuh"
#include "step_kernels.cuh"

namespace sl {

// device status words followed by the counters
constexpr size_t kReportBytes = sizeof(uint32_t) * kStatusWords + sizeof(unsigned long long) * kStatCounters;

#define SL_CUDA(call)                                                                        \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return fail(e_ == cudaErrorMemoryAllocation ? SL_E_NOMEM : SL_E_CUDA,            \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                 \
    } while (0)

// (hi, lo) float pair of a double: hi = fl32(v), lo = fl32(v - hi)
static void split_df(double v, float2 &o)
{
    const float h = (float)v;
    o.x = h;
    o.y = (float)(v - (double)h);
}

FastArgs make_fast_args(const sl_mesh *m, const FastProb *fp, const void *vin, void *vout, const sl_debug *dbg,
                        const FastProb *fh = nullptr);

// A coordinate in [0,1] as g + l: g = v rounded to the grid of 2^-24 (a float,
// exactly), l = fl32(v - g), |l| <= 2^-25, |v - g - l| <= 2^-49.  Differences
// of the g parts of two coordinates are exact in float (multiples of 2^-24
// below 1 in magnitude), which is what the certified test of the fast kernel
// builds on.
static void split_grid(double v, float2 &o)
{
    const double g = std::nearbyint(v * 16777216.0) / 16777216.0;
    o.x = (float)g;
    o.y = (float)(v - g);
}

void pack_fast_constants(int32_t kind, const double c[6], FastProb &f)
{
    for (int k = 0; k < 6; ++k) split_df(c[k], f.c[k]);
    if (kind == SL_FIELD_ROTATION && c[1] >= 0.0 && c[1] <= 1.0 && c[2] >= 0.0 && c[2] <= 1.0) {
        split_grid(c[1], f.c[1]);
        split_grid(c[2], f.c[2]);
        f.flags |= kFastCentreGrid;
    }
}

int32_t default_walk_cap(const sl_mesh *m)
{
    int32_t M = 1;
    for (int32_t c : m->cells) M = c > M ? c : M;
    int32_t cap = 4 * (M + 1);
    return cap < 64 ? 64 : cap;
}

void release_l2_window(sl_mesh *m)
{
    if (!m->l2_limit_set) return;
    cudaCtxResetPersistingL2Cache();
    cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, m->l2_limit_prev);
    m->l2_limit_set = false;
}

// Every kernel node of a recorded graph marks the walk records as
// persisting in L2 (SL_OPT_L2_WINDOW).
static sl_status apply_l2_window(sl_mesh *m, cudaGraph_t graph)
{
    int maxwin = 0, maxpers = 0;
    SL_CUDA(cudaDeviceGetAttribute(&maxwin, cudaDevAttrMaxAccessPolicyWindowSize, m->device));
    SL_CUDA(cudaDeviceGetAttribute(&maxpers, cudaDevAttrMaxPersistingL2CacheSize, m->device));
    void *base = m->d.he8 ? m->d.he8 : m->d.he;
    const size_t bytes = (m->d.he8 ? sizeof(uint2) : sizeof(float4)) * 3 * (size_t)m->Nt;
    const size_t win = bytes < (size_t)maxwin ? bytes : (size_t)maxwin;
    if (!base || win == 0 || maxpers <= 0) return SL_OK;
    if (!m->l2_limit_set) {
        SL_CUDA(cudaDeviceGetLimit(&m->l2_limit_prev, cudaLimitPersistingL2CacheSize));
        SL_CUDA(cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, (size_t)maxpers));
        m->l2_limit_set = true;
    }
    cudaKernelNodeAttrValue val;
    std::memset(&val, 0, sizeof(val));
    val.accessPolicyWindow.base_ptr = base;
    val.accessPolicyWindow.num_bytes = win;
    val.accessPolicyWindow.hitRatio = (float)maxpers >= (float)win ? 1.0f : (float)maxpers / (float)win;
    val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    size_t n = 0;
    SL_CUDA(cudaGraphGetNodes(graph, nullptr, &n));
    std::vector<cudaGraphNode_t> nodes(n);
    SL_CUDA(cudaGraphGetNodes(graph, nodes.data(), &n));
    for (cudaGraphNode_t node : nodes) {
        cudaGraphNodeType type;
        SL_CUDA(cudaGraphNodeGetType(node, &type));
        if (type == cudaGraphNodeTypeKernel)
            SL_CUDA(cudaGraphKernelNodeSetAttribute(node, cudaKernelNodeAttributeAccessPolicyWindow, &val));
    }
    return SL_OK;
}

void free_device(sl_mesh *m)
{
    release_l2_window(m);
    DeviceMesh &d = m->d;
    void *ptrs[] = {d.xy, d.tv[0], d.tv[1], d.tv[2], d.tn[0], d.tn[1], d.tn[2], d.t0, d.t0_init, d.extras, d.t0v, d.node_off, d.chunk_prob,
                    d.status, d.probs, d.fprobs, d.xyq, d.xyh, d.g1, d.g2, d.tparams, d.dfa, d.dfb, d.he, d.he8, d.weights, d.grid_t0v, d.tree_order, d.tree_parent, d.queue, d.queue_count,
                    m->host_v, m->host_v2};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    d = DeviceMesh();
    m->host_v = m->host_v2 = nullptr;
    if (m->graph.exec) cudaGraphExecDestroy((cudaGraphExec_t)m->graph.exec);
    m->graph = GraphCache();
    if (m->report) cudaFreeHost(m->report);
    m->report = nullptr;
    if (m->capture_stream) cudaStreamDestroy((cudaStream_t)m->capture_stream);
    m->capture_stream = nullptr;
}

// The longest edge of the mesh as |dx| + |dy| in the hop coordinates h of
// the double-float kernel (floats: the differences and sums are exact in
// double), rounded up to a float: the bound of the runs of lean hops
// (lean_walk).
static float hop_edge_bound(const sl_mesh *m, const std::vector<float2> &h)
{
    double L = 0.0;
    for (int32_t p = 0; p < m->n_problems; ++p) {
        const int64_t n0 = m->node_off[p];
        for (int64_t j = m->tri_off[p]; j < m->tri_off[p + 1]; ++j)
            for (int k = 0; k < 3; ++k) {
                const float2 a = h[n0 + m->tri[3 * j + k]], b = h[n0 + m->tri[3 * j + (k + 1) % 3]];
                const double d = std::fabs((double)a.x - (double)b.x) + std::fabs((double)a.y - (double)b.y);
                if (d > L) L = d;
            }
    }
    const float f = (float)L;
    return (double)f >= L ? f : std::nextafter(f, __builtin_inff());
}

static void alloc_extras(sl_mesh *m);
static sl_status build_jump_table(sl_mesh *m);

// Copy the host arrays (current numbering) to the device, converting local
// indices to global ones.
static sl_status upload_arrays(sl_mesh *m)
{
    DeviceMesh &d = m->d;
    const int64_t N = m->N, Nt = m->Nt;
    m->table_key.clear();   // the field node tables follow the numbering: rebuilt at the next step
    if (m->precision == SL_FP64) {
        SL_CUDA(cudaMemcpy(d.xy, m->xy.data(), sizeof(double) * 2 * N, cudaMemcpyHostToDevice));
        // (grid, remainder) float pairs of the coordinates for the double-float
        // kernel (split_grid); their grid parts are also the hop coordinates
        std::vector<float4> q(N);
        for (int64_t i = 0; i < N; ++i) {
            float2 a, b;
            split_grid(m->xy[2 * i], a);
            split_grid(m->xy[2 * i + 1], b);
            q[i] = make_float4(a.x, b.x, a.y, b.y);
        }
        SL_CUDA(cudaMemcpy(d.xyq, q.data(), sizeof(float4) * N, cudaMemcpyHostToDevice));
        std::vector<float2> hx(N);
        for (int64_t i = 0; i < N; ++i) hx[i] = make_float2(q[i].x, q[i].y);
        SL_CUDA(cudaMemcpy(d.xyh, hx.data(), sizeof(float2) * N, cudaMemcpyHostToDevice));
        m->hop_L = hop_edge_bound(m, hx);
    } else {
        std::vector<float> f(2 * N);
        for (int64_t q = 0; q < 2 * N; ++q) f[q] = (float)m->xy[q];
        SL_CUDA(cudaMemcpy(d.xy, f.data(), sizeof(float) * 2 * N, cudaMemcpyHostToDevice));
    }
    std::vector<int32_t> col(Nt);
    for (int k = 0; k < 3; ++k) {
        for (int32_t p = 0; p < m->n_problems; ++p)
            for (int64_t j = m->tri_off[p]; j < m->tri_off[p + 1]; ++j)
                col[j] = m->tri[3 * j + k] + (int32_t)m->node_off[p];
        SL_CUDA(cudaMemcpy(d.tv[k], col.data(), sizeof(int32_t) * Nt, cudaMemcpyHostToDevice));
        for (int32_t p = 0; p < m->n_problems; ++p)
            for (int64_t j = m->tri_off[p]; j < m->tri_off[p + 1]; ++j) {
                const int32_t nb = m->nbr[3 * j + k];
                if (nb >= 0) {
                    col[j] = nb + (int32_t)m->tri_off[p];
                } else {
                    // boundary edge opposite vertex k: the side of the square it lies on
                    const int64_t n0 = m->node_off[p];
                    const int64_t va = n0 + m->tri[3 * j + (k + 1) % 3], vb = n0 + m->tri[3 * j + (k + 2) % 3];
                    const double xa = m->xy[2 * va], ya = m->xy[2 * va + 1], xb = m->xy[2 * vb], yb = m->xy[2 * vb + 1];
                    int side = 3;
                    if (xa == 0.0 && xb == 0.0) side = 0;
                    else if (xa == 1.0 && xb == 1.0) side = 1;
                    else if (ya == 0.0 && yb == 0.0) side = 2;
                    col[j] = -1 - side;
                }
            }
        SL_CUDA(cudaMemcpy(d.tn[k], col.data(), sizeof(int32_t) * Nt, cudaMemcpyHostToDevice));
    }
    // half-edge walk records of the fast kernels
    sl_status st = build_walk_records(m);
    if (st != SL_OK) return st;
    SL_CUDA(cudaMemcpy(d.t0, m->t0.data(), sizeof(int32_t) * N, cudaMemcpyHostToDevice));
    SL_CUDA(cudaMemcpy(d.t0_init, m->t0_init.data(), sizeof(int32_t) * N, cudaMemcpyHostToDevice));
    SL_CUDA(cudaMemcpy(d.node_off, m->node_off.data(), sizeof(int64_t) * (m->n_problems + 1), cudaMemcpyHostToDevice));
    if (m->n_problems > 1) {
        // the problems of each chunk of 128 nodes (chunk_problem), one sweep
        const int64_t nc = (N + 127) >> 7;
        std::vector<int2> cp(nc);
        int32_t p = 0;
        for (int64_t c = 0; c < nc; ++c) {
            const int64_t first = c << 7, last = std::min(N, first + 128) - 1;
            while (m->node_off[p + 1] <= first) ++p;
            int32_t q = p;
            while (m->node_off[q + 1] <= last) ++q;
            cp[c] = make_int2(p, q);
        }
        if (!d.chunk_prob) SL_CUDA(cudaMalloc(&d.chunk_prob, sizeof(int2) * nc));
        SL_CUDA(cudaMemcpy(d.chunk_prob, cp.data(), sizeof(int2) * nc, cudaMemcpyHostToDevice));
    }
    alloc_extras(m);
    if (d.extras) {
        launch_build_tri(d.tv, Nt, (int4 *)d.tri, 0);
        SL_CUDA(cudaGetLastError());
        st = build_jump_table(m);
        if (st != SL_OK) return st;
    }
    if (d.pair_tri) {
        launch_pair_tri(make_fast_args(m, nullptr, nullptr, nullptr, nullptr), d.pair_tri, 0);
        SL_CUDA(cudaGetLastError());
    }
    launch_fill_t0v(d.t0, d.tv[0], d.tv[1], d.tv[2], (int4 *)d.t0v, N, 0);
    SL_CUDA(cudaGetLastError());
    SL_CUDA(cudaDeviceSynchronize());
    return SL_OK;
}

static size_t line_up(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

// Bytes of the weights of a run's steady fields (emit_weights).
static size_t weight_bytes(const sl_mesh *m)
{
    return line_up(sizeof(int4) * (size_t)m->N) +
           line_up((m->precision == SL_FP64 ? sizeof(float4) : sizeof(float)) * (size_t)m->N);
}

static void place_weights(sl_mesh *m, void *base)
{
    m->d.wq = base;
    m->d.wt = (char *)base + line_up(sizeof(int4) * (size_t)m->N);
}

// Up to this many nodes a handle has room for its weights from the start: an
// allocation takes 50 to 100 us whatever its size, which a first run of a few
// steps does not earn back (the first 10 steps of a rotation without weights,
// with weights allocated in the run, and with room from the start: 50 k nodes
// 110, 191 and 89 us, 200 k 126, 263 and 102, 1 M 272, 351 and 201; 2.3 M nodes in
// FP32, 4 steps, still 442 allocating them where locating at every step took
// 361).  Larger meshes allocate it in the first run that uses it (ensure_weights).
constexpr int64_t kEagerWeights = 1 << 22;

// Arrays that only make the steps faster: allocated where kSpareBytes per node
// stay free beside them, what a caller's buffers and the handle's later ones
// (tables 32, values 32, queue 4) may still need.  NULL otherwise, and the handle
// does without.
#ifndef SL_SPARE_BYTES      // a build that never has room for them sets more than any device has
#define SL_SPARE_BYTES 128
#endif
constexpr size_t kSpareBytes = SL_SPARE_BYTES;
static void *optional_malloc(const sl_mesh *m, size_t bytes)
{
    size_t avail = 0, total = 0;
    void *p = nullptr;
    if (cudaMemGetInfo(&avail, &total) == cudaSuccess && avail >= bytes + kSpareBytes * (size_t)m->N &&
        cudaMalloc(&p, bytes) == cudaSuccess)
        return p;
    cudaGetLastError();
    return nullptr;
}

// The problems' grids of the jump table, about one cell per four nodes, and the
// arrays that follow from the mesh, in one allocation.  Without them (d.tri is
// NULL) every step is the full node step.
static void alloc_extras(sl_mesh *m)
{
    DeviceMesh &d = m->d;
    const int32_t np = m->n_problems;
    if (d.extras) return;           // a renumbering: the same sizes
    m->jump_g.resize(np);
    m->jump_off.resize(np + 1);
    int64_t cells = 0;
    for (int32_t p = 0; p < np; ++p) {
        const double n = (double)(m->node_off[p + 1] - m->node_off[p]);
        const int32_t g = std::max(1, (int32_t)(0.5 * std::sqrt(n)));
        m->jump_g[p] = g;
        m->jump_off[p] = (int32_t)cells;
        cells += (int64_t)g * g;
    }
    m->jump_off[np] = (int32_t)cells;     // at most a quarter of the nodes: an int32
    // (on 256 bytes each: a warp's 512 bytes of weights from the middle of a line
    // are a line more, 1.5 % of a run)
    const size_t tri = line_up(sizeof(int4) * (size_t)m->Nt), jump = line_up(sizeof(int4) * (size_t)cells),
                 pair = m->precision == SL_FP64 ? sizeof(int32_t) * (size_t)m->N : 0,
                 w = m->N <= kEagerWeights ? weight_bytes(m) : 0;
    d.extras = w ? optional_malloc(m, tri + jump + pair + w) : nullptr;
    const bool weights = d.extras != nullptr;
    if (!d.extras) d.extras = optional_malloc(m, tri + jump + pair);
    if (!d.extras) return;
    char *p = (char *)d.extras;
    d.tri = p;
    d.jump = p + tri;
    if (pair) d.pair_tri = (int32_t *)(p + tri + jump + (weights ? w : 0));
    if (weights) place_weights(m, p + tri + jump);
}

// The jump table of every problem, built on the device (its scratch is the
// start-state cache, 16 bytes per node, filled afterwards: 2 bytes per node of
// seeds and two integers per problem of at least 3 nodes).
static sl_status build_jump_table(sl_mesh *m)
{
    DeviceMesh &d = m->d;
    const int32_t np = m->n_problems;
    const int64_t cells = m->jump_off[np];
    uint32_t *seed = (uint32_t *)d.t0v;
    int32_t *off = (int32_t *)(seed + 2 * (size_t)cells);
    std::vector<int32_t> hg(m->jump_off);
    hg.insert(hg.end(), m->jump_g.begin(), m->jump_g.end());
    SL_CUDA(cudaMemcpy(off, hg.data(), sizeof(int32_t) * hg.size(), cudaMemcpyHostToDevice));
    JumpBuildArgs a;
    for (int k = 0; k < 3; ++k) {
        a.tv[k] = d.tv[k];
        a.tn[k] = d.tn[k];
    }
    a.xyc = m->precision == SL_FP64 ? (const float2 *)d.xyh : (const float2 *)d.xy;
    a.t0_init = d.t0_init;
    a.node_off = d.node_off;
    a.off = off;
    a.gp = off + np + 1;
    a.nprob = np;
    a.cells = (int32_t)cells;
    a.max_g = *std::max_element(m->jump_g.begin(), m->jump_g.end());
    a.N = m->N;
    a.seed[0] = seed;
    a.seed[1] = a.seed[0] + cells;
    a.jump = (int4 *)d.jump;
    launch_build_jump(a, 0);
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

// Compact 8-byte records for FP64 meshes whose triangles are narrow enough
// (k_build_he8 reports an overflow otherwise), else 16-byte records; only
// one form is kept on the device.
sl_status build_walk_records(sl_mesh *m)
{
    DeviceMesh &d = m->d;
    const int64_t Nt = m->Nt;
    if (m->precision == SL_FP64 && m->opt_records == 1) {
        if (!d.he8) SL_CUDA(cudaMalloc(&d.he8, sizeof(uint2) * 3 * (Nt > 0 ? Nt : 1)));
        uint32_t *overflow = d.status + 1;   // a reserved status word, zero again afterwards
        SL_CUDA(cudaMemset(overflow, 0, sizeof(uint32_t)));
        launch_build_he8(d.tv, d.tn, (const float2 *)d.xyh, Nt, (uint2 *)d.he8, overflow, 0);
        SL_CUDA(cudaGetLastError());
        uint32_t h = 0;
        SL_CUDA(cudaMemcpy(&h, overflow, sizeof(h), cudaMemcpyDeviceToHost));
        SL_CUDA(cudaMemset(overflow, 0, sizeof(uint32_t)));
        if (!h) {
            if (d.he) cudaFree(d.he);
            d.he = nullptr;
            m->graph.valid = false;
            return SL_OK;
        }
    }
    if (d.he8) cudaFree(d.he8);
    d.he8 = nullptr;
    if (!d.he) SL_CUDA(cudaMalloc(&d.he, sizeof(float4) * 3 * (Nt > 0 ? Nt : 1)));
    launch_build_he(d.tv, d.tn, m->precision == SL_FP64 ? (const float2 *)d.xyh : (const float2 *)d.xy, Nt,
                    (float4 *)d.he, 0);
    SL_CUDA(cudaGetLastError());
    SL_CUDA(cudaDeviceSynchronize());
    m->graph.valid = false;
    return SL_OK;
}

sl_status upload(sl_mesh *m)
{
    SL_CUDA(cudaGetDevice(&m->device));
    SL_CUDA(cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, m->device));
    DeviceMesh &d = m->d;
    const int64_t N = m->N, Nt = m->Nt;
    const size_t cs = m->precision == SL_FP64 ? 2 * sizeof(double) : 2 * sizeof(float);
    SL_CUDA(cudaMalloc(&d.xy, cs * N));
    if (m->precision == SL_FP64) SL_CUDA(cudaMalloc(&d.xyq, sizeof(float4) * N));
    for (int k = 0; k < 3; ++k) {
        SL_CUDA(cudaMalloc(&d.tv[k], sizeof(int32_t) * Nt));
        SL_CUDA(cudaMalloc(&d.tn[k], sizeof(int32_t) * Nt));
    }
    SL_CUDA(cudaMalloc(&d.t0, sizeof(int32_t) * N));
    if (m->precision == SL_FP64) SL_CUDA(cudaMalloc(&d.xyh, sizeof(float2) * N));
    SL_CUDA(cudaMalloc(&d.t0_init, sizeof(int32_t) * N));
    SL_CUDA(cudaMalloc(&d.t0v, sizeof(int4) * N));
    SL_CUDA(cudaMalloc(&d.node_off, sizeof(int64_t) * (m->n_problems + 1)));
    // status words and counters in one block, read back in one copy
    SL_CUDA(cudaMalloc(&d.status, kReportBytes));
    SL_CUDA(cudaMemset(d.status, 0, kReportBytes));
    d.stats = (unsigned long long *)(d.status + kStatusWords);
    SL_CUDA(cudaMallocHost(&m->report, kReportBytes));
    return upload_arrays(m);
}

// Host-side evaluation of the time factors of each field at t_{n+1}.
// The constants of step n (t_{n+1} = (n+1) dt) of one problem, validated.
static sl_status fill_step_one(const sl_problem &q, int64_t n, int32_t p, ProbStep &s)
{
    const double pi = 3.14159265358979323846;
    if (q.kind < SL_FIELD_ZERO || q.kind > SL_FIELD_PAPER)
        return fail(SL_E_ARG, "problem " + std::to_string(p) + ": unknown field kind");
    if (!(std::isfinite(q.dt) && q.dt > 0.0))
        return fail(SL_E_ARG, "problem " + std::to_string(p) + ": dt must be finite and > 0");
    for (int k = 0; k < SL_NPARAMS; ++k)
        if (!std::isfinite(q.p[k])) return fail(SL_E_ARG, "problem " + std::to_string(p) + ": non-finite field parameter");
    if (q.kind == SL_FIELD_SWIRL && q.p[0] == 0.0) return fail(SL_E_ARG, "swirl period p0 must be nonzero");
    std::memset(&s, 0, sizeof(s));
    s.kind = q.kind;
    s.dt = q.dt;
    s.t = (double)(n + 1) * q.dt;
    std::memcpy(s.p, q.p, sizeof(s.p));
    if (q.kind == SL_FIELD_SWIRL) s.c[0] = std::cos(pi * s.t / q.p[0]);
    if (q.kind == SL_FIELD_FOURIER8)
        for (int mm = 0; mm < 8; ++mm) s.c[mm] = q.p[4 * mm + 2] * std::cos(2.0 * pi * s.t + q.p[4 * mm + 3]);
    if (q.kind == SL_FIELD_PAPER) s.c[0] = q.p[1] * s.t;
    return SL_OK;
}

static sl_status fill_step(const sl_mesh *m, const sl_problem *probs, int64_t n, ProbStep *out)
{
    for (int32_t p = 0; p < m->n_problems; ++p) {
        const sl_status st = fill_step_one(probs[p], n, p, out[p]);
        if (st != SL_OK) return st;
    }
    return SL_OK;
}

static sl_status ensure_probs(sl_mesh *m, size_t bytes)
{
    if (m->d.probs_bytes >= bytes) return SL_OK;
    cudaFree(m->d.probs);
    m->d.probs = nullptr;
    m->d.probs_bytes = 0;
    SL_CUDA(cudaMalloc(&m->d.probs, bytes));
    m->d.probs_bytes = bytes;
    return SL_OK;
}

static StepArgs make_args(const sl_mesh *m, const ProbStep *probs_dev, const void *vin, void *vout,
                          const sl_debug *dbg)
{
    StepArgs a;
    std::memset(&a, 0, sizeof(a));
    a.xy = m->d.xy;
    for (int k = 0; k < 3; ++k) {
        a.tv[k] = m->d.tv[k];
        a.tn[k] = m->d.tn[k];
    }
    a.t0v = (int4 *)m->d.t0v;
    a.vin = vin;
    a.vout = vout;
    a.probs = probs_dev;
    a.node_off = m->d.node_off;
    a.nprob = m->n_problems;
    a.walk_cap = m->opt_walk_cap > 0 ? m->opt_walk_cap : default_walk_cap(m);
    a.N = m->N;
    a.status = m->d.status;
    a.stats = m->d.stats;
    if (dbg) a.dbg = *dbg;
    a.keep_t0 = m->opt_strategy == 1 || m->opt_strategy == 2;   // (a), direct: T^0 kept
    a.exclude = m->opt_outside == 1;
    a.grid_M = m->opt_strategy == 2 ? m->grid_M : 0;
    a.grid_t0v = (const int4 *)m->d.grid_t0v;
    a.count = m->N;     // every node; the level launches of strategy (c) narrow it
    return a;
}

void fast_args_for(const sl_mesh *m, const FastProb *fp, const void *vin, void *vout, const sl_debug *dbg,
                   const FastProb *fh, FastArgs &out)
{
    out = make_fast_args(m, fp, vin, vout, dbg, fh);
}

// fp: the step's constants on the device; fh: the same on the host (or
// NULL), copied into the kernel parameters for a single problem.
FastArgs make_fast_args(const sl_mesh *m, const FastProb *fp, const void *vin, void *vout, const sl_debug *dbg,
                        const FastProb *fh)
{
    FastArgs a;
    std::memset(&a, 0, sizeof(a));
    a.xyq = (const float4 *)m->d.xyq;
    a.xyh = (const float2 *)m->d.xyh;
    a.xyf = m->precision == SL_FP32 ? (const float2 *)m->d.xy : nullptr;
    a.xyd = m->precision == SL_FP64 ? (const double2 *)m->d.xy : nullptr;
    for (int k = 0; k < 3; ++k) {
        a.tv[k] = m->d.tv[k];
        a.tn[k] = m->d.tn[k];
    }
    a.tri = (const int4 *)m->d.tri;
    a.he = (const float4 *)m->d.he;
    a.he8 = (const uint2 *)m->d.he8;
    // strategy (b) with the default hop cap may start a far walk at the jump
    // table; the other strategies and a cap set by the caller are about the
    // walk itself
    a.jump = m->opt_strategy == 0 && m->opt_walk_cap == 0 ? (const int4 *)m->d.jump : nullptr;
    a.t0_init = m->d.t0_init;
    a.pair_tri = m->d.pair_tri;
    a.initial = m->t0_initial;
    a.wq = (int4 *)m->d.wq;
    if (m->precision == SL_FP64) a.wt = (float4 *)m->d.wt;
    else a.wt2 = (float *)m->d.wt;
    a.t0v = (int4 *)m->d.t0v;
    a.vin = vin;
    a.vout = vout;
    if (m->precision == SL_FP64) {
        a.g1 = (const float4 *)m->d.g1;
        a.g2 = (const float4 *)m->d.g2;
    } else {
        a.g1f = (const float2 *)m->d.g1;
        a.g2f = (const float2 *)m->d.g2;
    }
    a.probs = fp;
    if (fh && m->n_problems == 1) {
        a.prob0 = fh[0];
        a.single = 1;
    }
    a.node_off = m->d.node_off;
    a.chunk_prob = (const int2 *)m->d.chunk_prob;
    a.nprob = m->n_problems;
    a.walk_cap = m->opt_walk_cap > 0 ? m->opt_walk_cap : default_walk_cap(m);
    a.lean_moves = m->opt_walk_cap > 0 ? 0 : 8;
    a.sms = m->sms;
    a.N = m->N;
    a.status = m->d.status;
    a.stats = m->d.stats;
    if (dbg) a.dbg = *dbg;
    a.keep_t0 = m->opt_strategy == 1 || m->opt_strategy == 2;   // (a), direct: T^0 kept
    a.exclude = m->opt_outside == 1;
    a.grid_M = m->opt_strategy == 2 ? m->grid_M : 0;
    a.grid_t0v = (const int4 *)m->d.grid_t0v;
    a.count = m->N;     // every node; the level launches of strategy (c) narrow it
    a.hop_L = m->hop_L;
    // G^2; +inf when the FP64 value path is off (no gradient exceeds it)
    a.steep_g2 = m->precision == SL_FP64 && m->opt_precise > 0
                     ? (float)((double)m->opt_precise * (double)m->opt_precise)
                     : __builtin_inff();
    return a;
}

// The fast kernels are the default; SL_OPT_KERNEL = 1 selects the plain FP64 one.
static bool use_fast(const sl_mesh *m) { return m->opt_kernel != 1 || m->precision == SL_FP32; }

// Per-step constants of the fast kernels (see FastProb), of one problem.
static void fill_fast_one(const sl_mesh *m, int32_t p, const ProbStep &q, FastProb &f)
{
    const double pi = 3.14159265358979323846;
    std::memset(&f, 0, sizeof(f));
    f.kind = q.kind;
    f.jump_g = m->jump_g[p];
    f.jump_off = m->jump_off[p];
    double c[6] = {0, 0, 0, 0, 0, 0};
    switch (q.kind) {
    case SL_FIELD_AFFINE:
        f.dc = make_float2((float)(q.dt * q.p[3] * q.dt), (float)(q.dt * q.p[7] * q.dt));
        c[0] = q.dt * (q.p[0] + q.p[3] * q.t);
        c[1] = q.dt * q.p[1];
        c[2] = q.dt * q.p[2];
        c[3] = q.dt * (q.p[4] + q.p[7] * q.t);
        c[4] = q.dt * q.p[5];
        c[5] = q.dt * q.p[6];
        break;
    case SL_FIELD_ROTATION:
        c[0] = q.dt * q.p[0];
        c[1] = q.p[1];
        c[2] = q.p[2];
        break;
    case SL_FIELD_SWIRL:
        c[0] = q.dt * q.c[0];
        f.dc.x = (float)(c[0] - q.dt * std::cos(pi * (q.t - q.dt) / q.p[0]));
        break;
    case SL_FIELD_PAPER:
    case SL_FIELD_FOURIER8: {
        const double w = q.kind == SL_FIELD_PAPER ? q.p[1] : 2.0 * pi;
        c[0] = q.dt * std::cos(w * q.t);
        c[1] = q.dt * std::sin(w * q.t);
        f.dc = make_float2((float)(c[0] - q.dt * std::cos(w * (q.t - q.dt))),
                           (float)(c[1] - q.dt * std::sin(w * (q.t - q.dt))));
        break;
    }
    default: break;
    }
    pack_fast_constants(q.kind, c, f);
}

static void fill_fast(const sl_mesh *m, const ProbStep *ps, FastProb *out)
{
    for (int32_t p = 0; p < m->n_problems; ++p) fill_fast_one(m, p, ps[p], out[p]);
}

sl_status fast_constants_one(const sl_mesh *m, const sl_problem &q, int64_t n, int32_t p, FastProb &f)
{
    ProbStep s;
    const sl_status st = fill_step_one(q, n, p, s);
    if (st != SL_OK) return st;
    fill_fast_one(m, p, s, f);
    return SL_OK;
}

std::vector<double> field_table_key(int32_t n_problems, const sl_problem *probs, bool &need1, bool &need2)
{
    need1 = need2 = false;
    std::vector<double> key((size_t)n_problems * kTableKeyStride);
    for (int32_t p = 0; p < n_problems; ++p) {
        const int kind = probs[p].kind;
        need1 |= kind == SL_FIELD_SWIRL || kind == SL_FIELD_PAPER || kind == SL_FIELD_FOURIER8;
        need2 |= kind == SL_FIELD_PAPER || kind == SL_FIELD_FOURIER8;
        key[kTableKeyStride * p] = kind;
        for (int k = 0; k < SL_NPARAMS; ++k) key[kTableKeyStride * p + 1 + k] = probs[p].p[k];
    }
    return key;
}

// Node tables of the trigonometric fields, rebuilt when the fields change.
static sl_status ensure_tables(sl_mesh *m, const sl_problem *probs, cudaStream_t s)
{
    bool need1 = false, need2 = false;
    const std::vector<double> key = field_table_key(m->n_problems, probs, need1, need2);
    if (!need1) return SL_OK;
    if (key == m->table_key && m->d.g1 && (!need2 || m->d.g2)) return SL_OK;
    // FP64 meshes keep (hi, lo) pairs, FP32 meshes the values rounded to float
    const size_t tsz = m->precision == SL_FP64 ? sizeof(float4) : sizeof(float2);
    if (!m->d.g1) SL_CUDA(cudaMalloc(&m->d.g1, tsz * m->N));
    if (need2 && !m->d.g2) SL_CUDA(cudaMalloc(&m->d.g2, tsz * m->N));
    if (!m->d.tparams) SL_CUDA(cudaMalloc(&m->d.tparams, sizeof(double) * key.size()));
    SL_CUDA(cudaStreamSynchronize(s));
    SL_CUDA(cudaMemcpy(m->d.tparams, key.data(), sizeof(double) * key.size(), cudaMemcpyHostToDevice));
    FieldTableArgs ta;
    ta.xyd = m->precision == SL_FP64 ? (const double2 *)m->d.xy : nullptr;
    ta.xyf = m->precision == SL_FP32 ? (const float2 *)m->d.xy : nullptr;
    ta.node_off = m->d.node_off;
    ta.nprob = m->n_problems;
    ta.N = m->N;
    ta.params = m->d.tparams;
    ta.g1 = ta.g2 = nullptr;
    ta.g1f = ta.g2f = nullptr;
    if (m->precision == SL_FP64) {
        ta.g1 = (float4 *)m->d.g1;
        ta.g2 = (float4 *)m->d.g2;
    } else {
        ta.g1f = (float2 *)m->d.g1;
        ta.g2f = (float2 *)m->d.g2;
    }
    launch_field_tables(ta, s);
    SL_CUDA(cudaGetLastError());
    SL_CUDA(cudaStreamSynchronize(s));
    m->table_key = key;
    m->graph.valid = false;
    return SL_OK;
}

// Strategy (c): one launch per spanning-tree level, in level order, so that
// every node starts from its parent's triangle of the same step.
template <class Args, class Launch>
static void for_levels(const sl_mesh *m, const Args &a0, Launch launch)
{
    if (m->opt_strategy != 3) {
        launch(a0);
        return;
    }
    Args a = a0;
    a.order = m->d.tree_order;
    a.parent = m->d.tree_parent;
    const std::vector<int64_t> &off = m->tree_level_off;
    for (size_t k = 0; k + 1 < off.size(); ++k) {
        a.base = off[k];
        a.count = off[k + 1] - off[k];
        launch(a);
    }
}

static sl_status launch_step(const sl_mesh *m, const StepArgs &a, bool debug, cudaStream_t s)
{
    if (m->precision != SL_FP64) return fail(SL_E_STATE, "the plain kernel is FP64 only");
    for_levels(m, a, [&](const StepArgs &x) { launch_plain_f64(x, m->opt_stats != 0, debug, m->opt_block, s); });
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

// Queue scratch of split steps (allocated before any recording).
static sl_status ensure_queue(sl_mesh *m)
{
    if (m->opt_split && m->precision == SL_FP64 && !m->d.queue) {
        SL_CUDA(cudaMalloc(&m->d.queue, sizeof(int32_t) * (m->N > 0 ? m->N : 1)));
        SL_CUDA(cudaMalloc(&m->d.queue_count, 2 * sizeof(uint32_t)));   // alternating, see launch_fast
    }
    return SL_OK;
}

static bool split_step(const sl_mesh *m, bool initial)
{
    return m->precision == SL_FP64 && m->opt_split && !initial && m->opt_strategy == 0 && !m->opt_outside;
}

// initial: the step starts from the initial start triangles (never split).
// split_seq: the number of split steps already enqueued in this sequence of
// steps (NULL: a sequence of one).  Split steps use the two queue counters
// in turn; the first one of a sequence zeroes its counter, and each settle
// pass zeroes the counter of the next step, so the steps between need no
// memset.  after_step: the last launch on the stream is a step kernel of
// the same sequence, so with SL_OPT_PDL this step's kernels are launched
// with programmatic serialization (launch_step_kernel); the experiment
// options keep plain launches.
static sl_status launch_fast(sl_mesh *m, const FastArgs &a, bool debug, int config, bool initial, cudaStream_t s,
                             int32_t *split_seq = nullptr, bool after_step = false)
{
    const bool pdl = m->opt_pdl && !(a.exclude || a.order || a.grid_M > 0 || a.keep_t0);
    if (split_step(m, initial)) {
        if (!m->d.queue) return fail(SL_E_STATE, "split step without its queue scratch");
        const int32_t q = split_seq ? *split_seq : 0;
        FastArgs x = a;
        x.queue = m->d.queue;
        x.queue_count = m->d.queue_count + (q & 1);
        x.queue_next = split_seq ? m->d.queue_count + ((q + 1) & 1) : nullptr;
        // the first split step of a sequence zeroes its counter with a memset
        x.pdl = pdl && after_step && q > 0;
        launch_settle_df(x, m->opt_stats != 0, debug, q == 0, s);
        x.pdl = pdl;     // the finish pass follows its settle pass
        launch_finish_df(x, m->opt_stats != 0, debug, m->sms, s);
        if (split_seq) ++*split_seq;
    } else {
        FastArgs y = a;
        y.pdl = pdl && after_step;
        for_levels(m, y, [&](const FastArgs &x) {
            if (m->precision == SL_FP64) launch_fast_df(x, m->opt_stats != 0, debug, config, s);
            else launch_fast_f32(x, m->opt_stats != 0, debug, config, s);
        });
    }
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

// Step k of a run of steady fields: the first one in the fused kernel (which
// stores the weights), the others apply them.
static sl_status launch_steady(sl_mesh *m, const FastArgs &a, int config, int32_t k, cudaStream_t s)
{
    FastArgs x = a;
    x.pdl = m->opt_pdl && k > 0;
    if (m->precision == SL_FP64) {
        if (k == 0) launch_fast_df(x, false, false, config, s);
        else launch_apply_df(x, s);
    } else {
        if (k == 0) launch_fast_f32(x, false, false, config, s);
        else launch_apply_f32(x, s);
    }
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

// Steps and runs that launch kernels on the caller's stream themselves are not
// for a stream that is being captured: the caller's graph would keep the
// address of the step's constants, which later calls rewrite or free, and the
// node tables, which follow the field.  (sl_run's own graphs end when these
// change; sl_step_noalloc owns what it hands to its kernels.)
static sl_status check_not_capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e == cudaSuccess && st == cudaStreamCaptureStatusNone) return SL_OK;
    cudaGetLastError();     // (an error: the legacy stream while another one is captured)
    return fail(SL_E_CUDA, "the stream is being captured (use sl_step_noalloc)");
}

static sl_status check_device(const sl_mesh *m)
{
    int dev = -1;
    SL_CUDA(cudaGetDevice(&dev));
    if (dev != m->device) return fail(SL_E_STATE, "the current device is not the device the mesh was created on");
    return SL_OK;
}

static void fill_stats(const unsigned long long *c, sl_stats *out)
{
    out->node_updates = c[0];
    out->walk_moves = c[1];
    out->max_moves = c[2];
    out->exact_tests = c[3];
    out->filter2_tests = c[4];
    out->clipped = c[5];
    out->fallbacks = c[6];
    out->walk_limit = c[7];
    out->excluded = c[8];
}

// The status words and the counters, one copy and one wait (page-locked, so
// that the copy is a queued one); the status words are cleared when one is set.
static sl_status read_report(sl_mesh *m, sl_stats *out, cudaStream_t s)
{
    SL_CUDA(cudaMemcpyAsync(m->report, m->d.status, kReportBytes, cudaMemcpyDeviceToHost, s));
    SL_CUDA(cudaStreamSynchronize(s));
    uint32_t st[kStatusWords];
    unsigned long long c[kStatCounters];
    std::memcpy(st, m->report, sizeof(st));
    std::memcpy(c, (const char *)m->report + sizeof(st), sizeof(c));
    if (st[0]) {
        SL_CUDA(cudaMemsetAsync(m->d.status, 0, sizeof(st), s));
        SL_CUDA(cudaStreamSynchronize(s));
    }
    if (out) fill_stats(c, out);
    if (st[0] & (1u << SL_E_WALK_LIMIT)) return fail(SL_E_WALK_LIMIT, "a barycentric walk exceeded its hop cap and its fallback");
    if (st[0] & (1u << SL_E_ARG))
        return fail(SL_E_ARG, "a coordinate fell outside the exact orientation predicate's range");
    return SL_OK;
}

static sl_status ensure_fprobs(sl_mesh *m, size_t bytes)
{
    if (m->d.fprobs_bytes >= bytes) return SL_OK;
    cudaFree(m->d.fprobs);
    m->d.fprobs = nullptr;
    m->d.fprobs_bytes = 0;
    SL_CUDA(cudaMalloc(&m->d.fprobs, bytes));
    m->d.fprobs_bytes = bytes;
    return SL_OK;
}

// Room for the weights (kEagerWeights); false: there is none, and the steps
// locate every time.
static bool ensure_weights(sl_mesh *m)
{
    if (m->d.wq) return true;
    if (m->d.tri) m->d.weights = optional_malloc(m, weight_bytes(m));
    if (!m->d.weights) return false;
    place_weights(m, m->d.weights);
    return true;
}

// Steady fields of a run (emit_weights): problems whose constants are the same
// at every one of the n_steps steps store their weights at the first step and
// use them at the others.  Marks them in fh and returns whether all of them
// are.  Storing costs about half a later step's time once and saves a third of
// one per step, so runs of fewer than 4 steps go without; so do the counting
// variants, the paper's experiments, split steps of a batch that is only
// partly steady, and a device without room for the weights.  The settle pass has
// no weights, and SL_OPT_SPLIT is the caller's choice or the tuner's, which weighs
// steps that locate: split against fused with weights, 1.2 M nodes, 50 steps, a
// third of them steady: 1.25 and 1.30 ms where feet move a third of a cell, 1.77 and
// 1.63 at 3 cells, 4.02 and 2.39 at 20; three quarters steady 1.20 and 0.87 at a
// third of a cell.  The tuner chose fused in each.
constexpr int32_t kSteadySteps = 4;
static bool mark_steady(sl_mesh *m, int32_t n_steps, bool split_rest, std::vector<FastProb> &fh)
{
    if (n_steps < kSteadySteps || m->opt_stats || m->opt_strategy != 0 || m->opt_outside) return false;
    const int32_t np = m->n_problems;
    std::vector<uint8_t> steady(np, 1);
    bool any = false, all = true;
    for (int32_t p = 0; p < np; ++p) {
        for (int32_t k = 1; k < n_steps && steady[p]; ++k)
            steady[p] = std::memcmp(&fh[(size_t)k * np + p], &fh[p], sizeof(FastProb)) == 0;
        any |= steady[p] != 0;
        all &= steady[p] != 0;
    }
    if (!any || (split_rest && !all)) return false;
    if (!ensure_weights(m)) return false;
    for (int32_t p = 0; p < np; ++p)
        for (int32_t k = 0; k < n_steps && steady[p]; ++k) fh[(size_t)k * np + p].flags |= k == 0 ? kFastEmit : kFastUse;
    return all;
}

// weights: steady fields may keep them (mark_steady); the tuners time steps that
// locate, which differ in what they choose between
static sl_status run_steps(sl_mesh *m, const sl_problem *probs, int64_t n0, int32_t n_steps, void *v, void *v2,
                           int32_t use_graph, cudaStream_t s, bool weights = true)
{
    const bool fast = use_fast(m);
    // strategy (c) launches once per spanning-tree level and step: far too
    // many nodes for a graph on large meshes, so it always runs eagerly
    if (m->opt_strategy == 3) use_graph = 0;
    const size_t per = sizeof(ProbStep) * m->n_problems;
    const size_t fper = sizeof(FastProb) * m->n_problems;
    const size_t elem = m->precision == SL_FP64 ? sizeof(double) : sizeof(float);
    GraphCache &g = m->graph;
    std::vector<uint8_t> key((const uint8_t *)probs, (const uint8_t *)(probs + m->n_problems));
    const bool first_initial = m->t0_initial;
    bool same = use_graph && g.valid && g.n0 == n0 && g.n_steps == n_steps && g.v == v && g.v_scratch == v2 &&
                g.probs == key && g.kernel == m->opt_kernel && g.stats == m->opt_stats && g.config == m->opt_config &&
                g.config_first == m->opt_config_first && g.t0_initial == first_initial && g.split == m->opt_split;
    // the steps' constants, which a replayed graph already holds
    std::vector<ProbStep> host;
    auto fill_host = [&]() -> sl_status {
        host.resize((size_t)m->n_problems * (size_t)n_steps);
        for (int32_t k = 0; k < n_steps; ++k) {
            sl_status st = fill_step(m, probs, n0 + k, host.data() + (size_t)k * m->n_problems);
            if (st != SL_OK) return st;
        }
        return SL_OK;
    };
    sl_status hs = same && g.exec ? SL_OK : fill_host();
    if (hs == SL_OK && fast) {
        hs = ensure_tables(m, probs, s);     // (a rebuilt table ends the recorded graph)
        if (hs == SL_OK) hs = ensure_queue(m);
    }
    if (hs == SL_OK && same && !g.valid) {
        same = false;
        if (host.empty()) hs = fill_host();
    }
    if (hs != SL_OK) return hs;
    const bool reuse = same && g.exec;
    // A run seen for the first time is launched step by step: recording and
    // instantiating a graph takes longer than launching its kernels (10 steps on
    // 91 k nodes: 218 us per run recorded, 116 us launched, readback of the status included), and a program that
    // reads its solution between runs repeats none of them.  The second run with
    // the same arguments records.  (The L2 window is an attribute of a graph's
    // nodes.)
    const bool record = use_graph && !reuse && (same || (m->opt_l2 && fast));
    auto remember = [&]() {
        g.valid = true;
        g.n0 = n0;
        g.n_steps = n_steps;
        g.v = v;
        g.v_scratch = v2;
        g.probs = key;
        g.kernel = m->opt_kernel;
        g.stats = m->opt_stats;
        g.config = m->opt_config;
        g.config_first = m->opt_config_first;
        g.t0_initial = first_initial;
        g.split = m->opt_split;
    };
    auto config_of = [&](int32_t k) { return (k == 0 && first_initial) ? first_config(m) : later_config(m); };
    std::vector<FastProb> fh;   // the fast kernels' constants, host copy (filled when recording)
    bool all_steady = false;
    if (!reuse) {
        const sl_status cst = check_not_capturing(s);
        if (cst != SL_OK) return cst;
        if (fast) {
            fh.resize((size_t)m->n_problems * (size_t)n_steps);
            for (int32_t k = 0; k < n_steps; ++k)
                fill_fast(m, host.data() + (size_t)k * m->n_problems, fh.data() + (size_t)k * m->n_problems);
            all_steady = weights && mark_steady(m, n_steps, split_step(m, false), fh);
            if (m->n_problems > 1) {
                // (a single problem's constants are kernel parameters.)  A
                // synchronous copy: a graph recorded below may replay them
                // later.  The one before reads the same buffer, rewritten here
                // and perhaps replaced.
                g.valid = false;
                SL_CUDA(cudaStreamSynchronize(s));
                sl_status st = ensure_fprobs(m, fper * n_steps);
                if (st != SL_OK) return st;
                SL_CUDA(cudaMemcpy(m->d.fprobs, fh.data(), fper * n_steps, cudaMemcpyHostToDevice));
            }
        } else {
            g.valid = false;     // likewise
            SL_CUDA(cudaStreamSynchronize(s));
            sl_status st = ensure_probs(m, per * n_steps);
            if (st != SL_OK) return st;
            SL_CUDA(cudaMemcpy(m->d.probs, host.data(), per * n_steps, cudaMemcpyHostToDevice));
        }
    }
    auto enqueue = [&](cudaStream_t q) -> sl_status {
        if (fast && m->precision == SL_FP64) {
            // values travel as (hi, lo) float pairs in the two caller buffers; a
            // first step reads the doubles itself and a last one writes them
            // where the number of steps puts them on the right buffers (the
            // passes of a split step take pairs only)
            const bool can_in = !split_step(m, first_initial) || all_steady,
                       can_out = !split_step(m, n_steps == 1 && first_initial) || all_steady;
            const bool in = can_in && (n_steps % 2 == 0 || !can_out), out = can_out && in == (n_steps % 2 == 0);
            void *a = v, *b = v2;
            if (!in) {
                launch_to_df((const double *)v, (float2 *)v2, m->N, q);
                a = v2;
                b = v;
            }
            int32_t split_seq = 0;
            for (int32_t k = 0; k < n_steps; ++k) {
                FastArgs args = make_fast_args(m, (const FastProb *)((char *)m->d.fprobs + fper * k), a, b, nullptr,
                                               fh.data() + (size_t)k * m->n_problems);
                args.initial = first_initial && k == 0;
                args.io = (in && k == 0 ? kIoIn : 0) | (out && k == n_steps - 1 ? kIoOut : 0);
                sl_status st = all_steady ? launch_steady(m, args, config_of(k), k, q)
                                          : launch_fast(m, args, false, config_of(k), k == 0 && first_initial, q,
                                                        &split_seq, k > 0);
                if (st != SL_OK) return st;
                void *t = a;
                a = b;
                b = t;
            }
            if (!out) launch_from_df((const float2 *)a, (double *)v, m->N, q);
            SL_CUDA(cudaGetLastError());
            return SL_OK;
        }
        void *a = v, *b = v2;
        int32_t split_seq = 0;
        for (int32_t k = 0; k < n_steps; ++k) {
            sl_status st;
            if (fast) {
                FastArgs args = make_fast_args(m, (const FastProb *)((char *)m->d.fprobs + fper * k), a, b, nullptr,
                                               fh.data() + (size_t)k * m->n_problems);
                args.initial = first_initial && k == 0;
                st = all_steady ? launch_steady(m, args, config_of(k), k, q)
                                : launch_fast(m, args, false, config_of(k), k == 0 && first_initial, q, &split_seq,
                                              k > 0);
            } else {
                StepArgs args = make_args(m, (const ProbStep *)((char *)m->d.probs + per * k), a, b, nullptr);
                st = launch_step(m, args, false, q);
            }
            if (st != SL_OK) return st;
            void *t = a;
            a = b;
            b = t;
        }
        if (a != v) SL_CUDA(cudaMemcpyAsync(v, a, elem * m->N, cudaMemcpyDeviceToDevice, q));
        return SL_OK;
    };
    if (!record && !reuse) {
        if (use_graph) {
            if (g.exec) cudaGraphExecDestroy((cudaGraphExec_t)g.exec);
            g = GraphCache();
            remember();
        }
        return enqueue(s);
    }
    if (!reuse) {
        if (g.exec) cudaGraphExecDestroy((cudaGraphExec_t)g.exec);
        g = GraphCache();
        // Record on a private stream: the caller's stream may be the legacy
        // default stream, which cannot be captured.  Recording executes
        // nothing; the graph is then launched on the caller's stream.
        if (!m->capture_stream) SL_CUDA(cudaStreamCreateWithFlags((cudaStream_t *)&m->capture_stream, cudaStreamNonBlocking));
        cudaStream_t cs = (cudaStream_t)m->capture_stream;
        cudaGraph_t graph;
        SL_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        sl_status st = enqueue(cs);
        cudaError_t ce = cudaStreamEndCapture(cs, &graph);
        if (st != SL_OK) {
            if (ce == cudaSuccess) cudaGraphDestroy(graph);
            return st;
        }
        if (ce != cudaSuccess) return fail(SL_E_CUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(ce));
        if (m->opt_l2 && fast) {
            st = apply_l2_window(m, graph);
            if (st != SL_OK) {
                cudaGraphDestroy(graph);
                return st;
            }
        }
        cudaGraphExec_t exec;
        ce = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (ce != cudaSuccess) return fail(SL_E_CUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(ce));
        remember();
        g.exec = exec;
    }
    SL_CUDA(cudaGraphLaunch((cudaGraphExec_t)g.exec, s));
    return SL_OK;
}

}  // namespace sl

using namespace sl;

extern "C" sl_status sl_step(sl_mesh *m, const sl_problem *probs, int64_t n, const void *v_in, void *v_out,
                             const sl_debug *dbg, void *stream)
{
    if (!m || !probs || !v_in || !v_out) return fail(SL_E_ARG, "sl_step: NULL argument");
    if (v_in == v_out) return fail(SL_E_ARG, "sl_step: v_in and v_out must not alias");
    if (n < 0) return fail(SL_E_ARG, "sl_step: n must be >= 0");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<ProbStep> host(m->n_problems);
    st = fill_step(m, probs, n, host.data());
    if (st == SL_OK) st = check_not_capturing(s);
    if (st != SL_OK) return st;
    const bool debug = dbg && (dbg->feet || dbg->tri || dbg->moves || dbg->flags || dbg->feet_lo);
    if (!use_fast(m)) {
        m->graph.valid = false;   // the per-step buffer is overwritten
        st = ensure_probs(m, sizeof(ProbStep) * m->n_problems);
        if (st != SL_OK) return st;
        SL_CUDA(cudaMemcpyAsync(m->d.probs, host.data(), sizeof(ProbStep) * m->n_problems, cudaMemcpyHostToDevice, s));
        SL_CUDA(cudaStreamSynchronize(s));   // the host staging vector goes out of scope
        StepArgs a = make_args(m, (const ProbStep *)m->d.probs, v_in, v_out, dbg);
        st = launch_step(m, a, debug, s);
        m->stepped = true;
        m->t0_initial = false;
        return st;
    }
    st = ensure_tables(m, probs, s);
    if (st == SL_OK) st = ensure_queue(m);
    if (st != SL_OK) return st;
    std::vector<FastProb> fh(m->n_problems);
    fill_fast(m, host.data(), fh.data());
    if (m->n_problems > 1) {
        // in the parameters of a small kernel, so that no host buffer outlives
        // the call and nothing waits (a single problem's are parameters of the
        // step itself)
        m->graph.valid = false;   // the per-step buffer is overwritten
        st = ensure_fprobs(m, sizeof(FastProb) * m->n_problems);
        if (st != SL_OK) return st;
        launch_put_constants(fh.data(), m->n_problems, (FastProb *)m->d.fprobs, s);
    }
    if (m->precision == SL_FP64 && split_step(m, m->t0_initial)) {
        // double values in and out; a split step works on (hi, lo) float pairs
        if (!m->d.dfa) SL_CUDA(cudaMalloc(&m->d.dfa, sizeof(float2) * m->N));
        if (!m->d.dfb) SL_CUDA(cudaMalloc(&m->d.dfb, sizeof(float2) * m->N));
        launch_to_df((const double *)v_in, (float2 *)m->d.dfa, m->N, s);
        FastArgs a = make_fast_args(m, (const FastProb *)m->d.fprobs, m->d.dfa, m->d.dfb, dbg, fh.data());
        st = launch_fast(m, a, debug, later_config(m), false, s);
        if (st != SL_OK) return st;
        launch_from_df((const float2 *)m->d.dfb, (double *)v_out, m->N, s);
        SL_CUDA(cudaGetLastError());
    } else {
        FastArgs a = make_fast_args(m, (const FastProb *)m->d.fprobs, v_in, v_out, dbg, fh.data());
        if (m->precision == SL_FP64) a.io = kIoIn | kIoOut;
        st = launch_fast(m, a, debug, m->t0_initial ? first_config(m) : later_config(m), m->t0_initial, s);
        if (st != SL_OK) return st;
    }
    m->stepped = true;
    m->t0_initial = false;
    return SL_OK;
}

extern "C" sl_status sl_run(sl_mesh *m, const sl_problem *probs, int64_t n0, int32_t n_steps, void *v,
                            void *v_scratch, int32_t use_graph, sl_stats *stats, void *stream)
{
    if (!m || !probs || !v || !v_scratch) return fail(SL_E_ARG, "sl_run: NULL argument");
    if (v == v_scratch) return fail(SL_E_ARG, "sl_run: v and v_scratch must not alias");
    if (n0 < 0 || n_steps < 0) return fail(SL_E_ARG, "sl_run: n0 and n_steps must be >= 0");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    if (n_steps > 0) {
        st = run_steps(m, probs, n0, n_steps, v, v_scratch, use_graph, s);
        if (st != SL_OK) return st;
        m->stepped = true;
        m->t0_initial = false;
    }
    if (m->opt_async && !stats) return SL_OK;   // status read by sl_mesh_status
    return read_report(m, stats, s);
}

extern "C" sl_status sl_run_host(sl_mesh *m, const sl_problem *probs, int64_t n0, int32_t n_steps, void *v_host,
                                 int32_t use_graph, sl_stats *stats, void *stream)
{
    if (!m || !probs || !v_host) return fail(SL_E_ARG, "sl_run_host: NULL argument");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t bytes = (m->precision == SL_FP64 ? sizeof(double) : sizeof(float)) * m->N;
    if (!m->host_v) {
        SL_CUDA(cudaMalloc(&m->host_v, bytes));
        SL_CUDA(cudaMalloc(&m->host_v2, bytes));
    }
    SL_CUDA(cudaMemcpyAsync(m->host_v, v_host, bytes, cudaMemcpyHostToDevice, s));
    if (n_steps > 0) {
        st = run_steps(m, probs, n0, n_steps, m->host_v, m->host_v2, use_graph, s);
        if (st != SL_OK) return st;
        m->stepped = true;
        m->t0_initial = false;
    }
    SL_CUDA(cudaMemcpyAsync(v_host, m->host_v, bytes, cudaMemcpyDeviceToHost, s));
    return read_report(m, stats, s);
}

extern "C" sl_status sl_mesh_get_t0(const sl_mesh *m, int32_t *t0_dev, void *stream)
{
    if (!m || !t0_dev) return fail(SL_E_ARG, "sl_mesh_get_t0: NULL argument");
    const sl_status st = check_device(m);
    if (st != SL_OK) return st;
    launch_export_t0((const int4 *)m->d.t0v, t0_dev, m->N, (cudaStream_t)stream);
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

extern "C" sl_status sl_mesh_set_t0(sl_mesh *m, const int32_t *t0_dev, void *stream)
{
    if (!m || !t0_dev) return fail(SL_E_ARG, "sl_mesh_set_t0: NULL argument");
    const sl_status st = check_device(m);
    if (st != SL_OK) return st;
    std::vector<int32_t> h(m->N);
    SL_CUDA(cudaMemcpyAsync(h.data(), t0_dev, sizeof(int32_t) * m->N, cudaMemcpyDeviceToHost, (cudaStream_t)stream));
    SL_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
    for (int32_t p = 0; p < m->n_problems; ++p)
        for (int64_t i = m->node_off[p]; i < m->node_off[p + 1]; ++i)
            if (h[i] < m->tri_off[p] || h[i] >= m->tri_off[p + 1])
                return fail(SL_E_ARG, "sl_mesh_set_t0: entry " + std::to_string(i) + " is not a triangle of its problem");
    m->t0_initial = false;
    launch_fill_t0v(t0_dev, m->d.tv[0], m->d.tv[1], m->d.tv[2], (int4 *)m->d.t0v, m->N, (cudaStream_t)stream);
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

extern "C" sl_status sl_mesh_reset_t0(sl_mesh *m, void *stream)
{
    if (!m) return fail(SL_E_ARG, "sl_mesh_reset_t0: mesh is NULL");
    const sl_status st = check_device(m);
    if (st != SL_OK) return st;
    m->t0_initial = true;
    if (m->d.tri)
        launch_reset_t0(m->d.t0_init, (const int4 *)m->d.tri, (int4 *)m->d.t0v, m->N, (cudaStream_t)stream);
    else
        launch_fill_t0v(m->d.t0_init, m->d.tv[0], m->d.tv[1], m->d.tv[2], (int4 *)m->d.t0v, m->N, (cudaStream_t)stream);
    SL_CUDA(cudaGetLastError());
    return SL_OK;
}

// Start states of the structured-grid triangles (direct location, Sec. 4):
// slot 2 (M m + l) + (lower ? 1 : 0) -> (3 t, T[0][t], T[1][t], T[2][t]).
sl_status sl::upload_grid_table(sl_mesh *m, const std::vector<int32_t> &slot_tri)
{
    SL_CUDA(cudaSetDevice(m->device));
    std::vector<int4> h(slot_tri.size());
    for (size_t k = 0; k < slot_tri.size(); ++k) {
        const int32_t t = slot_tri[k];
        h[k] = make_int4(3 * t, m->tri[3 * (size_t)t], m->tri[3 * (size_t)t + 1], m->tri[3 * (size_t)t + 2]);
    }
    if (m->d.grid_t0v) cudaFree(m->d.grid_t0v);
    m->d.grid_t0v = nullptr;
    SL_CUDA(cudaMalloc(&m->d.grid_t0v, sizeof(int4) * h.size()));
    SL_CUDA(cudaMemcpy(m->d.grid_t0v, h.data(), sizeof(int4) * h.size(), cudaMemcpyHostToDevice));
    m->graph.valid = false;
    return SL_OK;
}

// Spanning tree of strategy (c) on the device (node order by level, parents).
sl_status sl::upload_tree(sl_mesh *m, const std::vector<int32_t> &order, const std::vector<int32_t> &parent)
{
    SL_CUDA(cudaSetDevice(m->device));
    if (!m->d.tree_order) SL_CUDA(cudaMalloc(&m->d.tree_order, sizeof(int32_t) * m->N));
    if (!m->d.tree_parent) SL_CUDA(cudaMalloc(&m->d.tree_parent, sizeof(int32_t) * m->N));
    SL_CUDA(cudaMemcpy(m->d.tree_order, order.data(), sizeof(int32_t) * m->N, cudaMemcpyHostToDevice));
    SL_CUDA(cudaMemcpy(m->d.tree_parent, parent.data(), sizeof(int32_t) * m->N, cudaMemcpyHostToDevice));
    m->graph.valid = false;
    return SL_OK;
}

// T^0 back to the initial incident triangles, synchronously (option changes).
sl_status sl::reset_t0_sync(sl_mesh *m)
{
    SL_CUDA(cudaSetDevice(m->device));
    sl_status st = sl_mesh_reset_t0(m, nullptr);
    if (st != SL_OK) return st;
    SL_CUDA(cudaDeviceSynchronize());
    return SL_OK;
}

extern "C" sl_status sl_mesh_status(sl_mesh *m, void *stream)
{
    if (!m) return fail(SL_E_ARG, "sl_mesh_status: mesh is NULL");
    return read_report(m, nullptr, (cudaStream_t)stream);
}

extern "C" sl_status sl_mesh_stats(sl_mesh *m, sl_stats *out, int32_t reset, void *stream)
{
    if (!m) return fail(SL_E_ARG, "sl_mesh_stats: mesh is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    unsigned long long c[kStatCounters];
    SL_CUDA(cudaMemcpyAsync(c, m->d.stats, sizeof(c), cudaMemcpyDeviceToHost, s));
    SL_CUDA(cudaStreamSynchronize(s));
    if (reset) {
        SL_CUDA(cudaMemsetAsync(m->d.stats, 0, sizeof(c), s));
        SL_CUDA(cudaStreamSynchronize(s));
    }
    if (out) fill_stats(c, out);
    return SL_OK;
}

extern "C" sl_status sl_mesh_reorder(sl_mesh *m, int32_t curve, int32_t *node_perm, int32_t *tri_perm)
{
    if (!m) return fail(SL_E_ARG, "sl_mesh_reorder: mesh is NULL");
    if (curve < SL_CURVE_NONE || curve > SL_CURVE_MORTON) return fail(SL_E_ARG, "sl_mesh_reorder: unknown curve");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    if (m->stepped) {   // keep the walk state: bring the current T^0 back first
        SL_CUDA(cudaDeviceSynchronize());
        launch_export_t0((const int4 *)m->d.t0v, m->d.t0, m->N, 0);
        SL_CUDA(cudaMemcpy(m->t0.data(), m->d.t0, sizeof(int32_t) * m->N, cudaMemcpyDeviceToHost));
    }
    st = reorder_host(m, curve, node_perm, tri_perm);
    if (st != SL_OK) return st;
    if (m->graph.exec) cudaGraphExecDestroy((cudaGraphExec_t)m->graph.exec);
    m->graph = GraphCache();
    st = upload_arrays(m);
    // the structured-grid table follows the triangle numbering
    if (st == SL_OK && (m->opt_strategy == 2 || m->opt_strategy == 3))
        st = sl_mesh_set_option(m, SL_OPT_STRATEGY, m->opt_strategy);
    return st;
}

extern "C" void sl_mesh_destroy(sl_mesh *m)
{
    if (!m) return;
    free_device(m);
    delete m;
}

// After a renumbering: the recorded graph is stale, and the start tables of
// strategies 2 and 3 follow the triangle numbering.
static sl_status renumbered(sl_mesh *m)
{
    if (m->graph.exec) cudaGraphExecDestroy((cudaGraphExec_t)m->graph.exec);
    m->graph = GraphCache();
    sl_status st = upload_arrays(m);
    if (st == SL_OK && (m->opt_strategy == 2 || m->opt_strategy == 3))
        st = sl_mesh_set_option(m, SL_OPT_STRATEGY, m->opt_strategy);
    return st;
}

extern "C" sl_status sl_autotune_layout(sl_mesh *m, const sl_problem *probs, int32_t probe_steps, int32_t curves,
                                        void *v, void *v_scratch, int32_t *node_perm, int32_t *tri_perm, sl_tune *out,
                                        void *stream)
{
    if (!m || !probs || !v || !v_scratch || !out) return fail(SL_E_ARG, "sl_autotune_layout: NULL argument");
    if (probe_steps < 1 || probe_steps > 1000) return fail(SL_E_ARG, "sl_autotune_layout: probe_steps must be in [1, 1000]");
    if (curves < 1 || curves > 7) return fail(SL_E_ARG, "sl_autotune_layout: curves must be a non-empty set of sl_curve bits");
    if (!use_fast(m)) return fail(SL_E_STATE, "sl_autotune_layout: the plain kernel has no launch configurations");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t N = m->N, Nt = m->Nt;
    const size_t esz = m->precision == SL_FP64 ? sizeof(double) : sizeof(float);
    SL_CUDA(cudaStreamSynchronize(s));
    std::vector<uint8_t> v0(esz * N), vl(esz * N);
    SL_CUDA(cudaMemcpy(v0.data(), v, esz * N, cudaMemcpyDeviceToHost));
    if (m->stepped) {
        launch_export_t0((const int4 *)m->d.t0v, m->d.t0, N, s);
        SL_CUDA(cudaStreamSynchronize(s));
        SL_CUDA(cudaMemcpy(m->t0.data(), m->d.t0, sizeof(int32_t) * N, cudaMemcpyDeviceToHost));
    }
    // composite new -> old permutations (local) from the numbering at the call
    std::vector<int32_t> cn(N), ct(Nt), pn(N), pt(Nt);
    for (int32_t p = 0; p < m->n_problems; ++p) {
        for (int64_t i = m->node_off[p]; i < m->node_off[p + 1]; ++i) cn[i] = (int32_t)(i - m->node_off[p]);
        for (int64_t j = m->tri_off[p]; j < m->tri_off[p + 1]; ++j) ct[j] = (int32_t)(j - m->tri_off[p]);
    }
    auto compose = [&]() {   // cn <- cn o pn (pn: new -> old relative to the current numbering)
        for (int32_t p = 0; p < m->n_problems; ++p) {
            const int64_t n0 = m->node_off[p], t0 = m->tri_off[p];
            std::vector<int32_t> a(cn.begin() + n0, cn.begin() + m->node_off[p + 1]);
            for (int64_t i = n0; i < m->node_off[p + 1]; ++i) cn[i] = a[pn[i]];
            std::vector<int32_t> b(ct.begin() + t0, ct.begin() + m->tri_off[p + 1]);
            for (int64_t j = t0; j < m->tri_off[p + 1]; ++j) ct[j] = b[pt[j]];
        }
    };
    auto load_v = [&]() -> sl_status {   // V^0 in the current numbering
        for (int32_t p = 0; p < m->n_problems; ++p)
            for (int64_t i = m->node_off[p]; i < m->node_off[p + 1]; ++i)
                std::memcpy(&vl[esz * i], &v0[esz * (m->node_off[p] + cn[i])], esz);
        SL_CUDA(cudaMemcpy(v, vl.data(), esz * N, cudaMemcpyHostToDevice));
        return SL_OK;
    };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    SL_CUDA(cudaEventCreate(&e0));
    SL_CUDA(cudaEventCreate(&e1));
    auto time_layout = [&](float &ms) -> sl_status {
        sl_status r = load_v();
        if (r == SL_OK) r = sl_mesh_reset_t0(m, s);
        if (r != SL_OK) return r;
        SL_CUDA(cudaEventRecord(e0, s));
        r = run_steps(m, probs, 0, 1, v, v_scratch, 0, s, false);
        if (r != SL_OK) return r;
        m->t0_initial = false;
        r = run_steps(m, probs, 1, probe_steps, v, v_scratch, 0, s, false);
        if (r != SL_OK) return r;
        SL_CUDA(cudaEventRecord(e1, s));
        SL_CUDA(cudaEventSynchronize(e1));
        SL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        return SL_OK;
    };
    float times[3] = {-1.0f, -1.0f, -1.0f};
    int32_t best = -1, current = SL_CURVE_NONE;
    st = SL_OK;
    for (int32_t c = SL_CURVE_NONE; c <= SL_CURVE_MORTON && st == SL_OK; ++c) {
        if (!(curves >> c & 1)) continue;
        if (c != SL_CURVE_NONE) {
            st = reorder_host(m, c, pn.data(), pt.data());
            if (st == SL_OK) st = renumbered(m);
            if (st != SL_OK) break;
            compose();
            current = c;
        }
        {   // untimed first: lazy module loading, first touch of the new arrays
            float ms = 0.f;
            st = time_layout(ms);
            if (st != SL_OK) break;
        }
        st = time_layout(times[c]);
        if (st == SL_OK && (best < 0 || times[c] < times[best])) best = c;
    }
    if (st == SL_OK && best >= 0 && best != current) {
        if (best == SL_CURVE_NONE) {
            // back to the numbering at the call: the inverse of the composite
            for (int32_t p = 0; p < m->n_problems; ++p) {
                for (int64_t i = m->node_off[p]; i < m->node_off[p + 1]; ++i)
                    pn[m->node_off[p] + cn[i]] = (int32_t)(i - m->node_off[p]);
                for (int64_t j = m->tri_off[p]; j < m->tri_off[p + 1]; ++j)
                    pt[m->tri_off[p] + ct[j]] = (int32_t)(j - m->tri_off[p]);
            }
            st = permute_host(m, pn.data(), pt.data());
        } else {
            st = reorder_host(m, best, pn.data(), pt.data());
        }
        if (st == SL_OK) st = renumbered(m);
        if (st == SL_OK) compose();
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st == SL_OK) st = load_v();
    if (st == SL_OK) st = sl_mesh_reset_t0(m, s);
    if (st == SL_OK) SL_CUDA(cudaStreamSynchronize(s));
    if (node_perm) std::copy(cn.begin(), cn.end(), node_perm);
    if (tri_perm) std::copy(ct.begin(), ct.end(), tri_perm);
    if (st != SL_OK) return st;
    st = sl_autotune(m, probs, probe_steps, v, v_scratch, out, stream);
    out->curve = best;
    for (int k = 0; k < 3; ++k) out->curve_ms[k] = times[k];
    return st;
}

extern "C" sl_status sl_probe_gather(sl_mesh *m, const void *v, void *v_scratch, int32_t reps, float *ms_out,
                                     void *stream)
{
    if (!m || !v || !v_scratch || !ms_out) return fail(SL_E_ARG, "sl_probe_gather: NULL argument");
    if (reps < 1 || reps > 1000) return fail(SL_E_ARG, "sl_probe_gather: reps must be in [1, 1000]");
    if (v == v_scratch) return fail(SL_E_ARG, "sl_probe_gather: v and v_scratch must not alias");
    if (m->precision != SL_FP64) return fail(SL_E_ARG, "sl_probe_gather: FP64 meshes only");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    auto run = [&]() -> sl_status {
        SL_CUDA(cudaEventCreate(&e0));
        SL_CUDA(cudaEventCreate(&e1));
        const float4 *xyq = (const float4 *)m->d.xyq;
        const int4 *t0v = (const int4 *)m->d.t0v;
        launch_gather_probe(xyq, t0v, (const float2 *)v, (float2 *)v_scratch, m->N, s);
        SL_CUDA(cudaGetLastError());
        SL_CUDA(cudaEventRecord(e0, s));
        for (int32_t k = 0; k < reps; ++k) launch_gather_probe(xyq, t0v, (const float2 *)v, (float2 *)v_scratch, m->N, s);
        SL_CUDA(cudaEventRecord(e1, s));
        SL_CUDA(cudaEventSynchronize(e1));
        float ms = 0.f;
        SL_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        *ms_out = ms / (float)reps;
        return SL_OK;
    };
    st = run();
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    return st;
}

extern "C" sl_status sl_autotune(sl_mesh *m, const sl_problem *probs, int32_t probe_steps, void *v, void *v_scratch,
                                 sl_tune *out, void *stream)
{
    if (!m || !probs || !v || !v_scratch || !out) return fail(SL_E_ARG, "sl_autotune: NULL argument");
    if (probe_steps < 1 || probe_steps > 1000) return fail(SL_E_ARG, "sl_autotune: probe_steps must be in [1, 1000]");
    if (!use_fast(m)) return fail(SL_E_STATE, "sl_autotune: the plain kernel has no launch configurations");
    sl_status st = check_device(m);
    if (st != SL_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t vbytes = (m->precision == SL_FP64 ? sizeof(double) : sizeof(float)) * m->N;
    void *v_save = nullptr, *t_save = nullptr, *s_save = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
    const int32_t cfg0 = m->opt_config, cfgf0 = m->opt_config_first, split0 = m->opt_split, rec0 = m->opt_records;
    const bool init0 = m->t0_initial;
    std::memset(out, 0, sizeof(*out));
    for (int k = 0; k < SL_TUNE_MAX_CONFIGS; ++k) out->first_ms[k] = out->rest_ms[k] = out->split_ms[k] = -1.0f;
    out->compact_first_ms = out->compact_rest_ms = -1.0f;
    out->curve = -1;
    out->curve_ms[0] = out->curve_ms[1] = out->curve_ms[2] = -1.0f;
    auto cleanup = [&]() {
        if (v_save) cudaFree(v_save);
        if (t_save) cudaFree(t_save);
        if (s_save) cudaFree(s_save);
        if (e0) cudaEventDestroy(e0);
        if (e1) cudaEventDestroy(e1);
        if (e2) cudaEventDestroy(e2);
    };
    auto run = [&]() -> sl_status {
        SL_CUDA(cudaStreamSynchronize(s));
        SL_CUDA(cudaMalloc(&v_save, vbytes));
        SL_CUDA(cudaMalloc(&t_save, sizeof(int32_t) * m->N));
        SL_CUDA(cudaMalloc(&s_save, sizeof(unsigned long long) * kStatCounters));
        SL_CUDA(cudaMemcpy(v_save, v, vbytes, cudaMemcpyDeviceToDevice));
        launch_export_t0((const int4 *)m->d.t0v, (int32_t *)t_save, m->N, s);
        SL_CUDA(cudaMemcpy(s_save, m->d.stats, sizeof(unsigned long long) * kStatCounters, cudaMemcpyDeviceToDevice));
        SL_CUDA(cudaEventCreate(&e0));
        SL_CUDA(cudaEventCreate(&e1));
        SL_CUDA(cudaEventCreate(&e2));
        float best_first = 1e30f, best_rest = 1e30f;
        m->opt_split = 0;
        {   // one untimed step first: lazy module loading and first-touch costs
            sl_status r = sl_mesh_reset_t0(m, s);
            if (r == SL_OK) r = run_steps(m, probs, 0, 1, v, v_scratch, 0, s, false);
            if (r != SL_OK) return r;
            SL_CUDA(cudaStreamSynchronize(s));
        }
        for (int c = 0; c < kFastConfigs && c < SL_TUNE_MAX_CONFIGS; ++c) {
            m->opt_config = m->opt_config_first = c;
            SL_CUDA(cudaMemcpyAsync(v, v_save, vbytes, cudaMemcpyDeviceToDevice, s));
            sl_status r = sl_mesh_reset_t0(m, s);
            if (r != SL_OK) return r;
            SL_CUDA(cudaEventRecord(e0, s));
            r = run_steps(m, probs, 0, 1, v, v_scratch, 0, s, false);
            if (r != SL_OK) return r;
            m->t0_initial = false;
            SL_CUDA(cudaEventRecord(e1, s));
            r = run_steps(m, probs, 1, probe_steps, v, v_scratch, 0, s, false);
            if (r != SL_OK) return r;
            SL_CUDA(cudaEventRecord(e2, s));
            SL_CUDA(cudaEventSynchronize(e2));
            float f = 0.f, g = 0.f;
            SL_CUDA(cudaEventElapsedTime(&f, e0, e1));
            SL_CUDA(cudaEventElapsedTime(&g, e1, e2));
            g /= (float)probe_steps;
            out->first_ms[c] = f;
            out->rest_ms[c] = g;
            out->n_configs = c + 1;
            if (f < best_first) { best_first = f; out->config_first = c; }
            if (g < best_rest) { best_rest = g; out->config_rest = c; }
        }
        if (m->precision == SL_FP64) {
            // the later steps split into a settle pass and a finish pass (one
            // launch shape of their own; timed once, first step as chosen)
            m->opt_split = 1;
            sl_status r = ensure_queue(m);
            if (r != SL_OK) return r;
            for (int c = 0; c < 1; ++c) {
                m->opt_config = m->opt_config_first = out->config_first;
                SL_CUDA(cudaMemcpyAsync(v, v_save, vbytes, cudaMemcpyDeviceToDevice, s));
                r = sl_mesh_reset_t0(m, s);
                if (r != SL_OK) return r;
                r = run_steps(m, probs, 0, 1, v, v_scratch, 0, s, false);
                if (r != SL_OK) return r;
                m->t0_initial = false;
                SL_CUDA(cudaEventRecord(e1, s));
                r = run_steps(m, probs, 1, probe_steps, v, v_scratch, 0, s, false);
                if (r != SL_OK) return r;
                SL_CUDA(cudaEventRecord(e2, s));
                SL_CUDA(cudaEventSynchronize(e2));
                float g = 0.f;
                SL_CUDA(cudaEventElapsedTime(&g, e1, e2));
                g /= (float)probe_steps;
                out->split_ms[c] = g;
                if (g < best_rest) {
                    best_rest = g;
                    out->split = 1;
                }
            }
            m->opt_split = 0;
        }
        out->records = m->opt_records;
        if (m->precision == SL_FP64) {
            // the other walk-record form at the chosen configurations, scored
            // by a 50-step run (first step + 49 later ones)
            const float first_now = out->first_ms[out->config_first];
            const float rest_now = out->split ? out->split_ms[0] : out->rest_ms[out->config_rest];
            const int32_t other = m->opt_records ? 0 : 1;
            m->opt_records = other;
            sl_status r = build_walk_records(m);
            if (r != SL_OK) return r;
            if (other == 0 || m->d.he8) {
                m->opt_config_first = out->config_first;
                m->opt_config = out->config_rest;
                m->opt_split = out->split;
                SL_CUDA(cudaMemcpyAsync(v, v_save, vbytes, cudaMemcpyDeviceToDevice, s));
                r = sl_mesh_reset_t0(m, s);
                if (r != SL_OK) return r;
                SL_CUDA(cudaEventRecord(e0, s));
                r = run_steps(m, probs, 0, 1, v, v_scratch, 0, s, false);
                if (r != SL_OK) return r;
                m->t0_initial = false;
                SL_CUDA(cudaEventRecord(e1, s));
                r = run_steps(m, probs, 1, probe_steps, v, v_scratch, 0, s, false);
                if (r != SL_OK) return r;
                SL_CUDA(cudaEventRecord(e2, s));
                SL_CUDA(cudaEventSynchronize(e2));
                float f = 0.f, g = 0.f;
                SL_CUDA(cudaEventElapsedTime(&f, e0, e1));
                SL_CUDA(cudaEventElapsedTime(&g, e1, e2));
                g /= (float)probe_steps;
                out->compact_first_ms = other ? f : first_now;
                out->compact_rest_ms = other ? g : rest_now;
                if (f + 49.0f * g < first_now + 49.0f * rest_now) out->records = other;
                m->opt_split = 0;
            }
            if (m->opt_records != out->records) {
                m->opt_records = out->records;
                r = build_walk_records(m);
                if (r != SL_OK) return r;
            }
        }
        // restore values, T^0 and counters; keep the chosen configurations
        SL_CUDA(cudaMemcpyAsync(v, v_save, vbytes, cudaMemcpyDeviceToDevice, s));
        launch_fill_t0v((const int32_t *)t_save, m->d.tv[0], m->d.tv[1], m->d.tv[2], (int4 *)m->d.t0v, m->N, s);
        SL_CUDA(cudaMemcpyAsync(m->d.stats, s_save, sizeof(unsigned long long) * kStatCounters, cudaMemcpyDeviceToDevice, s));
        SL_CUDA(cudaMemsetAsync(m->d.status, 0, sizeof(uint32_t) * kStatusWords, s));
        SL_CUDA(cudaStreamSynchronize(s));
        m->opt_config = out->config_rest;
        m->opt_config_first = out->config_first;
        m->opt_split = out->split;
        m->t0_initial = init0;
        if (m->graph.exec) cudaGraphExecDestroy((cudaGraphExec_t)m->graph.exec);
        m->graph = GraphCache();
        return SL_OK;
    };
    st = run();
    if (st != SL_OK) {
        m->opt_config = cfg0;
        m->opt_config_first = cfgf0;
        m->opt_split = split0;
        m->t0_initial = init0;
        if (m->opt_records != rec0) {
            m->opt_records = rec0;
            build_walk_records(m);
        }
        if (m->graph.exec) cudaGraphExecDestroy((cudaGraphExec_t)m->graph.exec);
        m->graph = GraphCache();
    }
    cleanup();
    return st;
}
