// step_fast.cu -- the fast FP64-accuracy step kernel for GB300: launchers of
// the split step, the gather probe, value conversions, field tables and
// the walk records (the step kernels themselves are in step_fast_impl.cuh).
#include <cstring>

#include "step_fast_impl.cuh"

namespace sl {

template <bool kCompact>
static void launch_finish(const FastArgs &a, bool stats, bool debug, unsigned grid, cudaStream_t s)
{
    if (stats) {
        if (debug) launch_step_kernel(k_finish_df<true, true, kCompact>, grid, 128, s, a);
        else launch_step_kernel(k_finish_df<true, false, kCompact>, grid, 128, s, a);
    } else {
        if (debug) launch_step_kernel(k_finish_df<false, true, kCompact>, grid, 128, s, a);
        else launch_step_kernel(k_finish_df<false, false, kCompact>, grid, 128, s, a);
    }
}

template <int kBlock, int kMinBlocks>
static void launch_settle_cfg(const FastArgs &a, bool stats, bool debug, bool reset, cudaStream_t s)
{
    const unsigned grid = (unsigned)((a.N + kBlock - 1) / kBlock);
    if (grid == 0) return;
    if (reset) cudaMemsetAsync(a.queue_count, 0, sizeof(uint32_t), s);
    if (stats) {
        if (debug) launch_step_kernel(k_settle_df<true, true, kBlock, kMinBlocks, -1>, grid, kBlock, s, a);
        else launch_step_kernel(k_settle_df<true, false, kBlock, kMinBlocks, -1>, grid, kBlock, s, a);
    } else if (debug) {
        launch_step_kernel(k_settle_df<false, true, kBlock, kMinBlocks, -1>, grid, kBlock, s, a);
    } else if (!a.single) {
        launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, -1>, grid, kBlock, s, a);
    } else {
        // the timed path of a single mesh: the field kind compiled in
        switch (a.prob0.kind) {
        case SL_FIELD_AFFINE:
            launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_AFFINE>, grid, kBlock, s, a);
            break;
        case SL_FIELD_ROTATION:
            launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_ROTATION>, grid, kBlock, s, a);
            break;
        case SL_FIELD_SWIRL:
            launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_SWIRL>, grid, kBlock, s, a);
            break;
        case SL_FIELD_PAPER:
            launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_PAPER>, grid, kBlock, s, a);
            break;
        case SL_FIELD_FOURIER8:
            launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_FOURIER8>, grid, kBlock, s, a);
            break;
        default: launch_step_kernel(k_settle_df<false, false, kBlock, kMinBlocks, SL_FIELD_ZERO>, grid, kBlock, s, a); break;
        }
    }
}

// The settle pass needs 32 registers, so it runs at 128 x 14 (56 resident
// warps per SM): faster than at 48 or 64.  The caller provides a.queue (N
// entries) and a.queue_count (zeroed here when reset, else by the previous
// step's settle pass through its queue_next).
void launch_settle_df(const FastArgs &a, bool stats, bool debug, bool reset, cudaStream_t s)
{
    launch_settle_cfg<128, 14>(a, stats, debug, reset, s);
}

// The finish pass: a persistent grid of 8 blocks of 128 per SM over the queue.
void launch_finish_df(const FastArgs &a, bool stats, bool debug, int sms, cudaStream_t s)
{
    const unsigned g2 = (unsigned)(sms > 0 ? sms : 152) * 8u;
    if (a.he8) launch_finish<true>(a, stats, debug, g2, s);
    else launch_finish<false>(a, stats, debug, g2, s);
}


// Launch configurations (threads per block x resident blocks per SM the
// register budget is sized for): 0 = 256 x 4 (64 registers), 1 = 128 x 16 (32;
// 2 % faster than 128 x 12 on a batch of 2.8 M nodes, 4 % slower on 491 k), 2 =
// 128 x 8, 3 = 128 x 9 (56 registers), 4 = 256 x 5, 5 = 128 x 12.  Each
// is instantiated in a translation unit of its own pair (step_fast_c*.cu).
//
// They are configurations of the lean kernel.  Statistics, debug outputs,
// strategy (c) and a handle without its tables (a.tri) run the full node step in
// one configuration of its own.  A hop cap of the caller's holds in the lean
// kernel too: its hops are the full step's and end at the cap (a 1024^2-node swirl
// of 20 steps under a cap it never meets: 2.67 ms in the full step alone, 1.36
// here; 1.22 if the feet at their nodes were sent to the triangle known for them,
// past the walk that the cap is about).
void launch_fast_df(const FastArgs &a, bool stats, bool debug, int config, cudaStream_t s)
{
    if (stats || debug || a.order || !a.tri) {
        launch_full_df(a, stats, debug, s);
        return;
    }
    if (a.exclude || a.grid_M > 0 || a.keep_t0) {
        launch_lean_df_ext(a, s);
        return;
    }
    switch (config) {
    case 1: launch_lean_df_c1(a, s); break;
    case 2: launch_lean_df_c2(a, s); break;
    case 3: launch_lean_df_c3(a, s); break;
    case 4: launch_lean_df_c4(a, s); break;
    case 5: launch_lean_df_c5(a, s); break;
    default: launch_lean_df_c0(a, s); break;
    }
}

// A later step of steady fields (apply_weights) for every node.  Bound by
// memory: 48 bytes per node stream (weights, V^n, V^{n+1}) beside three value
// gathers that mostly hit L1, at 32 registers and 64 warps per SM: 0.118 ms on
// 16.8 M nodes, the measured copy bandwidth, where locating every node again
// (foot, certified test, quotient; also 48 bytes, 290 instructions, 64 bytes of
// gathered vertices) took 0.180 ms.  A 50-step rotation 9.60 -> 6.69 ms.  The
// weights past L1: they are read once.
//
// A node without weights yet (emit_open) takes the full node step, inline: called
// out of line it put saved registers on every node's path (50 steps 6.64 -> 6.73
// to 7.46 ms, four forms), inline the spills are its own (6.64 ms).
template <bool kCompact>
__global__ void __launch_bounds__(256, 8) k_apply_df(const __grid_constant__ FastArgs a)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (i >= a.N) return;
    float2 v;
    if (apply_weights(a, i, v)) {
        put_value(a, i, v);
        return;
    }
    NodeCounters c;
    step_node<false, true, false, kCompact>(a, i, a.nprob == 1 ? 0 : chunk_problem(a.chunk_prob, a.node_off, i), c);
}

void launch_apply_df(const FastArgs &a, cudaStream_t s)
{
    const unsigned grid = (unsigned)((a.N + 255) / 256);
    if (grid == 0) return;
    if (a.he8) launch_step_kernel(k_apply_df<true>, grid, 256, s, a);
    else launch_step_kernel(k_apply_df<false>, grid, 256, s, a);
}

// The triangle that holds node i's coordinate pair, the point a foot of no
// displacement (or one below the pair's rounding) is: within 2^-49 of the node,
// so among the node's triangles, found from the initial one over negative
// exact signs.  -1: the pair is on a vertex or between two triangles, where the
// step's own path decides.  Once per mesh and numbering, for the full step's
// foot_on_pair: with exact signs for every node of a step at which the field
// vanishes, and for a third of a swirl's boundary nodes at every step, 20 steps
// on 1.05 M nodes took 1.005 ms, 0.910 without; two single steps on 296 k nodes
// 70 -> 66 us.  (Asked in the lean pass instead it cost that pass 2 to 8 %.)
__global__ void k_pair_tri(const __grid_constant__ FastArgs a, int32_t *__restrict__ pair_tri)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.N) return;
    const float4 xq = a.xyq[i];
    const df X = df_make(xq.x, xq.z), Y = df_make(xq.y, xq.w);
    int32_t j = a.t0_init[i], found = -1;
    for (int hop = 0; hop < 64; ++hop) {
        const uint32_t r = exact_signs<false>(a.xyd, a.tv[0][j], a.tv[1][j], a.tv[2][j], X, Y, 7u);
        if (r & (1u << 12)) break;                       // a coordinate outside the exact range
        if (r & 0x2au) {
            const int32_t u = a.tn[r & 2u ? 0 : (r & 8u ? 1 : 2)][j];
            if (u < 0) break;
            j = u;
            continue;
        }
        const uint32_t pos = r & 0x15u;
        const int zeros = 3 - __popc(pos), k = !(pos & 1u) ? 0 : (!(pos & 4u) ? 1 : 2);
        if (zeros == 0 || (zeros == 1 && a.tn[k][j] < 0)) found = j;
        break;
    }
    pair_tri[i] = found;
}

void launch_pair_tri(const FastArgs &a, int32_t *pair_tri, cudaStream_t s)
{
    if (a.N > 0) k_pair_tri<<<(unsigned)((a.N + 127) / 128), 128, 0, s>>>(a, pair_tri);
}

// ---------------------------------------------------------------------------
// Gather probe: the memory accesses of a step whose feet stay in their start
// triangles, with only a sum as arithmetic (sl_probe_gather).

__global__ void __launch_bounds__(128, 14) k_gather_probe(const float4 *xyq, const int4 *t0v, const float2 *vin,
                                                          float2 *vout, int64_t N)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const float4 xq = xyq[i];
    const int4 tq = t0v[i];
    const float4 A = xyq[tq.y], B = xyq[tq.z], C = xyq[tq.w];
    const float2 V1 = vin[tq.y], V2 = vin[tq.z], V3 = vin[tq.w];
    const float s = ((xq.x + xq.y) + (xq.z + xq.w)) + ((A.x + A.y) + (A.z + A.w)) + ((B.x + B.y) + (B.z + B.w)) +
                    ((C.x + C.y) + (C.z + C.w)) + __int_as_float(tq.x & 0x007fffff);
    vout[i] = make_float2((V1.x + V2.x) + (V3.x + s), (V1.y + V2.y) + V3.y);
}

void launch_gather_probe(const float4 *xyq, const int4 *t0v, const float2 *vin, float2 *vout, int64_t N,
                         cudaStream_t s)
{
    if (N > 0) k_gather_probe<<<(unsigned)((N + 127) / 128), 128, 0, s>>>(xyq, t0v, vin, vout, N);
}

// ---------------------------------------------------------------------------
// Value format conversions (once per run, not per step)

__global__ void k_to_df(const double *__restrict__ src, float2 *__restrict__ dst, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        dst[i] = pair_of_double(src[i]);
    }
}

__global__ void k_from_df(const float2 *src, double *dst, int64_t n)
{
    // may run in place (src and dst alias, same 8-byte slots)
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        dst[i] = double_of_pair(src[i]);
    }
}

static unsigned grid_for(int64_t n, int block)
{
    int64_t g = (n + block - 1) / block;
    if (g > 152 * 32) g = 152 * 32;
    return (unsigned)(g > 0 ? g : 1);
}

void launch_to_df(const double *src, float2 *dst, int64_t n, cudaStream_t s)
{
    if (n > 0) k_to_df<<<grid_for(n, 256), 256, 0, s>>>(src, dst, n);
}

void launch_from_df(const float2 *src, double *dst, int64_t n, cudaStream_t s)
{
    if (n > 0) k_from_df<<<grid_for(n, 256), 256, 0, s>>>(src, dst, n);
}

namespace {
constexpr int kConstChunk = 56;     // 4 KiB of parameters
struct ConstChunk {
    FastProb *dst;
    int32_t count;
    FastProb p[kConstChunk];
};
__global__ void k_put_constants(const __grid_constant__ ConstChunk c)
{
    const int t = threadIdx.x;
    if (t < c.count) c.dst[t] = c.p[t];
}
}  // namespace

void launch_put_constants(const FastProb *src, int32_t n, FastProb *dst, cudaStream_t s)
{
    for (int32_t b = 0; b < n; b += kConstChunk) {
        ConstChunk c;
        c.dst = dst + b;
        c.count = n - b < kConstChunk ? n - b : kConstChunk;
        std::memcpy(c.p, src + b, sizeof(FastProb) * (size_t)c.count);
        k_put_constants<<<1, kConstChunk, 0, s>>>(c);
    }
}

// ---------------------------------------------------------------------------
// Node tables of the fields whose space dependence is costly (trigonometric):
//   SWIRL     g1 = (sin^2(pi x) sin(2 pi y), -sin^2(pi y) sin(2 pi x))
//   PAPER     g1 = (cos a, sin a), g2 = (-sin a, cos a), a = C0 |x - c|
//             (f = cos(C1 t) g1 + sin(C1 t) g2)
//   FOURIER8  g1 = sum_m a_m cos(phi_m) h_m, g2 = -sum_m a_m sin(phi_m) h_m,
//             h_m = (l_m pi sin(k_m pi x) cos(l_m pi y), -k_m pi cos(k_m pi x) sin(l_m pi y))
//             (f = cos(2 pi t) g1 + sin(2 pi t) g2)
// evaluated once per field in double and stored as (hi, lo) floats.

__device__ __forceinline__ float4 pack_df2(double gx, double gy)
{
    const float hx = __double2float_rn(gx), hy = __double2float_rn(gy);
    return make_float4(hx, hy, __double2float_rn(gx - (double)hx), __double2float_rn(gy - (double)hy));
}

__global__ void k_field_tables(FieldTableArgs a)
{
    const double pi = 3.14159265358979323846;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int pidx = a.nprob == 1 ? 0 : problem_of(a.node_off, a.nprob, i);
        const double *q = a.params + (1 + SL_NPARAMS) * (int64_t)pidx;
        const int kind = (int)q[0];
        const double *p = q + 1;
        const double2 xy = a.xyd ? a.xyd[i] : make_double2((double)a.xyf[i].x, (double)a.xyf[i].y);
        double g1x = 0, g1y = 0, g2x = 0, g2y = 0;
        if (kind == SL_FIELD_SWIRL) {
            double sx, cx, sy, cy;
            sincospi(xy.x, &sx, &cx);
            sincospi(xy.y, &sy, &cy);
            g1x = (sx * sx) * (2.0 * sy * cy);
            g1y = -(sy * sy) * (2.0 * sx * cx);
        } else if (kind == SL_FIELD_PAPER) {
            const double dx = xy.x - p[2], dy = xy.y - p[3];
            double s, c;
            sincos(p[0] * sqrt(dx * dx + dy * dy), &s, &c);
            g1x = c;
            g1y = s;
            g2x = -s;
            g2y = c;
        } else if (kind == SL_FIELD_FOURIER8) {
            for (int m = 0; m < 8; ++m) {
                const double k = p[4 * m], l = p[4 * m + 1], am = p[4 * m + 2], ph = p[4 * m + 3];
                double skx, ckx, sly, cly, sph, cph;
                sincospi(k * xy.x, &skx, &ckx);
                sincospi(l * xy.y, &sly, &cly);
                sincos(ph, &sph, &cph);
                const double hx = l * pi * skx * cly, hy = -k * pi * ckx * sly;
                g1x += am * cph * hx;
                g1y += am * cph * hy;
                g2x -= am * sph * hx;
                g2y -= am * sph * hy;
            }
        }
        if (a.g1) a.g1[i] = pack_df2(g1x, g1y);
        if (a.g2) a.g2[i] = pack_df2(g2x, g2y);
        if (a.g1f) a.g1f[i] = make_float2(__double2float_rn(g1x), __double2float_rn(g1y));
        if (a.g2f) a.g2f[i] = make_float2(__double2float_rn(g2x), __double2float_rn(g2y));
    }
}

// T^0 back to its initial triangles (sl_mesh_reset_t0).
__global__ void k_reset_t0(const int32_t *__restrict__ t0_init, const int4 *__restrict__ tri, int4 *__restrict__ t0v,
                           int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        t0v[i] = tri[t0_init[i]];
}

// T^0 as triangle indices.  The steps keep only the start states, 16 bytes per
// node that moved; with the index beside them they wrote 20 (an FP32 swirl on 4.2 M
// nodes 2.45 against 2.40 ms per 20 steps, a batch of 2.8 M 3.96 against 3.92 ms per
// 50, 8 single steps on 491 k 174 against 170 us).
__global__ void k_export_t0(const int4 *__restrict__ t0v, int32_t *__restrict__ t0, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        t0[i] = tri_of(t0v[i].x);
}

__global__ void k_fill_t0v(const int32_t *__restrict__ t0, const int32_t *__restrict__ tv0,
                           const int32_t *__restrict__ tv1, const int32_t *__restrict__ tv2, int4 *__restrict__ t0v,
                           int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t j = t0[i];
        t0v[i] = make_int4(3 * j, tv0[j], tv1[j], tv2[j]);
    }
}

// Jump table, pass 1: the least initial triangle of the nodes in each cell.
__global__ void k_jump_seed(JumpBuildArgs a)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int p = a.nprob == 1 ? 0 : problem_of(a.node_off, a.nprob, i);
        const int g = a.gp[p];
        const float2 x = a.xyc[i];
        atomicMin(&a.seed[0][a.off[p] + jump_cell(x.y, g) * g + jump_cell(x.x, g)], (uint32_t)a.t0_init[i]);
    }
}

// The problem of a cell (binary search over the cell offsets).
__device__ __forceinline__ int jump_problem(const int32_t *off, int nprob, int32_t c)
{
    int lo = 0, hi = nprob;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= c) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Pass 2, with r = 1, 2, 4, ...: a cell without a seed takes the least seed of
// the cells r away in the eight directions (any triangle will do; it should be
// near).
__global__ void k_jump_fill(JumpBuildArgs a, int r, int from)
{
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < a.cells; c += gridDim.x * blockDim.x) {
        uint32_t v = a.seed[from][c];
        if (v == 0xFFFFFFFFu) {
            const int p = a.nprob == 1 ? 0 : jump_problem(a.off, a.nprob, c);
            const int g = a.gp[p], q = c - a.off[p], m = q / g, l = q - m * g;
            for (int dm = -r; dm <= r; dm += r)
                for (int dl = -r; dl <= r; dl += r)
                    if (m + dm >= 0 && m + dm < g && l + dl >= 0 && l + dl < g)
                        v = min(v, a.seed[from][a.off[p] + (m + dm) * g + l + dl]);
        }
        a.seed[from ^ 1][c] = v;
    }
}

// Pass 3: from the seed triangle, cross the edge the cell's centre lies
// furthest beyond, at most 64 times (float: any triangle is a valid start).
// A cell that found no seed takes the initial triangle of its problem's first
// node.
__global__ void k_jump_walk(JumpBuildArgs a, int from)
{
    for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < a.cells; c += gridDim.x * blockDim.x) {
        const int p = a.nprob == 1 ? 0 : jump_problem(a.off, a.nprob, c);
        const int g = a.gp[p], q = c - a.off[p], m = q / g, l = q - m * g;
        const float X = ((float)l + 0.5f) / (float)g, Y = ((float)m + 0.5f) / (float)g;
        const uint32_t seed = a.seed[from][c];
        int32_t j = seed == 0xFFFFFFFFu ? a.t0_init[a.node_off[p]] : (int32_t)seed;
        int w[3];
        for (int hop = 0;; ++hop) {
            float2 V[3];
            for (int k = 0; k < 3; ++k) {
                w[k] = a.tv[k][j];
                V[k] = a.xyc[w[k]];
            }
            float best = 0.0f;
            int b = -1;
            for (int k = 0; k < 3; ++k) {
                const float2 A = V[(k + 1) % 3], B = V[(k + 2) % 3];
                const float o = (A.x - X) * (B.y - Y) - (A.y - Y) * (B.x - X);
                if (o < best) {
                    best = o;
                    b = k;
                }
            }
            if (b < 0 || hop == 64) break;
            const int32_t u = a.tn[b][j];
            if (u < 0) break;
            j = u;
        }
        a.jump[c] = make_int4(3 * j, w[0], w[1], w[2]);
    }
}

void launch_build_jump(const JumpBuildArgs &a, cudaStream_t s)
{
    if (a.N <= 0 || a.cells <= 0) return;
    cudaMemsetAsync(a.seed[0], 0xFF, sizeof(uint32_t) * (size_t)a.cells, s);
    k_jump_seed<<<grid_for(a.N, 256), 256, 0, s>>>(a);
    int from = 0;
    for (int r = 1; r < 2 * a.max_g; r *= 2, from ^= 1) k_jump_fill<<<grid_for(a.cells, 256), 256, 0, s>>>(a, r, from);
    k_jump_walk<<<grid_for(a.cells, 128), 128, 0, s>>>(a, from);
}

struct HalfEdgeArgs {
    const int32_t *tv[3];
    const int32_t *tn[3];
    const float2 *xyc;
    int64_t nt;
    float4 *he;
};

__global__ void k_build_he(HalfEdgeArgs a)
{
    const int64_t nh = 3 * a.nt;
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = (int32_t)(h / 3), k = (int32_t)(h - 3 * (int64_t)t);
        const int32_t u = a.tn[k][t];
        float4 r = make_float4(__int_as_float(0x7fc00000), __int_as_float(0x7fc00000),
                               __int_as_float(3 * t + (k == 2 ? 0 : k + 1)), __int_as_float(u));
        if (u >= 0) {
            int kp = 0;
            if (a.tn[1][u] == t) kp = 1;
            else if (a.tn[2][u] == t) kp = 2;
            const float2 q = a.xyc[a.tv[kp][u]];
            r = make_float4(q.x, q.y, __int_as_float(3 * u + (kp == 2 ? 0 : kp + 1)),
                            __int_as_float(3 * u + (kp == 0 ? 2 : kp - 1)));
        }
        a.he[h] = r;
    }
}

void launch_build_he(const int32_t *const tv[3], const int32_t *const tn[3], const float2 *xyc, int64_t nt,
                     float4 *he, cudaStream_t s)
{
    HalfEdgeArgs a;
    for (int k = 0; k < 3; ++k) {
        a.tv[k] = tv[k];
        a.tn[k] = tn[k];
    }
    a.xyc = xyc;
    a.nt = nt;
    a.he = he;
    if (nt > 0) k_build_he<<<grid_for(3 * nt, 256), 256, 0, s>>>(a);
}

struct HalfEdge8Args {
    const int32_t *tv[3];
    const int32_t *tn[3];
    const float2 *xyh;
    int64_t nt;
    uint2 *he8;
    uint32_t *overflow;
};

__global__ void k_build_he8(HalfEdge8Args a)
{
    const int64_t nh = 3 * a.nt;
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += (int64_t)gridDim.x * blockDim.x) {
        const int32_t t = (int32_t)(h / 3), k = (int32_t)(h - 3 * (int64_t)t);
        const int32_t u = a.tn[k][t];
        if (3 * (int64_t)t + 2 >= (1 << 27)) atomicOr(a.overflow, 1u);
        // boundary edge: zero offset, the exits of t itself
        int32_t e0 = 3 * t + (k == 2 ? 0 : k + 1);
        uint32_t bx = 1u << 17, by = 1u << 17;
        if (u >= 0) {
            int kp = 0;
            if (a.tn[1][u] == t) kp = 1;
            else if (a.tn[2][u] == t) kp = 2;
            // Q and the entered triangle's first vertex W0 = T[k'+1][u] (an
            // edge of u)
            const float2 q = a.xyh[a.tv[kp][u]], w = a.xyh[a.tv[kp == 2 ? 0 : kp + 1][u]];
            // grid values: the differences and their scaling by 2^24 are exact
            const float fx = __fmul_rn(__fsub_rn(q.x, w.x), 16777216.0f);
            const float fy = __fmul_rn(__fsub_rn(q.y, w.y), 16777216.0f);
            if (fabsf(fx) > 131070.0f || fabsf(fy) > 131070.0f || 3 * (int64_t)u + 2 >= (1 << 27)) {
                atomicOr(a.overflow, 1u);
            } else {
                bx = (uint32_t)(__float2int_rn(fx) + (1 << 17));
                by = (uint32_t)(__float2int_rn(fy) + (1 << 17));
                e0 = 3 * u + (kp == 2 ? 0 : kp + 1);
            }
        }
        const uint32_t f = (e0 % 3 == 2) ? 1u : 0u;
        const uint2 r = make_uint2(bx | ((by & 0x3FFFu) << 18), (by >> 14) | (f << 4) | ((uint32_t)e0 << 5));
        a.he8[h] = r;
    }
}

void launch_build_he8(const int32_t *const tv[3], const int32_t *const tn[3], const float2 *xyh, int64_t nt,
                      uint2 *he8, uint32_t *overflow, cudaStream_t s)
{
    HalfEdge8Args a;
    for (int k = 0; k < 3; ++k) {
        a.tv[k] = tv[k];
        a.tn[k] = tn[k];
    }
    a.xyh = xyh;
    a.nt = nt;
    a.he8 = he8;
    a.overflow = overflow;
    if (nt > 0) k_build_he8<<<grid_for(3 * nt, 256), 256, 0, s>>>(a);
}

__global__ void k_build_tri(const int32_t *__restrict__ tv0, const int32_t *__restrict__ tv1,
                            const int32_t *__restrict__ tv2, int4 *__restrict__ tri, int64_t nt)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x)
        tri[t] = make_int4(3 * (int32_t)t, tv0[t], tv1[t], tv2[t]);
}

void launch_build_tri(const int32_t *const tv[3], int64_t nt, int4 *tri, cudaStream_t s)
{
    if (nt > 0) k_build_tri<<<grid_for(nt, 256), 256, 0, s>>>(tv[0], tv[1], tv[2], tri, nt);
}

void launch_fill_t0v(const int32_t *t0, const int32_t *tv0, const int32_t *tv1, const int32_t *tv2, int4 *t0v,
                     int64_t n, cudaStream_t s)
{
    if (n > 0) k_fill_t0v<<<grid_for(n, 256), 256, 0, s>>>(t0, tv0, tv1, tv2, t0v, n);
}

void launch_reset_t0(const int32_t *t0_init, const int4 *tri, int4 *t0v, int64_t n, cudaStream_t s)
{
    if (n > 0) k_reset_t0<<<grid_for(n, 256), 256, 0, s>>>(t0_init, tri, t0v, n);
}

void launch_export_t0(const int4 *t0v, int32_t *t0, int64_t n, cudaStream_t s)
{
    if (n > 0) k_export_t0<<<grid_for(n, 256), 256, 0, s>>>(t0v, t0, n);
}

void launch_field_tables(const FieldTableArgs &a, cudaStream_t s)
{
    if (a.N > 0) k_field_tables<<<grid_for(a.N, 256), 256, 0, s>>>(a);
}

}  // namespace sl
