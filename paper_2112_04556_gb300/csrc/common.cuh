// Shared runtime pieces of the library: context, status handling, lattice geometry, link views,
// deterministic float64 reductions and the workspace pool.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <algorithm>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "../../include/rmhmc.h"
#include "su3.cuh"

namespace rm {

constexpr int kBlock = 128;           // threads per block of the site kernels
constexpr int kBlockMin = 64;         // smallest block of a tuned stencil launch
constexpr int kBlockMax = 256;        // largest block of a tuned stencil launch
constexpr int kRedSlots = 256;        // reduction slots per context (one per concurrent sum)

// ------------------------------------------------------------------------------------------------
// lattice geometry
// ------------------------------------------------------------------------------------------------
struct Geom {
    int L[4];
    int stride[4];
    int V;
    // division by L[d] as a multiply-high and shift (Granlund-Montgomery round-up method, exact for
    // numerators below 2^31 and therefore for every site index): q = (umulhi(mag, n) + n) >> shr
    unsigned mag[4];
    int shr[4];
};

__host__ inline void geom_init_divmod(Geom& g) {
    for (int d = 0; d < 4; d++) {
        int l = 0;
        while ((1u << l) < (unsigned)g.L[d]) l++;
        const unsigned long long m = ((1ull << 32) * ((1ull << l) - (unsigned long long)g.L[d])) / (unsigned long long)g.L[d] + 1ull;
        g.mag[d] = (unsigned)(m & 0xffffffffull);
        g.shr[d] = l;
    }
}

__device__ __forceinline__ int fast_div(const Geom& g, int n, int d) {
    return (int)((__umulhi(g.mag[d], (unsigned)n) + (unsigned)n) >> g.shr[d]);
}

__device__ __forceinline__ void neighbours(const Geom& g, int s, int fwd[4], int bwd[4]) {
    int r = s;
#pragma unroll
    for (int d = 0; d < 4; d++) {
        const int q = fast_div(g, r, d);
        const int c = r - q * g.L[d];
        r = q;
        fwd[d] = (c == g.L[d] - 1) ? s - c * g.stride[d] : s + g.stride[d];
        bwd[d] = (c == 0) ? s + (g.L[d] - 1) * g.stride[d] : s - g.stride[d];
    }
}

__device__ __forceinline__ void site_coords(const Geom& g, int s, int c[4]) {
#pragma unroll
    for (int d = 0; d < 4; d++) {
        const int q = fast_div(g, s, d);
        c[d] = s - q * g.L[d];
        s = q;
    }
}

// neighbour of site s one step (n = +1 or -1) along direction d, periodic
__device__ __forceinline__ int step_site(const Geom& g, int s, int d, int n) {
    int r = s, c = 0;
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int q = fast_div(g, r, e);
        if (e == d) c = r - q * g.L[e];
        r = q;
    }
    if (n > 0) return c == g.L[d] - 1 ? s - c * g.stride[d] : s + g.stride[d];
    return c == 0 ? s + (g.L[d] - 1) * g.stride[d] : s - g.stride[d];
}

// site reached from coordinates c by n steps along direction d (periodic), without changing c
__device__ __forceinline__ int shifted(const Geom& g, const int c[4], int d, int n) {
    int s = 0;
#pragma unroll
    for (int e = 3; e >= 0; e--) {
        int ce = c[e];
        if (e == d) { ce = (ce + n) % g.L[e]; if (ce < 0) ce += g.L[e]; }
        s = s * g.L[e] + ce;
    }
    return s;
}

// ------------------------------------------------------------------------------------------------
// internal link layouts
//   FP64: u64[(mu*9 + 3i + j) * V + s]            double2 (re, im)
//   FP32: u32a[(mu*3 + r) * V + s]  float4, r=0: (u00,u01) r=1: (u02,u10) r=2: (u11,u12)
//         u32b[(mu*3 + j) * V + s]  float2, u2j (third row; unused by the 12-real format)
// ------------------------------------------------------------------------------------------------
//   FP64, adjoint table (link "format" kLinkAd): ad[(mu*32 + 4b + h) * V + s]  double2 (Ad[2h][b], Ad[2h+1][b])
constexpr int kLinkAd = 64;
struct Links64 { const double2* u; int V; const double2* ad; };
struct Links32 { const float4* a; const float2* b; int V; };

template <typename T, int LF> struct LinkLoad;

template <int LF> struct LinkLoad<double, LF> {
    __device__ __forceinline__ static mat3<double> load(const Links64& U, int s, int mu) {
        mat3<double> m;
        const int rows = LF == 12 ? 2 : 3;
#pragma unroll
        for (int i = 0; i < rows; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const double2 v = __ldg(&U.u[(size_t)(mu * 9 + 3 * i + j) * U.V + s]);
                m.e[i][j] = cmk(v.x, v.y);
            }
        if (LF == 12) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
                cplx<double> c = csub(cmul(m.e[0][j1], m.e[1][j2]), cmul(m.e[0][j2], m.e[1][j1]));
                m.e[2][j] = cconj(c);
            }
        }
        return m;
    }
};

template <int LF> struct LinkLoad<float, LF> {
    __device__ __forceinline__ static mat3<float> load(const Links32& U, int s, int mu) {
        mat3<float> m;
        const float4 r0 = __ldg(&U.a[(size_t)(mu * 3 + 0) * U.V + s]);
        const float4 r1 = __ldg(&U.a[(size_t)(mu * 3 + 1) * U.V + s]);
        const float4 r2 = __ldg(&U.a[(size_t)(mu * 3 + 2) * U.V + s]);
        m.e[0][0] = cmk(r0.x, r0.y); m.e[0][1] = cmk(r0.z, r0.w);
        m.e[0][2] = cmk(r1.x, r1.y); m.e[1][0] = cmk(r1.z, r1.w);
        m.e[1][1] = cmk(r2.x, r2.y); m.e[1][2] = cmk(r2.z, r2.w);
        if (LF == 12) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
                cplx<float> c = csub(cmul(m.e[0][j1], m.e[1][j2]), cmul(m.e[0][j2], m.e[1][j1]));
                m.e[2][j] = cconj(c);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const float2 v = __ldg(&U.b[(size_t)(mu * 3 + j) * U.V + s]);
                m.e[2][j] = cmk(v.x, v.y);
            }
        }
        return m;
    }
};

// ------------------------------------------------------------------------------------------------
// field component access: AoS [V][4][8]
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void load8(const double* p, double* x) {
    const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
    for (int i = 0; i < 4; i++) { double2 v = __ldg(q + i); x[2 * i] = v.x; x[2 * i + 1] = v.y; }
}
__device__ __forceinline__ void load8(const float* p, float* x) {
    const float4* q = reinterpret_cast<const float4*>(p);
    float4 a = __ldg(q), b = __ldg(q + 1);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
// a * b + c on a pair of float32 values in one instruction (each rounded as fmaf rounds)
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ void store8(double* p, const double* x) {
    double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
    for (int i = 0; i < 4; i++) q[i] = make_double2(x[2 * i], x[2 * i + 1]);
}
__device__ __forceinline__ void store8(float* p, const float* x) {
    float4* q = reinterpret_cast<float4*>(p);
    q[0] = make_float4(x[0], x[1], x[2], x[3]);
    q[1] = make_float4(x[4], x[5], x[6], x[7]);
}

// ------------------------------------------------------------------------------------------------
// Krylov vectors (the basis r_k and q) are chunk-planar: [8][V][4], plane c = 2 mu + h holding the colours 4 h .. 4 h + 3
// of component mu.  Consecutive sites are adjacent in a plane, so a warp of 32 consecutive sites reads a component of
// any of their neighbours as two contiguous 512-byte segments, and its links without duplicates; with the sites' 128-byte
// rows of the [V][4][8] layout either the links are read four times (four lanes per site) or every load touches 32
// lines (one).
// ------------------------------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ const T* plane_at(const T* X, int V, int s, int c) {
    return X + ((size_t)c * V + s) * 4;
}
template <typename T> __device__ __forceinline__ T* plane_at(T* X, int V, int s, int c) {
    return X + ((size_t)c * V + s) * 4;
}
__device__ __forceinline__ void load4(const float* p, float* x) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double* x) {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p)), b = __ldg(reinterpret_cast<const double2*>(p) + 1);
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
}
__device__ __forceinline__ void store4(float* p, const float* x) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void store4(double* p, const double* x) {
    reinterpret_cast<double2*>(p)[0] = make_double2(x[0], x[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(x[2], x[3]);
}
// the eight colours of component mu at site s
template <typename T> __device__ __forceinline__ void load_plane8(const T* X, int V, int s, int mu, T* x) {
    load4(plane_at(X, V, s, 2 * mu), x);
    load4(plane_at(X, V, s, 2 * mu + 1), x + 4);
}

// ------------------------------------------------------------------------------------------------
// deterministic reductions: every block writes its partial sums to a slot array; the last block
// to finish (ticket counter) adds them in block order in float64 and writes the result.
// ------------------------------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double* sh /* N * (kBlock/32) */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int n = 0; n < N; n++) {
        double x = v[n];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sh[n * (blockDim.x >> 5) + warp] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int n = 0; n < N; n++) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += sh[n * (blockDim.x >> 5) + w];
            v[n] = s;
        }
    }
}

// float partials summed within a warp in float, then across warps and blocks in double
template <int N>
__device__ __forceinline__ void block_sum_f(float (&v)[N], double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int n = 0; n < N; n++) {
        float x = v[n];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sh[n * (blockDim.x >> 5) + warp] = (double)x;
    }
    __syncthreads();
}

// Called by EVERY thread of every block; v[] holds the block's N sums in thread 0.  partials:
// [nblocks][N] for this reduction, counter: its ticket.  The last block to arrive adds all partials:
// thread t takes blocks t, t + blockDim, ... in that order, then a fixed shuffle/shared-memory tree, so
// the result does not depend on scheduling.  Returns true in thread 0 of the last block, with out[0..N-1]
// written; sh needs N * (blockDim / 32) doubles.
template <int N>
__device__ __forceinline__ bool grid_sum_finish(const double* v, double* partials, unsigned* counter, double* out,
                                                int nblocks, int bid, double* sh) {
    __shared__ int am_last;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int n = 0; n < N; n++) partials[(size_t)bid * N + n] = v[n];
        __threadfence();
        const unsigned ticket = atomicAdd(counter, 1u);
        am_last = ticket == (unsigned)(nblocks - 1);
    }
    __syncthreads();
    if (!am_last) return false;
    __threadfence();
    double t[N];
#pragma unroll
    for (int n = 0; n < N; n++) t[n] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
#pragma unroll
        for (int n = 0; n < N; n++) t[n] += __ldcg(partials + (size_t)b * N + n);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int n = 0; n < N; n++) {
        double x = t[n];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if (lane == 0) sh[n * nw + warp] = x;
    }
    __syncthreads();
    if (threadIdx.x != 0) return false;
#pragma unroll
    for (int n = 0; n < N; n++) {
        double x = 0.0;
        for (int w = 0; w < nw; w++) x += sh[n * nw + w];
        out[n] = x;
    }
    *counter = 0u;
    return true;
}

// ------------------------------------------------------------------------------------------------
// buffer of device memory owned by the context
// ------------------------------------------------------------------------------------------------
struct DevBuf { void* p = nullptr; size_t bytes = 0; };

constexpr int kWaitPolls = 1 << 21;

}  // namespace rm

// ------------------------------------------------------------------------------------------------
// the context
// ------------------------------------------------------------------------------------------------
struct rmhmc_ctx {
    int device = 0;
    rm::Geom g{};
    std::string err;
    // links
    double2* u64 = nullptr;
    float4* u32a = nullptr;
    float2* u32b = nullptr;
    bool links_valid = false;
    unsigned long long link_gen = 1;   // bumped whenever the internal link copies change
    unsigned long long import_gen = 0; // bumped by every import of the caller's links
    // import_gen whose links were last looked at, and whether they are unitary, for float64 and float32 (links_su3)
    unsigned long long su3_gen[2] = {0, 0};
    bool su3[2] = {false, false};
    bool own_capture = false;          // the library's streams are capturing a trajectory
    bool links_in_graph = false;       // a graph of the caller's imports links: the host no longer sees when they change
    unsigned long long adj_gen = 0;    // link_gen the float32-pair adjoint table was built for
    unsigned long long adj64_gen = 0;  // and the float64 one
    bool loops_off = false;            // no memory for the gauge force's loops
    bool adj64_off = false;            // no memory for the float64 one
    // reductions
    double* red_partials = nullptr;   // [kRedSlots][max_blocks * 2]
    unsigned* red_counters = nullptr; // [kRedSlots]
    double* red_out = nullptr;        // [kRedSlots][8]
    int max_blocks = 0;
    double* h_pinned = nullptr;       // pinned host staging (kPinned doubles)
    // workspace pool
    std::map<std::string, rm::DevBuf> bufs;
    size_t num_sms = 0;
    size_t smem_optin = 0;              // most shared memory a block may have
    // pinned upload ring (kRingSlots slots of kRingBytes) and the events that guard slot reuse
    char* ring = nullptr;
    cudaEvent_t ring_ev[4] = {};
    unsigned ring_idx = 0;
    // events of the look-behind convergence check of the Krylov loop, and the iteration count of the
    // last run per (precision, shift, tolerance, cap)
    cudaEvent_t kr_ev[2] = {};
    std::map<std::string, int> kr_pred;
    // CUDA graph of the molecular dynamics: executable, the parameters and workspace generation it was
    // captured for, capture streams, and whether graphs are used (fallback reason when not)
    cudaGraphExec_t md_exec = nullptr;
    std::string md_key;
    bool md_cg_run = false;             // its Krylov runs are cooperative (one kernel each)
    bool md_loops = false;              // its gauge forces come from shared loops
    unsigned long long md_gen = 0;
    unsigned long long ws_gen = 0;      // bumped whenever a workspace buffer is (re)allocated
    cudaStream_t cap_st[3] = {};
    bool use_graphs = true;
    std::string graph_note;
    // autotuned stencil shapes per (precision bytes * 100 + link format): components per lane, block size
    std::map<int, std::pair<int, int>> tune;
    std::set<int> pinned;              // keys of tune that the caller set (rmhmc_set_stencil_shape)
    // kernel of the kinetic-force contraction (rmhmc_set_stencil_shape, RMHMC_SHAPE_KFORCE): 4 the fused one (the default),
    // 0 four lanes per link
    int lg_mode = 4;
    // float64 link update in float-float arithmetic (rmhmc_set_stencil_shape, RMHMC_SHAPE_LINKUPDATE)
    bool link_update_ff = true;
    // gauge force from shared loops, float64 stencils from the table of adjoint matrices (RMHMC_SHAPE_LOOPS, _TABLE)
    bool use_loops = true, use_table = true;
    // z-extent of the multi-field adjoint kernel's slabs (rmhmc_set_stencil_shape, RMHMC_SHAPE_ADJOINT); 0 chosen
    // from the lattice and the field count
    int ad_slab = 0;
    // set when the device refuses the cooperative CG run
    bool cg_run_off = false;
    // polls of a device-side wait before it gives up (rmhmc_set_wait_limit)
    int wait_limit = rm::kWaitPolls;
    // incremented by every rmhmc_set_stencil_shape and rmhmc_set_wait_limit: part of the key of a captured trajectory graph
    int shape_gen = 0;
    std::string tune_report;
    // counters: kernels launched; optional timing of the conjugate-gradient stencil launches
    long long launches = 0;
    long long krylov_iters = 0;
    bool prof = false;
    long long prof_count = 0;
    double prof_ms = 0.0;
    cudaEvent_t* prof_ev = nullptr;   // 2 * kProfEvents events, created when profiling is switched on
};

namespace rm {

constexpr int kPinned = 1 << 16;
constexpr int kRingSlots = 4;
constexpr int kProfEvents = 256;
constexpr size_t kRingBytes = 1 << 20;
// copy host bytes to device memory asynchronously through the pinned ring
int upload(rmhmc_ctx* ctx, void* dst, const void* src, size_t bytes, cudaStream_t st);

int set_err(rmhmc_ctx* ctx, int code, const char* fmt, ...);
int cuda_check(rmhmc_ctx* ctx, cudaError_t e, const char* what);
void* workspace(rmhmc_ctx* ctx, const char* name, size_t bytes, int* status);
// a form that the context does without for want of memory (&ctx->adj64_off or &ctx->loops_off), noted in rmhmc_tuning
void without(rmhmc_ctx* ctx, bool* off);
int import_links(rmhmc_ctx* ctx, const double* U, cudaStream_t st);
int ensure_links(rmhmc_ctx* ctx, const double* U, cudaStream_t st);
void links_imported(rmhmc_ctx* ctx);
inline size_t field_elems(const rmhmc_ctx* ctx) { return (size_t)ctx->g.V * 32; }
inline int site_blocks(const rmhmc_ctx* ctx) { return (ctx->g.V + kBlock - 1) / kBlock; }
// blocks of the stencil kernels: four lanes per site (one per field component mu)
inline int lane_blocks(const rmhmc_ctx* ctx) { return (int)(((size_t)ctx->g.V * 4 + kBlock - 1) / kBlock); }
// grids of the reduced kernels hold at most one full wave (2048 threads per SM) and stride over the rest:
// the deterministic final sum then has at most 16 * SMs block partials.  Above one wave the grid is trimmed
// so that every thread strides the same number of times (no tail pass with a partly idle grid, whose blocks
// would wait at the final reduction)
inline int capped_grid(const rmhmc_ctx* ctx, size_t threads, int block) {
    const size_t need = (threads + block - 1) / block;
    const size_t cap = (size_t)ctx->num_sms * (2048 / block);
    if (need <= cap) return (int)std::max<size_t>(1, need);
    const size_t passes = (need + cap - 1) / cap;
    const size_t sms = std::max<size_t>(1, ctx->num_sms);
    const size_t g = (need + passes - 1) / passes;
    return (int)std::min(cap, (g + sms - 1) / sms * sms);   // whole blocks per SM
}
inline Links64 links64(const rmhmc_ctx* ctx) { return Links64{ctx->u64, ctx->g.V, nullptr}; }
// whether st is being captured into a graph of the caller's: such a graph reads the links it finds when it is replayed, so
// that it must not hold what the host derived from those of today (the float64 table, whether they are unitary)
inline bool caller_captures(const rmhmc_ctx* ctx, cudaStream_t st) {
    if (ctx->own_capture) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) cudaGetLastError();   // (the legacy stream beside a capture)
    return cs == cudaStreamCaptureStatusActive;
}
inline bool links_tracked(const rmhmc_ctx* ctx, cudaStream_t st) { return !ctx->links_in_graph && !caller_captures(ctx, st); }
// the links with their float64 adjoint table, built if the links changed since; ad is null where a table is not used
// (more than kAdTableMax sites, no memory for it, links that change behind the host's back)
constexpr int kAdTableMax = 1 << 22;   // 2 KB a site
int links64_adjoint(rmhmc_ctx* ctx, Links64* U, cudaStream_t st);
// ensure_links for a call that goes on to use the table (table): on up to kImportTableMax sites new links and their table come
// from one launch (float64 lap_apply with links, two launches -> one: 4^4 37.0 -> 30.9 us, 8^4 46.2 -> 41.1, 12^4 153 -> 148;
// by 3x3 products 39.0, 40.3 and 162 us)
constexpr int kImportTableMax = 1 << 15;
int ensure_links_table(rmhmc_ctx* ctx, const double* U, bool table, cudaStream_t st);
inline Links32 links32(const rmhmc_ctx* ctx) { return Links32{ctx->u32a, ctx->u32b, ctx->g.V}; }
double* red_slot_partials(rmhmc_ctx* ctx, int slot);
unsigned* red_slot_counter(rmhmc_ctx* ctx, int slot);
double* red_slot_out(rmhmc_ctx* ctx, int slot);
// copy n doubles from device to host through pinned memory and synchronise the stream
int fetch(rmhmc_ctx* ctx, const double* dsrc, double* hdst, int n, cudaStream_t st);

}  // namespace rm

#define RM_CHECK(ctx, call)                                                  \
    do {                                                                     \
        cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess) return rm::cuda_check((ctx), e_, #call);      \
    } while (0)
#define RM_LAUNCH_CHECK(ctx) RM_CHECK(ctx, cudaGetLastError())
#define RM_TRY(x)                     \
    do {                              \
        int s_ = (x);                 \
        if (s_ != RMHMC_OK) return s_; \
    } while (0)
