// A whole conjugate-gradient run (krylov.cu: q_k = (A + sigma) r_k + beta q_{k-1}, r_{k+1} = r_k - alpha_k q_k, every
// r_k kept) as one cooperative launch, for lattices whose q fits in the shared memory of the chip.
//
// What bounds it.  On a small lattice an iteration of the two-kernel form is latency, not work: at 8^4 the stencil launch
// takes 11 us and the update 7 us, most of it the ends of the kernels (block sums, a ticket, the last block's sum of
// all partials, the next launch).  Here the blocks stay: two grid barriers an iteration, q in shared memory,
// r_{k+1} published to L2 for the neighbours, every block adding up the same partials in the same order, so that all take
// the same decisions without a broadcast.  The run starts from the caller's field and needs no host or graph loop.
// A mixed kinetic evaluation at tolerance 3e-7, two-kernel form -> this: 8^4 458 -> 333 us (10.5 us an iteration),
// 13 x 11 x 9 x 17 695 -> 508 us, 16^4 977 -> 773 us, 16^3 x 32 1430 -> 1145 us, 16^2 x 32^2 2396 -> 2223 us; float64 at 16^4
// 27.0 -> 26.1 ms.
//
// Work: units of 32 consecutive sites and one component, a contiguous range of units per block, one warp per unit.
#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "krylov.cuh"
#include "stencil.cuh"
#include "tune.cuh"

namespace rm {

// Grid barrier with the sum of the blocks' values v (valid in thread 0) returned to all threads; the blocks' global
// writes before it are visible after it.  The partials are added by the first warp of every block in a fixed order.
// bar[0] counts arrivals (wrapping), bar[1] is the generation; part holds two arrays of gridDim.x, used in turn (a block
// that runs ahead writes the other one, and comes back to this one only after all have left it).  Returns false in
// every thread of a block whose wait ran out.  (Polling the partials themselves, tagged with the generation, saves the
// counter's round trip but floods L2: 350 against 333 us for a kinetic evaluation at 8^4.)  limit: polls before a block
// gives up (the default, kWaitPolls, is about two seconds at an L2 round trip each); a cooperative launch has all its
// blocks resident, so that only a lost block can run it out.
struct GridSum {
    unsigned* bar;
    double* part;
    int limit;
    unsigned gen;
    __device__ __forceinline__ GridSum(unsigned* b, double* p, int l) : bar(b), part(p), limit(l) {
        gen = *reinterpret_cast<volatile unsigned*>(bar + 1);   // cannot change before this block has arrived
    }
    __device__ __forceinline__ bool operator()(double v, double& sum, double* sh) {
        __shared__ int failed;
        double* const p = part + (gen & 1) * gridDim.x;
        if (threadIdx.x == 0) {
            p[blockIdx.x] = v;
            failed = 0;
            __threadfence();
            if (atomicInc(bar, gridDim.x - 1) == gridDim.x - 1) {
                __threadfence();
                asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(bar + 1), "r"(gen + 1) : "memory");
            } else {
                unsigned now = gen;
                for (int n = 0; n < limit && now == gen; n++)
                    asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(now) : "l"(bar + 1) : "memory");
                if (now == gen) failed = 1;
            }
            __threadfence();
        }
        gen++;
        __syncthreads();
        if (failed) return false;
        if (threadIdx.x < 32) {
            double t = 0.0;
            for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) t += __ldcg(p + b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (threadIdx.x == 0) *sh = t;
        }
        __syncthreads();
        sum = *sh;
        return true;
    }
};

// field values that other blocks write during the kernel: ordinary loads, ordered by the barriers
__device__ __forceinline__ void load4_shared(const float* p, float* x) {
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void load4_shared(const double* p, double* x) {
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(x[0]), "=d"(x[1]) : "l"(p) : "memory");
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(x[2]), "=d"(x[3]) : "l"(p + 2) : "memory");
}
template <typename T> struct SrcShared {
    const T* X;
    int V;
    __device__ __forceinline__ void operator()(int s, int mu, T* x) const {
        load4_shared(plane_at(X, V, s, 2 * mu), x);
        load4_shared(plane_at(X, V, s, 2 * mu + 1), x + 4);
    }
};

// a thread's chunk of four values of q in shared memory
__device__ __forceinline__ void q_load(const float* p, float* x) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void q_load(const double* p, double* x) {
    const double2 v = reinterpret_cast<const double2*>(p)[0], w = reinterpret_cast<const double2*>(p)[1];
    x[0] = v.x; x[1] = v.y; x[2] = w.x; x[3] = w.y;
}

// sum over the block of the lanes' values, in thread 0 (float lanes add within their warp in float, as the kernels of
// the two-kernel form do)
template <typename T> __device__ __forceinline__ double block_total(T x, double* shw) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0) shw[threadIdx.x >> 5] = (double)x;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += shw[w];
    return t;
}

// NMU: 1, or 0 with the neighbours of a unit loaded ahead (hop_sum_shape); BLOCK: largest block; iters (nullable) counts
// iterations.  flags[0] is the largest of what the blocks say, 4 (a barrier gave up) above every outcome of block 0: a block
// can give up on a barrier that the others still pass.  (Block 0 clears it first.  A 4 from before that is lost only
// where all blocks then pass the first barrier, and with it the run if it ends there: its work is complete.)
// status (nullable): the trajectory's status word.  After a run that gave up the barrier's counter is off until the host
// clears it, so that the graph's later runs return at once.
template <typename T, typename TI, int NMU, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 1)
    k_cg_run(Geom g, typename LinksOf<T>::type U, const TI* __restrict__ b, T* R, size_t fs, T diag, int* flags, double* vals,
             int maxit, double tol2, long long* iters, int units_per_block, double* part, unsigned* bar, int limit,
             const int* status) {
    // float32 blocks of 256 and 768 threads have a unit per warp and nothing to add up
    using Sum = std::conditional_t<sizeof(T) == 4 && BLOCK == 512, CompSum, PlainSum<T>>;
    extern __shared__ __align__(16) unsigned char cgs[];
    T* const qs = reinterpret_cast<T*>(cgs);   // [item][chunk][thread][4]
    __shared__ double shw[BLOCK / 32], sh[3];
    GridSum gsum(bar, part, limit);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int nunit = (g.V + 31) / 32 * 4;
    const int u0 = blockIdx.x * units_per_block + warp, u1 = min(nunit, (blockIdx.x + 1) * units_per_block);
    double* const rho = vals;
    double* const gamma = vals + (maxit + 1);
    double* const alpha = gamma + maxit;
    double* const beta = alpha + maxit;
    const bool writer = blockIdx.x == 0 && threadIdx.x == 0;
    if (status && *status == kStatusGaveUp) return;   // flags still say so
    if (writer) flags[0] = flags[1] = 0;   // readers of the vectors' number see 0 or the run's
    // r_0 = b in T, |r_0|^2 accurate to float64
    double rr;
    {
        SumSq32 sf;
        double sd = 0.0;
        for (int u = u0; u < u1; u += wpb) {
            const int s = u / 4 * 32 + lane, mu = u & 3;
            if (s >= g.V) continue;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                TI v[4];
                T x[4];
                load4(b + (size_t)s * 32 + mu * 8 + h * 4, v);
                if constexpr (sizeof(T) == 4) to_f32_n(v, x);
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    if constexpr (sizeof(T) == 4) {
                        sf.add(x[a]);
                    } else {
                        x[a] = v[a];
                        sd = fma(x[a], x[a], sd);
                    }
                }
                store4(plane_at(R, g.V, s, 2 * mu + h), x);
            }
        }
        const double t = block_total(sizeof(T) == 4 ? sf.value() : sd, shw);
        if (!gsum(t, rr, sh)) {
            if (threadIdx.x == 0) atomicMax(flags, 4);
            return;
        }
    }
    if (writer) rho[0] = rr;
    const double stop = tol2 * rr;
    int k = 0, done = isfinite(rr) ? (rr == 0.0 ? 1 : 0) : 3;
    double bk = 0.0;
    while (!done) {
        const SrcShared<T> src{R + (size_t)k * fs, g.V};
        T* const rn = R + (size_t)(k + 1) * fs;
        const T bt = (T)bk;
        Sum dot;
        T* q = qs + threadIdx.x * 4;
        for (int u = u0; u < u1; u += wpb, q += 8 * blockDim.x) {
            const int s = u / 4 * 32 + lane, mu = u & 3;
            if (s >= g.V) continue;
            T hc[1][8], x[8], y[8], o[8];
            hop_coefs<T, sizeof(T) == 8 ? kLinkAd : 18, NMU>(g, U, s, mu, src, hc);
            const T(&h)[8] = hc[0];
            src(s, mu, x);
            if (k > 0) {
                q_load(q, o);
                q_load(q + 4 * blockDim.x, o + 4);
            }
            T d = T(0);
#pragma unroll
            for (int a = 0; a < 8; a++) {
                y[a] = fma(T(-0.0625), h[a], diag * x[a]);
                if (k > 0) y[a] = fma(bt, o[a], y[a]);
                d = fma(x[a], y[a], d);
            }
            dot.add(d);
            store4(q, y);
            store4(q + 4 * blockDim.x, y + 4);
        }
        double gm;
        if (!gsum(block_total(dot.value(), shw), gm, sh + 1)) { done = 4; break; }
        const double al = rr / gm;
        const T at = (T)al;
        dot = Sum();
        q = qs + threadIdx.x * 4;
        for (int u = u0; u < u1; u += wpb, q += 8 * blockDim.x) {
            const int s = u / 4 * 32 + lane, mu = u & 3;
            if (s >= g.V) continue;
            T x[8], o[8];
            src(s, mu, x);
            q_load(q, o);
            q_load(q + 4 * blockDim.x, o + 4);
            T d = T(0);
#pragma unroll
            for (int a = 0; a < 8; a++) {
                x[a] = fma(-at, o[a], x[a]);
                d = fma(x[a], x[a], d);
            }
            dot.add(d);
            store4(plane_at(rn, g.V, s, 2 * mu), x);
            store4(plane_at(rn, g.V, s, 2 * mu + 1), x + 4);
        }
        double rn2;
        if (!gsum(block_total(dot.value(), shw), rn2, sh + 2)) { done = 4; break; }
        bk = rn2 / rr;
        if (writer) {
            gamma[k] = gm;
            alpha[k] = al;
            rho[k + 1] = rn2;
            beta[k] = bk;
        }
        rr = rn2;
        k++;
        if (!isfinite(rr) || !isfinite(al)) done = 3;
        else if (rr <= stop) done = 1;
        else if (k >= maxit) done = 2;
    }
    if (done == 4) {
        if (threadIdx.x == 0) atomicMax(flags, 4);
    } else if (writer) {
        flags[1] = k;
        atomicMax(flags, done);
        if (iters) *iters += k;
    }
}

struct CgRunShape { int grid, warps, units, maxw; size_t smem; };

// One block per SM with an equal share of the units.  Up to 8 units a block run a warp each with 255 registers, up to 24 a
// warp each with 80, both loading the neighbours ahead; more go in rounds of 16 warps at 128 registers (16^4, 54 units:
// 765 us a kinetic evaluation against 806 and 809 us in rounds of 24 and 32 warps).  float64 is bound by its arithmetic
// from a few units on: 8 warps of 255 registers.
template <typename T> static CgRunShape cg_run_shape(const rmhmc_ctx* ctx) {
    const int nunit = (ctx->g.V + 31) / 32 * 4, sms = (int)ctx->num_sms;
    CgRunShape s;
    s.units = (nunit + sms - 1) / sms;
    s.grid = (nunit + s.units - 1) / s.units;
    s.maxw = sizeof(T) == 8 || s.units <= 8 ? 8 : s.units <= 24 ? 24 : 16;
    const int items = (s.units + s.maxw - 1) / s.maxw;
    s.warps = (s.units + items - 1) / items;
    s.smem = (size_t)items * s.warps * 32 * 8 * sizeof(T);
    return s;
}

// static shared memory of the kernel (the block's partial sums and the barrier's words), rounded up
constexpr size_t kCgRunStatic = 1024;

// q has to fit next to it: ceil(units / warps) rounds of 1 or 2 KB a warp, which depends on how many SMs share the sites
template <typename T> bool cg_run_fits(const rmhmc_ctx* ctx, bool captured) {
    return !ctx->cg_run_off && (captured || !ctx->prof) && !ctx->pinned.count(10000 + (int)sizeof(T) * 100 + 18) &&
           ctx->g.V <= (sizeof(T) == 4 ? kCgRunMax32 : kCgRunMax64) &&
           cg_run_shape<T>(ctx).smem + kCgRunStatic <= ctx->smem_optin;
}

// the barrier words (64 bytes; they wrap and count on from launch to launch) and two arrays of partials
int cg_run_reset(rmhmc_ctx* ctx, cudaStream_t st) {
    auto it = ctx->bufs.find("cg_run");
    if (it != ctx->bufs.end() && it->second.p) RM_CHECK(ctx, cudaMemsetAsync(it->second.p, 0, 64, st));
    return RMHMC_OK;
}

int cg_run_prepare(rmhmc_ctx* ctx, unsigned** bar) {
    int status = RMHMC_OK;
    const unsigned long long gen = ctx->ws_gen;
    void* p = workspace(ctx, "cg_run", 64 + sizeof(double) * 2 * ctx->num_sms, &status);
    if (!p) return status;
    if (ctx->ws_gen != gen) {   // a new buffer
        RM_CHECK(ctx, cudaMemset(p, 0, 64));
        RM_CHECK(ctx, cudaDeviceSynchronize());   // the caller's stream may not follow the legacy stream
    }
    if (bar) *bar = (unsigned*)p;
    return RMHMC_OK;
}

template <typename T, typename TI>
int cg_run_launch(rmhmc_ctx* ctx, const typename LinksOf<T>::type& links, const TI* b, T* R, double diag, int* flags,
                  double* vals, int maxit, double tol2, long long* iters, cudaStream_t st, const int* status) {
    const CgRunShape s = cg_run_shape<T>(ctx);
    unsigned* bar = nullptr;
    RM_TRY(cg_run_prepare(ctx, &bar));
    double* part = (double*)((char*)bar + 64);
    typename LinksOf<T>::type U = links;
    Geom g = ctx->g;
    size_t fs = field_elems(ctx);
    T d = (T)diag;
    int units = s.units, limit = ctx->wait_limit;
    void* args[] = {&g, &U, &b, &R, &fs, &d, &flags, &vals, &maxit, &tol2, &iters, &units, &part, &bar, &limit, &status};
    const void* kern = (const void*)k_cg_run<T, TI, sizeof(T) == 8 ? 1 : 0, 256>;
    if constexpr (sizeof(T) == 4) {
        if (s.maxw == 24) kern = (const void*)k_cg_run<T, TI, 0, 768>;
        if (s.maxw == 16) kern = (const void*)k_cg_run<T, TI, 1, 512>;
    }
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
    const bool refused = e != cudaSuccess;
    if (!refused) e = cudaLaunchCooperativeKernel(kern, dim3(s.grid), dim3(s.warps * 32), args, s.smem, st);
    if (refused || e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        // fewer SMs than the device reports are ours (a partitioned GPU): the two-kernel form from here on
        cudaGetLastError();
        ctx->cg_run_off = true;
        return RMHMC_OK;
    }
    RM_CHECK(ctx, e);
    ++ctx->launches;
    return RMHMC_OK;
}

template bool cg_run_fits<float>(const rmhmc_ctx*, bool);
template bool cg_run_fits<double>(const rmhmc_ctx*, bool);
template int cg_run_launch<float, float>(rmhmc_ctx*, const Links32&, const float*, float*, double, int*, double*, int, double,
                                         long long*, cudaStream_t, const int*);
template int cg_run_launch<float, double>(rmhmc_ctx*, const Links32&, const double*, float*, double, int*, double*, int, double,
                                          long long*, cudaStream_t, const int*);
template int cg_run_launch<double, double>(rmhmc_ctx*, const Links64&, const double*, double*, double, int*, double*, int,
                                           double, long long*, cudaStream_t, const int*);

}  // namespace rm
