// Gauge force and action from shared loops (Sec. 2; gauge.cu has the definitions): every plaquette and rectangle is
// multiplied out once and its coefficients are carried to the links it holds, instead of a staple product per link.
//
// With C_mn(x) = P Q^dag, P = U_m(x) U_n(x+m), Q = U_n(x) U_m(x+n), the plaquette based at x (C_nm = C_mn^dag), the long
// rectangle is R_mn(x) = [U_m(x) C_mn(x+m) U_m(x)^dag] C_mn(x).  A loop based at the far end y of a step along its own side is
// the loop conjugated by the link of that step, so that its coefficients (k of -i(C - C^dag)/2, r of R) move by
//   (T_d f)(y) = coefficients of U_d(y-d)^dag f(y-d) U_d(y-d),   108 FMA.
// Sorting the loops that hold U_m(y) by their base point gives, with -(beta/6) in front,
//   F_m = sum_n { c0 (1 - T_n) k_mn + c1 [ (1 + T_m)(1 - T_n) r_mn - r_nm + T_n T_n r_nm ] }(y).
// Per site that is 6 x 324 + 12 x 108 = 3240 FMA for the plaquette action and about 10,200 with rectangles, where the
// staples take 5616 and 36,700; the action reads the traces of the same products.  The transport and the rectangles use
// U U^dag = 1: links that are not unitary to 2^-43 (say, read from single precision; 2^-20 for the float32 force) keep the
// staples, which take any matrices (links_su3; once per import, 24^3 x 48: 170 us, float32 45 us).
//
// float64 (0.55 TFMA/s) is bound by the operations, float32 was by re-reading the links of every staple from L2.  Measured at
// 24^3 x 48, float32 Iwasaki force with its float64 action: 9.70 ms with staples, 6.84 ms here; float64 Wilson flow at 16^4,
// 8 steps: 23.8 -> 15.6 ms.
#include <algorithm>

#include "df.cuh"
#include "krylov.cuh"
#include "ops.cuh"
#include "stencil.cuh"

namespace rm {

template <typename T> struct C2;
template <> struct C2<float> { using type = float2; };
template <> struct C2<double> { using type = double2; };

// plane index of the pair m < n, and of the ordered pair (m, n)
__host__ __device__ __forceinline__ int pair_of(int m, int n) { return m * (7 - m) / 2 + n - m - 1; }
__device__ __forceinline__ int ordered_of(int m, int n) { return 3 * m + (n < m ? n : n - 1); }

template <typename T> __device__ __forceinline__ mat3<T> load_mat(const typename C2<T>::type* M, int V, int p, int s) {
    mat3<T> m;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        const typename C2<T>::type v = M[((size_t)p * 9 + e) * V + s];
        m.e[e / 3][e % 3] = cmk<T>(v.x, v.y);
    }
    return m;
}
// field f of a set of chunk-planar coefficient fields
template <typename T> __device__ __forceinline__ void load_f(const T* K, int V, int f, int s, T* x) {
    load_plane8(K + (size_t)f * 8 * V, V, s, 0, x);
}
template <typename T> __device__ __forceinline__ void store_f(T* K, int V, int f, int s, const T* x) {
    T* p = K + (size_t)f * 8 * V;
    store4(plane_at(p, V, s, 0), x);
    store4(plane_at(p, V, s, 1), x + 4);
}
template <typename T> __device__ __forceinline__ mat3<T> link(const typename LinksOf<T>::type& U, int s, int mu) {
    return LinkLoad<T, 18>::load(U, s, mu);
}

// C_mn(x) of every pair: the matrices to M, the coefficients to K (either may be null); ACT: sums of 1 - ReTr C/3 and of
// ReTr C/3 to out
template <typename T, bool ACT>
__global__ void __launch_bounds__(kBlock) k_plaquettes(Geom g, typename LinksOf<T>::type U, typename C2<T>::type* M, T* K,
                                                       double* partials, unsigned* counter, double* out) {
    double act = 0.0, plaq = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 6 * g.V; i += gridDim.x * blockDim.x) {
        const int p = i / g.V, s = i - p * g.V;
        const int m = p < 3 ? 0 : p < 5 ? 1 : 2, n = p < 3 ? p + 1 : p < 5 ? p - 1 : 3;
        const mat3<T> P = m_mul(link<T>(U, s, m), link<T>(U, step_site(g, s, m, 1), n));
        const mat3<T> Q = m_mul(link<T>(U, s, n), link<T>(U, step_site(g, s, n, 1), m));
        if (M || K) {
            const mat3<T> C = m_mul_nd(P, Q);
            if (M)
#pragma unroll
                for (int e = 0; e < 9; e++) {
                    typename C2<T>::type v;
                    v.x = C.e[e / 3][e % 3].re;
                    v.y = C.e[e / 3][e % 3].im;
                    M[((size_t)p * 9 + e) * g.V + s] = v;
                }
            if (K) {
                T k[8];
                antiherm_coef(C, k);
                store_f(K, g.V, p, s, k);
            }
        }
        if (ACT) {
            T tr = T(0);
#pragma unroll
            for (int e = 0; e < 9; e++)
                tr = fma(P.e[e / 3][e % 3].re, Q.e[e / 3][e % 3].re, fma(P.e[e / 3][e % 3].im, Q.e[e / 3][e % 3].im, tr));
            const double rt = (double)tr / 3.0;
            act += 1.0 - rt;
            plaq += rt;
        }
    }
    if (ACT) {
        __shared__ double sh[2 * (kBlock / 32)];
        double v[2] = {act, plaq};
        block_sum<2>(v, sh);
        grid_sum_finish<2>(v, partials, counter, out, gridDim.x, blockIdx.x, sh);
    }
}

// r_mn(x) of every ordered pair (m the long side) to K (null: none); ACT: sum of 1 - ReTr R/3 to out
template <typename T, bool ACT>
__global__ void __launch_bounds__(kBlock) k_rectangles(Geom g, typename LinksOf<T>::type U, const typename C2<T>::type* M, T* K,
                                                       double* partials, unsigned* counter, double* out) {
    double act = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 12 * g.V; i += gridDim.x * blockDim.x) {
        const int o = i / g.V, s = i - o * g.V;
        const int m = o / 3, j = o - 3 * m, n = j < m ? j : j + 1;
        const int p = m < n ? pair_of(m, n) : pair_of(n, m);
        const mat3<T> u = link<T>(U, s, m);
        // for m > n the planes hold C_nm = C_mn^dag: R^dag = C_nm(x) [U C_nm(x+m) U^dag]
        mat3<T> t = m_mul_nd(m_mul(u, load_mat<T>(M, g.V, p, step_site(g, s, m, 1))), u);
        const mat3<T> c = load_mat<T>(M, g.V, p, s);
        if (K) {
            const mat3<T> R = m < n ? m_mul(t, c) : m_mul(c, t);
            T k[8];
            antiherm_coef(R, k);
            if (m > n)
#pragma unroll
                for (int a = 0; a < 8; a++) k[a] = -k[a];
            store_f(K, g.V, o, s, k);
        }
        if (ACT) {
            T tr = T(0);   // ReTr(t c)
#pragma unroll
            for (int a = 0; a < 3; a++)
#pragma unroll
                for (int b = 0; b < 3; b++) tr = fma(t.e[a][b].re, c.e[b][a].re, fma(-t.e[a][b].im, c.e[b][a].im, tr));
            act += 1.0 - (double)tr / 3.0;
        }
    }
    if (ACT) {
        __shared__ double sh[kBlock / 32];
        double v[1] = {act};
        block_sum<1>(v, sh);
        grid_sum_finish<1>(v, partials, counter, out, gridDim.x, blockIdx.x, sh);
    }
}

// acc += (T_d f)(s) from the field f at y = s - d
template <typename T>
__device__ __forceinline__ void add_moved(herm<T>& acc, const mat3<T>& u, const T* f) {
    acc_udxu_tl(acc, u, coef_to_herm2(f));
}

// what the rectangles move twice, from k and r: c1 G_m = c1 sum_n (1 - T_n) r_mn (fields 12 + m), and
// w_mn = -c0 k_mn + c1 T_n r_nm (fields ordered_of(m, n)).  Lane: site, direction m per blockIdx.y
template <typename T>
__global__ void __launch_bounds__(kBlock) k_rect_move(Geom g, typename LinksOf<T>::type U, const T* __restrict__ K,
                                                      const T* __restrict__ R, T* __restrict__ W, T c0, T c1) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
    if (s >= g.V) return;
    T G[8];
#pragma unroll
    for (int a = 0; a < 8; a++) G[a] = T(0);
    for (int n = 0; n < 4; n++) {
        if (n == m) continue;
        const int y = step_site(g, s, n, -1);
        const mat3<T> u = link<T>(U, y, n);
        T f[8], r[8], h[8];
        herm<T> e = h_zero<T>();
        load_f(R, g.V, ordered_of(m, n), y, f);
        add_moved(e, u, f);
        herm2_to_coef_tl(e, h);
        load_f(R, g.V, ordered_of(m, n), s, r);
#pragma unroll
        for (int a = 0; a < 8; a++) G[a] = fma(c1, r[a] - h[a], G[a]);
        e = h_zero<T>();
        load_f(R, g.V, ordered_of(n, m), y, f);
        add_moved(e, u, f);
        herm2_to_coef_tl(e, h);
        T k[8];
        load_f(K, g.V, m < n ? pair_of(m, n) : pair_of(n, m), s, k);
        const T c = m < n ? c0 : -c0;
#pragma unroll
        for (int a = 0; a < 8; a++) h[a] = fma(c1, h[a], -c * k[a]);
        store_f(W, g.V, ordered_of(m, n), s, h);
    }
    store_f(W, g.V, 12 + m, s, G);
}

// the force: plaquette action (RECT false: k in K) or with rectangles (k, r and the fields of k_rect_move)
template <typename T, bool RECT>
__global__ void __launch_bounds__(kBlock) k_loop_force(Geom g, typename LinksOf<T>::type U, const T* __restrict__ K,
                                                       const T* __restrict__ R, const T* __restrict__ W, T c0, T c1, double scale,
                                                       double* __restrict__ F) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x, m = blockIdx.y;
    if (s >= g.V) return;
    T v[8], f[8];
#pragma unroll
    for (int a = 0; a < 8; a++) v[a] = T(0);
    herm<T> e = h_zero<T>();
    if (RECT) {
        load_f(W, g.V, 12 + m, s, v);
        const int y = step_site(g, s, m, -1);
        load_f(W, g.V, 12 + m, y, f);
        add_moved(e, link<T>(U, y, m), f);
    }
    for (int n = 0; n < 4; n++) {
        if (n == m) continue;
        const int y = step_site(g, s, n, -1);
        const int p = m < n ? pair_of(m, n) : pair_of(n, m);
        const T c = m < n ? c0 : -c0;
        load_f(K, g.V, p, s, f);
#pragma unroll
        for (int a = 0; a < 8; a++) v[a] = fma(c, f[a], v[a]);
        if (RECT) {
            load_f(R, g.V, ordered_of(n, m), s, f);
#pragma unroll
            for (int a = 0; a < 8; a++) v[a] = fma(-c1, f[a], v[a]);
            load_f(W, g.V, ordered_of(m, n), y, f);
        } else {
            load_f(K, g.V, p, y, f);
#pragma unroll
            for (int a = 0; a < 8; a++) f[a] *= -c;
        }
        add_moved(e, link<T>(U, y, n), f);
    }
    T h[8];
    herm2_to_coef_tl(e, h);
    double* out = F + (size_t)s * 32 + m * 8;
#pragma unroll
    for (int a = 0; a < 8; a++) out[a] = scale * (double)(v[a] + h[a]);
}

// scratch: matrices of 6 plaquettes, coefficients of 6 + 12 loops and 16 moved fields
template <typename T> struct LoopBufs {
    typename C2<T>::type* M = nullptr;
    T *K = nullptr, *R = nullptr, *W = nullptr;
};
template <typename T> static int loop_bufs(rmhmc_ctx* ctx, bool rect, bool force, LoopBufs<T>& b) {
    int status = RMHMC_OK;
    const size_t V = ctx->g.V;
    const bool f32 = sizeof(T) == 4;
    if (rect) {
        b.M = (typename C2<T>::type*)workspace(ctx, f32 ? "gl_m32" : "gl_m64", sizeof(T) * 2 * 54 * V, &status);
        if (!b.M) return status;
    }
    if (!force) return RMHMC_OK;
    const size_t nf = rect ? 34 : 6;
    T* p = (T*)workspace(ctx, f32 ? (rect ? "gl_r32" : "gl_k32") : (rect ? "gl_r64" : "gl_k64"), sizeof(T) * 8 * nf * V, &status);
    if (!p) return status;
    b.K = p;
    b.R = p + 6 * 8 * V;
    b.W = p + 18 * 8 * V;
    return RMHMC_OK;
}

template <typename T>
static int loops_t(rmhmc_ctx* ctx, const typename LinksOf<T>::type& U, double beta, double c1, double* F, bool act,
                   cudaStream_t st) {
    const bool rect = c1 != 0.0;
    const double c0 = 1.0 - 8.0 * c1;
    LoopBufs<T> b;
    RM_TRY((loop_bufs<T>(ctx, rect, F != nullptr, b)));
    double* part = red_slot_partials(ctx, kSlotLoops);
    unsigned* cnt = red_slot_counter(ctx, kSlotLoops);
    double* out = red_slot_out(ctx, kSlotLoops);
    // blocks: at most what the partials of the slots from kSlotLoops on hold
    auto grid = [&](int loops) {
        return std::min(capped_grid(ctx, (size_t)loops * ctx->g.V, kBlock), ctx->max_blocks * (kSlotLoopsEnd - kSlotLoops));
    };
    if (act) k_plaquettes<T, true><<<grid(6), kBlock, 0, st>>>(ctx->g, U, b.M, b.K, part, cnt, out);
    else k_plaquettes<T, false><<<grid(6), kBlock, 0, st>>>(ctx->g, U, b.M, b.K, nullptr, nullptr, nullptr);
    ++ctx->launches;
    if (rect) {
        if (act) k_rectangles<T, true><<<grid(12), kBlock, 0, st>>>(ctx->g, U, b.M, b.R, part, cnt, out + 2);
        else k_rectangles<T, false><<<grid(12), kBlock, 0, st>>>(ctx->g, U, b.M, b.R, nullptr, nullptr, nullptr);
        ++ctx->launches;
    }
    if (F) {
        const dim3 sites(site_blocks(ctx), 4);
        const double scale = -(double)((T)beta / T(6));
        if (rect) {
            k_rect_move<T><<<sites, kBlock, 0, st>>>(ctx->g, U, b.K, b.R, b.W, (T)c0, (T)c1);
            k_loop_force<T, true><<<sites, kBlock, 0, st>>>(ctx->g, U, b.K, b.R, b.W, (T)c0, (T)c1, scale, F);
            ++ctx->launches;
        } else {
            k_loop_force<T, false><<<sites, kBlock, 0, st>>>(ctx->g, U, b.K, nullptr, nullptr, (T)c0, T(0), scale, F);
        }
        ++ctx->launches;
    }
    RM_LAUNCH_CHECK(ctx);
    return RMHMC_OK;
}

// Number of links with an entry of U U^dag - 1 above 2^-43 or not a number.  Thread per link; float-float (errors of about
// 1e-14), since float64 would take 0.35 ms at 24^3 x 48 (this: 0.17 ms).
__global__ void __launch_bounds__(kBlock) k_su3_check(Links64 U, double* partials, unsigned* counter, double* out) {
    int bad = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 4 * U.V; i += gridDim.x * blockDim.x) {
        const int mu = i / U.V, s = i - mu * U.V;
        cdfl u[9];
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const double2 v = __ldg(U.u + (size_t)(mu * 9 + e) * U.V + s);
            u[e] = cdf_make(df_split(v.x), df_split(v.y));
        }
        bool ok = true;
        auto within = [&](dfl x) { ok = ok && fabsf(x.hi + x.lo) <= 0x1p-43f; };
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = a; b < 3; b++) {
                cdfl t = cdf_mul(u[3 * a], cdf_conj(u[3 * b]));
                t = cdf_add(t, cdf_mul(u[3 * a + 1], cdf_conj(u[3 * b + 1])));
                t = cdf_add(t, cdf_mul(u[3 * a + 2], cdf_conj(u[3 * b + 2])));
                within(a == b ? df_sub(t.re, df_make(1.f, 0.f)) : t.re);
                if (a != b) within(t.im);
            }
        bad += !ok;
    }
    __shared__ double sh[kBlock / 32];
    double v[1] = {(double)bad};
    block_sum<1>(v, sh);
    grid_sum_finish<1>(v, partials, counter, out, gridDim.x, blockIdx.x, sh);
}

// the same of the float32 copies, above 2^-20 (the sums here are off by less than 2^-21)
__global__ void __launch_bounds__(kBlock) k_su3_check32(Links32 U, double* partials, unsigned* counter, double* out) {
    int bad = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 4 * U.V; i += gridDim.x * blockDim.x) {
        const int mu = i / U.V, s = i - mu * U.V;
        const mat3<float> u = LinkLoad<float, 18>::load(U, s, mu);
        const mat3<float> p = m_mul_nd(u, u);
        bool ok = true;
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const cplx<float> z = p.e[e / 3][e % 3];
            ok = ok && fabsf(z.re - (e % 4 == 0 ? 1.f : 0.f)) <= 0x1p-20f && fabsf(z.im) <= 0x1p-20f;
        }
        bad += !ok;
    }
    __shared__ double sh[kBlock / 32];
    double v[1] = {(double)bad};
    block_sum<1>(v, sh);
    grid_sum_finish<1>(v, partials, counter, out, gridDim.x, blockIdx.x, sh);
}

int su3_check_launch(rmhmc_ctx* ctx, int prec, cudaStream_t st) {
    const int grid = capped_grid(ctx, (size_t)4 * ctx->g.V, kBlock);
    double* part = red_slot_partials(ctx, kSlotSu3);
    unsigned* cnt = red_slot_counter(ctx, kSlotSu3);
    double* out = red_slot_out(ctx, kSlotSu3) + prec;
    if (prec == RMHMC_FP64) k_su3_check<<<grid, kBlock, 0, st>>>(links64(ctx), part, cnt, out);
    else k_su3_check32<<<grid, kBlock, 0, st>>>(links32(ctx), part, cnt, out);
    ++ctx->launches;
    RM_LAUNCH_CHECK(ctx);
    return RMHMC_OK;
}

void su3_known(rmhmc_ctx* ctx, int prec, bool su3) {
    ctx->su3[prec] = su3;
    ctx->su3_gen[prec] = ctx->import_gen;
}

int su3_state(const rmhmc_ctx* ctx, int prec) {
    const bool known64 = ctx->su3_gen[RMHMC_FP64] == ctx->import_gen, known32 = ctx->su3_gen[RMHMC_FP32] == ctx->import_gen;
    if (prec == RMHMC_FP64) return known64 ? ctx->su3[RMHMC_FP64] : known32 && !ctx->su3[RMHMC_FP32] ? 0 : -1;
    return known32 ? ctx->su3[RMHMC_FP32] : known64 && ctx->su3[RMHMC_FP64] ? 1 : -1;
}

int links_su3(rmhmc_ctx* ctx, int prec, cudaStream_t st, bool* su3) {
    int state = su3_state(ctx, prec);
    if (state < 0) {
        double bad = 0.0;
        RM_TRY(su3_check_launch(ctx, prec, st));
        RM_TRY(fetch(ctx, red_slot_out(ctx, kSlotSu3) + prec, &bad, 1, st));
        su3_known(ctx, prec, bad == 0.0);
        state = bad == 0.0;
    }
    *su3 = state == 1;
    return RMHMC_OK;
}

int gauge_loops_launch(rmhmc_ctx* ctx, double beta, double c1, int prec, double* F, bool act, bool defer, bool* used,
                       cudaStream_t st) {
    *used = false;
    if (!loops_usable(ctx) || !links_tracked(ctx, st)) return RMHMC_OK;
    if (F || c1 != 0.0) {
        bool su3 = true;
        if (!defer || su3_state(ctx, prec) >= 0) RM_TRY(links_su3(ctx, prec, st, &su3));
        if (!su3) return RMHMC_OK;
    }
    const int s = prec == RMHMC_FP64 ? loops_t<double>(ctx, links64(ctx), beta, c1, F, act, st)
                                     : loops_t<float>(ctx, links32(ctx), beta, c1, F, false, st);
    if (s == RMHMC_ENOMEM) {
        // no room for the loops: the staples serve as before
        ctx->err.clear();
        without(ctx, &ctx->loops_off);
        return RMHMC_OK;
    }
    RM_TRY(s);
    *used = true;
    return RMHMC_OK;
}

int gauge_loops_prepare(rmhmc_ctx* ctx, double c1, int prec) {
    if (!loops_usable(ctx)) return RMHMC_OK;
    LoopBufs<float> f;
    LoopBufs<double> d;
    const int s = prec == RMHMC_FP64 ? loop_bufs<double>(ctx, c1 != 0.0, true, d) : loop_bufs<float>(ctx, c1 != 0.0, true, f);
    if (s == RMHMC_ENOMEM) {
        ctx->err.clear();
        without(ctx, &ctx->loops_off);
        return RMHMC_OK;
    }
    return s;
}

}  // namespace rm
