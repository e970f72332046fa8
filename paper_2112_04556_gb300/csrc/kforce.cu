// Kinetic (mass-term) force, Sec. 3 (the force F_M below Eq. 5), and the link-adjoint of the
// Laplacian stencil it is built from.
//
// With T = 1/2 |R(A) P|^2, R(lam) = c + sum_j alpha_j/(lam + sigma_j):
//   dT = -sum_j alpha_j <Z_j, (dA) X_j>,  X_j = (A+sigma_j)^{-1} P,  Z_j = (A+sigma_j)^{-1} R(A) P,
// so F_K = -dT/dw = sum_j alpha_j <Z_j, (dA/dw) X_j>.  Only two hops of A contain U = U_nu(y): the
// forward hop at y and the backward hop at y+nu.  With W1 = U X(y+nu) U^dag, W2 = U Z(y+nu) U^dag,
//   d<Z, A X>/dw^a = -(1/16) 2i sum_mu Tr(T^a D),   D = [W1, Z(y)] - [X(y), W2] = M - M^dag,
//   M = W1 Z(y) - X(y) W2,
// and with K = -i D:  d<Z, A X>/dw^a = (1/16) sum_mu Tr(lambda^a K) = (1/8) sum_mu coef_a(M)
// where coef_a(M) = Tr(lambda^a (-i)(M - M^dag)/2) (antiherm_coef).
#include <algorithm>

#include "df.cuh"
#include "fcontract.cuh"
#include "krylov.cuh"
#include "ops.cuh"
#include "stencil.cuh"

namespace rm {

constexpr int kMaxPairs = 24;
struct PairWeights { double w[kMaxPairs]; };

// The same in the adjoint representation R = Ad(U): with x, z the coefficients at y and x', z' those at y + nu,
//   G^a = (1/16) sum_cd f_acd (R C)_cd,   C = sum_pairs w sum_mu (x' z^T + z' x^T),
// so that a pair costs two outer products per component (576 operations per link with the weights) and the conjugation
// by U comes once, for C.  The form above takes two conjugations and two matrix products per pair and component, 2016 FMA
// a link, which float64 (0.55 TFMA/s) is bound by: float64 at 16^4, 12 pairs 11.5 -> 3.5 ms, one pair 1.01 -> 0.7 ms.
// Four lanes per link, two columns d of C each; the contraction with f meets in shared memory.  Where the stencils have the
// table of R (LF = kLinkAd; built once per set of links) a column costs its 64 FMA instead of a conjugation's 108 and its
// expansions: differentiated Laplacian at 16^4 1.623 -> 1.590 ms, kinetic force with 12 pairs 13.35 -> 13.20 ms, and the error
// against 64 bits 4.6e-16 -> 3.5e-16.
template <int LF>
__global__ void __launch_bounds__(kBlock) k_link_grad(Geom g, Links64 U, const double* __restrict__ X,
                                                       const double* __restrict__ Z, size_t fs, int nf, PairWeights w,
                                                       double* __restrict__ G) {
    __shared__ double rcs[kBlock / 4][65];   // R C of the block's links
    const int lane = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = lane >> 2, q = lane & 3;
    const int nu = blockIdx.y;
    const bool live = y < g.V;
    double* const rc = rcs[threadIdx.x >> 2];
    if (live) {
        const size_t yo = (size_t)y * 32 + 2 * q, yn = (size_t)step_site(g, y, nu, 1) * 32;
        double C[2][8];
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int b = 0; b < 8; b++) C[i][b] = 0.0;
        for (int f = 0; f < nf; f++) {
            const double wf = w.w[f];
            const double *Xf = X + f * fs, *Zf = Z + f * fs;
#pragma unroll 2
            for (int mu = 0; mu < 4; mu++) {
                double xp[8], zp[8];
                load8(Xf + yn + mu * 8, xp);
                load8(Zf + yn + mu * 8, zp);
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    const double x = wf * __ldg(Xf + yo + mu * 8 + i), z = wf * __ldg(Zf + yo + mu * 8 + i);
#pragma unroll
                    for (int b = 0; b < 8; b++) C[i][b] = fma(xp[b], z, fma(zp[b], x, C[i][b]));
                }
            }
        }
        double r[2][8];
        if constexpr (LF == kLinkAd) {
            const double2* t = U.ad + (size_t)nu * 32 * U.V + y;
#pragma unroll
            for (int i = 0; i < 2; i++)
#pragma unroll
                for (int c = 0; c < 8; c++) r[i][c] = 0.0;
#pragma unroll
            for (int b = 0; b < 8; b++)
#pragma unroll
                for (int a = 0; a < 4; a++) {
                    const double2 v = __ldg(t + (size_t)(4 * b + a) * U.V);
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        r[i][2 * a] = fma(v.x, C[i][b], r[i][2 * a]);
                        r[i][2 * a + 1] = fma(v.y, C[i][b], r[i][2 * a + 1]);
                    }
                }
        } else {
            const mat3<double> u = LinkLoad<double, LF>::load(U, y, nu);
#pragma unroll
            for (int i = 0; i < 2; i++) {
                herm<double> E = h_zero<double>();
                acc_uxud(E, u, coef_to_herm2(C[i]));   // (with its trace: exact for any matrix, as the table)
                herm2_to_coef(E, r[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
            for (int c = 0; c < 8; c++) rc[c * 8 + 2 * q + i] = r[i][c];
    }
    __syncwarp();
    if (live) {
        double* out = G + (size_t)y * 32 + nu * 8 + 2 * q;
#pragma unroll
        for (int i = 0; i < 2; i++) {
            double v = 0.0;
#pragma unroll
            for (int t = 0; t < 4; t++) {
                const FTerm f = kFTerms[2 * q + i][t];
                if (f.v != 0.0) v = fma(f.v, rc[f.c * 8 + f.d] - rc[f.d * 8 + f.c], v);
            }
            out[i] = v * (1.0 / 16.0);
        }
    }
}

// The form of the file's head, four lanes per link with a component each, for float32: there the operations are not what bounds
// it, and a lane reads its own component's rows only, where a lane of the kernel above reads all four.  The form above took
// 1.3 to 1.4 times as long at any number of pairs: 24^3 x 48 672 against 499 us for one pair, 4547 against 3524 us for 12;
// 16^4 76 against 57 us; 8^4 with 12 pairs 45 against 35 us
template <int LF>
__global__ void __launch_bounds__(kBlock) k_link_grad_direct(Geom g, Links32 U, const float* __restrict__ X,
                                                              const float* __restrict__ Z, size_t fs, int nf, PairWeights w,
                                                              double* __restrict__ G) {
    const int lane = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = lane >> 2, mu = lane & 3;
    const int nu = blockIdx.y;
    const bool live = y < g.V;
    float k[8];
#pragma unroll
    for (int a = 0; a < 8; a++) k[a] = 0.f;
    if (live) {
        int fwd[4], bwd[4];
        neighbours(g, y, fwd, bwd);
        const int yp = fwd[nu];
        const mat3<float> u = LinkLoad<float, LF>::load(U, y, nu);
        for (int f = 0; f < nf; f++) {
            const float wf = (float)w.w[f];
            const float* Xf = X + f * fs;
            const float* Zf = Z + f * fs;
            float xb[8];
            load8(Xf + (size_t)yp * 32 + mu * 8, xb);
            herm<float> W1 = h_zero<float>();
            acc_uxud(W1, u, coef_to_herm2(xb));          // 2 W1
            load8(Zf + (size_t)yp * 32 + mu * 8, xb);
            herm<float> W2 = h_zero<float>();
            acc_uxud(W2, u, coef_to_herm2(xb));          // 2 W2
            load8(Zf + (size_t)y * 32 + mu * 8, xb);
            const mat3<float> Zy = herm_full(coef_to_herm2(xb));   // 2 Z(y)
            load8(Xf + (size_t)y * 32 + mu * 8, xb);
            const mat3<float> Xy = herm_full(coef_to_herm2(xb));   // 2 X(y)
            mat3<float> M = m_mul(herm_full(W1), Zy);              // 4 W1 Z
            const mat3<float> M2 = m_mul(Xy, herm_full(W2));       // 4 X W2
#pragma unroll
            for (int i = 0; i < 3; i++)
#pragma unroll
                for (int j = 0; j < 3; j++) M.e[i][j] = csub(M.e[i][j], M2.e[i][j]);
            float kk[8];
            antiherm_coef(M, kk);                               // 4 coef(M)
#pragma unroll
            for (int a = 0; a < 8; a++) k[a] = fma(wf, kk[a], k[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 8; a++) {
        k[a] += __shfl_xor_sync(0xffffffffu, k[a], 1);
        k[a] += __shfl_xor_sync(0xffffffffu, k[a], 2);
    }
    if (live && mu == 0) {
        double* out = G + (size_t)y * 32 + nu * 8;
        // d<Z,AX>/dw = (1/8) coef(M) and the doubled expansions gave 4 coef(M): scale by 1/32
#pragma unroll
        for (int a = 0; a < 8; a++) out[a] = (double)k[a] * (1.0 / 32.0);
    }
}

int link_grad_launch(rmhmc_ctx* ctx, int prec, const void* X, const void* Z, int nf, const double* w, double* G,
                     cudaStream_t st) {
    if (nf > kMaxPairs) return set_err(ctx, RMHMC_EINVAL, "at most %d field pairs", kMaxPairs);
    PairWeights pw{};
    for (int f = 0; f < nf; f++) pw.w[f] = w[f];
    const dim3 grid(lane_blocks(ctx), 4);
    if (prec == RMHMC_FP64) {
        Links64 U = links64(ctx);
        RM_TRY(links64_adjoint(ctx, &U, st));
        if (U.ad)
            k_link_grad<kLinkAd><<<grid, kBlock, 0, st>>>(ctx->g, U, (const double*)X, (const double*)Z,
                                                                  field_elems(ctx), nf, pw, G);
        else
            k_link_grad<18><<<grid, kBlock, 0, st>>>(ctx->g, U, (const double*)X, (const double*)Z,
                                                             field_elems(ctx), nf, pw, G);
    } else
        k_link_grad_direct<18><<<grid, kBlock, 0, st>>>(ctx->g, links32(ctx), (const float*)X, (const float*)Z,
                                                        field_elems(ctx), nf, pw, G);
    ++ctx->launches;
    RM_LAUNCH_CHECK(ctx);
    return RMHMC_OK;
}

// ------------------------------------------------------------------------------------------------
// Kinetic force straight from the Krylov basis.  With X_j = sum_k cx_jk r_k and Z_j = sum_k cz_jk r_k on the
// stored residuals r_k, the force on U = U_nu(y) is, in the adjoint representation R = Ad(U)
// (U T^b U^dag = sum_c R_cb T^c) and with the su(3) structure constants f,
//   G^a = (1/16) sum_cd f_acd (R C)_cd,   C = sum_mu sum_kl S_kl r_k,mu(y+nu) r_l,mu(y)^T,
//   S_kl = sum_j alpha_j (cx_jk cz_jl + cz_jk cx_jl),
// because coef_a(W Z - X W') = (1/2) f_acd [R (x' z^T + z' x^T)]_cd for W = U X' U^dag, W' = U Z' U^dag
// (x, z, x', z' the coefficient vectors of X(y), Z(y), X(y+nu), Z(y+nu)).  One pass over the n basis
// vectors replaces forming the 2 npole fields X_j, Z_j and the per-pole conjugations: per site about
// 8 n^2 + 256 n + 1400 FMA per link against 576 npole per link for the direct form.
// ------------------------------------------------------------------------------------------------

// eight values from shared memory (plain loads: the read-only global path does not apply to shared memory)
__device__ __forceinline__ void lds8(const float* p, float* x) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void lds8(const double* p, double* x) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const double2 v = reinterpret_cast<const double2*>(p)[i];
        x[2 * i] = v.x; x[2 * i + 1] = v.y;
    }
}

constexpr int kLgSites = 32;   // sites per block (4 lanes each)
constexpr int kLgKC = 4;       // basis vectors per chunk of W
constexpr int kLgPad = kLgKC * 32 + 4;

// S_kl (row stride ld) from the basis rows of X_j (rows j) and Z_j (rows ns + j), row stride ldr;
// n from flags[1] when flags is given
__global__ void __launch_bounds__(256) k_pair_matrix(const double* __restrict__ rows, int ldr, int ns, PairWeights w,
                                                     const int* __restrict__ flags, int n, double* __restrict__ S, int ld) {
    if (flags) n = flags[1];
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n * n; idx += gridDim.x * blockDim.x) {
        const int k = idx / n, l = idx % n;
        double s = 0.0;
#pragma unroll 4
        for (int j = 0; j < ns; j++) {
            const double* X = rows + (size_t)j * ldr;
            const double* Z = rows + (size_t)(ns + j) * ldr;
            s = fma(w.w[j], fma(X[k], Z[l], Z[k] * X[l]), s);
        }
        S[(size_t)k * ld + l] = s;
    }
}

// one block: kLgSites sites x 4 lanes.  Per chunk of kLgKC basis vectors: lane (y, mu) forms
// W_k,mu(y) = sum_l S_kl r_l,mu(y) into shared memory; then lane (y, nu) accumulates
// C += sum_mu r_k,mu(y+nu) W_k,mu(y)^T.  Finally lane (y, nu) conjugates the columns of C by U_nu(y) and
// contracts with f.  n from flags[1] when flags is given.
template <typename T, int LF>
__global__ void __launch_bounds__(kLgSites * 4, 4) k_link_grad_krylov(Geom g, typename LinksOf<T>::type U, const T* __restrict__ R,
                                                                   size_t fs, const int* __restrict__ flags, int n,
                                                                   const double* __restrict__ S, int ld, double* __restrict__ G) {
    __shared__ __align__(16) T Ws[kLgSites * kLgPad];
    __shared__ T Ss[kLgKC * kBasisCap];
    if (flags) n = flags[1];
    const int sl = threadIdx.x >> 2, q = threadIdx.x & 3;
    T* const wrow = Ws + sl * kLgPad;
    for (int base = blockIdx.x * kLgSites; base < g.V; base += gridDim.x * kLgSites) {
        const int y = base + sl;
        const bool live = y < g.V;
        int yn = 0;
        if (live) {
            int fwd[4], bwd[4];
            neighbours(g, y, fwd, bwd);
            yn = fwd[q];
        }
        T C[8][8];
#pragma unroll
        for (int b = 0; b < 8; b++)
#pragma unroll
            for (int d = 0; d < 8; d++) C[b][d] = T(0);
        for (int k0 = 0; k0 < n; k0 += kLgKC) {
            __syncthreads();
            for (int t = threadIdx.x; t < kLgKC * n; t += blockDim.x) {
                const int kk = t / n, l = t - kk * n;
                Ss[kk * kBasisCap + l] = k0 + kk < n ? (T)S[(size_t)(k0 + kk) * ld + l] : T(0);
            }
            __syncthreads();
            T w[kLgKC][8];
#pragma unroll
            for (int kk = 0; kk < kLgKC; kk++)
#pragma unroll
                for (int a = 0; a < 8; a++) w[kk][a] = T(0);
            if (live) {
                for (int l = 0; l < n; l++) {
                    T r[8];
                    load_plane8(R + (size_t)l * fs, g.V, y, q, r);
#pragma unroll
                    for (int kk = 0; kk < kLgKC; kk++) {
                        const T s = Ss[kk * kBasisCap + l];
#pragma unroll
                        for (int a = 0; a < 8; a++) w[kk][a] = fma(s, r[a], w[kk][a]);
                    }
                }
            }
#pragma unroll
            for (int kk = 0; kk < kLgKC; kk++) store8(wrow + kk * 32 + q * 8, w[kk]);
            __syncthreads();
            if (live) {
                const int kc = min(kLgKC, n - k0);
                for (int kk = 0; kk < kc; kk++) {
                    const T* rk = R + (size_t)(k0 + kk) * fs;
#pragma unroll
                    for (int mu = 0; mu < 4; mu++) {
                        T rp[8], wv[8];
                        load_plane8(rk, g.V, yn, mu, rp);
                        lds8(wrow + kk * 32 + mu * 8, wv);
#pragma unroll
                        for (int b = 0; b < 8; b++)
#pragma unroll
                            for (int d = 0; d < 8; d++) C[b][d] = fma(rp[b], wv[d], C[b][d]);
                    }
                }
            }
        }
        if (live) {
            const mat3<T> u = LinkLoad<T, LF>::load(U, y, q);
            T Gk[8];
#pragma unroll
            for (int a = 0; a < 8; a++) Gk[a] = T(0);
#pragma unroll
            for (int d = 0; d < 8; d++) {
                T col[8], rc[8];
#pragma unroll
                for (int b = 0; b < 8; b++) col[b] = C[b][d];
                herm<T> E = h_zero<T>();
                acc_uxud_tl(E, u, coef_to_herm2(col));   // 2 sum_c (R C)_cd T^c
                herm2_to_coef_tl(E, rc);                  // (R C)_cd
                f_contract(d, rc, Gk);
            }
            double* out = G + (size_t)y * 32 + q * 8;
#pragma unroll
            for (int a = 0; a < 8; a++) out[a] = (double)Gk[a] * (1.0 / 16.0);
        }
    }
}

// The contraction in one pass with the velocity and the energy (the default).  Block: 32 consecutive sites, one per
// lane; warp: component mu (phase W) or link direction nu (phase C), so that every load of the planes is two contiguous
// 512-byte segments.  Phase W holds the site's own row of up to kLbN basis vectors in registers, four colours at a time, and
// leaves W_k,mu = sum_l S_kl r_l,mu of all of them in shared memory; phase C adds r_k,mu(y+nu) W_k,mu(y)^T to the lane's
// 8 x 8 accumulator, the neighbours' rows loaded one vector ahead.
//
// What bounds it.  The kernel above re-reads the own rows and S for every four vectors, between two barriers each, with
// its accumulators live: at 128 registers it waits on that chain of loads (long scoreboard 5.5 per issue, 34 % of the
// FMA pipe).  Here the own rows are read once, all in flight together, and 8 warps with 255 registers each take the
// place of 16 with 128.  At 32^4 and 18 vectors: 2.47 ms with the velocity and the energy, against 2.75 ms and two
// combinations of 0.48 ms each; at 16^4 0.164 ms (40 % of the FMA pipe; 42 % of the issue slots).
// VEL: Vel = sum_k cvel[k] r_k; EN: |sum_k cen[k] r_k|^2 to *out (float64-accurate sum): both from the rows in registers.
// Runs longer than kLbN take a pass per kLbN x kLbN block of S.  Tiles are taken in the order (z block of bz planes, t,
// position in the slab): the t + 1 rows of a slab are then still in L2 when the sweep reaches them.
constexpr int kLbSites = 32;
constexpr int kLbN = 20;           // the workloads' runs have 13 to 18 vectors
constexpr int kLbSmem = (kLbN * kLbN + 2 * kBasisCap + kLbN * 32 * kLbSites) * (int)sizeof(float);

template <int LF, bool VEL, bool EN>
__global__ void __launch_bounds__(128, 2)
    k_link_grad_basis(Geom g, Links32 U, const float* __restrict__ R, size_t fs, const int* __restrict__ flags, int n,
                      const double* __restrict__ S, int ld, double* __restrict__ G, const double* __restrict__ cvel,
                      double* __restrict__ Vel, const double* __restrict__ cen, int bz, double* partials, unsigned* counter,
                      double* out) {
    extern __shared__ __align__(16) float lbs[];
    float* Ss = lbs;                                      // [k][l] of the current block of S
    float* cv = Ss + kLbN * kLbN;
    float* ce = cv + kBasisCap;
    float4* W = reinterpret_cast<float4*>(ce + kBasisCap);   // [k][plane][site]
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (flags) n = flags[1];
    auto load_s = [&](int k0, int l0) {
        for (int i = threadIdx.x; i < kLbN * kLbN; i += blockDim.x) {
            const int k = k0 + i / kLbN, l = l0 + i % kLbN;
            Ss[i] = k < n && l < n ? (float)S[(size_t)k * ld + l] : 0.f;
        }
    };
    const bool single = n <= kLbN;
    if (single) load_s(0, 0);
    for (int k = threadIdx.x; k < kBasisCap; k += blockDim.x) {
        if (VEL) cv[k] = k < n ? (float)cvel[k] : 0.f;
        if (EN) ce[k] = k < n ? (float)cen[k] : 0.f;
    }
    __syncthreads();
    SumSq32 energy;
    const int P = g.stride[2], V3 = g.stride[3];
    const int nts = (P * bz + kLbSites - 1) / kLbSites;
    const int nunit = nts * g.L[3] * ((g.L[2] + bz - 1) / bz);
    const size_t ps = (size_t)g.V * 4;                    // plane stride
    for (int u = blockIdx.x; u < nunit; u += gridDim.x) {
        const int jt = u % nts, ru = u / nts, tt = ru % g.L[3], z0 = (ru / g.L[3]) * bz;
        const int first = jt * kLbSites + lane;
        const bool live = first < P * min(bz, g.L[2] - z0);
        const int y = live ? tt * V3 + z0 * P + first : 0;
        const float* const own = R + (size_t)y * 4 + 2 * w * ps;
        const float* const nbr = R + (size_t)step_site(g, y, w, 1) * 4;
        float2 C[8][4];                                   // C[b][d], pairs of d
#pragma unroll
        for (int b = 0; b < 8; b++)
#pragma unroll
            for (int d = 0; d < 4; d++) C[b][d] = make_float2(0.f, 0.f);
        const int nk = max(n, 1);   // an empty run (zero momenta) still writes its zeros
        for (int k0 = 0; k0 < nk; k0 += kLbN) {
            const int kc = min(kLbN, n - k0);
            // neighbours' rows of the first vector, on their way during phase W
            const float* rk = nbr + (size_t)k0 * fs;
            float4 ra[4][2];
            if (kc > 0)
#pragma unroll
                for (int mu = 0; mu < 4; mu++)
#pragma unroll
                    for (int h = 0; h < 2; h++) ra[mu][h] = __ldg(reinterpret_cast<const float4*>(rk + (2 * mu + h) * ps));
#pragma unroll 1
            for (int h = 0; h < 2; h++) {
                float4 va = make_float4(0.f, 0.f, 0.f, 0.f), ea = va;
                for (int l0 = 0; l0 < nk; l0 += kLbN) {
                    if (!single) {
                        __syncthreads();
                        load_s(k0, l0);
                        __syncthreads();
                    }
                    float4 r[kLbN];
#pragma unroll
                    for (int l = 0; l < kLbN; l++)
                        r[l] = l0 + l < n ? __ldg(reinterpret_cast<const float4*>(own + h * ps + (size_t)(l0 + l) * fs))
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int k = 0; k < kc; k++) {
                        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                        float4* dst = W + (k * 8 + 2 * w + h) * kLbSites + lane;
                        if (l0 > 0) a = *dst;
#pragma unroll
                        for (int l = 0; l < kLbN; l += 4) {
                            const float4 s = *reinterpret_cast<const float4*>(Ss + k * kLbN + l);
                            const float sv[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
                            for (int q = 0; q < 4; q++) {
                                a.x = fmaf(sv[q], r[l + q].x, a.x); a.y = fmaf(sv[q], r[l + q].y, a.y);
                                a.z = fmaf(sv[q], r[l + q].z, a.z); a.w = fmaf(sv[q], r[l + q].w, a.w);
                            }
                        }
                        *dst = a;
                    }
                    if ((VEL || EN) && k0 == 0)
#pragma unroll
                        for (int l = 0; l < kLbN; l++) {
                            if (VEL) {
                                const float c = cv[l0 + l];
                                va.x = fmaf(c, r[l].x, va.x); va.y = fmaf(c, r[l].y, va.y);
                                va.z = fmaf(c, r[l].z, va.z); va.w = fmaf(c, r[l].w, va.w);
                            }
                            if (EN) {
                                const float c = ce[l0 + l];
                                ea.x = fmaf(c, r[l].x, ea.x); ea.y = fmaf(c, r[l].y, ea.y);
                                ea.z = fmaf(c, r[l].z, ea.z); ea.w = fmaf(c, r[l].w, ea.w);
                            }
                        }
                }
                if ((VEL || EN) && k0 == 0 && live) {
                    if (VEL) {
                        const double o[4] = {(double)va.x, (double)va.y, (double)va.z, (double)va.w};
                        store4(Vel + (size_t)y * 32 + w * 8 + h * 4, o);
                    }
                    if (EN) {
                        energy.add(ea.x); energy.add(ea.y);
                        energy.add(ea.z); energy.add(ea.w);
                    }
                }
            }
            __syncthreads();
            for (int k = 0; k < kc; k++) {
                rk += fs;
#pragma unroll
                for (int mu = 0; mu < 4; mu++) {
                    const float a[8] = {ra[mu][0].x, ra[mu][0].y, ra[mu][0].z, ra[mu][0].w,
                                        ra[mu][1].x, ra[mu][1].y, ra[mu][1].z, ra[mu][1].w};
                    if (k + 1 < kc)
#pragma unroll
                        for (int h = 0; h < 2; h++) ra[mu][h] = __ldg(reinterpret_cast<const float4*>(rk + (2 * mu + h) * ps));
                    const float4 w0 = W[(k * 8 + 2 * mu) * kLbSites + lane], w1 = W[(k * 8 + 2 * mu + 1) * kLbSites + lane];
                    const float2 wp[4] = {make_float2(w0.x, w0.y), make_float2(w0.z, w0.w), make_float2(w1.x, w1.y),
                                          make_float2(w1.z, w1.w)};
#pragma unroll
                    for (int b = 0; b < 8; b++)
#pragma unroll
                        for (int d = 0; d < 4; d++) C[b][d] = ffma2(make_float2(a[b], a[b]), wp[d], C[b][d]);
                }
            }
            __syncthreads();   // W is rewritten
        }
        if (live) {
            const mat3<float> m = LinkLoad<float, LF>::load(U, y, w);
            float Gk[8];
#pragma unroll
            for (int a = 0; a < 8; a++) Gk[a] = 0.f;
#pragma unroll
            for (int d = 0; d < 8; d++) {
                float col[8], rc[8];
#pragma unroll
                for (int b = 0; b < 8; b++) col[b] = d & 1 ? C[b][d >> 1].y : C[b][d >> 1].x;
                herm<float> E = h_zero<float>();
                acc_uxud_tl(E, m, coef_to_herm2(col));   // 2 sum_c (R C)_cd T^c
                herm2_to_coef_tl(E, rc);                  // (R C)_cd
                f_contract(d, rc, Gk);
            }
            double o[8];
#pragma unroll
            for (int a = 0; a < 8; a++) o[a] = (double)Gk[a] * (1.0 / 16.0);
            store8(G + (size_t)y * 32 + w * 8, o);
        }
    }
    if (EN) {
        __shared__ double sh[4];
        double v[1] = {energy.value()};
        block_sum<1>(v, sh);
        grid_sum_finish<1>(v, partials, counter, out, gridDim.x, blockIdx.x, sh);
    }
}

template <bool VEL, bool EN>
static int launch_basis(rmhmc_ctx* ctx, const float* R, const int* flags, int n, const double* S, double* G,
                        const double* cvel, double* Vel, const double* cen, int slot, cudaStream_t st) {
    auto kern = k_link_grad_basis<18, VEL, EN>;
    RM_CHECK(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kLbSmem));
    // slabs of z whose two t-slices of 20 basis vectors take at most a third of L2
    const size_t slice = (size_t)ctx->g.stride[3] * 32 * sizeof(float) * 20 * 2, room = (size_t)40 << 20;
    const int nzb = (int)std::min<size_t>(ctx->g.L[2], (slice + room - 1) / room);
    const int bz = (ctx->g.L[2] + nzb - 1) / nzb;
    const int nunit = (ctx->g.stride[2] * bz + kLbSites - 1) / kLbSites * ctx->g.L[3] * ((ctx->g.L[2] + bz - 1) / bz);
    const int grid = std::max(1, std::min(std::min(nunit, (int)ctx->num_sms * 2), ctx->max_blocks * 2));
    kern<<<grid, 128, kLbSmem, st>>>(ctx->g, links32(ctx), R, field_elems(ctx), flags, n, S, kBasisCap, G, cvel, Vel, cen, bz,
                                     EN ? red_slot_partials(ctx, slot) : nullptr,
                                     EN ? red_slot_counter(ctx, slot) : nullptr, EN ? red_slot_out(ctx, slot) : nullptr);
    ++ctx->launches;
    RM_LAUNCH_CHECK(ctx);
    return RMHMC_OK;
}

// F_K from the basis rows (X_j rows 0..ns-1, Z_j rows ns..2ns-1, row stride ldr, device float64) of the
// float32 basis R; n on the host, or read on the device from flags[1] when flags is given
int link_grad_krylov_launch(rmhmc_ctx* ctx, const float* R, const double* rows, int ldr, int ns, const double* alpha,
                            const int* flags, int n, double* F, const double* cvel, double* Vel, const double* cen,
                            int slot, cudaStream_t st) {
    if (ns > kMaxPairs) return set_err(ctx, RMHMC_EINVAL, "at most %d poles", kMaxPairs);
    int status = RMHMC_OK;
    double* S = (double*)workspace(ctx, "kf_pairs", sizeof(double) * kBasisCap * kBasisCap, &status);
    if (!S) return status;
    if (rows) {
        PairWeights pw{};
        for (int j = 0; j < ns; j++) pw.w[j] = alpha[j];
        k_pair_matrix<<<ctx->num_sms / 4 > 1 ? ctx->num_sms / 4 : 1, 256, 0, st>>>(rows, ldr, ns, pw, flags, n, S, kBasisCap);
        ++ctx->launches;
    }
    if (ctx->lg_mode == kLgFused) {
        if (Vel && cen) return launch_basis<true, true>(ctx, R, flags, n, S, F, cvel, Vel, cen, slot, st);
        if (Vel) return launch_basis<true, false>(ctx, R, flags, n, S, F, cvel, Vel, cen, slot, st);
        if (cen) return launch_basis<false, true>(ctx, R, flags, n, S, F, cvel, Vel, cen, slot, st);
        return launch_basis<false, false>(ctx, R, flags, n, S, F, cvel, Vel, cen, slot, st);
    }
    const int grid = capped_grid(ctx, (size_t)ctx->g.V * 4, kLgSites * 4);
    k_link_grad_krylov<float, 18><<<grid, kLgSites * 4, 0, st>>>(ctx->g, links32(ctx), R, field_elems(ctx), flags, n, S,
                                                                 kBasisCap, F);
    ++ctx->launches;
    RM_LAUNCH_CHECK(ctx);
    return RMHMC_OK;
}

// ------------------------------------------------------------------------------------------------
// kinetic pieces from a single Krylov run on P
// ------------------------------------------------------------------------------------------------
template <typename T>
static int kinetic_t(rmhmc_ctx* ctx, const MassTerm& m, const double* P, double tol, int maxiter, double* F, double* Vel,
                     double* Tkin, int* iters, cudaStream_t st) {
    const int ns = m.npole();
    const size_t fs = field_elems(ctx);
    int status = RMHMC_OK;
    if (ns == 0) {
        // M = c^{-2}: V = c^2 P, F_K = 0, T = c^2 |P|^2 / 2
        if (F) RM_CHECK(ctx, cudaMemsetAsync(F, 0, sizeof(double) * fs, st));
        if (Vel) RM_TRY(axpby64(ctx, m.c * m.c, P, 0.0, nullptr, Vel, fs, st));
        if (Tkin) {
            double n2 = 0.0;
            RM_TRY(norm2_64(ctx, P, fs, &n2, st));
            *Tkin = 0.5 * m.c * m.c * n2;
        }
        if (iters) *iters = 0;
        return RMHMC_OK;
    }
    const double s0 = *std::min_element(m.sigma.begin(), m.sigma.end());
    KrylovResult kr;
    RM_TRY((krylov_run<T, double>(ctx, P, s0, tol, maxiter, kr, st)));
    if (kr.status == 2) return set_err(ctx, RMHMC_ENOCONV, "kinetic force: Krylov run hit its cap (%d)", kr.n);
    if (iters) *iters = kr.n;
    Tridiag tri;
    tri.build(kr);
    const int n = tri.n;
    // Galerkin coefficient vectors: y_j = (T+D_j)^{-1} e1|b|, g = R(T) e1|b|, z_j = (T+D_j)^{-1} g, v = R(T) g
    std::vector<double> e1(n, 0.0), g(n, 0.0), v(n, 0.0);
    if (n > 0) e1[0] = tri.bnorm;
    std::vector<std::vector<double>> ys(ns), zs(ns);
    for (int j = 0; j < ns; j++) tri.solve(m.sigma[j] - s0, e1, ys[j]);
    for (int k = 0; k < n; k++) {
        g[k] = m.c * e1[k];
        for (int j = 0; j < ns; j++) g[k] += m.alpha[j] * ys[j][k];
    }
    for (int j = 0; j < ns; j++) tri.solve(m.sigma[j] - s0, g, zs[j]);
    for (int k = 0; k < n; k++) {
        v[k] = m.c * g[k];
        for (int j = 0; j < ns; j++) v[k] += m.alpha[j] * zs[j][k];
    }
    // float32 basis: force, velocity and energy in one pass over the basis
    const bool fused = F && sizeof(T) == 4 && ctx->lg_mode == kLgFused;
    if (Tkin && !fused) {
        // T = 1/2 |R P|^2 from the explicitly formed R P (float64 sum), not from |g|, which would
        // assume exactly orthonormal Lanczos vectors
        double* Y = (double*)workspace(ctx, "kf_y", sizeof(double) * fs, &status);
        if (!Y) return status;
        CombineSpec spec;
        spec.n = n;
        spec.M = 1;
        spec.coef.assign(n, 0.0);
        tri.to_basis(g, spec.coef.data());
        double* o[1] = {Y};
        RM_TRY((krylov_combine<T, double>(ctx, spec, o, st)));
        double y2 = 0.0;
        RM_TRY(norm2_64(ctx, Y, fs, &y2, st));
        *Tkin = 0.5 * y2;
    }
    if (Vel && !fused) {
        CombineSpec spec;
        spec.n = n;
        spec.M = 1;
        spec.coef.assign(n, 0.0);
        tri.to_basis(v, spec.coef.data());
        double* o[1] = {Vel};
        RM_TRY((krylov_combine<T, double>(ctx, spec, o, st)));
    }
    if (!F) return RMHMC_OK;
    if constexpr (sizeof(T) == 4) {
        // float32 basis: the force straight from the basis (rows of X_j and Z_j on the stored residuals)
        double* rows = (double*)workspace(ctx, "kf_rows", sizeof(double) * (size_t)(2 * ns + 2) * kBasisCap, &status);
        if (!rows) return status;
        std::vector<double> h((size_t)(2 * ns + 2) * n, 0.0);
        for (int j = 0; j < ns; j++) {
            tri.to_basis(ys[j], h.data() + (size_t)j * n);
            tri.to_basis(zs[j], h.data() + (size_t)(ns + j) * n);
        }
        tri.to_basis(v, h.data() + (size_t)2 * ns * n);
        tri.to_basis(g, h.data() + (size_t)(2 * ns + 1) * n);
        RM_TRY(upload(ctx, rows, h.data(), sizeof(double) * h.size(), st));
        RM_TRY(link_grad_krylov_launch(ctx, (const float*)krylov_basis<T>(ctx), rows, n, ns, m.alpha.data(), nullptr, n, F,
                                       rows + (size_t)2 * ns * n, Vel, Tkin ? rows + (size_t)(2 * ns + 1) * n : nullptr,
                                       kSlotNorm, st));
        if (fused && Tkin) {
            // |R P|^2 of the explicitly formed R P, as above
            double y2 = 0.0;
            RM_TRY(fetch(ctx, red_slot_out(ctx, kSlotNorm), &y2, 1, st));
            *Tkin = 0.5 * y2;
        }
    } else {
        T* XZ = (T*)workspace(ctx, "kf_xz64", sizeof(T) * fs * 2 * ns, &status);
        if (!XZ) return status;
        CombineSpec spec;
        spec.n = n;
        spec.M = 2 * ns;
        spec.coef.assign((size_t)2 * ns * n, 0.0);
        std::vector<T*> outs(2 * ns);
        for (int j = 0; j < ns; j++) {
            tri.to_basis(ys[j], spec.coef.data() + (size_t)j * n);
            tri.to_basis(zs[j], spec.coef.data() + (size_t)(ns + j) * n);
            outs[j] = XZ + (size_t)j * fs;
            outs[ns + j] = XZ + (size_t)(ns + j) * fs;
        }
        RM_TRY((krylov_combine<T, T>(ctx, spec, outs.data(), st)));
        RM_TRY(link_grad_launch(ctx, RMHMC_FP64, XZ, XZ + (size_t)ns * fs, ns, m.alpha.data(), F, st));
    }
    return RMHMC_OK;
}

int kinetic_from_krylov(rmhmc_ctx* ctx, const MassTerm& m, const double* P, double tol, int maxiter, int prec,
                        double* F, double* Vel, double* T, int* iters, cudaStream_t st) {
    if (prec == RMHMC_FP64) return kinetic_t<double>(ctx, m, P, tol, maxiter, F, Vel, T, iters, st);
    return kinetic_t<float>(ctx, m, P, tol, maxiter, F, Vel, T, iters, st);
}

}  // namespace rm

using namespace rm;

extern "C" int lap_link_grad(rmhmc_ctx* ctx, const double* U, const double* X, const double* Z, int nfield,
                             const double* w, int prec, double* G, cudaStream_t stream) {
    if (!ctx) return RMHMC_EINVAL;
    ctx->err.clear();
    if (!X || !Z || !G || (nfield > 0 && !w)) return set_err(ctx, RMHMC_EINVAL, "lap_link_grad: null argument");
    if (nfield < 0 || nfield > kMaxPairs) return set_err(ctx, RMHMC_EINVAL, "lap_link_grad: nfield in [0, %d]", kMaxPairs);
    if (prec != RMHMC_FP64 && prec != RMHMC_FP32) return set_err(ctx, RMHMC_EINVAL, "lap_link_grad: bad prec");
    RM_TRY(ensure_links_table(ctx, U, prec == RMHMC_FP64 && nfield > 0, stream));
    const size_t fs = field_elems(ctx);
    if (nfield == 0) {
        RM_CHECK(ctx, cudaMemsetAsync(G, 0, sizeof(double) * fs, stream));
        return RMHMC_OK;
    }
    if (prec == RMHMC_FP64) return link_grad_launch(ctx, prec, X, Z, nfield, w, G, stream);
    int status = RMHMC_OK;
    float* buf = (float*)workspace(ctx, "lg_xz32", sizeof(float) * fs * 2 * nfield, &status);
    if (!buf) return status;
    RM_TRY(to_float(ctx, X, buf, fs * nfield, stream));
    RM_TRY(to_float(ctx, Z, buf + fs * nfield, fs * nfield, stream));
    return link_grad_launch(ctx, prec, buf, buf + fs * nfield, nfield, w, G, stream);
}

extern "C" int kinetic_force(rmhmc_ctx* ctx, const double* U, const double* P, const rmhmc_mass* mass, double tol,
                             int prec, double* F, double* Vout, double* T, cudaStream_t stream) {
    if (!ctx) return RMHMC_EINVAL;
    ctx->err.clear();
    if (!P) return set_err(ctx, RMHMC_EINVAL, "kinetic_force: null momenta");
    if (!(tol > 0.0)) return set_err(ctx, RMHMC_EINVAL, "kinetic_force: tol must be > 0");
    if (prec != RMHMC_FP64 && prec != RMHMC_MIXED) return set_err(ctx, RMHMC_EINVAL, "kinetic_force: bad prec");
    MassTerm m;
    RM_TRY(parse_mass(ctx, mass, m));
    RM_TRY(ensure_links(ctx, U, stream));
    // the kernels read and write float64 fields 16 bytes at a time: a field at an odd multiple of 8 bytes goes through
    // the workspace
    const size_t bytes = sizeof(double) * field_elems(ctx);
    int status = RMHMC_OK;
    auto aligned = [&](const void* p, const char* name) -> double* {
        return (uintptr_t)p % 16 ? (double*)workspace(ctx, name, bytes, &status) : (double*)p;
    };
    const double* Pa = aligned(P, "kf_p16");
    double *Fa = aligned(F, "kf_f16"), *Va = aligned(Vout, "kf_v16");
    RM_TRY(status);
    if (Pa != P) RM_CHECK(ctx, cudaMemcpyAsync((void*)Pa, P, bytes, cudaMemcpyDeviceToDevice, stream));
    RM_TRY(kinetic_from_krylov(ctx, m, Pa, tol, 1000, prec, Fa, Va, T, nullptr, stream));
    if (Fa != F) RM_CHECK(ctx, cudaMemcpyAsync(F, Fa, bytes, cudaMemcpyDeviceToDevice, stream));
    if (Va != Vout) RM_CHECK(ctx, cudaMemcpyAsync(Vout, Va, bytes, cudaMemcpyDeviceToDevice, stream));
    return RMHMC_OK;
}

extern "C" int rmhmc_heatbath(rmhmc_ctx* ctx, const double* U, const double* xi, const rmhmc_mass* mass, double tol,
                              int prec, double* P, cudaStream_t stream) {
    if (!ctx) return RMHMC_EINVAL;
    ctx->err.clear();
    if (!xi || !P) return set_err(ctx, RMHMC_EINVAL, "rmhmc_heatbath: null field");
    if (!(tol > 0.0)) return set_err(ctx, RMHMC_EINVAL, "rmhmc_heatbath: tol must be > 0");
    if (prec != RMHMC_FP64 && prec != RMHMC_MIXED) return set_err(ctx, RMHMC_EINVAL, "rmhmc_heatbath: bad prec");
    MassTerm m;
    RM_TRY(parse_mass(ctx, mass, m));
    RM_TRY(ensure_links(ctx, U, stream));
    return heatbath_apply(ctx, m, xi, tol, 1000, prec, P, stream);
}
