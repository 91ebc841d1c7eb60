// Spectral-side kernels of the RHS F (Eq. (ode)) on CUDA cores:
//   prep32     coefficient sets of the FP32 ensembles' synthesis (Eqs.
//              (stok_eig), (vort_app))
//   analysis   per-order Legendre sums of the quadrature-weighted Fourier
//              profiles (Eq. (disc_vec_orth_proj)), FP32, for numbers of
//              northern latitudes that legendre_f32.cu does not take
//   finish     degree-shift recombination and the diagonal Stokes update
//              (Sec. 4.2: nu lambda_L alpha_{L,m}) plus forcing.
// The coefficient state in and out is always FP64.
#include <cuda_runtime.h>

#include "finish.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace sph {

// ---------------------------------------------------------------------------
// prep: one thread per ext row (m, K), K = m..N+1.
//   field 0 (zeta):  lambda_K^{1/2} alpha_K
//   field 1 (theta): a_K = lambda_K^{-1/2} alpha_K
//   field 2 (phi):   (K-1) eps_{K,m} a_{K-1} - (K+2) eps_{K+1,m} a_{K+1}
// (sin(theta) d/dtheta Pt_L^m = L eps_{L+1,m} Pt_{L+1}^m - (L+1) eps_{L,m} Pt_{L-1}^m
//  regrouped by degree).  The coefficients come precomputed per row, c =
// (lam^{1/2}, lam^{-1/2}, c_down, c_up).  alpha_K is converted once per row and its degree
// neighbours come from shared memory; the arithmetic is FP32 (the FP32 path
// contracts in FP32 anyway), keeping the weak FP64 pipe for the state only.
__global__ void __launch_bounds__(128) k_prep32(const double2* __restrict__ alpha, const float4* __restrict__ prepc,
                                                float* __restrict__ bsyn, int N, int ncoef, size_t bstride) {
    __shared__ float2 sa[130];
    pdl_launch();
    pdl_wait();   // alpha may be the predecessor's output
    // batch of instances along gridDim.z (fixed strides between instances)
    alpha += size_t(blockIdx.z) * ncoef;
    bsyn += size_t(blockIdx.z) * bstride;
    const int m = blockIdx.y, t = threadIdx.x;
    const int K0 = m + blockIdx.x * 128, K = K0 + t;
    const int lo = m > 0 ? m : 1;
    auto ld = [&](int Kp) -> float2 {
        if (Kp < lo || Kp > N) return make_float2(0.f, 0.f);
        const double2 c = alpha[packed_index(N, m, Kp)];
        return make_float2(float(c.x), float(c.y));
    };
    sa[t + 1] = ld(K);
    if (t == 0) sa[0] = ld(K0 - 1);
    if (t == 127) sa[129] = ld(K0 + 128);
    __syncthreads();
    if (K > N + 1) return;
    const int row = ext_row(N, m, K);
    const float4 c = prepc[row];
    float* out = bsyn + size_t(row) * 6;
    const float2 a0 = sa[t + 1], am = sa[t], ap = sa[t + 2];
    out[0] = c.x * a0.x;
    out[1] = c.x * a0.y;
    out[2] = c.y * a0.x;
    out[3] = c.y * a0.y;
    out[4] = fmaf(c.z, am.x, c.w * ap.x);
    out[5] = fmaf(c.z, am.y, c.w * ap.y);
}

// ---------------------------------------------------------------------------
// analysis: block (j-tile, m, parity); thread = one ext row (degree K).
//   H_{f,K} = sum_{north p} Pt_K^m(x_p) [G_f(p) + (-1)^{K+m} G_f(p')],
// p' the mirror row; the table block is [nh][rows] so that threads of a warp
// read consecutive degrees.  G already carries (2 pi / M) w_p / sin(theta_p)
// (and sin(theta_p) for the scalar adjoint field).
template <int NF>
__global__ void __launch_bounds__(128) k_analysis(const float* __restrict__ pana, const float* __restrict__ gana,
                                                   float* __restrict__ hana, int N, int nh, int nlat) {
    pdl_launch();
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* S = reinterpret_cast<float*>(smem_raw);  // [nh][2 NF]
    const int m = blockIdx.y, par = blockIdx.z;
    const int ne = ext_even(N, m), no = ext_odd(N, m);
    const int nrows = par ? no : ne;
    if (int(blockIdx.x * blockDim.x) >= nrows) return;
    const int rowstart = ext_off(N, m) + (par ? ne : 0);
    for (int i = threadIdx.x; i < nh * NF; i += blockDim.x) {
        const int p = i / NF, f = i % NF;
        const int pr = nlat - 1 - p;
        const float* a = gana + gsyn_index(0, f, m, p, N, nlat) * 2;
        float ar = a[0], ai = a[1], br = 0.f, bi = 0.f;
        if (pr != p) {
            const float* b = gana + gsyn_index(0, f, m, pr, N, nlat) * 2;
            br = b[0];
            bi = b[1];
        }
        S[p * 2 * NF + 2 * f] = par ? ar - br : ar + br;
        S[p * 2 * NF + 2 * f + 1] = par ? ai - bi : ai + bi;
    }
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nrows) return;
    float acc[2 * NF];
#pragma unroll
    for (int f = 0; f < 2 * NF; ++f) acc[f] = 0.f;
    const float* Pa = pana + size_t(rowstart) * nh + j;
#pragma unroll 4
    for (int p = 0; p < nh; ++p) {
        const float pv = __ldg(Pa + size_t(p) * nrows);
        const float* sp = S + p * 2 * NF;
#pragma unroll
        for (int f = 0; f < 2 * NF; ++f) acc[f] = fma(pv, sp[f], acc[f]);
    }
    float* dst = hana + size_t(rowstart + j) * 2 * NF;
#pragma unroll
    for (int f = 0; f < 2 * NF; ++f) dst[f] = acc[f];
}

// ---------------------------------------------------------------------------
// finish: one thread per packed (L, m).
//   N_{L,m} = lambda^{-1/2} [ -i m H^theta_L
//             - (L eps_{L+1,m} H^phi_{L+1} - (L+1) eps_{L,m} H^phi_{L-1}) ]
// with the FP64 coefficients precomputed per entry:
// c = (lambda^{-1/2}, L eps_{L+1,m} lambda^{-1/2}, (L+1) eps_{L,m} lambda^{-1/2}, lambda).
// kind 0: out = forcing - nu lambda alpha - N              (Eq. (ode));
//         + 2 i omega_d m / lambda alpha, the Coriolis diagonal of
//         Eq. (Coriolis_ZLm), when the product leaves it out (omega_d = Omega)
// kind 1: out = N                                          (projection)
// kind 2: out = -nu lambda w - s_m (N + lambda^{1/2} H^rho_L)  (J^T w; alpha = w)
// One more use of the adjoint's operands: with part, the block's sum of
// <lambda dot_with, w>, the derivative in nu (as a kernel of its own after the
// finish, with its launch, 3.9 us).
__device__ __forceinline__ double lam_dot(int L, double2 a, double2 b) {
    return double(L) * (L + 1.0) * (a.x * b.x + a.y * b.y);
}

__global__ void k_finish(int kind, const double* __restrict__ hana, int nf, const double2* __restrict__ alpha,
                         const double2* __restrict__ forcing, double2* __restrict__ out,
                         const int2* __restrict__ lm, const double4_32a* __restrict__ finc, int N, double nu,
                         int n, double omega_d, int* __restrict__ emax, const double2* dot_with,
                         double* __restrict__ part) {
    pdl_launch();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // the analysis is done with the column exponents: zero for the next ring
    for (int j = i; j < 3 * (N + 1); j += gridDim.x * blockDim.x) emax[j] = 0;
    if (part) block_sum256(i < n ? lam_dot(lm[i].x, dot_with[i], alpha[i]) : 0.0, part);
    if (i >= n) return;
    const int L = lm[i].x, m = lm[i].y;
    const double4_32a c = finc[i];
    const double* hL = hana + size_t(ext_row(N, m, L)) * 2 * nf;
    const double* hU = hana + size_t(ext_row(N, m, L + 1)) * 2 * nf;
    const double htr = hL[0], hti = hL[1];
    const double hur = hU[2], hui = hU[3];
    double hdr = 0.0, hdi = 0.0;
    if (L - 1 >= m) {
        const double* hD = hana + size_t(ext_row(N, m, L - 1)) * 2 * nf;
        hdr = hD[2];
        hdi = hD[3];
    }
    const double cm = c.x * m;
    const double nr = cm * hti - (c.y * hur - c.z * hdr);
    const double ni = -cm * htr - (c.y * hui - c.z * hdi);
    const double lam = c.w;
    double2 r;
    if (kind == 0) {
        const double2 a = alpha[i];
        const double2 f = forcing ? forcing[i] : make_double2(0.0, 0.0);
        r.x = f.x - nu * lam * a.x - nr;
        r.y = f.y - nu * lam * a.y - ni;
        if (omega_d != 0.0) {
            const double cor = 2.0 * omega_d * m / lam;
            r.x -= cor * a.y;
            r.y += cor * a.x;
        }
    } else if (kind == 1) {
        r = make_double2(nr, ni);
    } else {
        const double2 wv = alpha[i];
        const double sm = m == 0 ? 1.0 : 2.0;
        const double sl = lam * c.x;  // lambda^{1/2}
        r.x = -nu * lam * wv.x - sm * (nr + sl * hL[4]);
        r.y = -nu * lam * wv.y - sm * (ni + sl * hL[5]);
    }
    out[i] = r;
}

// FP32-path finish: the recombination runs in FP32 on the FP32 projections
// (coefficients in FP32); only the state update f - nu lambda alpha - N is
// FP64.
__global__ void k_finish32(int kind, const float* __restrict__ hana, int nf, const double2* __restrict__ alpha,
                           const double2* __restrict__ forcing, double2* __restrict__ out,
                           const int2* __restrict__ lm, const float4* __restrict__ finc, int N, double nu, int n,
                           size_t hstride, const double* __restrict__ nu_inst, double omega_d,
                           const double2* dot_with, double* __restrict__ part) {
    pdl_launch();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n && !part) return;
    // the plan's constants are read before the wait for the predecessor
    int L, m;
    packed_lm(N, min(i, n - 1), L, m);
    (void)lm;
    const float4 c = finc[min(i, n - 1)];
    pdl_wait();
    if (part) {
        block_sum256(i < n ? lam_dot(L, dot_with[i], alpha[i]) : 0.0, part);
        if (i >= n) return;
    }
    // batch of instances along gridDim.y: per-instance vectors, projections, nu
    {
        const size_t b = blockIdx.y;
        hana += b * hstride;
        alpha += b * n;
        out += b * n;
        if (forcing) forcing += b * n;
        if (nu_inst) nu = nu_inst[b];
    }
    const float* hL = hana + size_t(ext_row(N, m, L)) * 2 * nf;
    const float* hU = hana + size_t(ext_row(N, m, L + 1)) * 2 * nf;
    const float* hD = L - 1 >= m ? hana + size_t(ext_row(N, m, L - 1)) * 2 * nf : nullptr;
    double2 r;
    if (kind < 2) {
        const double2 a = kind == 0 ? alpha[i] : make_double2(0.0, 0.0);
        const double2 f = kind == 0 && forcing ? forcing[i] : make_double2(0.0, 0.0);
        r = finish32_entry(kind, L, m, c, hL, hU, hD, a, f, nu, omega_d);
    } else {
        const float hdr = hD ? hD[2] : 0.f, hdi = hD ? hD[3] : 0.f;
        const float cm = c.x * float(m);
        const float nr = cm * hL[1] - (c.y * hU[2] - c.z * hdr);
        const float ni = -cm * hL[0] - (c.y * hU[3] - c.z * hdi);
        const double lam = double(L) * double(L + 1);
        const double2 wv = alpha[i];
        const float sm = m == 0 ? 1.f : 2.f;
        const float sl = c.w * c.x;  // lambda^{1/2}
        const double nl = nu * lam;
        r.x = -nl * wv.x - double(sm * (nr + sl * hL[4]));
        r.y = -nl * wv.y - double(sm * (ni + sl * hL[5]));
    }
    out[i] = r;
}

// ---------------------------------------------------------------------------
// launchers

template <int NF>
static int anal_t(sphnse_plan* P) {
    const int maxrows = ext_even(P->N, 0);
    dim3 blk(128), grd((maxrows + 127) / 128, P->N + 1, 2);
    size_t sm = size_t(P->nh) * 2 * NF * sizeof(float);
    if (sm > 48 * 1024) {
        allow_dynamic_smem(reinterpret_cast<const void*>(k_analysis<NF>), sm);
    }
    stage_begin(P, SPHNSE_STAGE_ANALYSIS);
    launch_pdl_small(P->n_cta, k_analysis<NF>, grd, blk, sm, P->stream,
               reinterpret_cast<const float*>(P->tab[SPHNSE_FP32].ana),
               reinterpret_cast<const float*>(P->d_gana), reinterpret_cast<float*>(P->d_hana), P->N, P->nh, P->nlat);
    stage_end(P, SPHNSE_STAGE_ANALYSIS);
    return check_cuda(cudaGetLastError());
}

int launch_analysis(sphnse_plan* P, int nfields) {
    if (ana32_ok(P)) return launch_analysis32(P, nfields);
    return nfields == 3 ? anal_t<3>(P) : anal_t<2>(P);
}

int launch_finish(sphnse_plan* P, int kind, int prec, const double* alpha, const double* forcing,
                  double* out, const double* dot_with) {
    const int n = P->n_coeff;
    const double2* dw = reinterpret_cast<const double2*>(dot_with);
    double* part = dot_with ? P->h_part : nullptr;
    const int nf = kind == 2 ? 3 : 2;
    dim3 blk(256), grd((n + 255) / 256);
    stage_begin(P, SPHNSE_STAGE_FINISH);
    if (prec == SPHNSE_FP64)
        launch_pdl_small(P->n_cta, k_finish, grd, blk, 0, P->stream, kind, static_cast<const double*>(P->d_hana), nf,
                                                     reinterpret_cast<const double2*>(alpha),
                                                     reinterpret_cast<const double2*>(forcing),
                                                     reinterpret_cast<double2*>(out), P->d_lm, P->d_finc, P->N, P->nu, n,
                                                     kind == 0 && P->coriolis_split ? P->Omega : 0.0, P->dig.emax, dw, part);
    else
        launch_pdl(k_finish32, grd, blk, 0, P->stream, kind, static_cast<const float*>(P->d_hana), nf,
                   reinterpret_cast<const double2*>(alpha), reinterpret_cast<const double2*>(forcing),
                   reinterpret_cast<double2*>(out), static_cast<const int2*>(P->d_lm),
                   static_cast<const float4*>(P->d_finc32), P->N, P->nu, n, size_t(0),
                   static_cast<const double*>(nullptr), kind == 0 && P->coriolis_split ? P->Omega : 0.0, dw, part);
    stage_end(P, SPHNSE_STAGE_FINISH);
    return check_cuda(cudaGetLastError());
}

// batched FP32 launchers over nb instances with fixed strides (ensemble)
int launch_prep32_batch(sphnse_plan* P, int nb, const double* alpha, float* bsyn, size_t bstride) {
    dim3 blk(128), grd((P->N + 2 + 127) / 128, P->N + 1, nb);
    stage_begin(P, SPHNSE_STAGE_PREP);
    launch_pdl(k_prep32, grd, blk, 0, P->stream, reinterpret_cast<const double2*>(alpha),
               static_cast<const float4*>(P->d_prepc32), bsyn, P->N, P->n_coeff, bstride);
    stage_end(P, SPHNSE_STAGE_PREP);
    return check_cuda(cudaGetLastError());
}

int launch_finish32_batch(sphnse_plan* P, int nb, const float* hana, size_t hstride, const double* alpha,
                          double* out, const double* nu_inst) {
    const int n = P->n_coeff;
    dim3 blk(256), grd((n + 255) / 256, nb);
    stage_begin(P, SPHNSE_STAGE_FINISH);
    launch_pdl(k_finish32, grd, blk, 0, P->stream, 0, hana, 2, reinterpret_cast<const double2*>(alpha),
               static_cast<const double2*>(nullptr), reinterpret_cast<double2*>(out),
               static_cast<const int2*>(P->d_lm), static_cast<const float4*>(P->d_finc32), P->N, P->nu, n, hstride,
               nu_inst, 0.0, static_cast<const double2*>(nullptr), static_cast<double*>(nullptr));
    stage_end(P, SPHNSE_STAGE_FINISH);
    return check_cuda(cudaGetLastError());
}

}  // namespace sph
