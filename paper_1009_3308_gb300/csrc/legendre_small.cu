// FP64 Legendre synthesis and analysis for small plans (SMALL_NH northern
// latitudes at most): one block per order, multiply-adds on the FP64 pipe.
//
// These calls are latency: the digit-split tensor-core sums (legendre_dig.cu)
// spend their time on column scales, digits, TMEM and barriers, ten times their
// MMAs at L = 31, while the whole table is 24 x 560 entries.  Here a block
// holds everything of its order: it requests its part of the table before it
// waits for the predecessor, builds the coefficient sets itself, splits the
// degrees (latitudes) over its threads and, in the analysis, goes on to the
// recombination and diagonal update of its order, so an RHS is three launches.
// Larger plans are bound by the FP64 pipe here (two operations per clock per
// SM) and take the tensor cores.
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace sph {

struct SmallArgs {
    const double* table;   // [n_ext][nh]
    const double2* alpha;
    const double2* beta;   // adjoint: fields 3, 4 (scaled by 1 / s_m)
    const double4_32a* prepc;
    const double* isin;    // 1 / sin(theta_p)
    double* gsyn;          // [nf][pair][N+1][2] complex
    const double* gana;
    const double2* forcing;
    double2* out;
    const double2* dot_with;   // kind 2, with part: sums of <lambda dot_with, alpha>
    double* part;
    const double4_32a* finc;
    int N, nh, nlat, kind;
    double nu, omega_d;
};

constexpr int SM_U = 8;               // synthesis: table entries a thread requests ahead
constexpr int SM_P = SMALL_NH / 4;    // analysis: latitudes of a thread (four threads per row)

template <int NF>
__global__ void __launch_bounds__(256) k_syn_small(SmallArgs a) {
    constexpr int C = 2 * NF;
    extern __shared__ __align__(16) double sms[];
    const int N = a.N, nh = a.nh, nlat = a.nlat, m = blockIdx.x, tid = threadIdx.x;
    const int ne = ext_even(N, m), no = ext_odd(N, m), cnt = ne + no, e0 = ext_off(N, m);
    double* B = sms;              // [cnt][C]
    double* part = B + cnt * C;   // [split][even and odd columns][C]
    const int ncol = 2 * nh, S = 256 / ncol, col = tid % ncol, sp = tid / ncol;
    const int par = col >= nh, p = col - par * nh, n = sp < S ? (par ? no : ne) : 0;
    const double* src = a.table + size_t(e0 + (par ? ne : 0)) * nh + p;
    // this thread's degrees: a run, and the runs are added from the highest on, so
    // that few roundings happen at the size of the low degrees' terms, which cancel
    // in u_phi (dealt out in turn, u_phi at L = 31 had a mean error of 7.4e-16, this
    // way 5.7e-16, one sequential sum 6.1e-16)
    const int len = (n + S - 1) / S, jb = sp * len, je = min(jb + len, n);
    pdl_launch();
    // the table does not depend on the predecessor
    double pv[SM_U];
#pragma unroll
    for (int u = 0; u < SM_U; ++u) {
        const int j = jb + u;
        pv[u] = j >= jb && j < je ? src[size_t(j) * nh] : 0.0;
    }
    pdl_wait();
    const int lo = m > 0 ? m : 1, pk = packed_off(N, m) - lo;
    const double sc = m == 0 ? 1.0 : 0.5;
    for (int i = tid; i < cnt; i += 256) {
        const int K = i < ne ? m + 2 * i : m + 1 + 2 * (i - ne);
        const double4_32a c = a.prepc[e0 + i];
        auto A = [&](const double2* v, int Kp) -> double2 {
            return (Kp < lo || Kp > N) ? make_double2(0.0, 0.0) : v[pk + Kp];
        };
        double* o = B + i * C;
        const double2 a0 = A(a.alpha, K), am = A(a.alpha, K - 1), ap = A(a.alpha, K + 1);
        o[0] = c.x * a0.x;
        o[1] = c.x * a0.y;
        o[2] = c.y * a0.x;
        o[3] = c.y * a0.y;
        o[4] = c.z * am.x + c.w * ap.x;
        o[5] = c.z * am.y + c.w * ap.y;
        if constexpr (NF == 5) {
            const double2 b0 = A(a.beta, K), bm = A(a.beta, K - 1), bp = A(a.beta, K + 1);
            o[6] = sc * (c.y * b0.x);
            o[7] = sc * (c.y * b0.y);
            o[8] = sc * (c.z * bm.x + c.w * bp.x);
            o[9] = sc * (c.z * bm.y + c.w * bp.y);
        }
    }
    __syncthreads();
    double acc[C];
#pragma unroll
    for (int f = 0; f < C; ++f) acc[f] = 0.0;
    const double* bb = B + (par ? ne : 0) * C;
    for (int t0 = 0; t0 < je - jb; t0 += SM_U) {
        if (t0 > 0)
#pragma unroll
            for (int u = 0; u < SM_U; ++u) {
                const int j = jb + t0 + u;
                pv[u] = j >= jb && j < je ? src[size_t(j) * nh] : 0.0;
            }
#pragma unroll
        for (int u = 0; u < SM_U; ++u) {
            const int j = jb + t0 + u;
            if (t0 + u >= je - jb) break;
#pragma unroll
            for (int f = 0; f < C; ++f) acc[f] = fma(pv[u], bb[j * C + f], acc[f]);
        }
    }
    if (sp < S)
#pragma unroll
        for (int f = 0; f < C; ++f) part[(sp * ncol + col) * C + f] = acc[f];
    __syncthreads();
    // north = E + O, south = E - O
    for (int t = tid; t < ncol * NF; t += 256) {
        const int q = t % nh, hemi = (t / nh) & 1, f = t / ncol;
        const int row = hemi ? nlat - 1 - q : q;
        if (hemi && row == q) continue;   // equator of an odd grid
        double gr = 0.0, gi = 0.0, hr = 0.0, hi = 0.0;
        for (int s = S - 1; s >= 0; --s) {
            const double* E = part + (s * ncol + q) * C + 2 * f;
            const double* O = E + nh * C;
            gr += E[0];
            gi += E[1];
            hr += O[0];
            hi += O[1];
        }
        gr = hemi ? gr - hr : gr + hr;
        gi = hemi ? gi - hi : gi + hi;
        const double inv = a.isin[q];
        double2 o;
        if (f == 0) o = make_double2(gr, gi);
        else if (f == 1 || f == 3) o = make_double2(-gi * (inv * m), gr * (inv * m));   // (i m / sin) g
        else o = make_double2(-gr * inv, -gi * inv);                                    // -(1 / sin) g
        *reinterpret_cast<double2*>(a.gsyn + gsyn_index(1, f, m, row, N, nlat) * 2) = o;
    }
}

// Analysis and finish (kind 0: F, 1: projection, 2: J^T w; see k_finish).
template <int NF>
__global__ void __launch_bounds__(256) k_ana_small(SmallArgs a) {
    constexpr int C = 2 * NF;
    extern __shared__ __align__(16) double sms[];
    const int N = a.N, nh = a.nh, nlat = a.nlat, m = blockIdx.x, tid = threadIdx.x;
    const int ne = ext_even(N, m), cnt = ext_count(N, m), e0 = ext_off(N, m);
    static_assert((4 * SMALL_NH - 2) / 3 + 2 <= 64, "rows per block");
    double* S = sms;               // [parity][C][nh]: G(p) + G(p'), G(p) - G(p')
    double* H = S + 2 * C * nh;    // [cnt][C]
    // four threads per row; every row of the order (at most 55) and every degree
    // (at most 53) has its threads
    const int sp = tid & 3, row = tid >> 2;
    const double* tab = a.table + size_t(e0 + min(row, cnt - 1)) * nh;
    const int lo = m > 0 ? m : 1, L = lo + tid, i = packed_off(N, m) + tid;
    pdl_launch();
    double pv[SM_P];
#pragma unroll
    for (int u = 0; u < SM_P; ++u) {
        const int p = sp + 4 * u;
        pv[u] = p < nh ? tab[p] : 0.0;
    }
    double4_32a c = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    if (L <= N) c = a.finc[i];
    pdl_wait();
    double2 x = make_double2(0.0, 0.0), fo = x;
    if (L <= N && a.kind != 1) x = a.alpha[i];
    if (L <= N && a.forcing) fo = a.forcing[i];
    for (int t = tid; t < nh * NF; t += 256) {
        const int f = t / nh, p = t % nh, pr = nlat - 1 - p;
        const double2 v = *reinterpret_cast<const double2*>(a.gana + gsyn_index(1, f, m, p, N, nlat) * 2);
        double2 y = make_double2(0.0, 0.0);
        if (pr != p) y = *reinterpret_cast<const double2*>(a.gana + gsyn_index(1, f, m, pr, N, nlat) * 2);
        S[(2 * f) * nh + p] = v.x + y.x;
        S[(2 * f + 1) * nh + p] = v.y + y.y;
        S[(C + 2 * f) * nh + p] = v.x - y.x;
        S[(C + 2 * f + 1) * nh + p] = v.y - y.y;
    }
    __syncthreads();
    {
        const double* s = S + (row >= ne ? C * nh : 0) + sp;
        double acc[C];
#pragma unroll
        for (int f = 0; f < C; ++f) acc[f] = 0.0;
#pragma unroll
        for (int u = 0; u < SM_P; ++u)
            if (sp + 4 * u < nh)
#pragma unroll
                for (int f = 0; f < C; ++f) acc[f] = fma(pv[u], s[f * nh + 4 * u], acc[f]);
#pragma unroll
        for (int f = 0; f < C; ++f)
#pragma unroll
            for (int o = 2; o > 0; o >>= 1) acc[f] += __shfl_xor_sync(0xffffffffu, acc[f], o);
        if (sp == 0 && row < cnt)
#pragma unroll
            for (int f = 0; f < C; ++f) H[row * C + f] = acc[f];
    }
    __syncthreads();
    if (a.part) {
        double s = 0.0;
        if (L <= N) {
            const double2 v = a.dot_with[i];
            s = double(L) * (L + 1.0) * (v.x * x.x + v.y * x.y);
        }
        block_sum256(s, a.part);
    }
    if (L > N) return;
    const double* hL = H + (ext_row(N, m, L) - e0) * C;
    const double* hU = H + (ext_row(N, m, L + 1) - e0) * C;
    double hdr = 0.0, hdi = 0.0;
    if (L - 1 >= m) {
        const double* hD = H + (ext_row(N, m, L - 1) - e0) * C;
        hdr = hD[2];
        hdi = hD[3];
    }
    const double cm = c.x * m;
    const double nr = cm * hL[1] - (c.y * hU[2] - c.z * hdr);
    const double ni = -cm * hL[0] - (c.y * hU[3] - c.z * hdi);
    const double lam = c.w;
    double2 r;
    if (a.kind == 0) {
        r.x = fo.x - a.nu * lam * x.x - nr;
        r.y = fo.y - a.nu * lam * x.y - ni;
        if (a.omega_d != 0.0) {
            const double cor = 2.0 * a.omega_d * m / lam;
            r.x -= cor * x.y;
            r.y += cor * x.x;
        }
    } else if (a.kind == 1) {
        r = make_double2(nr, ni);
    } else {
        const double sm = m == 0 ? 1.0 : 2.0, sl = lam * c.x;
        double rho0 = 0.0, rho1 = 0.0;
        if constexpr (NF == 3) {
            rho0 = hL[4];
            rho1 = hL[5];
        }
        r.x = -a.nu * lam * x.x - sm * (nr + sl * rho0);
        r.y = -a.nu * lam * x.y - sm * (ni + sl * rho1);
    }
    a.out[i] = r;
}

// ---------------------------------------------------------------------------

static SmallArgs small_args(sphnse_plan* P) {
    SmallArgs a{};
    a.table = static_cast<const double*>(P->tab[SPHNSE_FP64].syn);
    a.prepc = P->d_prepc;
    a.isin = P->d_isin;
    a.gsyn = static_cast<double*>(P->d_gsyn);
    a.gana = static_cast<const double*>(P->d_gana);
    a.finc = P->d_finc;
    a.N = P->N;
    a.nh = P->nh;
    a.nlat = P->nlat;
    a.nu = P->nu;
    return a;
}

int launch_synthesis_small(sphnse_plan* P, const double* alpha, const double* beta) {
    SmallArgs a = small_args(P);
    a.alpha = reinterpret_cast<const double2*>(alpha);
    a.beta = reinterpret_cast<const double2*>(beta);
    const int C = beta ? 10 : 6, S = 256 / (2 * P->nh);
    const size_t sm = size_t(C) * (P->N + 2 + S * 2 * P->nh) * sizeof(double);
    stage_begin(P, SPHNSE_STAGE_SYNTHESIS);
    const cudaError_t e = beta ? launch_pdl(k_syn_small<5>, dim3(P->N + 1), dim3(256), sm, P->stream, a)
                               : launch_pdl(k_syn_small<3>, dim3(P->N + 1), dim3(256), sm, P->stream, a);
    stage_end(P, SPHNSE_STAGE_SYNTHESIS);
    return check_cuda(e);
}

int launch_analysis_small(sphnse_plan* P, int kind, const double* alpha, const double* forcing, double* out,
                          const double* dot_with) {
    SmallArgs a = small_args(P);
    a.dot_with = reinterpret_cast<const double2*>(dot_with);
    a.part = dot_with ? P->h_part : nullptr;
    a.alpha = reinterpret_cast<const double2*>(alpha);
    a.forcing = reinterpret_cast<const double2*>(forcing);
    a.out = reinterpret_cast<double2*>(out);
    a.kind = kind;
    a.omega_d = kind == 0 && P->coriolis_split ? P->Omega : 0.0;
    const int C = kind == 2 ? 6 : 4;
    const size_t sm = size_t(C) * (P->N + 2 + 2 * P->nh) * sizeof(double);
    stage_begin(P, SPHNSE_STAGE_ANALYSIS);
    const cudaError_t e = kind == 2 ? launch_pdl(k_ana_small<3>, dim3(P->N + 1), dim3(256), sm, P->stream, a)
                                    : launch_pdl(k_ana_small<2>, dim3(P->N + 1), dim3(256), sm, P->stream, a);
    stage_end(P, SPHNSE_STAGE_ANALYSIS);
    return check_cuda(e);
}

}  // namespace sph
