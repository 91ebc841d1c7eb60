// Longitude ("ring") kernel of the FP64 path in 64-bit fixed point (fx64.cuh),
// one CTA per pair of Gauss latitudes 2 j, 2 j + 1.
//
// RHS (Sec. 4.2: the phi sums of Eqs. (app_soln_rep), (eval_nonlin1) are
// Fourier sums, evaluated by FFT):
//   1. inverse FFTs of the Hermitian spectra g_m, |m| <= N (zero-padded to
//      M): zeta + i u_theta per ring, and u_phi of both rings in one signal
//   2. pointwise product (Eqs. (short_nonlin1), (C)):
//      q = zeta + 2 Omega cos(theta_p),  W_theta = -q u_phi,  W_phi = q u_theta
//   3. forward FFT of W_theta + i W_phi per ring, separation of the two real
//      spectra, truncation to m = 0..N, scaling by (2 pi / M) w_p / sin(theta_p)
// GRID writes zeta, u_theta, u_phi to grid rows; PROJECT transforms given grid
// rows of a tangential field; ADJOINT evaluates the transposed linearised
// product (fields zeta, u_theta, u_phi, v_theta, v_phi).
//
// M = nlon = 2^a 3^b; in-place Stockham autosort stages of radix 8, 4, 2, 9
// and 3 in shared memory.  Every thread holds its butterflies of a stage in
// registers (8 TPT complex values), the block synchronises, and writes them
// back.  Spectra are read and written in the latitude-pair-major layout
// [f][row / 2][m][row % 2] (a CTA's data are contiguous runs, and the
// order-major side of the Legendre kernels still moves whole 32-byte
// sectors), so no transpose runs between this kernel and the Legendre sums.
//
// Scaling: every real field of a ring is scaled by its own power of two so
// that the sum of its spectrum's magnitudes is below 2^60 (two shared-memory
// reductions: the largest exponent, then the sum of the leading 16 bits).
// Measured on the GB300 (event pairs, RHS): 369 us in FP64 arithmetic, 110 us
// here at L = 511 (1536 longitudes); 94 and 45 us at L = 255; 41 and 26 us at
// L = 100 (324 longitudes); 24.5 and 18.4 us at L = 31.  The FP64 form was
// bound by the FP64 pipe; this one by the integer multiply-adds and, for grids
// of less than a wave, by the chain of stages.  Against 64-bit references the
// errors of F, the fields and the projection are those of the FP64 form or
// smaller (u_theta at L = 511: 1.09e-15 against 1.31e-15).
// On the grid each factor of the product is shifted up to 2^61, and the
// products are rescaled by the sum of their magnitudes in the same way, so
// that no FFT intermediate overflows and all 60 bits are used.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>

#include "fx64.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace sph {

struct FxPlan {
    int n = 0, nst = 0;
    int radix[12];
};

static bool make_fx_plan(int n, FxPlan* p) {
    p->n = n;
    p->nst = 0;
    int r = n;
    for (int R : {8, 4, 2, 9, 3})
        while (r % R == 0 && p->nst < 12) {
            p->radix[p->nst++] = R;
            r /= R;
        }
    return r == 1;
}

// e^{-2 pi i t / M} as split Q62 pairs (cos hi, cos lo, -sin hi, -sin lo)
std::vector<int> ring_fx_twiddles(int M) {
    std::vector<int> tw(4 * size_t(M));
    for (int t = 0; t < M; ++t) {
        const long double ang = 2.0L * 3.14159265358979323846264338327950288L * t / M;
        const fx2 c = fx_split(llroundl(std::cos(ang) * 4611686018427387904.0L));
        long long sq = llroundl(-std::sin(ang) * 4611686018427387904.0L);
        // the inverse transform negates both halves of the sine
        if (fx_split(sq).l == INT_MIN) ++sq;
        const fx2 s = fx_split(sq);
        tw[4 * t] = c.h;
        tw[4 * t + 1] = c.l;
        tw[4 * t + 2] = s.h;
        tw[4 * t + 3] = s.l;
    }
    return tw;
}

struct RingFxArgs {
    int N, M, nlat;
    double two_omega;
    const double* x;       // cos(theta)
    const double* s;       // sin(theta)
    const double* rw;      // (2 pi / M) w_p / sin(theta_p)
    const double* gsyn;    // [nf][pair][N+1][2] complex
    double* gana;          // [nf][pair][N+1][2] complex
    const double* gin0;    // grid input rows (PROJECT)
    const double* gin1;
    double* gout0;         // grid output rows (GRID)
    double* gout1;
    double* gout2;
    const int4* tw;
    int* emax;             // [nf][N+1] largest biased exponents of gana (atomic maxima)
    FxPlan plan;
    int early;             // let the successor start its prologue at once
};

// one 16-byte slot of padding per eight, so that the stride-8 writes of the
// first radix-8 stage fall into different banks
__device__ __forceinline__ int fxp(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int fx_stride(int M) { return M + ((M + 7) >> 3); }

__device__ __forceinline__ cx<fx> fx_ld(const longlong2* p) {
    const longlong2 v = *p;
    return {{v.x}, {v.y}};
}
__device__ __forceinline__ void fx_st(longlong2* p, cx<fx> v) { *p = make_longlong2(v.x.v, v.y.v); }

// One in-place stage of radix R over NSIG signals; a thread's butterflies are
// t = tid + b NT (signal t / nb, butterfly t mod nb).
template <int R, int NSIG, int TPT, int S>
__device__ __forceinline__ void fx_stage(longlong2* buf, int M, int Ns, const int4* tw) {
    constexpr int MAXB = (8 * TPT + R - 1) / R;
    // the stage loop holds one copy of this body per radix: without this the
    // compiler hoists every copy's addresses out of the loop and spills them
    // (for the same reason an idle thread's values are set to zero below: left
    // undefined, they count as live around the loop)
    asm volatile("" : "+r"(M));
    const int nb = M / R, ld = fx_stride(M), step = M / (Ns * R);
    cx<fx> v[MAXB][R];
    int to[MAXB];   // base of the outputs; stride Ns
#pragma unroll
    for (int b = 0; b < MAXB; ++b) {
        int t = threadIdx.x + b * blockDim.x;
        if (t < NSIG * nb) {
            int sg = 0;
#pragma unroll
            for (int i = 1; i < NSIG; ++i)
                if (t >= nb) {
                    t -= nb;
                    ++sg;
                }
            const longlong2* src = buf + sg * ld;
            const int q = t / Ns, k = t - q * Ns;
            to[b] = sg * M + q * Ns * R + k;   // signal and index, unpadded
#pragma unroll
            for (int r = 0; r < R; ++r) v[b][r] = fx_ld(src + fxp(t + r * nb));
            if (Ns > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const int4 w = tw[k * r * step];
                    v[b][r] = S > 0 ? fx_cmul(v[b][r], {w.x, w.y}, {-w.z, -w.w})
                                    : fx_cmul(v[b][r], {w.x, w.y}, {w.z, w.w});
                }
            }
            fx_dft<R, S>(v[b]);
        } else {
            to[b] = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) v[b][r] = {{0}, {0}};
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < MAXB; ++b) {
        const int t = threadIdx.x + b * blockDim.x;
        if (t < NSIG * nb) {
            int i = to[b], sg = 0;
#pragma unroll
            for (int j = 1; j < NSIG; ++j)
                if (i >= M) {
                    i -= M;
                    ++sg;
                }
            longlong2* dst = buf + sg * ld;
#pragma unroll
            for (int r = 0; r < R; ++r) fx_st(dst + fxp(i + r * Ns), v[b][r]);
        }
    }
    __syncthreads();
}

template <int NSIG, int TPT, int S>
__device__ __forceinline__ void fx_fft(longlong2* buf, const FxPlan& plan, const int4* tw) {
    int Ns = 1;
    for (int st = 0; st < plan.nst; ++st) {
        const int R = plan.radix[st];
        if (R == 8) fx_stage<8, NSIG, TPT, S>(buf, plan.n, Ns, tw);
        else if (R == 4) fx_stage<4, NSIG, TPT, S>(buf, plan.n, Ns, tw);
        else if (R == 2) fx_stage<2, NSIG, TPT, S>(buf, plan.n, Ns, tw);
        else if (R == 9) fx_stage<9, NSIG, TPT, S>(buf, plan.n, Ns, tw);
        else fx_stage<3, NSIG, TPT, S>(buf, plan.n, Ns, tw);
        Ns *= R;
    }
}

// Block reductions of NV small integers per thread into shared slots
// (zeroed, and read after the next barrier).
template <int NV>
__device__ __forceinline__ void red_max(const int* v, int* slot) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int w = __reduce_max_sync(0xffffffffu, v[i]);
        if ((threadIdx.x & 31) == 0) atomicMax(slot + i, w);
    }
}
template <int NV>
__device__ __forceinline__ void red_add(const unsigned* v, unsigned* slot) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const unsigned w = __reduce_add_sync(0xffffffffu, v[i]);
        if ((threadIdx.x & 31) == 0) atomicAdd(slot + i, w);
    }
}
template <int NV>
__device__ __forceinline__ void red_or(const unsigned* v, unsigned* slot) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const unsigned w = __reduce_or_sync(0xffffffffu, v[i]);
        if ((threadIdx.x & 31) == 0) atomicOr(slot + i, w);
    }
}
__device__ __forceinline__ int bitlen(unsigned v) { return 32 - __clz(v); }
__device__ __forceinline__ unsigned hi_abs(long long v) { return unsigned((v ^ (v >> 63)) >> 32); }
__device__ __forceinline__ unsigned top16_abs(long long v) { return unsigned((v ^ (v >> 63)) >> 44) + 1u; }

// signals of a ring pair: inverse transforms, forward transforms
template <int MODE> struct FxMode {
    static constexpr int NF = MODE == RING_ADJOINT ? 5 : (MODE == RING_PROJECT ? 2 : 3);   // input fields
    static constexpr int NI = MODE == RING_ADJOINT ? 5 : (MODE == RING_PROJECT ? 0 : 3);   // inverse signals
    static constexpr int NO = MODE == RING_ADJOINT ? 3 : 2;                                // forward signals
    static constexpr int NS = NI > NO ? NI : NO;
};

// MODE and TPT (butterfly values per thread / 8) fix the launch shape:
// blockDim >= NS M / (8 TPT).
template <int MODE, int TPT>
__global__ void __launch_bounds__(MODE == RING_ADJOINT ? 512 : 288, MODE == RING_ADJOINT ? 1 : 2) k_ring_fx(RingFxArgs a) {
    using Q = FxMode<MODE>;
    constexpr int NF = Q::NF, NS = Q::NS;
    extern __shared__ __align__(16) unsigned char smem_fx[];
    __shared__ int s_emax[2 * NF];
    __shared__ unsigned s_sum[2 * NF], s_or[2 * NF], s_sum2[6];
    const int M = a.M, N = a.N, nlat = a.nlat, ld = fx_stride(M), tid = threadIdx.x, NT = blockDim.x;
    longlong2* buf = reinterpret_cast<longlong2*>(smem_fx);
    int4* tw = reinterpret_cast<int4*>(buf + NS * ld);
    const int pair = blockIdx.x, npair = (nlat + 1) / 2, row0 = 2 * pair;
    const bool two = row0 + 1 < nlat;
    if (a.early) pdl_launch();
    // the plan's constants do not depend on the predecessor
    for (int t = tid; t < M; t += NT) tw[t] = a.tw[t];
    if (tid < 2 * NF) {
        s_emax[tid] = 0;
        s_sum[tid] = 0u;
        s_or[tid] = 0u;
    }
    if (tid < 6) s_sum2[tid] = 0u;
    const double fc[2] = {a.two_omega * a.x[row0], two ? a.two_omega * a.x[row0 + 1] : 0.0};
    double scale[2] = {MODE == RING_GRID ? 1.0 : a.rw[row0], MODE == RING_GRID ? 1.0 : (two ? a.rw[row0 + 1] : 0.0)};
    pdl_wait();
    int kf[2 * NF];   // fixed point = value 2^kf, of field f of ring r at 2 f + r

    if constexpr (MODE != RING_PROJECT) {
        // a thread owns the orders m = tid + i NT of every field and both rings
        constexpr int NM = TPT;
        double x[NM][NF][4];
        int em[2 * NF];
#pragma unroll
        for (int i = 0; i < 2 * NF; ++i) em[i] = 0;
#pragma unroll
        for (int i = 0; i < NM; ++i) {
            const int m = tid + i * NT;
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                double4_32a g = make_double4_32a(0.0, 0.0, 0.0, 0.0);
                if (m <= N)
                    g = *reinterpret_cast<const double4_32a*>(a.gsyn +
                                                              ((size_t(f) * npair + pair) * size_t(N + 1) + m) * 4);
                x[i][f][0] = g.x;
                x[i][f][1] = m == 0 ? 0.0 : g.y;   // fields are real
                x[i][f][2] = two ? g.z : 0.0;
                x[i][f][3] = two && m != 0 ? g.w : 0.0;
                if (f == 0 && m == 0 && MODE != RING_GRID) {   // q = zeta + 2 Omega cos(theta)
                    x[i][f][0] += fc[0];
                    x[i][f][2] += fc[1];
                }
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    em[2 * f + r] = max(em[2 * f + r], max(f64_bexp(x[i][f][2 * r]), f64_bexp(x[i][f][2 * r + 1])));
            }
        }
        __syncthreads();   // the slots are zero
        red_max<2 * NF>(em, s_emax);
        __syncthreads();
        unsigned sm[2 * NF];
#pragma unroll
        for (int j = 0; j < 2 * NF; ++j) {
            const int E = max(s_emax[j], 1);
            em[j] = E;
            sm[j] = 0u;
#pragma unroll
            for (int i = 0; i < NM; ++i) {
                const int m = tid + i * NT;
                const unsigned v = f64_top16(x[i][j / 2][2 * (j & 1)], E) + f64_top16(x[i][j / 2][2 * (j & 1) + 1], E);
                if (m <= N) sm[j] += m == 0 ? v : 2u * v;
            }
        }
        red_add<2 * NF>(sm, s_sum);
        // the zero-padded middle of every inverse signal
        for (int m = N + 1 + tid; m < M - N; m += NT)
#pragma unroll
            for (int sg = 0; sg < Q::NI; ++sg) buf[sg * ld + fxp(m)] = make_longlong2(0, 0);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 2 * NF; ++j) {
            kf[j] = 1072 - em[j] + 26 - bitlen(s_sum[j]);
            // a non-finite input makes its ring's outputs NaN
            if (em[j] == 2047) scale[j & 1] = __longlong_as_double(0x7FF8000000000000LL);
        }
        // signals: RHS, GRID: (zeta, u_theta) of each ring, (u_phi, u_phi) of
        // both; ADJOINT: (zeta, u_theta), (u_phi, v_theta) of each ring,
        // (v_phi, v_phi) of both
#pragma unroll
        for (int i = 0; i < NM; ++i) {
            const int m = tid + i * NT;
            if (m > N) continue;
            auto put = [&](int sg, int fa, int ra, int fb, int rb) {
                const long long ax = f64_to_fx(x[i][fa][2 * ra], kf[2 * fa + ra]);
                const long long ay = f64_to_fx(x[i][fa][2 * ra + 1], kf[2 * fa + ra]);
                const long long bx = f64_to_fx(x[i][fb][2 * rb], kf[2 * fb + rb]);
                const long long by = f64_to_fx(x[i][fb][2 * rb + 1], kf[2 * fb + rb]);
                buf[sg * ld + fxp(m)] = make_longlong2(ax - by, ay + bx);
                if (m > 0) buf[sg * ld + fxp(M - m)] = make_longlong2(ax + by, bx - ay);
            };
            put(0, 0, 0, 1, 0);
            put(1, 0, 1, 1, 1);
            if constexpr (MODE == RING_ADJOINT) {
                put(2, 2, 0, 3, 0);
                put(3, 2, 1, 3, 1);
                put(4, 4, 0, 4, 1);
            } else {
                put(2, 2, 0, 2, 1);
            }
        }
        __syncthreads();
        fx_fft<Q::NI, TPT, +1>(buf, a.plan, tw);
    }

    if constexpr (MODE == RING_GRID) {
        for (int q = tid; q < M; q += NT) {
            const longlong2 B = buf[2 * ld + fxp(q)];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (r == 1 && !two) break;
                const longlong2 A = buf[r * ld + fxp(q)];
                const size_t o = size_t(row0 + r) * M + q;
                if (a.gout0) a.gout0[o] = f64_scale(__ll2double_rn(A.x) * scale[r], -kf[r]);
                if (a.gout1) a.gout1[o] = f64_scale(__ll2double_rn(A.y) * scale[r], -kf[2 + r]);
                if (a.gout2) a.gout2[o] = f64_scale(__ll2double_rn(r ? B.y : B.x) * scale[r], -kf[4 + r]);
            }
        }
        return;
    }

    // W (fields to transform): value j = 2 c + r, c = 0, 1: the two components
    // of ring r's signal; ADJOINT also c = 2: rho of ring r
    constexpr int NW = MODE == RING_ADJOINT ? 6 : 4;
    constexpr int NQ = (8 * TPT + NS - 1) / NS;   // grid points per thread
    int kw[NW];
    long long w[NQ][NW];
    if constexpr (MODE == RING_PROJECT) {
        double x[NQ][4];
        int em[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = tid + i * NT;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = j / 2, r = j & 1;
                x[i][j] = 0.0;
                if (q < M && (r == 0 || two)) x[i][j] = (c ? a.gin1 : a.gin0)[size_t(row0 + r) * M + q];
                em[j] = max(em[j], f64_bexp(x[i][j]));
            }
        }
        __syncthreads();
        red_max<4>(em, s_emax);
        __syncthreads();
        unsigned sm[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            em[j] = max(s_emax[j], 1);
            sm[j] = 0u;
#pragma unroll
            for (int i = 0; i < NQ; ++i)
                if (tid + i * NT < M) sm[j] += f64_top16(x[i][j], em[j]);
        }
        red_add<4>(sm, s_sum);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            kw[j] = 1072 - em[j] + 26 - bitlen(s_sum[j]);
            if (em[j] == 2047) scale[j & 1] = __longlong_as_double(0x7FF8000000000000LL);
#pragma unroll
            for (int i = 0; i < NQ; ++i) w[i][j] = f64_to_fx(x[i][j], kw[j]);
        }
    } else {
        // the grid values of point q: fields 2 f + r
        auto fields = [&](int q, long long* v) {
            const longlong2 A0 = buf[fxp(q)], A1 = buf[ld + fxp(q)];
            v[0] = A0.x; v[1] = A1.x; v[2] = A0.y; v[3] = A1.y;
            if constexpr (MODE == RING_ADJOINT) {
                const longlong2 B0 = buf[2 * ld + fxp(q)], B1 = buf[3 * ld + fxp(q)], C = buf[4 * ld + fxp(q)];
                v[4] = B0.x; v[5] = B1.x; v[6] = B0.y; v[7] = B1.y; v[8] = C.x; v[9] = C.y;
            } else {
                const longlong2 B = buf[2 * ld + fxp(q)];
                v[4] = B.x; v[5] = B.y;
            }
        };
        unsigned om[2 * NF];
#pragma unroll
        for (int j = 0; j < 2 * NF; ++j) om[j] = 0u;
        for (int q = tid; q < M; q += NT) {
            long long v[2 * NF];
            fields(q, v);
#pragma unroll
            for (int j = 0; j < 2 * NF; ++j) om[j] |= hi_abs(v[j]);
        }
        red_or<2 * NF>(om, s_or);
        __syncthreads();
        int up[2 * NF];   // left shift of a field to |v| < 2^61
#pragma unroll
        for (int j = 0; j < 2 * NF; ++j) {
            up[j] = max(0, 29 - bitlen(s_or[j]));
            kf[j] += up[j];
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if constexpr (MODE == RING_RHS) {
                kw[r] = kf[r] + kf[4 + r] - 62;        // W_theta = -q u_phi
                kw[2 + r] = kf[r] + kf[2 + r] - 62;    // W_phi = q u_theta
            } else {
                kw[r] = kf[r] + kf[8 + r] - 62;        // X_theta = q v_phi
                kw[2 + r] = kf[r] + kf[6 + r] - 62;    // X_phi = -q v_theta
                // rho = -v_theta u_phi + v_phi u_theta, at the coarser scale of the two
                kw[4 + r] = min(kf[6 + r] + kf[4 + r], kf[8 + r] + kf[2 + r]) - 62;
            }
        }
        unsigned sm[NW];
#pragma unroll
        for (int j = 0; j < NW; ++j) sm[j] = 0u;
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = tid + i * NT;
#pragma unroll
            for (int j = 0; j < NW; ++j) w[i][j] = 0;
            if (q < M) {
                long long v[2 * NF];
                fields(q, v);
#pragma unroll
                for (int j = 0; j < 2 * NF; ++j) v[j] <<= up[j];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if constexpr (MODE == RING_RHS) {
                        w[i][r] = -fx_mul62(v[r], v[4 + r]);
                        w[i][2 + r] = fx_mul62(v[r], v[2 + r]);
                    } else {
                        w[i][r] = fx_mul62(v[r], v[8 + r]);
                        w[i][2 + r] = -fx_mul62(v[r], v[6 + r]);
                        const int d1 = kw[4 + r] + 62 - kf[6 + r] - kf[4 + r];
                        const int d2 = kw[4 + r] + 62 - kf[8 + r] - kf[2 + r];
                        w[i][4 + r] = fx_shift(fx_mul62(v[8 + r], v[2 + r]), d2) -
                                      fx_shift(fx_mul62(v[6 + r], v[4 + r]), d1);
                    }
                }
#pragma unroll
                for (int j = 0; j < NW; ++j) sm[j] += top16_abs(w[i][j]);
            }
        }
        red_add<NW>(sm, s_sum2);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NW; ++j) {
            const int sh = 16 - bitlen(s_sum2[j]);
            kw[j] += sh;
#pragma unroll
            for (int i = 0; i < NQ; ++i) w[i][j] = fx_shift(w[i][j], sh);
        }
    }
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const int q = tid + i * NT;
        if (q >= M) continue;
        buf[fxp(q)] = make_longlong2(w[i][0], w[i][2]);
        buf[ld + fxp(q)] = make_longlong2(w[i][1], w[i][3]);
        if constexpr (MODE == RING_ADJOINT) buf[2 * ld + fxp(q)] = make_longlong2(w[i][4], w[i][5]);
    }
    __syncthreads();
    fx_fft<Q::NO, TPT, -1>(buf, a.plan, tw);

    // separate the real spectra: of Z = A + i B, A_m = (Z_m + conj Z_{M-m}) / 2,
    // B_m = (Z_m - conj Z_{M-m}) / (2 i); truncate, weight, store
    const double sn[2] = {MODE == RING_ADJOINT ? a.s[row0] : 0.0, MODE == RING_ADJOINT && two ? a.s[row0 + 1] : 0.0};
    for (int m = tid; m <= N; m += NT) {
        const int mr = m == 0 ? 0 : M - m;
        double4_32a o[3];
        auto cv = [&](long long v, double sc, int k) { return f64_scale(__ll2double_rn(v) * sc, -k - 1); };
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const longlong2 p = buf[r * ld + fxp(m)], z = buf[r * ld + fxp(mr)];
            const double tx = cv(p.x + z.x, scale[r], kw[r]), ty = cv(p.y - z.y, scale[r], kw[r]);
            const double fx_ = cv(p.y + z.y, scale[r], kw[2 + r]), fy = cv(z.x - p.x, scale[r], kw[2 + r]);
            if (r == 0) {
                o[0].x = tx; o[0].y = ty; o[1].x = fx_; o[1].y = fy;
            } else {
                o[0].z = tx; o[0].w = ty; o[1].z = fx_; o[1].w = fy;
            }
        }
        if constexpr (MODE == RING_ADJOINT) {
            // rho of the two rings: plain quadrature weight (2 pi / M) w_p
            const longlong2 p = buf[2 * ld + fxp(m)], z = buf[2 * ld + fxp(mr)];
            o[2].x = cv(p.x + z.x, scale[0] * sn[0], kw[4]);
            o[2].y = cv(p.y - z.y, scale[0] * sn[0], kw[4]);
            o[2].z = cv(p.y + z.y, scale[1] * sn[1], kw[5]);
            o[2].w = cv(z.x - p.x, scale[1] * sn[1], kw[5]);
        }
#pragma unroll
        for (int f = 0; f < (MODE == RING_ADJOINT ? 3 : 2); ++f)
        {
            *reinterpret_cast<double4_32a*>(a.gana + ((size_t(f) * npair + pair) * size_t(N + 1) + m) * 4) = o[f];
            // the column scales of the analysis
            atomicMax(a.emax + f * (N + 1) + m,
                      max(max(f64_bexp(o[f].x), f64_bexp(o[f].y)), max(f64_bexp(o[f].z), f64_bexp(o[f].w))));
        }
    }
}

template <int MODE, int TPT>
static cudaError_t ring_fx_t(sphnse_plan* P, RingFxArgs a) {
    constexpr int NS = FxMode<MODE>::NS;
    const int threads = ((NS * a.M + 8 * TPT - 1) / (8 * TPT) + 31) / 32 * 32;
    const size_t sm = size_t(NS) * fx_stride(a.M) * 16 + size_t(a.M) * 16;
    allow_dynamic_smem(reinterpret_cast<const void*>(k_ring_fx<MODE, TPT>), sm);
    const int grid = (a.nlat + 1) / 2;
    a.early = grid <= 2 * P->nsm;
    return launch_pdl(k_ring_fx<MODE, TPT>, dim3(grid), dim3(threads), sm, P->stream, a);
}

template <int MODE>
static cudaError_t ring_fx_m(sphnse_plan* P, const RingFxArgs& a) {
    // one butterfly of eight per thread while the block fits its bound
    constexpr int most = MODE == RING_ADJOINT ? 512 : 288;
    return FxMode<MODE>::NS * a.M <= 8 * most ? ring_fx_t<MODE, 1>(P, a) : ring_fx_t<MODE, 2>(P, a);
}

int launch_ring_fx(sphnse_plan* P, int mode, const double* gin0, const double* gin1, double* gout0, double* gout1,
                   double* gout2) {
    RingFxArgs a;
    if (!make_fx_plan(P->nlon, &a.plan)) return SPHNSE_E_UNSUPPORTED;
    a.N = P->N;
    a.M = P->nlon;
    a.nlat = P->nlat;
    a.two_omega = mode == RING_RHS && P->coriolis_split ? 0.0 : 2.0 * P->Omega;
    a.x = P->d_x;
    a.s = P->d_s;
    a.rw = P->d_rw;
    a.gsyn = static_cast<const double*>(P->d_gsyn);
    a.gana = static_cast<double*>(P->d_gana);
    a.gin0 = gin0;
    a.gin1 = gin1;
    a.gout0 = gout0;
    a.gout1 = gout1;
    a.gout2 = gout2;
    a.tw = P->d_fxtw;
    a.emax = P->dig.emax;
    stage_begin(P, SPHNSE_STAGE_RING);
    cudaError_t e;
    switch (mode) {
        case RING_RHS: e = ring_fx_m<RING_RHS>(P, a); break;
        case RING_GRID: e = ring_fx_m<RING_GRID>(P, a); break;
        case RING_PROJECT: e = ring_fx_m<RING_PROJECT>(P, a); break;
        default: e = ring_fx_m<RING_ADJOINT>(P, a); break;
    }
    stage_end(P, SPHNSE_STAGE_RING);
    return check_cuda(e);
}

}  // namespace sph
