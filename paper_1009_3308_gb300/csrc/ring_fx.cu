// Longitude ("ring") kernel of the FP64 path in 64-bit fixed point (fx64.cuh),
// one CTA per pair of Gauss latitudes 2 j, 2 j + 1 (ADJOINT: per latitude).
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
// M = nlon = 2^a 3^b; Stockham autosort stages of radix 8, 4, 2, 9 and 3 from
// one shared-memory buffer to the other, one barrier each.  Small grids are
// bound by instruction fetch (each instruction runs a few times per CTA: half
// of the issue slots of the first form, whose in-place stages were unrolled
// per direction and signal count, waited for instructions at L = 31 .. 255),
// so one rolled copy of each radix serves both directions: the inverse
// transform is the forward one with real and imaginary parts exchanged.
// Spectra are read and written in the latitude-pair-major layout
// [f][row / 2][m][row % 2] (a CTA's data are contiguous runs, and the
// order-major side of the Legendre kernels still moves whole 32-byte
// sectors), so no transpose runs between this kernel and the Legendre sums.
//
// Scaling: every real field of a ring is scaled by its own power of two so
// that the sum of its spectrum's magnitudes is below 2^60 (two shared-memory
// reductions: the largest exponent, then the sum of the leading 16 bits).
// Measured on the GB300 (event pairs, RHS): 369 us in FP64 arithmetic, 99 us
// here at L = 511 (1536 longitudes); 94 and 37 us at L = 255; 41 and 20 us at
// L = 100 (324 longitudes); 24.5 and 14.4 us at L = 31.  The FP64 form was
// bound by the FP64 pipe; this one by the integer multiply-adds and, for grids
// of less than a wave, by the chain of stages.  Against 64-bit references the
// errors of F, the fields and the projection are those of the FP64 form or
// smaller (u_theta at L = 511: 1.09e-15 against 1.31e-15).
// On the grid each factor of the product is shifted up to 2^61, and the
// products are rescaled by the sum of their magnitudes in the same way, so
// that no FFT intermediate overflows and all 60 bits are used.
#include <cuda_runtime.h>

#include <algorithm>
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

// e^{-2 pi i t / M} as split Q62 pairs (cos hi, cos lo, -sin hi, -sin lo); M is
// even.  The extended-precision functions, slow where long double is emulated,
// run at about 2 sqrt(M / 4) angles: a quarter (half) of the circle is their
// products, the rest reflections.
std::vector<int> ring_fx_twiddles(int M) {
    typedef long double ld;
    std::vector<long long> c(M), s(M);   // cos, sin in Q62
    const int H = M / 2, top = M % 4 == 0 ? M / 4 : H, B = int(std::sqrt(double(top))) + 1;
    const ld step = 2.0L * 3.14159265358979323846264338327950288L / M, one = 4611686018427387904.0L;
    std::vector<ld> uc(B), us(B);
    for (int a = 0; a < B; ++a) {
        uc[a] = std::cos(step * a);
        us[a] = std::sin(step * a);
    }
    for (int b = 0; b <= top; b += B) {
        const ld vc = std::cos(step * b), vs = std::sin(step * b);
        for (int a = 0; a < B && a + b <= top; ++a) {
            c[a + b] = llroundl((uc[a] * vc - us[a] * vs) * one);
            s[a + b] = llroundl((us[a] * vc + uc[a] * vs) * one);
        }
    }
    for (int t = top + 1; t <= H; ++t) {   // reflect at pi / 2
        c[t] = -c[H - t];
        s[t] = s[H - t];
    }
    for (int t = H + 1; t < M; ++t) {      // and at pi
        c[t] = c[M - t];
        s[t] = -s[M - t];
    }
    std::vector<int> tw(4 * size_t(M));
    for (int t = 0; t < M; ++t) {
        const fx2 a = fx_split(c[t]), b = fx_split(-s[t]);
        tw[4 * t] = a.h;
        tw[4 * t + 1] = a.l;
        tw[4 * t + 2] = b.h;
        tw[4 * t + 3] = b.l;
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
    int* emax;             // [nf][N+1] largest biased exponents of gana (atomic maxima); null: not needed
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

// One stage of radix R over nsig signals from entry `from` of the shared array
// to entry `to`; step = M / (Ns R).
template <int R>
__device__ __forceinline__ void fx_stage(longlong2* sm, int from, int to, int nsig, int M, int Ns, int step,
                                         const int4* tw) {
    const int nb = M / R, ld = fx_stride(M);
    const float rns = 1.f / float(Ns);
#pragma unroll 1
    for (int u = threadIdx.x; u < nsig * nb; u += blockDim.x) {
        int t = u, o = 0;   // butterfly and its signal's offset
        while (t >= nb) {
            t -= nb;
            o += ld;
        }
        // t / Ns: exact, as t + 1/2 is at least 1 / (2 Ns) away from every multiple
        const int q = int((float(t) + 0.5f) * rns), k = t - q * Ns;
        cx<fx> v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = fx_ld(sm + from + o + fxp(t + r * nb));
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                const int4 w = tw[k * r * step];
                v[r] = fx_cmul(v[r], {w.x, w.y}, {w.z, w.w});
            }
        }
        fx_dft<R, -1>(v);
#pragma unroll
        for (int r = 0; r < R; ++r) fx_st(sm + to + o + fxp(q * Ns * R + k + r * Ns), v[r]);
    }
    __syncthreads();
}

// Forward transform of nsig signals at entry `from`, `to` the other buffer;
// returns the entry of the result.
__device__ __forceinline__ int fx_fft(longlong2* sm, int from, int to, int nsig, const FxPlan& plan, const int4* tw) {
    int Ns = 1, step = plan.n;
#pragma unroll 1
    for (int st = 0; st < plan.nst; ++st) {
        const int R = plan.radix[st];
        if (R == 8) fx_stage<8>(sm, from, to, nsig, plan.n, Ns, step /= 8, tw);
        else if (R == 4) fx_stage<4>(sm, from, to, nsig, plan.n, Ns, step /= 4, tw);
        else if (R == 2) fx_stage<2>(sm, from, to, nsig, plan.n, Ns, step /= 2, tw);
        else if (R == 9) fx_stage<9>(sm, from, to, nsig, plan.n, Ns, step /= 9, tw);
        else fx_stage<3>(sm, from, to, nsig, plan.n, Ns, step /= 3, tw);
        Ns *= R;
        const int t = from;
        from = to;
        to = t;
    }
    return from;
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

// Signals: RHS, GRID: (zeta, u_theta) of each of the CTA's two rings and
// (u_phi, u_phi) of both; PROJECT: (v_theta, v_phi) of two rings; ADJOINT, one
// ring per CTA (its shared memory): (zeta, u_theta), (u_phi, v_theta), (v_phi, 0)
// in, (X_theta, X_phi), (rho, 0) out.
template <int MODE> struct FxMode {
    static constexpr int NF = MODE == RING_ADJOINT ? 5 : (MODE == RING_PROJECT ? 2 : 3);   // input fields
    static constexpr int RPC = MODE == RING_ADJOINT ? 1 : 2;                               // rings per CTA
    static constexpr int NS = MODE == RING_PROJECT ? 2 : 3;                                // signals
    static constexpr int NV = NF * RPC;                                                    // value f of ring r: RPC f + r
};

template <int MODE>
__global__ void __launch_bounds__(576, 1) k_ring_fx(RingFxArgs a) {
    using Q = FxMode<MODE>;
    constexpr int NF = Q::NF, NS = Q::NS, RPC = Q::RPC, NV = Q::NV;
    extern __shared__ __align__(16) unsigned char smem_fx[];
    __shared__ int s_emax[NV];
    __shared__ unsigned s_sum[NV], s_or[NV], s_sum2[4];
    const int M = a.M, N = a.N, nlat = a.nlat, ld = fx_stride(M), tid = threadIdx.x, NT = blockDim.x;
    longlong2* sm = reinterpret_cast<longlong2*>(smem_fx);
    int cur = 0;   // the buffer that holds the signals: entries 0 or NS ld
    int4* tw = reinterpret_cast<int4*>(sm + 2 * NS * ld);
    const int npair = (nlat + 1) / 2, row0 = RPC * blockIdx.x, pair = row0 / 2;
    const bool two = RPC == 2 && row0 + 1 < nlat;
    if (a.early) pdl_launch();
    // the plan's constants do not depend on the predecessor
    for (int t = tid; t < M; t += NT) tw[t] = a.tw[t];
    if (tid < NV) {
        s_emax[tid] = 0;
        s_sum[tid] = 0u;
        s_or[tid] = 0u;
    }
    if (tid < 4) s_sum2[tid] = 0u;
    double fc[RPC], scale[RPC];
#pragma unroll
    for (int r = 0; r < RPC; ++r) {
        const int row = min(row0 + r, nlat - 1);
        fc[r] = MODE == RING_GRID ? 0.0 : a.two_omega * a.x[row];
        scale[r] = MODE == RING_GRID ? 0.0 : a.rw[row];
    }
    pdl_wait();
    int kf[NV];   // fixed point = value 2^kf
    unsigned bad = 0;   // GRID: fields (bits, in the order of kf) with a non-finite input
    const double nan = __longlong_as_double(0x7FF8000000000000LL);

    if constexpr (MODE != RING_PROJECT) {
        // a thread owns the order m = tid (N < M / 3 <= blockDim) of every field and ring
        const int m = tid;
        double x[NV][2];
        int em[NV];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const double* g = a.gsyn + ((size_t(f) * npair + pair) * size_t(N + 1) + m) * 4;
            if constexpr (RPC == 2) {
                double4_32a v = make_double4_32a(0.0, 0.0, 0.0, 0.0);
                if (m <= N) v = *reinterpret_cast<const double4_32a*>(g);
                x[2 * f][0] = v.x;
                x[2 * f][1] = v.y;
                x[2 * f + 1][0] = two ? v.z : 0.0;
                x[2 * f + 1][1] = two ? v.w : 0.0;
            } else {
                double2 v = make_double2(0.0, 0.0);
                if (m <= N) v = *reinterpret_cast<const double2*>(g + 2 * (row0 & 1));
                x[f][0] = v.x;
                x[f][1] = v.y;
            }
        }
        if (m == 0) {
#pragma unroll
            for (int j = 0; j < NV; ++j) x[j][1] = 0.0;   // fields are real
            x[0][0] += fc[0];                             // q = zeta + 2 Omega cos(theta)
            if constexpr (RPC == 2)
                if (two) x[1][0] += fc[1];
        }
#pragma unroll
        for (int j = 0; j < NV; ++j) em[j] = max(f64_bexp(x[j][0]), f64_bexp(x[j][1]));
        __syncthreads();   // the reduction slots are zero, the twiddles in place
        red_max<NV>(em, s_emax);
        __syncthreads();
        unsigned sum[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            em[j] = max(s_emax[j], 1);
            const unsigned v = f64_top16(x[j][0], em[j]) + f64_top16(x[j][1], em[j]);
            sum[j] = m > N ? 0u : (m == 0 ? v : 2u * v);
        }
        red_add<NV>(sum, s_sum);
        // the zero-padded middle of every signal
        for (int q = N + 1 + tid; q < M - N; q += NT)
#pragma unroll
            for (int sg = 0; sg < NS; ++sg) sm[sg * ld + fxp(q)] = make_longlong2(0, 0);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            kf[j] = 1072 - em[j] + 26 - bitlen(s_sum[j]);
            // a non-finite input: NaN for its ring, on the grid for that field of it
            if (MODE == RING_GRID) bad |= em[j] == 2047 ? 1u << j : 0u;
            else if (em[j] == 2047) scale[j % RPC] = nan;
        }
        if (m <= N) {
            long long v[NV][2];
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                v[j][0] = f64_to_fx(x[j][0], kf[j]);
                v[j][1] = f64_to_fx(x[j][1], kf[j]);
            }
            // Z = a + i b of two Hermitian spectra, Z_{M-m} = conj(a_m) + i conj(b_m);
            // stored with real and imaginary parts exchanged (inverse transform)
            auto put = [&](int sg, long long ax, long long ay, long long bx, long long by) {
                sm[sg * ld + fxp(m)] = make_longlong2(ay + bx, ax - by);
                if (m > 0) sm[sg * ld + fxp(M - m)] = make_longlong2(bx - ay, ax + by);
            };
            if constexpr (RPC == 2) {
                put(0, v[0][0], v[0][1], v[2][0], v[2][1]);
                put(1, v[1][0], v[1][1], v[3][0], v[3][1]);
                put(2, v[4][0], v[4][1], v[5][0], v[5][1]);
            } else {
                put(0, v[0][0], v[0][1], v[1][0], v[1][1]);
                put(1, v[2][0], v[2][1], v[3][0], v[3][1]);
                put(2, v[4][0], v[4][1], 0, 0);
            }
        }
    }

    // W = the fields to transform forward: component c of ring r's signal (ADJOINT: X_theta,
    // X_phi, rho) at RPC c + r
    constexpr int NW = MODE == RING_ADJOINT ? 3 : 4;
    int kw[NW];
    if constexpr (MODE == RING_PROJECT) {
        auto grid = [&](int j, int q) {
            return (j & 1) == 0 || two ? (j / 2 ? a.gin1 : a.gin0)[size_t(row0 + (j & 1)) * M + q] : 0.0;
        };
        int em[4] = {0, 0, 0, 0};
        for (int q = tid; q < M; q += NT)
#pragma unroll
            for (int j = 0; j < 4; ++j) em[j] = max(em[j], f64_bexp(grid(j, q)));
        __syncthreads();
        red_max<4>(em, s_emax);
        __syncthreads();
        unsigned sum[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int j = 0; j < 4; ++j) em[j] = max(s_emax[j], 1);
        for (int q = tid; q < M; q += NT)
#pragma unroll
            for (int j = 0; j < 4; ++j) sum[j] += f64_top16(grid(j, q), em[j]);
        red_add<4>(sum, s_sum);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            kw[j] = 1072 - em[j] + 26 - bitlen(s_sum[j]);
            if (em[j] == 2047) scale[j & 1] = nan;
        }
        for (int q = tid; q < M; q += NT)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                sm[r * ld + fxp(q)] = make_longlong2(f64_to_fx(grid(r, q), kw[r]), f64_to_fx(grid(2 + r, q), kw[2 + r]));
    }
    __syncthreads();

    // pass 0: inverse transform and product; pass 1: forward transform
#pragma unroll 1
    for (int pass = MODE == RING_PROJECT ? 1 : 0; pass < 2; ++pass) {
        cur = fx_fft(sm, cur, NS * ld - cur, pass == 0 ? NS : 2, a.plan, tw);
        if (pass == 1) break;
        const longlong2* in = sm + cur;
        if constexpr (MODE == RING_GRID) {
            for (int q = tid; q < M; q += NT) {
                const longlong2 B = in[2 * ld + fxp(q)];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (r == 1 && !two) break;
                    const longlong2 A = in[r * ld + fxp(q)];   // (u_theta, zeta)
                    const size_t o = size_t(row0 + r) * M + q;
                    auto val = [&](long long v, int j) { return bad >> j & 1 ? nan : f64_scale(__ll2double_rn(v), -kf[j]); };
                    if (a.gout0) a.gout0[o] = val(A.y, r);
                    if (a.gout1) a.gout1[o] = val(A.x, 2 + r);
                    if (a.gout2) a.gout2[o] = val(r ? B.x : B.y, 4 + r);
                }
            }
            return;
        } else if constexpr (MODE != RING_PROJECT) {
            // the grid values of point q (real and imaginary parts exchanged)
            auto fields = [&](int q, long long* v) {
                const longlong2 A = in[fxp(q)], B = in[ld + fxp(q)], C = in[2 * ld + fxp(q)];
                if constexpr (RPC == 2) {
                    v[0] = A.y; v[1] = B.y; v[2] = A.x; v[3] = B.x; v[4] = C.y; v[5] = C.x;
                } else {
                    v[0] = A.y; v[1] = A.x; v[2] = B.y; v[3] = B.x; v[4] = C.y;
                }
            };
            unsigned om[NV];
#pragma unroll
            for (int j = 0; j < NV; ++j) om[j] = 0u;
            for (int q = tid; q < M; q += NT) {
                long long v[NV];
                fields(q, v);
#pragma unroll
                for (int j = 0; j < NV; ++j) om[j] |= hi_abs(v[j]);
            }
            red_or<NV>(om, s_or);
            __syncthreads();
            int up[NV];   // left shift of a field to |v| < 2^61
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                up[j] = max(0, 29 - bitlen(s_or[j]));
                kf[j] += up[j];
            }
            int d1 = 0, d2 = 0;
            if constexpr (MODE == RING_RHS) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    kw[r] = kf[r] + kf[4 + r] - 62;        // W_theta = -q u_phi
                    kw[2 + r] = kf[r] + kf[2 + r] - 62;    // W_phi = q u_theta
                }
            } else {
                kw[0] = kf[0] + kf[4] - 62;   // X_theta = q v_phi
                kw[1] = kf[0] + kf[3] - 62;   // X_phi = -q v_theta
                // rho = -v_theta u_phi + v_phi u_theta, at the coarser scale of the two
                kw[2] = min(kf[3] + kf[2], kf[4] + kf[1]) - 62;
                d1 = kw[2] + 62 - kf[3] - kf[2];
                d2 = kw[2] + 62 - kf[4] - kf[1];
            }
            longlong2* out = sm + (NS * ld - cur);
            unsigned sum[NW];
#pragma unroll
            for (int j = 0; j < NW; ++j) sum[j] = 0u;
            for (int q = tid; q < M; q += NT) {
                long long v[NV], w[4];
                fields(q, v);
#pragma unroll
                for (int j = 0; j < NV; ++j) v[j] <<= up[j];
                if constexpr (MODE == RING_RHS) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        w[r] = -fx_mul62(v[r], v[4 + r]);
                        w[2 + r] = fx_mul62(v[r], v[2 + r]);
                    }
                    out[fxp(q)] = make_longlong2(w[0], w[2]);
                    out[ld + fxp(q)] = make_longlong2(w[1], w[3]);
                } else {
                    w[0] = fx_mul62(v[0], v[4]);
                    w[1] = -fx_mul62(v[0], v[3]);
                    w[2] = fx_shift(fx_mul62(v[4], v[1]), d2) - fx_shift(fx_mul62(v[3], v[2]), d1);
                    out[fxp(q)] = make_longlong2(w[0], w[1]);
                    out[ld + fxp(q)] = make_longlong2(w[2], 0);
                }
#pragma unroll
                for (int j = 0; j < NW; ++j) sum[j] += top16_abs(w[j]);
            }
            red_add<NW>(sum, s_sum2);
            __syncthreads();
            int sh[4] = {0, 0, 0, 0};
#pragma unroll
            for (int j = 0; j < NW; ++j) {
                sh[j] = 16 - bitlen(s_sum2[j]);
                kw[j] += sh[j];
            }
            // every thread rescales the points it wrote
            for (int q = tid; q < M; q += NT)
#pragma unroll
                for (int sg = 0; sg < 2; ++sg) {
                    const longlong2 w = out[sg * ld + fxp(q)];
                    const int jx = RPC == 2 ? sg : 2 * sg, jy = RPC == 2 ? 2 + sg : 1 + 2 * sg;
                    out[sg * ld + fxp(q)] = make_longlong2(fx_shift(w.x, sh[jx]), fx_shift(w.y, sh[jy]));
                }
            cur = NS * ld - cur;
            __syncthreads();
        }
    }

    // separate the real spectra: of Z = A + i B, A_m = (Z_m + conj Z_{M-m}) / 2,
    // B_m = (Z_m - conj Z_{M-m}) / (2 i); truncate, weight, store
    const int m = tid;
    if (m > N) return;
    const longlong2* in = sm + cur;
    const int mr = m == 0 ? 0 : M - m;
    auto cv = [&](long long v, double sc, int k) { return f64_scale(__ll2double_rn(v) * sc, -k - 1); };
    // field f of every ring, and the column scales of the analysis
    auto store = [&](int f, const double4_32a& o) {
        double* g = a.gana + ((size_t(f) * npair + pair) * size_t(N + 1) + m) * 4;
        int e = max(f64_bexp(o.x), f64_bexp(o.y));
        if constexpr (RPC == 2) {
            *reinterpret_cast<double4_32a*>(g) = o;
            e = max(e, max(f64_bexp(o.z), f64_bexp(o.w)));
        } else {
            *reinterpret_cast<double2*>(g + 2 * (row0 & 1)) = make_double2(o.x, o.y);
        }
        if (a.emax) atomicMax(a.emax + f * (N + 1) + m, e);
    };
    double4_32a o0 = make_double4_32a(0.0, 0.0, 0.0, 0.0), o1 = o0;
#pragma unroll
    for (int r = 0; r < RPC; ++r) {
        if (r == 1 && !two) break;
        const longlong2 p = in[r * ld + fxp(m)], z = in[r * ld + fxp(mr)];
        const double tx = cv(p.x + z.x, scale[r], kw[r]), ty = cv(p.y - z.y, scale[r], kw[r]);
        const double fx_ = cv(p.y + z.y, scale[r], kw[RPC + r]), fy = cv(z.x - p.x, scale[r], kw[RPC + r]);
        if (r == 0) {
            o0.x = tx; o0.y = ty; o1.x = fx_; o1.y = fy;
        } else {
            o0.z = tx; o0.w = ty; o1.z = fx_; o1.w = fy;
        }
    }
    store(0, o0);
    store(1, o1);
    if constexpr (MODE == RING_ADJOINT) {
        // rho: plain quadrature weight (2 pi / M) w_p
        const longlong2 p = in[ld + fxp(m)], z = in[ld + fxp(mr)];
        const double sc = scale[0] * a.s[row0];
        o0.x = cv(p.x + z.x, sc, kw[2]);
        o0.y = cv(p.y - z.y, sc, kw[2]);
        store(2, o0);
    }
}

template <int MODE>
static cudaError_t ring_fx_t(sphnse_plan* P, RingFxArgs a) {
    using Q = FxMode<MODE>;
    // a radix-8 butterfly per thread; a grid of at most one CTA per SM, whose time
    // is one thread's chain, takes a radix-3 butterfly and a grid point per thread
    // (RHS at L = 100, 81 CTAs: 56 -> 46 us; at L = 255, 192 CTAs, 86 -> 92 us);
    // every order m <= N < M / 3 needs its own thread
    const int grid = (a.nlat + Q::RPC - 1) / Q::RPC;
    const int want = grid <= P->nsm ? std::min(Q::NS * a.M / 3, 576) : Q::NS * a.M / 8;
    const int threads = (std::max(want, a.N + 1) + 31) / 32 * 32;
    const size_t sm = size_t(2) * Q::NS * fx_stride(a.M) * 16 + size_t(a.M) * 16;
    allow_dynamic_smem(reinterpret_cast<const void*>(k_ring_fx<MODE>), sm);
    // a grid of more than one wave must not start its successor early
    a.early = grid <= P->nsm * std::max(1, std::min(int((227 * 1024) / (sm + 1024)), 576 / threads));
    return launch_pdl(k_ring_fx<MODE>, dim3(grid), dim3(threads), sm, P->stream, a);
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
        case RING_RHS: e = ring_fx_t<RING_RHS>(P, a); break;
        case RING_GRID: e = ring_fx_t<RING_GRID>(P, a); break;
        case RING_PROJECT: e = ring_fx_t<RING_PROJECT>(P, a); break;
        default: e = ring_fx_t<RING_ADJOINT>(P, a); break;
    }
    stage_end(P, SPHNSE_STAGE_RING);
    return check_cuda(e);
}

}  // namespace sph
