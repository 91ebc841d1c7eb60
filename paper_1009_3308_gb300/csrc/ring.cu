// Longitude ("ring") kernels of the FP32 and BF16x3 paths (the FP64 path's
// kernel is in ring_fx.cu).  General kernel: one CTA per pair of Gauss
// latitudes.  It reads the latitude-pair-major
// spectra [f][row / 2][m][row % 2] (a CTA's data are contiguous) and writes the
// order-major ones of the analysis (16 bytes, two latitudes, at a time), so it
// needs no transposes.  With one latitude per CTA and a transpose kernel on
// either side the adjoint's ring took 22.5 + 13.5 us at L = 255 (event pairs).
//
// RHS mode (Sec. 4.2: the phi sums of Eqs. (app_soln_rep), (eval_nonlin1)
// are Fourier sums, evaluated by FFT):
//   1. inverse FFT of the Hermitian spectra g_m, |m| <= N (zero-padded to M):
//      z1 = zeta + i u_theta, z2 = u_phi              (two complex M-point FFTs)
//   2. pointwise product (Eqs. (short_nonlin1), (C)):
//      q = zeta + 2 Omega cos(theta_p),  W_theta = -q u_phi,  W_phi = q u_theta
//   3. forward FFT of W_theta + i W_phi, separation of the two real spectra,
//      truncation to m = 0..N, scaling by (2 pi / M) w_p / sin(theta_p)
//      (the quadrature weight of Eq. (quadrule) and the 1/sin of the basis).
// M = nlon = 2^a 3^b; Stockham autosort radix-8/4/2/3 stages (radix 3 last)
// from one shared-memory buffer to the other, a butterfly of one signal per
// thread at a time, one barrier per stage; twiddles e^{-2 pi i t / M} computed
// in FP64 on the host, staged in shared memory.  (In-place stages holding every
// signal's butterflies in registers spilled 276 bytes per thread and left half
// of the threads idle: the adjoint's ring took 24.1 us at L = 255, now 14.3.)
// Products keep |m| <= 2N and M >= 3N + 2 > 3N, so the truncated m <= N
// coefficients are alias-free.
//
// Other modes reuse the same machinery: GRID writes zeta, u_theta, u_phi to
// grid rows; PROJECT transforms given grid rows of a tangential field;
// ADJOINT evaluates the transposed linearised product (see rhs_adjoint).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "fft_small.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "ring4.cuh"

namespace sph {

// entry i of a signal: one slot of padding per sixteen keeps the stride-8
// writes of the first radix-8 stage out of one another's banks
__device__ __forceinline__ int rpad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int ring_stride(int M) { return M + ((M + 15) >> 4); }

// One stage of radix R over the 2 ns signals (ns per ring, rings rs apart),
// from -> to; Ns = product of the earlier radices, step = M / (Ns R).  FIRST:
// Ns = 1, every twiddle is 1.
template <int R, int SIGN, bool FIRST = false>
__device__ __forceinline__ void stage(cx<float>* sm, int from, int to, int ns, int rs, int M, int Ns, int step,
                                      const float* tw) {
    const int nb = M / R, ld = ring_stride(M);
    const float rns = 1.f / float(Ns);
#pragma unroll 1
    for (int u = threadIdx.x; u < 2 * ns * nb; u += blockDim.x) {
        int j = u, sg = 0;
        while (j >= nb) {
            j -= nb;
            ++sg;
        }
        const int o = sg < ns ? sg * ld : rs + (sg - ns) * ld;
        // j / Ns: exact, as j + 1/2 is at least 1 / (2 Ns) away from every multiple
        const int q = int((float(j) + 0.5f) * rns), k = j - q * Ns;
        cx<float> v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = sm[from + o + rpad(j + r * nb)];
        if constexpr (!FIRST) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                // which product of a sum is rounded is spelled out, or the compiler picks
                // it anew for each instance of this loop and results differ between them
                const cx<float> a = v[r], w = twiddle<float>(tw, k * r * step, SIGN);
                v[r] = {fmaf(a.x, w.x, -__fmul_rn(a.y, w.y)),
                        R == 2 && SIGN < 0 ? fmaf(a.x, w.y, __fmul_rn(a.y, w.x)) : fmaf(a.y, w.x, __fmul_rn(a.x, w.y))};
            }
        }
        dft<float, R>(v, SIGN);
#pragma unroll
        for (int r = 0; r < R; ++r) sm[to + o + rpad(q * Ns * R + k + r * Ns)] = v[r];
    }
    __syncthreads();
}

// Full M-point transforms (SIGN -1 forward, +1 inverse) of the signals at entry
// `from` of the shared array, `to` the other buffer; returns the result's entry.
template <int SIGN>
__device__ __forceinline__ int fft(cx<float>* sm, int from, int to, int ns, int rs, const FFTPlan& plan, const float* tw) {
    int Ns = 1, step = plan.n;
#pragma unroll 1
    for (int st = 0; st < plan.nstages; ++st) {
        const int R = plan.radix[st];
        if (R == 8 && st == 0) stage<8, SIGN, true>(sm, from, to, ns, rs, plan.n, 1, step /= 8, tw);
        else if (R == 8) stage<8, SIGN>(sm, from, to, ns, rs, plan.n, Ns, step /= 8, tw);
        else if (R == 4) stage<4, SIGN>(sm, from, to, ns, rs, plan.n, Ns, step /= 4, tw);
        else if (R == 2) stage<2, SIGN>(sm, from, to, ns, rs, plan.n, Ns, step /= 2, tw);
        else stage<3, SIGN>(sm, from, to, ns, rs, plan.n, Ns, step /= 3, tw);
        Ns *= R;
        const int t = from;
        from = to;
        to = t;
    }
    return from;
}

struct RingArgs {
    int N, M, nlat;
    double two_omega;
    const double* x;       // cos(theta)
    const double* s;       // sin(theta)
    const double* rw;      // (2 pi / M) w_p / sin(theta_p)
    const void* gsyn;      // [nf][pair][N+1][2] complex float
    void* gana;            // [nf][N+1][nlat] complex float
    const double* gin0;    // grid input rows (PROJECT)
    const double* gin1;
    double* gout0;         // grid output rows (GRID)
    double* gout1;
    double* gout2;
    size_t sgs, sga;       // per-instance strides (complex entries) along gridDim.y
    int early;             // a grid of one wave: the successor may start its prologue at once
};

template <int MODE>
__global__ void __launch_bounds__(512) k_ring(RingArgs a, const __grid_constant__ FFTPlan plan,
                                              const float* __restrict__ tw) {
    if (a.early) pdl_launch();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NBUF = MODE == RING_ADJOINT ? 3 : (MODE == RING_PROJECT ? 1 : 2);
    const int M = a.M, N = a.N, nlat = a.nlat, pair = blockIdx.x, npair = (nlat + 1) / 2, row0 = 2 * pair;
    const int ls = ring_stride(M), rs = NBUF * ls;     // signal and ring strides
    cx<float>* sm = reinterpret_cast<cx<float>*>(smem_raw);    // [2 rings][NBUF][ls], twice
    int cur = 0;                                       // the buffer that holds the signals: entry 0 or 2 rs
    // the twiddle table e^{-2 pi i t / M} lives in shared memory after the buffers
    float* tws = reinterpret_cast<float*>(sm + 4 * rs);
    for (int t = threadIdx.x; t < 2 * M; t += blockDim.x) tws[t] = tw[t];
    const bool two = row0 + 1 < nlat;                  // an odd grid's last pair has one ring
    const size_t ld = size_t(N + 1);
    const cx<float>* gs = reinterpret_cast<const cx<float>*>(a.gsyn) + size_t(blockIdx.y) * a.sgs;
    cx<float>* ga = reinterpret_cast<cx<float>*>(a.gana) + size_t(blockIdx.y) * a.sga;
    pdl_wait();

    if constexpr (MODE != RING_PROJECT) {
        // Hermitian spectra of two real fields packed as a + i b:
        //   Z_m = g^a_m + i g^b_m (m <= N);  Z_{M-m} = conj(g^a_m) + i conj(g^b_m)
        const int nsig = MODE == RING_ADJOINT ? 3 : 2;
        for (int m = threadIdx.x; m < M - N; m += blockDim.x) {
            for (int sgi = 0; sgi < nsig; ++sgi) {
                // fields packed per signal: RHS/GRID (0,1),(2,-); ADJOINT (0,1),(2,3),(4,-)
                const int fa = 2 * sgi, fb = 2 * sgi + 1;
                const bool has_b = (MODE == RING_ADJOINT) ? fb <= 4 : fb <= 2;
                // order m of both rings
                cx<float> A[2] = {{0.f, 0.f}, {0.f, 0.f}}, Bv[2] = {{0.f, 0.f}, {0.f, 0.f}};
                if (m <= N) {
                    const cx<float>* g = gs + ((size_t(fa) * npair + pair) * ld + m) * 2;
                    const float4 u = *reinterpret_cast<const float4*>(g);
                    A[0] = {u.x, u.y};
                    if (two) A[1] = {u.z, u.w};
                    if (has_b) {
                        const float4 w = *reinterpret_cast<const float4*>(g + size_t(npair) * ld * 2);
                        Bv[0] = {w.x, w.y};
                        if (two) Bv[1] = {w.z, w.w};
                    }
                }
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    cx<float> ga_ = A[r], gb_ = Bv[r];
                    if (m == 0) { ga_.y = 0.f; gb_.y = 0.f; }
                    cx<float>* z = sm + r * rs + sgi * ls;
                    z[rpad(m)] = {ga_.x - gb_.y, ga_.y + gb_.x};
                    if (m > 0 && m <= N) z[rpad(M - m)] = {ga_.x + gb_.y, gb_.x - ga_.y};
                }
            }
        }
        __syncthreads();
        cur = fft<+1>(sm, cur, 2 * rs - cur, nsig, rs, plan, tws);
    }

    // point q of ring r, both rings over the CTA's threads
    auto points = [&](auto&& f) {
        for (int u = threadIdx.x; u < 2 * M; u += blockDim.x) {
            const int r = u >= M, q = u - r * M;
            f(r, q, sm + cur + r * rs + rpad(q));
        }
    };
    if constexpr (MODE == RING_GRID) {
        points([&](int r, int q, const cx<float>* z) {
            if (r && !two) return;
            const size_t o = size_t(row0 + r) * M + q;
            if (a.gout0) a.gout0[o] = double(z[0].x);
            if (a.gout1) a.gout1[o] = double(z[0].y);
            if (a.gout2) a.gout2[o] = double(z[ls].x);
        });
        return;
    }

    constexpr int nout = MODE == RING_ADJOINT ? 2 : 1;
    const float fc0 = float(a.two_omega * a.x[row0]), fc1 = float(a.two_omega * a.x[min(row0 + 1, nlat - 1)]);
    if constexpr (MODE == RING_RHS) {
        points([&](int r, int q, cx<float>* z) {
            const float zeta = z[0].x, uth = z[0].y, uph = z[ls].x;
            const float qq = zeta + (r ? fc1 : fc0);
            z[0] = {-qq * uph, qq * uth};
        });
    } else if constexpr (MODE == RING_PROJECT) {
        points([&](int r, int q, cx<float>* z) {
            const size_t o = size_t(row0 + r) * M + q;
            z[0] = r && !two ? cx<float>{0.f, 0.f} : cx<float>{float(a.gin0[o]), float(a.gin1[o])};
        });
    } else {  // RING_ADJOINT: fields zeta, u_th, u_ph, v_th, v_ph
        points([&](int r, int q, cx<float>* z) {
            const float zeta = z[0].x, uth = z[0].y;
            const float uph = z[ls].x, vth = z[ls].y, vph = z[2 * ls].x;
            const float qq = zeta + (r ? fc1 : fc0);
            // X = -q xhat x v = (q v_phi, -q v_theta); rho = v . (xhat x u) = -v_th u_ph + v_ph u_th
            z[0] = {qq * vph, -qq * vth};
            z[ls] = {-vth * uph + vph * uth, 0.f};
        });
    }
    __syncthreads();
    cur = fft<-1>(sm, cur, 2 * rs - cur, nout, rs, plan, tws);

    // both rings of order m at once: two latitudes are 16 bytes of the order-major output
    float scale[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) scale[r] = float(a.rw[min(row0 + r, nlat - 1)]);
    auto put = [&](int f, int m, const cx<float> (&v)[2]) {
        cx<float>* d = ga + (size_t(f) * ld + m) * nlat + row0;
        if (nlat % 2 == 0) {
            *reinterpret_cast<float4*>(d) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        } else {   // rows of an odd grid are 8-byte aligned
            d[0] = v[0];
            if (two) d[1] = v[1];
        }
    };
    for (int m = threadIdx.x; m <= N; m += blockDim.x) {
        cx<float> oA[2], oB[2], oC[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const cx<float>* Z = sm + cur + r * rs;
            const cx<float> p = Z[rpad(m)];
            const cx<float> q = Z[rpad(m == 0 ? 0 : M - m)];
            // W = A + i B with A, B real fields: A_m = (Z_m + conj Z_{M-m}) / 2,
            // B_m = (Z_m - conj Z_{M-m}) / (2 i)
            cx<float> A{0.5f * (p.x + q.x), 0.5f * (p.y - q.y)};
            cx<float> Bv{0.5f * (p.y + q.y), 0.5f * (q.x - p.x)};
            oA[r] = {A.x * scale[r], A.y * scale[r]};
            oB[r] = {Bv.x * scale[r], Bv.y * scale[r]};
            if constexpr (nout == 2) {
                // scalar field rho: plain quadrature weight (2 pi / M) w_p
                const float sc2 = scale[r] * float(a.s[min(row0 + r, nlat - 1)]);
                const cx<float> z = Z[ls + rpad(m)];
                oC[r] = {z.x * sc2, z.y * sc2};
            }
        }
        put(0, m, oA);
        put(1, m, oB);
        if constexpr (nout == 2) put(2, m, oC);
    }
}

template <int MODE>
static void ring_t(sphnse_plan* P, RingArgs a, const float* tw, int nb = 1) {
    const int nbuf = MODE == RING_ADJOINT ? 3 : (MODE == RING_PROJECT ? 1 : 2);
    // Two threads per butterfly of the average stage: half of them idle in the
    // stages, all of them load and store.  One thread per radix-8 butterfly was
    // right for radix-8 plans only: the projection at L = 153 on 486 = 2 3^5
    // longitudes took 32.1 us, with this rule 16.7, at 324 FP32 F 28.6, now 20.8.
    int nb_sum = 0;
    for (int i = 0; i < P->fft.nstages; ++i) nb_sum += P->nlon / P->fft.radix[i];
    const int threads = std::min(512, std::max(64, (4 * nbuf * nb_sum / P->fft.nstages + 31) / 32 * 32));
    const size_t sm = size_t(4 * nbuf) * ring_stride(P->nlon) * sizeof(cx<float>) + size_t(P->nlon) * 2 * sizeof(float);
    allow_dynamic_smem(reinterpret_cast<const void*>(k_ring<MODE>), sm);
    a.early = long(P->nlat + 1) / 2 * nb <= long(P->nsm) * std::min<long>(512 / threads, (227 << 10) / long(sm + 1024));
    launch_pdl(k_ring<MODE>, dim3((P->nlat + 1) / 2, nb), dim3(threads), sm, P->stream, a, P->fft, tw);
}

// FP32 RHS ring pass over nb instances (latitude-pair-major in, order-major out, with strides)
int launch_ring_batch(sphnse_plan* P, int nb, const float* gsyn, size_t sgs, float* gana, size_t sga) {
    RingArgs a{};
    a.N = P->N;
    a.M = P->nlon;
    a.nlat = P->nlat;
    a.two_omega = 2.0 * P->Omega;
    a.x = P->d_x;
    a.s = P->d_s;
    a.rw = P->d_rw;
    a.gsyn = gsyn;
    a.gana = gana;
    a.sgs = sgs / 2;
    a.sga = sga / 2;
    stage_begin(P, SPHNSE_STAGE_RING);
    ring_t<RING_RHS>(P, a, P->d_tw32, nb);
    stage_end(P, SPHNSE_STAGE_RING);
    return check_cuda(cudaGetLastError());
}

static void ring_mode(sphnse_plan* P, int mode, const RingArgs& a, const float* tw) {
    switch (mode) {
        case RING_RHS: ring_t<RING_RHS>(P, a, tw); break;
        case RING_GRID: ring_t<RING_GRID>(P, a, tw); break;
        case RING_PROJECT: ring_t<RING_PROJECT>(P, a, tw); break;
        default: ring_t<RING_ADJOINT>(P, a, tw); break;
    }
}

int launch_ring(sphnse_plan* P, int mode, const double* gin0, const double* gin1,
                double* gout0, double* gout1, double* gout2) {
    RingArgs a;
    a.N = P->N;
    a.M = P->nlon;
    a.nlat = P->nlat;
    a.two_omega = mode == RING_RHS && P->coriolis_split ? 0.0 : 2.0 * P->Omega;
    a.x = P->d_x;
    a.s = P->d_s;
    a.rw = P->d_rw;
    a.gsyn = P->d_gsyn;
    a.gana = P->d_gana;
    a.gin0 = gin0;
    a.gin1 = gin1;
    a.gout0 = gout0;
    a.gout1 = gout1;
    a.gout2 = gout2;
    a.sgs = a.sga = 0;
    stage_begin(P, SPHNSE_STAGE_RING);
    ring_mode(P, mode, a, P->d_tw32);
    stage_end(P, SPHNSE_STAGE_RING);
    return check_cuda(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Four-step ring kernel (the transform itself is in ring4.cuh)

template <int M2>
__global__ void __launch_bounds__(128, 4) k_ring4(Ring4Args a) {
    extern __shared__ __align__(16) float2 sm4[];
    __shared__ float s_rw[128 / M2];
    pdl_launch();
    pdl_wait();
    ring4_rings<M2>(a, blockIdx.x * (128 / M2), blockIdx.y, threadIdx.x, sm4, s_rw);
}

// 256 threads per G = 128 / M2 rings (grids of less than a wave)
template <int M2>
__global__ void __launch_bounds__(256, 3) k_ring4w(Ring4Args a) {
    extern __shared__ __align__(16) float2 sm4[];
    __shared__ float s_rw[128 / M2];
    pdl_launch();
    pdl_wait();
    ring4w_rings<M2>(a, blockIdx.x * (128 / M2), blockIdx.y, threadIdx.x, sm4, s_rw);
}

template <int M2>
static int ring4_t(sphnse_plan* P, int nb, const float* gsyn, size_t sgs, float* gana, size_t sga, int pairs) {
    constexpr size_t sm = ring4_smem<M2>();
    static_assert(sm <= 227 * 1024, "ring4 shared memory");
    allow_dynamic_smem(reinterpret_cast<const void*>(k_ring4<M2>), sm);
    Ring4Args a;
    a.N = P->N;
    a.nlat = P->nlat;
    a.two_omega = P->coriolis_split ? 0.f : float(2.0 * P->Omega);
    a.x = P->d_x;
    a.rw = P->d_rw;
    a.gsyn = reinterpret_cast<const float2*>(gsyn);
    a.gana = reinterpret_cast<float2*>(gana);
    a.ftw = reinterpret_cast<const float2*>(P->d_ftw);
    a.sgs = sgs / 2;
    a.sga = sga / 2;
    a.pairs = pairs;
    constexpr int G = 128 / M2;
    const dim3 grid((P->nlat + G - 1) / G, nb);
    if constexpr (M2 >= 16) {
        // a grid of less than four CTAs per SM is latency-bound: twice the
        // threads per ring shorten each thread's chain of passes
        const bool wide = P->ring_threads == 256 ||
                          (P->ring_threads == 0 && size_t(grid.x) * grid.y <= size_t(4) * P->nsm);
        if (wide) {
            allow_dynamic_smem(reinterpret_cast<const void*>(k_ring4w<M2>), sm);
            return check_cuda(launch_pdl(k_ring4w<M2>, grid, dim3(256), sm, P->stream, a));
        }
    }
    return check_cuda(launch_pdl(k_ring4<M2>, grid, dim3(128), sm, P->stream, a));
}

int ring4_m2(int nlon, int nlat) {
    if (nlon % 24 || nlat % 2) return 0;
    const int M2 = nlon / 24;
    return (M2 == 4 || M2 == 8 || M2 == 16 || M2 == 32 || M2 == 64) ? M2 : 0;
}

bool ring4_ok(const sphnse_plan* P) { return ring4_m2(P->nlon, P->nlat) != 0 && P->d_ftw != nullptr; }

// twiddle tables of the four-step kernel (FP64 -> FP32), in its padded layout
std::vector<float> ring4_twiddles(int nlon) {
    const int M2 = ring4_m2(nlon, 2);
    if (!M2) return {};
    int A = 0, P1 = 0;
    switch (M2) {
        case 64: A = R4<64>::A; P1 = R4<64>::P1; break;
        case 32: A = R4<32>::A; P1 = R4<32>::P1; break;
        case 16: A = R4<16>::A; P1 = R4<16>::P1; break;
        case 8: A = R4<8>::A; P1 = R4<8>::P1; break;
        default: A = R4<4>::A; P1 = R4<4>::P1; break;
    }
    const int B = M2 / A, B2 = B + 1;
    std::vector<float> tw(2 * (size_t(24) * P1 + size_t(A) * B2), 0.f);
    for (int k1 = 0; k1 < 24; ++k1)
        for (int t = 0; t < M2; ++t) {
            const double ang = 2.0 * M_PI * double((long(t) * k1) % nlon) / double(nlon);
            tw[2 * (k1 * P1 + t)] = float(std::cos(ang));
            tw[2 * (k1 * P1 + t) + 1] = float(std::sin(ang));
        }
    float* t2 = tw.data() + 2 * 24 * P1;
    for (int c = 0; c < A; ++c)
        for (int bb = 0; bb < B; ++bb) {
            const double ang = 2.0 * M_PI * double((bb * c) % M2) / double(M2);
            t2[2 * (c * B2 + bb)] = float(std::cos(ang));
            t2[2 * (c * B2 + bb) + 1] = float(std::sin(ang));
        }
    return tw;
}

// FP32 RHS ring pass over nb instances, order-major buffers
int launch_ring4(sphnse_plan* P, int nb, const float* gsyn, size_t sgs, float* gana, size_t sga, int pairs) {
    stage_begin(P, SPHNSE_STAGE_RING);
    int rc;
    switch (ring4_m2(P->nlon, P->nlat)) {
        case 64: rc = ring4_t<64>(P, nb, gsyn, sgs, gana, sga, pairs); break;
        case 32: rc = ring4_t<32>(P, nb, gsyn, sgs, gana, sga, pairs); break;
        case 16: rc = ring4_t<16>(P, nb, gsyn, sgs, gana, sga, pairs); break;
        case 8: rc = ring4_t<8>(P, nb, gsyn, sgs, gana, sga, pairs); break;
        case 4: rc = ring4_t<4>(P, nb, gsyn, sgs, gana, sga, pairs); break;
        default: rc = SPHNSE_E_UNSUPPORTED;
    }
    stage_end(P, SPHNSE_STAGE_RING);
    return rc;
}

}  // namespace sph
