// FP32 Legendre synthesis and analysis of one instance on CUDA cores (the
// batched ensemble streams are in legendre_stream.cu).
//
// The table is read once, straight into registers: a block owns one order and
// 64 northern latitudes (synthesis: two warps for the even, two for the odd
// degrees) or 32 rows of one (order, parity) (analysis: four rows per warp),
// so that even at L = 255 every SM holds 20 to 30 warps with 16 (12) loads in
// flight each.  The persistent one-CTA-per-SM streams before it gave a whole
// order to one CTA: at L = 255 two orders per CTA, their start and tail and
// the imbalance between them took 4/5 of the time.  The synthesis builds its
// coefficient sets from alpha itself (three blocks per order repeat that at
// L = 255), which saves the prep launch.
//
// Every sum runs in the order of the streaming kernels (synthesis: degrees in
// sequence; analysis: four consecutive latitudes per lane, then across the
// warp), so results are bit for bit theirs.
#include <cuda_runtime.h>

#include <algorithm>

#include "f64cvt.h"
#include "internal.h"
#include "ptx.cuh"

namespace sph {

__device__ __forceinline__ float ld_tab(const float* p, uint64_t pol) {
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ float4 ld_tab4(const float* p, uint64_t pol) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}

struct F32Args {
    const float* table;    // [n_ext][nh]
    const double2* alpha;
    const double2* beta;   // adjoint: fields 3, 4 (scaled by 1 / s_m)
    const float4* prepc;
    const float* isin;     // 1 / sin(theta_p)
    float* gsyn;           // [NF] spectra, layout gsyn_index(pairs, ...)
    const float* gana;     // [NF][N+1][nlat] complex
    float* hana;           // [n_ext][2 NF]
    int N, nh, nlat, pairs, evict_first;
    int rb;                // analysis: groups of 32 rows per block
    // a grid of about one wave (eight synthesis blocks of 128 threads and 64
    // registers an SM, three analysis blocks of 256 and 80): the successor may start
    // its prologue at once.  From larger grids its CTAs take the slots of later
    // blocks: F 22.6 us against 18.9 at L = 170, 34.4 against 28.8 at L = 255; never
    // early is as fast from L = 100 on, below that calls are bound by the host.
    int early;
};

constexpr int F32_U = 16;   // table rows in flight per thread

// NF = 3: the fields of alpha; 5: and the two of beta; 2: those of beta alone
template <int NF>
__global__ void __launch_bounds__(128) k_syn32(F32Args a) {
    constexpr int NA = NF == 2 ? 0 : 3, C = 2 * NF, LD = (C + 3) / 4 * 4;   // coefficient rows padded to 16 bytes
    extern __shared__ __align__(16) float sm32[];
    const int N = a.N, nh = a.nh, nlat = a.nlat, m = blockIdx.y, tid = threadIdx.x;
    const int ne = ext_even(N, m), no = ext_odd(N, m), cnt = ne + no, e0 = ext_off(N, m);
    float* B = sm32;
    float* red = B + size_t(cnt) * LD;                // [2][64][C]
    const int par = tid >> 6, pl = tid & 63, p = blockIdx.x * 64 + pl, pc = min(p, nh - 1);
    const uint64_t pol = a.evict_first ? policy_evict_first() : policy_evict_last();
    const int n = par ? no : ne;
    const float* src = a.table + size_t(e0 + (par ? ne : 0)) * nh + pc;
    if (a.early) pdl_launch();
    // the table does not depend on the predecessor
    float pv[F32_U];
#pragma unroll
    for (int u = 0; u < F32_U; ++u) pv[u] = u < n ? ld_tab(src + size_t(u) * nh, pol) : 0.f;
    const float inv_s = a.isin[pc];
    pdl_wait();
    {
        const int lo = m > 0 ? m : 1, pk = packed_off(N, m) - lo;
        const float sc = m == 0 ? 1.f : 0.5f;
        for (int i = tid; i < cnt; i += 128) {
            const int K = i < ne ? m + 2 * i : m + 1 + 2 * (i - ne);
            const float4 c = a.prepc[e0 + i];
            float* out = B + size_t(i) * LD;
            auto ld = [&](const double2* v, int Kp, float scale) -> float2 {
                if (Kp < lo || Kp > N) return make_float2(0.f, 0.f);
                const double2 x = v[pk + Kp];
                return make_float2(f64_to_f32_rn(x.x) * scale, f64_to_f32_rn(x.y) * scale);
            };
            if constexpr (NA == 3) {
                const float2 a0 = ld(a.alpha, K, 1.f), am = ld(a.alpha, K - 1, 1.f), ap = ld(a.alpha, K + 1, 1.f);
                out[0] = c.x * a0.x;
                out[1] = c.x * a0.y;
                out[2] = c.y * a0.x;
                out[3] = c.y * a0.y;
                out[4] = fmaf(c.z, am.x, c.w * ap.x);
                out[5] = fmaf(c.z, am.y, c.w * ap.y);
            }
            if constexpr (NF != 3) {
                const float2 b0 = ld(a.beta, K, sc), bm = ld(a.beta, K - 1, sc), bp = ld(a.beta, K + 1, sc);
                out[2 * NA] = c.y * b0.x;
                out[2 * NA + 1] = c.y * b0.y;
                out[2 * NA + 2] = fmaf(c.z, bm.x, c.w * bp.x);
                out[2 * NA + 3] = fmaf(c.z, bm.y, c.w * bp.y);
            }
        }
    }
    __syncthreads();
    float acc[C];
#pragma unroll
    for (int f = 0; f < C; ++f) acc[f] = 0.f;
    const float* bb = B + size_t(par ? ne : 0) * LD;
    for (int j = 0; j < n; j += F32_U) {
        float nx[F32_U];
#pragma unroll
        for (int u = 0; u < F32_U; ++u) {
            const int r = j + F32_U + u;
            nx[u] = r < n ? ld_tab(src + size_t(r) * nh, pol) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < F32_U; ++u) {
            if (j + u >= n) break;
            const float4* b4 = reinterpret_cast<const float4*>(bb + size_t(j + u) * LD);
            float b[LD];
#pragma unroll
            for (int q = 0; q < LD / 4; ++q) reinterpret_cast<float4*>(b)[q] = b4[q];
#pragma unroll
            for (int f = 0; f < C; ++f) acc[f] = fmaf(pv[u], b[f], acc[f]);
        }
#pragma unroll
        for (int u = 0; u < F32_U; ++u) pv[u] = nx[u];
    }
    // even and odd sums meet: the even warps write north = E + O, the odd ones south = E - O
    float* mine = red + (par * 64 + pl) * C;
    const float* other = red + ((1 - par) * 64 + pl) * C;
#pragma unroll
    for (int f = 0; f < C; ++f) mine[f] = acc[f];
    __syncthreads();
    const int row = par ? nlat - 1 - p : p;
    if (p >= nh || (par && row == p)) return;
    const float mm = float(m);
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        const float gr = par ? other[2 * q] - acc[2 * q] : acc[2 * q] + other[2 * q];
        const float gi = par ? other[2 * q + 1] - acc[2 * q + 1] : acc[2 * q + 1] + other[2 * q + 1];
        const int f = q + 3 - NA;
        float2 o;
        if (f == 0) o = make_float2(gr, gi);
        else if (f == 1 || f == 3) o = make_float2(-mm * gi * inv_s, mm * gr * inv_s);   // (i m / sin) g
        else o = make_float2(-gr * inv_s, -gi * inv_s);                                  // -(1 / sin) g
        *reinterpret_cast<float2*>(a.gsyn + gsyn_index(a.pairs, f, m, row, N, nlat) * 2) = o;
    }
}

// Transpose-reduction of NV per-lane partial sums across a warp: afterwards
// lane l holds the total of index (NV == 32 ? l : l >> 1).
template <int NV>
__device__ __forceinline__ float warp_transpose_sum(float* v) {
    const int lane = threadIdx.x & 31;
    int n = NV;
#pragma unroll
    for (int mask = 16; mask >= 1; mask >>= 1) {
        if (n == 1) {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], mask);
            continue;
        }
        const int half = n / 2;
        const bool b = (lane & mask) != 0;
#pragma unroll
        for (int i = 0; i < NV / 2; ++i) {
            if (i < half) {
                const float keep = b ? v[half + i] : v[i];
                const float send = b ? v[i] : v[half + i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
            }
        }
        n = half;
    }
    return v[0];
}

// block (row chunk, order, parity), four rows per warp; NP = ceil(nh / 128):
// latitude steps of a lane.  A chunk is 32 rows, for the adjoint's three fields
// on the largest grids 32 a.rb: there a block would spend as long on its profile
// S as on 32 rows (L = 511 adjoint 235 us with 32 rows, 223 with 96).  Looping in
// every shape, or holding the next rows in registers, cost resident blocks and
// time (FP32 RHS 77 against 73 us at L = 340).
template <int NF, int NP>
__global__ void __launch_bounds__(256) k_ana32(F32Args a) {
    constexpr int C = 2 * NF;
    constexpr int NV = 4 * C <= 16 ? 16 : 32, FS = NV / 4;
    extern __shared__ __align__(16) float sm32[];     // S[C][nh]
    const int N = a.N, nh = a.nh, nlat = a.nlat, m = blockIdx.y, par = blockIdx.z;
    const int ne = ext_even(N, m), n = par ? ext_odd(N, m) : ne;
    if (a.early) pdl_launch();
    constexpr bool MULTI = NF == 3 && NP == 3;
    const int rb = MULTI ? a.rb : 1, jb = blockIdx.x * 32 * rb, je = min(n, jb + 32 * rb);
    if (jb >= n) return;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const int base = ext_off(N, m) + (par ? ne : 0);
    int j = jb + warp * 4;
    const uint64_t pol = a.evict_first ? policy_evict_first() : policy_evict_last();
    auto request = [&](int jr, float4 (&v)[NP][4]) {
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int p = 4 * lane + 128 * i;
                v[i][r] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (jr + r < je && p < nh) v[i][r] = ld_tab4(a.table + size_t(base + jr + r) * nh + p, pol);
            }
    };
    // the table does not depend on the predecessor
    float4 pv[NP][4];
    request(j, pv);
    pdl_wait();
    for (int i = threadIdx.x; i < nh * NF; i += 256) {
        const int f = i / nh, p = i % nh, pr = nlat - 1 - p;
        const float2 x = *reinterpret_cast<const float2*>(a.gana + gsyn_index(0, f, m, p, N, nlat) * 2);
        float2 y = make_float2(0.f, 0.f);
        if (pr != p) y = *reinterpret_cast<const float2*>(a.gana + gsyn_index(0, f, m, pr, N, nlat) * 2);
        sm32[size_t(2 * f) * nh + p] = par ? x.x - y.x : x.x + y.x;
        sm32[size_t(2 * f + 1) * nh + p] = par ? x.y - y.y : x.y + y.y;
    }
    __syncthreads();
    for (; j < je; j += 32) {
        float acc[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] = 0.f;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int p = 4 * lane + 128 * i;
            if (p < nh) {
#pragma unroll
                for (int f = 0; f < C; ++f) {
                    const float4 s4 = *reinterpret_cast<const float4*>(sm32 + size_t(f) * nh + p);
                    const float sf[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
                    for (int v = 0; v < 4; ++v)
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float pe = v == 0 ? pv[i][r].x : v == 1 ? pv[i][r].y : v == 2 ? pv[i][r].z : pv[i][r].w;
                            acc[r * FS + f] = fmaf(pe, sf[v], acc[r * FS + f]);
                        }
                }
            }
        }
        const float tot = warp_transpose_sum<NV>(acc);
        const int idx = NV == 32 ? lane : (lane >> 1), r = idx / FS, f = idx % FS;
        if ((NV == 32 || (lane & 1) == 0) && f < C && j + r < je) a.hana[size_t(base + j + r) * C + f] = tot;
        if (!MULTI) break;
        if (j + 32 < je) request(j + 32, pv);
    }
}

// ---------------------------------------------------------------------------

static F32Args f32_args(sphnse_plan* P) {
    F32Args a{};
    a.table = static_cast<const float*>(P->tab[SPHNSE_FP32].syn);
    a.prepc = P->d_prepc32;
    a.isin = P->d_isin32;
    a.gsyn = static_cast<float*>(P->d_gsyn);
    a.gana = static_cast<const float*>(P->d_gana);
    a.hana = static_cast<float*>(P->d_hana);
    a.N = P->N;
    a.nh = P->nh;
    a.nlat = P->nlat;
    // synthesis and analysis read the same table: up to half of L2 it stays
    // there between them and the next call (F at L = 340, 60 MB: 45.5 us, 49.1
    // without), a larger one must not displace the grid fields (L = 511, 202 MB:
    // 104.6 us, 109.4 if it did; at L = 383, 85 MB, 67.4 and 66.2)
    a.evict_first = size_t(P->n_ext) * P->nh * sizeof(float) > (size_t(64) << 20);
    return a;
}

// without alpha, the fields of beta only (the others keep their values in d_gsyn)
int launch_synthesis32(sphnse_plan* P, const double* alpha, const double* beta, int pairs) {
    F32Args a = f32_args(P);
    a.alpha = reinterpret_cast<const double2*>(alpha);
    a.beta = reinterpret_cast<const double2*>(beta);
    a.pairs = pairs;
    const dim3 grid((P->nh + 63) / 64, P->N + 1);
    a.early = int(grid.x * grid.y) <= 8 * P->nsm;
    const int C = (alpha ? 6 : 0) + (beta ? 4 : 0);
    const size_t sm = (size_t(P->N + 2) * ((C + 3) / 4 * 4) + 128 * C) * sizeof(float);
    stage_begin(P, SPHNSE_STAGE_SYNTHESIS);
    const cudaError_t e = !alpha ? launch_pdl(k_syn32<2>, grid, dim3(128), sm, P->stream, a)
                          : beta ? launch_pdl(k_syn32<5>, grid, dim3(128), sm, P->stream, a)
                                 : launch_pdl(k_syn32<3>, grid, dim3(128), sm, P->stream, a);
    stage_end(P, SPHNSE_STAGE_SYNTHESIS);
    return check_cuda(e);
}

template <int NF>
static cudaError_t ana32_t(sphnse_plan* P, F32Args a) {
    // at least eight blocks per SM
    const long groups = long(P->n_ext) / 32;
    a.rb = NF == 3 && P->nh > 256 ? int(std::max(1L, std::min(4L, groups / (8L * P->nsm)))) : 1;
    const dim3 grid((ext_even(P->N, 0) + 32 * a.rb - 1) / (32 * a.rb), P->N + 1, 2);
    a.early = int(grid.x * grid.y * grid.z) <= 3 * P->nsm;
    const size_t sm = size_t(2 * NF) * P->nh * sizeof(float);
    switch ((P->nh + 127) / 128) {
        case 1: return launch_pdl(k_ana32<NF, 1>, grid, dim3(256), sm, P->stream, a);
        case 2: return launch_pdl(k_ana32<NF, 2>, grid, dim3(256), sm, P->stream, a);
        default: return launch_pdl(k_ana32<NF, 3>, grid, dim3(256), sm, P->stream, a);
    }
}

// rows of whole 16-byte vectors, at most three latitude steps (nlon <= 1536)
bool ana32_ok(const sphnse_plan* P) { return P->nh % 4 == 0 && P->nh >= 32 && P->nh <= 384; }

int launch_analysis32(sphnse_plan* P, int nf) {
    const F32Args a = f32_args(P);
    // a table larger than L2 streams faster through the persistent kernel's bulk copies (projection at
    // L = 511, 202 MB: 68 us against 76); smaller ones are latency-bound there (L = 383: 47 against 44)
    if (nf == 2 && size_t(P->n_ext) * P->nh * sizeof(float) > (size_t(128) << 20)) return launch_analysis_stream(P);
    stage_begin(P, SPHNSE_STAGE_ANALYSIS);
    const cudaError_t e = nf == 3 ? ana32_t<3>(P, a) : ana32_t<2>(P, a);
    stage_end(P, SPHNSE_STAGE_ANALYSIS);
    return check_cuda(e);
}

}  // namespace sph
