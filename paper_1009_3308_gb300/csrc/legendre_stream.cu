// Persistent streaming Legendre kernels of the FP32 ensembles, and of single
// analyses whose table exceeds L2 (CUDA cores).
//
// The per-order Legendre sums of the RHS (Sec. 4.2; synthesis of the fields
// of Eq. (app_soln_rep) and (vort_app), analysis = the discrete projection of
// Eq. (disc_vec_orth_proj)) stream the table Pt_K^m(x_p) once per pass; the
// table (>= 200 MB at L = 511) is far larger than L2, so the kernels are
// HBM-bound.  Design:
//   * one CTA per SM, persistent; the orders m are dealt to CTAs by a host
//     LPT schedule on the per-order row counts (L + 2 - m rows each);
//   * a producer warp streams rows with 1-D bulk async copies (TMA engine)
//     into an NST-stage shared-memory ring (evict-first L2 policy, so the
//     L2-resident intermediates survive); each stage holds HR even-parity and
//     HR odd-parity rows (K - m even / odd) of the current order;
//   * consumer warps wait on the stage's full mbarrier, compute, and release
//     it through its empty mbarrier;
//   * synthesis: two thread groups (even rows -> E, odd rows -> O) each own V
//     consecutive latitudes per thread, epilogue north = E + O, south = E - O;
//   * analysis: teams of warps take whole stages; a warp reduces 4 rows at a
//     time over the latitudes (lanes split p) with a transpose-reduction.
// Table layout [ext row][nh]: row (m, K) holds Pt_K^m at the nh northern nodes.
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace sph {

constexpr int NST = 6;   // pipeline depth: 6 stages of 24 KB
constexpr int V = 4;     // consecutive latitudes of a thread
constexpr int HR = 8;    // rows of each parity per stage

__device__ __forceinline__ void vload(const float* p, float* out) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    out[0] = v.x;
    out[1] = v.y;
    out[2] = v.z;
    out[3] = v.w;
}

struct StreamArgs {
    const void* table;   // [n_ext][nh]
    const void* bsyn;    // synthesis coefficient sets [n_ext][2 NF]
    void* gsyn;          // [NF][N+1][nlat] complex (m-major)
    const void* gana;    // [NF][N+1][nlat] complex (m-major)
    void* hana;          // [n_ext][2 NF]
    const double* sinth;
    const int* items;    // orders m, grouped per CTA
    const int* item_off; // [gridDim + 1]
    unsigned* status;
    int N, nh, nlat;
    // batches: an item v stands for instance v / (N+1) and order v % (N+1);
    // per-instance strides (elements) of bsyn, gsyn, gana, hana
    size_t sb, sg, sa, sh;
    int pairs;           // gsyn layout (gsyn_index)
};

// chunk c of order m: rows [c HR, c HR + HR) of the even and of the odd block
__device__ __forceinline__ void chunk_rows(int ne, int no, int c, int HR, int* cnt_e, int* cnt_o) {
    int ce = ne - c * HR, co = no - c * HR;
    *cnt_e = ce < 0 ? 0 : (ce > HR ? HR : ce);
    *cnt_o = co < 0 ? 0 : (co > HR ? HR : co);
}

// Producer: lane 0 of warp 0 walks the CTA's (order, chunk) sequence.
__device__ void produce(const StreamArgs& a, float* stages, uint64_t* full, uint64_t* empty, volatile int* abort,
                        int n_items_begin, int n_items_end) {
    const uint64_t pol = policy_evict_first();
    const float* tab = reinterpret_cast<const float*>(a.table);
    const size_t rowb = size_t(a.nh) * sizeof(float);
    int it = 0, end = 0;   // stages, and those requested
    for (int ii = n_items_begin; ii < n_items_end; ++ii) {
        const int m = a.items[ii] % (a.N + 1);
        const int ne = ext_even(a.N, m), no = ext_odd(a.N, m), e0 = ext_off(a.N, m);
        const int nch = ((ne > no ? ne : no) + HR - 1) / HR;
        for (int c = 0; c < nch; ++c, ++it) {
            const int s = it % NST;
            const uint32_t ph = (it / NST) & 1;
            if (it >= NST && !mbar_wait(&empty[s], ph ^ 1, abort, a.status)) continue;
            if (*abort) continue;
            end = it + 1;
            int ce, co;
            chunk_rows(ne, no, c, HR, &ce, &co);
            float* dst = stages + size_t(s) * 2 * HR * a.nh;
            mbar_arrive_expect_tx(&full[s], uint32_t((ce + co) * rowb));
            if (ce) bulk_g2s(dst, tab + size_t(e0 + c * HR) * a.nh, uint32_t(ce * rowb), &full[s], pol);
            if (co) bulk_g2s(dst + size_t(HR) * a.nh, tab + size_t(e0 + ne + c * HR) * a.nh, uint32_t(co * rowb),
                             &full[s], pol);
        }
    }
    // wait for the copies still in flight before leaving (bounded)
    for (int k = max(0, end - NST); k < end; ++k) mbar_drain(&full[k % NST], (k / NST) & 1, a.status);
}

// ---------------------------------------------------------------------------
// synthesis

template <int NF>
__global__ void __launch_bounds__(512, 1) k_syn_stream(StreamArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + NST;
    volatile int* abort = reinterpret_cast<volatile int*>(empty + NST);
    float* stages = reinterpret_cast<float*>(smem + 128);
    const int nh = a.nh, N = a.N, nlat = a.nlat;
    float* Bsm = stages + size_t(NST) * 2 * HR * nh;                 // 2 x [N+2][2 NF]
    float* red = Bsm + size_t(2) * (N + 2) * 2 * NF;                  // [nh][2 NF]
    const int tpg = (blockDim.x - 32) / 2;                        // threads per group
    const int n_cwarps = (blockDim.x - 32) / 32;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], n_cwarps);
        }
        *abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    pdl_launch();
    const int ib = a.item_off[blockIdx.x], iend = a.item_off[blockIdx.x + 1];
    if (threadIdx.x < 32) {
        // the tables do not depend on the predecessor: stream them right away
        if (threadIdx.x == 0) produce(a, stages, full, empty, abort, ib, iend);
        return;
    }
    pdl_wait();
    const int ct = threadIdx.x - 32;
    const int g = ct / tpg;               // 0: even rows, 1: odd rows
    const int p0 = (ct % tpg) * V;
    const bool act = p0 < nh;
    const int ncons = blockDim.x - 32;
    const float* bsyn = reinterpret_cast<const float*>(a.bsyn);
    float* gsyn = reinterpret_cast<float*>(a.gsyn);
    int it = 0;
    for (int ii = ib; ii < iend; ++ii) {
        const int inst = a.items[ii] / (N + 1), m = a.items[ii] % (N + 1);
        const int ne = ext_even(N, m), no = ext_odd(N, m), e0 = ext_off(N, m), cnt = ne + no;
        float* B = Bsm + size_t(ii & 1) * (N + 2) * 2 * NF;
        const float* bsrc = bsyn + inst * a.sb;
        float* gdst = gsyn + inst * a.sg;
        for (int i = ct; i < cnt * 2 * NF; i += ncons) B[i] = bsrc[size_t(e0) * 2 * NF + i];
        named_bar_sync(1, ncons);
        float acc[V][2 * NF];
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int f = 0; f < 2 * NF; ++f) acc[v][f] = 0.f;
        const int nch = ((ne > no ? ne : no) + HR - 1) / HR;
        for (int c = 0; c < nch; ++c, ++it) {
            const int s = it % NST;
            const bool ok = mbar_wait(&full[s], (it / NST) & 1, abort, a.status);
            int ce, co;
            chunk_rows(ne, no, c, HR, &ce, &co);
            const int nrow = g ? co : ce;
            if (ok && act) {
                const float* st = stages + (size_t(s) * 2 + g) * HR * nh + p0;
                const float* bb = B + size_t((g ? ne : 0) + c * HR) * 2 * NF;
#pragma unroll 2
                for (int r = 0; r < nrow; ++r) {
                    float pv[V];
                    vload(st + size_t(r) * nh, pv);
                    const float* b = bb + r * 2 * NF;
#pragma unroll
                    for (int f = 0; f < 2 * NF; ++f) {
                        const float bf = b[f];
#pragma unroll
                        for (int v = 0; v < V; ++v) acc[v][f] = fma(pv[v], bf, acc[v][f]);
                    }
                }
            }
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(&empty[s]);
        }
        // epilogue: odd group hands O over through shared memory
        if (g == 1 && act)
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int f = 0; f < 2 * NF; ++f) red[(p0 + v) * 2 * NF + f] = acc[v][f];
        named_bar_sync(1, ncons);
        if (g == 0 && act && !*abort) {
            const float mm = float(m);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int p = p0 + v;
                if (p >= nh) break;
                const float inv_s = float(1.0 / a.sinth[p]);
#pragma unroll
                for (int hemi = 0; hemi < 2; ++hemi) {
                    const int row = hemi == 0 ? p : nlat - 1 - p;
                    if (hemi == 1 && row == p) break;
                    const float sg = hemi == 0 ? 1.f : -1.f;
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const float gr = acc[v][2 * f] + sg * red[p * 2 * NF + 2 * f];
                        const float gi = acc[v][2 * f + 1] + sg * red[p * 2 * NF + 2 * f + 1];
                        float o0, o1;
                        if (f == 0) { o0 = gr; o1 = gi; }
                        else if (f == 1 || f == 3) { o0 = -mm * gi * inv_s; o1 = mm * gr * inv_s; }
                        else { o0 = -gr * inv_s; o1 = -gi * inv_s; }
                        float* d = gdst + gsyn_index(a.pairs, f, m, row, N, nlat) * 2;
                        d[0] = o0;
                        d[1] = o1;
                    }
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// analysis

// Transpose-reduction of NV per-lane partial sums across a warp: afterwards
// lane l holds the total of index (NV == 32 ? l : l >> 1).
template <int NV>
__device__ __forceinline__ float transpose_reduce(float* v) {
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

template <int NF, int NTEAM>
__global__ void __launch_bounds__(288, 1) k_ana_stream(StreamArgs a) {
    constexpr int QPS = 2 * HR / 4;               // row quads per stage = warps per team
    constexpr int NVR = 4 * 2 * NF;               // values per lane per quad
    constexpr int NV = NVR <= 16 ? 16 : 32;
    constexpr int FS = NV / 4;                    // slot stride per row in the reduced index
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + NST;
    volatile int* abort = reinterpret_cast<volatile int*>(empty + NST);
    float* stages = reinterpret_cast<float*>(smem + 128);
    const int nh = a.nh, N = a.N, nlat = a.nlat;
    float* Ssm = stages + size_t(NST) * 2 * HR * nh;   // 2 buffers x 2 parities x [nh][2 NF]
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], QPS);
        }
        *abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    pdl_launch();
    const int ib = a.item_off[blockIdx.x], iend = a.item_off[blockIdx.x + 1];
    if (threadIdx.x < 32) {
        // the tables do not depend on the predecessor: stream them right away
        if (threadIdx.x == 0) produce(a, stages, full, empty, abort, ib, iend);
        return;
    }
    pdl_wait();
    const int ct = threadIdx.x - 32, ncons = blockDim.x - 32;
    const int warp = ct / 32, lane = ct & 31;
    const int team = warp / QPS, q = warp % QPS;
    const int par = (q * 4) / HR;                 // quad -> parity block
    const int r0 = (q * 4) % HR;                  // first row of the quad in its block
    const float* gana = reinterpret_cast<const float*>(a.gana);
    float* hana = reinterpret_cast<float*>(a.hana);
    int it = 0;
    for (int ii = ib; ii < iend; ++ii) {
        const int inst = a.items[ii] / (N + 1), m = a.items[ii] % (N + 1);
        const int ne = ext_even(N, m), no = ext_odd(N, m), e0 = ext_off(N, m);
        const float* gsrc = gana + inst * a.sa;
        float* hdst = hana + inst * a.sh;
        // S is field-major: S[par][f][p] (par 0: G(p) + G(p'), 1: G(p) - G(p'))
        // so that a lane's V consecutive latitudes are one conflict-free vector load
        float* S = Ssm + size_t(ii & 1) * 2 * nh * 2 * NF;
        for (int i = ct; i < nh * NF; i += ncons) {
            const int f = i / nh, p = i % nh, pr = nlat - 1 - p;
            const float* ga = gsrc + gsyn_index(0, f, m, p, N, nlat) * 2;
            float ar = ga[0], ai = ga[1], br = 0.f, bi = 0.f;
            if (pr != p) {
                const float* gb = gsrc + gsyn_index(0, f, m, pr, N, nlat) * 2;
                br = gb[0];
                bi = gb[1];
            }
            S[size_t(2 * f) * nh + p] = ar + br;
            S[size_t(2 * f + 1) * nh + p] = ai + bi;
            S[size_t(2 * NF + 2 * f) * nh + p] = ar - br;
            S[size_t(2 * NF + 2 * f + 1) * nh + p] = ai - bi;
        }
        named_bar_sync(1, ncons);
        const int nch = ((ne > no ? ne : no) + HR - 1) / HR;
        for (int c = 0; c < nch; ++c, ++it) {
            if (it % NTEAM != team) continue;
            const int s = it % NST;
            const bool ok = mbar_wait(&full[s], (it / NST) & 1, abort, a.status);
            int ce, co;
            chunk_rows(ne, no, c, HR, &ce, &co);
            const int nrow = (par ? co : ce) - r0;   // rows of this quad present
            if (ok && nrow > 0) {
                float acc[NV];
#pragma unroll
                for (int i = 0; i < NV; ++i) acc[i] = 0.f;
                const float* st = stages + (size_t(s) * 2 + par) * HR * nh + size_t(r0) * nh;
                const float* Sp = S + size_t(par) * nh * 2 * NF;
                for (int p = lane * V; p < nh; p += 32 * V) {
                    float pv[4][V];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        if (r < nrow) vload(st + size_t(r) * nh + p, pv[r]);
                        else
#pragma unroll
                            for (int v = 0; v < V; ++v) pv[r][v] = 0.f;
                    }
#pragma unroll
#pragma unroll
                    for (int f = 0; f < 2 * NF; ++f) {
                        float sf[V];
                        vload(Sp + size_t(f) * nh + p, sf);
#pragma unroll
                        for (int v = 0; v < V; ++v)
#pragma unroll
                            for (int r = 0; r < 4; ++r) acc[r * FS + f] = fma(pv[r][v], sf[v], acc[r * FS + f]);
                    }
                }
                const float tot = transpose_reduce<NV>(acc);
                const int idx = NV == 32 ? lane : (lane >> 1);
                const int r = idx / FS, f = idx % FS;
                const bool writer = (NV == 32 || (lane & 1) == 0) && f < 2 * NF && r < nrow;
                if (writer && !*abort) {
                    const int row = e0 + (par ? ne : 0) + c * HR + r0 + r;
                    hdst[size_t(row) * 2 * NF + f] = tot;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
    }
}

// ---------------------------------------------------------------------------
// host launchers

bool stream_ok(const sphnse_plan* P) { return P->d_items != nullptr && P->nh % 4 == 0 && P->nh >= 32; }

// FP32 batched streaming passes over instances (items = inst * (N+1) + m)
int launch_synthesis_stream_batch(sphnse_plan* P, const int* items, const int* item_off, int ncta,
                                  const float* bsyn, size_t sb, float* gsyn, size_t sg, int pairs) {
    const int tpg = ((P->nh / 4 + 31) / 32) * 32;
    const int threads = 32 + 2 * tpg;
    const size_t sm = 128 + sizeof(float) * (size_t(NST) * 2 * HR * P->nh + size_t(2) * (P->N + 2) * 6 +
                                             size_t(P->nh) * 6);
    if (threads > 512 || sm > 227 * 1024 || !stream_ok(P)) return SPHNSE_E_UNSUPPORTED;
    allow_dynamic_smem(reinterpret_cast<const void*>(k_syn_stream<3>), sm);
    StreamArgs a{P->tab[SPHNSE_FP32].syn, bsyn, gsyn, nullptr, nullptr, P->d_s, items, item_off, P->d_status,
                 P->N, P->nh, P->nlat, sb, sg, 0, 0, pairs};
    stage_begin(P, SPHNSE_STAGE_SYNTHESIS);
    launch_pdl(k_syn_stream<3>, dim3(ncta), dim3(threads), sm, P->stream, a);
    stage_end(P, SPHNSE_STAGE_SYNTHESIS);
    return check_cuda(cudaGetLastError());
}

int launch_analysis_stream(sphnse_plan* P) {
    return launch_analysis_stream_batch(P, P->d_items, P->d_item_off, P->n_cta, static_cast<const float*>(P->d_gana), 0,
                                        static_cast<float*>(P->d_hana), 0);
}

int launch_analysis_stream_batch(sphnse_plan* P, const int* items, const int* item_off, int ncta,
                                 const float* gana, size_t sa, float* hana, size_t sh) {
    constexpr int QPS = 2 * HR / 4;
    constexpr int NTEAM = 8 / QPS;
    const int threads = 32 + 32 * QPS * NTEAM;
    const size_t sm = 128 + sizeof(float) * (size_t(NST) * 2 * HR * P->nh + size_t(2) * 2 * P->nh * 4);
    if (sm > 227 * 1024 || !stream_ok(P)) return SPHNSE_E_UNSUPPORTED;
    allow_dynamic_smem(reinterpret_cast<const void*>(k_ana_stream<2, NTEAM>), sm);
    StreamArgs a{P->tab[SPHNSE_FP32].syn, nullptr, nullptr, gana, hana, P->d_s, items, item_off, P->d_status,
                 P->N, P->nh, P->nlat, 0, 0, sa, sh, 0};
    stage_begin(P, SPHNSE_STAGE_ANALYSIS);
    launch_pdl(k_ana_stream<2, NTEAM>, dim3(ncta), dim3(threads), sm, P->stream, a);
    stage_end(P, SPHNSE_STAGE_ANALYSIS);
    return check_cuda(cudaGetLastError());
}

}  // namespace sph
