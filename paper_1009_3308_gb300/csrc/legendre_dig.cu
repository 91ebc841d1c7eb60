// FP64 Legendre synthesis and analysis on the tcgen05 tensor cores, by exact
// digit splitting (the error-free splitting of matrix products of Ozaki,
// Ogita, Oishi and Rump, Numer. Algorithms 59 (2012)).
//
// Every table row is scaled by a power of two to |a| < 0.993, every coefficient
// (or profile) column to |b| <= 1/2, and both are cut into eight balanced
// base-256 digits:  a = sum_i a_i 2^(1 - 8 i),  b = sum_j b_j 2^(1 - 8 j),
// |a_i|, |b_j| <= 128.  The products of i + j = s share one accumulator group,
// s = 2 .. 10:
//     sum_k a b = sum_s 2^(2 - 8 s) D_s,   D_s = sum_{i + j = s} sum_k a_i b_j,
// and the epilogue adds the groups in integers.  Digits are exact in FP16, their
// products are integers of at most 2^14.  For the digits of these tables (14
// orders at L = 511) no column makes |D_s| reach 2^24 in the synthesis, nor in
// the analysis up to s = 6, so that the FP32 accumulators hold it exactly; the
// bound of the analysis' last groups is 2^24.6, where a rounding is worth 2^-54
// of max|a| max|b| at most (no such sum has been seen: digits past the first
// are spread out and sums stay near 2^20).
//
// Error.  Relative to max|a| max|b| of a row and a column, digits end at 2^-64
// and the products left out (i + j > 10) add up to about 2^-67.  A multiply-add
// chain errs relative to the largest product |a_k b_k|, which is far smaller
// where a state's low degrees meet polar rows: there Pt_K^m rises with K like
// K^(m + 1/2), the spectrum falls, and the result is divided by sin(theta).
// Eight table digits cover the 2^9 of 1/sin(theta) at L = 511; with seven the
// largest error of u_theta for the mode (9, 8) was 5.1e-15 of its maximum, with
// eight 2.5e-16 as in a multiply-add chain.  For the columns the degrees of an
// order are balanced: table entries of degree K are divided, coefficient sets
// multiplied by 2^t, t = floor(log2(K + 1)) up to a constant (dig_shift); without it
// a spectrum falling like l^-4 lost a factor of four (order 1 at L = 511).  What stays below
// the chain's precision are results smaller than 2^-60 of max|a| max|b|: the
// projection of a field that lives on polar rows in one order above about ten.
//
// Per K = 16 step one tile of 128 table rows takes eight MMAs, digit i of the
// table against digits 1 .. 10 - i of the columns (N = G (10 - i), G
// columns per group): with the columns of a group adjacent, those digits are a prefix of
// the B rows and land on the groups from i + 1 on, a contiguous run of accumulator
// columns.  The table digits are stored once per plan as bytes (digit + 128) in
// the order the kernels consume them: one 16 KB block per (tile, K step) = 8
// planes of 128 x 16, one bulk copy each; blocks whose digits are all zero
// (polar latitudes at high order) are left out.  Four warps expand a block to
// FP16 (a byte under 0x64 is 1024 + byte; one packed subtraction) straight into
// tensor memory, where the MMAs take their A operand: written to shared memory
// instead, the expanded digits cost more than the halved HBM stream saved.
//
// Bound: the single-K-step stages, whose barrier waits (150 to 200 cycles even
// when they pass at once), expansion and MMAs take about 1070 (synthesis) and 890
// (analysis) cycles per 16 KB block, which streams in 760 at the measured copy rate
// (6.8 TB/s).  The FP64 pipe (two operations per clock per SM) would need 10 multiply-adds per
// entry and RHS: 0.8 ms at L = 511.
// Measured (event pairs, GB300) against the FP64 multiply-add kernels and their
// prep: L = 511 synthesis 558 -> 94 us, analysis 429 -> 80; L = 255 96 -> 30,
// 74 -> 22; L = 100 41 -> 15, 22 -> 13.  Errors of the sums against extended
// precision, emulated for single modes, exponential and power-law spectra at L =
// 53, 100, 255 and 511, 8 to 18 orders each: the largest and the mean error of
// every field are at most 1.1 times those of the multiply-add chain and mostly
// smaller (two states of order 0 at L = 100: 1.2 times).
//
// Synthesis tiles: rows 0 .. 63 the even, rows 64 .. 127 the odd degrees of one
// order on 64 northern latitudes (columns 0 .. G/2-1 of a group belong to the
// even, the others to the odd degrees), so north = E + O and south = E - O
// meet in one epilogue.  Analysis tiles: four pieces of up to 32 rows of one
// (order, parity), one per epilogue warp, each with its own G / 4 columns.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "fx64.cuh"
#include "internal.h"
#include "tc.cuh"

namespace sph {

constexpr int DG_ND = 8;                     // digits of the table and of the columns
constexpr int DG_NG = 9;                     // accumulator groups i + j = 2 .. 10
constexpr int DG_RPLANE = 128 * 16;          // a digit of 128 rows x 16 of the contracted index: bytes digit + 128
constexpr int DG_RBYTES = DG_ND * DG_RPLANE; // one block of the stored table
constexpr int DG_ACOLS = DG_ND * 8;          // the same in FP16: columns of tensor memory, a row per lane
constexpr int DG_NX = 3;                     // stages of it
constexpr int DG_MINEXP = -22;               // row scales are at least 2^-22 (smaller rows lose digits below 2^-86)
constexpr int DG_NAN = 1 << 20;              // exponent of a column with a non-finite entry

// byte offset of element (row, k) of a K = 16 tile: rows of 32 bytes, the two
// halves swapped in every second group of four rows (32-byte swizzle)
__host__ __device__ constexpr int dg_off(int row, int k) {
    return row * 32 + (((k >> 3) ^ (row >> 2)) & 1) * 16 + (k & 7) * 2;
}
// shared-memory descriptor of that layout: K-major, 32-byte swizzle
__device__ __forceinline__ uint64_t dg_desc(const void* smem_ptr) {
    uint64_t d = 0;
    d |= uint64_t((smem_u32(smem_ptr) & 0x3FFFF) >> 4);
    d |= uint64_t(1) << 16;          // leading byte offset (unused with swizzle)
    d |= uint64_t(256 >> 4) << 32;   // to the next 8 rows
    d |= uint64_t(1) << 46;
    d |= uint64_t(6) << 61;          // 32-byte swizzle
    return d;
}

// two bytes digit + 128 under 0x64 are the FP16 numbers 1152 + digit
__device__ __forceinline__ uint32_t dg_half2(uint32_t w) {
    const __half2 bias = __half2half2(__ushort_as_half(0x6480));
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), bias);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ int dg_steps(int n) { return (n + 15) / 16; }

// ---------------------------------------------------------------------------
// table digits (once per plan)

// row exponents: |P| < (1 - 2^-7) 2^e over a row, so that the top digit stays below 128.  Synthesis rows are (m, latitude p)
// over all degrees of the order, analysis rows are the ext rows over p.
__device__ __forceinline__ int dg_bexp(double x) { return f64_bexp(fma(x, 0x1p-7, x)); }
__global__ void k_dig_syn_scale(const double* __restrict__ tab, int* __restrict__ ea, int N, int nh) {
    const int m = blockIdx.y, p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nh) return;
    const int ne = ext_even(N, m), cnt = ext_count(N, m);
    const double* t = tab + size_t(ext_off(N, m)) * nh + p;
    int e = 0;
    for (int r = 0; r < cnt; ++r) {
        const int K = r < ne ? m + 2 * r : m + 1 + 2 * (r - ne);
        e = max(e, dg_bexp(t[size_t(r) * nh]) - dig_shift(N, K));
    }
    ea[m * nh + p] = max(e - 1022, DG_MINEXP - dig_shift(N, 0));   // of entries scaled up by -dig_shift
}
__global__ void k_dig_ana_scale(const double* __restrict__ tab, int* __restrict__ ea, int n_ext, int nh) {
    const int r = blockIdx.x * 4 + threadIdx.x / 32;
    if (r >= n_ext) return;
    int e = 0;
    for (int p = threadIdx.x & 31; p < nh; p += 32) e = max(e, dg_bexp(tab[size_t(r) * nh + p]));
    e = __reduce_max_sync(0xffffffffu, e);
    if ((threadIdx.x & 31) == 0) ea[r] = max(e - 1022, DG_MINEXP);
}

// the digits of eight scaled entries -> eight bytes of each plane; returns whether any is nonzero
__device__ __forceinline__ bool dig_store(const double (&x)[8], const int (&e)[8], unsigned char* dst) {
    unsigned long long w[DG_ND] = {};
    bool any = false;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const long long v = f64_to_fx(x[i], 63 - e[i]);
        any = any || v != 0;
        const unsigned long long u = (unsigned long long)v + 0x8080808080808080ULL;
#pragma unroll
        for (int d = 0; d < DG_ND; ++d) w[d] |= ((u >> (56 - 8 * d)) & 255) << (8 * i);
    }
#pragma unroll
    for (int d = 0; d < DG_ND; ++d) *reinterpret_cast<unsigned long long*>(dst + d * DG_RPLANE) = w[d];
    return any;
}

// block = (step, latitude tile, order): thread = (row, half of the step)
__global__ void __launch_bounds__(256) k_dig_syn(const double* __restrict__ tab, const int* __restrict__ ea,
                                                 const int* __restrict__ base, unsigned char* __restrict__ out,
                                                 int* __restrict__ used, int N, int nh, int ntile) {
    const int m = blockIdx.z, t = blockIdx.y, ks = blockIdx.x, ne = ext_even(N, m);
    if (ks >= dg_steps(ne)) return;
    const int row = threadIdx.x & 127, h = threadIdx.x >> 7, par = row >> 6, p = t * 64 + (row & 63);
    const int n = par ? ext_odd(N, m) : ne;
    const double* src = tab + size_t(ext_off(N, m) + (par ? ne : 0)) * nh + p;
    double x[8];
    int e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int j = ks * 16 + h * 8 + i;
        x[i] = j < n && p < nh ? src[size_t(j) * nh] : 0.0;
        e[i] = p < nh ? ea[m * nh + p] + dig_shift(N, m + par + 2 * j) : 0;
    }
    const int blk = base[m * ntile + t] + ks;
    const bool any = dig_store(x, e, out + size_t(blk) * DG_RBYTES + row * 16 + h * 8);
    if (__syncthreads_or(any) && threadIdx.x == 0) used[blk] = 1;
}
__global__ void __launch_bounds__(256) k_dig_ana(const double* __restrict__ tab, const int* __restrict__ ea,
                                                 const int4* __restrict__ pieces, unsigned char* __restrict__ out,
                                                 int* __restrict__ used, int nh) {
    const int tile = blockIdx.y, ks = blockIdx.x, nks = gridDim.x;
    const int h = threadIdx.x & 1, row = threadIdx.x >> 1;
    const int4 pc = pieces[4 * tile + (row >> 5)];
    const bool in = (row & 31) < pc.w;
    const int r = pc.z + (row & 31);
    double x[8];
    int e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int p = ks * 16 + h * 8 + i;
        x[i] = in && p < nh ? tab[size_t(r) * nh + p] : 0.0;
        e[i] = in ? ea[r] : 0;
    }
    const int blk = tile * nks + ks;
    const bool any = dig_store(x, e, out + size_t(blk) * DG_RBYTES + row * 16 + h * 8);
    if (__syncthreads_or(any) && threadIdx.x == 0) used[blk] = 1;
}

// ---------------------------------------------------------------------------

struct DigArgs {
    const unsigned char* blocks;  // table digits, DG_RBYTES per (tile, step)
    const int4* items;            // (m or analysis tile, latitude tile, first step | end step << 16,
                                  //  first block)
    const int* cnt;               // items of every CTA, at c * istride
    int istride;
    int evict_first;              // the digits exceed what L2 can keep
    const int* ea;                // row exponents
    unsigned* status;
    int N, nh, nlat;
    // synthesis
    const double2* alpha;
    const double2* beta;          // adjoint: fields 3, 4
    const double4_32a* prepc;
    const short4* eoff;           // exponents of the coefficient sets per packed entry
    double* gsyn;                 // [nf][pair][N+1][2] complex
    const double* isin;           // 1 / sin(theta_p)
    // analysis
    const int4* pieces;           // (m, parity, first ext row, rows) x 4 per tile
    const double* gana;           // [nf][pair][N+1][2] complex
    const int* emax;              // largest biased exponent of gana per (field, order)
    double* hana;                 // [n_ext][2 nf]
};

// two scaled values of a column (contracted indexes 2 w, 2 w + 1) -> word w of the column's
// rows of all eight digits; stride: bytes between the digits
__device__ __forceinline__ void dig_put(unsigned char* dst, int stride, long long b0, long long b1) {
    const unsigned long long u0 = (unsigned long long)b0 + 0x8080808080808080ULL;
    const unsigned long long u1 = (unsigned long long)b1 + 0x8080808080808080ULL;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint32_t s0 = j < 4 ? uint32_t(u0 >> 32) : uint32_t(u0), s1 = j < 4 ? uint32_t(u1 >> 32) : uint32_t(u1);
        const int q = 3 - (j & 3);
        const uint32_t w = __byte_perm(s0, s1, q | (4 + q) << 8);   // bytes 0 and 2
        *reinterpret_cast<uint32_t*>(dst + j * stride) = dg_half2(__byte_perm(w, 0x64646464u, 0x4240));
    }
}

// the sum over an item without a nonzero digit block, whose accumulator holds no
// data: 0, but NaN for a column with a non-finite entry (its product with a zero)
__device__ __forceinline__ double dig_none(int e) {
    return e >= DG_NAN / 2 ? __longlong_as_double(0x7FF8000000000000LL) : 0.0;
}

// sum_s D_s 2^(2 - 8 s) 2^e: the groups of one output added exactly, as
// h 2^-54 + r 2^-70, and rounded once to binary64
__device__ __forceinline__ double dig_val(const uint32_t* d, int stride, int e) {
    int g[DG_NG];
#pragma unroll
    for (int s = 0; s < DG_NG; ++s) g[s] = __float2int_rn(__uint_as_float(d[s * stride]));
    const long long h = ((long long)g[0] << 40) + ((long long)g[1] << 32) + ((long long)g[2] << 24) +
                        ((long long)g[3] << 16) + ((long long)g[4] << 8) + g[5];
    const long long r = (long long)g[6] * 256 + g[7] + ((g[8] + 128) >> 8);
    if (e >= DG_NAN / 2) return dig_none(e);
    // as many of r's bits as fit below h (|h| < 2^62: 384 terms of at most 1/2)
    const int sh = min(16, max(0, __clzll(h ^ (h >> 63)) - 3));
    const long long v = (h << sh) + (r >> (16 - sh));
    return v == 0 ? 0.0 : f64_scale(__ll2double_rn(v), e - 54 - sh);
}

// position in a ring of n slots: slot and the parity of its uses
struct DigRing {
    int slot = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void next(int n) {
        if (++slot == n) {
            slot = 0;
            phase ^= 1;
        }
    }
};

template <bool SYN, int NF> struct DigShape {
    // columns of one order and parity, padded; group width; pipeline stages
    static constexpr int C = 2 * NF;
    static constexpr int CP = SYN ? (C <= 8 ? 8 : 16) : (C <= 4 ? 4 : 8);
    static constexpr int G = SYN ? 2 * CP : 4 * CP;
    static constexpr int BBYTES = DG_NG * G * 32;            // eight digits of the columns and a zero digit
    static constexpr int NACC = 2 * DG_NG * G + DG_NX * DG_ACOLS <= 512 ? 2 : 1;   // accumulator buffers
    static_assert(NACC * DG_NG * G + DG_NX * DG_ACOLS <= 512, "tensor memory");
    // ring of stored table blocks (what is in flight from memory) and of column digits
    static constexpr int NR = SYN && G == 32 ? 8 : 10;
    static constexpr int NS = SYN ? (NF == 3 ? 9 : 6) : (NF == 2 ? 10 : 6);
    static constexpr int XCH = SYN ? 2 * 128 * C * 8 : 0;   // even and odd sums meet here
    // Copy, MMA, 4 epilogue, builder, 4 expander warps, and SYN: column exponents.
    // A builder takes 4000 to 6000 cycles per stage (load latency, FP64 and 64-bit
    // integer chains), so there are as many as the registers allow: 20 warps of 96,
    // where that does not spill, else 16 of 128.
    static constexpr int NB = SYN ? (NF == 3 ? 9 : 5) : (NF == 2 ? 10 : 6);
    static constexpr int WARPS = 10 + NB + (SYN ? 1 : 0);
    static constexpr size_t smem(int istride) {
        return 1024 + size_t(NR) * DG_RBYTES + size_t(NS) * BBYTES + XCH + 512 + size_t(istride) * (16 + 8 + 20);
    }
};

template <bool SYN, int NF>
__global__ void __launch_bounds__(32 * DigShape<SYN, NF>::WARPS, 1) k_dig(DigArgs a) {
    using Q = DigShape<SYN, NF>;
    constexpr int NS = Q::NS, NR = Q::NR, NX = DG_NX, G = Q::G, C = Q::C, CP = Q::CP, NG = DG_NG, NACC = Q::NACC;
    static_assert(8 * (2 * (NR + NX + NS) + 4) + 8 <= 512, "barriers");
    constexpr int NB = Q::NB, NBW = NS < NB ? NS : NB;   // a builder per stage, none a full ring ahead
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                           ~uintptr_t(1023));
    unsigned char* Rs = smem;
    unsigned char* Bs = Rs + NR * DG_RBYTES;
    double* xch = reinterpret_cast<double*>(Bs + NS * Q::BBYTES);
    uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(xch) + Q::XCH);
    uint64_t* r_full = bars;
    uint64_t* r_empty = r_full + NR;
    uint64_t* a_full = r_empty + NR;
    uint64_t* a_empty = a_full + NX;
    uint64_t* b_full = a_empty + NX;
    uint64_t* b_empty = b_full + NS;
    uint64_t* acc_full = b_empty + NS;
    uint64_t* acc_empty = acc_full + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int4* s_items = reinterpret_cast<int4*>(reinterpret_cast<unsigned char*>(bars) + 512);
    uint64_t* sc_full = reinterpret_cast<uint64_t*>(s_items + a.istride);   // SYN: column exponents of an item ready
    int* s_eb = reinterpret_cast<int*>(sc_full + a.istride);               // [item][5]
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const int N = a.N, nh = a.nh, nlat = a.nlat, npair = (nlat + 1) / 2;
    const int nI = a.cnt[blockIdx.x];
    for (int i = threadIdx.x; i < a.istride; i += blockDim.x) {
        s_items[i] = a.items[blockIdx.x * a.istride + i];
        mbar_init(&sc_full[i], 1);
    }
    for (int i = threadIdx.x; i < NS * Q::BBYTES / 16; i += blockDim.x)
        reinterpret_cast<uint4*>(Bs)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_proxy_async_smem();
    if (threadIdx.x == 0) {
        for (int s = 0; s < NR; ++s) {
            mbar_init(&r_full[s], 1);
            mbar_init(&r_empty[s], 4);
        }
        for (int s = 0; s < NX; ++s) {
            mbar_init(&a_full[s], 4);
            mbar_init(&a_empty[s], 1);
        }
        for (int s = 0; s < NS; ++s) {
            mbar_init(&b_full[s], 1);
            mbar_init(&b_empty[s], 1);
        }
        for (int b = 0; b < NACC; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 128);
        }
        *abort = 0;
    }
    fence_barrier_init();
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_launch();
    const uint32_t tmem = *tmem_slot, tmemA = tmem + NACC * NG * G;

    if (warp == 0) {
        if (elect_one()) {
            // the table does not depend on the predecessor: stream right away
            const uint64_t pol = a.evict_first ? policy_evict_first() : policy_evict_last();
            DigRing r;
            int it = 0, end = 0;   // blocks, and those requested (all, unless a wait ran out)
            for (int i = 0; i < nI; ++i) {
                const int4 itm = s_items[i];
                const unsigned char* src = a.blocks + size_t(itm.w) * DG_RBYTES;
                const int k1 = itm.z >> 16;
                for (int ks = itm.z & 0xFFFF; ks < k1; ++ks, ++it, r.next(NR)) {
                    if (it >= NR && !mbar_wait(&r_empty[r.slot], r.phase ^ 1, abort, a.status)) continue;
                    if (*abort) continue;
                    end = it + 1;
                    mbar_arrive_expect_tx(&r_full[r.slot], DG_RBYTES);
                    bulk_g2s(Rs + r.slot * DG_RBYTES, src + size_t(ks) * DG_RBYTES, DG_RBYTES, &r_full[r.slot], pol);
                }
            }
            for (int k = max(0, end - NR); k < end; ++k) mbar_drain(&r_full[k % NR], (k / NR) & 1, a.status);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            DigRing ra, rb;
            for (int i = 0; i < nI; ++i) {
                const int4 itm = s_items[i];
                const int buf = i % NACC, k0 = itm.z & 0xFFFF, k1 = itm.z >> 16;
                bool ok = true;
                if (i >= NACC) ok = mbar_wait(&acc_empty[buf], (i / NACC - 1) & 1, abort, a.status);
                tc_fence_after();
                const uint32_t d = tmem + uint32_t(buf * NG * G);
                for (int ks = k0; ks < k1; ++ks, ra.next(NX), rb.next(NS)) {
                    ok = mbar_wait2(&a_full[ra.slot], ra.phase, &b_full[rb.slot], rb.phase, abort, a.status) && ok;
                    tc_fence_after();
                    if (ok) {
                        const unsigned char* B = Bs + rb.slot * Q::BBYTES;
                        const uint64_t bd = dg_desc(B);
                        const uint32_t ad = tmemA + ra.slot * DG_ACOLS;
                        // the first digit's MMA starts groups 0 .. 7, the zero digit group 8
                        if (ks == k0)
                            mma_f16_ta(d + 8 * G, ad, dg_desc(B + 8 * G * 32), idesc_f16(128, G), 0);
#pragma unroll
                        for (int g = 0; g < DG_ND; ++g)
                            mma_f16_ta(d + g * G, ad + g * 8, bd, idesc_f16(128, G * (NG - g < 8 ? NG - g : 8)),
                                       ks > k0 || g > 0);
                    }
                    mma_commit(&a_empty[ra.slot]);
                    mma_commit(&b_empty[rb.slot]);
                }
                mma_commit(&acc_full[buf]);
            }
            if (nI > 0) mbar_drain(&acc_full[(nI - 1) % NACC], ((nI - 1) / NACC) & 1, a.status);
        }
    } else if (warp < 6) {
        pdl_wait();
        const int quarter = warp & 3;
        const uint32_t lanes = uint32_t(quarter * 32) << 16;
        int xb = 0;    // exchange buffer
        for (int i = 0; i < nI; ++i) {
            const int4 itm = s_items[i];
            const int buf = i % NACC;
            const bool none = (itm.z & 0xFFFF) >= (itm.z >> 16);   // no nonzero block
            const uint32_t d0 = tmem + lanes + uint32_t(buf * NG * G);
            if constexpr (SYN) {
                const int m = itm.x, par = quarter >> 1, pl = (quarter & 1) * 32 + lane, p = itm.y * 64 + pl;
                const double inv = p < nh ? a.isin[p] : 0.0, minv = inv * double(m);
                const int ea = p < nh ? a.ea[m * nh + p] : 0;
                double V[C];   // this row's sums
                mbar_wait(&acc_full[buf], (i / NACC) & 1, abort, a.status);
                tc_fence_after();
                mbar_wait(&sc_full[i], 0, abort, a.status);
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    uint32_t d[2 * NG];
#pragma unroll
                    for (int s = 0; s < NG; ++s) tmem_ld2_nowait(d0 + uint32_t(s * G + par * CP + 2 * f), d + 2 * s);
                    tmem_wait_ld();
                    const int e = ea + s_eb[5 * i + f];
                    V[2 * f] = none ? dig_none(e) : dig_val(d, 2, e);
                    V[2 * f + 1] = none ? dig_none(e) : dig_val(d + 1, 2, e);
                }
                tc_fence_before();
                mbar_arrive(&acc_empty[buf]);
                // even and odd sums meet: the even warps write north = E + O, the odd ones south = E - O
                double* mine = xch + ((size_t(xb) * 2 + par) * 64 + pl) * C;
                const double* other = xch + ((size_t(xb) * 2 + 1 - par) * 64 + pl) * C;
                xb ^= 1;
#pragma unroll
                for (int c = 0; c < C; ++c) mine[c] = V[c];
                named_bar_sync(1, 128);
                const int row = par ? nlat - 1 - p : p;
                if (p >= nh || (par && row == p) || *abort) continue;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const double gr = par ? other[2 * f] - V[2 * f] : V[2 * f] + other[2 * f];
                    const double gi = par ? other[2 * f + 1] - V[2 * f + 1] : V[2 * f + 1] + other[2 * f + 1];
                    double2 o;
                    if (f == 0) o = make_double2(gr, gi);
                    else if (f == 1 || f == 3) o = make_double2(-gi * minv, gr * minv);   // (i m / sin) g
                    else o = make_double2(-gr * inv, -gi * inv);                          // -(1 / sin) g
                    *reinterpret_cast<double2*>(a.gsyn + gsyn_index(1, f, m, row, N, nlat) * 2) = o;
                }
            } else {
                const int4 pc = a.pieces[4 * itm.x + quarter];
                const int row = pc.z + lane;
                const bool in = lane < pc.w;
                const int ea = in ? a.ea[row] : 0;
                int eb[NF];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const int b = a.emax[f * (N + 1) + pc.x];
                    eb[f] = b == 2047 ? DG_NAN : b - 1020;
                }
                mbar_wait(&acc_full[buf], (i / NACC) & 1, abort, a.status);
                tc_fence_after();
                double H[C];
                if constexpr (CP == 4) {
                    uint32_t d[NG * CP];
#pragma unroll
                    for (int s = 0; s < NG; ++s) tmem_ld4_nowait(d0 + uint32_t(s * G + quarter * CP), d + CP * s);
                    tmem_wait_ld();
                    tc_fence_before();
                    mbar_arrive(&acc_empty[buf]);
#pragma unroll
                    for (int c = 0; c < C; ++c) H[c] = none ? dig_none(ea + eb[c / 2]) : dig_val(d + c, CP, ea + eb[c / 2]);
                } else {
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        uint32_t d[2 * NG];
#pragma unroll
                        for (int s = 0; s < NG; ++s) tmem_ld2_nowait(d0 + uint32_t(s * G + quarter * CP + 2 * f), d + 2 * s);
                        tmem_wait_ld();
                        H[2 * f] = none ? dig_none(ea + eb[f]) : dig_val(d, 2, ea + eb[f]);
                        H[2 * f + 1] = none ? dig_none(ea + eb[f]) : dig_val(d + 1, 2, ea + eb[f]);
                    }
                    tc_fence_before();
                    mbar_arrive(&acc_empty[buf]);
                }
                if (!in || *abort) continue;
#pragma unroll
                for (int f = 0; f < NF; ++f)
                    *reinterpret_cast<double2*>(a.hana + size_t(row) * C + 2 * f) = make_double2(H[2 * f], H[2 * f + 1]);
            }
        }
    } else if (warp < 6 + NB) {
        // builders: warp 6 + it % NBW writes stage it's column digits
        const int bw = warp - 6;
        // Synthesis: task = (parity, field, contracted index), a value per lane, and
        // two lanes of adjacent indexes exchange real and imaginary parts to write
        // a word of two each (a word's two indexes per lane left a quarter of the
        // lanes idle: L = 511 99 us, now 94, L = 255 34, now 32).  Analysis: task = (piece, field, two latitudes).
        constexpr int NT = SYN ? 2 * NF * 16 : 4 * NF * 8, TR = (NT + 31) / 32;
        static_assert(NT % 32 == 0 || !SYN, "whole warps");
        constexpr int XV = SYN ? 2 : 4;   // values loaded per task
        pdl_wait();
        int it = 0;
        if (bw < NBW)
            for (int i = 0; i < nI; ++i) {
                const int4 itm = s_items[i];
                const int k1 = itm.z >> 16;
                int4 pc[TR];
                int kb[TR];
                bool big = false;   // analysis: a sum of two x may exceed the largest number
                if constexpr (!SYN) {
#pragma unroll
                    for (int r = 0; r < TR; ++r) {
                        const int task = r * 32 + lane;
                        pc[r] = task < NT ? a.pieces[4 * itm.x + (task >> 3) / NF] : make_int4(0, 0, 0, 0);
                    }
#pragma unroll
                    for (int r = 0; r < TR; ++r)
                        kb[r] = 63 - (a.emax[((r * 32 + lane) >> 3) % NF * (N + 1) + pc[r].x] - 1020);
#pragma unroll
                    for (int r = 0; r < TR; ++r) big = big || kb[r] < 63 - 1025;
#pragma unroll
                    for (int r = 0; r < TR; ++r) kb[r] += big;
                }
                for (int ks = itm.z & 0xFFFF; ks < k1; ++ks, ++it) {
                    if (it % NBW != bw) continue;
                    const int s = it % NS;
                    // every load of the stage before the first use of one, and before the wait for the slot
                    double2 x[TR][XV];
                    double sg[TR];
                    double2 cf[TR];
                    if constexpr (SYN) {
                        const int m = itm.x, ne = ext_even(N, m), lo = m > 0 ? m : 1, pk = packed_off(N, m) - lo;
#pragma unroll
                        for (int r = 0; r < TR; ++r) {
                            const int task = r * 32 + lane, f = (task >> 4) % NF, par = (task >> 4) / NF;
                            const int n = par ? ext_odd(N, m) : ne, r0 = ext_off(N, m) + (par ? ne : 0);
                            const bool deg = f == 2 || f == 4;   // the degree-shift set
                            const double2* src = f < 3 ? a.alpha : a.beta;
                            const int j = ks * 16 + (task & 15), K = m + par + 2 * j, K1 = deg ? K - 1 : K, K2 = K + 1;
                            const double2 z = make_double2(0.0, 0.0);
                            const double2* c = reinterpret_cast<const double2*>(a.prepc + r0 + j) + deg;
                            cf[r] = j < n ? *c : z;
                            x[r][0] = j < n && K1 >= lo && K1 <= N ? src[pk + K1] : z;
                            x[r][1] = deg && j < n && K2 <= N ? src[pk + K2] : z;
                        }
                        mbar_wait(&sc_full[i], 0, abort, a.status);
                    } else {
#pragma unroll
                        for (int r = 0; r < TR; ++r) {
                            const int w = lane & 7, f = ((r * 32 + lane) >> 3) % NF, p = ks * 16 + 2 * w;
                            const double* g = a.gana + (size_t(f) * npair * size_t(N + 1) + pc[r].x) * 4;
                            const size_t ld = size_t(N + 1) * 4;
                            const double2 z = make_double2(0.0, 0.0);
                            sg[r] = pc[r].y ? -1.0 : 1.0;
                            x[r][0] = x[r][1] = x[r][2] = x[r][3] = z;   // p, p + 1 and their mirrors
                            if (pc[r].w > 0 && p < nh) {
                                const double4_32a no = *reinterpret_cast<const double4_32a*>(g + size_t(p / 2) * ld);
                                x[r][0] = make_double2(no.x, no.y);
                                if (p + 1 < nh) x[r][1] = make_double2(no.z, no.w);
                                if (nlat % 2 == 0) {
                                    const double4_32a so =
                                        *reinterpret_cast<const double4_32a*>(g + size_t((nlat - 2 - p) / 2) * ld);
                                    x[r][2] = make_double2(so.z, so.w);
                                    if (p + 1 < nh) x[r][3] = make_double2(so.x, so.y);
                                } else {
                                    // mirrors in different pairs; the equator is its own mirror
                                    const int q0 = nlat - 1 - p, q1 = nlat - 2 - p;
                                    auto row = [&](int q) {
                                        return *reinterpret_cast<const double2*>(g + size_t(q / 2) * ld + 2 * (q & 1));
                                    };
                                    if (q0 != p) x[r][2] = row(q0);
                                    if (q1 > p + 1) x[r][3] = row(q1);
                                }
                            }
                        }
                    }
                    if (!SYN && big) {
#pragma unroll
                        for (int r = 0; r < TR; ++r)
#pragma unroll
                            for (int e = 0; e < XV; ++e) x[r][e] = make_double2(0.5 * x[r][e].x, 0.5 * x[r][e].y);
                    }
                    // SYN: the words of a column (even lanes the real, odd lanes the imaginary part's);
                    // else (re, im) of latitude 2 w, then 2 w + 1
                    long long v[TR][XV];
                    int col[TR];
#pragma unroll
                    for (int r = 0; r < TR; ++r) {
                        const int task = r * 32 + lane;
                        if constexpr (!SYN) {
                            const int f = (task >> 3) % NF, h = (task >> 3) / NF;
                            col[r] = h * CP + 2 * f;
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                v[r][2 * e] = f64_to_fx(fma(sg[r], x[r][2 + e].x, x[r][e].x), kb[r]);
                                v[r][2 * e + 1] = f64_to_fx(fma(sg[r], x[r][2 + e].y, x[r][e].y), kb[r]);
                            }
                        } else {
                            const int f = (task >> 4) % NF, par = (task >> 4) / NF, odd = lane & 1;
                            const bool deg = f == 2 || f == 4;
                            col[r] = par * CP + 2 * f + odd;
                            // beta is scaled by 1 / s_m
                            const int k = 63 - s_eb[5 * i + f] - (f >= 3 && itm.x > 0);
                            const double c1 = f == 0 || deg ? cf[r].x : cf[r].y, c2 = cf[r].y;
                            const long long re = f64_to_fx(fma(c1, x[r][0].x, c2 * x[r][1].x), k);
                            const long long im = f64_to_fx(fma(c1, x[r][0].y, c2 * x[r][1].y), k);
                            const long long got = __shfl_xor_sync(0xffffffffu, odd ? re : im, 1);
                            v[r][0] = odd ? got : re;
                            v[r][1] = odd ? im : got;
                        }
                    }
                    if (it >= NS) mbar_wait(&b_empty[s], ((it / NS) - 1) & 1, abort, a.status);
#pragma unroll
                    for (int r = 0; r < TR; ++r)
                        if (r * 32 + lane < NT && !*abort) {
                            unsigned char* t = Bs + s * Q::BBYTES;
                            if constexpr (SYN) {
                                dig_put(t + dg_off(col[r], lane & 14), G * 32, v[r][0], v[r][1]);
                            } else {
                                const int w = lane & 7;
                                dig_put(t + dg_off(col[r], 2 * w), G * 32, v[r][0], v[r][2]);
                                dig_put(t + dg_off(col[r] + 1, 2 * w), G * 32, v[r][1], v[r][3]);
                            }
                        }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&b_full[s]);
                }
            }
    } else if (warp < 10 + NB) {
        // expanders: 32 rows of every digit from bytes to FP16 in tensor memory
        const int row = (warp & 3) * 32 + lane;
        const uint32_t lanes = uint32_t((warp & 3) * 32) << 16;
        DigRing rr, ra;
        for (int i = 0; i < nI; ++i) {
            const int4 itm = s_items[i];
            const int k1 = itm.z >> 16;
            for (int ks = itm.z & 0xFFFF; ks < k1; ++ks, rr.next(NR), ra.next(NX)) {
                // (a barrier still in its first phase passes for the one before)
                mbar_wait2(&r_full[rr.slot], rr.phase, &a_empty[ra.slot], ra.phase ^ 1, abort, a.status);
                tc_fence_after();
#pragma unroll
                for (int d0 = 0; d0 < DG_ND; d0 += 4) {
                    uint4 q[4];
#pragma unroll
                    for (int d = 0; d < 4; ++d)
                        q[d] = *reinterpret_cast<const uint4*>(Rs + rr.slot * DG_RBYTES + (d0 + d) * DG_RPLANE + row * 16);
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const uint32_t in[4] = {q[d].x, q[d].y, q[d].z, q[d].w};
                        uint32_t h[8];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            h[2 * e] = dg_half2(__byte_perm(in[e], 0x64646464u, 0x4140));
                            h[2 * e + 1] = dg_half2(__byte_perm(in[e], 0x64646464u, 0x4342));
                        }
                        tmem_st8_nowait(tmemA + lanes + uint32_t(ra.slot * DG_ACOLS + (d0 + d) * 8), h);
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&a_full[ra.slot]);
                    mbar_arrive(&r_empty[rr.slot]);
                }
            }
        }
    } else if constexpr (SYN) {
        // column exponents of every item: |b| <= 2^(eb - 1) from the exponents
        // of alpha and of the coefficient sets; NaN for a column that may hold a
        // number beyond the largest (see dig_shift; looking at the products here
        // cost 2.5 us at L = 511)
        pdl_wait();
        for (int i = 0; i < nI; ++i) {
            const int m = s_items[i].x, lo = m > 0 ? m : 1, pk = packed_off(N, m) - lo;
            int e[5] = {0, 0, 0, 0, 0}, top = 0;
#pragma unroll 8
            for (int K = lo + lane; K <= N; K += 32) {
                const short4 c = a.eoff[pk + K];
                const double2 x = a.alpha[pk + K];
                const int b = max(f64_bexp(x.x), f64_bexp(x.y));
                top = max(top, b);
                e[0] = max(e[0], b + c.x);
                e[1] = max(e[1], b + c.y);
                e[2] = max(e[2], b + c.z);
                if constexpr (NF == 5) {
                    const double2 y = a.beta[pk + K];
                    const int d = max(f64_bexp(y.x), f64_bexp(y.y));
                    top = max(top, d);
                    e[3] = max(e[3], d + c.y);
                    e[4] = max(e[4], d + c.z);
                }
            }
            top = __reduce_max_sync(0xffffffffu, top);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const int v = __reduce_max_sync(0xffffffffu, e[f]) - 2 * 1022 + 1;
                if (lane == 0) s_eb[5 * i + f] = top == 2047 || v > 1024 ? DG_NAN : v;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sc_full[i]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ---------------------------------------------------------------------------
// host side

// LPT over one CTA per SM, CTA lists at a fixed stride
static void dig_schedule(sphnse_plan* P, const std::vector<int4>& items, DigSide* D, std::vector<int4>& flat,
                         std::vector<int>& cnt) {
    std::vector<int> order(items.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = int(i);
    // an item costs its steps plus about one for its epilogue and start
    auto cost = [&](int i) { return (items[i].z >> 16) - (items[i].z & 0xFFFF) + 1; };
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost(x) > cost(y); });
    const int nc = std::min<int>(P->nsm, int(items.size()));
    std::vector<std::vector<int4>> bins(nc);
    std::vector<long> load(nc, 0);
    for (int idx : order) {
        const int b = int(std::min_element(load.begin(), load.end()) - load.begin());
        bins[b].push_back(items[idx]);
        load[b] += cost(idx);
    }
    D->ncta = nc;
    D->istride = 1;
    for (auto& b : bins) D->istride = std::max(D->istride, int(b.size()));
    flat.assign(size_t(nc) * D->istride, make_int4(0, 0, 0, 0));
    cnt.resize(nc);
    for (int c = 0; c < nc; ++c) {
        cnt[c] = int(bins[c].size());
        std::copy(bins[c].begin(), bins[c].end(), flat.begin() + size_t(c) * D->istride);
    }
}

void dig_free(sphnse_plan* P) {
    for (void* q : {static_cast<void*>(P->dig.syn.blocks), P->dig.arena, P->dig.sched})
        if (q) cudaFree(q);
    P->dig = DigState();
}

// parts of one device allocation, 256-byte aligned, with a host image
struct DigArena {
    std::vector<unsigned char> host;
    template <typename T>
    size_t add(const T* src, size_t n) {   // src null: zeros
        const size_t o = (host.size() + 255) / 256 * 256;
        host.resize(o + n * sizeof(T), 0);
        if (src && n) std::memcpy(host.data() + o, src, n * sizeof(T));
        return o;
    }
    int upload(void** d) const {
        if (cudaMalloc(d, host.size()) != cudaSuccess) return SPHNSE_E_NOMEM;
        return cudaMemcpy(*d, host.data(), host.size(), cudaMemcpyHostToDevice) == cudaSuccess ? SPHNSE_OK : SPHNSE_E_CUDA;
    }
};

// Digits, schedules and constants, from the FP64 table [n_ext][nh] on the
// device (which the digits replace).
int dig_setup(sphnse_plan* P, const double* d_tab) {
    const int N = P->N, nh = P->nh, ntile = (nh + 63) / 64;
    DigState& T = P->dig;
    // synthesis tiles (m, 64 latitudes), steps of 16 degrees of each parity
    std::vector<int> base(size_t(N + 1) * ntile);
    int nblk = 0;
    for (int m = 0; m <= N; ++m)
        for (int t = 0; t < ntile; ++t) {
            base[size_t(m) * ntile + t] = nblk;
            nblk += (ext_even(N, m) + 15) / 16;
        }
    // analysis tiles: four pieces of up to 32 rows of one (m, parity)
    std::vector<int4> pieces;
    for (int m = 0; m <= N; ++m)
        for (int par = 0; par < 2; ++par) {
            const int ne = ext_even(N, m), n = par ? ext_odd(N, m) : ne, r0 = ext_off(N, m) + (par ? ne : 0);
            for (int r = 0; r < n; r += 32) pieces.push_back(make_int4(m, par, r0 + r, std::min(32, n - r)));
        }
    while (pieces.size() % 4) pieces.push_back(make_int4(0, 0, 0, 0));
    const int atile = int(pieces.size() / 4), aks = (nh + 15) / 16, ablk = atile * aks;

    // exponents of the coefficient sets applied to alpha_{K,m}: zeta, theta, and the larger of
    // alpha_K's two places in the degree-shift set
    auto bexp = [](double v) { return v == 0.0 ? 0 : std::ilogb(v) + 1023; };
    auto eps = [](int l, int m) {
        return l <= m ? 0.0 : std::sqrt((double(l) * l - double(m) * m) / (4.0 * l * l - 1.0));
    };
    std::vector<short4> eoff(P->n_coeff);
    for (int m = 0, i = 0; m <= N; ++m)
        for (int l = (m > 0 ? m : 1); l <= N; ++l, ++i) {
            const double sl = std::sqrt(double(l) * (l + 1.0));
            // alpha_l enters row l + 1 with l eps_{l+1}, row l - 1 with (l + 1) eps_l; the sum of a
            // row's two terms takes one more bit; the sets of degree K are scaled by 2^dig_shift(N, K)
            const double dn = std::max(std::ldexp(l * eps(l + 1, m), dig_shift(N, l + 1)),
                                       std::ldexp((l + 1) * eps(l, m), dig_shift(N, l - 1))) / sl;
            const int t = dig_shift(N, l);
            eoff[i] = make_short4(short(bexp(sl) + t), short(bexp(1.0 / sl) + t), short(bexp(dn) + 1), 0);
        }
    DigArena A;
    const size_t o_eas = A.add<int>(nullptr, size_t(N + 1) * nh), o_eaa = A.add<int>(nullptr, P->n_ext);
    const size_t o_pc = A.add(pieces.data(), pieces.size()), o_base = A.add(base.data(), base.size());
    const size_t o_eoff = A.add(eoff.data(), eoff.size()), o_emax = A.add<int>(nullptr, size_t(3) * (N + 1));
    const size_t o_used = A.add<int>(nullptr, size_t(nblk) + ablk);
    int rc = A.upload(&T.arena);
    if (rc) return rc;
    unsigned char* d = static_cast<unsigned char*>(T.arena);
    T.syn.ea = reinterpret_cast<int*>(d + o_eas);
    T.ana.ea = reinterpret_cast<int*>(d + o_eaa);
    T.ana.pieces = reinterpret_cast<int4*>(d + o_pc);
    T.eoff = reinterpret_cast<short4*>(d + o_eoff);
    T.emax = reinterpret_cast<int*>(d + o_emax);
    const int* d_base = reinterpret_cast<const int*>(d + o_base);
    int* d_used = reinterpret_cast<int*>(d + o_used);
    T.syn.bytes = size_t(nblk) * DG_RBYTES;
    T.ana.bytes = size_t(ablk) * DG_RBYTES;
    if (cudaMalloc(reinterpret_cast<void**>(&T.syn.blocks), T.syn.bytes + T.ana.bytes) != cudaSuccess)
        return SPHNSE_E_NOMEM;
    T.ana.blocks = T.syn.blocks + T.syn.bytes;
    k_dig_syn_scale<<<dim3((nh + 127) / 128, N + 1), 128>>>(d_tab, T.syn.ea, N, nh);
    k_dig_ana_scale<<<(P->n_ext + 3) / 4, 128>>>(d_tab, T.ana.ea, P->n_ext, nh);
    k_dig_syn<<<dim3((ext_even(N, 0) + 15) / 16, ntile, N + 1), 256>>>(d_tab, T.syn.ea, d_base, T.syn.blocks, d_used, N,
                                                                      nh, ntile);
    k_dig_ana<<<dim3(aks, atile), 256>>>(d_tab, T.ana.ea, T.ana.pieces, T.ana.blocks, d_used + nblk, nh);
    std::vector<int> used(size_t(nblk) + ablk);
    if (cudaMemcpy(used.data(), d_used, used.size() * sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return SPHNSE_E_CUDA;
    // leading steps without a nonzero digit are skipped
    std::vector<int4> items;
    for (int m = 0; m <= N; ++m)
        for (int t = 0; t < ntile; ++t) {
            const int b = base[size_t(m) * ntile + t], k1 = (ext_even(N, m) + 15) / 16;
            int k0 = 0;
            while (k0 < k1 && !used[size_t(b) + k0]) ++k0;
            items.push_back(make_int4(m, t, k0 | (k1 << 16), b));
        }
    std::vector<int4> fs, fa;
    std::vector<int> cs, ca;
    dig_schedule(P, items, &T.syn, fs, cs);
    items.clear();
    for (int t = 0; t < atile; ++t) {
        int k0 = 0;
        while (k0 < aks && !used[size_t(nblk) + size_t(t) * aks + k0]) ++k0;
        items.push_back(make_int4(t, 0, k0 | (aks << 16), t * aks));
    }
    dig_schedule(P, items, &T.ana, fa, ca);
    DigArena Q;
    const size_t o_fs = Q.add(fs.data(), fs.size()), o_fa = Q.add(fa.data(), fa.size());
    const size_t o_cs = Q.add(cs.data(), cs.size()), o_ca = Q.add(ca.data(), ca.size());
    if ((rc = Q.upload(&T.sched))) return rc;
    d = static_cast<unsigned char*>(T.sched);
    T.syn.items = reinterpret_cast<int4*>(d + o_fs);
    T.ana.items = reinterpret_cast<int4*>(d + o_fa);
    T.syn.cnt = reinterpret_cast<int*>(d + o_cs);
    T.ana.cnt = reinterpret_cast<int*>(d + o_ca);
    return SPHNSE_OK;   // (ensure_tables waits for the copies)
}

static DigArgs dig_args(sphnse_plan* P, const DigSide& D) {
    DigArgs a{};
    a.blocks = D.blocks;
    a.items = D.items;
    a.cnt = D.cnt;
    a.istride = D.istride;
    // tables that fit L2 beside the grid fields stay there between calls (either
    // way 45.8 us for F at L = 150, 32 MB; kept at L = 200, 74 MB, F took 72.2 us
    // against 69.5, at L = 255, 120 MB, 85.8 against 81.1)
    a.evict_first = P->dig.syn.bytes + P->dig.ana.bytes > (size_t(48) << 20);
    a.ea = D.ea;
    a.status = P->d_status;
    a.N = P->N;
    a.nh = P->nh;
    a.nlat = P->nlat;
    a.alpha = nullptr;
    a.prepc = P->d_prepc;
    a.eoff = P->dig.eoff;
    a.gsyn = static_cast<double*>(P->d_gsyn);
    a.isin = P->d_isin;
    a.pieces = P->dig.ana.pieces;
    a.gana = static_cast<const double*>(P->d_gana);
    a.emax = P->dig.emax;
    a.hana = static_cast<double*>(P->d_hana);
    return a;
}

template <bool SYN, int NF>
static int dig_launch(sphnse_plan* P, const DigSide& D, const DigArgs& a) {
    using Q = DigShape<SYN, NF>;
    const size_t sm = Q::smem(D.istride);
    if (sm > 227 * 1024) return SPHNSE_E_UNSUPPORTED;
    allow_dynamic_smem(reinterpret_cast<const void*>(k_dig<SYN, NF>), sm);
    const int stage = SYN ? SPHNSE_STAGE_SYNTHESIS : SPHNSE_STAGE_ANALYSIS;
    stage_begin(P, stage);
    const cudaError_t e = launch_pdl(k_dig<SYN, NF>, dim3(D.ncta), dim3(32 * Q::WARPS), sm, P->stream, a);
    stage_end(P, stage);
    return check_cuda(e);
}

int launch_synthesis_dig(sphnse_plan* P, const double* alpha, const double* beta) {
    DigArgs a = dig_args(P, P->dig.syn);
    a.alpha = reinterpret_cast<const double2*>(alpha);
    a.beta = reinterpret_cast<const double2*>(beta);
    return beta ? dig_launch<true, 5>(P, P->dig.syn, a) : dig_launch<true, 3>(P, P->dig.syn, a);
}

void dig_clear_exponents(sphnse_plan* P) {
    cudaMemsetAsync(P->dig.emax, 0, size_t(3) * (P->N + 1) * sizeof(int), P->stream);
}

int launch_analysis_dig(sphnse_plan* P, int nf) {
    const DigArgs a = dig_args(P, P->dig.ana);
    return nf == 3 ? dig_launch<false, 3>(P, P->dig.ana, a) : dig_launch<false, 2>(P, P->dig.ana, a);
}

}  // namespace sph
