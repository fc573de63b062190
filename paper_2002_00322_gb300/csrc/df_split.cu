// Density-fitted exchange in FP64 on the sm_103a tensor cores, by the digit
// splitting of jk_split.cu:
//   Y_k[P][p][s] = sum_r B[P][p][r] D_k[r][s],   K_k[p][q] = sum_{P,s} Y_k[P][p][s] B[P][q][s]
// (GB300's FP64 pipe runs two FMA per clock and SM, so cuBLAS DGEMMs of the two
// products took 426 of the 430 ms of a 16-density build over 200 functions and
// 700 auxiliaries; the digit products take 28 times the multiply-adds at 800
// times the rate.)
//
// Every operand is a set of rows over a summed index.  A row has one power of
// two 2^e above its largest element and is kept as seven digits of base 512
// (63 bits), FP16 each, in tiles of 128 rows x 64 summed elements laid out as
//   [group of 8 summed elements][digit][row][8 elements]           (112 KB)
// which are K-major tensor-core operands for M = 128 rows as they lie, and whose
// 64-row halves are N operands.  B is symmetric in (p, r), so its tiles serve
// as the first operand of Y (rows p, for every P) and as the second of K (rows
// q); they are laid out once, at create.  The kernel of the first product
// writes Y as tiles for the second: |Y| <= max_P |B_P[p]|_2 max_s |D_k[:, s]|_2
// bounds the rows, so no pass over Y is needed to find their exponents.
//
// k_df_gemm forms tiles of 128 x 64 outputs.  For each block of 64 summed
// elements the digit products with i + j = t < 7 are summed in FP32 tensor
// memory (7 x 64 columns), read and added to two 64-bit integers per output in
// registers, SH for t < 3 and SL for the rest: a product is
// 2^(e_a + e_b - 70) (2^36 SH + SL).  The sums of a block are exact for t <= 3 (at
// most 4 * 64 terms of 2^16, below 2^24 or equal); those of t >= 4 are too unless
// their digits line up (up to 7 * 64 terms of 2^16), and an addition above 2^24
// then rounds by 1, 2^-52 of the rows' largest product.  A block adds at most
// 2^51 + 2^43 to SL, so the integers hold 2048 blocks, and no CTA sums more
// (df_ranges).  The digit pairs left out weigh 2^-63 of that product each.  A row
// spans all auxiliaries, whose elements differ by decades: with six digits and
// t < 6 the error of K against 64-bit references was 5e-13 over 200 functions
// (DGEMM 3.9e-14).  The bound is normwise: an element of B 2^-k of its row's
// largest over all auxiliaries keeps 63 - k bits, one of D likewise in its column,
// and Y is rounded to 2^-62 of its bound, which all columns share.
//
// Digits serve densities whose largest element lies in [2^-500, 2^500), where
// the squares behind the bound on Y stay in FP64's range; plain_row takes the
// others (and those with infinities or NaN) in FP64 arithmetic.  The factor's
// elements are at most 2^250 (the handle keeps to cuBLAS otherwise).
//
// What bounds it: the MMAs (3.6K cycles per block of full size) and the
// tensor-memory reads after each block (448 of the 512 columns are one
// accumulator, so they do not overlap): at 120 functions the tensor pipe is busy 32
// and 41 % of the two products, the ALU 41 and 16 %.  Sixteen warps read, a quarter of the
// columns each (c_0 past the conversion unit): 200 functions, 700 auxiliaries, 16
// densities 26.1 -> 23.7 ms against eight.
//
// Warp roles (576 threads, one CTA per SM): warp 0 producer (bulk copies into
// five stages of 16 summed elements), warp 1 MMA issuer, warps 2-17 epilogue.
#include "esmf_internal.cuh"
#include "split.cuh"
#include "umma.cuh"

namespace esmf {

using namespace split;
using namespace umma;

namespace {

constexpr int ND = 7, NT = 7;                 // digits per operand, column groups t = i + j
constexpr int BITS = 9 * ND - 1;              // |fixed-point value| <= 2^BITS
constexpr int GROUP = ND * 128 * 16;          // 8 summed elements of a tile, all digits: 14 KB
constexpr int TILE = 8 * GROUP;               // 112 KB
constexpr int STAGES = 5;
constexpr int A_STAGE = 2 * GROUP, B_STAGE = 2 * ND * 64 * 16;
constexpr int OFF_CTRL = STAGES * (A_STAGE + B_STAGE);
constexpr int DF_SMEM = OFF_CTRL + 1024;
constexpr int EPI_WARPS = 16;
constexpr int DF_THREADS = 64 + 32 * EPI_WARPS;
constexpr int EMIN = 1022 - 600;              // smallest exponent field of a row
constexpr int BMAX = 250;                     // largest exponent of the factor
constexpr unsigned long long SL_MASK = (1ull << 36) - 1;   // SL below 2^36 SH
constexpr int MAX_BLOCKS = 2048;              // blocks of 64 summed elements that SL and SH hold

struct DfCtrl {
    uint64_t full[STAGES], empty[STAGES], accfull, accfree;
    uint32_t tmem_base;
    int abort_flag, never;
};
static_assert(sizeof(DfCtrl) <= 1024 && DF_SMEM <= 227 * 1024, "shared memory");

// 32 lanes x 32-bit, 4 consecutive columns per thread
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float *v) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// exponent field of x: |x| < 2^(field - 1022)
__device__ __forceinline__ int exp_field(double x) { return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7ffu); }

// digits of eight fixed-point values as the eight-element pieces of a tile's
// group: digit i at dst + i * 2048 (dst addresses the row)
__device__ __forceinline__ void store_digits(unsigned char *dst, const long long *X) {
    uint32_t w[8][3];
#pragma unroll
    for (int j = 0; j < 8; ++j) digit_words<ND>(X[j], w[j]);
    auto put = [&](int i, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
        *reinterpret_cast<uint4 *>(dst + i * 2048) = make_uint4(a, b, c, d);
    };
    put(0, digit_pair<0>(w[0], w[1]), digit_pair<0>(w[2], w[3]), digit_pair<0>(w[4], w[5]), digit_pair<0>(w[6], w[7]));
    put(1, digit_pair<1>(w[0], w[1]), digit_pair<1>(w[2], w[3]), digit_pair<1>(w[4], w[5]), digit_pair<1>(w[6], w[7]));
    put(2, digit_pair<2>(w[0], w[1]), digit_pair<2>(w[2], w[3]), digit_pair<2>(w[4], w[5]), digit_pair<2>(w[6], w[7]));
    put(3, digit_pair<3>(w[0], w[1]), digit_pair<3>(w[2], w[3]), digit_pair<3>(w[4], w[5]), digit_pair<3>(w[6], w[7]));
    put(4, digit_pair<4>(w[0], w[1]), digit_pair<4>(w[2], w[3]), digit_pair<4>(w[4], w[5]), digit_pair<4>(w[6], w[7]));
    put(5, digit_pair<5>(w[0], w[1]), digit_pair<5>(w[2], w[3]), digit_pair<5>(w[4], w[5]), digit_pair<5>(w[6], w[7]));
    put(6, digit_pair<6>(w[0], w[1]), digit_pair<6>(w[2], w[3]), digit_pair<6>(w[4], w[5]), digit_pair<6>(w[6], w[7]));
}

}  // namespace

// ---------------------------------------------------------------- operands
// eB[p]: exponent of max over P, r of |B[P][p][r]|; nB[p]: exponent above
// max_P |B_P[p]|_2 (one more, for the rounding of the norm).  Rows so small that
// the squares leave FP64's range: |B_P[p]|_2 <= sqrt(n) max |B_P[p][r]|, n < 2^18.
// One block per p.
__global__ void __launch_bounds__(256) k_df_brows(const double *B, int naux, int n, int16_t *eB, int16_t *nB) {
    __shared__ double red[8];
    __shared__ int rede[8];
    const int p = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double top = 0.0;
    int e = EMIN;
    for (int P = w; P < naux; P += 8) {
        const double *row = B + ((int64_t)P * n + p) * n;
        double s = 0.0;
        for (int r = lane; r < n; r += 32) {
            s = fma(row[r], row[r], s);
            e = max(e, exp_field(row[r]));
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        top = fmax(top, s);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) { red[w] = top; rede[w] = e; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) { top = fmax(top, red[i]); e = max(e, rede[i]); }
        eB[p] = (int16_t)(e - 1022);
        nB[p] = (int16_t)(e < 1022 + DMIN ? e - 1022 + 10 : exp_field(sqrt(top)) - 1022 + 1);
    }
}

// digit tiles of B: [P][128 rows p][64 r] (zero beyond n); one thread per
// (P, p, group of 8 r)
__global__ void k_df_btiles(const double *B, int naux, int n, int npb, int nkb, const int16_t *eB, unsigned char *tiles) {
    const int64_t total = (int64_t)naux * npb * nkb * 8 * 128;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(t & 127), g = (int)(t >> 7 & 7);
        const int64_t tile = t >> 10;
        const int kb = (int)(tile % nkb), pb = (int)(tile / nkb % npb);
        const int64_t P = tile / nkb / npb;
        const int p = pb * 128 + row, r0 = kb * 64 + g * 8;
        long long X[8];
        const int e = p < n ? eB[p] + 1022 : EMIN;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const double v = (p < n && r0 + j < n) ? B[(P * n + p) * n + r0 + j] : 0.0;
            X[j] = fixed_point<BITS>((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), e);
        }
        store_digits(tiles + tile * TILE + g * GROUP + row * 16, X);
    }
}

// Per density k and column s: exponent eD[k * ldD + s] of max_r |D_k[r][s]|;
// per density the exponent above max_s |D_k[:, s]|_2 in ED[k] (any smaller value
// at launch; the column of the largest element has a norm in range and bounds the
// columns whose squares underflow) and the exponent field of its largest element
// in top[k] (below 0 at launch; subnormal elements count as 1).
__global__ void k_df_dcols(const double *D, int n, int ldD, int16_t *eD, int *ED, int *top) {
    const int k = blockIdx.y, s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= ldD) return;
    int e = 0;
    double q = 0.0;
    if (s < n)
        for (int r = 0; r < n; ++r) {
            const double v = D[((int64_t)k * n + r) * n + s];
            q = fma(v, v, q);
            e = max(e, field_of(v));
        }
    eD[(int64_t)k * ldD + s] = (int16_t)(max(e, EMIN) - 1022);
    if (e == 0) return;
    atomicMax(top + k, e);
    atomicMax(ED + k, exp_field(sqrt(q)) - 1022 + 1);
}

// digit tiles of the densities, rows s over r: [k][128 rows s][64 r]
__global__ void k_df_dtiles(const double *D, int n, int m, int npb, int nkb, int ldD, const int16_t *eD, unsigned char *tiles) {
    const int64_t total = (int64_t)m * npb * nkb * 8 * 128;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(t & 127), g = (int)(t >> 7 & 7);
        const int64_t tile = t >> 10;
        const int kb = (int)(tile % nkb), sb = (int)(tile / nkb % npb);
        const int64_t k = tile / nkb / npb;
        const int s = sb * 128 + row, r0 = kb * 64 + g * 8;
        long long X[8];
        const int e = s < n ? min(eD[k * ldD + s] + 1022, 1022 + DMAX) : EMIN;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const double v = (s < n && r0 + j < n) ? D[(k * n + r0 + j) * n + s] : 0.0;
            X[j] = exp_field(v) > e ? 0 : fixed_point<BITS>((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v), e);
        }
        store_digits(tiles + tile * TILE + g * GROUP + row * 16, X);
    }
}

// ---------------------------------------------------------------- products
struct DfGemm {
    const unsigned char *A, *B;    // digit tiles of the two operands
    unsigned char *Y;              // first product: tiles of Y out
    unsigned long long *S;         // second product: SH, then SL, n x n per density of the group, added to
    const int16_t *eB, *nB, *eD;
    const int *ED, *top;
    int n, naux, npb, nkb, nsb;    // nsb: blocks of 64 output columns
    int k0, kc, splits, ldD;
    int64_t items;
    int *error;
};

// SECOND = false: Y (item: P, 128 p, density, 64 s); true: K (item: range of the
// blocks (P, 64 s), density, 128 p, 64 q)
template <bool SECOND>
__global__ void __launch_bounds__(DF_THREADS, 1) k_df_gemm(const __grid_constant__ DfGemm G) {
    extern __shared__ __align__(1024) unsigned char sm[];
    DfCtrl &c = *reinterpret_cast<DfCtrl *>(sm + OFF_CTRL);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int *abort_flag = &c.abort_flag;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&c.full[s], 1);
            mbar_init(&c.empty[s], 1);
        }
        mbar_init(&c.accfull, 1);
        mbar_init(&c.accfree, EPI_WARPS);
        c.abort_flag = 0;
        c.never = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(&c.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    auto fail = [&](int code) {
        *abort_flag = 1;
        if (G.error) atomicExch(G.error, code);
    };
    // an item: its tiles' base indices, output column block and blocks of 64
    struct Item {
        int64_t a, b;              // tile index of block 0 (first product), or of block (0, 0)
        int k, pb, ob;             // density of the group, 128 rows, 64 columns
        int64_t P;
        int64_t j0, j1;            // blocks
    };
    auto item_of = [&](int64_t it) {
        Item x;
        if (!SECOND) {
            x.ob = (int)(it % G.nsb); it /= G.nsb;
            x.k = (int)(it % G.kc); it /= G.kc;
            x.pb = (int)(it % G.npb);
            x.P = it / G.npb;
            x.a = (x.P * G.npb + x.pb) * G.nkb;
            x.b = ((int64_t)(G.k0 + x.k) * G.npb + (x.ob >> 1)) * G.nkb;
            x.j0 = 0; x.j1 = G.nkb;
        } else {
            x.ob = (int)(it % G.nsb); it /= G.nsb;
            x.pb = (int)(it % G.npb); it /= G.npb;
            x.k = (int)(it % G.kc);
            const int64_t sp = it / G.kc, blocks = (int64_t)G.naux * G.nkb;
            x.P = 0; x.a = 0; x.b = 0;
            x.j0 = blocks * sp / G.splits; x.j1 = blocks * (sp + 1) / G.splits;
        }
        return x;
    };
    // tiles of block j, its steps of 16 summed elements
    auto tiles_of = [&](const Item &x, int64_t j, int64_t &ta, int64_t &tb, int &ks) {
        int kb;
        if (!SECOND) {
            kb = (int)j;
            ta = x.a + j;
            tb = x.b + j;
        } else {
            const int64_t P = j / G.nkb;
            kb = (int)(j - P * G.nkb);
            ta = (((int64_t)x.k * G.naux + P) * G.npb + x.pb) * G.nkb + kb;
            tb = (P * G.npb + (x.ob >> 1)) * G.nkb + kb;
        }
        ks = min(4, (G.n - kb * 64 + 15) / 16);
    };
    // columns of an output block, padded to 16
    auto width = [&](int ob) { return min(64, (G.n - ob * 64 + 15) / 16 * 16); };

    if (warp == 0) {
        // ------------------------------------------------ producer
        int st = 0;
        bool ok = true;
        for (int64_t it = blockIdx.x; ok && it < G.items; it += gridDim.x) {
            const Item x = item_of(it);
            const int W = width(x.ob), half = x.ob & 1;
            for (int64_t j = x.j0; ok && j < x.j1; ++j) {
                int64_t ta, tb;
                int ks;
                tiles_of(x, j, ta, tb, ks);
                for (int h = 0; h < ks; ++h, ++st) {
                    const int s = st % STAGES;
                    if (st >= STAGES && !__all_sync(~0u, wait_for(&c.empty[s], (st / STAGES - 1) & 1, abort_flag))) { fail(41); ok = false; break; }
                    unsigned char *dst = sm + s * (A_STAGE + B_STAGE);
                    if (lane == 0) mbar_arrive_expect_tx(&c.full[s], 2 * (GROUP + ND * W * 16));
                    __syncwarp();
                    if (lane == 31) bulk_g2s(dst, G.A + ta * TILE + h * 2 * GROUP, 2 * GROUP, &c.full[s]);
                    if (lane < 2 * ND)
                        bulk_g2s(dst + A_STAGE + lane * W * 16, G.B + tb * TILE + h * 2 * GROUP + lane * 2048 + half * 1024, W * 16,
                                 &c.full[s]);
                }
            }
        }
        // no copy may still be landing when the CTA leaves
        for (int k = st > STAGES ? st - STAGES : 0; k < st; ++k) wait_for(&c.full[k % STAGES], (k / STAGES) & 1, &c.never);
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        const uint32_t lead = elect_one() ? 1u : 0u, sbase = smem_u32(sm);
        int st = 0, blk = 0;
        bool ok = true;
        for (int64_t it = blockIdx.x; ok && it < G.items; it += gridDim.x) {
            const Item x = item_of(it);
            const uint32_t W = uniform(width(x.ob));
            const uint32_t first = uniform(256u / W < (uint32_t)ND ? 256u / W : (uint32_t)ND);   // digits of one MMA
            const uint32_t id = uniform(idesc_f16(128, 0, 0, 0)), wid = uniform((W >> 3) << 17);
            for (int64_t j = x.j0; ok && j < x.j1; ++j, ++blk) {
                int64_t ta, tb;
                int ks;
                tiles_of(x, j, ta, tb, ks);
                if (blk >= 1 && !__all_sync(~0u, wait_for(&c.accfree, (blk - 1) & 1, abort_flag))) { fail(42); ok = false; break; }
                for (int h = 0; h < ks; ++h, ++st) {
                    const int s = st % STAGES;
                    if (!__all_sync(~0u, wait_for(&c.full[s], (st / STAGES) & 1, abort_flag))) { fail(43); ok = false; break; }
                    tc_fence_after();
                    const uint32_t dst = sbase + s * (A_STAGE + B_STAGE);
                    const uint64_t a0 = sdesc(dst, GROUP, 128), b0 = sdesc(dst + A_STAGE, ND * W * 16, 128);
                    const uint32_t ahi = uniform((uint32_t)(a0 >> 32)), bhi = uniform((uint32_t)(b0 >> 32));
                    const uint32_t a = uniform((uint32_t)a0), b = uniform((uint32_t)b0);
#pragma unroll
                    for (int i = 0; i < ND; ++i) {
                        // digit i of A against the digits 0 .. 6-i of B, into the columns of t = i ..
                        const uint32_t acc = (i > 0 || h > 0) ? 1u : 0u;
                        const uint32_t nj = NT - i, n1 = nj < first ? nj : first;
                        mma_pred(lead, tmem + i * W, a + i * 128, ahi, b, bhi, id + n1 * wid, acc);
                        if (n1 < nj)
                            mma_pred(lead, tmem + (i + n1) * W, a + i * 128, ahi, b + n1 * W, bhi, id + (nj - n1) * wid, acc);
                    }
                    if (lead) {
                        mma_commit(&c.empty[s]);
                        if (h + 1 == ks) mma_commit(&c.accfull);
                    }
                    __syncwarp();
                }
            }
        }
        // MMAs in flight must end before tensor memory is released
        if (blk > 0) wait_for(&c.accfull, (blk - 1) & 1, &c.never);
    } else {
        // ------------------------------------------------ epilogue
        const int quarter = warp & 3, ch = (warp - 2) >> 2;       // lane quarter, every fourth group of 8 columns
        const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16);
        const int row = quarter * 32 + lane;
        int blk = 0;
        bool ok = true;
        for (int64_t it = blockIdx.x; ok && it < G.items; it += gridDim.x) {
            const Item x = item_of(it);
            const int W = width(x.ob), p = x.pb * 128 + row;
            const int groups = (W / 8 - ch + 3) / 4;              // groups ch and ch + 4 as far as the block has them
            long long SH[2][8], SL[2][8];
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
                for (int i = 0; i < 8; ++i) SH[g][i] = SL[g][i] = 0;
            const int ap = p < G.n ? G.eB[p] : 0;
            const int yp = p < G.n ? G.nB[p] + G.ED[G.k0 + x.k] : 4096;
            for (int64_t j = x.j0; j < x.j1; ++j, ++blk) {
                if (!__all_sync(~0u, wait_for(&c.accfull, blk & 1, abort_flag))) { fail(44); ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    if (g < groups) {
#pragma unroll
                        for (int i0 = 0; i0 < 8; i0 += 4) {
                            float v[NT][4];
#pragma unroll
                            for (int t = 0; t < NT; ++t) tmem_ld4(tl + t * W + (ch + 4 * g) * 8 + i0, v[t]);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                // |c_0| <= 2^22: through the bits of c_0 + 1.5 2^23, off the conversion unit
                                auto ci = [&](int t) { return (long long)__float2int_rn(v[t][i]); };
                                const long long z0 = (int)(__float_as_uint(__fadd_rn(v[0][i], 12582912.f)) - 0x4b400000u);
                                SH[g][i0 + i] += z0 * (1 << 18) + ci(1) * 512 + ci(2);
                                SL[g][i0 + i] += ci(3) * (1 << 27) + ci(4) * (1 << 18) + ci(5) * 512 + ci(6);
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.accfree);
            }
            if (SECOND && ok) {
#pragma unroll
                for (int g = 0; g < 2; ++g)
                    if (g < groups)
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const int q = x.ob * 64 + (ch + 4 * g) * 8 + i;
                            if (p < G.n && q < G.n) {
                                // the ranges' sums join as integers: any order gives the same bits
                                unsigned long long *o = G.S + ((int64_t)x.k * G.n + p) * G.n + q;
                                atomicAdd(o, (unsigned long long)(SH[g][i] + (SL[g][i] >> 36)));
                                atomicAdd(o + (int64_t)G.kc * G.n * G.n, (unsigned long long)SL[g][i] & SL_MASK);
                            }
                        }
            }
            if (!SECOND && ok) {
                // Y = 2^(ap + eD - 70) (2^36 SH + SL) as a fixed-point value of its row's exponent yp
                unsigned char *out = G.Y + ((((int64_t)x.k * G.naux + x.P) * G.npb + x.pb) * G.nkb + x.ob) * TILE +
                                     ch * GROUP + row * 16;
                const int16_t *ed = G.eD + (int64_t)(G.k0 + x.k) * G.ldD + x.ob * 64 + ch * 8;
#pragma unroll
                for (int g = 0; g < 2; ++g)
                    if (g < groups) {
                        long long X[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            // right shift: nB > eB and ED > eD make it 10 at least (rows beyond n and
                            // densities that plain_row takes get zeros)
                            const int r = yp - ap - ed[g * 32 + i] + 70 - BITS;
                            const __int128 S = ((__int128)SH[g][i] << 36) + SL[g][i];
                            X[i] = r > 100 || r < 1 ? 0 : (long long)((S + ((__int128)1 << (r - 1))) >> r);
                        }
                        store_digits(out + 4 * g * GROUP, X);
                    }
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Row p of K of a density beyond the digits' range, in FP64 arithmetic:
// y[s] = sum_r B[P][p][r] D[r][s] for a piece of s at a time, then K[p][q] += sum_s
// y[s] B[P][s][q] (B is symmetric; both sums read whole rows).  200 functions, 700
// auxiliaries: 41 ms a density (the two cuBLAS products took 27 ms).
__device__ void plain_row(const double *B, const double *Dk, int n, int naux, int p, double *Kp) {
    constexpr int PIECE = 1024;
    __shared__ double y[PIECE];
    for (int q = threadIdx.x; q < n; q += blockDim.x) Kp[q] = 0.0;
    for (int P = 0; P < naux; ++P) {
        const double *BP = B + (int64_t)P * n * n, *bp = BP + (int64_t)p * n;
        for (int s0 = 0; s0 < n; s0 += PIECE) {
            const int len = min(PIECE, n - s0);
            __syncthreads();
            for (int s = threadIdx.x; s < len; s += blockDim.x) {
                double a = 0.0;
                for (int r = 0; r < n; ++r) a = fma(bp[r], Dk[(int64_t)r * n + s0 + s], a);
                y[s] = a;
            }
            __syncthreads();
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                double a = Kp[q];
                for (int s = 0; s < len; ++s) a = fma(y[s], BP[(int64_t)(s0 + s) * n + q], a);
                Kp[q] = a;
            }
        }
    }
}

// K of a group's densities, one block per row: from their integer sums (each range
// adds less than 2^36 to SL, and 2^18 blocks, more than the device has room for,
// 2^59 to SH), or by plain_row.
__global__ void __launch_bounds__(256) k_df_kout(const __grid_constant__ DfGemm G, const double *B, const double *D, double *K) {
    const int p = blockIdx.x, k = G.k0 + blockIdx.y;
    const int64_t nn = (int64_t)G.n * G.n;
    double *Kp = K + k * nn + (int64_t)p * G.n;
    if (G.top[k] > 0 && beyond_digits(G.top[k])) {
        plain_row(B, D + k * nn, G.n, G.naux, p, Kp);
        return;
    }
    const unsigned long long *row = G.S + blockIdx.y * nn + (int64_t)p * G.n;
    const int e = G.nB[p] + G.ED[k] - 70;
    for (int q = threadIdx.x; q < G.n; q += blockDim.x) {
        const unsigned long long lo = row[q + G.kc * nn];
        const long long hi = (long long)(row[q] + (lo >> 36));
        Kp[q] = scalbn(fma((double)hi, 0x1p36, (double)(lo & SL_MASK)), e + G.eB[q]);
    }
}

// ---------------------------------------------------------------- host side
namespace {

#define CKS(call)                                                                  \
    do {                                                                           \
        cudaError_t e_ = (call);                                                   \
        if (e_ != cudaSuccess) {                                                   \
            set_error("%s: %s", #call, cudaGetErrorString(e_));                    \
            return ESMF_ERR_CUDA;                                                  \
        }                                                                          \
    } while (0)

int row_blocks(int n) { return (n + 127) / 128; }
int sum_blocks(int n) { return (n + 63) / 64; }
int grid_for(int64_t work) {
    const int64_t g = (work + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

// Ranges that the naux * sum_blocks(n) summed blocks of the second product are
// cut into: about four items per SM, 4 blocks or more each, never above MAX_BLOCKS.
int df_ranges(int n, int naux, int kc, int num_sms) {
    const int64_t tiles = (int64_t)kc * row_blocks(n) * sum_blocks(n), blocks = (int64_t)naux * sum_blocks(n);
    int64_t sp = (4 * num_sms + tiles - 1) / tiles;
    if (sp > blocks / 4) sp = blocks / 4;
    const int64_t least = (blocks + MAX_BLOCKS - 1) / MAX_BLOCKS;
    return (int)(sp < least ? least : sp);
}

template <bool SECOND>
int df_gemm(const DfGemm &g, int num_sms, cudaStream_t s) {
    CKS(cudaFuncSetAttribute(k_df_gemm<SECOND>, cudaFuncAttributeMaxDynamicSharedMemorySize, DF_SMEM));
    k_df_gemm<SECOND><<<(int)(g.items < num_sms ? g.items : num_sms), DF_THREADS, DF_SMEM, s>>>(g);
    CKS(cudaGetLastError());
    return ESMF_OK;
}

}  // namespace

// df_ranges for the tests
extern "C" int esmf_df_exchange_ranges(int n, int naux, int kc, int num_sms) { return df_ranges(n, naux, kc, num_sms); }

size_t df_split_tile_bytes(int n, int64_t matrices) { return (size_t)matrices * row_blocks(n) * sum_blocks(n) * TILE; }

size_t df_split_sum_bytes(int n, int group) { return (size_t)group * n * n * 2 * sizeof(unsigned long long); }

int launch_df_split_rows(const double *B, int naux, int n, int16_t *eB, int16_t *nB, cudaStream_t s) {
    k_df_brows<<<n, 256, 0, s>>>(B, naux, n, eB, nB);
    CKS(cudaGetLastError());
    return ESMF_OK;
}

bool df_split_rows_fit(int n, const int16_t *eB) {
    int top = EMIN - 1022;
    for (int p = 0; p < n; ++p) top = eB[p] > top ? eB[p] : top;
    return top >= -BMAX && top <= BMAX && sum_blocks(n) <= MAX_BLOCKS;
}

int launch_df_split_factor(const double *B, int naux, int n, const int16_t *eB, unsigned char *tiles, cudaStream_t s) {
    const int npb = row_blocks(n), nkb = sum_blocks(n);
    k_df_btiles<<<grid_for((int64_t)naux * npb * nkb * 1024), 256, 0, s>>>(B, naux, n, npb, nkb, eB, tiles);
    CKS(cudaGetLastError());
    return ESMF_OK;
}

int launch_df_split_exchange(const DfSplit &a, cudaStream_t s) {
    const int n = a.n, npb = row_blocks(n), nkb = sum_blocks(n), ldD = nkb * 64;
    CKS(cudaMemsetAsync(a.ED, 0x80, sizeof(int) * 2 * a.m, s));       // top follows
    k_df_dcols<<<dim3((ldD + 63) / 64, a.m), 64, 0, s>>>(a.D, n, ldD, a.eD, a.ED, a.top);
    CKS(cudaGetLastError());
    k_df_dtiles<<<grid_for((int64_t)a.m * npb * nkb * 1024), 256, 0, s>>>(a.D, n, a.m, npb, nkb, ldD, a.eD, a.Dtiles);
    CKS(cudaGetLastError());
    for (int k0 = 0; k0 < a.m; k0 += a.group) {
        DfGemm g;
        g.eB = a.eB; g.nB = a.nB; g.eD = a.eD; g.ED = a.ED; g.top = a.top;
        g.n = n; g.naux = a.naux; g.npb = npb; g.nkb = nkb; g.nsb = nkb; g.ldD = ldD;
        g.k0 = k0; g.kc = a.m - k0 < a.group ? a.m - k0 : a.group;
        g.Y = a.Ytiles; g.S = a.S; g.error = a.error;
        g.A = a.Btiles; g.B = a.Dtiles; g.splits = 1;
        g.items = (int64_t)a.naux * npb * g.kc * nkb;
        int rc = df_gemm<false>(g, a.num_sms, s);
        if (rc != ESMF_OK) return rc;
        g.splits = df_ranges(n, a.naux, g.kc, a.num_sms);
        g.A = a.Ytiles; g.B = a.Btiles;
        g.items = (int64_t)g.kc * npb * nkb * g.splits;
        CKS(cudaMemsetAsync(a.S, 0, df_split_sum_bytes(n, g.kc), s));
        rc = df_gemm<true>(g, a.num_sms, s);
        if (rc != ESMF_OK) return rc;
        k_df_kout<<<dim3(n, g.kc), n <= 128 ? 128 : 256, 0, s>>>(g, a.B, a.D, a.K);
        CKS(cudaGetLastError());
    }
    return ESMF_OK;
}

}  // namespace esmf
