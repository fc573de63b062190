// FP64 grouped J/K contraction on the sm_103a tensor cores (tcgen05) for FP64 and
// double-FP32 integral stores: every operand is rounded to a fixed-point number
// relative to its block's largest element, whose digits the FP16 tensor pipe
// multiplies and sums exactly (the splitting of Ozaki, Ogita, Oishi and Rump 2012,
// in its fixed-point form).
//
// A brick (P Q | R S) feeds the six GEMM views of jk_umma.cu (64 output rows,
// 64 terms, all densities as columns).  With one power of two 2^eV per brick
// and one 2^eD per density and 8 x 8 density block,
//   V = 2^(eV-8) sum_i x_i 2^(-9 i), i < 7,   D = 2^(eD-8) sum_j y_j 2^(-9 j), j < 6
// where the digits x_i, y_j are integers in [-256, 256], exact in FP16: 63 bits
// below the brick's largest integral, 54 below the block's largest density.  The
// integrals have a digit more because a brick's span decades while a block's
// densities mostly do not (with six digits K of 24 functions was further from
// 64-bit references than FP64 arithmetic's, 7.0e-16 against 5.2e-16).  Then
//   V . D = 2^(eV+eD-16) sum_t 2^(-9 t) c_t,   c_t = sum_{i+j=t} x_i . y_j
// and each c_t is an integer that FP32 accumulation in tensor memory holds
// exactly: 64 terms of at most 2^16 per digit pair, below 2^24 for t <= 3; a
// last place rounded in a later t weighs less than 2^-51 of the largest
// product.  All digit pairs with t <= 6 are formed; the others are below 2^-60
// of the largest product.
//
// Accuracy: with Vb the largest integral of a brick and Db the largest density of
// an 8 x 8 block, each product V D of a sum is off by at most 2^-53 |V| Db +
// 2^-58 Vb Db, and every brick sum is rounded once.  In the norm of J or K that is
// less than FP64 arithmetic's rounding: against 113-bit sums, means over eight
// molecules of 24 functions, J 4.1e-16 and K 3.8e-16 (k_jk_cuda<double> 5.1e-16 and
// 4.6e-16), three of 40 functions 3.7e-16 and 3.9e-16 (4.4e-16 and 4.7e-16).  Single
// outputs that only products far below Vb Db feed keep fewer digits than there: J of
// functions that hardly overlap (products below 2^-58) none.  (Scaling the Coulomb operands by the
// Schwarz bounds kept those, but digits of their own for W cost 16 % of a build of
// 200 functions and raised the error of J in the norm to 5.4e-16.)
//
// MMA N covers the digits: with the density digits of a block as consecutive
// operand rows [y_0 | y_1 | ...], the digit x_i multiplies a run of them at
// once into the columns of t = i, i+1, ... (one MMA per 16 terms and digit of
// V instead of one per digit pair).
//
// What bounds it: at 16 densities the MMAs of a brick take 8.8K cycles of the
// tensor pipe (M = 64 runs at 2,048 MAC per clock) and fetch 940 KB of operands
// from shared memory (7.3K cycles at 128 B per clock) beside 350 KB of other
// traffic there; the CUDA-core FP64 form of the same brick takes 327K cycles
// (GB300 has two FP64 FMA per clock and SM).  200 functions, 16 densities, 53K
// bricks: 54.7 ms with k_jk_cuda<double>, 2.78 ms here (15.4K cycles a brick).
// Recombining into one 62-bit integer per output was faster (2.62 ms against
// 3.02 when that was tried), but rounds every output at 2^-56 of the brick's
// largest product, also one a thousand times smaller, where FP64 arithmetic
// would not.
//
// Warp roles (832 threads, 576 at 8 densities; one CTA per SM): warp 0 producer
// (bulk copies of the packed record one brick ahead and of one density tile per
// view through a two-slot ring), warp 1 tensor-memory owner and MMA issuer, warps 2-9
// converters (packed record -> digits in registers -> tiles V and, with r and q
// swapped, W, which the Coulomb views read), the others epilogue in two groups
// that take the views alternately: tensor-memory load, integer
// recombination of the c_t, one FP64 reduction per output.  V
// and W are single tiles (shared memory holds no second pair): the digits of
// the next brick wait in registers, V is written while the Coulomb MMAs (over
// W) run, W while the exchange MMAs (over V) run.  The D^T outputs go to an
// accumulator of their own in the same orientation as the D outputs, so that
// every reduction of a warp covers 2 x 16 consecutive values; the finalisation
// adds its transpose.
//
// Digits serve densities whose largest element lies in [2^-500, 2^500).  A pass
// with another one (k_split_dbank finds the largest exponents), infinities and NaN
// among them, runs a plain FP64 loop over the same bricks (200 functions, 16
// densities: 79 ms; 54.6 ms with k_jk_cuda<double>).
#include <cuda_fp16.h>

#include "esmf_internal.cuh"
#include "split.cuh"
#include "umma.cuh"

namespace esmf {

using namespace split;
using namespace umma;

namespace {

constexpr int NV = 7, ND = 6;                     // digits of an integral, of a density
constexpr int NT = 7;                             // column groups t = i + j
constexpr int SLICE = 8192;                       // one digit of a brick, 4096 x FP16
constexpr int REC_BYTES = MASK_BYTES + 8 * BRICK; // keep mask + packed values
constexpr int MPM = 16;                           // densities per pass
constexpr int RING_SLOT = ND * 2 * MPM * 128;     // largest density tile (exchange)
constexpr int OFF_V = 0, OFF_W = NV * SLICE, OFF_REC = 2 * NV * SLICE;
constexpr int OFF_RING = OFF_REC + 2 * REC_BYTES;
constexpr int OFF_CTRL = OFF_RING + 2 * RING_SLOT;
constexpr int CTRL_BYTES = 2048;
constexpr int SPLIT_SMEM = OFF_CTRL + CTRL_BYTES;     // all of the 227 KB a CTA can have
constexpr int CONV_WARPS = 8, CONV_THREADS = 32 * CONV_WARPS;
// Epilogue warps: at 16 densities two groups of eight, the warps of a group
// sharing a view's densities (200 functions 2.99 -> 2.78 ms against groups of
// four; a view's 224 columns are read, recombined and reduced by them); at 8
// densities groups of four (2.00 ms against 2.09 with eight: half the work, and
// more warps then only contend with the converters and the MMA issuer).
template <int MP>
constexpr int epi_warps = MP == 16 ? 16 : 8;
template <int MP>
constexpr int split_threads = 64 + CONV_THREADS + 32 * epi_warps<MP>;
// Smallest exponent fields of a tile: bricks below 2^-300 and density blocks
// below 2^-640 lose their low digits, then vanish, and no product's exponent
// leaves FP64's normal range.  Neither is seen beside the handle's largest
// integrals, which are above 2^-260 (a basis' exponents have squares in FP64's
// range), and the densities' largest elements, above 2^DMIN.
constexpr int EMIN_V = 1022 - 300, EMIN_D = 1022 - 640;
constexpr int REGION = 256;                       // tensor-memory columns per view buffer
static_assert(OFF_RING % 1024 == 0 && OFF_REC % 16 == 0, "operand tiles");
static_assert(NT * 2 * MPM <= REGION, "view region");

struct SplitCtrl {
    uint64_t recfull[2], recfree[2];   // packed records: landed / read
    uint64_t convV, convW;             // digit tiles written (once per brick)
    uint64_t vfree, wfree;             // their MMAs done (once per brick)
    uint64_t dfull[2], mmad[2], accfree[2];   // per view: tile landed, MMAs done, accumulators read
    uint32_t tmem_base;
    int abort_flag;
    int never;                         // zero: waits that an abort must not cut short
    int decide;
    int scan[CONV_WARPS], emax[CONV_WARPS];
    unsigned epub;                     // bricks whose exponent is published in ev[]
    int ev[4];
    uint16_t vpos[512];
};
static_assert(SPLIT_SMEM <= 227 * 1024 && sizeof(SplitCtrl) <= CTRL_BYTES, "control block");

// Views of a brick in the order they run: 0-3 exchange V1..V4, 4 Coulomb J1, 5
// Coulomb J2 (see jk_umma.cu); the next one after v that the brick has.
__device__ __forceinline__ bool has_view(const BrickDesc &d, int v) {
    if (v == 1) return d.P != d.Q;
    if (v == 2) return d.R != d.S;
    if (v == 3) return d.P != d.Q && d.R != d.S;
    return v < 6;
}

// ---- recombination: sum_t c_t 2^(9 (3 - t)) as a double, rounded once.  The
// part of t <= 3 is an integer of at most 50 bits, formed on the integer pipe
// and read as a double through the bits of 1.5 2^52 + itself (|c_0| <= 2^22
// likewise from c_0 + 1.5 2^23); the c_t of t >= 4 are summed in FP32, whose
// bits widen to FP64 on the integer pipe too.  Two FP64 additions remain.
__device__ __forceinline__ double recombine(const float *c, int stride) {
    float f = fmaf(c[6 * stride], 0x1p-9f, c[5 * stride]);
    f = fmaf(f, 0x1p-18f, c[4 * stride] * 0x1p-9f);
    long long S = (long long)__float2int_rn(c[2 * stride]) * 512 + __float2int_rn(c[3 * stride]);
    S += (long long)__float2int_rn(c[1 * stride]) * (1 << 18);
    const int c0 = (int)(__float_as_uint(__fadd_rn(c[0], 12582912.f)) - 0x4b400000u);
    S += (long long)c0 * (1 << 27) + 0x4338000000000000ll;
    const uint32_t b = __float_as_uint(f);
    const uint32_t fhi = f == 0.0f ? 0u : (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u);
    return (__longlong_as_double(S) - 0x1.8p52) + __hiloint2double((int)fhi, (int)(b << 29));
}

// *p += (value_hi, lo) as a double unless hi is zero (a zero value): a predicated
// reduction, so that the outputs of a loop are scheduled across each other
__device__ __forceinline__ void red_nonzero(double *p, int hi, int value_hi, int lo) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.s32 q, %1, 0;\n@q red.global.add.f64 [%0], %2;\n}" ::"l"(p), "r"(hi),
                 "d"(__hiloint2double(value_hi, lo))
                 : "memory");
}

// four columns for lanes 0-15, the next four for lanes 16-31 of 16 accumulator rows
__device__ __forceinline__ void tmem_ld_half4(uint32_t taddr, float *v) {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.16x32bx2.x4.b32 {%0,%1,%2,%3}, [%4], 4;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// canonical K-major operand tile: row n (density column of the MMA), k = b*8 + d
__device__ __forceinline__ int tile_off(int row, int k) {
    return (row & 7) * 16 + (k & 7) * 2 + (k >> 3) * 128 + (row >> 3) * 1024;
}

}  // namespace

// ---------------------------------------------------------------- density tiles
// Digit tiles of one pass (densities d0 .. d0+mp-1; those >= m are zero) and
// their exponents.  K bank, tile (X,Y) of nb*nb: row j*2mp + kk holds digit j
// of D[X*8+b][Y*8+d] at k = b*8 + d, row j*2mp + mp + kk that of
// D[Y*8+d][X*8+b]; exponent eK[(X*nb+Y)*16 + kk] of block (X,Y) (the
// transposed part of the tile has that of (Y,X)).  J bank, X >= Y: row j*mp +
// kk of D[X,Y] + [X != Y] D[Y,X]^T, exponent eJ.  top[kk]: the density's largest
// exponent field (0 at launch).  One warp per (X, Y, kk), lane l the two elements
// b = l / 4, d = 2 (l % 4) + {0, 1}.
__global__ void __launch_bounds__(256) k_split_dbank(const double *D, int n, int nb, int m, int d0, int mp,
                                                     unsigned char *kbank, unsigned char *jbank, int16_t *eK,
                                                     int16_t *eJ, int *top) {
    const int tile = blockIdx.x, X = tile / nb, Y = tile % nb;
    const int lane = threadIdx.x & 31, kk = blockIdx.y * 8 + (threadIdx.x >> 5);
    const int b = lane >> 2, d = 2 * (lane & 3);
    const double *Dk = D + (int64_t)(d0 + kk) * n * n;
    const int p = X * 8 + b, q = Y * 8 + d;
    const bool live = kk < m;
    double v[2], t[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool in = live && p < n && q + h < n;
        v[h] = in ? Dk[(int64_t)p * n + q + h] : 0.0;
        t[h] = in ? Dk[(int64_t)(q + h) * n + p] : 0.0;
    }
    const int f = __reduce_max_sync(0xffffffffu, max(field_of(v[0]), field_of(v[1])));
    if (lane == 0 && live && f) atomicMax(top + kk, f);
    auto emit = [&](const double *x, unsigned char *base, int row, int rows, int16_t *eout) {
        const uint32_t h0 = (uint32_t)__double2hiint(x[0]), h1 = (uint32_t)__double2hiint(x[1]);
        int e = max((int)((h0 >> 20) & 0x7ffu), (int)((h1 >> 20) & 0x7ffu));
        e = max(__reduce_max_sync(0xffffffffu, e), EMIN_D);
        uint32_t wa[3], wb[3];
        digit_words<ND>(fixed_point<53>((uint32_t)__double2loint(x[0]), h0, e), wa);
        digit_words<ND>(fixed_point<53>((uint32_t)__double2loint(x[1]), h1, e), wb);
        const int o = tile_off(row, b * 8 + d), step = rows * 128;   // rows of one digit: rows * 128 bytes
        *reinterpret_cast<uint32_t *>(base + o) = digit_pair<0>(wa, wb);
        *reinterpret_cast<uint32_t *>(base + o + step) = digit_pair<1>(wa, wb);
        *reinterpret_cast<uint32_t *>(base + o + 2 * step) = digit_pair<2>(wa, wb);
        *reinterpret_cast<uint32_t *>(base + o + 3 * step) = digit_pair<3>(wa, wb);
        *reinterpret_cast<uint32_t *>(base + o + 4 * step) = digit_pair<4>(wa, wb);
        *reinterpret_cast<uint32_t *>(base + o + 5 * step) = digit_pair<5>(wa, wb);
        if (lane == 0 && eout) *eout = (int16_t)(e - 1022);
    };
    unsigned char *kt = kbank + (size_t)tile * (ND * 2 * mp * 128);
    emit(v, kt, kk, 2 * mp, eK + (size_t)tile * MPM + kk);
    emit(t, kt, mp + kk, 2 * mp, nullptr);
    if (X >= Y) {
        double s[2] = {v[0], v[1]};
        if (X != Y) { s[0] += t[0]; s[1] += t[1]; }
        const size_t jt = (size_t)X * (X + 1) / 2 + Y;
        emit(s, jbank + jt * (ND * mp * 128), kk, mp, eJ + jt * MPM + kk);
    }
}

// ---------------------------------------------------------------- main kernel
struct SplitParams {
    const BrickDesc *bricks;
    int64_t nbricks;
    const int64_t *offsets;        // record start, in 8-byte elements
    const unsigned char *store;
    const unsigned char *kbank, *jbank;
    const int16_t *eK, *eJ;
    const double *D;               // caller's densities (the plain path)
    int n, nb, m, d0, mtot;
    double *Jacc, *Kacc, *KTacc;   // block-major [X][Y][k][x][y], k < mtot
    const int *top;                // largest exponent fields of the pass's densities
    int *error;                    // the handle's device error flag
};

namespace {

// Plain FP64 form of the kernel's bricks, for densities beyond the digits'
// range: the dense tile in shared memory, one output per thread and step, the
// sums in the order of the CUDA-core kernel.
template <int SRC>
__device__ void plain_bricks(const SplitParams &P, unsigned char *sm) {
    double *V = reinterpret_cast<double *>(sm);
    unsigned short *pos = reinterpret_cast<unsigned short *>(sm + 8 * BRICK);
    const int64_t nn = (int64_t)P.n * P.n;
    for (int64_t bi = blockIdx.x; bi < P.nbricks; bi += gridDim.x) {
        const BrickDesc d = P.bricks[bi];
        const unsigned char *rec = P.store + P.offsets[bi] * 8;
        __syncthreads();
        for (int v = threadIdx.x; v < 512; v += blockDim.x) {
            int c = 0;
            for (int u = 0; u < v; ++u) c += __popc(rec[u]);
            pos[v] = (unsigned short)c;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < BRICK; e += blockDim.x) {
            const unsigned mk = rec[e >> 3];
            double x = 0.0;
            if (mk & (1u << (e & 7))) {
                const int i = pos[e >> 3] + __popc(mk & ((1u << (e & 7)) - 1u));
                if (SRC == 0) x = reinterpret_cast<const double *>(rec + MASK_BYTES)[i];
                else {
                    const float2 u = reinterpret_cast<const float2 *>(rec + MASK_BYTES)[i];
                    x = (double)u.x + (double)u.y;
                }
            }
            V[e] = x;
        }
        __syncthreads();
        const bool diag = d.R == d.P && d.S == d.Q;
        const int blk[4] = {d.P, d.Q, d.R, d.S}, str[4] = {512, 64, 8, 1};
        // per view: positions of the output row, output column and the two summed indices
        const int vw[6][4] = {{0, 2, 1, 3}, {1, 2, 0, 3}, {0, 3, 1, 2}, {1, 3, 0, 2}, {0, 1, 2, 3}, {2, 3, 0, 1}};
        for (int v = 0; v < 6; ++v) {
            if (!has_view(d, v) || (v == 5 && diag)) continue;
            const int A = vw[v][0], C = vw[v][1], X = vw[v][2], Y = vw[v][3];
            const bool coul = v >= 4;
            const int parts = (coul || diag) ? 1 : 2;
            for (int t = threadIdx.x; t < parts * 64 * P.m; t += blockDim.x) {
                const int e = t & 63, k = (t >> 6) % P.m, part = (t >> 6) / P.m;
                const double *Dk = P.D + (int64_t)(P.d0 + k) * nn;
                double acc = 0.0;
                for (int x = 0; x < 8; ++x)
                    for (int y = 0; y < 8; ++y) {
                        const int gx = blk[X] * 8 + x, gy = blk[Y] * 8 + y;
                        double dv = 0.0;
                        if (gx < P.n && gy < P.n) {
                            dv = part ? Dk[(int64_t)gy * P.n + gx] : Dk[(int64_t)gx * P.n + gy];
                            if (coul && blk[X] != blk[Y]) dv += Dk[(int64_t)gy * P.n + gx];
                        }
                        acc = fma(V[(e >> 3) * str[A] + (e & 7) * str[C] + x * str[X] + y * str[Y]], dv, acc);
                    }
                double *out = coul ? P.Jacc : (part ? P.KTacc : P.Kacc);
                atomicAdd(out + ((int64_t)(blk[A] * P.nb + blk[C]) * P.mtot + P.d0 + k) * 64 + e, acc);
            }
        }
    }
}

}  // namespace

// SRC: 0 FP64 store, 1 double-FP32 store; MP: density columns of the pass (8 or 16)
// JN: a thread's densities that are recombined, three of four when the pass has
// no more (the GVP and energy builds): 200 functions, 3 densities 2.01 -> 1.93 ms.
// A run-time test instead cost 1 % at 4 to 8 densities and 2 % at 16.
template <int SRC, int MP, int JN>
__global__ void __launch_bounds__(split_threads<MP>, 1) k_jk_split(const __grid_constant__ SplitParams P) {
    extern __shared__ __align__(1024) unsigned char sm[];
    SplitCtrl &c = *reinterpret_cast<SplitCtrl *>(sm + OFF_CTRL);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (__any_sync(0xffffffffu, lane < P.m && beyond_digits(P.top[lane]))) {
        plain_bricks<SRC>(P, sm);
        return;
    }
    constexpr uint32_t KBYTES = ND * 2 * MP * 128, JBYTES = ND * MP * 128;
    volatile int *abort_flag = &c.abort_flag;
    const int64_t step = gridDim.x;
    const int nloc = (int)((P.nbricks - blockIdx.x + step - 1) / step);   // bricks of this CTA

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&c.recfull[s], 1);
            mbar_init(&c.recfree[s], CONV_WARPS);
            mbar_init(&c.dfull[s], 1);
            mbar_init(&c.mmad[s], 1);
            mbar_init(&c.accfree[s], epi_warps<MP> / 2);
        }
        mbar_init(&c.convV, CONV_WARPS);
        mbar_init(&c.convW, CONV_WARPS);
        mbar_init(&c.vfree, 1);
        mbar_init(&c.wfree, 1);
        c.abort_flag = 0;
        c.never = 0;
        c.epub = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc(&c.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    auto fail = [&](int code) {
        *abort_flag = 1;
        if (P.error) atomicExch(P.error, code);
    };
    auto brick = [&](int i) { return P.bricks[blockIdx.x + (int64_t)i * step]; };

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------ producer
        int recs = 0, views = 0;
        auto load_record = [&](int i, const BrickDesc &d) -> bool {
            const int s = i & 1;
            if (i >= 2 && !wait_for(&c.recfree[s], ((i - 2) >> 1) & 1, abort_flag)) { fail(21); return false; }
            const uint32_t rec = ((uint32_t)MASK_BYTES + 8u * (uint32_t)d.nkept + 15u) & ~15u;
            mbar_arrive_expect_tx(&c.recfull[s], rec);
            bulk_g2s(sm + OFF_REC + s * REC_BYTES, P.store + P.offsets[blockIdx.x + (int64_t)i * step] * 8, rec,
                     &c.recfull[s]);
            recs = i + 1;
            return true;
        };
        BrickDesc d = brick(0), dn = d;
        bool ok = load_record(0, d);
        for (int i = 0; ok && i < nloc; ++i, d = dn) {
            if (i + 1 < nloc) {
                dn = brick(i + 1);
                ok = load_record(i + 1, dn);
            }
            for (int v = 0; ok && v < 6; ++v) {
                if (!has_view(d, v)) continue;
                const int s = views & 1;
                if (views >= 2 && !wait_for(&c.mmad[s], ((views - 2) >> 1) & 1, abort_flag)) { fail(22); ok = false; break; }
                const int tx = (v == 0 || v == 2) ? d.Q : d.P, ty = (v < 2) ? d.S : d.R;   // D[Q,S] D[P,S] D[Q,R] D[P,R]
                const unsigned char *src;
                if (v < 4) src = P.kbank + ((size_t)tx * P.nb + ty) * KBYTES;
                else if (v == 4) src = P.jbank + ((size_t)d.R * (d.R + 1) / 2 + d.S) * JBYTES;
                else src = P.jbank + ((size_t)d.P * (d.P + 1) / 2 + d.Q) * JBYTES;
                const uint32_t bytes = v < 4 ? KBYTES : JBYTES;
                mbar_arrive_expect_tx(&c.dfull[s], bytes);
                bulk_g2s(sm + OFF_RING + s * RING_SLOT, src, bytes, &c.dfull[s]);
                ++views;
            }
        }
        // no copy may still be landing when the CTA leaves
        for (int k = recs > 2 ? recs - 2 : 0; k < recs; ++k) wait_for(&c.recfull[k & 1], (k >> 1) & 1, &c.never);
        for (int k = views > 2 ? views - 2 : 0; k < views; ++k) wait_for(&c.dfull[k & 1], (k >> 1) & 1, &c.never);
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        // One lane leads; every MMA carries it as a predicate, so that the converged
        // warp forms the descriptors in uniform registers (200 functions, 16
        // densities: 7 % less time than with the MMAs in the elected lane's branch)
        const uint32_t lead = elect_one() ? 1u : 0u, sbase = smem_u32(sm);
        int views = 0;
        BrickDesc dn = brick(0);
        bool ok = true;
        for (int i = 0; ok && i < nloc; ++i) {
            const BrickDesc d = dn;
            if (i + 1 < nloc) dn = brick(i + 1);
            const int lastx = (d.R != d.S) ? (d.P != d.Q ? 3 : 2) : (d.P != d.Q ? 1 : 0);
            for (int v = 0; v < 6; ++v) {
                if (!has_view(d, v)) continue;
                const int s = views & 1;
                if (v == 0 && !__all_sync(~0u, wait_for(&c.convV, i & 1, abort_flag))) { fail(23); ok = false; break; }
                if (v == 4 && !__all_sync(~0u, wait_for(&c.convW, i & 1, abort_flag))) { fail(24); ok = false; break; }
                if (!__all_sync(~0u, wait_for(&c.dfull[s], (views >> 1) & 1, abort_flag))) { fail(25); ok = false; break; }
                if (views >= 2 && !__all_sync(~0u, wait_for(&c.accfree[s], ((views - 2) >> 1) & 1, abort_flag))) { fail(26); ok = false; break; }
                tc_fence_after();
                // A: views 0, 2, 4 step 256 B per 16 terms, the others 2048 B; views 0, 1, 4
                // are K-major, 2, 3, 5 MN-major
                const bool even = v == 0 || v == 2 || v == 4;
                const uint32_t lbo = even ? 128u : 1024u, sbo = even ? 1024u : 128u;
                const uint32_t W = v < 4 ? 2 * MP : MP;              // columns (and operand rows) of one digit
                const uint64_t a0 = sdesc(sbase + (v < 4 ? OFF_V : OFF_W), lbo, sbo), b0 = sdesc(sbase + OFF_RING + s * RING_SLOT, 128, 1024);
                const uint32_t alo = uniform((uint32_t)a0), ahi = uniform((uint32_t)(a0 >> 32));
                const uint32_t blo = uniform((uint32_t)b0), bhi = uniform((uint32_t)(b0 >> 32));
                const uint32_t ks = uniform((even ? 256u : 2048u) >> 4), col = uniform(tmem + s * REGION);
                const uint32_t Wu = uniform(W), wid = uniform((W >> 3) << 17);
                const uint32_t id0 = uniform(idesc_f16(64, 0, (v == 2 || v == 3 || v == 5) ? 1 : 0, 0));
#pragma unroll
                for (int x = 0; x < NV; ++x) {
                    // digit x of V against the density digits 0 .. nj-1, into the columns of t = x ..
                    const uint32_t nj = x < 2 ? ND : NT - x;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t a = alo + x * (SLICE >> 4) + j * ks, bd = blo + 16 * j;
                        if (x == 1 && j == 0) {
                            // t = 6 starts here: its columns are written, those of t < 6 added to
                            mma_pred(lead, col + Wu, a, ahi, bd, bhi, id0 + 5 * wid, 1u);
                            mma_pred(lead, col + 6 * Wu, a, ahi, bd + 40 * Wu, bhi, id0 + wid, 0u);
                        } else {
                            mma_pred(lead, col + x * Wu, a, ahi, bd, bhi, id0 + nj * wid, (x > 0 || j > 0) ? 1u : 0u);
                        }
                    }
                }
                if (lead) {
                    mma_commit(&c.mmad[s]);
                    if (v == lastx) mma_commit(&c.vfree);
                    if (v == 5) mma_commit(&c.wfree);
                }
                __syncwarp();
                ++views;
            }
        }
        // MMAs in flight must end before tensor memory is released
        for (int k = views > 2 ? views - 2 : 0; k < views; ++k) wait_for(&c.mmad[k & 1], (k >> 1) & 1, &c.never);
    } else if (warp >= 2 && warp < 2 + CONV_WARPS) {
        // ------------------------------------------------ converters
        const int ct = threadIdx.x - 64, cw = ct >> 5;
        BrickDesc dn = brick(0);
        for (int i = 0; i < nloc; ++i) {
            const int s = i & 1;
            const int nkept = dn.nkept;
            if (i + 1 < nloc) dn = brick(i + 1);
            if (!wait_for(&c.recfull[s], (i >> 1) & 1, abort_flag)) fail(27);
            // leave together: every converter thread must reach the same named barriers
            named_bar_sync(1, CONV_THREADS);
            if (ct == 0) c.decide = *abort_flag;
            const unsigned char *mask = sm + OFF_REC + s * REC_BYTES;
            const uint2 *vals = reinterpret_cast<const uint2 *>(mask + MASK_BYTES);
            // packed positions (exclusive scan of the per-vector counts) and the largest exponent
            const uint32_t mk2 = reinterpret_cast<const uint16_t *>(mask)[ct];
            const int tot = __popc(mk2);
            int incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            uint32_t hmax = 0;
            for (int k = ct; k < nkept; k += CONV_THREADS) hmax = max(hmax, (SRC == 0 ? vals[k].y : vals[k].x) & 0x7fffffffu);
            int em = SRC == 0 ? (int)(hmax >> 20) : (hmax >> 23 ? (int)(hmax >> 23) + 896 : 0);
            em = __reduce_max_sync(0xffffffffu, em);
            if (lane == 31) { c.scan[cw] = incl; c.emax[cw] = em; }
            named_bar_sync(1, CONV_THREADS);
            if (c.decide) break;
            int base = incl - tot, emax = SRC == 0 ? EMIN_V : 897;
#pragma unroll
            for (int w = 0; w < CONV_WARPS; ++w) {
                base += w < cw ? c.scan[w] : 0;
                emax = max(emax, c.emax[w]);
            }
            c.vpos[2 * ct] = (uint16_t)base;
            c.vpos[2 * ct + 1] = (uint16_t)(base + __popc(mk2 & 0xffu));
            if (ct == 0) {
                c.ev[i & 3] = emax - 1022;
                counter_release_add(&c.epub);
            }
            named_bar_sync(1, CONV_THREADS);
            // two s-vectors per thread, mapped so that the stores of 8 neighbouring
            // threads hit distinct bank groups in V and in W; their digits wait in
            // registers until the operand tiles are free
            uint32_t dg[2][NV][4];
            int vv[2], ww[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int u = k * CONV_THREADS + ct;
                const int q = u & 7, p = u >> 6, r = (q + ((u >> 3) & 7)) & 7;
                vv[k] = p * 64 + q * 8 + r;
                ww[k] = p * 64 + r * 8 + q;
                const uint32_t m8 = mask[vv[k]];
                const uint2 *src = vals + c.vpos[vv[k]];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    long long x[2];
#pragma unroll
                    for (int z = 0; z < 2; ++z) {
                        const int e = 2 * h + z;
                        uint2 w = make_uint2(0u, 0u);
                        if (m8 & (1u << e)) w = src[__popc(m8 & ((1u << e) - 1u))];
                        if (SRC == 0) x[z] = fixed_point<62>(w.x, w.y, emax);
                        else x[z] = fixed_point_f<62>(__uint_as_float(w.x), emax) + fixed_point_f<62>(__uint_as_float(w.y), emax);
                    }
                    uint32_t wa[3], wb[3];
                    digit_words<NV>(x[0], wa);
                    digit_words<NV>(x[1], wb);
                    dg[k][0][h] = digit_pair<0>(wa, wb);
                    dg[k][1][h] = digit_pair<1>(wa, wb);
                    dg[k][2][h] = digit_pair<2>(wa, wb);
                    dg[k][3][h] = digit_pair<3>(wa, wb);
                    dg[k][4][h] = digit_pair<4>(wa, wb);
                    dg[k][5][h] = digit_pair<5>(wa, wb);
                    dg[k][6][h] = digit_pair<6>(wa, wb);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.recfree[s]);
            auto store = [&](int off, const int *at) {
#pragma unroll
                for (int k = 0; k < 2; ++k)
#pragma unroll
                    for (int x = 0; x < NV; ++x)
                        *reinterpret_cast<uint4 *>(sm + off + x * SLICE + at[k] * 16) =
                            make_uint4(dg[k][x][0], dg[k][x][1], dg[k][x][2], dg[k][x][3]);
                fence_proxy_async();
                __syncwarp();
            };
            if (i >= 1 && !wait_for(&c.vfree, (i - 1) & 1, abort_flag)) fail(28);
            store(OFF_V, vv);
            if (lane == 0) mbar_arrive(&c.convV);
            if (i >= 1 && !wait_for(&c.wfree, (i - 1) & 1, abort_flag)) fail(29);
            store(OFF_W, ww);
            if (lane == 0) mbar_arrive(&c.convW);
        }
    } else if (warp >= 2 + CONV_WARPS) {
        // ------------------------------------------------ epilogue
        // group g takes the views with index parity g (tensor-memory region g); four
        // of its warps cover the four lane quarters for eight densities
        constexpr int GW = epi_warps<MP> / 2, H = 4;         // warps of a group, densities of a thread
        const int ew = warp - 2 - CONV_WARPS, g = ew / GW, slice = warp & 3;
        const int c0 = (ew % GW) / 4 * 2 * H;                // the warp's densities: c0 .. c0 + 7
        const uint32_t tl = tmem + ((uint32_t)(slice * 32) << 16) + g * REGION + c0;
        const int row = slice * 16 + (lane & 15), cb = c0 + (lane < 16 ? 0 : H);
        int views = 0;
        BrickDesc dn = brick(0);
        bool ok = true;
        for (int i = 0; ok && i < nloc; ++i) {
            const BrickDesc d = dn;
            if (i + 1 < nloc) dn = brick(i + 1);
            const bool diag = d.R == d.P && d.S == d.Q;
            int ev = 0;
            bool have = false;
            for (int v = 0; v < 6; ++v) {
                if (!has_view(d, v)) continue;
                const int vi = views++;
                if ((vi & 1) != g) continue;
                // the view's output block (A, C) and its density block (tx, ty)
                const int A = v == 5 ? d.R : ((v == 0 || v == 2 || v == 4) ? d.P : d.Q);
                const int C = v == 5 ? d.S : (v == 4 ? d.Q : (v < 2 ? d.R : d.S));
                const int tx = v == 4 ? d.R : ((v == 0 || v == 2) ? d.Q : d.P);
                const int ty = v == 5 ? d.Q : ((v < 2 || v == 4) ? d.S : d.R);
                const bool coul = v >= 4;
                // exponents of the parts' density blocks: the D part, then (exchange) the D^T part
                uint2 xq[2];
                {
                    const int16_t *ex = coul ? P.eJ + ((size_t)tx * (tx + 1) / 2 + ty) * MPM
                                             : P.eK + ((size_t)tx * P.nb + ty) * MPM;
                    const int16_t *et = coul ? ex : P.eK + ((size_t)ty * P.nb + tx) * MPM;
                    xq[0] = *reinterpret_cast<const uint2 *>(ex + cb);
                    xq[1] = *reinterpret_cast<const uint2 *>(et + cb);
                }
                if (!__all_sync(~0u, wait_for(&c.mmad[g], (vi >> 1) & 1, abort_flag))) { fail(30); ok = false; break; }
                if (!have) {
                    if (!__all_sync(~0u, counter_wait(&c.epub, (unsigned)i + 1u, abort_flag, POLLS))) { fail(31); ok = false; break; }
                    ev = c.ev[i & 3] - 43;
                    have = true;
                }
                tc_fence_after();
                const uint32_t W = coul ? MP : 2 * MP;
                const int64_t out = ((int64_t)(A * P.nb + C) * P.mtot + P.d0 + cb) * 64 + row;
                // no D^T part and no J2 for the (PQ|PQ) brick
                const int parts = (coul || diag) ? 1 : 2;
                const bool none = v == 5 && diag;
#pragma unroll 1
                for (int part = 0; part < parts; ++part) {
                    alignas(8) int16_t xp[H];
                    *reinterpret_cast<uint2 *>(xp) = part ? xq[1] : xq[0];
                    float a[NT * H];
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < NT; ++t) tmem_ld_half4(tl + part * MP + t * W, a + t * H);
                    tmem_wait_ld();
                    if (part == parts - 1) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&c.accfree[g]);
                    }
                    double *dst = (coul ? P.Jacc : (part ? P.KTacc : P.Kacc)) + out;
                    if (!none) {
#pragma unroll
                        for (int j = 0; j < JN; ++j) {
                            // the power of two is added to the exponent field; columns without a
                            // density have zeros
                            const double x = recombine(a + j, H);
                            const int hi = __double2hiint(x);
                            red_nonzero(dst + j * 64, hi, hi + ((ev + xp[j]) << 20), __double2loint(x));
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ---------------------------------------------------------------- host side
size_t split_kbank_bytes(int nb) { return (size_t)nb * nb * (ND * 2 * MPM * 128 + MPM * sizeof(int16_t)); }
size_t split_jbank_bytes(int nb) { return (size_t)nb * (nb + 1) / 2 * (ND * MPM * 128 + MPM * sizeof(int16_t)); }

template <int SRC, int MP, int JN = 4>
static int split_pass(const SplitParams &p, int grid, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_jk_split<SRC, MP, JN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SPLIT_SMEM);
    if (e != cudaSuccess) { set_error("smem attribute: %s", cudaGetErrorString(e)); return ESMF_ERR_CUDA; }
    k_jk_split<SRC, MP, JN><<<grid, split_threads<MP>, SPLIT_SMEM, s>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) { set_error("k_jk_split: %s", cudaGetErrorString(e)); return ESMF_ERR_CUDA; }
    return ESMF_OK;
}

int launch_jk_split(const SplitLaunch &L, cudaStream_t s) {
    if (L.ev_start) cudaEventRecord(L.ev_start, s);
    for (int d0 = 0; d0 < L.m; d0 += MPM) {
        const int mc = L.m - d0 < MPM ? L.m - d0 : MPM;
        const int mp = mc <= 8 ? 8 : MPM;
        SplitParams p;
        p.bricks = L.bricks; p.nbricks = L.nbricks; p.offsets = L.offsets;
        p.store = (const unsigned char *)L.store;
        // exponents behind the operand tiles of each bank
        unsigned char *kb = (unsigned char *)L.kbank, *jb = (unsigned char *)L.jbank;
        int16_t *eK = (int16_t *)(kb + (size_t)L.nb * L.nb * (ND * 2 * MPM * 128));
        int16_t *eJ = (int16_t *)(jb + (size_t)L.nb * (L.nb + 1) / 2 * (ND * MPM * 128));
        p.kbank = kb; p.jbank = jb; p.eK = eK; p.eJ = eJ;
        p.D = L.D; p.n = L.n; p.nb = L.nb; p.m = mc; p.d0 = d0; p.mtot = L.m;
        p.Jacc = L.Jacc; p.Kacc = L.Kacc; p.KTacc = L.KTacc; p.top = L.top + d0; p.error = L.error;
        k_split_dbank<<<dim3(L.nb * L.nb, mp / 8), 256, 0, s>>>(L.D, L.n, L.nb, mc, d0, mp, kb, jb, eK, eJ, L.top + d0);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) { set_error("k_split_dbank: %s", cudaGetErrorString(e)); return ESMF_ERR_CUDA; }
        const int grid = L.nbricks < L.num_sms ? (int)L.nbricks : L.num_sms;
        int rc;
        if (L.f32x2) rc = mc <= 3 ? split_pass<1, 8, 3>(p, grid, s) : mp == 8 ? split_pass<1, 8>(p, grid, s) : split_pass<1, 16>(p, grid, s);
        else rc = mc <= 3 ? split_pass<0, 8, 3>(p, grid, s) : mp == 8 ? split_pass<0, 8>(p, grid, s) : split_pass<0, 16>(p, grid, s);
        if (rc != ESMF_OK) return rc;
    }
    if (L.ev_stop) cudaEventRecord(L.ev_stop, s);
    return ESMF_OK;
}

}  // namespace esmf
