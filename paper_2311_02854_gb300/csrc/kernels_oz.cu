// FP64-accurate segmented grouped GEMM on the bf16 tensor cores of sm_103a.
//
// GB300 runs FP64 at ~1.2 TFLOP/s, so the products that must be FP64-accurate
// (the FP64 operator store, the residuals of the defect correction, FP64
// Rayleigh quotients) are emulated on the bf16 tensor cores by an error-free
// splitting of the operands (Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012):
//
//  * every 32-deep K stage of an output tile of up to 128 x 64 is converted by
//    loader warps: row r of A and column c of B get a power-of-two scale 2^E from the
//    largest magnitude in their 32 elements, the element is rounded to a
//    48-bit integer Q = round(|x| 2^(48-E)), and Q is cut into six 8-bit
//    slices q_0..q_5 (q_0 <= 256) stored as bf16 (exact: at most 9 significant
//    bits), so that x = sign * sum_i q_i 2^(E - 8(i+1)) up to 2^(E-49);
//  * the slice products with i + j = g <= 5 are issued as tcgen05.mma
//    (M = 128, K = 16 per instruction) into one FP32 accumulator per
//    order g in tensor memory.  Every product is an integer below 2^16 and
//    each order's sum over the 32-deep stage stays below 2^24 for g <= 5, so
//    the accumulations are exact whatever the order of the additions;
//  * the epilogue warps read the six orders, combine them with the row and
//    column scales and the segment's alpha into a double-float (two FP32)
//    accumulator per element (FP32 arithmetic only: GB300's FP32 rate is ~64x
//    its FP64 rate), and at the end of the tile write or atomically add the
//    FP64 result.
//
// The work list is the FP64 engine's (Tile / Seg records over FP64 buffers of
// a BufTable), lowered with 128 x 64 tiles (stacked products: Tile::sn) and
// uploaded longest first.  Persistent CTAs, one per SM, walk (tile, vector)
// items with the vectors innermost, so the CTAs that run at the same time share
// their operator tiles in L2.  Slices are kept in 128B-swizzled rows 64 deep
// that hold two stages, so stage q+1 is converted into the other half while the
// tensor cores consume stage q.
//
// Bound: the instruction streams of the conversion and of the combination, not
// the tensor pipe.  Hence the split: two groups of six loader warps convert
// alternate stages, each thread eight values of one row that it keeps in
// registers from the scale to the slices (two to four lanes share a row, by the
// depth of the stage); rows and columns outside the block are neither loaded nor
// converted; the slices of B follow each other along N, so that one instruction
// multiplies a slice of A with all the slices of B it meets (6 instructions per
// 16-deep step instead of 21); a tile of up to 32 columns has two sets of
// accumulators, and only its columns are combined, by two warps per 32 rows.  A
// warp reads the tensor memory of its own scheduler's quarter only, so tiles of
// up to 32 rows keep one of the four schedulers busy: the loaders stay off the
// first scheduler, and lists stack up to four such products in a tile.  The code
// of each role is kept short: with the column loops unrolled (accumulators in
// registers) a warp spent ~1900 cycles per four columns and 22 000 on writing a
// tile out, fetching instructions.  FP64-pipe instructions take a scheduler ~74
// cycles each, so floats are widened by their bits.  (Four warps that converted
// all 128 rows of every stage, one row per thread, and 42 instructions per stage
// took ~7 us per stage.)
// Warps 0-7 epilogue (warp w: tile rows 32 (w % 4) .., half w / 4 of the
// columns), warp 8 lane 0 issues the MMAs, the other warps but 12, 16 and 20 loaders.  Every
// wait is bounded; a timeout sets the device error word.
#include <cuda_bf16.h>

#include <algorithm>

#include "engine.h"
#include "ptx.h"

namespace dmrg {
namespace {

using namespace ptx;

constexpr int OTM = 128, OTN = 64, OTK = 32;   // tile rows, columns, stage depth
constexpr int ROWB = 128;                      // bytes of a swizzled slice row (64 deep: two stages)
constexpr int NSL = 6;                         // slices per operand
constexpr int NORD = 6;                        // accumulated orders g = i + j = 0..5
constexpr int A_SLICE = OTM * ROWB;            // 16 KB
constexpr int SLICE_BYTES = NSL * (OTM + OTN) * ROWB;
constexpr int NREC = 4;
constexpr uint32_t TMEM_COLS = 512;            // 6 orders x 64 columns (or twice 6 x 32), rounded to a power of two
constexpr int NEPI = 8;                        // epilogue warps
constexpr int MMA_WARP = NEPI;
constexpr int NLDW = 6;                        // loader warps of a group
constexpr int OZ_THREADS = (NEPI + 16) * 32;   // warps 12, 16 and 20 idle (the first scheduler's)
constexpr int EPI_COLS = OTN / 2;

// per-stage record shared by loaders (write), MMA issuer and epilogue (read)
struct OzStage {
    int32_t ea[OTM];   // row scales of A (exponent E: |x| < 2^E), -1000 for a zero row
    int32_t eb[OTN];   // column scales of B
    float ah, al;      // alpha as a double-float pair
    int32_t flags;     // 2 last stage of the tile, 4 no MMA (tile without products)
    int32_t ksteps;    // 16-deep MMA steps
    int32_t n16;       // MMA N / 16
    int32_t pad;
};
// the epilogue's double-float accumulators live in shared memory ([column][thread],
// conflict-free), so that the loop over the columns need not be unrolled
constexpr int ACC_BYTES = NEPI * 32 * EPI_COLS * 8;
constexpr int OZ_SMEM = 1024 + SLICE_BYTES + NREC * (int)sizeof(OzStage) + ACC_BYTES;
static_assert(OZ_SMEM <= 232448, "shared memory of one SM");

// biased exponent field of a double (0 for zero and subnormals)
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// 48-bit integer magnitude of |x| 2^(48-E) (rounded half up), with E = ebias - 1023
__device__ __forceinline__ uint64_t q48(double x, int ebias) {
    const uint64_t bits = (uint64_t)__double_as_longlong(x);
    const int eb = (int)((bits >> 52) & 0x7FF);
    const uint64_t m = (bits & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const int sh = ebias + 4 - eb;  // right shift, >= 5
    if (eb == 0 || sh >= 54) return 0;  // zero / subnormal: below every scale used here
    return (m + (1ull << (sh - 1))) >> sh;
}

// Slices of eight values at 16-byte column c of row `row` of the six slice tiles
// at dst + i * slice (128B-swizzled, K-major)
__device__ __forceinline__ void store_slices(const double (&x)[8], int ebias, uint32_t dst, uint32_t slice, int row,
                                             int c) {
    uint32_t w[NSL][4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        uint32_t f[2][NSL];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint64_t Q = q48(x[2 * p + h], ebias);
            const uint32_t ql = (uint32_t)Q, qh = (uint32_t)(Q >> 32);
            // 2^23 + slice as FP32 bits, minus 2^23: the slice (0..256), exact in bf16
            const uint32_t t[NSL] = {0x4B000000u | (qh >> 8), __byte_perm(qh, 0x4B000000u, 0x7650),
                                     __byte_perm(ql, 0x4B000000u, 0x7653), __byte_perm(ql, 0x4B000000u, 0x7652),
                                     __byte_perm(ql, 0x4B000000u, 0x7651), __byte_perm(ql, 0x4B000000u, 0x7650)};
#pragma unroll
            for (int i = 0; i < NSL; ++i) f[h][i] = __float_as_uint(__uint_as_float(t[i]) - 8388608.0f);
        }
        const uint32_t sign = (((uint32_t)__double2hiint(x[2 * p]) >> 16) & 0x8000u) |
                              ((uint32_t)__double2hiint(x[2 * p + 1]) & 0x80000000u);
#pragma unroll
        for (int i = 0; i < NSL; ++i) w[i][p] = __byte_perm(f[0][i], f[1][i], 0x7632) | sign;
    }
    const uint32_t off = dst + (uint32_t)((row >> 3) * 1024 + (row & 7) * ROWB + (((c ^ (row & 7)) & 7) << 4));
#pragma unroll
    for (int i = 0; i < NSL; ++i)
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(off + i * slice), "r"(w[i][0]), "r"(w[i][1]),
                     "r"(w[i][2]), "r"(w[i][3])
                     : "memory");
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// exactly representable FP32 power of two 2^k (0 below the normal range)
__device__ __forceinline__ float pow2f(int k) {
    if (k < -126) return 0.0f;
    if (k > 127) k = 127;
    return __uint_as_float((uint32_t)(k + 127) << 23);
}

__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_gemm_kernel(const Tile* __restrict__ tiles, int ntiles, int nvec, int single, const Seg* __restrict__ segs,
                   BufTable bt) {
    extern __shared__ uint8_t smem_raw[];
    // full[h]: loaders -> MMA (slices of K half h and the stage record written);
    // rec[h]: MMA -> epilogue (record visible); done[h]: MMA completion -> loaders
    // (half h free) and epilogue (orders ready); free[h]: epilogue -> MMA (orders read)
    __shared__ __align__(8) uint64_t full_bar[2], rec_bar[2], done_bar[2], free_bar[2], drain_bar;
    __shared__ uint32_t tmem_base_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = sbase, sB = sbase + NSL * A_SLICE;
    OzStage* recs = reinterpret_cast<OzStage*>(smem_raw + (sbase - smem_u32(smem_raw)) + SLICE_BYTES);
    float2* acc_s = reinterpret_cast<float2*>(recs + NREC);

    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), TMEM_COLS);
    if (tid == 0) {
        for (int h = 0; h < 2; ++h) {
            mbar_init(smem_u32(&full_bar[h]), NLDW);
            mbar_init(smem_u32(&rec_bar[h]), 1);
            mbar_init(smem_u32(&done_bar[h]), 1);
            mbar_init(smem_u32(&free_bar[h]), NEPI);
        }
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    const uint32_t total = (uint32_t)ntiles * (uint32_t)nvec, NV = (uint32_t)nvec;  // total < 2^31
    // the CTA's r-th item: dealt back and forth, since the items are ordered longest first
    const uint32_t G = gridDim.x;
    auto item = [&](uint32_t r) { return r * G + ((r & 1u) ? G - 1u - blockIdx.x : blockIdx.x); };
    bool failed = false;

    if (warp > MMA_WARP && (warp & 3) != 0) {
        // ---------------- loaders / converters ----------------
        const int li = warp - MMA_WARP - 1 - ((warp - MMA_WARP) >> 2);
        const uint32_t grp = (uint32_t)(li / NLDW);
        const int gw = li % NLDW;
        uint32_t d = 0;  // stages so far (all tiles, both groups)
        // The lanes hold the records of the next 32 segments of a tile (or, of lists
        // whose tiles have one segment each, of the next 32 tiles of this CTA): the
        // dependent loads tile -> segment are paid once per 32, not by every stage.
        uint32_t cr = 0;  // round of the next tile
        int cs = 0;       // segments of it already taken
        while (item(cr) < total && !failed) {
            const uint32_t t = item(single ? cr + (uint32_t)lane : cr);
            Tile T{};
            Seg S{};
            bool valid = false, last = true;
            if (t < total) {
                T = tiles[t / NV];
                const int idx = T.seg_beg + (single ? 0 : cs + lane);
                valid = idx < T.seg_end || (idx == T.seg_beg && T.seg_beg == T.seg_end);
                last = idx + 1 >= T.seg_end;
                if (idx < T.seg_end) S = segs[idx];
            }
            const int nseg = __shfl_sync(0xffffffffu, T.seg_end - T.seg_beg, 0);
            cs += 32;
            if (single) {
                cr += 32;
            } else if (cs >= nseg) {
                ++cr;
                cs = 0;
            }
            const int vt = (int)(t % NV);
            const int nl = __popc(__ballot_sync(0xffffffffu, valid));  // the valid lanes are the first nl
            for (int l = 0; l < nl && !failed; ++l) {
                const auto at = [&](auto x) { return __shfl_sync(0xffffffffu, x, l); };
                const int k = at(S.k), end = at((int)last);
                // a segment without depth only matters where it ends a tile
                const int nst = k > 0 ? (k + OTK - 1) / OTK : end;
                if (nst == 0) continue;
                if (nst == 1 && (d & 1u) != grp) {  // the other group's
                    ++d;
                    continue;
                }
                const int m = at(T.m), m0 = at(T.m0), n0 = at(T.n0), sn = at((int)T.sn), srows = 16 * at((int)T.sb);
                const int astride = at(T.astride), v = at(vt);
                const int mrem = min(OTM, m - m0), nrem = min(OTN, at(T.n) - n0), n16 = (nrem + 15) / 16;
                const uint32_t b_slice = (uint32_t)n16 * 16u * ROWB;  // the slices of B follow each other along N
                const int form = at(S.a_buf | (S.b_buf << 8) | (S.a_tr ? 1 << 16 : 0) | (S.b_tr ? 1 << 17 : 0));
                const int lda = at(S.lda), ldb = at(S.ldb);
                const int64_t ak = form >> 16 & 1 ? lda : 1, ar = form >> 16 & 1 ? 1 : lda;
                const int64_t bk = form >> 17 & 1 ? 1 : ldb, br = form >> 17 & 1 ? ldb : 1;
                const double* A0 = bt.p[form & 255] + at((long long)S.a_off) + (int64_t)v * bt.vstride[form & 255] + m0 * ar;
                const double* B0 = bt.p[form >> 8 & 255] + at((long long)S.b_off) + (int64_t)v * bt.vstride[form >> 8 & 255] + n0 * br;
                const double alpha = at(S.alpha);
                for (int st = 0; st < nst; ++st) {
                    const uint32_t slot = d & 1u, use = d >> 1;
                    OzStage& R = recs[d % NREC];
                    ++d;
                    if (slot != grp) continue;
                    const int kb = st * OTK, kn = max(0, min(OTK, k - kb)), steps = (kn + 15) / 16;
                    // a task: rt rows of one product's A or columns of B, 32 / rt K groups of eight
                    const int lg = kn > 16 ? 3 : 4, rt = 1 << lg;
                    const int lr = lane & (rt - 1), cg = lane >> lg;
                    const int nap = (mrem + rt - 1) >> lg;  // tasks of a product
                    const int na = kn > 0 ? nap * max(sn, 1) : 0, nb = kn > 0 ? (nrem + rt - 1) >> lg : 0;
                    const int kv = kn - 8 * cg;  // K values of this lane's group that exist
                    int ok = 1;
                    bool waited = false;
#pragma unroll 1
                    for (int t1 = gw; t1 < na + nb || !waited; t1 += NLDW) {
                        const bool isb = t1 >= na;
                        const int pi = isb || sn == 0 ? 0 : t1 / nap;  // stacked product
                        int row = ((isb ? t1 - na : t1 - pi * nap) << lg) + lr;
                        const double* q = isb ? B0 + row * br + (kb + 8 * cg) * bk
                                              : A0 + (int64_t)pi * astride + row * ar + (kb + 8 * cg) * ak;
                        const int64_t ks = isb ? bk : ak;
                        const int n = t1 < na + nb && row < (isb ? nrem : mrem) ? kv : 0;
                        row += pi * srows;
                        double x[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) x[j] = j < n ? q[j * ks] : 0.0;
                        if (!waited) {  // (the loads are in flight) half free: the MMAs of stage d - 2 completed
                            waited = true;
                            if (lane == 0 && use > 0) ok = mbar_wait(smem_u32(&done_bar[slot]), (use - 1) & 1u) ? 1 : 0;
                            ok = __shfl_sync(0xffffffffu, ok, 0);
                            if (!ok || t1 >= na + nb) break;
                        }
                        int emax = 0;
#pragma unroll
                        for (int j = 0; j < 8; ++j) emax = max(emax, exp_field(x[j]));
                        for (int o = rt; o < 32; o *= 2) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
                        const bool in = row < (isb ? 16 * n16 : OTM);  // (a task's last rows may lie beyond the buffers)
                        if (cg == 0 && in) (isb ? R.eb : R.ea)[row] = emax ? emax + 1 - 1023 : -1000;
                        if (cg < 2 * steps && in)
                            store_slices(x, emax + 1, isb ? sB : sA, isb ? b_slice : (uint32_t)A_SLICE, row,
                                         (int)slot * (OTK / 8) + cg);
                    }
                    if (!ok) {
                        failed = true;
                        break;
                    }
                    if (gw == 0 && lane == 0) {
                        R.ah = (float)alpha;
                        R.al = (float)(alpha - (double)R.ah);
                        R.flags = (end && st == nst - 1 ? 2 : 0) | (kn == 0 ? 4 : 0);
                        R.ksteps = steps;
                        R.n16 = n16;
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&full_bar[slot]));
                }
            }
        }
    } else if (warp == MMA_WARP) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            uint32_t d = 0;
            bool wide = false;  // the previous stage used all the accumulators
            for (uint32_t r = 0; item(r) < total && !failed; ++r) {
                for (;;) {
                    const uint32_t slot = d & 1u, use = d >> 1;
                    if (!mbar_wait(smem_u32(&full_bar[slot]), use & 1u)) { failed = true; break; }
                    const OzStage& R = recs[d % NREC];
                    const int flags = R.flags, steps = R.ksteps, n16 = R.n16;
                    // accumulators: the set of the stage's parity (up to 32 columns), or all
                    const bool w = n16 > 2;
                    if (use > 0 && !mbar_wait(smem_u32(&free_bar[slot]), (use - 1) & 1u)) { failed = true; break; }
                    if ((w || wide) && d >= 1 && !mbar_wait(smem_u32(&free_bar[slot ^ 1u]), ((d - 1) >> 1) & 1u)) {
                        failed = true;
                        break;
                    }
                    wide = w;
                    mbar_arrive(smem_u32(&rec_bar[slot]));
                    tc_fence_after();
                    if (!(flags & 4)) {
                        // slice i of A times the slices 0 .. 5 - i of B adds to the orders
                        // i .. 5: one instruction of N = (6 - i) cs (two above 256)
                        const uint32_t cs = 16u * (uint32_t)n16, dt0 = tmem + (w ? 0u : slot * 256u);
                        const uint32_t most = 256u / cs;  // slices of B per instruction
                        const uint32_t khalf = slot * (OTK * 2);
                        const uint64_t ad0 = sdesc(sA + khalf, 16, 1024), bd0 = sdesc(sB + khalf, 16, 1024);
                        for (int kk = 0; kk < steps; ++kk) {
#pragma unroll
                            for (uint32_t i = 0; i < NSL; ++i) {
                                const uint64_t ad = ad0 + (uint64_t)((i * A_SLICE) >> 4) + 2u * kk;
                                const uint32_t n0 = min((uint32_t)NSL - i, most), n1 = NSL - i - n0;
                                const uint32_t acc = (i == 0 && kk == 0) ? 0u : 1u;
                                mma_bf16(dt0 + i * cs, ad, bd0 + 2u * kk, idesc_mn(0, 0, 0, (int)(n0 * cs), OTM), acc);
                                if (n1 > 0)
                                    mma_bf16(dt0 + (i + n0) * cs, ad, bd0 + 2u * kk + (uint64_t)((n0 * cs * ROWB) >> 4),
                                             idesc_mn(0, 0, 0, (int)(n1 * cs), OTM), acc);
                            }
                        }
                    }
                    mma_commit(smem_u32(&done_bar[slot]));
                    ++d;
                    if (flags & 2) break;
                }
            }
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0)) failed = true;
        }
    } else if (warp < NEPI) {
        // ---------------- epilogue ----------------
        const int quarter = warp & 3, chalf = warp >> 2;
        const int row = quarter * 32 + lane;
        float2* acc = acc_s + tid;  // acc[c * NEPI * 32]: (high, low)
        uint32_t d = 0;
        Tile nT{};
        if (blockIdx.x < total) nT = tiles[blockIdx.x / NV];
        for (uint32_t round = 0; item(round) < total && !failed; ++round) {
            const uint32_t it = item(round), in = item(round + 1);
            const Tile T = nT;
            if (in < total) nT = tiles[in / NV];
            const int v = (int)(it % NV);
            const int nrem = min(OTN, T.n - T.n0);
            // this thread's output row (stacked products: m * ldc apart, their rows run on)
            int64_t orow = T.m0 + row;
            bool rok = orow < T.m, any = T.m0 + quarter * 32 < T.m;
            if (T.sn) {
                const int sr = 16 * T.sb, i = row / sr;
                rok = i < T.sn && row - i * sr < T.m;
                any = quarter * 32 < T.sn * sr;
                orow = (int64_t)i * T.m + row - i * sr;
            }
            // columns of this half (a multiple of four apart), none for rows outside
            const int hc = ((nrem + 1) / 2 + 3) & ~3, c0 = chalf * hc;
            const int ncol = any ? min(hc, nrem - c0) : 0;
            const uint32_t cs = (uint32_t)((nrem + 15) / 16) * 16u;  // columns of an order
            for (int c = 0; c < ((ncol + 3) & ~3); ++c) acc[c * NEPI * 32] = make_float2(0.f, 0.f);
            for (;;) {
                const uint32_t slot = d & 1u, use = d >> 1;
                int ok = 1;
                if (lane == 0)
                    ok = (mbar_wait(smem_u32(&rec_bar[slot]), use & 1u) && mbar_wait(smem_u32(&done_bar[slot]), use & 1u))
                             ? 1
                             : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) { failed = true; break; }
                __syncwarp();
                tc_fence_after();
                const OzStage& R = recs[d % NREC];
                const int flags = R.flags;
                ++d;
                if ((flags & 4) || ncol <= 0) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&free_bar[slot]));
                    if (flags & 2) break;
                    continue;
                }
                const int er = R.ea[row];
                const float ah = R.ah, al = R.al;
                const bool unit = (ah == 1.f || ah == -1.f) && al == 0.f;  // alpha = +-1: a sign only
                const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (cs > 32u ? 0u : slot * 256u) + (uint32_t)c0;
#pragma unroll 1
                for (int cc = 0; cc * 4 < ncol; ++cc) {
                    uint32_t a[NORD][4];
#pragma unroll
                    for (int g = 0; g < NORD; ++g) tmem_ld4(tb + (uint32_t)g * cs + (uint32_t)(cc * 4), a[g]);
                    int ec[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) ec[j] = R.eb[min(c0 + cc * 4 + j, OTN - 1)];
                    tmem_wait_ld();
                    if (cc * 4 + 4 >= ncol) {  // every order and scale of this stage is in registers: release them
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&free_bar[slot]));
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float2& sum = acc[(cc * 4 + j) * NEPI * 32];
                        // sum of the orders, order g weighted 2^-8g, as a double-float
                        float sh = __uint_as_float(a[0][j]), sl = 0.f, e;
#pragma unroll
                        for (int g = 1; g < NORD; ++g) {
                            two_sum(sh, __uint_as_float(a[g][j]) * pow2f(-8 * g), sh, e);
                            sl += e;
                        }
                        // unit of order 0: 2^(E_r - 8) 2^(E_c - 8)
                        const float sc = pow2f(er + ec[j] - 16);
                        sh *= sc;
                        sl *= sc;
                        float p, pe;
                        if (unit) {
                            p = sh * ah;
                            pe = sl * ah;
                        } else {  // times alpha (double-float product)
                            p = sh * ah;
                            pe = fmaf(sh, ah, -p);
                            pe = fmaf(sh, al, pe);
                            pe = fmaf(sl, ah, pe);
                        }
                        float2 t = sum;
                        float nh;
                        two_sum(t.x, p, nh, e);
                        t.y += e + pe;
                        t.x = nh;
                        sum = t;
                    }
                }
                if (flags & 2) break;
            }
            if (failed) break;
            // the tile's FP64 result
            if (rok && ncol > 0) {
                double* C = bt.p[T.c_buf] + T.c_off + (int64_t)v * bt.vstride[T.c_buf] + orow * T.ldc + T.n0 + c0;
#pragma unroll 1
                for (int c = 0; c < ncol; ++c) {
                    const float2 t = acc[c * NEPI * 32];
                    const double r = widen(t.x) + widen(t.y);
                    if (T.mode == TILE_ATOMIC) atomicAdd(C + c, r);
                    else C[c] = r;
                }
            }
        }
    }
    if (failed) atomicExch(bt.err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace

int oz_tile_rows() { return OTM; }
int oz_tile_cols() { return OTN; }
int oz_stage_depth() { return OTK; }

void launch_seg_gemm_oz(const WorkList& w, const BufTable& bt, int nvec, cudaStream_t st) {
    if (w.tiles.empty()) return;
    DMRG_REQUIRE(w.tile_m == OTM && w.tile_n == OTN, DMRG_EINVAL, "work list not lowered for the FP64 tensor-core engine");
    DMRG_REQUIRE(bt.pmask == 0, DMRG_EINVAL, "the FP64 tensor-core engine reads FP64 buffers only");
    DMRG_REQUIRE(bt.err != nullptr, DMRG_EINVAL, "the FP64 tensor-core engine needs an error word");
    const int64_t total = (int64_t)w.tiles.size() * nvec;
    DMRG_REQUIRE(total < (1LL << 31), DMRG_EINVAL, "work list too large for one launch");
    static bool attr = false;
    if (!attr) {
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
        attr = true;
    }
    int dev = 0, nsm = 0;
    DMRG_CHECK_CUDA(cudaGetDevice(&dev));
    DMRG_CHECK_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int grid = (int)std::min<int64_t>(total, std::max(nsm, 1));
    oz_gemm_kernel<<<grid, OZ_THREADS, OZ_SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, (int)w.single, w.d_segs, bt);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

}  // namespace dmrg
