// Tensor-core segmented grouped GEMM for sm_103a (5th-generation tensor cores):
// operands staged in shared memory (128B-swizzled canonical layouts, K-major
// or MN-major), tcgen05.mma kind::f16 with bf16 inputs and FP32 accumulation
// in tensor memory, completion tracked by mbarriers, persistent
// warp-specialised CTAs (one or two per SM) walking the tiles round-robin, the
// vectors of a launch innermost (the copies of one tile for every vector run
// back to back on neighbouring CTAs, so that the operator boxes they share are
// read from DRAM once and then served from L2).  One output
// tile (128 x 128) accumulates the K-segments of its block (the term sum of
// the sigma reduction happens in the accumulator).  bf16 "pieces": an operand x is held as hi + lo; with
// nsplit = 2 each product runs as hi*hi + hi*lo + lo*hi.
#include <cuda_bf16.h>

#include <algorithm>

#include "ptx.h"
#include "tc.h"

namespace dmrg {
namespace {

using namespace ptx;

constexpr int TM = 128, TN = 128, TK = 64;
static_assert(sizeof(Tile) % 4 == 0 && sizeof(TSeg) % 4 == 0, "work-list records are moved by 32-bit shuffles");
static_assert(sizeof(TSeg) % 16 == 0, "segment records stay 16-byte aligned");
constexpr int PIECE_BYTES = TM * TK * 2;  // one 128 x 64 bf16 operand tile
constexpr uint32_t TMEM_COLS = 128;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// instruction descriptor of a full 128 x 128 tile
__device__ __forceinline__ uint32_t idesc(int a_mn, int b_mn, int neg) { return idesc_mn(a_mn, b_mn, neg, TN, TM); }

// Stage one 128 x 64 (M x K) operand piece into shared memory in the 128B-swizzled
// canonical layout the MMA descriptors describe.  Element (r, k) of the
// operand is base[r*ld + k] (mn = 0: K-major) or base[k*ld + r] (mn = 1:
// MN-major), valid for r < R, k < K; chunks outside are zero-filled (no global
// read).  Producer thread p always handles the same 16-byte column chunk of 8
// rows 16 (K-major) or 8 (MN-major) apart, so the swizzle and the validity of
// the chunk's columns are loop invariant and each copy costs a few instructions.
__device__ __forceinline__ void load_piece(uint32_t sdst, const __nv_bfloat16* base, int ld, int mn, int r0, int R,
                                           int k0, int K, int p) {
    if (!mn) {
        const int c = p & 7, rr = p >> 3;  // chunk, first row (0..15)
        const int kk = k0 + c * 8;
        const int cvalid = kk < K ? min(8, K - kk) * 2 : 0;
        uint32_t dst = sdst + (uint32_t)((rr >> 3) * 1024 + (rr & 7) * 128 + ((c ^ (rr & 7)) << 4));
        const __nv_bfloat16* src = base + (int64_t)(r0 + rr) * ld + kk;
        const int64_t step = (int64_t)16 * ld;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const bool ok = (r0 + rr + 16 * j < R) && cvalid > 0;
            cp_async16(dst, ok ? (const void*)src : (const void*)base, ok ? cvalid : 0);
            dst += 2048;
            src += step;
        }
    } else {
        const int c = p & 15, kr = p >> 4;  // chunk along M, first K row (0..7)
        const int rr = r0 + c * 8;
        const int cvalid = rr < R ? min(8, R - rr) * 2 : 0;
        uint32_t dst = sdst + (uint32_t)((c >> 3) * 1024 + kr * 128 + (((c & 7) ^ kr) << 4));
        const __nv_bfloat16* src = base + (int64_t)(k0 + kr) * ld + rr;
        const int64_t step = (int64_t)8 * ld;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const bool ok = (k0 + kr + 8 * j < K) && cvalid > 0;
            cp_async16(dst, ok ? (const void*)src : (const void*)base, ok ? cvalid : 0);
            dst += 2048;
            src += step;
        }
    }
}

__device__ __forceinline__ void cp_async_wait_n(int n) {
    // wait until at most n committed groups are pending (n is 0..2 here)
    if (n <= 0) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    else if (n == 1) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    else asm volatile("cp.async.wait_group 2;\n" ::: "memory");
}
// Roles of the persistent kernel (one CTA per SM):
//   warps 0-3  epilogue: TMEM -> registers -> global (warp w owns TMEM lanes 32w..32w+31)
//   warps 4-7  producers: cp.async of the operand pieces of each 64-deep K stage
//   warp  8    MMA issuer (lane 0): tcgen05.mma into one of two TMEM accumulators
// Stages flow through a ring of STAGES shared-memory slots (full / empty
// mbarriers); tiles alternate between two 128-column TMEM accumulators
// (tmem_full / tmem_empty), so loads of the next stages, the MMAs of one tile
// and the epilogue of the previous tile overlap.  Every wait is bounded; on a
// timeout the CTA sets the error word and winds down.
constexpr int kEpiWarps = 4, kProdWarps = 4;
constexpr int NPROD = kProdWarps * 32;
constexpr int THREADS2 = (kEpiWarps + kProdWarps + 1) * 32;
template <int NSPLIT>
struct Cfg2 {
    static constexpr int STAGES = (NSPLIT == 1) ? 6 : (NSPLIT == 2 ? 3 : 2);
    static constexpr int STAGE_BYTES = 2 * NSPLIT * PIECE_BYTES;
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
    // the producers publish a stage's full barrier LAG stages after issuing it
    static constexpr int LAG = STAGES - 1 < 2 ? STAGES - 1 : 2;
};

// Piece products of a split-precision MMA: x = sum_i x_i with |x_i| ~ 2^-8i |x|;
// products x_i y_j with i + j <= NSPLIT - 1 are kept (1, 3 or 6 of them).
template <int NSPLIT>
struct Prods {
    static constexpr int N = NSPLIT == 1 ? 1 : (NSPLIT == 2 ? 3 : 6);
};
__device__ __forceinline__ int prod_a(int pr) { return (0x210100 >> (4 * pr)) & 0xF; }  // 0,0,1,0,1,2
__device__ __forceinline__ int prod_b(int pr) { return (0x012010 >> (4 * pr)) & 0xF; }  // 0,1,0,2,1,0

struct StageMeta {
    uint8_t a_mn, b_mn, neg, flags;  // flags: 1 first stage of a tile, 2 last, 4 no MMA (empty tile)
    int32_t k16;                     // 16-deep MMA steps holding data (1..4)
};

__device__ __forceinline__ int tile_stages(const Tile& T, const Seg* __restrict__ segs) {
    int nst = 0;
    for (int s = T.seg_beg; s < T.seg_end; ++s) nst += (segs[s].k + TK - 1) / TK;
    return nst;
}

// Epilogue of one tile by warps 0-3 (warp w owns TMEM lanes / tile rows
// 32w..32w+31): accumulator columns at TMEM address tacc -> registers, release
// of the accumulator (one arrive per warp on `tempty`), then alpha * acc
// written or accumulated into the output in the tile's mode.
template <int NSPLIT>
__device__ __forceinline__ void epilogue_tile(const Tile& T, int v, int nst, uint32_t tacc, int warp, int lane,
                                              const TcBufs& B, uint32_t tempty) {
    const int row = warp * 32 + lane;
    const int r = T.m0 + row;
    const bool rok = r < T.m;
    const float alpha = T.alpha;
    uint32_t acc[TN];
    if (nst > 0) {
#pragma unroll
        for (int cg = 0; cg < TN / 32; ++cg) {
            uint32_t (&a32)[32] = *reinterpret_cast<uint32_t(*)[32]>(&acc[cg * 32]);
            tmem_ld32(tacc + ((uint32_t)(warp * 32) << 16) + (uint32_t)(cg * 32), a32);
        }
        tmem_wait_ld();
    } else {
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[j] = 0u;
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(tempty);
    if (!rok || (nst == 0 && (T.mode == TC_ATOMIC_F64 || T.mode == TC_ATOMIC_F32))) return;
    const int ncol = min(TN, T.n - T.n0);
    const int64_t off = T.c_off + (int64_t)r * T.ldc + T.n0 + (int64_t)v * B.out_vstride[T.c_buf];
    if (T.mode == TC_ATOMIC_F64) {
        double* o = (double*)B.out[T.c_buf] + off;
#pragma unroll
        for (int j = 0; j < TN; ++j)
            if (j < ncol) atomicAdd(o + j, (double)alpha * (double)__uint_as_float(acc[j]));
    } else if (T.mode == TC_ATOMIC_F32) {
        float* o = (float*)B.out[T.c_buf] + off;
#pragma unroll
        for (int j = 0; j < TN; ++j)
            if (j < ncol) atomicAdd(o + j, alpha * __uint_as_float(acc[j]));
    } else if (T.mode == TC_STORE_F32) {
        float* o = (float*)B.out[T.c_buf] + off;
#pragma unroll
        for (int j = 0; j < TN; ++j)
            if (j < ncol) o[j] = alpha * __uint_as_float(acc[j]);
    } else {  // TC_STORE_SPLIT: chunks of 8 (rows padded to multiples of 8)
        __nv_bfloat16* oh = (__nv_bfloat16*)B.out[T.c_buf] + off;
        __nv_bfloat16* ol = (__nv_bfloat16*)B.out_lo[T.c_buf] + off;
#pragma unroll
        for (int j0 = 0; j0 < TN; j0 += 8) {
            if (j0 >= ncol) break;
            __align__(16) __nv_bfloat16 h8[8], l8[8], m8[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float x = alpha * __uint_as_float(acc[j0 + j]);
                const __nv_bfloat16 h = __float2bfloat16_rn(x);
                h8[j] = h;
                const float r = x - __bfloat162float(h);
                l8[j] = __float2bfloat16_rn(r);
                m8[j] = __float2bfloat16_rn(r - __bfloat162float(l8[j]));
            }
            *(uint4*)(oh + j0) = *(const uint4*)h8;
            if (NSPLIT >= 2) *(uint4*)(ol + j0) = *(const uint4*)l8;
            if (NSPLIT == 3) *(uint4*)(ol + B.out_pstride[T.c_buf] + j0) = *(const uint4*)m8;
        }
    }
}

template <int NSPLIT>
__global__ void __launch_bounds__(THREADS2, 1)
    tc_seg_gemm_kernel(const Tile* __restrict__ tiles, int ntiles, int nvec, const Seg* __restrict__ segs, TcBufs B) {
    using C = Cfg2<NSPLIT>;
    constexpr int S = C::STAGES;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], tfull_bar[2], tempty_bar[2], drain_bar;
    __shared__ StageMeta meta[S];
    __shared__ uint32_t tmem_base_s;
    __shared__ int fail_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         smem_u32(&tmem_base_s)),
                     "r"(2 * TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full_bar[s]), NPROD);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&tfull_bar[b]), 1);
            mbar_init(smem_u32(&tempty_bar[b]), kEpiWarps);
        }
        mbar_init(smem_u32(&drain_bar), 1);
        fail_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    const int total = ntiles * nvec;
    bool failed = false;

    if (warp >= kEpiWarps && warp < kEpiWarps + kProdWarps) {
        // ---------------- producers ----------------
        const int p = tid - kEpiWarps * 32;
        uint32_t q = 0;
        auto finish_stage = [&](uint32_t qs) {  // stage qs's copies are complete: publish it
            fence_proxy_async();
            mbar_arrive(smem_u32(&full_bar[qs % S]));
        };
        auto begin_stage = [&](uint32_t qs) -> bool {  // wait until slot of stage qs is free
            if (qs >= (uint32_t)S && !mbar_wait(smem_u32(&empty_bar[qs % S]), ((qs / S) - 1) & 1u)) return false;
            return true;
        };
        constexpr int LAG = C::LAG;
        auto end_issue = [&]() {  // after committing stage q: publish stage q - LAG
            cp_async_commit();
            if (q >= (uint32_t)LAG) {
                cp_async_wait_n(LAG);
                finish_stage(q - LAG);
            }
            ++q;
        };
        for (int t = blockIdx.x; t < total && !failed; t += gridDim.x) {
            const int tix = t / nvec, v = t % nvec;
            const Tile T = tiles[tix];
            const int nst = tile_stages(T, segs);
            if (nst == 0) {
                if (!begin_stage(q)) { failed = true; break; }
                if (p == 0) meta[q % S] = StageMeta{0, 0, 0, 1 | 2 | 4, 0};
                end_issue();
                continue;
            }
            int done = 0;
            for (int s = T.seg_beg; s < T.seg_end && !failed; ++s) {
                const Seg Sg = segs[s];
                const int a_mn = Sg.a_tr ? 1 : 0, b_mn = Sg.b_tr ? 0 : 1;
                const int64_t ao = Sg.a_off + (int64_t)v * B.vstride[Sg.a_buf];
                const int64_t bo = Sg.b_off + (int64_t)v * B.vstride[Sg.b_buf];
                for (int k0 = 0; k0 < Sg.k; k0 += TK) {
                    if (!begin_stage(q)) { failed = true; break; }
                    const uint32_t sa = sbase + (q % S) * C::STAGE_BYTES;
                    const uint32_t sb = sa + NSPLIT * PIECE_BYTES;
                    load_piece(sa, B.hi[Sg.a_buf] + ao, Sg.lda, a_mn, T.m0, T.m, k0, Sg.k, p);
                    load_piece(sb, B.hi[Sg.b_buf] + bo, Sg.ldb, b_mn, T.n0, T.n, k0, Sg.k, p);
                    if (NSPLIT >= 2) {
                        load_piece(sa + PIECE_BYTES, B.lo[Sg.a_buf] + ao, Sg.lda, a_mn, T.m0, T.m, k0, Sg.k, p);
                        load_piece(sb + PIECE_BYTES, B.lo[Sg.b_buf] + bo, Sg.ldb, b_mn, T.n0, T.n, k0, Sg.k, p);
                    }
                    if (NSPLIT == 3) {
                        load_piece(sa + 2 * PIECE_BYTES, B.lo[Sg.a_buf] + B.pstride[Sg.a_buf] + ao, Sg.lda, a_mn, T.m0,
                                   T.m, k0, Sg.k, p);
                        load_piece(sb + 2 * PIECE_BYTES, B.lo[Sg.b_buf] + B.pstride[Sg.b_buf] + bo, Sg.ldb, b_mn, T.n0,
                                   T.n, k0, Sg.k, p);
                    }
                    if (p == 0) {
                        const int kv = min(TK, Sg.k - k0);
                        meta[q % S] = StageMeta{(uint8_t)a_mn, (uint8_t)b_mn, (uint8_t)(Sg.alpha < 0.0 ? 1 : 0),
                                                (uint8_t)((done == 0 ? 1 : 0) | (done == nst - 1 ? 2 : 0)),
                                                (kv + 15) / 16};
                    }
                    end_issue();
                    ++done;
                }
            }
        }
        // publish the last LAG stages (or wind down after a failure)
        cp_async_wait0();
        for (uint32_t qs = (q >= (uint32_t)LAG ? q - LAG : 0); qs < q; ++qs) finish_stage(qs);
    } else if (warp == kEpiWarps + kProdWarps) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            uint32_t q = 0, tc = 0;
            for (int t = blockIdx.x; t < total && !failed; t += gridDim.x, ++tc) {
                const uint32_t buf = tc & 1u, use = tc >> 1;
                if (use > 0 && !mbar_wait(smem_u32(&tempty_bar[buf]), (use - 1) & 1u)) { failed = true; break; }
                tc_fence_after();
                const uint32_t dt = tmem + buf * TMEM_COLS;
                for (;;) {
                    const uint32_t slot = q % S;
                    if (!mbar_wait(smem_u32(&full_bar[slot]), (q / S) & 1u)) { failed = true; break; }
                    tc_fence_after();
                    const StageMeta M = meta[slot];
                    if (!(M.flags & 4)) {
                        const uint32_t sa = sbase + slot * C::STAGE_BYTES;
                        const uint32_t sb = sa + NSPLIT * PIECE_BYTES;
                        const uint32_t id = idesc(M.a_mn, M.b_mn, M.neg);
                        for (int kk = 0; kk < M.k16; ++kk) {
#pragma unroll
                            for (int pr = 0; pr < Prods<NSPLIT>::N; ++pr) {
                                const int pa = prod_a(pr), pb = prod_b(pr);
                                const uint32_t a_s = sa + pa * PIECE_BYTES;
                                const uint32_t b_s = sb + pb * PIECE_BYTES;
                                const uint64_t ad =
                                    M.a_mn ? sdesc(a_s + kk * 4096, 1024, 2048) : sdesc(a_s + kk * 32, 16, 1024);
                                const uint64_t bd =
                                    M.b_mn ? sdesc(b_s + kk * 4096, 1024, 2048) : sdesc(b_s + kk * 32, 16, 1024);
                                const uint32_t acc = ((M.flags & 1) && kk == 0 && pr == 0) ? 0u : 1u;
                                mma_bf16(dt, ad, bd, id, acc);
                            }
                        }
                    }
                    mma_commit(smem_u32(&empty_bar[slot]));
                    ++q;
                    if (M.flags & 2) break;
                }
                if (failed) break;
                mma_commit(smem_u32(&tfull_bar[buf]));
            }
            // every MMA issued by this thread has completed once this commit arrives
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0)) failed = true;
        }
    } else {
        // ---------------- epilogue ----------------
        uint32_t tc = 0;
        for (int t = blockIdx.x; t < total && !failed; t += gridDim.x, ++tc) {
            const uint32_t buf = tc & 1u, use = tc >> 1;
            int ok = 1;
            if (lane == 0) ok = mbar_wait(smem_u32(&tfull_bar[buf]), use & 1u) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);  // warp-uniform (tcgen05.ld is warp-collective)
            if (!ok) { failed = true; break; }
            __syncwarp();
            tc_fence_after();
            const int tix = t / nvec, v = t % nvec;
            const Tile T = tiles[tix];
            const int nst = tile_stages(T, segs);
            epilogue_tile<NSPLIT>(T, v, nst, tmem + buf * TMEM_COLS, warp, lane, B, smem_u32(&tempty_bar[buf]));
        }
    }
    if (failed) {
        fail_s = 1;
        atomicExch(B.err, 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(2 * TMEM_COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// TMA-staged kernel
// ---------------------------------------------------------------------------

__device__ __forceinline__ void mbar_arrive_tx(uint32_t addr, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(addr), "r"(bytes) : "memory");
}
// box of a 5-D tensor map (all its pieces) into shared memory, completion on an mbarrier
__device__ __forceinline__ void tma_load5(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w,
                                          uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(0), "r"(bar)
        : "memory");
}

// Rows of 128 bytes that one piece of an operand takes in shared memory: one box,
// of 128 rows for a K-major operand beyond 64 rows; an MN-major one beyond 64
// columns (halves = 2) has two boxes, every piece's halves NSPLIT * rows apart.
__device__ __forceinline__ int piece_rows(int mn, int halves, int box) { return !mn && halves == 2 ? 128 : box; }

// One operand (all pieces) of a stage from coordinates (x, y) of its map.  K-major
// (mn = 0): rows of the block at x = k0; MN-major (mn = 1): its columns at rows k0..
// (two: 128 of them).  A block that ends within the first 64 rows / columns brings
// no more: the MMA reads don't-care data beyond, which only reaches output rows /
// columns the epilogue drops.
template <int NSPLIT>
__device__ __forceinline__ void tma_operand(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w, uint32_t bar,
                                            uint32_t ps, bool two) {
    tma_load5(dst, map, x, y, z, w, bar);
    if (NSPLIT == 3) tma_load5(dst + ps, map + 1, x, y, z, w, bar);
    if (two) {
        tma_load5(dst + NSPLIT * ps, map, x + 64, y, z, w, bar);
        if (NSPLIT == 3) tma_load5(dst + 4 * ps, map + 1, x + 64, y, z, w, bar);
    }
}

// Roles: warps 0-7 epilogue in two groups of four that take the CTA's tiles
// alternately, warp 8 TMA producer (all lanes), warp 9 lane 0 MMA issuer.
//
// Bound: not by data.  The producer and the MMA lane spend their time issuing (waits,
// descriptors, copies, 6 to 12 MMAs, commits; ~1000 cycles per stage each, counted with
// one CTA per SM and a copy per piece), whatever the stage holds, so two CTAs share an
// SM, half of shared and tensor memory each, and issue in parallel (one CTA with everything:
// K = 24, D = 500, four vectors 20.4 ms, two: 11.6 ms; K = 36, D = 1000
// 16.4 -> 13.5 ms), and one copy brings all pieces of an operand (two per small
// stage instead of four: K = 8, D = 64 233 -> 185 us, K = 24 8.5 -> 7.7 ms).
// Large sectors come near what L2 hands to the SMs (K = 14 and K = 36: 8 to 10
// TB/s of operands while it runs), small ones stay with the issuing lanes.
constexpr int kCtas3 = 2;
constexpr int kEpiGroups = 2;
constexpr int kProdWarp3 = 4 * kEpiGroups;
constexpr int THREADS3 = (kProdWarp3 + 2) * 32;
constexpr uint32_t kAcc = 2;             // accumulators in tensor memory (2 x 128 of the 512 columns)

// Shared memory is a ring of UNITS units of 2 KB (16 rows of 128 bytes).  A stage
// takes the units that its boxes fill, [A pieces | B pieces] in one stretch, and
// up to SLOTS stages are in flight.  With fixed units of 32 KB (one for a stage
// within 64 x 64, else two) a stage of 48 x 48 or of 128 x 16 took 32 or 64 KB
// instead of 24 or 36, and two or three of them filled the ring: K = 14, D = 600
// 1.81 -> 1.52 ms, K = 36, D = 1000 11.0 -> 10.0, K = 24, D = 500, four vectors
// 7.7 -> 7.35.  (Tiny stages, which never filled it, pay for the bookkeeping:
// K = 8, D = 64 189 -> 197 us.  More than four slots gave nothing more there.)
template <int NSPLIT>
struct Cfg3 {
    static constexpr int UNITS = 55;
    static constexpr int SLOTS = 16;
    static constexpr int SMEM = UNITS * 2048 + 1024;
};

// stage record of the TMA kernel (one 8-byte word)
struct __align__(8) StageMeta3 {
    uint8_t form;        // 1 A MN-major, 2 B MN-major, 4 negate A, 8 cross terms swapped,
                         // 16 first stage of a tile, 32 last, 64 no MMA (empty tile)
    uint8_t kn;          // 16-deep K steps holding data | 16 * (MMA N / 16)
    uint8_t a_ps, b_ps;  // units between the pieces of an operand ...
    uint8_t a_lb, b_lb;  // ... and between the 64-wide halves of an MN-major one
    uint8_t a_at, b_at;  // first unit of each operand
};

__device__ __forceinline__ uint32_t idesc_n(int a_mn, int b_mn, int neg, int n) { return idesc_mn(a_mn, b_mn, neg, n, TM); }

// Epilogue of one tile by one group of four warps: the tile's columns 32 at a
// time from tensor memory, then alpha * acc in the tile's mode.  Warps whose 32
// rows lie outside the block only release the accumulator.
template <int NSPLIT>
__device__ __forceinline__ void epilogue_tma(const Tile& T, int v, uint32_t tacc, int w4, int lane, const TcBufs& B,
                                             uint32_t tempty) {
    const int row = w4 * 32 + lane;
    const int ncol = min((int)T.tn, T.n - T.n0);
    // row r of product i of a stack
    bool any, rok;
    int i = 0, r = T.m0 + row;
    if (T.sn) {
        i = row / (16 * T.sb);
        r = row - i * 16 * T.sb;
        any = w4 * 32 < T.sn * 16 * T.sb;
        rok = i < T.sn && r < T.m;
    } else {
        any = T.nst > 0 && T.m0 + w4 * 32 < T.m;
        rok = r < T.m;
    }
    const float alpha = T.alpha;
    const int64_t off = T.c_off + (int64_t)v * B.out_vstride[T.c_buf] +
                        (T.tr ? ((int64_t)i * T.n + T.n0) * T.ldc + r : ((int64_t)i * T.m + r) * T.ldc + T.n0);
    if (T.nst == 0 && T.mode == TC_STORE_SPLIT && rok) {  // a stored block without products is zero
        for (int j0 = 0; j0 < ncol; j0 += 8) {
            *(uint4*)((__nv_bfloat16*)B.out[T.c_buf] + off + j0) = make_uint4(0, 0, 0, 0);
            if (NSPLIT >= 2) *(uint4*)((__nv_bfloat16*)B.out_lo[T.c_buf] + off + j0) = make_uint4(0, 0, 0, 0);
            if (NSPLIT == 3)
                *(uint4*)((__nv_bfloat16*)B.out_lo[T.c_buf] + B.out_pstride[T.c_buf] + off + j0) = make_uint4(0, 0, 0, 0);
        }
    }
    if (any) {
        for (int c0 = 0; c0 < ncol; c0 += 32) {
            uint32_t acc[32];
            __syncwarp();
            tmem_ld32(tacc + ((uint32_t)(w4 * 32) << 16) + (uint32_t)c0, acc);
            tmem_wait_ld();
            if (c0 + 32 >= ncol) {  // the last columns are in registers: release the accumulator
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty);
            }
            if (!rok) continue;
            if (T.mode == TC_ATOMIC_F64) {
                double* o = (double*)B.out[T.c_buf] + off + c0;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (c0 + j < ncol) atomicAdd(o + j, (double)alpha * (double)__uint_as_float(acc[j]));
            } else if (T.tr) {  // TC_STORE_SPLIT, transposed: the lanes' elements of a column lie side by side
                __nv_bfloat16* oh = (__nv_bfloat16*)B.out[T.c_buf] + off + (int64_t)c0 * T.ldc;
                __nv_bfloat16* ol = (__nv_bfloat16*)B.out_lo[T.c_buf] + off + (int64_t)c0 * T.ldc;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    if (c0 + j >= ncol) break;
                    const float x = alpha * __uint_as_float(acc[j]);
                    const __nv_bfloat16 h = __float2bfloat16_rn(x);
                    *oh = h;
                    const float d = x - __bfloat162float(h);
                    const __nv_bfloat16 l = __float2bfloat16_rn(d);
                    if (NSPLIT >= 2) *ol = l;
                    if (NSPLIT == 3) ol[B.out_pstride[T.c_buf]] = __float2bfloat16_rn(d - __bfloat162float(l));
                    oh += T.ldc;
                    ol += T.ldc;
                }
            } else {  // TC_STORE_SPLIT: chunks of 8 (rows padded to multiples of 8)
                __nv_bfloat16* oh = (__nv_bfloat16*)B.out[T.c_buf] + off + c0;
                __nv_bfloat16* ol = (__nv_bfloat16*)B.out_lo[T.c_buf] + off + c0;
#pragma unroll
                for (int j0 = 0; j0 < 32; j0 += 8) {
                    if (c0 + j0 >= ncol) break;
                    __align__(16) __nv_bfloat16 h8[8], l8[8], m8[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float x = alpha * __uint_as_float(acc[j0 + j]);
                        const __nv_bfloat16 h = __float2bfloat16_rn(x);
                        h8[j] = h;
                        const float d = x - __bfloat162float(h);
                        l8[j] = __float2bfloat16_rn(d);
                        m8[j] = __float2bfloat16_rn(d - __bfloat162float(l8[j]));
                    }
                    *(uint4*)(oh + j0) = *(const uint4*)h8;
                    if (NSPLIT >= 2) *(uint4*)(ol + j0) = *(const uint4*)l8;
                    if (NSPLIT == 3) *(uint4*)(ol + B.out_pstride[T.c_buf] + j0) = *(const uint4*)m8;
                }
            }
        }
    } else {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
    }
}

// The lanes of the producer warp each hold the record of one segment (and of
// its tile): the tile / segment loads of 32 segments are in flight together,
// one batch ahead of the copies, and the lanes then issue their stages in
// order.  (One lane walking tile -> segment -> copies spent ~1 us per stage on
// the dependent loads, whatever the stage held: K = 24, D = 500 ran 5 % of the
// operand bytes per second that the same kernel reached on 400-wide sectors.)
struct ProdRec {
    int32_t a_map, b_map, a_z, b_z, k;
    int32_t m0, n0, v;
    uint8_t a_mn, b_mn, a_pv, b_pv, a_br, b_br, neg, flags;  // flags: 1 first segment of a tile, 2 last, 4 empty tile
    uint8_t nA, nB, n16, valid, a_bz, swap;
};

template <int NSPLIT>
__global__ void __launch_bounds__(THREADS3, kCtas3)
    tc_tma_kernel(const Tile* __restrict__ tiles, int ntiles, int nvec, const TSeg* __restrict__ segs,
                  const CUtensorMap* __restrict__ maps, int single, TcBufs B) {
    using C = Cfg3<NSPLIT>;
    constexpr uint32_t U = C::UNITS, SL = C::SLOTS;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[SL], empty_bar[SL], tfull_bar[kAcc], tempty_bar[kAcc], drain_bar;
    __shared__ StageMeta3 meta[SL];
    __shared__ uint32_t tmem_base_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), kAcc * TMEM_COLS);
    if (tid == 0) {
        for (uint32_t s = 0; s < SL; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (uint32_t b = 0; b < kAcc; ++b) {
            mbar_init(smem_u32(&tfull_bar[b]), 1);
            mbar_init(smem_u32(&tempty_bar[b]), 4);
        }
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    const uint32_t total = (uint32_t)ntiles * (uint32_t)nvec, G = gridDim.x, NV = (uint32_t)nvec;  // total < 2^31
    // The CTA's r-th item.  The items are ordered longest first; dealt in one
    // direction only, the first CTAs would get the longest of every round.
    auto item = [&](uint32_t r) { return r * G + ((r & 1u) ? G - 1u - blockIdx.x : blockIdx.x); };
    bool failed = false;

    if (warp == kProdWarp3) {
        // ---------------- TMA producer ----------------
        // cursor: the round of the next tile (single: of lane 0) and, for lists whose
        // tiles sum several segments, its record, the next segment and the record after it
        uint32_t cr = 0, ct = item(0);
        int cs = 0;
        Tile cT{}, nT{};
        if (!single) {
            if (ct < total) {
                cT = tiles[ct / NV];
                cs = cT.seg_beg;
            }
            if (item(1) < total) nT = tiles[item(1) / NV];
        }
        auto fetch = [&]() {
            ProdRec r{};
            Tile T = cT;
            int idx, v;
            if (single) {
                const uint32_t t = item(cr + (uint32_t)lane);
                r.valid = t < total;
                v = r.valid ? (int)(t % NV) : 0;
                if (r.valid) T = tiles[t / NV];
                idx = T.seg_beg;
                r.flags = 1 | 2;
                if (item(cr) < total) cr += 32;
            } else {
                idx = cs + lane;
                v = (int)(ct % NV);
                r.valid = ct < total && (idx < cT.seg_end || (lane == 0 && cT.seg_beg == cT.seg_end));
                r.flags = (idx == cT.seg_beg ? 1 : 0) | (idx + 1 >= cT.seg_end ? 2 : 0);
                cs += 32;
                if (ct < total && cs >= cT.seg_end) {
                    ct = item(++cr);
                    cT = nT;
                    cs = cT.seg_beg;
                    if (item(cr + 1) < total) nT = tiles[item(cr + 1) / NV];
                }
            }
            if (r.valid && idx < T.seg_end) {
                const TSeg S = segs[idx];
                r.a_map = S.a_map;
                r.b_map = S.b_map;
                r.a_z = S.a_z;
                r.b_z = S.b_z;
                r.k = S.k;
                r.a_mn = S.a_tr ? 1 : 0;
                r.b_mn = S.b_tr ? 0 : 1;
                r.a_pv = S.a_pv;
                r.b_pv = S.b_pv;
                r.a_br = S.a_br;
                r.b_br = S.b_br;
                r.a_bz = S.a_bz;
                r.swap = S.swap;
                r.neg = S.sign < 0.f ? 1 : 0;
            } else {
                r.flags = 1 | 2 | 4;
            }
            // a second 64-row (or 64-column) half only when the block extends past the first
            const int ncol = min((int)T.tn, T.n - T.n0);
            r.m0 = T.m0;
            r.n0 = T.n0;
            r.v = v;
            r.nA = (T.m - T.m0 > 64 && !T.sn) ? 2 : 1;
            r.nB = (ncol > 64) ? 2 : 1;
            r.n16 = (uint8_t)((ncol + 15) / 16);
            return r;
        };
        // The same in all lanes: stages issued, stages known to be free again, units
        // handed out (or skipped) and given back, and the ring position of head.
        // Lane i holds where the stage in slot i ends.
        uint32_t si = 0, tail = 0, head = 0, back = 0, pos = 0, end = 0;
        ProdRec next = fetch();
        while (!failed) {
            const ProdRec R = next;
            const unsigned live = __ballot_sync(0xffffffffu, R.valid);
            if (!live) break;
            next = fetch();
            const bool none = (R.flags & 4) != 0;
            const int nst = !R.valid ? 0 : (none ? 1 : (R.k + TK - 1) / TK);
            const int abox = R.a_bz * R.a_br;
            const int arows = piece_rows(R.a_mn, R.nA, abox), brows = piece_rows(R.b_mn, R.nB, R.b_br);
            const int au = NSPLIT * arows * (R.a_mn ? R.nA : 1) / 16, bu = NSPLIT * brows * (R.b_mn ? R.nB : 1) / 16;
            const uint32_t n = none ? 0 : au + bu;
            // the MMAs read 128 rows of A whatever the box holds: those units lie in the ring too
            // (but for stacked MN-major operators, whose two boxes are those 128 rows)
            const int areach = !R.a_mn ? (NSPLIT - 1) * arows / 16 + 8 : (R.a_bz > 1 ? au : 2 * NSPLIT * arows / 16);
            const uint32_t reach = none ? 0 : max((int)n, areach);
            const uint32_t need_l = n | reach << 8 | (uint32_t)nst << 16;
            // this segment's StageMeta3 but for the flags of first and last, the K steps
            // of its last stage and the ring position (the record is two words)
            const uint32_t form = R.a_mn | R.b_mn << 1 | R.neg << 2 | R.swap << 3;
            const uint32_t m0 = form | (uint32_t)(4 | R.n16 << 4) << 8 | (uint32_t)arows / 16 << 16 | (uint32_t)brows / 16 << 24;
            const uint32_t a_lb = R.a_bz > 1 ? R.a_br / 16 : NSPLIT * arows / 16;  // (stacked MN-major: one box apart)
            const uint32_t m1 = a_lb | (uint32_t)(NSPLIT * brows / 16) << 8 | (uint32_t)au << 24;
            const uint32_t klast = (uint32_t)(4 - (R.k - TK * (nst - 1) + 15) / 16) << 8;
            const CUtensorMap* am = maps + kMapsPerKey * R.a_map + (!R.a_mn && R.nA == 2 ? 2 : 0);
            const CUtensorMap* bm = maps + kMapsPerKey * R.b_map + (!R.b_mn && R.nB == 2 ? 2 : 0);
            const int av = R.a_pv ? R.v : 0, bv = R.b_pv ? R.v : 0;
            const bool a2 = R.a_mn && R.nA == 2, b2 = R.b_mn && R.nB == 2;
            const int nl = __popc(live);  // the valid lanes are the first nl
            for (int l = 0; l < nl && !failed; ++l) {
                const uint32_t w = __shfl_sync(0xffffffffu, need_l, l), un = w & 255u, ur = w >> 8 & 255u, us = w >> 16;
                for (uint32_t st = 0; st < us; ++st) {
                    if (pos + ur > U) {
                        head += U - pos;
                        pos = 0;
                    }
                    // units before head + un - U must be free (with no stage in flight all are)
                    while (si - tail >= SL || (tail != si && (int)(back + U - un - head) < 0)) {
                        const uint32_t t = tail % SL;
                        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&empty_bar[t]), (tail / SL) & 1u))) {
                            failed = true;
                            break;
                        }
                        back = __shfl_sync(0xffffffffu, end, t);
                        ++tail;
                    }
                    if (failed) break;
                    const uint32_t slot = si % SL;
                    if (lane == l) {
                        const uint32_t bar = smem_u32(&full_bar[slot]);
                        uint2* rec = reinterpret_cast<uint2*>(&meta[slot]);
                        if (none) {
                            *rec = make_uint2(16 | 32 | 64, 0);
                            mbar_arrive(bar);
                        } else {
                            const bool last = st + 1 == us;
                            *rec = make_uint2(m0 + ((R.flags & 1) && st == 0 ? 16 : 0) + ((R.flags & 2) && last ? 32 : 0) -
                                                  (last ? klast : 0),
                                              m1 + pos * 0x01010000u);
                            mbar_arrive_tx(bar, 2048u * n);
                            const uint32_t sa = sbase + 2048u * pos;
                            const int k0 = (int)st * TK;
                            tma_operand<NSPLIT>(sa, am, R.a_mn ? R.m0 : k0, R.a_mn ? k0 : R.m0, R.a_z, av, bar,
                                                128u * arows, a2);
                            tma_operand<NSPLIT>(sa + 2048u * au, bm, R.b_mn ? R.n0 : k0, R.b_mn ? k0 : R.n0, R.b_z, bv, bar,
                                                128u * brows, b2);
                        }
                    }
                    __syncwarp();
                    head += un;
                    pos += un;
                    if (lane == (int)slot) end = head;
                    ++si;
                }
            }
        }
    } else if (warp == kProdWarp3 + 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            uint32_t q = 0;
            for (uint32_t tc = 0; item(tc) < total && !failed; ++tc) {
                const uint32_t buf = tc % kAcc, use = tc / kAcc;
                if (use > 0 && !mbar_wait(smem_u32(&tempty_bar[buf]), (use - 1) & 1u)) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const uint32_t dt = tmem + buf * TMEM_COLS;
                for (;;) {
                    const uint32_t slot = q % SL;
                    if (!mbar_wait(smem_u32(&full_bar[slot]), (q / SL) & 1u)) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    const StageMeta3 M = meta[slot];
                    if (!(M.form & 64)) {
                        const uint32_t sa = sbase + M.a_at * 2048u, sb = sbase + M.b_at * 2048u;
                        const int a_mn = M.form & 1, b_mn = M.form >> 1 & 1, swap = M.form >> 3 & 1;
                        const uint32_t aps = M.a_ps * 2048u, bps = M.b_ps * 2048u;
                        const uint32_t id = idesc_n(a_mn, b_mn, M.form >> 2 & 1, M.kn & 0xF0);
                        // bits of a descriptor besides its address, and the address step of a 16-deep K step
                        const uint64_t ab = a_mn ? sdesc(0, M.a_lb * 2048u, 1024) : sdesc(0, 16, 1024);
                        const uint64_t bb = b_mn ? sdesc(0, M.b_lb * 2048u, 1024) : sdesc(0, 16, 1024);
                        const uint32_t ak = a_mn ? 2048 : 32, bk = b_mn ? 2048 : 32;
                        for (int kk = 0; kk < (M.kn & 15); ++kk) {
#pragma unroll
                            for (int pr = 0; pr < Prods<NSPLIT>::N; ++pr) {
                                const uint32_t a_s = sa + (swap ? prod_b(pr) : prod_a(pr)) * aps + kk * ak;
                                const uint32_t b_s = sb + (swap ? prod_a(pr) : prod_b(pr)) * bps + kk * bk;
                                const uint32_t acc = ((M.form & 16) && kk == 0 && pr == 0) ? 0u : 1u;
                                mma_bf16(dt, ab | ((a_s & 0x3FFFFu) >> 4), bb | ((b_s & 0x3FFFFu) >> 4), id, acc);
                            }
                        }
                    }
                    mma_commit(smem_u32(&empty_bar[slot]));
                    ++q;
                    if (M.form & 32) break;
                }
                if (failed) break;
                mma_commit(smem_u32(&tfull_bar[buf]));
            }
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0)) failed = true;
        }
    } else {
        // ---------------- epilogue ----------------
        const int grp = warp >> 2, w4 = warp & 3;
        Tile Tn{};
        if (item(grp) < total) Tn = tiles[item(grp) / NV];
        for (uint32_t tc = grp; item(tc) < total && !failed; tc += kEpiGroups) {
            const uint32_t t = item(tc), tn = item(tc + kEpiGroups);
            const uint32_t buf = tc % kAcc, use = tc / kAcc;
            const Tile T = Tn;  // fetched one tile ahead, while the MMAs of this one run
            if (tn < total) Tn = tiles[tn / NV];
            int ok = 1;
            if (lane == 0) ok = mbar_wait(smem_u32(&tfull_bar[buf]), use & 1u) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);  // warp-uniform (tcgen05.ld is warp-collective)
            if (!ok) {
                failed = true;
                break;
            }
            __syncwarp();
            tc_fence_after();
            epilogue_tma<NSPLIT>(T, (int)(t % NV), tmem + buf * TMEM_COLS, w4, lane, B, smem_u32(&tempty_bar[buf]));
        }
    }
    if (failed) atomicExch(B.err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, kAcc * TMEM_COLS);
}

// ---------------------------------------------------------------------------
// TMA-staged kernel, one tile and one stage after the other
// ---------------------------------------------------------------------------
//
// The sums of short lists inside Davidson.  An output region receives one FP64 atomic
// addition per K-chunk, and from the third chunk on their order decides the last place
// of an element.  Davidson makes any figure of its vector out of such a place: its
// corrections r / (theta - H_ii) lie almost in the space that it has already, and what
// Gram-Schmidt leaves of them is normalised (K = 14, D = 600, eight steps from a random
// vector: 1e-16 becomes 1).  tc_tma_kernel finishes chunks in an order that changes from
// call to call in many regions; here one lane walks tile -> segment -> copies, so that a
// tile takes a time of its own (490 ns per 64-deep stage, 245 per segment, 3.9 us),
// repeatable to 0.3 us, and 99.4 % of all pairs of chunks keep their order: of 72
// calls (24 problems) 6 differ from their plan's first by over 1e-9, with tc_tma_kernel
// 17; and 100 of 108 give the vector that this schedule gave when it was the only one
// (101 of its own repeats did).  It costs 0.41 ms per sigma there (1.45 -> 1.86).
// Lists of more than kSerialItems products stay with tc_tma_kernel: no order repeats
// there (K = 24, D = 500, 550 000 products: two calls differ by order one after eight
// steps with either kernel).
//
// Its tiles are ordered by their stages alone and dealt in one direction, one CTA per
// SM, fixed stages of 128 x 64 rows per piece.

// 64 x 64 box of a 4-D tensor map (one piece) into shared memory, completion on an mbarrier
__device__ __forceinline__ void tma_load4(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w,
                                          uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
        : "memory");
}

// One 128 x 64 operand piece as (up to) two 64-row boxes, 8 KB apart.  K-major
// (mn = 0): rows r0.. of the map at x = k0; MN-major (mn = 1): columns r0.. of the map
// at rows k0..  halves = 1: the block ends within the first 64 (see tma_operand).
__device__ __forceinline__ void tma_piece(uint32_t dst, const CUtensorMap* map, int mn, int r0, int k0, int z, int w,
                                          uint32_t bar, int halves) {
    if (!mn) {
        tma_load4(dst, map, k0, r0, z, w, bar);
        if (halves == 2) tma_load4(dst + 8192, map, k0, r0 + 64, z, w, bar);
    } else {
        tma_load4(dst, map, r0, k0, z, w, bar);
        if (halves == 2) tma_load4(dst + 8192, map, r0 + 64, k0, z, w, bar);
    }
}

// Roles: warps 0-3 epilogue (as in tc_seg_gemm_kernel), warp 4 lane 0 TMA
// producer, warp 5 lane 0 MMA issuer.
constexpr int THREADS4 = (kEpiWarps + 2) * 32;

// stage record
struct StageMeta4 {
    uint8_t a_mn, b_mn, neg, flags;  // flags: 1 first stage of a tile, 2 last, 4 no MMA (empty tile)
    uint8_t k16, n16, pad[2];        // 16-deep K steps holding data; MMA N / 16
};

template <int NSPLIT>
__global__ void __launch_bounds__(THREADS4, 1)
    tc_serial_kernel(const Tile* __restrict__ tiles, int ntiles, int nvec, const TSeg* __restrict__ segs,
                     const CUtensorMap* __restrict__ maps, TcBufs B) {
    using C = Cfg2<NSPLIT>;
    constexpr int S = C::STAGES;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], tfull_bar[2], tempty_bar[2], drain_bar;
    __shared__ StageMeta4 meta[S];
    __shared__ uint32_t tmem_base_s;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (warp == 0) tmem_alloc(smem_u32(&tmem_base_s), 2 * TMEM_COLS);
    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&tfull_bar[b]), 1);
            mbar_init(smem_u32(&tempty_bar[b]), kEpiWarps);
        }
        mbar_init(smem_u32(&drain_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    const int total = ntiles * nvec;
    bool failed = false;

    if (warp == kEpiWarps) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t q = 0;
            for (int t = blockIdx.x; t < total && !failed; t += gridDim.x) {
                const int v = t % nvec;
                const Tile T = tiles[t / nvec];
                const int nst = T.nst;
                // a second 64-row (or 64-column) half only when the block extends past the first
                const int ncol = min((int)T.tn, T.n - T.n0);  // columns of this tile
                const int nA = (T.m - T.m0 > 64) ? 2 : 1, nB = (ncol > 64) ? 2 : 1;
                const int n16 = (ncol + 15) / 16;
                if (nst == 0) {
                    if (q >= (uint32_t)S && !mbar_wait(smem_u32(&empty_bar[q % S]), ((q / S) - 1) & 1u)) {
                        failed = true;
                        break;
                    }
                    meta[q % S] = StageMeta4{0, 0, 0, 1 | 2 | 4, 0, 0, {0, 0}};
                    mbar_arrive(smem_u32(&full_bar[q % S]));
                    ++q;
                    continue;
                }
                int done = 0;
                for (int s = T.seg_beg; s < T.seg_end && !failed; ++s) {
                    const TSeg Sg = segs[s];
                    const int a_mn = Sg.a_tr ? 1 : 0, b_mn = Sg.b_tr ? 0 : 1;
                    const int aw = Sg.a_pv ? v : 0, bw = Sg.b_pv ? v : 0;
                    const CUtensorMap* am = maps + NSPLIT * Sg.a_map;
                    const CUtensorMap* bm = maps + NSPLIT * Sg.b_map;
                    const uint32_t bytes = (uint32_t)NSPLIT * 128u * (uint32_t)(nA * Sg.a_br + nB * Sg.b_br);
                    for (int k0 = 0; k0 < Sg.k; k0 += TK) {
                        const uint32_t slot = q % S;
                        if (q >= (uint32_t)S && !mbar_wait(smem_u32(&empty_bar[slot]), ((q / S) - 1) & 1u)) {
                            failed = true;
                            break;
                        }
                        const int kv = min(TK, Sg.k - k0);
                        meta[slot] = StageMeta4{(uint8_t)a_mn, (uint8_t)b_mn, (uint8_t)(Sg.sign < 0.f ? 1 : 0),
                                                (uint8_t)((done == 0 ? 1 : 0) | (done == nst - 1 ? 2 : 0)),
                                                (uint8_t)((kv + 15) / 16), (uint8_t)n16, {0, 0}};
                        const uint32_t bar = smem_u32(&full_bar[slot]);
                        mbar_arrive_tx(bar, bytes);
                        const uint32_t sa = sbase + slot * C::STAGE_BYTES;
                        const uint32_t sb = sa + NSPLIT * PIECE_BYTES;
#pragma unroll
                        for (int pc = 0; pc < NSPLIT; ++pc) {
                            tma_piece(sa + pc * PIECE_BYTES, am + pc, a_mn, T.m0, k0, Sg.a_z, aw, bar, nA);
                            tma_piece(sb + pc * PIECE_BYTES, bm + pc, b_mn, T.n0, k0, Sg.b_z, bw, bar, nB);
                        }
                        ++q;
                        ++done;
                    }
                }
            }
        }
    } else if (warp == kEpiWarps + 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            uint32_t q = 0, tc = 0;
            for (int t = blockIdx.x; t < total && !failed; t += gridDim.x, ++tc) {
                const uint32_t buf = tc & 1u, use = tc >> 1;
                if (use > 0 && !mbar_wait(smem_u32(&tempty_bar[buf]), (use - 1) & 1u)) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const uint32_t dt = tmem + buf * TMEM_COLS;
                for (;;) {
                    const uint32_t slot = q % S;
                    if (!mbar_wait(smem_u32(&full_bar[slot]), (q / S) & 1u)) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    const StageMeta4 M = meta[slot];
                    if (!(M.flags & 4)) {
                        const uint32_t sa = sbase + slot * C::STAGE_BYTES;
                        const uint32_t sb = sa + NSPLIT * PIECE_BYTES;
                        const uint32_t id = idesc_n(M.a_mn, M.b_mn, M.neg, 16 * M.n16);
                        for (int kk = 0; kk < M.k16; ++kk) {
#pragma unroll
                            for (int pr = 0; pr < Prods<NSPLIT>::N; ++pr) {
                                const int pa = prod_a(pr), pb = prod_b(pr);
                                const uint32_t a_s = sa + pa * PIECE_BYTES;
                                const uint32_t b_s = sb + pb * PIECE_BYTES;
                                const uint64_t ad =
                                    M.a_mn ? sdesc(a_s + kk * 2048, 8192, 1024) : sdesc(a_s + kk * 32, 16, 1024);
                                const uint64_t bd =
                                    M.b_mn ? sdesc(b_s + kk * 2048, 8192, 1024) : sdesc(b_s + kk * 32, 16, 1024);
                                const uint32_t acc = ((M.flags & 1) && kk == 0 && pr == 0) ? 0u : 1u;
                                mma_bf16(dt, ad, bd, id, acc);
                            }
                        }
                    }
                    mma_commit(smem_u32(&empty_bar[slot]));
                    ++q;
                    if (M.flags & 2) break;
                }
                if (failed) break;
                mma_commit(smem_u32(&tfull_bar[buf]));
            }
            mma_commit(smem_u32(&drain_bar));
            if (!mbar_wait(smem_u32(&drain_bar), 0)) failed = true;
        }
    } else {
        // ---------------- epilogue ----------------
        uint32_t tc = 0;
        Tile Tn{};
        if (blockIdx.x < total) Tn = tiles[blockIdx.x / nvec];
        for (int t = blockIdx.x; t < total && !failed; t += gridDim.x, ++tc) {
            const uint32_t buf = tc & 1u, use = tc >> 1;
            const Tile T = Tn;  // fetched one tile ahead, while the MMAs of this one run
            if (t + (int)gridDim.x < total) Tn = tiles[(t + gridDim.x) / nvec];
            int ok = 1;
            if (lane == 0) ok = mbar_wait(smem_u32(&tfull_bar[buf]), use & 1u) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);  // warp-uniform (tcgen05.ld is warp-collective)
            if (!ok) {
                failed = true;
                break;
            }
            __syncwarp();
            tc_fence_after();
            epilogue_tile<NSPLIT>(T, t % nvec, T.nst, tmem + buf * TMEM_COLS, warp, lane, B,
                                  smem_u32(&tempty_bar[buf]));
        }
    }
    if (failed) atomicExch(B.err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 2 * TMEM_COLS);
}

// ---------------------------------------------------------------------------
// conversions
// ---------------------------------------------------------------------------

// x -> hi + lo + lo2: each piece is the bf16 rounding (through FP32) of what the
// previous ones leave.  Bound: HBM (14 bytes per element with two pieces) once
// the FP64 pipe is out of the way: conversions between FP64 and FP32 run there
// at ~2 per cycle and SM, and four of them per element took 180 us for 26
// million elements (79 us at the copy rate).  So x is rounded to FP32 by integer
// operations on its bits, and what that leaves, an integer of 29 bits in units
// of x's last place, is converted as an integer; the sums below are then those
// of FP32 numbers, exact but for their own rounding.
struct Pieces {
    __nv_bfloat16 h, l, m;
};
__device__ __forceinline__ Pieces split_pieces(double xd, bool three) {
    const uint32_t hi = (uint32_t)__double2hiint(xd), lo = (uint32_t)__double2loint(xd);
    const int eb = (int)((hi >> 20) & 0x7FFu);
    Pieces p;
    if (eb >= 1023 - 90 && eb < 1023 + 126) {
        uint32_t f = (hi & 0x80000000u) | ((uint32_t)(eb - 896) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
        const uint32_t rem = lo & 0x1FFFFFFFu;
        const uint32_t up = (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;  // to nearest even
        f += up;
        int left = (int)rem - (up ? 0x20000000 : 0);  // |x| - |f| in units of 2^(eb - 1075)
        if (hi >> 31) left = -left;
        const float xf = __uint_as_float(f);
        const float e = __int2float_rn(left) * 0x1p-52f * __uint_as_float((uint32_t)(eb - 896) << 23);
        p.h = __float2bfloat16_rn(xf);
        const float d = __fsub_rn(xf, __bfloat162float(p.h));
        p.l = __float2bfloat16_rn(__fadd_rn(d, e));
        p.m = __ushort_as_bfloat16((unsigned short)0);
        if (three) {
            const float t = __fadd_rn(__fsub_rn(d, __bfloat162float(p.l)), e);
            p.m = __float2bfloat16_rn(t);
            // e is off by up to 2^-25 of itself where left has more than 24 bits: too
            // little to matter unless t is close to the middle of two pieces or tiny
            // (0.1 % of random values; without this 7 third pieces in 10 million were
            // rounded the other way, enough to move a BF16X6 store by 1e-7)
            const uint32_t tb = __float_as_uint(t);
            if (abs(left) >= 1 << 24 && ((tb & 0xFFFFu) - 0x7FF8u <= 0x10u || (int)(tb >> 23 & 0xFFu) < eb - 896 - 28)) {
                const double r = xd - (double)__bfloat162float(p.h);
                p.m = __float2bfloat16_rn((float)(r - (double)__bfloat162float(p.l)));
            }
        }
    } else if ((hi << 1 | lo) == 0u) {
        p.h = __ushort_as_bfloat16((unsigned short)(hi >> 16));
        p.l = p.m = __ushort_as_bfloat16((unsigned short)0);
    } else {  // outside FP32's comfortable range, infinities, NaN
        p.h = __float2bfloat16_rn((float)xd);
        const double r = xd - (double)__bfloat162float(p.h);
        p.l = __float2bfloat16_rn((float)r);
        p.m = __float2bfloat16_rn((float)(r - (double)__bfloat162float(p.l)));
    }
    return p;
}
__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// n elements, then zeros up to ldd; VEC: four elements per thread and step
// (src 16-byte, pieces 8-byte aligned)
template <bool VEC>
__global__ void split_f64_flat_kernel(const double* __restrict__ src, int64_t n, int64_t ldd,
                                      __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                      __nv_bfloat16* __restrict__ lo2) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    const int64_t nv = VEC ? n / 4 : 0;
    const bool three = lo2 != nullptr;
    if (VEC) {
        for (int64_t i = t0; i < nv; i += nt) {
            const double2 a = ((const double2*)src)[2 * i], b = ((const double2*)src)[2 * i + 1];
            const Pieces p[4] = {split_pieces(a.x, three), split_pieces(a.y, three), split_pieces(b.x, three),
                                 split_pieces(b.y, three)};
            ((uint2*)hi)[i] = make_uint2(pack2(p[0].h, p[1].h), pack2(p[2].h, p[3].h));
            if (lo) ((uint2*)lo)[i] = make_uint2(pack2(p[0].l, p[1].l), pack2(p[2].l, p[3].l));
            if (lo2) ((uint2*)lo2)[i] = make_uint2(pack2(p[0].m, p[1].m), pack2(p[2].m, p[3].m));
        }
    }
    for (int64_t i = 4 * nv + t0; i < ldd; i += nt) {
        const Pieces p = split_pieces(i < n ? src[i] : 0.0, three);
        hi[i] = p.h;
        if (lo) lo[i] = p.l;
        if (lo2) lo2[i] = p.m;
    }
}

// one job per blockIdx.x, its rows dealt to the warps of gridDim.y blocks (one
// block per job left most SMs idle: K = 14, D = 600 has sectors of 13 000
// elements on 1.8 waves of blocks, 104 us for 0.6 million elements)
__global__ void split_blocks_kernel(const double* __restrict__ src, const SplitJob* __restrict__ jobs,
                                    __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                    __nv_bfloat16* __restrict__ lo2) {
    const SplitJob J = jobs[blockIdx.x];
    const int nw = blockDim.x / 32, lane = threadIdx.x & 31;
    const bool three = lo2 != nullptr;
    for (int r = blockIdx.y * nw + threadIdx.x / 32; r < J.rows; r += gridDim.y * nw) {
        const double* q = src + J.src_off + (int64_t)r * J.ld_src;
        const int64_t o = J.dst_off + (int64_t)r * J.ld_dst;  // offsets and leading dimensions are multiples of 8
        for (int c = 2 * lane; c < J.ld_dst; c += 64) {
            const Pieces a = split_pieces(c < J.cols ? q[c] : 0.0, three),
                         b = split_pieces(c + 1 < J.cols ? q[c + 1] : 0.0, three);
            *(uint32_t*)(hi + o + c) = pack2(a.h, b.h);
            if (lo) *(uint32_t*)(lo + o + c) = pack2(a.l, b.l);
            if (lo2) *(uint32_t*)(lo2 + o + c) = pack2(a.m, b.m);
        }
    }
}

int grid_for(int64_t n) {
    int64_t g = (n + 255) / 256;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

int tc_num_sms() {
    static int n = 0;
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 148;
    }
    return n;
}

void launch_seg_gemm_tc(const WorkList& w, const TcBufs& b, int nvec, int nsplit, cudaStream_t st) {
    if (w.tiles.empty()) return;
    const int64_t total = (int64_t)w.tiles.size() * nvec;
    DMRG_REQUIRE(total < (1LL << 31), DMRG_EINVAL, "tensor-core work list too large");
    DMRG_CHECK_CUDA(cudaMemsetAsync(b.counter, 0, sizeof(int), st));
    const int grid = (int)std::min<int64_t>(total, tc_num_sms());
    if (nsplit == 3) {
        static bool attr = false;
        if (!attr) {
            DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_seg_gemm_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 Cfg2<3>::SMEM));
            attr = true;
        }
        tc_seg_gemm_kernel<3><<<grid, THREADS2, Cfg2<3>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs, b);
    } else if (nsplit == 2) {
        static bool attr = false;
        if (!attr) {
            DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_seg_gemm_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 Cfg2<2>::SMEM));
            attr = true;
        }
        tc_seg_gemm_kernel<2><<<grid, THREADS2, Cfg2<2>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs, b);
    } else {
        static bool attr = false;
        if (!attr) {
            DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_seg_gemm_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 Cfg2<1>::SMEM));
            attr = true;
        }
        tc_seg_gemm_kernel<1><<<grid, THREADS2, Cfg2<1>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs, b);
    }
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// TMA work lists and tensor maps (host)
// ---------------------------------------------------------------------------

void TmaWorkList::add_block(int64_t c_off, int c_buf, int m, int n, int ldc, const std::vector<TSeg>& s, uint8_t mode,
                            int64_t kchunk, float alpha, int tn, bool tr) {
    if (m <= 0 || n <= 0) return;
    DMRG_REQUIRE(tn == 64 || tn == TN, DMRG_EINVAL, "tile width must be 64 or 128");
    DMRG_REQUIRE(!tr || (mode == TC_STORE_SPLIT && !s.empty()), DMRG_EINVAL, "only stored products are transposed");
    std::vector<std::pair<int, int>> chunks;
    const bool atomic = (mode == TC_ATOMIC_F64 || mode == TC_ATOMIC_F32);
    if (atomic && kchunk > 0) {
        int beg = 0;
        int64_t acc = 0;
        for (int i = 0; i < (int)s.size(); ++i) {
            if (acc > 0 && acc + s[i].k > kchunk) {
                chunks.push_back({beg, i});
                beg = i;
                acc = 0;
            }
            acc += s[i].k;
        }
        chunks.push_back({beg, (int)s.size()});
    } else {
        chunks.push_back({0, (int)s.size()});
    }
    for (auto& ch : chunks) {
        const int sb = (int)segs.size();
        int64_t nst = 0;
        for (int i = ch.first; i < ch.second; ++i) {
            segs.push_back(s[i]);
            nst += (s[i].k + TK - 1) / TK;
        }
        DMRG_REQUIRE(nst < 65536, DMRG_EINVAL, "tile with too many K stages (use a K-chunk)");
        const int se = (int)segs.size();
        for (int m0 = 0; m0 < m; m0 += TM)
            for (int n0 = 0; n0 < n; n0 += tn) {
                Tile t{};
                t.tn = (uint8_t)tn;
                t.alpha = alpha;
                t.c_off = c_off;
                t.ldc = ldc;
                t.m = m;
                t.n = n;
                t.m0 = m0;
                t.n0 = n0;
                t.seg_beg = sb;
                t.seg_end = se;
                t.c_buf = (uint8_t)c_buf;
                t.mode = mode;
                t.nst = (uint16_t)nst;
                t.tr = tr ? 1 : 0;
                tiles.push_back(t);
            }
    }
}

void TmaWorkList::add_stack(int64_t c_off, int c_buf, int m, int n, int ldc, const TSeg& s, float alpha, int sn, int sb,
                            int tn, bool tr) {
    if (m <= 0 || n <= 0 || sn <= 0) return;
    const int sbeg = (int)segs.size();
    segs.push_back(s);
    for (int n0 = 0; n0 < n; n0 += tn) {
        Tile t{};
        t.tn = (uint8_t)tn;
        t.sn = (uint8_t)sn;
        t.sb = (uint8_t)sb;
        t.tr = tr ? 1 : 0;
        t.alpha = alpha;
        t.c_off = c_off;
        t.ldc = ldc;
        t.m = m;
        t.n = n;
        t.n0 = n0;
        t.seg_beg = sbeg;
        t.seg_end = sbeg + 1;
        t.c_buf = (uint8_t)c_buf;
        t.mode = TC_STORE_SPLIT;
        t.nst = (uint16_t)((s.k + TK - 1) / TK);
        tiles.push_back(t);
    }
}

namespace {
// largest work first: a stable counting sort, two linear passes instead of an n log n
// sort of millions of records on every bond
template <typename Work>
std::vector<Tile> sorted_down(const std::vector<Tile>& tiles, const Work& work) {
    int maxn = 0;
    for (const Tile& t : tiles) maxn = std::max(maxn, work(t));
    std::vector<size_t> pos((size_t)maxn + 2, 0);
    for (const Tile& t : tiles) ++pos[(size_t)(maxn - work(t)) + 1];
    for (size_t i = 1; i < pos.size(); ++i) pos[i] += pos[i - 1];
    std::vector<Tile> sorted(tiles.size());
    for (const Tile& t : tiles) sorted[pos[(size_t)(maxn - work(t))]++] = t;
    return sorted;
}
}  // namespace

void TmaWorkList::order_tiles(bool serial) {
    single = true;
    for (const Tile& t : tiles) single = single && t.seg_end - t.seg_beg == 1;
    // Longest tiles first (stages, weighted by the rows and columns they load):
    // CTAs take the tiles in turn, back and forth, so the short ones fill in at
    // the end of the launch instead of a few long ones trailing.  (By stages alone
    // and in one direction the SMs idled 19 % of a K = 14, D = 600 phase 2: sigma
    // 1.52 -> 1.47 ms, K = 8, D = 64 199 -> 176 us.)
    by_stages.clear();
    if (serial) by_stages = sorted_down(tiles, [](const Tile& t) { return (int)t.nst; });
    tiles = sorted_down(tiles, [](const Tile& t) {
        const int rows = t.sn ? t.sn * 16 * t.sb : std::min(t.m - t.m0, TM);
        return (int)((int64_t)t.nst * (64 + rows + std::min<int>(t.tn, t.n - t.n0)) / 64);
    });
}

void TmaWorkList::upload(cudaStream_t st) {
    if (tiles.size() > cap_tiles) {
        if (d_tiles) cudaFree(d_tiles);
        cap_tiles = tiles.size() + 16;
        DMRG_CHECK_CUDA(dev_malloc(&d_tiles, cap_tiles * sizeof(Tile)));
    }
    if (segs.size() > cap_segs) {
        if (d_segs) cudaFree(d_segs);
        cap_segs = segs.size() + 16;
        DMRG_CHECK_CUDA(dev_malloc(&d_segs, cap_segs * sizeof(TSeg)));
    }
    if (by_stages.size() > cap_stages) {
        if (d_by_stages) cudaFree(d_by_stages);
        cap_stages = by_stages.size() + 16;
        DMRG_CHECK_CUDA(dev_malloc(&d_by_stages, cap_stages * sizeof(Tile)));
    }
    if (!by_stages.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_by_stages, by_stages.data(), by_stages.size() * sizeof(Tile),
                                        cudaMemcpyHostToDevice, st));
    if (!tiles.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_tiles, tiles.data(), tiles.size() * sizeof(Tile), cudaMemcpyHostToDevice, st));
    if (!segs.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_segs, segs.data(), segs.size() * sizeof(TSeg), cudaMemcpyHostToDevice, st));
}

void TmaWorkList::release() {
    if (d_tiles) cudaFree(d_tiles);
    if (d_segs) cudaFree(d_segs);
    if (d_by_stages) cudaFree(d_by_stages);
    d_tiles = nullptr;
    d_segs = nullptr;
    d_by_stages = nullptr;
    cap_tiles = cap_segs = cap_stages = 0;
}

int MapTable::get(const MapKey& k) {
    auto it = index.find(k);
    if (it != index.end()) return it->second;
    DMRG_REQUIRE(k.cols >= 1 && k.rows >= 1 && k.nz >= 1 && k.nv >= 1, DMRG_EINVAL, "empty tensor-map extent");
    DMRG_REQUIRE(k.off % 8 == 0 && k.ld % 8 == 0 && k.zstride % 8 == 0 && k.vstride % 8 == 0, DMRG_EINVAL,
                 "tensor-map operand not 16-byte aligned");
    DMRG_REQUIRE(k.ld >= k.cols && k.zstride >= k.rows * k.ld && k.vstride >= k.nz * k.zstride, DMRG_EINVAL,
                 "tensor-map strides overlap");
    const int i = (int)keys.size();
    keys.push_back(k);
    index[k] = i;
    return i;
}

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        DMRG_CHECK_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
        DMRG_REQUIRE(q == cudaDriverEntryPointSuccess && p, DMRG_ECUDA, "cuTensorMapEncodeTiled unavailable");
        fn = (EncodeTiledFn)p;
    }
    return fn;
}
}  // namespace

void MapTable::encode_upload(const TcBufs& tb, int nsplit, cudaStream_t st, bool serial) {
    const size_t n = kMapsPerKey * keys.size();
    std::vector<CUtensorMap> h(std::max<size_t>(n, 1));
    EncodeTiledFn fn = encode_fn();
    const auto encode = [fn](CUtensorMap& map, int nd, const __nv_bfloat16* base, const cuuint64_t* dims,
                             const cuuint64_t* strides, const cuuint32_t* box) {
        const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        const CUresult r = fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, nd, (void*)base, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        DMRG_REQUIRE(r == CUDA_SUCCESS, DMRG_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    };
    for (size_t i = 0; i < keys.size(); ++i) {
        const MapKey& k = keys[i];
        for (int m = 0; m < kMapsPerKey; ++m) {
            const bool tall = m >= 2, rest = m & 1;
            if ((tall && (k.rows <= 64 || k.bz > 1)) || (rest && nsplit != 3)) {  // unused: a copy of the first map
                h[kMapsPerKey * i + m] = h[kMapsPerKey * i];
                continue;
            }
            const __nv_bfloat16 *hi = tb.hi[k.buf], *lo = tb.lo[k.buf];
            const __nv_bfloat16* base = rest ? lo : hi;
            const int pieces = rest || nsplit == 2 ? 2 : 1;
            DMRG_REQUIRE(base && (nsplit == 1 || lo), DMRG_EINVAL, "tensor map over an unset buffer");
            const int64_t pst = pieces == 1 ? k.vstride : (rest ? tb.pstride[k.buf] : (int64_t)(lo - hi));
            DMRG_REQUIRE(pst > 0 && pst % 8 == 0 && pst * 2 < (1LL << 40), DMRG_EINVAL, "pieces not in one allocation");
            const cuuint64_t dims[5] = {(cuuint64_t)k.cols, (cuuint64_t)k.rows, (cuuint64_t)k.nz, (cuuint64_t)k.nv,
                                        (cuuint64_t)pieces};
            const cuuint64_t strides[4] = {(cuuint64_t)k.ld * 2, (cuuint64_t)k.zstride * 2, (cuuint64_t)k.vstride * 2,
                                           (cuuint64_t)pst * 2};
            const cuuint32_t box[5] = {64, tall ? 128u : (cuuint32_t)box_rows(k.rows), (cuuint32_t)k.bz, 1,
                                       (cuuint32_t)pieces};
            encode(h[kMapsPerKey * i + m], 5, base + k.off, dims, strides, box);
        }
    }
    // one piece per map, for launch_seg_gemm_serial (which runs no stacked products)
    std::vector<CUtensorMap> h1(serial ? (size_t)nsplit * keys.size() : 0);
    for (size_t i = 0; serial && i < keys.size(); ++i) {
        const MapKey& k = keys[i];
        if (k.bz > 1) continue;
        const cuuint64_t dims[4] = {(cuuint64_t)k.cols, (cuuint64_t)k.rows, (cuuint64_t)k.nz, (cuuint64_t)k.nv};
        const cuuint64_t strides[3] = {(cuuint64_t)k.ld * 2, (cuuint64_t)k.zstride * 2, (cuuint64_t)k.vstride * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)box_rows(k.rows), 1, 1};
        for (int pc = 0; pc < nsplit; ++pc) {
            const __nv_bfloat16* base = pc == 0 ? tb.hi[k.buf] : tb.lo[k.buf] + (pc == 2 ? tb.pstride[k.buf] : 0);
            encode(h1[(size_t)nsplit * i + pc], 4, base + k.off, dims, strides, box);
        }
    }
    if (h1.size() > cap1) {
        if (d_maps1) cudaFree(d_maps1);
        cap1 = h1.size() + 64;
        DMRG_CHECK_CUDA(dev_malloc(&d_maps1, cap1 * sizeof(CUtensorMap)));
    }
    if (!h1.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_maps1, h1.data(), h1.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice, st));
    if (n > cap) {
        if (d_maps) cudaFree(d_maps);
        cap = n + 64;
        DMRG_CHECK_CUDA(dev_malloc(&d_maps, cap * sizeof(CUtensorMap)));
    }
    if (n > 0) DMRG_CHECK_CUDA(cudaMemcpyAsync(d_maps, h.data(), n * sizeof(CUtensorMap), cudaMemcpyHostToDevice, st));
    DMRG_CHECK_CUDA(cudaStreamSynchronize(st));
    for (int b = 0; b < kMaxBufs; ++b) {
        enc_ptr[b][0] = tb.hi[b];
        enc_ptr[b][1] = tb.lo[b];
        enc_ptr[b][2] = tb.lo[b] ? tb.lo[b] + tb.pstride[b] : nullptr;
    }
}

bool MapTable::stale(const TcBufs& tb) const {
    if (!d_maps) return true;
    for (const MapKey& k : keys)
        if (enc_ptr[k.buf][0] != tb.hi[k.buf] || enc_ptr[k.buf][1] != tb.lo[k.buf] ||
            enc_ptr[k.buf][2] != (tb.lo[k.buf] ? tb.lo[k.buf] + tb.pstride[k.buf] : nullptr))
            return true;
    return false;
}

void MapTable::release() {
    if (d_maps) cudaFree(d_maps);
    if (d_maps1) cudaFree(d_maps1);
    d_maps = d_maps1 = nullptr;
    cap = cap1 = 0;
    clear();
}

void tc_prepare(int nsplit) {
    static bool done[4] = {false, false, false, false};
    if (nsplit < 1 || nsplit > 3 || done[nsplit]) return;
    if (nsplit == 1) {
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_tma_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg3<1>::SMEM));
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_serial_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg2<1>::SMEM));
    } else if (nsplit == 2) {
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_tma_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg3<2>::SMEM));
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_serial_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg2<2>::SMEM));
    } else {
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_tma_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg3<3>::SMEM));
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(tc_serial_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg2<3>::SMEM));
    }
    done[nsplit] = true;
}

void launch_seg_gemm_tma(const TmaWorkList& w, const MapTable& maps, const TcBufs& b, int nvec, int nsplit,
                         cudaStream_t st) {
    tc_prepare(nsplit);
    if (w.tiles.empty()) return;
    const int64_t total = (int64_t)w.tiles.size() * nvec;
    DMRG_REQUIRE(total < (1LL << 31), DMRG_EINVAL, "tensor-core work list too large");
    DMRG_REQUIRE(maps.d_maps != nullptr, DMRG_EINVAL, "tensor maps not uploaded");
    const int grid = (int)std::min<int64_t>(total, kCtas3 * tc_num_sms());
    const int single = w.single ? 1 : 0;
    if (nsplit == 3) {
        tc_tma_kernel<3><<<grid, THREADS3, Cfg3<3>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs,
                                                                maps.d_maps, single, b);
    } else if (nsplit == 2) {
        tc_tma_kernel<2><<<grid, THREADS3, Cfg3<2>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs,
                                                                maps.d_maps, single, b);
    } else {
        tc_tma_kernel<1><<<grid, THREADS3, Cfg3<1>::SMEM, st>>>(w.d_tiles, (int)w.tiles.size(), nvec, w.d_segs,
                                                                maps.d_maps, single, b);
    }
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void launch_seg_gemm_serial(const TmaWorkList& w, const MapTable& maps, const TcBufs& b, int nvec, int nsplit,
                            cudaStream_t st) {
    tc_prepare(nsplit);
    if (w.by_stages.empty()) return;
    const int64_t total = (int64_t)w.by_stages.size() * nvec;
    DMRG_REQUIRE(total < (1LL << 30), DMRG_EINVAL, "tensor-core work list too large");
    DMRG_REQUIRE(maps.d_maps1 != nullptr, DMRG_EINVAL, "tensor maps not uploaded");
    const int grid = (int)std::min<int64_t>(total, tc_num_sms()), n = (int)w.by_stages.size();
    if (nsplit == 3) tc_serial_kernel<3><<<grid, THREADS4, Cfg2<3>::SMEM, st>>>(w.d_by_stages, n, nvec, w.d_segs, maps.d_maps1, b);
    else if (nsplit == 2) tc_serial_kernel<2><<<grid, THREADS4, Cfg2<2>::SMEM, st>>>(w.d_by_stages, n, nvec, w.d_segs, maps.d_maps1, b);
    else tc_serial_kernel<1><<<grid, THREADS4, Cfg2<1>::SMEM, st>>>(w.d_by_stages, n, nvec, w.d_segs, maps.d_maps1, b);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_split_f64_flat(const double* src, int64_t n, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st,
                        __nv_bfloat16* lo2, int64_t n_pad) {
    n_pad = std::max(n, n_pad);
    if (n_pad <= 0) return;
    const bool vec = ((uintptr_t)src & 15) == 0 && (((uintptr_t)hi | (uintptr_t)lo | (uintptr_t)lo2) & 7) == 0;
    if (vec) split_f64_flat_kernel<true><<<grid_for((n_pad + 3) / 4), 256, 0, st>>>(src, n, n_pad, hi, lo, lo2);
    else split_f64_flat_kernel<false><<<grid_for(n_pad), 256, 0, st>>>(src, n, n_pad, hi, lo, lo2);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_split_blocks(const double* src, const SplitJob* d_jobs, int njobs, __nv_bfloat16* hi, __nv_bfloat16* lo,
                      cudaStream_t st, __nv_bfloat16* lo2) {
    if (njobs <= 0) return;
    split_blocks_kernel<<<dim3(njobs, 16), 256, 0, st>>>(src, d_jobs, hi, lo, lo2);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

}  // namespace dmrg
