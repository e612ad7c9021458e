// FP64 kernels of libdmrg: the segmented grouped GEMM (every block product of
// the sigma step, the renormalisation, the intermediates and the density
// matrices; Sec. 2.2 "GEMM step" with the "reduction" fused into the
// accumulator) and the vector / Jacobi kernels of Davidson and decimation.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "engine.h"

namespace dmrg {

int64_t& launch_counter() {
    static int64_t c = 0;
    return c;
}

// ---------------------------------------------------------------------------
// Work lists
// ---------------------------------------------------------------------------

void WorkList::add_block(int64_t c_off, int c_buf, int m, int n, int ldc, const std::vector<Seg>& s,
                         uint8_t mode, int64_t kchunk, int tile, float alpha) {
    if (m <= 0 || n <= 0) return;
    // split segments into K-chunks (only for atomically accumulated blocks)
    std::vector<std::pair<int, int>> chunks;
    const bool atomic = (mode == TILE_ATOMIC || mode == 2 || mode == 4);
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
        int sb = (int)segs.size();
        for (int i = ch.first; i < ch.second; ++i) {
            segs.push_back(s[i]);
            flops += 2.0 * m * n * (double)s[i].k;
        }
        int se = (int)segs.size();
        const int tm = tile_m > 0 ? tile_m : tile, tn = tile_n > 0 ? tile_n : tile;
        for (int m0 = 0; m0 < m; m0 += tm)
            for (int n0 = 0; n0 < n; n0 += tn) {
                Tile t{};
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
                tiles.push_back(t);
            }
    }
}

void WorkList::add_stack(int64_t c_off, int c_buf, int m, int n, int ldc, const Seg& s, int64_t astride, int sn, int sb) {
    if (m <= 0 || n <= 0 || sn <= 0) return;
    DMRG_REQUIRE(std::abs(astride) < (1LL << 31), DMRG_EINVAL, "operators too far apart to be stacked");
    const int sbeg = (int)segs.size();
    segs.push_back(s);
    flops += 2.0 * sn * m * n * (double)s.k;
    for (int n0 = 0; n0 < n; n0 += tile_n) {
        Tile t{};
        t.astride = (int32_t)astride;
        t.sn = (uint8_t)sn;
        t.sb = (uint8_t)sb;
        t.c_off = c_off;
        t.ldc = ldc;
        t.m = m;
        t.n = n;
        t.n0 = n0;
        t.seg_beg = sbeg;
        t.seg_end = sbeg + 1;
        t.c_buf = (uint8_t)c_buf;
        t.mode = TILE_STORE;
        tiles.push_back(t);
    }
}

namespace {
constexpr int kSplitWarps = 4;  // warps of a CTA that share a part's term sum (FP64 units)
}

void WorkList::arrange() {
    // lists of the bf16-piece engine keep their order: its K-chunks are added as they
    // finish, and the rules below know the FP64 engines only
    if (!tiles.empty() && tiles[0].mode > TILE_ATOMIC) return;
    // work of a tile: 64-deep (FP64-accurate engine: oz_stage_depth) K steps, times
    // its rows and columns to convert plus a constant (by stages alone K = 24,
    // D = 500 took 18.8 ms instead of 17.8) or its 8 x 8 groups (FP64 units)
    const bool oz = tile_m == oz_tile_rows();
    const int tk = oz ? oz_stage_depth() : 64;
    std::vector<int> cost(tiles.size());
    int64_t total = 0;
    int maxn = 0;
    for (size_t i = 0; i < tiles.size(); ++i) {
        const Tile& t = tiles[i];
        int64_t n = 0;
        for (int s = t.seg_beg; s < t.seg_end; ++s) n += (segs[s].k + tk - 1) / tk;
        const int rows = t.sn ? t.sn * 16 * t.sb : std::min(t.m - t.m0, 128);
        if (oz) n = (n * (32 + rows + std::min(t.n - t.n0, 128)) + 31) / 32;
        else n *= (int64_t)((std::min(t.m - t.m0, 64) + 7) / 8) * ((std::min(t.n - t.n0, 64) + 7) / 8);
        cost[i] = (int)std::min<int64_t>(n, 1 << 20);
        total += cost[i];
        maxn = std::max(maxn, cost[i]);
    }
    // FP64 units.  Part of a tile per warp: 16 or 32 square where every tile ends
    // there, else 32 square, four per tile.  Several warps per part (split: CTAs of
    // four) when there are fewer parts than two per warp slot (12 on each of the
    // 152 SMs), or when the longest sum, on one warp, would take more than a
    // quarter of the launch; eight CTAs where even four warps per part do not fill
    // the slots and the sums are long (K = 10, D = 100: 250 outputs of ~300
    // products; 2.0 ms with four warps per part, see seg_split_f64_kernel).
    constexpr int64_t kSlots = 152 * 12;
    int mmax = 0, nmax = 0;
    int64_t parts = 0, segsum = 0, ksum = 0;
    for (const Tile& t : tiles) {
        const int m = std::min(t.m - t.m0, 64), n = std::min(t.n - t.n0, 64);
        mmax = std::max(mmax, m);
        nmax = std::max(nmax, n);
        parts += (int64_t)((m + 31) / 32) * ((n + 31) / 32);
        segsum += t.seg_end - t.seg_beg;
    }
    for (const Seg& g : segs) ksum += g.k;
    single = true;
    for (const Tile& t : tiles) single = single && t.seg_end - t.seg_beg == 1;
    part = std::max(mmax, nmax) <= 16 ? 16 : (std::max(mmax, nmax) <= 32 ? 32 : 64);
    split = 0;
    byk = false;
    if (!oz && !rank1 && !tiles.empty() && !segs.empty()) {
        const int64_t nt = (int64_t)tiles.size(), ns = (int64_t)segs.size();
        const bool few = parts < 2 * kSlots, longest = (int64_t)maxn * kSlots > total;
        byk = ksum / ns >= 32;  // a segment's K-blocks then feed four warps
        if ((few || longest) && (byk || segsum >= 8 * nt)) split = 1;
        if (split && !byk && parts * kSplitWarps < kSlots && segsum >= 64 * nt) split = 8;
    }
    // chains (seg_chain_f64_kernel): parts of 32 x 32, or smaller ones (16 x 16, 8 x 8,
    // 8 x 4) where that leaves the SMs without warps (fewer parts than kFill) or one warp
    // with a sum that outlasts its SM's share of the launch
    chain_part = 32;
    if (!oz && !rank1) {
        constexpr int64_t kSMs = 152, kFill = 8 * kSMs;
        for (; chain_part > 4; chain_part /= 2) {
            const int rows = std::max(chain_part, 8);
            int64_t np_all = 0, worst = 0;
            for (size_t i = 0; i < tiles.size(); ++i) {
                const int m = std::min(tiles[i].m - tiles[i].m0, 64), n = std::min(tiles[i].n - tiles[i].n0, 64);
                const int64_t np = (int64_t)((m + rows - 1) / rows) * ((n + chain_part - 1) / chain_part);
                np_all += np;
                worst = std::max(worst, cost[i] / np);
            }
            if (np_all >= kFill && worst * kSMs <= total) break;
        }
    }
    sub_m = (mmax + std::max(chain_part, 8) - 1) / std::max(chain_part, 8);
    sub_n = (nmax + chain_part - 1) / chain_part;
    if ((oz || split) && tiles.size() > 1) {
        // longest first (stable counting sort), so that short tiles fill in at the
        // end instead of a few long ones trailing
        std::vector<size_t> pos((size_t)maxn + 2, 0);
        for (int n : cost) ++pos[(size_t)(maxn - n) + 1];
        for (size_t i = 1; i < pos.size(); ++i) pos[i] += pos[i - 1];
        std::vector<Tile> sorted(tiles.size());
        for (size_t i = 0; i < tiles.size(); ++i) sorted[pos[(size_t)(maxn - cost[i])]++] = tiles[i];
        tiles.swap(sorted);
    }
}

void WorkList::upload(cudaStream_t st) {
    arrange();
    if (tiles.size() > cap_tiles) {
        if (d_tiles) cudaFree(d_tiles);
        cap_tiles = tiles.size() + tiles.size() / 4 + 16;
        DMRG_CHECK_CUDA(dev_malloc(&d_tiles, cap_tiles * sizeof(Tile)));
    }
    if (segs.size() > cap_segs) {
        if (d_segs) cudaFree(d_segs);
        cap_segs = segs.size() + segs.size() / 4 + 16;
        DMRG_CHECK_CUDA(dev_malloc(&d_segs, cap_segs * sizeof(Seg)));
    }
    if (!tiles.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_tiles, tiles.data(), tiles.size() * sizeof(Tile),
                                        cudaMemcpyHostToDevice, st));
    if (!segs.empty())
        DMRG_CHECK_CUDA(cudaMemcpyAsync(d_segs, segs.data(), segs.size() * sizeof(Seg),
                                        cudaMemcpyHostToDevice, st));
}

void WorkList::release() {
    if (d_tiles) cudaFree(d_tiles);
    if (d_segs) cudaFree(d_segs);
    d_tiles = nullptr;
    d_segs = nullptr;
    cap_tiles = cap_segs = 0;
}

// ---------------------------------------------------------------------------
// Segmented grouped GEMM on the FP64 units (64 x 64 tiles, 32 x 32 per warp)
// ---------------------------------------------------------------------------
//
// Bound: the FP64 units (1.05 TFLOP/s measured, as FMA or as mma.m8n8k4: one
// 8 x 8 x 4 product per ~140 cycles and SM).  The split follows from that:
// work is cut in 8 x 8 x 4 products and the ones outside the block are not
// issued (a 64 x 64 x 16 step computed in full spends 21 times a 10 x 10 x 10
// product, the usual size at small bonds, and 2.3 times a 42 x 42 one), and
// operands go from global memory to the fragments directly: at that rate the
// loads cost nothing and neither shared memory nor barriers are needed.  A warp
// owns a 32 x 32 part of a tile and is a CTA of its own, so that no warp's slot
// waits for a larger neighbour (2 x 2 warps per 64 x 64 tile kept the units 79 %
// busy, the ratio of the mean to the largest share of a 52 x 64 tile).

namespace {
constexpr int PT = 32;  // part of a tile per warp: 4 x 4 groups of 8 x 8 (2 x 2 where all tiles end within 16 x 16)

// element idx of buffer buf (FP64, or bf16 pieces read as hi + lo)
__device__ __forceinline__ double ld_elem(const BufTable& bt, int buf, int64_t idx) {
    if (bt.pmask & (1u << buf)) {
        const __nv_bfloat16* h = (const __nv_bfloat16*)bt.p[buf];
        double x = (double)__bfloat162float(h[idx]);
        if (bt.lo[buf]) {
            const __nv_bfloat16* l = (const __nv_bfloat16*)bt.lo[buf];
            x += (double)__bfloat162float(l[idx]);
            if (bt.pstride[buf]) x += (double)__bfloat162float(l[bt.pstride[buf] + idx]);
        }
        return x;
    }
    return bt.p[buf][idx];
}

// D (8 x 8) += A (8 x 4) B (4 x 8): lane l holds A(l / 4, l % 4), B(l % 4, l / 4)
// and D(l / 4, 2 (l % 4) + {0, 1})
__device__ __forceinline__ void mma884(double (&d)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};\n"
                 : "+d"(d[0]), "+d"(d[1])
                 : "d"(a), "d"(b));
}

// part `sub` (0: the only one of a tile within 32 x 32; else 2 x 2 per tile) of
// tile T: its origin in the block and its extents (not positive: nothing there)
struct Part {
    int m0, n0, mr, nr;
};
__device__ __forceinline__ Part tile_part(const Tile& T, int sub) {
    Part p;
    p.m0 = T.m0 + (sub >> 1) * PT;
    p.n0 = T.n0 + (sub & 1) * PT;
    p.mr = min(PT, T.m - p.m0);
    p.nr = min(PT, T.n - p.n0);
    return p;
}

// Sums to the part's output.  TILE_ATOMIC outputs are added to without atomics:
// one CTA owns each part, and the lists that add to the same output run one
// after the other, so every element's sum has one order and two calls agree to
// the bit.
template <int GR>
__device__ __forceinline__ void store_part(const Tile& T, const BufTable& bt, int v, const Part& p,
                                           const double (&acc)[GR][GR][2]) {
    const int lane = threadIdx.x & 31;
    double* C = bt.p[T.c_buf] + T.c_off + (int64_t)v * bt.vstride[T.c_buf];
#pragma unroll
    for (int i = 0; i < GR; ++i) {
        const int r = 8 * i + (lane >> 2);
        if (r >= p.mr) continue;
#pragma unroll
        for (int j = 0; j < GR; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = 8 * j + 2 * (lane & 3) + e;
                if (c >= p.nr) continue;
                double* dst = C + (int64_t)(p.m0 + r) * T.ldc + p.n0 + c;
                *dst = T.mode == TILE_ATOMIC ? *dst + acc[i][j][e] : acc[i][j][e];
            }
    }
}

// acc += the segments [sb, se) over part p; of each segment the K-blocks of
// 4 KU that are kf, kf + ks, ... of its own
template <int GR, int KU>
__device__ __forceinline__ void part_sum(const Seg* __restrict__ segs, const BufTable& bt, int v, int sb, int se,
                                         int kf, int ks, const Part& p, double (&acc)[GR][GR][2]) {
    const int lane = threadIdx.x & 31;
    const int lr = lane >> 2, lk = lane & 3;
    Seg N{};
    if (sb < se) N = segs[sb];
    for (int s = sb; s < se; ++s) {
        const Seg S = N;
        if (s + 1 < se) N = segs[s + 1];  // in flight during this segment
        // element (row, k) of op(A) at A + row * ra + k * ka, (k, col) of op(B) at B + k * kb + col * cb
        const int64_t ra = S.a_tr ? 1 : S.lda, ka = S.a_tr ? S.lda : 1;
        const int64_t cb = S.b_tr ? S.ldb : 1, kb = S.b_tr ? 1 : S.ldb;
        const int64_t A = S.a_off + (int64_t)v * bt.vstride[S.a_buf] + (p.m0 + lr) * ra + lk * ka;
        const int64_t B = S.b_off + (int64_t)v * bt.vstride[S.b_buf] + (p.n0 + lr) * cb + lk * kb;
        for (int k0 = 4 * KU * kf; k0 < S.k; k0 += 4 * KU * ks) {
            double a[KU][GR], b[KU][GR];
#pragma unroll
            for (int u = 0; u < KU; ++u) {
                const bool kv = k0 + 4 * u + lk < S.k;
#pragma unroll
                for (int i = 0; i < GR; ++i) {
                    a[u][i] = 0.0;
                    b[u][i] = 0.0;
                    if (kv && lr + 8 * i < p.mr) a[u][i] = ld_elem(bt, S.a_buf, A + 8 * i * ra + (k0 + 4 * u) * ka);
                    if (kv && lr + 8 * i < p.nr) b[u][i] = ld_elem(bt, S.b_buf, B + 8 * i * cb + (k0 + 4 * u) * kb);
                }
            }
            if (S.alpha != 1.0) {
#pragma unroll
                for (int u = 0; u < KU; ++u)
#pragma unroll
                    for (int i = 0; i < GR; ++i) a[u][i] *= S.alpha;
            }
#pragma unroll
            for (int u = 0; u < KU; ++u) {
                if (k0 + 4 * u >= S.k) break;
#pragma unroll
                for (int i = 0; i < GR; ++i)
#pragma unroll
                    for (int j = 0; j < GR; ++j)
                        if (8 * i < p.mr && 8 * j < p.nr) mma884(acc[i][j], a[u][i], b[u][j]);
            }
        }
    }
}

template <int GR, int KU>
__global__ void __launch_bounds__(32, GR == 2 ? 24 : 12)
    seg_gemm_f64_kernel(const Tile* __restrict__ tiles, int subs, const Seg* __restrict__ segs, BufTable bt) {
    const Tile T = tiles[blockIdx.x / subs];
    const Part p = tile_part(T, (int)(blockIdx.x % subs));
    if (p.mr <= 0 || p.nr <= 0) return;
    const int v = blockIdx.y;
    double acc[GR][GR][2] = {};
    part_sum<GR, KU>(segs, bt, v, T.seg_beg, T.seg_end, 0, 1, p, acc);
    store_part<GR>(T, bt, v, p, acc);
}

// The same with several warps per part: kSplit in a CTA, and with a cluster of
// CTAs that many times more.  Each takes a range of the tile's segments, or
// (byk: segments of some depth) its share of every segment's K-blocks; the
// partial sums are added in warp, then in rank order (through distributed
// shared memory).  For lists with fewer parts than the chip has warps, or whose
// longest term sums would outlast the rest of the launch: the sigma of a small
// bond has a few hundred outputs, each the sum of hundreds to thousands of
// products.
constexpr int kSplit = kSplitWarps;
template <int GR, int KU>
__global__ void __launch_bounds__(32 * kSplit, GR == 2 ? 5 : 3)
    seg_split_f64_kernel(const Tile* __restrict__ tiles, int subs, int nrank, int byk, const Seg* __restrict__ segs,
                         BufTable bt) {
    __shared__ double part[kSplit][GR * GR * 2][32];
    const int rank = (int)(blockIdx.x % nrank);  // clusters are runs of nrank blocks
    const uint32_t pi = blockIdx.x / nrank;
    const Tile T = tiles[pi / subs];
    const Part p = tile_part(T, (int)(pi % subs));
    if (p.mr <= 0 || p.nr <= 0) return;  // the whole cluster leaves
    const int v = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ns = T.seg_end - T.seg_beg;
    const int w = rank * kSplit + warp, nw = nrank * kSplit;
    double acc[GR][GR][2] = {};
    if (byk) part_sum<GR, KU>(segs, bt, v, T.seg_beg, T.seg_end, w, nw, p, acc);
    else part_sum<GR, KU>(segs, bt, v, T.seg_beg + (int)(ns * w / nw), T.seg_beg + (int)(ns * (w + 1) / nw), 0, 1, p, acc);
#pragma unroll
    for (int i = 0; i < GR; ++i)
#pragma unroll
        for (int j = 0; j < GR; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) part[warp][(i * GR + j) * 2 + e][lane] = acc[i][j][e];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int i = 0; i < GR; ++i)
#pragma unroll
            for (int j = 0; j < GR; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int q = 1; q < kSplit; ++q) acc[i][j][e] += part[q][(i * GR + j) * 2 + e][lane];
    }
    if (nrank > 1) {
        if (warp == 0) {
#pragma unroll
            for (int i = 0; i < GR; ++i)
#pragma unroll
                for (int j = 0; j < GR; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) part[0][(i * GR + j) * 2 + e][lane] = acc[i][j][e];
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
        if (warp == 0 && rank == 0) {
#pragma unroll
            for (int i = 0; i < GR; ++i)
#pragma unroll
                for (int j = 0; j < GR; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint32_t a = (uint32_t)__cvta_generic_to_shared(&part[0][(i * GR + j) * 2 + e][lane]);
                        for (int q = 1; q < nrank; ++q) {
                            uint32_t ra;
                            double x;
                            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(ra) : "r"(a), "r"(q));
                            asm volatile("ld.shared::cluster.f64 %0, [%1];\n" : "=d"(x) : "r"(ra) : "memory");
                            acc[i][j][e] += x;
                        }
                    }
        }
        // the partial sums stay until rank 0 has read them
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    }
    if (warp == 0 && rank == 0) store_part<GR>(T, bt, v, p, acc);
}

// The same product with one chain of fused multiply-adds per element, segment after
// segment and k after k (cut where its depth reaches the list's K-chunk, the pieces
// added in order): the sigma inside an FP64 Davidson call, which makes any figure of its
// vector out of a last place (see seg_outer_f64_kernel; products of four k's on the
// mma units with long sums shared among warps are off by 2e-15 of a sigma, and eight
// steps turned that into 1e-7 to 1e-2 of the vector in three of four problems).
//
// Bound: the FP64 units (89 % busy on K = 14, D = 600 first products), or for small
// bonds the longest chain, 63 ns per k.  What is shared among warps is the elements of a
// sum: a warp owns a part of 32 x 32 down to 8 x 4 of a tile.  Lane l = 4 r + c sums rows
// 8 i + r of columns 4 j + c.  Batches of KU k's, the next one in flight: of their operand
// elements a lane loads (and scales) KA of A and KB of B, one row and one column of its
// own at every few k's, and the lanes hand them to each other, so that a multiply-add
// comes with one or two other instructions (eighteen where each lane loaded all of its
// operands: sigma K = 14, D = 600 173 ms, now 93; 89 on the mma units).  Rows and columns
// outside the part read its last one and are dropped.
template <int GI, int GJ, int KU>
__global__ void __launch_bounds__(32, GI == 4 ? 12 : 20)
    seg_chain_f64_kernel(const Tile* __restrict__ tiles, int sub_m, int sub_n, int kchunk, const Seg* __restrict__ segs,
                        BufTable bt) {
    constexpr int UA = 4 / GI, UB = 8 / GJ;  // a lane's elements of A (B) are UA (UB) k's apart
    constexpr int KA = KU / UA, KB = KU / UB;
    const int subs = sub_m * sub_n;
    const Tile T = tiles[blockIdx.x / subs];
    const int sub = (int)(blockIdx.x % subs);
    Part p;
    p.m0 = T.m0 + sub / sub_n * 8 * GI;
    p.n0 = T.n0 + sub % sub_n * 4 * GJ;
    p.mr = min(8 * GI, min(T.m, T.m0 + 64) - p.m0);
    p.nr = min(4 * GJ, min(T.n, T.n0 + 64) - p.n0);
    if (p.mr <= 0 || p.nr <= 0) return;
    const int v = blockIdx.y, lane = threadIdx.x & 31, lr = lane >> 2, lc = lane & 3;
    const int arow = min(8 * (lc % GI) + lr, p.mr - 1), au = lc / GI;  // the lane's row of A, its first k
    const int bcol = min(4 * (lr % GJ) + lc, p.nr - 1), bu = lr / GJ;  // column of B
    double acc[GI][GJ] = {};
    // the chain so far to the output.  TILE_ATOMIC: added without atomics (one warp owns
    // the elements, and lists that add to the same output run one after the other)
    auto flush = [&]() {
        double* C = bt.p[T.c_buf] + T.c_off + (int64_t)v * bt.vstride[T.c_buf] + (int64_t)(p.m0 + lr) * T.ldc + p.n0 + lc;
#pragma unroll
        for (int i = 0; i < GI; ++i)
#pragma unroll
            for (int j = 0; j < GJ; ++j)
                if (8 * i + lr < p.mr && 4 * j + lc < p.nr) {
                    double* c = C + (int64_t)8 * i * T.ldc + 4 * j;
                    *c = T.mode == TILE_ATOMIC ? *c + acc[i][j] : acc[i][j];
                }
    };
    struct Batch {
        double a[KA], b[KB], alpha;
        int n;       // k's
        bool first;  // a new chain begins with it
    };
    // cursor: segment s (records one ahead in N), k's left of it, depth of the chain
    int s = T.seg_beg, left = 0, depth = 0;
    Seg N{};
    if (s < T.seg_end) N = segs[s];
    const double *pa = nullptr, *pb = nullptr;
    int64_t ka = 0, kb = 0;
    double alpha = 0.0;
    bool cut = false;
    auto open = [&]() {  // the next segment with products, if any
        left = 0;
        while (s < T.seg_end) {
            const Seg S = N;
            if (s + 1 < T.seg_end) N = segs[s + 1];
            if (kchunk > 0 && depth > 0 && depth + S.k > kchunk) {
                cut = true;
                depth = 0;
            }
            depth += S.k;
            if (S.k <= 0) {
                ++s;
                continue;
            }
            // element (row, k) of op(A) at A + row * ra + k * ka, (k, col) of op(B) at B + k * kb + col * cb
            const int64_t ra = S.a_tr ? 1 : S.lda, cb = S.b_tr ? S.ldb : 1;
            ka = S.a_tr ? S.lda : 1;
            kb = S.b_tr ? 1 : S.ldb;
            pa = bt.p[S.a_buf] + S.a_off + (int64_t)v * bt.vstride[S.a_buf] + (p.m0 + arow) * ra + au * ka;
            pb = bt.p[S.b_buf] + S.b_off + (int64_t)v * bt.vstride[S.b_buf] + (p.n0 + bcol) * cb + bu * kb;
            alpha = S.alpha;
            left = S.k;
            break;
        }
    };
    auto fetch = [&](Batch& x) {
        x.n = min(KU, left);
        x.first = cut;
        x.alpha = alpha;
        cut = false;
        if (left <= 0) return;
#pragma unroll
        for (int q = 0; q < KA; ++q) {
            x.a[q] = au + q * UA < left ? *pa : 0.0;
            pa += UA * ka;
        }
#pragma unroll
        for (int q = 0; q < KB; ++q) {
            x.b[q] = bu + q * UB < left ? *pb : 0.0;
            pb += UB * kb;
        }
        left -= KU;
        if (left <= 0) {
            ++s;
            open();
        }
    };
    Batch next;
    open();
    fetch(next);
    while (next.n > 0) {
        Batch x = next;
        fetch(next);
        if (x.first) {
            flush();
#pragma unroll
            for (int i = 0; i < GI; ++i)
#pragma unroll
                for (int j = 0; j < GJ; ++j) acc[i][j] = 0.0;
        }
        if (x.alpha != 1.0) {
#pragma unroll
            for (int q = 0; q < KA; ++q) x.a[q] *= x.alpha;
        }
#pragma unroll
        for (int u = 0; u < KU; ++u) {
            if (u >= x.n) break;
            double b[GJ];
#pragma unroll
            for (int j = 0; j < GJ; ++j) b[j] = __shfl_sync(0xffffffffu, x.b[u / UB], ((u % UB) * GJ + j) * 4 + lc);
#pragma unroll
            for (int i = 0; i < GI; ++i) {
                const double a = __shfl_sync(0xffffffffu, x.a[u / UA], (lane & 28) | ((u % UA) * GI + i));
                if (i > 0 && 8 * i >= p.mr) break;
#pragma unroll
                for (int j = 0; j < GJ; ++j)
                    if (j == 0 || 4 * j < p.nr) acc[i][j] = fma(a, b[j], acc[i][j]);
            }
        }
    }
    flush();
}

// The same product for lists whose segments all have K = 1 (rank-1 updates:
// the diagonal of H_eff as sums of diag(O_L) diag(O_R)^T, the two-electron
// integrals as a sum over Cholesky vectors).  Every element is one chain of fused
// multiply-adds in segment order: the correction step of Davidson divides by
// theta - H_ii, so a last place of the diagonal, or of the integrals behind it,
// can end up as any figure of its vector.  (Integrals summed by four warps each and
// a diagonal on mma.m8n8k4 moved the last place of one element in 14 000 at K = 14,
// D = 600, and took 396 us instead of 370 at K = 24, D = 500.)  Bound: the latency of the strided gathers (a diagonal is
// read with stride ld + 1) and, behind it, the FP64 units.  A CTA gathers the
// elements of 64 segments into shared memory with all its threads, one segment
// and operand each (32 loads in flight per thread); a thread then sums two rows,
// 16 apart, of four columns, 8 apart.
constexpr int kOuter = 64;
__global__ void __launch_bounds__(2 * kOuter)
    seg_outer_f64_kernel(const Tile* __restrict__ tiles, int subs, const Seg* __restrict__ segs, BufTable bt) {
    __shared__ double As[kOuter][PT + 1], Bs[kOuter][PT + 1];  // odd rows: a gathering warp writes without conflicts
    const Tile T = tiles[blockIdx.x / subs];
    const Part p = tile_part(T, (int)(blockIdx.x % subs));
    if (p.mr <= 0 || p.nr <= 0) return;
    const int v = blockIdx.y, tid = threadIdx.x;
    const int r0 = tid >> 3, c0 = tid & 7;  // the thread's first row and column
    const int ls = tid % kOuter;
    const bool isb = tid >= kOuter;
    double acc[2][4] = {};
    for (int s0 = T.seg_beg; s0 < T.seg_end; s0 += kOuter) {
        double x[PT];
        const bool sv = s0 + ls < T.seg_end;
        if (sv) {
            const Seg S = segs[s0 + ls];
            const int buf = isb ? S.b_buf : S.a_buf;
            const int64_t st = isb ? (S.b_tr ? S.ldb : 1) : (S.a_tr ? 1 : S.lda);
            const int64_t o = (isb ? S.b_off + p.n0 * st : S.a_off + p.m0 * st) + (int64_t)v * bt.vstride[buf];
            const int nx = isb ? p.nr : p.mr;
            const double al = isb ? 1.0 : S.alpha;
#pragma unroll
            for (int i = 0; i < PT; ++i) x[i] = i < nx ? ld_elem(bt, buf, o + i * st) * al : 0.0;
        } else {
#pragma unroll
            for (int i = 0; i < PT; ++i) x[i] = 0.0;
        }
        __syncthreads();  // the previous 64 segments have been used
#pragma unroll
        for (int i = 0; i < PT; ++i) (isb ? Bs : As)[ls][i] = x[i];
        __syncthreads();
        const int ne = min(kOuter, T.seg_end - s0);
        if ((r0 & ~3) < p.mr) {  // (a warp has four consecutive rows)
            for (int k = 0; k < ne; ++k) {
                double a[2], b[4];
#pragma unroll
                for (int i = 0; i < 2; ++i) a[i] = As[k][r0 + 16 * i];
#pragma unroll
                for (int j = 0; j < 4; ++j) b[j] = Bs[k][c0 + 8 * j];
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if ((r0 & ~3) + 16 * i < p.mr && 8 * j < p.nr) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
    }
    double* C = bt.p[T.c_buf] + T.c_off + (int64_t)v * bt.vstride[T.c_buf];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = r0 + 16 * i, c = c0 + 8 * j;
            if (r >= p.mr || c >= p.nr) continue;
            double* dst = C + (int64_t)(p.m0 + r) * T.ldc + p.n0 + c;
            *dst = T.mode == TILE_ATOMIC ? *dst + acc[i][j] : acc[i][j];
        }
}
}  // namespace

static void launch_chains(const WorkList& w, dim3 grid, const Tile* tiles, const BufTable& bt, cudaStream_t st) {
    auto kernel = w.chain_part == 32   ? seg_chain_f64_kernel<4, 8, 4>
                  : w.chain_part == 16 ? seg_chain_f64_kernel<2, 4, 4>
                  : w.chain_part == 8  ? seg_chain_f64_kernel<1, 2, 16>
                                       : seg_chain_f64_kernel<1, 1, 16>;
    kernel<<<grid, 32, 0, st>>>(tiles, w.sub_m, w.sub_n, w.kchunk, w.d_segs, bt);
}

void launch_seg_gemm_f64(const WorkList& w, const BufTable& bt, int nvec, cudaStream_t st, bool chains) {
    if (w.tiles.empty()) return;
    if (w.tile_m == oz_tile_rows() && !w.rank1) {
        launch_seg_gemm_oz(w, bt, nvec, st);
        return;
    }
    DMRG_REQUIRE(w.tile_m == 0, DMRG_EINVAL, "work list tile shape not runnable on the FP64 engine");
    DMRG_REQUIRE(nvec <= 65535, DMRG_EINVAL, "too many vectors for one launch");
    chains = chains && !w.rank1;
    DMRG_REQUIRE(!chains || bt.pmask == 0, DMRG_EINVAL, "chains are summed over FP64 buffers only");
    const int subs = chains ? w.sub_m * w.sub_n : (w.part == 64 ? 4 : 1);
    const bool tiny = w.part == 16;
    const int nrank = w.split && !chains ? w.split : 1;
    const int64_t n = (int64_t)w.tiles.size(), maxt = 2147483647LL / (subs * nrank);
    for (int64_t t0 = 0; t0 < n; t0 += maxt) {
        const int64_t nt = std::min(n - t0, maxt);
        const dim3 grid((unsigned)(nt * subs * nrank), (unsigned)nvec);
        const Tile* tl = w.d_tiles + t0;
        if (w.rank1) {
            seg_outer_f64_kernel<<<grid, 2 * kOuter, 0, st>>>(tl, subs, w.d_segs, bt);
        } else if (chains) {
            launch_chains(w, grid, tl, bt, st);
        } else if (w.split) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = grid;
            cfg.blockDim = dim3(32 * kSplit);
            cfg.stream = st;
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = (unsigned)nrank;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            DMRG_CHECK_CUDA(cudaLaunchKernelEx(&cfg, tiny ? seg_split_f64_kernel<2, 4> : seg_split_f64_kernel<4, 2>, tl, subs,
                                               nrank, (int)w.byk, (const Seg*)w.d_segs, bt));
        } else {
            (tiny ? seg_gemm_f64_kernel<2, 4> : seg_gemm_f64_kernel<4, 2>)<<<grid, 32, 0, st>>>(tl, subs, w.d_segs, bt);
        }
        ++launch_counter();
    }
    DMRG_CHECK_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Vector kernels
// ---------------------------------------------------------------------------

namespace {

__device__ double block_sum(double x, double* sh) {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = x;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sh[i];
    return t;  // valid in thread 0
}

__global__ void dots_stage1(const double* __restrict__ X, int64_t ldx, const double* __restrict__ y,
                            int64_t n, double* __restrict__ part, int nblk) {
    __shared__ double sh[32];
    const int i = blockIdx.y;
    double acc = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)nblk * blockDim.x)
        acc = fma(X[(int64_t)i * ldx + k], y[k], acc);
    double t = block_sum(acc, sh);
    if (threadIdx.x == 0) part[(int64_t)i * nblk + blockIdx.x] = t;
}

__global__ void dots_stage2(const double* __restrict__ part, int nblk, double* __restrict__ out) {
    __shared__ double sh[32];
    const int i = blockIdx.x;
    double acc = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) acc += part[(int64_t)i * nblk + b];
    double t = block_sum(acc, sh);
    if (threadIdx.x == 0) out[i] = t;
}

__global__ void combine_kernel(const double* __restrict__ X, int64_t ldx, int m, const double* __restrict__ c,
                               int64_t n, double* __restrict__ y) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int i = 0; i < m; ++i) acc = fma(c[i], X[(int64_t)i * ldx + k], acc);
        y[k] = acc;
    }
}

__global__ void axpby_kernel(double a, const double* __restrict__ x, double b, double* __restrict__ y, int64_t n) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        y[k] = a * x[k] + b * y[k];
}

__global__ void precond_kernel(const double* __restrict__ r, const double* __restrict__ d, double theta,
                               double* __restrict__ t, int64_t n) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        double den = d[k] - theta;
        if (fabs(den) < 1e-8) den = (den < 0.0) ? -1e-8 : 1e-8;
        t[k] = -r[k] / den;
    }
}

__global__ void fill_kernel(double* x, double v, int64_t n) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        x[k] = v;
}

__global__ void perturb_kernel(double* x, int64_t n, uint32_t seed, double amp) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t h = (uint32_t)k * 2654435761u ^ (seed * 2246822519u);
        h ^= h >> 15;
        h *= 2246822519u;
        h ^= h >> 13;
        h *= 3266489917u;
        h ^= h >> 16;
        x[k] += amp * ((double)h * (1.0 / 4294967296.0) - 0.5);
    }
}

__global__ void identity_kernel(double* x, int n) {
    const int64_t nn = (int64_t)n * n;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nn; k += (int64_t)gridDim.x * blockDim.x)
        x[k] = (k / n == k % n) ? 1.0 : 0.0;
}

int grid_for(int64_t n, int threads = 256) {
    int64_t g = (n + threads - 1) / threads;
    if (g > 152 * 32) g = 152 * 32;
    return (int)(g < 1 ? 1 : g);
}

}  // namespace

void dev_dots(const double* X, int64_t ldx, int m, const double* y, int64_t n, double* out, double* work,
              cudaStream_t st) {
    if (m <= 0) return;
    int nblk = (int)((n + 256 * 8 - 1) / (256 * 8));
    if (nblk > 256) nblk = 256;
    if (nblk < 1) nblk = 1;
    dots_stage1<<<dim3(nblk, m), 256, 0, st>>>(X, ldx, y, n, work, nblk);
    dots_stage2<<<m, 256, 0, st>>>(work, nblk, out);
    launch_counter() += 2;
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_combine(const double* X, int64_t ldx, int m, const double* c, int64_t n, double* y, cudaStream_t st) {
    combine_kernel<<<grid_for(n), 256, 0, st>>>(X, ldx, m, c, n, y);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_axpby(double a, const double* x, double b, double* y, int64_t n, cudaStream_t st) {
    axpby_kernel<<<grid_for(n), 256, 0, st>>>(a, x, b, y, n);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_jacobi_precond(const double* r, const double* d, double theta, double* t, int64_t n, cudaStream_t st) {
    precond_kernel<<<grid_for(n), 256, 0, st>>>(r, d, theta, t, n);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_fill(double* x, double v, int64_t n, cudaStream_t st) {
    if (n <= 0) return;
    fill_kernel<<<grid_for(n), 256, 0, st>>>(x, v, n);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_perturb(double* x, int64_t n, uint32_t seed, double amp, cudaStream_t st) {
    perturb_kernel<<<grid_for(n), 256, 0, st>>>(x, n, seed, amp);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

void dev_identity(double* x, int n, cudaStream_t st) {
    identity_kernel<<<grid_for((int64_t)n * n), 256, 0, st>>>(x, n);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Batched cyclic Jacobi eigensolver (round-robin ordering), one CTA per matrix
// (Golub & Van Loan, Alg. 8.4.3 with parallel ordering).
// ---------------------------------------------------------------------------

namespace {
constexpr int kJacThreads = 512;

__global__ void __launch_bounds__(kJacThreads) jacobi_eigh_kernel(const EigJob* __restrict__ jobs, int max_sweeps) {
    const EigJob J = jobs[blockIdx.x];
    const int n = J.n, lda = J.lda;
    double* __restrict__ A = J.A;
    double* __restrict__ V = J.V;
    extern __shared__ double sm[];
    const int ne = n + (n & 1);
    const int np = ne / 2;
    double* cs = sm;            // np
    double* sn = sm + np;       // np
    int* pp = (int*)(sm + 2 * np);
    int* qq = pp + np;
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int64_t idx = tid; idx < (int64_t)n * n; idx += nt) {
        int i = (int)(idx / n), j = (int)(idx % n);
        V[(int64_t)i * lda + j] = (i == j) ? 1.0 : 0.0;
    }
    __syncthreads();
    if (n <= 1) {
        if (tid == 0 && n == 1) J.w[0] = A[0];
        return;
    }
    // threshold Jacobi: a pair is rotated only if |a_pq| > eps * sqrt(|a_pp a_qq|)
    // (relative accuracy of small eigenvalues); stop after a sweep without rotations
    __shared__ int rotated;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        if (tid == 0) rotated = 0;
        __syncthreads();
        for (int r = 0; r < ne - 1; ++r) {
            for (int t = tid; t < np; t += nt) {
                int a, b;
                if (t == 0) {
                    a = r % (ne - 1);
                    b = ne - 1;
                } else {
                    a = (r + t) % (ne - 1);
                    b = (r + ne - 1 - t) % (ne - 1);
                }
                int p = a < b ? a : b, q = a < b ? b : a;
                double c = 1.0, s = 0.0;
                if (q < n) {
                    const double apq = A[(int64_t)p * lda + q];
                    const double app = A[(int64_t)p * lda + p], aqq = A[(int64_t)q * lda + q];
                    if (fabs(apq) > 1e-15 * sqrt(fabs(app * aqq)) && fabs(apq) > 1e-300) {
                        double tau = (aqq - app) / (2.0 * apq);
                        double tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                        c = 1.0 / sqrt(1.0 + tt * tt);
                        s = tt * c;
                        rotated = 1;
                    }
                }
                cs[t] = c;
                sn[t] = s;
                pp[t] = p;
                qq[t] = (q < n) ? q : -1;
            }
            __syncthreads();
            // rows: A <- J^T A
            for (int64_t idx = tid; idx < (int64_t)np * n; idx += nt) {
                int t = (int)(idx / n), k = (int)(idx % n);
                int q = qq[t];
                double s = sn[t];
                if (q < 0 || s == 0.0) continue;
                int p = pp[t];
                double c = cs[t];
                double x = A[(int64_t)p * lda + k], y = A[(int64_t)q * lda + k];
                A[(int64_t)p * lda + k] = c * x - s * y;
                A[(int64_t)q * lda + k] = s * x + c * y;
            }
            __syncthreads();
            // columns: A <- A J, V <- V J
            for (int64_t idx = tid; idx < (int64_t)np * n; idx += nt) {
                int t = (int)(idx / n), k = (int)(idx % n);
                int q = qq[t];
                double s = sn[t];
                if (q < 0 || s == 0.0) continue;
                int p = pp[t];
                double c = cs[t];
                double x = A[(int64_t)k * lda + p], y = A[(int64_t)k * lda + q];
                A[(int64_t)k * lda + p] = c * x - s * y;
                A[(int64_t)k * lda + q] = s * x + c * y;
                x = V[(int64_t)k * lda + p];
                y = V[(int64_t)k * lda + q];
                V[(int64_t)k * lda + p] = c * x - s * y;
                V[(int64_t)k * lda + q] = s * x + c * y;
            }
            __syncthreads();
        }
        if (!rotated) break;
        __syncthreads();
    }
    for (int i = tid; i < n; i += nt) J.w[i] = A[(int64_t)i * lda + i];
}
}  // namespace

void dev_jacobi_eigh_batched(const EigJob* d_jobs, int njobs, int max_sweeps, cudaStream_t st) {
    if (njobs <= 0) return;
    // shared memory sized for matrices up to 4096
    const int maxn = 4096;
    size_t smem = (size_t)(maxn / 2) * (2 * sizeof(double) + 2 * sizeof(int));
    static bool attr = false;
    if (!attr) {
        DMRG_CHECK_CUDA(cudaFuncSetAttribute(jacobi_eigh_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem));
        attr = true;
    }
    jacobi_eigh_kernel<<<njobs, kJacThreads, smem, st>>>(d_jobs, max_sweeps);
    ++launch_counter();
    DMRG_CHECK_CUDA(cudaGetLastError());
}

}  // namespace dmrg
