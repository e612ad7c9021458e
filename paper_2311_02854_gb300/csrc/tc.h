// Tensor-core (tcgen05, sm_103a) segmented grouped GEMM on bf16 operand pieces.
#pragma once

#include <cuda.h>  // CUtensorMap (the encoder is fetched from the driver at run time)
#include <cuda_bf16.h>

#include <map>
#include <tuple>
#include <unordered_map>

#include "engine.h"

namespace dmrg {

// Output modes of the tensor-core engine (Tile::mode)
enum TcMode : uint8_t {
    TC_ATOMIC_F64 = 2,   // atomicAdd(double) of alpha * acc
    TC_STORE_SPLIT = 3,  // store alpha * acc as bf16 pieces (hi, lo) with the same offsets
    TC_ATOMIC_F32 = 4,   // atomicAdd(float)
    TC_STORE_F32 = 5,
};

// Operands: every buffer id holds `nsplit` bf16 pieces with identical layouts
// (x ~ hi + lo).  A segment's A / B are K-major (tr = 0) or MN-major (tr = 1).
struct TcBufs {
    const __nv_bfloat16* hi[kMaxBufs];
    const __nv_bfloat16* lo[kMaxBufs];
    int64_t pstride[kMaxBufs];  // three pieces: piece 2 at lo + pstride
    int64_t vstride[kMaxBufs];
    void* out[kMaxBufs];       // double* / float* / bf16 hi pieces (by mode)
    void* out_lo[kMaxBufs];    // bf16 lo pieces for TC_STORE_SPLIT
    int64_t out_pstride[kMaxBufs];
    int64_t out_vstride[kMaxBufs];
    int* counter;              // dynamic tile counter (zeroed before each launch)
    int* err;                  // device error word (0 = ok)
};

// Launch over the tiles of `w` (Seg::alpha must be +1 or -1: a sign applied
// through the MMA negate bit; Tile::alpha scales the epilogue).
void launch_seg_gemm_tc(const WorkList& w, const TcBufs& b, int nvec, int nsplit, cudaStream_t st);

int tc_num_sms();
// one-time kernel attributes (dynamic shared memory) of the nsplit kernels
void tc_prepare(int nsplit);

// ---------------------------------------------------------------------------
// TMA-staged variant: every operand is addressed through a tensor map.
// ---------------------------------------------------------------------------

// A segment whose operands are read through tensor maps.  Each map is 5-D:
// x = column, y = row, z = operator row of a stored family (0 otherwise), w =
// vector index (for per-vector buffers), then the bf16 piece, so that one copy
// brings both pieces.  A key has kMapsPerKey maps: boxes of up to 64 rows and, at
// 2, of 128 rows; with three pieces hi alone and, one further, (lo, lo2).
constexpr int kMapsPerKey = 4;
struct TSeg {
    int32_t a_map, b_map;  // map keys
    int32_t a_z, b_z;      // z coordinates
    int32_t k;             // K extent of the segment
    uint8_t a_tr, b_tr;    // a_tr: A held as K x M (MN-major); b_tr: B held as N x K (K-major)
    uint8_t a_pv, b_pv;    // 1: the operand's w coordinate is the vector index
    uint8_t a_br, b_br;    // rows of the maps' boxes (min(64, rows rounded up to 16))
    uint8_t a_bz;          // operator rows of A's boxes (stacked products: up to 8, else 1)
    uint8_t swap;          // the factors of the product trade sides: its cross terms run in the other order
    float sign;            // +1 or -1 (MMA negate bit)
};

struct TmaWorkList {
    std::vector<Tile> tiles;
    std::vector<TSeg> segs;
    Tile* d_tiles = nullptr;
    TSeg* d_segs = nullptr;
    size_t cap_tiles = 0, cap_segs = 0;
    bool single = false;  // every tile has one segment (set by order_tiles)
    // the tiles by stages alone, for launch_seg_gemm_serial (empty where that is not used)
    std::vector<Tile> by_stages;
    Tile* d_by_stages = nullptr;
    size_t cap_stages = 0;
    // output block (m x n, ld ldc) at c_off of c_buf, 128 x tn tiles (tn = 64 or
    // 128), split into K-chunks of at most kchunk (atomic modes only); tr: stored
    // transposed (TC_STORE_SPLIT only)
    void add_block(int64_t c_off, int c_buf, int m, int n, int ldc, const std::vector<TSeg>& s, uint8_t mode,
                   int64_t kchunk, float alpha, int tn = 128, bool tr = false);
    // sn stored products (m x n, ld ldc, one behind another from c_off on) of one tile
    // row: product i in accumulator rows i * 16 * sb ...
    void add_stack(int64_t c_off, int c_buf, int m, int n, int ldc, const TSeg& s, float alpha, int sn, int sb, int tn,
                   bool tr);
    void order_tiles(bool serial = false);  // longest tiles first (stable); serial: by_stages too
    void upload(cudaStream_t st);
    void release();
};

// A matrix as a tensor-map key: element (z, y, x) of vector w of buffer `buf`
// lives at off + w*vstride + z*zstride + y*ld + x (elements), x < cols, y < rows.
// Its boxes are 64 columns x box_rows(rows) rows x bz operator rows.
inline int box_rows(int64_t rows) { return rows >= 64 ? 64 : (int)((rows + 15) / 16 * 16); }
struct MapKey {
    int buf;
    int64_t off;
    int64_t cols, rows, ld, nz, zstride, nv, vstride;
    int bz = 1;  // operator rows of a box
    auto tie() const { return std::tie(buf, off, cols, rows, ld, nz, zstride, nv, vstride, bz); }
    bool operator<(const MapKey& o) const { return tie() < o.tie(); }
};

struct MapKeyHash {
    size_t operator()(const MapKey& k) const {
        uint64_t h = 0x9e3779b97f4a7c15ull ^ (uint64_t)k.buf;
        const int64_t v[9] = {k.off, k.cols, k.rows, k.ld, k.nz, k.zstride, k.nv, k.vstride, k.bz};
        for (int i = 0; i < 9; ++i) {
            h ^= (uint64_t)v[i] + 0x9e3779b97f4a7c15ull + (h << 6) + (h >> 2);
            h *= 0xff51afd7ed558ccdull;
        }
        return (size_t)(h ^ (h >> 33));
    }
};
struct MapKeyEq {
    bool operator()(const MapKey& a, const MapKey& b) const { return a.tie() == b.tie(); }
};

struct MapTable {
    std::vector<MapKey> keys;
    std::unordered_map<MapKey, int, MapKeyHash, MapKeyEq> index;
    CUtensorMap* d_maps = nullptr;   // kMapsPerKey per key
    CUtensorMap* d_maps1 = nullptr;  // 4-D, one per piece and key (launch_seg_gemm_serial)
    size_t cap = 0, cap1 = 0;
    const void* enc_ptr[kMaxBufs][3] = {};  // piece pointers the device maps were encoded with
    int get(const MapKey& k);  // validates alignment; returns the key index
    bool stale(const TcBufs& tb) const;  // a piece pointer moved since the last encode
    // encode the maps of every key (serial: those of launch_seg_gemm_serial too) and copy
    // them to the device
    void encode_upload(const TcBufs& tb, int nsplit, cudaStream_t st, bool serial);
    void clear() {
        keys.clear();
        index.clear();
    }
    void release();
};

// Launch the TMA-staged kernel over the tiles of `w` (maps on the device).
void launch_seg_gemm_tma(const TmaWorkList& w, const MapTable& maps, const TcBufs& b, int nvec, int nsplit,
                         cudaStream_t st);
// The same for the phase-2 tiles of lists of up to kSerialItems products, in an order of
// arrival that repeats from call to call (see tc_serial_kernel).
constexpr size_t kSerialItems = 1 << 18;
void launch_seg_gemm_serial(const TmaWorkList& w, const MapTable& maps, const TcBufs& b, int nvec, int nsplit,
                            cudaStream_t st);

// FP64 -> bf16 pieces (hi, lo, optionally lo2), same layout, n elements, then
// zeros up to n_pad (0: none); lo2 receives the third piece x - hi - lo
void dev_split_f64_flat(const double* src, int64_t n, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t st,
                        __nv_bfloat16* lo2 = nullptr, int64_t n_pad = 0);
// batched block copy FP64 -> pieces: for each job (src_off, dst_off, rows, cols, ld_src, ld_dst)
struct SplitJob {
    int64_t src_off, dst_off;
    int rows, cols, ld_src, ld_dst;
};
void dev_split_blocks(const double* src, const SplitJob* d_jobs, int njobs, __nv_bfloat16* hi, __nv_bfloat16* lo,
                      cudaStream_t st, __nv_bfloat16* lo2 = nullptr);

}  // namespace dmrg
