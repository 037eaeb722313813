#pragma once
// fxpq_conv_tc.cuh -- the C-Block contraction (Sec. IV-B) on the 5th-generation tensor cores.
//
// Implicit GEMM: rows = output pixels (N*P*Q), columns = output channels K, reduction over the
// flattened (r, s, c) taps of one code plane.  Operands are fp16 values that are exact integer
// codes (|code| <= 255 per limb), multiplied by tcgen05.mma .kind::f16 into fp32 TMEM
// accumulators.  fp32 accumulation is exact while every partial sum stays below 2^24, so the host
// splits the reduction into groups ("chunks") whose worst-case magnitude max|a| * max|w| * K_chunk
// is below 2^24; after each group the epilogue warps drain the accumulator, convert it to an
// integer (exact) and add it, shifted by the limb weight (0, 8 or 16 bits), into integer running
// sums.  The same grouping carries the two-limb split of 9..16-bit codes
// (v = 256 * v_hi + v_lo): one pass per (A limb, W limb) pair.
//
// CTA (one per SM, persistent over tiles):
//   warps 0-3  producers, into 128-byte swizzled K-major shared-memory stages.  The B tile
//              (BN channels x 64 taps) always comes by TMA.  The A tile takes one of these forms:
//              row tiles (128 consecutive output pixels): cp.async gather by 128 threads, with
//              zero fill for padding and ragged edges, or one box where the layer's im2col rows are
//              the stored activations;
//              patch tiles: a TH x TW patch of output pixels of TN images, whose inputs for one tap
//              and 64 channels are a single 5-D TMA box, strided like the convolution (the
//              hardware zero-fills the padding); the warps that issue copies own the stages in turn;
//              windows: see the patch values 3 and 4 of TcParams.
//   next 8 to 16 (BN / 8; 16 in the window instances)
//              epilogue: drain TMEM (tcgen05.ld), integer running sums, final bias / ReLU /
//              FxP-QLayer (shared with the CUDA-core kernel), or fp32 codes where the sums allow it.
//   then one   TMEM allocation and MMA issue (the whole warp, one elected lane per instruction),
//   one more   the TMA stores of staged tiles (BN <= 128), or five converters of packed weights.
// Every wait is bounded: on expiry the kernel latches FXPQ_ERR_TIMEOUT, stops issuing work,
// drains its own copies and MMAs, frees TMEM and returns.
// The kernel is a template over the tile width, the integer type of the running sums and whether
// the layer carries a Scale layer (SC): fxpq_conv_tc.cu instantiates the SC = false kernels and the
// host side, fxpq_conv_tc_scale.cu the SC = true ones, so that the two compile in parallel and the
// Scale layer's epilogue costs the other layers nothing.
#include <cuda.h>  // CUtensorMap and its enums (the encoder is fetched through the runtime)
#include <climits>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "fxpq_common.cuh"
#include "fxpq_conv.cuh"

namespace fxpq {
namespace tc {


constexpr int TC_BM = 128;
constexpr int TC_BK = 64;  // fp16 elements per k-block row = 128 bytes (one swizzle atom row)
// Pipeline depth: 6 stages of 24 or 32 KB (BN <= 128); 4 of 48 KB for BN = 256, whose one-plane codes are
// stored through per-warp 2 KB slices (no TMA-store staging of the whole tile) so that the output
// staging keeps only 32 KB; 3 for the packed-weight instance, whose packed stages take the 64 KB
// staging region.  (The 256-column layers lose about a fifth of their speed from 3 stages to 2: the
// copies' latency, not the tensor pipe, bounds them at this depth.)
__host__ __device__ constexpr int tc_stages(int BN, bool PK = false) { return BN == 256 ? (PK ? 3 : 4) : 6; }
// Output staging: tiles of BN / 64 boxes of 128 rows x 128 bytes for the TMA-store epilogue, two of them for
// BN = 64 (the sixth stage is worth more than a second 32 KB tile for BN = 128), 32 KB where
// the codes are stored directly (BN = 256 without packed weights).
__host__ __device__ constexpr int tc_out_bytes(int BN, bool PK = false) { return (BN == 256 && PK) ? 65536 : 32768; }
__host__ __device__ constexpr int tc_stg_tiles(int BN) { return BN == 64 ? 2 : 1; }
// Row-tile producers arrive on a stage this many k-blocks after issuing its copies (cp.async groups
// in flight).  It must stay below the stage count: a producer waiting for a stage to be consumed
// must already have arrived on it.
__host__ __device__ constexpr int tc_lag(int BN, bool PK = false) { return tc_stages(BN, PK) - 1 < 3 ? tc_stages(BN, PK) - 1 : 3; }
// Warps: 4 producers, epilogue warps (four per 32-column chunk group: one per TMEM lane quadrant;
// BN / 8 of them up to 16, each then draining BN / 128 chunks), one MMA / TMEM-allocation warp.
__host__ __device__ constexpr int tc_epi_warps(int BN) { return BN / 8 < 16 ? BN / 8 : 16; }
// and, where whole tiles are stored by TMA (BN <= 128), one warp that issues these stores.
__host__ __device__ constexpr int tc_threads(int BN) { return (5 + (BN <= 128 ? 1 : 0) + tc_epi_warps(BN)) * 32; }
// Packed weights (PK instances, BN = 256 only): the weights arrive as k-bit records (k <= 8) and these
// extra warps after the MMA warp, with producer warps 1-3, expand every k-block's records into the
// fp16 B stage.  The packed stages live in the output staging region, which PK layers do not use.
constexpr int TC_PK_WARPS = 5;
constexpr int TC_PK_CONVERTERS = 3 + TC_PK_WARPS;  // converter warps
__host__ __device__ constexpr int tc_threads_pk(int BN, bool pk) { return tc_threads(BN) + (pk ? 32 * TC_PK_WARPS : 0); }
// Window-mode instance (WIN, BN = 64, two-limb x and w, 32-bit epilogue): 16 epilogue warps of 16 columns
// each and two output staging tiles.
constexpr int TC_WIN_EPI_WARPS = 16;
// W64 instance (64-channel window mode) shared memory: resident weights (up to 9 taps of 8 KiB) and two
// window slots of up to 3 copies of 18 rows x 8 pixels x 128 bytes from the start, the two staging tiles
// at W64_SO.
constexpr int TC_W64_SO = 180 * 1024;
constexpr size_t tc_smem_w64() { return 1024 + TC_W64_SO + 2 * 64 * TC_BM * 2 + 256; }
__host__ __device__ constexpr int tc_threads_win() { return (6 + TC_WIN_EPI_WARPS) * 32; }
// Dynamic shared memory: barriers, the stages (A and B tiles), the output staging tile.
template <int BN, bool PK = false>
constexpr size_t tc_smem_bytes() {
    return 1024 + tc_stages(BN, PK) * (TC_BM * TC_BK * 2 + BN * TC_BK * 2) + tc_out_bytes(BN, PK) + 256;
}
static_assert(tc_smem_bytes<256>() <= 232448 && tc_smem_bytes<256, true>() <= 232448 && tc_smem_bytes<128>() <= 232448,
              "dynamic shared memory within the 227 KB a CTA may use");
constexpr int TC_MAX_GROUPS = 64;
constexpr int TC_MAX_SPLIT = 16;
constexpr long long TC_WAIT_CYCLES = 4000000000LL;  // ~2 s at 2 GHz
// TMA-issuing warps of patch and TMA row tiles (warps 0 .. n-1).  Producer p issues the k-blocks of the
// stages s with s % n == p (n divides the stage count), so every use of a stage comes from one warp, in
// order, and its parity wait on the stage's `empty` barrier is never more than one phase ahead of it.
// (A parity wait two phases ahead reads as complete: with k-blocks dealt round-robin, more producers
// than stages could refill a stage before its data was consumed.)  A warp's latency per k-block (the
// barrier round, two copies) would bound the rate: one warp for the A and one for the B boxes of every
// stage took 880 cycles per k-block of 128-column tiles where two that share the stages take 650.
__host__ __device__ constexpr int tc_producers(int BN, bool PK = false) {
    return tc_stages(BN, PK) <= 4 ? tc_stages(BN, PK) : 2;
}

struct TcGroup {
    int kb0, kb1;          // k-block range within a plane
    int a_plane, w_plane;  // limb planes (0 = hi or the only plane, 1 = lo)
    int shift;             // weight of this pass: 0, 8 or 16 bits
};

struct TcParams {
    CUtensorMap tmap_w;  // weights as [planes][K][R*S*Cp] fp16, box {64, BN, 1}, 128-byte swizzle
    CUtensorMap tmap_w2; // rows2 > 0: the same with a box of rows2 channels, for the last column tile (a TMA box is
    int rows2;           // slow where it lies outside the tensor: 72 channels of 3 x 3 x 64, 1568 row tiles, 54.9 us with
    uint32_t idesc2;     // 56 of a box's 64 rows past the end, 31.4 without); idesc2: MMAs of rows2 columns, rounded to 16
    CUtensorMap tmap_y;  // output codes: [M][K] box {64, 128} (linear tiles) or [N][P][Q][K] box {64, TW, TH, 1}
    CUtensorMap tmap_x;  // patch tiles: activations [planes][N][H][W][Cp], box {64, TW, TH, 1, 1}; window mode:
                         // [planes][N][H][W * 8], box {8 WW, WH, 1, 1} (a window row is one 16 WW-byte run)
    int fast_store;      // 1: one-plane codes staged in shared memory and written by TMA stores
    int nbuf;            // fp32 accumulator buffers in TMEM: 2, or 1 when BN = 256 needs running sums
    int patch;           // a tile is a TH x TW patch of TN images and the A tile comes by TMA:
                         // 1: one 64-channel box per k-block (128-byte swizzle), kbt k-blocks per tap;
                         // 2: Cp == 8 (one 8-channel box per tap, 8 taps per k-block, no swizzle);
                         // 3: Cp == 8, window mode (one input window per tile and limb plane, taps as
                         //    shifted descriptors, weights resident in shared memory)
                         // 4: Cp == 64, window mode of one-plane layers (W64 instance): the 8 x 16 patch's
                         //    input window, one 128-byte-swizzled TMA box per tile, weights resident,
                         //    every tap and 16-channel step one shifted swizzled MMA
    int rows_tma;        // 128-row tiles whose A tile is one 2-D TMA box of the activations seen as
                         // [planes][M][R*S*Cp] (1x1 stride-1 layers without padding, and kernels that
                         // cover the whole unpadded map: FC layers), box {64, rows, 1}, 128-byte
                         // swizzle, taps past R*S*Cp zero filled
    int rows;            // output rows of a row tile: 128, or with TMA rows M's equal parts (a box is slow where it lies
                         // outside the tensor; the tile's other rows hold whatever the stage does and are not stored):
                         // 136 x 4096 outputs of 4096 products 47.8 us with 128-row tiles, 33.4 with two of 72
    int nacc;            // fp32 accumulators per TMEM buffer (window mode: one per limb pair)
    int WW, WH, S2;      // window mode: window width / height in pixels, taps per row rounded up to even
    int w32;             // window mode, two-limb x and w, one-plane codes out: the 32-bit epilogue (the
                         // host proved its bounds; see the epilogue), with m = sh - 16 in [0, 30]
    int fepi;            // the fp32 epilogue (codes: a.vf and fast_store; fp32 image: a.vi; one exact group, no split)
    float win_c[3], win_eps;  // w32 in fp32: 2^(16 - sh), 2^(8 - sh), 2^-sh; the most that the fp32 sum is off
                              // (0: integer arithmetic throughout)
    int wf32;            // the same window instance writing the fp32 image of v = 2^16 T + Lo
    int win_bytes;       // window mode: bytes of one window (128-byte aligned; patch 4: 16-byte aligned)
    int w64_slot0;       // patch 4: offset of window slot 0 (after the resident weights)
    int w64_slot_stride; // bytes between the two window slots (S copies of WH KiB)
    int TH, TW, TN;      // patch shape: TH x TW pixels of TN images (TH * TW * TN <= 128)
    int tiles_p, tiles_q;  // patches per image along P and Q (128-row tiles: 1)
    int step_n, step_q, step_p, step_g;  // the grid size in the tile index's digits (TileIter)
    int kbt;             // patch 1: k-blocks per tap (the 64-channel blocks of Cp, the last one zero filled)
    ConvArgs a;
    int RSC;       // R * S * Cp: reduction length of one plane
    int tiles_m, tiles_n, n_tiles;
    int n_groups;
    // Split reduction: every tile's reduction is shared by ksplit work units, unit share s taking the
    // groups g[gs[s]] .. g[gs[s + 1] - 1] (sub-ranges of every exact group, or whole groups); a unit
    // writes its exact integer sums to part[s][M][K] (ACC) and a second kernel adds the shares and
    // applies the epilogue.  Without a split, gs = {0, n_groups}.
    int ksplit, n_units;
    int gs[TC_MAX_SPLIT + 1];
    void* part;
    // Packed weights (pk = 1, one plane of wk <= 8 bits, wsigned): fxpq_pack_weights' tiles, words
    // [ceil(R*S*Cp / 64)][K_pad / 256][wk][256][2]: word (kb, t, b, o, h) bit i = bit b of code
    // 64 kb + 32 h + i of output channel 256 t + o.
    const uint32_t* wpack;
    int pk, wk, wsigned, K_pad;
    int* status;
    TcGroup g[TC_MAX_GROUPS];
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The copy- and MMA-issuing instructions below are executed by a whole, converged warp and carry their own
// elect.sync predicate: one (always the same) lane issues.  The operands then stay in uniform registers and
// the loops around them in uniform control flow.  Issued from a branch of one thread instead, every operand
// was moved there per instruction: 44 cycles per MMA and about 230 more after each barrier probe (four
// M = 128, N = 128 MMAs, a commit and a wait: 472 cycles, 256 in this form, the tensor core's own rate), and
// about 1300 cycles per pair of tensor copies.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes) : "memory");
}

// 2-D tiled TMA store from shared memory (bulk-group completion).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, int x, int y, int z, int w, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(w), "r"(src)
                 : "memory");
}

// 5-D tiled TMA load completing on mbarrier `bar` (coordinates innermost first; out-of-range
// positions, e.g. the convolution's padding, read as zero).
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            int c4, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];\n\t}" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

// 4-D tiled TMA load (coordinates innermost first) completing on mbarrier `bar`.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n\t}" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}

// Position of a CTA's current tile, stepped by the grid size with carries instead of divisions: tile index
// = ((image group * tiles_p + patch row) * tiles_q + patch column) * tiles_n + column tile (128-row tiles: the
// row tile takes the image group's place).  A division is about 30 instructions, and every epilogue warp
// would need five per tile.
struct TileIter {
    int tn, iq, ip, ng;
    __device__ __forceinline__ TileIter(const TcParams& P, int t0) { split(P, t0, tn, iq, ip, ng); }
    static __host__ __device__ __forceinline__ void split(const TcParams& P, int t, int& n, int& q, int& p, int& g) {
        n = t % P.tiles_n;
        t /= P.tiles_n;
        q = t % P.tiles_q;
        t /= P.tiles_q;
        p = t % P.tiles_p;
        g = t / P.tiles_p;
    }
    __device__ __forceinline__ void next(const TcParams& P) {
        tn += P.step_n;
        int c = tn >= P.tiles_n;
        tn -= c ? P.tiles_n : 0;
        iq += P.step_q + c;
        c = iq >= P.tiles_q;
        iq -= c ? P.tiles_q : 0;
        ip += P.step_p + c;
        c = ip >= P.tiles_p;
        ip -= c ? P.tiles_p : 0;
        ng += P.step_g + c;
    }
};

// A tile row's place within its tile, decoded once per thread: image, row and column offsets of a patch pixel
// in bytes 2, 1 and 0 (each below 128), or -1 for a row past the patch.
__device__ __forceinline__ int row_in_tile(const TcParams& P, int row) {
    const int pix = P.TH * P.TW, ti = row / pix, r = row - ti * pix, j = r / P.TW;
    return ti < P.TN ? (ti << 16) | (j << 8) | (r - j * P.TW) : -1;
}
// Linear output row of that place in the tile at T (`row` itself in 128-row tiles), or -1 outside the map.
__device__ __forceinline__ long long row_at(const TcParams& P, const TileIter& T, int place, int row) {
    if (!P.patch) {
        const long long m = (long long)T.ng * P.rows + row;
        return row < P.rows && m < P.a.M ? m : -1;
    }
    const int n = T.ng * P.TN + (place >> 16), p = T.ip * P.TH + ((place >> 8) & 255), q = T.iq * P.TW + (place & 255);
    if (place < 0 || n >= P.a.N || p >= P.a.P || q >= P.a.Q) return -1;
    return ((long long)n * P.a.P + p) * P.a.Q + q;
}

// Output row (linear index into N*P*Q, or -1 when outside the map) of row i of the window instances' patch tm.
__device__ __forceinline__ long long tile_row(const TcParams& P, int tm, int i) {
    const int per_img = P.tiles_p * P.tiles_q, pix = P.TH * P.TW;
    const int ti = i / pix, j = i - ti * pix;
    if (ti >= P.TN) return -1;
    const int ng = tm / per_img, r = tm - ng * per_img, n = ng * P.TN + ti;
    const int p = (r / P.tiles_q) * P.TH + j / P.TW, q = (r % P.tiles_q) * P.TW + j % P.TW;
    if (n >= P.a.N || p >= P.a.P || q >= P.a.Q) return -1;
    return ((long long)n * P.a.P + p) * P.a.Q + q;
}

// 3-D tiled TMA load (coordinates innermost first) completing on mbarrier `bar`.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];\n\t}" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// 1-D bulk copy global -> shared completing on mbarrier `bar` (both addresses 16-byte aligned, bytes a
// multiple of 16).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// Bit-plane bytes -> fp16 codes.  (lo, hi): an 8 x 8 bit matrix, byte b = plane b (bytes 0-3 in lo,
// 4-7 in hi), bit c = code c of eight consecutive codes.  Three delta swaps transpose it (Hacker's
// Delight, 7-3: byte c then holds code c's k bits).  Signed codes have bit k-1 flipped (`flip`), which
// maps them to u = code + 2^(k-1) in [0, 2^k); each byte then becomes the fp16 1024 + u (exponent
// byte 0x64, u in the mantissa) and one half2 subtraction of `off` = 1024 (+ 2^(k-1) if signed)
// leaves the code itself, exactly.  Returns the 16-byte chunk of the eight fp16 codes.
__device__ __forceinline__ uint4 planes_to_f16(uint32_t lo, uint32_t hi, uint32_t flip, uint32_t off) {
    uint32_t t;
    t = (lo ^ (lo >> 7)) & 0x00AA00AAu;
    lo ^= t ^ (t << 7);
    t = (hi ^ (hi >> 7)) & 0x00AA00AAu;
    hi ^= t ^ (t << 7);
    t = (lo ^ (lo >> 14)) & 0x0000CCCCu;
    lo ^= t ^ (t << 14);
    t = (hi ^ (hi >> 14)) & 0x0000CCCCu;
    hi ^= t ^ (t << 14);
    t = (lo ^ (hi << 4)) & 0xF0F0F0F0u;  // the 4 x 4 blocks across the two words
    lo ^= t;
    hi ^= t >> 4;
    lo ^= flip;
    hi ^= flip;
    const __half2 o2 = *reinterpret_cast<const __half2*>(&off);
    uint32_t h[4] = {__byte_perm(lo, 0x64646464u, 0x5140), __byte_perm(lo, 0x64646464u, 0x5342),
                     __byte_perm(hi, 0x64646464u, 0x5140), __byte_perm(hi, 0x64646464u, 0x5342)};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&h[q]), o2);
        h[q] = *reinterpret_cast<const uint32_t*>(&v);
    }
    return make_uint4(h[0], h[1], h[2], h[3]);
}

// 4 x 4 byte transpose: out[m] byte b = in[b] byte m.
__device__ __forceinline__ void byte_transpose4(const uint32_t (&in)[4], uint32_t (&out)[4]) {
    const uint32_t t0 = __byte_perm(in[0], in[1], 0x5140), t1 = __byte_perm(in[0], in[1], 0x7362);
    const uint32_t t2 = __byte_perm(in[2], in[3], 0x5140), t3 = __byte_perm(in[2], in[3], 0x7362);
    out[0] = __byte_perm(t0, t2, 0x5410);
    out[1] = __byte_perm(t0, t2, 0x7632);
    out[2] = __byte_perm(t1, t3, 0x5410);
    out[3] = __byte_perm(t1, t3, 0x7632);
}

// Expands one k-block's packed tile (`pk`: k bit planes of BN rows x 2 words, word (b, o, h) at
// 2 (b BN + o) + h, bit i = bit b of code 32 h + i of row o) into the fp16 B stage `sb` (BN rows of
// 128 bytes, 128-byte swizzle: chunk j of row o at 16 ((j ^ o) & 7)).  Thread tid of nthreads takes
// rows tid, tid + nthreads, ...: one 8-byte load per plane (consecutive rows: no bank conflicts), then
// eight chunks.
template <int BN>
__device__ __forceinline__ void pk_convert_stage(const uint32_t* pk, unsigned char* sb, int k, uint32_t flip,
                                                 uint32_t off, int tid, int nthreads) {
    for (int o = tid; o < BN; o += nthreads) {
        uint32_t w[2][8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            uint2 v = make_uint2(0u, 0u);
            if (b < k) v = *reinterpret_cast<const uint2*>(pk + 2 * (b * BN + o));
            w[0][b] = v.x;
            w[1][b] = v.y;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t lo[4], hi[4];
            byte_transpose4({w[h][0], w[h][1], w[h][2], w[h][3]}, lo);
            byte_transpose4({w[h][4], w[h][5], w[h][6], w[h][7]}, hi);
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int j = 4 * h + m;
                *reinterpret_cast<uint4*>(sb + o * 128 + ((j ^ (o & 7)) << 4)) = planes_to_f16(lo[m], hi[m], flip, off);
            }
        }
    }
}

// Bounded wait for the phase of `bar` with the given parity.  Returns false (and latches the
// timeout status, sets the CTA abort flag) if it gave up or another role already aborted.
__device__ __forceinline__ bool wait_bounded_for(uint32_t bar, uint32_t parity, volatile int* abort, int* status,
                                                 long long limit) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > limit) {
            *abort = 1;
            latch_status(status, FXPQ_ERR_TIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
    return wait_bounded_for(bar, parity, abort, status, TC_WAIT_CYCLES);
}
// The same for a whole converged warp (the MMA- and copy-issuing ones); the result is uniform by votes, which
// keeps the caller's control flow uniform.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort, int* status) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    while (true) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (__any_sync(0xffffffffu, *abort)) return false;
        if (__any_sync(0xffffffffu, clock64() - t0 > TC_WAIT_CYCLES)) {
            *abort = 1;
            latch_status(status, FXPQ_ERR_TIMEOUT);
            return false;
        }
    }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
// Shared-memory matrix descriptor, K-major without swizzle: core matrices of 8 rows x 16 bytes;
// lbo = bytes between core matrices adjacent in K, sbo = bytes between 8-row groups.
__device__ __forceinline__ uint64_t make_sdesc_noswz(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1u << 46;  // descriptor version; layout type 0 = no swizzle
    return d;
}

__device__ __forceinline__ uint64_t make_sdesc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);          // start address
    d |= (uint64_t)1u << 16;                          // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024u >> 4) << 32;                // stride byte offset: 8 rows x 128 B
    d |= (uint64_t)1u << 46;                          // descriptor version
    d |= (uint64_t)2u << 61;                          // SWIZZLE_128B
    return d;
}

// Instruction descriptor, kind::f16: fp16 A and B (K-major), fp32 accumulator, M x N.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
    return (1u << 4)                        // D format F32
           | (0u << 7) | (0u << 10)         // A, B format F16
           | ((uint32_t)(N >> 3) << 17)     // N / 8
           | ((uint32_t)(M >> 4) << 24);    // M / 16
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
        : "memory");
}

// Loads / stores without their completion wait, so that several TMEM accesses share one round trip.
// After tmem_wait_ld(), reg_fence() on each loaded array orders every use of its registers after the
// wait (the empty asm redefines them).
__device__ __forceinline__ void tmem_ld16_nw(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void reg_fence(uint32_t (&r)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}
__device__ __forceinline__ void tmem_st16_nw(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 32 one-plane codes per lane (row m, channels k0 ..) through a 2 KB shared-memory slice of the warp: each
// lane puts its row's 64 bytes there (16-byte pieces rotated against bank conflicts), then every store
// instruction writes whole 64-byte row segments of eight rows.  One-plane codes have K % 8 == 0, so a
// 16-byte piece lies wholly inside or past K.  Rows with m < 0 store nothing.
__device__ __forceinline__ void store_codes_direct(const ConvArgs& a, long long m, int k0, const uint32_t (&w)[16],
                                                   unsigned char* wbuf, int lane) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        *reinterpret_cast<uint4*>(wbuf + lane * 64 + 16 * (q ^ ((lane >> 1) & 3))) =
            make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
    __syncwarp();
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int r = (lane >> 2) + 8 * it, pc = lane & 3;
        const long long mr = __shfl_sync(0xffffffffu, m, r);
        const uint4 v = *reinterpret_cast<const uint4*>(wbuf + r * 64 + 16 * (pc ^ ((r >> 1) & 3)));
        const int kk = k0 + pc * 8;
        if (mr >= 0 && kk < a.K) *reinterpret_cast<uint4*>(static_cast<__half*>(a.y) + mr * a.K + kk) = v;
    }
    __syncwarp();
}

// The same for 32 fp32 values per lane (channels k0 ..), in two rounds of 64 bytes of a row.  K % 4 == 0.
__device__ __forceinline__ void store_f32_direct(const ConvArgs& a, long long m, int k0, const float (&v)[32],
                                                 unsigned char* wbuf, int lane) {
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = 16 * hf + 4 * q;
            *reinterpret_cast<float4*>(wbuf + lane * 64 + 16 * (q ^ ((lane >> 1) & 3))) =
                make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int r = (lane >> 2) + 8 * it, pc = lane & 3;
            const long long mr = __shfl_sync(0xffffffffu, m, r);
            const uint4 x = *reinterpret_cast<const uint4*>(wbuf + r * 64 + 16 * (pc ^ ((r >> 1) & 3)));
            const int kk = k0 + 16 * hf + pc * 4;
            if (mr >= 0 && kk < a.K) *reinterpret_cast<uint4*>(static_cast<float*>(a.y) + mr * a.K + kk) = x;
        }
        __syncwarp();
    }
}

// Uniform constants of the 32-bit FxP-QLayer epilogue (the same arithmetic as qlayer_code32, with
// the bias alignment split into a left and a right shift so that it has no branches).
struct Epi32 {
    int bsl, bsr, fmask;  // bias term (b << bsl) >> bsr; fraction bits b & fmask (bias finer than acc)
    int sh, hm1;          // requantizing right shift and 2^(sh-1) - 1
    int floor;            // 0 with ReLU, INT_MIN without
    int lo, hi;
    int has_bias;
};

__host__ __device__ __forceinline__ Epi32 make_epi32(const ConvArgs& a) {
    Epi32 e;
    e.bsl = a.bsh > 0 ? a.bsh : 0;
    e.bsr = a.bsh < 0 ? -a.bsh : 0;
    e.fmask = (1 << e.bsr) - 1;
    e.sh = a.sh32;
    e.hm1 = (1 << (a.sh32 - 1)) - 1;
    e.floor = a.relu ? 0 : INT_MIN;
    e.lo = (int)a.lo;
    e.hi = (int)a.hi;
    e.has_bias = a.has_bias;
    return e;
}

// One code: N = acc + aligned bias; ReLU; N / 2^sh rounded half to even, then clipped.  With
// q = floor(N / 2^sh) and x = (q & 1) | phi, floor((N + 2^(sh-1) - 1 + x) / 2^sh) is q + 1 exactly
// when the remainder is above one half, or equal to it with q odd or phi set (phi: the bias had
// nonzero bits below the accumulator's scale, so the true value lies above the tie).  After a ReLU
// clamp N = 0 and the sum stays below 2^sh whatever phi is.  The host keeps |N| + 2^(sh-1) < 2^31.
__host__ __device__ __forceinline__ int epi32_code(const Epi32& e, int acc, int bterm, int phi) {
    const int N = max(acc + bterm, e.floor);
    const int x = ((N >> e.sh) & 1) | phi;
    return min(max((N + e.hm1 + x) >> e.sh, e.lo), e.hi);
}

// The same FxP-QLayer on 64-bit values (wide sums, two-limb layers, Scale layers), valid for
// 1 <= sh <= 62: the bias alignment is v = (acc << dr) + (B << dl) (one of dl, dr is zero), a Scale
// layer (SC) makes it ((v * aleph1) << dr2) + (aleph2 << dl2), and the code is
// round_half_even(v / 2^sh) = floor((v + 2^(sh-1) - 1 + ((v >> sh) & 1)) / 2^sh), clipped.  The host
// keeps |v| < 2^62 at every step, so neither the product nor the rounding sum can overflow.
struct Epi64 {
    int dl, dr, sh;
    long long hm1, floor;
    int lo, hi, has_bias, ok;  // ok: 1 <= sh <= 62 (otherwise the generic path runs)
    int dl2, dr2;
};

__host__ __device__ __forceinline__ Epi64 make_epi64(const ConvArgs& a) {
    Epi64 e;
    e.dl = a.delta > 0 ? a.delta : 0;
    e.dr = a.delta < 0 ? -a.delta : 0;
    e.sh = a.sh;
    e.ok = a.sh >= 1 && a.sh <= 62;
    e.hm1 = e.ok ? (1LL << (a.sh - 1)) - 1 : 0;
    e.floor = a.relu ? 0LL : LLONG_MIN;
    e.lo = (int)a.lo;
    e.hi = (int)a.hi;
    e.has_bias = a.has_bias;
    e.dl2 = a.delta2 > 0 ? a.delta2 : 0;
    e.dr2 = a.delta2 < 0 ? -a.delta2 : 0;
    return e;
}

// m, h: aleph1 and aleph2 codes of the channel (read only when SC)
template <bool SC>
__host__ __device__ __forceinline__ int epi64_code(const Epi64& e, long long acc, int32_t b, int32_t m, int32_t h) {
    long long v = (acc << e.dr) + ((long long)b << e.dl);
    if (SC) v = ((v * (long long)m) << e.dr2) + ((long long)h << e.dl2);
    v = max(v, e.floor);
    const long long c = (v + e.hm1 + ((v >> e.sh) & 1)) >> e.sh;
    return (int)min(max(c, (long long)e.lo), (long long)e.hi);
}

// aleph1 / aleph2 codes of channel k for the SC epilogue (0 past K)
__device__ __forceinline__ int32_t scale_code(const ConvArgs& a, int k) { return k < a.K ? __ldg(a.scale + k) : 0; }
__device__ __forceinline__ int32_t shift_code(const ConvArgs& a, int k) { return k < a.K ? __ldg(a.shift + k) : 0; }

// Two codes in [-512, 511] as a packed fp16 pair: 1536 + c has the bit pattern 0x6600 + c (the
// binade [1024, 2048) has unit spacing), and one packed subtraction of 1536 leaves c exactly.
__device__ __forceinline__ uint32_t pack_codes_f16(int c0, int c1) {
    // 0x6600 + c0 >= 0x6400 never borrows from the high half
    const uint32_t bits = (uint32_t)c1 * 65536u + (uint32_t)c0 + 0x66006600u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&bits), __halves2half2(__ushort_as_half(0x6600),
                                                                                        __ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// Final epilogue of 32 consecutive output channels k0.. of row m, every output that the staged tiles of one-plane codes do
// not carry (two-plane codes, int64 sums, fp32 images, codes of packed-weight layers): bias alignment, Scale layer, ReLU,
// FxP-QLayer.  All 32 lanes take part; rows with m < 0 (outside the output) store nothing.  wbuf: epi_buf_bytes<ACC>() of
// shared memory of the warp, or null.
//   codes: 16-byte pieces of eight codes per plane (K % 8 == 0);
//   fp32 (K % 4 == 0) and int64 (K % 2 == 0) with wbuf: every round each lane puts 16 of its row's sums there (16-byte
//     pieces rotated against bank conflicts), then takes four channels in four rows, four lanes side by side, so that the
//     warp writes whole row segments rather than 32 rows at one value per lane;
//   else one value per store.
// Lane j holds the constants of channel k0 + j, aligned: one load serves the chunk, and shuffles hand them out.  (Loading
// them per value, one after the other, the 9- to 16-bit codes of a small layer took 10 to 20 us more, and those of 4 x 98 x
// 98 x 208 outputs 376 us; 172 with one code per store in unrolled code, 66 so.)
// It is a call, its values passed in local memory: inlined, it made the 128-column kernels spill 1.2 KB around every path,
// the codes of several groups among them.  It runs in short loops: unrolled over the 32 channels, the int64 logits of a
// 512 -> 1000 layer, one tile per CTA and each instruction run once, took 25 us, most of it for fetching code and
// re-reading parameters; 13 us so.
template <typename ACC>
__host__ __device__ constexpr int epi_buf_bytes() {
    return 32 * 16 * (int)sizeof(ACC);
}
// a is a copy of what it needs: read through a reference, the kernel's parameters cost a trip to memory each.
struct EpiBlock {
    void* y;
    const int32_t *bias, *scale, *shift;
    long long M;
    int K, out_mode, py;
    float f32_scale;
    Epi64 e;
};
__device__ __forceinline__ EpiBlock make_epi_block(const ConvArgs& a) {
    return EpiBlock{a.y, a.bias, a.scale, a.shift, a.M, a.K, a.out_mode, a.py, a.f32_scale, make_epi64(a)};
}
template <typename ACC, bool SC>
__device__ __noinline__ void epilogue_block32(const EpiBlock a, long long m, int k0, const ACC (&acc)[32], unsigned char* wbuf,
                                              int lane) {
    if (!__any_sync(0xffffffffu, m >= 0)) return;
    const int mode = a.out_mode, K = a.K;
    const long long M = a.M;
    const Epi64& e = a.e;
    const long long bl = (long long)(e.has_bias && k0 + lane < K ? __ldg(a.bias + k0 + lane) : 0) << e.dl;
    int32_t ms = 0;
    long long hl = 0;
    if constexpr (SC) {
        ms = k0 + lane < K ? __ldg(a.scale + k0 + lane) : 0;
        hl = (long long)(k0 + lane < K ? __ldg(a.shift + k0 + lane) : 0) << e.dl2;
    }
    auto form = [&](long long v, long long b, int32_t s, long long h) -> long long {
        v = (v << e.dr) + b;
        if constexpr (SC) v = ((v * (long long)s) << e.dr2) + h;
        return max(v, e.floor);
    };
    auto value = [&](int j) -> long long {  // of the lane's own row
        return form((long long)acc[j], __shfl_sync(0xffffffffu, bl, j), SC ? __shfl_sync(0xffffffffu, ms, j) : 0,
                    SC ? __shfl_sync(0xffffffffu, hl, j) : 0ll);
    };
    if (mode == FXPQ_OUT_CODES) {
        const int py = a.py;
        const int left = min(-e.sh, 31);  // sh <= 0: past 2^17, or with 31 bits to the left, every value is clipped
        __half* const y = static_cast<__half*>(a.y) + m * K;
#pragma unroll 1
        for (int c0 = 0; c0 < 32 && k0 + c0 < K; c0 += 8) {
            int c[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const long long v = value(c0 + j);
                const long long q = e.ok ? (v + e.hm1 + ((v >> e.sh) & 1)) >> e.sh : min(max(v, -(1ll << 17)), 1ll << 17) << left;
                c[j] = (int)min(max(q, (long long)e.lo), (long long)e.hi);
            }
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                hi[j] = py == 2 ? pack_codes_f16(c[2 * j] >> 8, c[2 * j + 1] >> 8) : pack_codes_f16(c[2 * j], c[2 * j + 1]);
                lo[j] = pack_codes_f16(c[2 * j] & 255, c[2 * j + 1] & 255);
            }
            if (m >= 0) {
                *reinterpret_cast<uint4*>(y + k0 + c0) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                if (py == 2) *reinterpret_cast<uint4*>(y + M * K + k0 + c0) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
        }
        return;
    }
    const bool f32 = mode == FXPQ_OUT_F32;
    const float f32_scale = a.f32_scale;
    float* const yf = static_cast<float*>(a.y);
    long long* const yl = static_cast<long long*>(a.y);
    if (!wbuf || K % (f32 ? 4 : 2) != 0) {
#pragma unroll 1
        for (int c0 = 0; c0 < 32 && k0 + c0 < K; c0 += 8) {
            long long v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = value(c0 + j);
            if (m >= 0) {
                const long long o = m * K + k0 + c0;
                const int n = min(K - k0 - c0, 8);
                if (f32) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < n) yf[o + j] = __ll2float_rn(v[j]) * f32_scale;
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < n) yl[o + j] = v[j];
                }
            }
            __syncwarp();
        }
        return;
    }
    // a row's 16 sums take U pieces of 16 bytes, piece u at u ^ swz(row)
    constexpr int U = (int)sizeof(ACC), ROW = 16 * U;
    auto swz = [](int row) { return U == 8 ? row & 7 : (row >> 1) & 3; };
    const int pc = lane & 3;
#pragma unroll 1
    for (int c0 = 0; c0 < 32 && k0 + c0 < K; c0 += 16) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint4 w;
            if constexpr (U == 4) {
                w = make_uint4((uint32_t)acc[c0 + 4 * u], (uint32_t)acc[c0 + 4 * u + 1], (uint32_t)acc[c0 + 4 * u + 2],
                               (uint32_t)acc[c0 + 4 * u + 3]);
            } else {
                const unsigned long long w0 = (unsigned long long)acc[c0 + 2 * u], w1 = (unsigned long long)acc[c0 + 2 * u + 1];
                w = make_uint4((uint32_t)w0, (uint32_t)(w0 >> 32), (uint32_t)w1, (uint32_t)(w1 >> 32));
            }
            *reinterpret_cast<uint4*>(wbuf + lane * ROW + 16 * (u ^ swz(lane))) = w;
        }
        __syncwarp();
        const int kk = k0 + c0 + 4 * pc;
        long long bv[4], hv[4];
        int32_t sv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            bv[i] = __shfl_sync(0xffffffffu, bl, c0 + 4 * pc + i);
            sv[i] = SC ? __shfl_sync(0xffffffffu, ms, c0 + 4 * pc + i) : 0;
            hv[i] = SC ? __shfl_sync(0xffffffffu, hl, c0 + 4 * pc + i) : 0ll;
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int r = (lane >> 2) + 8 * it;
            const long long mr = __shfl_sync(0xffffffffu, m, r);
            ACC raw[4];
#pragma unroll
            for (int h = 0; h < U / 4; ++h)
                *reinterpret_cast<uint4*>(raw + 4 * h / (U / 4)) =
                    *reinterpret_cast<const uint4*>(wbuf + r * ROW + 16 * ((U / 4 * pc + h) ^ swz(r)));
            long long v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = form((long long)raw[i], bv[i], sv[i], hv[i]);
            if (mr >= 0 && kk < K) {
                if (f32) {
                    *reinterpret_cast<float4*>(yf + mr * K + kk) =
                        make_float4(__ll2float_rn(v[0]) * f32_scale, __ll2float_rn(v[1]) * f32_scale,
                                    __ll2float_rn(v[2]) * f32_scale, __ll2float_rn(v[3]) * f32_scale);
                } else {
                    longlong2* const d = reinterpret_cast<longlong2*>(yl + mr * K + kk);
                    d[0] = make_longlong2(v[0], v[1]);
                    if (kk + 2 < K) d[1] = make_longlong2(v[2], v[3]);
                }
            }
        }
        __syncwarp();
    }
}

// One code of the two-limb window epilogue in exact 32-bit arithmetic.  With the limb sums S_hh, S_mid = S_hl + S_lh, S_ll
// and the aligned bias B' = 2^16 Bh + Bl (0 <= Bl < 2^16; bt = (Bh, Bl)):
//   v = 2^16 S_hh + 2^8 S_mid + S_ll + B' = 2^16 T + Lo,
//   L = 2^8 S_mid + S_ll + Bl,  T = S_hh + Bh + (L >> 16),  Lo = L & 0xFFFF
// (the host keeps |L| and |T| below 2^31).  With sh = 16 + m, floor(v / 2^sh) = T >> m and the remainder is 2^16 (T mod
// 2^m) + Lo, so round half to even needs T mod 2^m (mmask = 2^m - 1) against half = 2^(m-1), and Lo only to tell a tie
// (Lo = 0) from above it.  ReLU: v < 0 exactly when T < 0.
__device__ __forceinline__ int win_code(uint32_t fhh, uint32_t fhl, uint32_t flh, uint32_t fll, int2 bt, int m, int half,
                                        int mmask, int relu, int lo, int hi) {
    const int mid = __float2int_rn(__uint_as_float(fhl)) + __float2int_rn(__uint_as_float(flh));
    const int L = mid * 256 + __float2int_rn(__uint_as_float(fll)) + bt.y;
    const int T = __float2int_rn(__uint_as_float(fhh)) + bt.x + (L >> 16);
    const int Lo = L & 0xFFFF;
    int q, up;
    if (m > 0) {
        q = T >> m;
        const int rem = T & mmask;
        up = (rem > half) | ((rem == half) & ((Lo != 0) | (q & 1)));
    } else {
        q = T;
        up = (Lo > 0x8000) | ((Lo == 0x8000) & (q & 1));
    }
    return min(max((relu && T < 0) ? 0 : q + up, lo), hi);
}

__device__ __forceinline__ uint64_t f32x2_splat(float c) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %1};" : "=l"(v) : "f"(c));
    return v;
}

// Two accumulators to packed codes in fp32 (fepi_bias): one packed fused multiply-add, clip, the packed
// rounding addition of f32_codes_f16x2.  About 4.5 instructions per code, none of them a conversion (those
// run at a quarter of the rate); the integer form took 20 to 30.
__device__ __forceinline__ uint32_t fepi_pair(uint32_t a0, uint32_t a1, uint64_t cc, float t0, float t1, float lo, float hi) {
    uint64_t av, tv, v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(av) : "r"(a0), "r"(a1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(tv) : "f"(t0), "f"(t1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(av), "l"(cc), "l"(tv));
    float x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
    x = fminf(fmaxf(x, lo), hi);
    y = fminf(fmaxf(y, lo), hi);
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(v) : "l"(f32x2_splat(12609024.0f)));
    uint32_t r0, r1;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(r0), "=r"(r1) : "l"(v));
    const uint32_t w = __byte_perm(r0, r1, 0x5410);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w),
                              __halves2half2(__ushort_as_half(0x6600), __ushort_as_half(0x6600)));
    return *reinterpret_cast<const uint32_t*>(&h);
}

// One output of a Scale layer in exact 64-bit arithmetic, for the rare value next to a rounding boundary.
static __device__ __noinline__ int scale_code_exact(const ConvArgs& a, int k, uint32_t f) {
    const Epi64 e = make_epi64(a);
    const int32_t b = (e.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
    return epi64_code<true>(e, (long long)__float2int_rn(__uint_as_float(f)), b, scale_code(a, k), shift_code(a, k));
}
// Two outputs (channels k, k + 1) of a Scale layer to packed codes: fepi_scale, exact arithmetic within vs_eps of a
// rounding boundary (one value in some ten thousand).
__device__ __forceinline__ uint32_t fepi_scale_pair(const ConvArgs& a, int k, uint32_t f0, uint32_t f1, float m0, float m1,
                                                    float t0, float t1) {
    const float x = fminf(fmaxf(fmaf(__uint_as_float(f0), m0, t0), a.vf_lo), a.vf_hi);
    const float y = fminf(fmaxf(fmaf(__uint_as_float(f1), m1, t1), a.vf_lo), a.vf_hi);
    const float rx = (x + 12582912.0f) - 12582912.0f, ry = (y + 12582912.0f) - 12582912.0f;
    if (fmaxf(fabsf(x - rx), fabsf(y - ry)) > 0.5f - a.vs_eps)
        return pack_codes_f16(scale_code_exact(a, k, f0), scale_code_exact(a, k + 1, f1));
    return f32_codes_f16x2(x, y);
}

// ------------------------------------------------------------------ kernel
// PK converter warp `cid` (of TC_PK_CONVERTERS): walks the same k-block sequence as the issuing thread;
// for each k-block waits until its A box and packed records have landed (pkfull), expands its share of
// the records into the B stage, makes the writes visible to the tensor cores' async proxy and arrives
// on the stage's full barrier (one arrival per warp).
template <int BN, bool SPLIT>
__device__ __forceinline__ void pk_convert_loop(const TcParams& P, int cid, int lane, const unsigned char* sP,
                                                unsigned char* sB, uint32_t pkfull0, uint32_t full0, volatile int* abort) {
    constexpr int STAGES = tc_stages(BN, true);
    constexpr int B_BYTES = BN * TC_BK * 2;
    const int k = P.wk;
    const uint32_t flip = P.wsigned ? 0x01010101u * (1u << (k - 1)) : 0u;
    const uint32_t o1 = 0x6400u + (P.wsigned ? (1u << (k - 1)) : 0u);  // fp16 bits of 1024 (+ 2^(k-1))
    const uint32_t off = o1 | (o1 << 16);
    uint32_t it = 0;
    for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles); ut += gridDim.x) {
        const int t = SPLIT ? ut / P.ksplit : ut, sp = SPLIT ? ut - t * P.ksplit : 0;
        (void)t;
        (void)sp;
        for (int gi = SPLIT ? P.gs[sp] : 0; gi < (SPLIT ? P.gs[sp + 1] : P.n_groups); ++gi) {
            for (int kb = P.g[gi].kb0; kb < P.g[gi].kb1; ++kb, ++it) {
                const uint32_t stage = it % STAGES, phase = (it / STAGES) & 1;
                if (!wait_bounded(pkfull0 + 8 * stage, phase, abort, P.status)) return;
                pk_convert_stage<BN>(reinterpret_cast<const uint32_t*>(sP + stage * (BN * 64)), sB + stage * B_BYTES, k,
                                     flip, off, cid * 32 + lane, TC_PK_CONVERTERS * 32);
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + 8 * stage);
            }
        }
    }
}

// SPLIT: the instantiation that runs split reductions (P.ksplit >= 1, unit share ranges P.gs); without it
// the unit loop is the tile loop and every tile takes all P.n_groups groups.
// PK: the instantiation that reads packed k-bit weights (P.pk = 1; BN = 256, TMA A tiles, no output
// staging): one thread issues every copy and TC_PK_CONVERTERS warps expand the weights.
// WIN: the window-mode instance of the 32-bit two-limb epilogue (P.patch == 3, P.w32): 16 epilogue warps and
// two staging tiles; only window mode's roles are compiled into it.
// W64: the same for the 64-channel window mode (P.patch == 4) with one-plane codes out.
// FE: the instance of layers whose epilogue is the fp32 FxP-QLayer (P.fepi): nothing else is compiled into it,
// which keeps its epilogue out of local memory (beside the integer forms the 128-column one spilled 320 bytes).
template <int BN, typename ACC, bool SC, bool SPLIT = false, bool PK = false, bool WIN = false, bool W64 = false, bool FE = false>
__global__ void __launch_bounds__((WIN || W64) ? tc_threads_win() : tc_threads_pk(BN, PK), 1)
    conv_tc_kernel(const __grid_constant__ TcParams P) {
    constexpr int TC_STAGES = tc_stages(BN, PK);
    constexpr int TC_LAG = tc_lag(BN, PK);
    // 256-column tiles without packed weights store their one-plane codes with plain stores through
    // each warp's 2 KB slice of the staging region rather than by TMA stores of a whole staged tile
    constexpr bool DIRECT = BN == 256 && !PK;
    static_assert(TC_LAG >= 1 && TC_LAG < TC_STAGES, "producer lag must be below the stage count");
    static_assert(!PK || (BN == 256 && sizeof(ACC) == 4 && !SC), "packed weights: 256-column int32 tiles only");
    static_assert(!PK || TC_STAGES * BN * 64 <= tc_out_bytes(BN, PK), "packed stages must fit the staging region");
    // PK: one issuing warp (producer warp 0), so its stage waits are in order by construction
    constexpr int TC_PRODUCERS = PK ? 1 : tc_producers(BN, PK);
    static_assert(TC_STAGES % TC_PRODUCERS == 0 && TC_PRODUCERS <= 4,
                  "each stage must have one producer among warps 0..3");
    constexpr int NSTG = tc_stg_tiles(BN);  // staging tiles of the TMA stores
    static_assert(!WIN || (BN == 64 && sizeof(ACC) == 8 && !SC && !SPLIT && !PK), "window instance: BN = 64, int64");
    static_assert(!W64 || (BN == 64 && sizeof(ACC) == 4 && !SC && !SPLIT && !PK && !WIN), "W64 instance: BN = 64, int32");
    static_assert(!FE || (sizeof(ACC) == 4 && !SPLIT && !PK && !WIN && !W64), "fp32 epilogue: plain int32 instances");
    constexpr bool WEPI = WIN || W64;  // the window instances' epilogue (16 warps, two staging tiles)
    constexpr int EPI_WARPS = WEPI ? TC_WIN_EPI_WARPS : tc_epi_warps(BN);
    static_assert(tc_out_bytes(BN, PK) >= EPI_WARPS * (int)(32 * 16 * sizeof(ACC)) || WEPI, "epilogue_block32's buffers fit");
    constexpr int MMA_WARP = 4 + EPI_WARPS;
    constexpr bool STORE_WARP = BN <= 128;  // warp MMA_WARP + 1 stores the staged tiles
    constexpr int STG_BYTES = BN * TC_BM * 2;  // one staging tile
    constexpr int CPW = WEPI ? 1 : (BN / 32) / (EPI_WARPS / 4);  // 32-column chunks per epilogue warp
    constexpr int A_BYTES = TC_BM * TC_BK * 2;  // 16 KB
    constexpr int B_BYTES = BN * TC_BK * 2;
    constexpr uint32_t IDESC = make_idesc(TC_BM, BN);
    // fp32 accumulator buffers + integer running sums, rounded up to a power of two (BN = 256: two
    // buffers without running sums, or one buffer with them)
    // (the int64 instance also serves window mode: two buffers of up to four limb-pair accumulators)
    constexpr uint32_t USED_COLS = (BN == 256 || sizeof(ACC) == 8) ? 512u : 2 * BN + BN * (uint32_t)(sizeof(ACC) / 4);
    constexpr uint32_t TMEM_COLS = USED_COLS <= 256 ? 256u : 512u;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* sA = base;
    unsigned char* sB = base + TC_STAGES * A_BYTES;
    unsigned char* sO = W64 ? base + TC_W64_SO : sB + TC_STAGES * B_BYTES;  // output staging: BN/64 halves of
                                                                         // [128 rows][64 codes]
    uint64_t* bars = reinterpret_cast<uint64_t*>(sO + tc_out_bytes(BN, PK));
    // bars: full[STAGES], empty[STAGES], accfull[2], accempty[2], done
    volatile int* abort = reinterpret_cast<volatile int*>(bars + 2 * TC_STAGES + 5);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * TC_STAGES + 6);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + TC_STAGES);
    const uint32_t accfull0 = smem_u32(bars + 2 * TC_STAGES), accempty0 = smem_u32(bars + 2 * TC_STAGES + 2);
    const uint32_t done_bar = smem_u32(bars + 2 * TC_STAGES + 4);
    const uint32_t stg_full = smem_u32(bars + 2 * TC_STAGES + 7);  // staging written by every epilogue warp
    const uint32_t stg_free = smem_u32(bars + 2 * TC_STAGES + 8);  // staging read by the previous TMA store
    const uint32_t wbar = smem_u32(bars + 2 * TC_STAGES + 9);      // window mode: resident weights loaded
    const uint32_t stg_full2 = smem_u32(bars + 2 * TC_STAGES + 10);  // the second staging tile
    const uint32_t stg_free2 = smem_u32(bars + 2 * TC_STAGES + 11);
    // PK: pkfull[s] completes when stage s's A box and packed weight records have landed; the
    // converters then fill the B stage and arrive on full[s]
    const uint32_t pkfull0 = smem_u32(bars + 2 * TC_STAGES + 10);
    unsigned char* sP = sO;  // PK: packed stages of BN * 64 bytes (k <= 8 words per 32 codes)

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // warp: uniform
    const ConvArgs& a = P.a;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            // patch and TMA row tiles: one expect_tx arrival for both TMAs; gathered row tiles: one arrival per
            // producer warp + the weight TMA's expect_tx
            mbar_init(full0 + 8 * s, PK ? TC_PK_CONVERTERS : (P.patch || P.rows_tma) ? 1 : 4 + 1);
            mbar_init(empty0 + 8 * s, 1);
            if (PK) mbar_init(pkfull0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accfull0 + 8 * b, 1);
            mbar_init(accempty0 + 8 * b, EPI_WARPS);  // one arrival per epilogue warp
        }
        mbar_init(done_bar, 1);
        mbar_init(stg_full, EPI_WARPS);
        mbar_init(stg_free, 1);
        if (STORE_WARP) {
            mbar_init(stg_full2, EPI_WARPS);
            mbar_init(stg_free2, 1);
        }
        mbar_init(wbar, 1);
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x == 32) {  // the descriptors that this launch uses, fetched while the kernel sets up
        prefetch_tmap(&P.tmap_w);
        if (P.rows2) prefetch_tmap(&P.tmap_w2);
        if (P.patch || P.rows_tma) prefetch_tmap(&P.tmap_x);
        if (P.fast_store) prefetch_tmap(&P.tmap_y);
    }
    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    pdl_wait();
    // window mode, 32-bit epilogue: per output channel the aligned bias B' = b 2^delta split as
    // (B' >> 16, B' & 0xFFFF), in the last 512 bytes of the B region (the resident weights stay below)
    int2* wtab = reinterpret_cast<int2*>(sB + TC_STAGES * B_BYTES - 512);
    float* wtabf = reinterpret_cast<float*>(sB + TC_STAGES * B_BYTES - 768);  // B' 2^-sh, the 256 bytes before it
    if (WIN && P.patch == 3 && (P.w32 || P.wf32) && warp == 1) {
        for (int k = lane; k < 64; k += 32) {
            const long long bb = (a.has_bias && k < a.K) ? ((long long)__ldg(a.bias + k) << (a.delta > 0 ? a.delta : 0)) : 0;
            wtab[k] = make_int2((int)(bb >> 16), (int)(bb & 0xFFFF));
            wtabf[k] = (float)bb * P.win_c[2];
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (!WIN && warp < 4 && P.patch == 4) {
        // ============================================================ producer, 64-channel window mode
        // The weights, one 128-byte-swizzled box {64 ch, 64 out ch} per tap (8 KiB, the layout of a B
        // stage), are loaded once to the start of shared memory.  Per tile and tap column s, the input
        // window of the 16 x 8 patch shifted by s pixels, TH + R - 1 rows of 8 pixels of 64 channels (one
        // swizzle pattern per row, padding zero filled), is one box into window slot (tile count mod 2):
        // every tap's A operand then starts on a pattern boundary.
        if (warp == 0) {
            mbar_arrive_expect_tx(wbar, (uint32_t)(a.R * a.S) * 8192u);
            for (int t = 0; t < a.R * a.S; ++t)
                tma_load_3d(smem_u32(sA) + (uint32_t)t * 8192u, &P.tmap_w, t * TC_BK, 0, 0, wbar);
            const uint32_t copyb = (uint32_t)P.WH * 1024u;
            const int per_img = P.tiles_p * P.tiles_q;
            uint32_t it = 0, stage = 0, phase = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < P.n_tiles && ok; t += gridDim.x) {
                const int n_img = t / per_img, r = t - n_img * per_img;
                const int hp0 = (r / P.tiles_q) * P.TH - a.pad, wq0 = (r % P.tiles_q) * P.TW - a.pad;
                if (!wait_warp(empty0 + 8 * stage, phase ^ 1, abort, P.status)) {
                    ok = false;
                    break;
                }
                const uint32_t fb = full0 + 8 * stage;
                mbar_arrive_expect_tx(fb, (uint32_t)a.S * copyb);
                const uint32_t dst = smem_u32(sA) + (uint32_t)P.w64_slot0 + stage * (uint32_t)P.w64_slot_stride;
                for (int q = 0; q < a.S; ++q) tma_load_4d(dst + (uint32_t)q * copyb, &P.tmap_x, 0, wq0 + q, hp0, n_img, fb);
                ++it;
                if (++stage == 2) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            const uint32_t from = it >= 2 ? it - 2 : 0;
            for (uint32_t j = from; j < it; ++j) {
                const long long t0 = clock64();
                while (!mbar_try_wait(full0 + 8 * (j % 2), (j / 2) & 1) && clock64() - t0 < TC_WAIT_CYCLES) {
                }
            }
            const long long t0 = clock64();
            while (!mbar_try_wait(wbar, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
            }
        }
    } else if (!W64 && warp < 4 && P.patch == 3) {
        // ============================================================ producer, window mode
        // Stride 1, Cp == 8: the weights are loaded once into the B region, per kernel row r and tap
        // pair sp a block of the two taps, each tap the BN output channels of every limb plane in turn
        // (rows [W_hi | W_lo] of one B operand of N = pw BN: one MMA forms both limb sums of an x limb;
        // one box {8 ch, BN out ch} per tap and plane, taps past S zero filled); per tile, one box per
        // x limb plane holds the input window of TH + R - 1 rows by TW + S2 - 1 pixels (padding zero
        // filled).
        if (warp == 0) {
            const int np = P.S2 / 2;
            const uint32_t tapb = (uint32_t)(BN * 16);  // one tap of one plane
            mbar_arrive_expect_tx(wbar, (uint32_t)(a.pw * a.R * np * 2) * tapb);
            for (int r = 0; r < a.R; ++r)
                for (int t = 0; t < 2 * np; ++t)
                    for (int iw = 0; iw < a.pw; ++iw)
                        tma_load_5d(smem_u32(sB) + (uint32_t)(((r * np + t / 2) * 2 + (t & 1)) * a.pw + iw) * tapb,
                                    &P.tmap_w, 0, 0, t, r, iw, wbar);
            const uint32_t win_tx = (uint32_t)(P.WW * P.WH * 16);
            const int per_img = P.tiles_p * P.tiles_q;
            uint32_t it = 0, stage = 0, phase = 0;
            bool ok = true;
            for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
                const int t = SPLIT ? ut / P.ksplit : ut, sp = SPLIT ? ut - t * P.ksplit : 0;
                (void)sp;
                const int tm = t / P.tiles_n;
                const int n_img = tm / per_img, r = tm - n_img * per_img;
                const int hp0 = (r / P.tiles_q) * P.TH - a.pad, wq0 = (r % P.tiles_q) * P.TW - a.pad;
                if (!wait_warp(empty0 + 8 * stage, phase ^ 1, abort, P.status)) {
                    ok = false;
                    break;
                }
                const uint32_t fb = full0 + 8 * stage;
                mbar_arrive_expect_tx(fb, (uint32_t)a.px * win_tx);
                // (pixels and channels of a row are one inner dimension: x = 8 * pixel, a multiple of 8)
                for (int ia = 0; ia < a.px; ++ia)
                    tma_load_4d(smem_u32(sA + stage * A_BYTES) + (uint32_t)(ia * P.win_bytes), &P.tmap_x, 8 * wq0, hp0,
                                n_img, ia, fb);
                ++it;
                if (++stage == TC_STAGES) {
                    stage = 0;
                    phase ^= 1;
                }
            }
            // bounded wait until the copies of the last stages and the weights have landed
            const uint32_t from = it >= TC_STAGES ? it - TC_STAGES : 0;
            for (uint32_t j = from; j < it; ++j) {
                const long long t0 = clock64();
                while (!mbar_try_wait(full0 + 8 * (j % TC_STAGES), (j / TC_STAGES) & 1) &&
                       clock64() - t0 < TC_WAIT_CYCLES) {
                }
            }
            const long long t0 = clock64();
            while (!mbar_try_wait(wbar, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
            }
        }
    } else if (!WEPI && warp < 4 && (P.patch || P.rows_tma)) {
        // ============================================================ producer, patch tiles
        // The A tile of tap (r, s) and channels c0..c0+63 is the box {64, TW, TH, TN} of the input at
        // (c0, q0 st + s - pad, p0 st + r - pad, n0), traversed with the convolution's stride; the padding
        // and channels past Cp read as zeros, so that the weight columns of the next tap, which the B box
        // then holds in their place, count for nothing.
        // Cp == 8: a k-block is 8 taps of 8 channels; tap tl's box {8, TW, TH} lands at byte
        // 2048 tl of the stage (a 16-byte K column of the no-swizzle layout), and taps past R*S
        // are boxes wholly outside the tensor (zero filled).
        if (warp < TC_PRODUCERS) {
            const uint32_t me = warp;
            const bool narrow = P.patch == 2;
            const uint32_t a_bytes = P.rows_tma ? (uint32_t)P.rows * 128u : (uint32_t)(P.TH * P.TW * P.TN * (narrow ? 8 * 16 : 128));
            uint32_t it = 0, stage = 0, phase = 0;
            bool ok = true;
            TileIter T(P, SPLIT ? 0 : blockIdx.x);
            for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
                const int sp = SPLIT ? ut % P.ksplit : 0;
                if (SPLIT) TileIter::split(P, ut / P.ksplit, T.tn, T.iq, T.ip, T.ng);
                const int tm = T.ng, tn = T.tn, n_img = T.ng * P.TN;  // tm: TMA row tiles
                const int hp0 = T.ip * P.TH * a.stride - a.pad, wq0 = T.iq * P.TW * a.stride - a.pad;
                const bool last_n = P.rows2 && tn == P.tiles_n - 1;
                const CUtensorMap* const mw = last_n ? &P.tmap_w2 : &P.tmap_w;
                const uint32_t b_bytes = last_n ? (uint32_t)P.rows2 * (TC_BK * 2) : (uint32_t)B_BYTES;
                if (!SPLIT) T.next(P);
                for (int gi = SPLIT ? P.gs[sp] : 0; gi < (SPLIT ? P.gs[sp + 1] : P.n_groups) && ok; ++gi) {
                    const TcGroup g = P.g[gi];
                    // tap (rr, ss) and channel offset cc of the group's first k-block, then stepped by
                    // TC_BK channels; wx: the weights' column
                    const int tp0 = g.kb0 / P.kbt;
                    int cc = (g.kb0 - tp0 * P.kbt) * TC_BK;
                    int rr = tp0 / a.S, ss = tp0 - rr * a.S;
                    int wx = P.patch == 1 ? tp0 * a.Cp + cc : g.kb0 * TC_BK;
                    for (int kb = g.kb0; kb < g.kb1; ++kb, ++it) {
                        if (stage % TC_PRODUCERS == me) {
                            if (!wait_warp(empty0 + 8 * stage, phase ^ 1, abort, P.status)) {
                                ok = false;
                                break;
                            }
                            const uint32_t fb = PK ? pkfull0 + 8 * stage : full0 + 8 * stage;
                            const uint32_t pk_bytes = PK ? (uint32_t)(BN * 8 * P.wk) : 0u;
                            mbar_arrive_expect_tx(fb, a_bytes + (PK ? pk_bytes : b_bytes));
                            if (narrow) {
                                for (int tl = 0; tl < 8; ++tl) {
                                    const int tap = kb * 8 + tl;
                                    const bool in = tap < a.R * a.S;
                                    const int r8 = in ? tap / a.S : 0, s8 = in ? tap - (tap / a.S) * a.S : 0;
                                    tma_load_5d(smem_u32(sA + stage * A_BYTES + tl * 2048), &P.tmap_x, in ? 0 : 8,
                                                wq0 + s8, hp0 + r8, n_img, g.a_plane, fb);
                                }
                            } else if (P.rows_tma) {
                                tma_load_3d(smem_u32(sA + stage * A_BYTES), &P.tmap_x, kb * TC_BK, tm * P.rows, g.a_plane,
                                            fb);
                            } else {
                                tma_load_5d(smem_u32(sA + stage * A_BYTES), &P.tmap_x, cc, wq0 + ss, hp0 + rr, n_img,
                                            g.a_plane, fb);
                            }
                            if (PK)
                                bulk_load(smem_u32(sP + stage * (BN * 64)),
                                          P.wpack + ((size_t)kb * P.K_pad + (size_t)tn * BN) * 2 * P.wk, pk_bytes, fb);
                            else
                                tma_load_3d(smem_u32(sB + stage * B_BYTES), mw, wx, tn * BN, g.w_plane, fb);
                        }
                        if (++stage == TC_STAGES) {
                            stage = 0;
                            phase ^= 1;
                        }
                        wx += TC_BK;
                        if (!narrow) {
                            cc += TC_BK;
                            if (cc >= a.Cp) {
                                if (P.patch == 1) wx += a.Cp - cc;  // the next tap's first column
                                cc = 0;
                                if (++ss == a.S) {
                                    ss = 0;
                                    ++rr;
                                }
                            }
                        }
                    }
                }
            }
            // bounded wait until the copies of the last stages have landed (PK: on pkfull, which only
            // the copies complete)
            const uint32_t drain0 = PK ? pkfull0 : full0;
            const uint32_t from = it >= TC_STAGES ? it - TC_STAGES : 0;
            for (uint32_t j = from; j < it; ++j) {
                const long long t0 = clock64();
                while (!mbar_try_wait(drain0 + 8 * (j % TC_STAGES), (j / TC_STAGES) & 1) &&
                       clock64() - t0 < TC_WAIT_CYCLES) {
                }
            }
        }
        if (PK && warp >= 1) pk_convert_loop<BN, SPLIT>(P, warp - 1, lane, sP, sB, pkfull0, full0, abort);
    } else if (!WEPI && warp < 4) {
        // ============================================================ producers, row tiles
        // Thread t copies 16-byte chunk c = t % 8 of rows t/8, t/8 + 16, ...: eight consecutive
        // threads cover one 128-byte row, so every warp instruction reads four whole rows.
        const int c = threadIdx.x & 7;
        const int r0 = threadIdx.x >> 3;  // 0..15
        constexpr int AR = TC_BM / 16;    // A rows per thread
        const __half* xb = a.x;
        uint32_t it = 0;
        bool ok = true;
        for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
            const int t = SPLIT ? ut / P.ksplit : ut, sp = SPLIT ? ut - t * P.ksplit : 0;
            (void)sp;
            const int tm = t / P.tiles_n, tn = t % P.tiles_n;
            const bool last_n = P.rows2 && tn == P.tiles_n - 1;
            long long rowoff[AR];  // element offset of the (r, s) = (0, 0) tap of each row (may be negative)
            int p0[AR], q0[AR];
#pragma unroll
            for (int i = 0; i < AR; ++i) {
                const long long m = (long long)tm * TC_BM + r0 + 16 * i;
                const long long mm = m < a.M ? m : 0;
                const int n_img = (int)(mm / ((long long)a.P * a.Q));
                const int pq = (int)(mm - (long long)n_img * a.P * a.Q);
                p0[i] = (pq / a.Q) * a.stride - a.pad;
                q0[i] = (pq % a.Q) * a.stride - a.pad;
                if (m >= a.M) p0[i] = -(1 << 20);  // rows past the end read zeros
                rowoff[i] = (((long long)n_img * a.H + p0[i]) * a.W + q0[i]) * a.Cp;
            }
            for (int gi = SPLIT ? P.gs[sp] : 0; gi < (SPLIT ? P.gs[sp + 1] : P.n_groups) && ok; ++gi) {
                const TcGroup g = P.g[gi];
                const __half* xp = xb + (long long)g.a_plane * a.x_ps;
                for (int kb = g.kb0; kb < g.kb1; ++kb) {
                    const int stage = it % TC_STAGES;
                    const uint32_t ph = (it / TC_STAGES) & 1;
                    if (!wait_warp(empty0 + 8 * stage, ph ^ 1, abort, P.status)) {
                        ok = false;
                        break;
                    }
                    const uint32_t dA = smem_u32(sA + stage * A_BYTES);
                    if (warp == 0) {  // the weight tile: one TMA, zero-filled past R*S*Cp
                        __syncwarp();
                        mbar_arrive_expect_tx(full0 + 8 * stage, last_n ? (uint32_t)P.rows2 * (TC_BK * 2) : (uint32_t)B_BYTES);
                        tma_load_3d(smem_u32(sB + stage * B_BYTES), last_n ? &P.tmap_w2 : &P.tmap_w, kb * TC_BK, tn * BN,
                                    g.w_plane, full0 + 8 * stage);
                    }
                    const int f = kb * TC_BK + 8 * c;  // this thread's chunk of the flattened (r, s, c) index
                    const bool fvalid = f < P.RSC;
                    const int tp = f / a.Cp;
                    const int cc = f - tp * a.Cp;
                    const int rr = tp / a.S, ss = tp - rr * a.S;
                    const long long toff = ((long long)rr * a.W + ss) * a.Cp + cc;
#pragma unroll
                    for (int i = 0; i < AR; ++i) {
                        const int row = r0 + 16 * i;
                        const int h = p0[i] + rr, w = q0[i] + ss;
                        const bool v = fvalid && (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
                        const __half* src = v ? xp + rowoff[i] + toff : xb;
                        cp_async16(dA + row * 128 + (uint32_t)((c ^ (row & 7)) << 4), src, v ? 16u : 0u);
                    }
                    cp_async_commit();
                    if (it >= TC_LAG) {
                        // this warp's copies of stage it - TC_LAG have landed: one arrival for the warp
                        cp_async_wait<TC_LAG>();
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(full0 + 8 * ((it - TC_LAG) % TC_STAGES));
                    }
                    ++it;
                }
            }
        }
        cp_async_wait<0>();
        fence_proxy_async();
        __syncwarp();
        const uint32_t first = it >= TC_LAG ? it - TC_LAG : 0;
        if (lane == 0)
            for (uint32_t j = first; j < it; ++j) mbar_arrive(full0 + 8 * (j % TC_STAGES));
        if (threadIdx.x == 0) {
            // Every weight TMA this thread issued has landed once its stage's phase completes (the MMA
            // thread already waited for them unless the kernel aborted): bounded wait on the last ones.
            const uint32_t from = it >= TC_STAGES ? it - TC_STAGES : 0;
            for (uint32_t j = from; j < it; ++j) {
                const long long t0 = clock64();
                while (!mbar_try_wait(full0 + 8 * (j % TC_STAGES), (j / TC_STAGES) & 1) &&
                       clock64() - t0 < TC_WAIT_CYCLES) {
                }
            }
        }
    } else if (WEPI && warp < MMA_WARP) {
        // ============================================================ epilogue, window instances
        // Warp w drains TMEM lanes 32 (w % 4) .. + 31 and the 16 columns 16 cw .., cw = (w - 4) / 4: WIN of
        // the four limb accumulators, with the 32-bit arithmetic of the generic window epilogue below;
        // W64 of the one int32-exact accumulator, with the FxP-QLayer of the generic epilogue.  Tile u
        // goes through staging tile u % 2, whose previous store must have read it (at most the other
        // tile's store is then in flight).
        const int quad = warp & 3, cw = (warp - 4) >> 2;
        const int row = quad * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const int m = a.sh - 16;
        const int half = m > 0 ? 1 << (m - 1) : 0;
        const int mmask = (int)((1u << m) - 1u);
        const int lo = (int)a.lo, hi = (int)a.hi;
        const float flo = a.relu && lo < 0 ? 0.0f : (float)lo, fhi = (float)hi;
        const bool f32out = a.out_mode == FXPQ_OUT_F32;  // the fp32 image (calibration) instead of codes
        // W64, 32-bit codes: a thread's 16 output channels are the same in every tile, so their aligned
        // bias terms and the flags of bias bits below the accumulator's scale are formed once
        const Epi32 e32w = make_epi32(a);
        int btw[16];  // (P.fepi: the fp32 terms' bits)
        uint32_t phiw = 0u;
        const uint64_t cc2 = f32x2_splat(a.vf_c);
        if (W64) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const int k = cw * 16 + j;
                const int32_t b = (a.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                btw[j] = !P.fepi  ? (b << e32w.bsl) >> e32w.bsr
                         : f32out ? __float_as_int((float)b * a.vi_b)
                                  : __float_as_int(a.has_bias ? fepi_bias(a, b) : 0.0f);
                phiw |= ((b & e32w.fmask) != 0 ? 1u : 0u) << j;
            }
        }
        bool ok = true;
        uint32_t u = 0;
        for (int t = blockIdx.x; t < P.n_tiles && ok; t += gridDim.x, ++u) {
            const uint32_t buf = u & 1;
            if (!wait_bounded(accfull0 + 8 * buf, (u >> 1) & 1, abort, P.status)) {
                ok = false;
                break;
            }
            tc_fence_after();
            uint32_t w[16];  // codes: 8 words of fp16 pairs; fp32 image: 16 values
            if (W64) {
                uint32_t f[16];
                tmem_ld16_nw(lane_base + buf * (uint32_t)BN + (uint32_t)(cw * 16), f);
                tmem_wait_ld();
                reg_fence(f);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
                if (f32out && P.fepi) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        w[j] = __float_as_uint(fepi_image(a, __uint_as_float(f[j]), a.vi_c, __int_as_float(btw[j])));
                } else if (f32out) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int k = cw * 16 + j;
                        const int acc = __float2int_rn(__uint_as_float(f[j]));
                        const int32_t b = (a.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                        w[j] = __float_as_uint(__ll2float_rn(cblock_value<false>(a, k, (long long)acc, b)) * a.f32_scale);
                    }
                }
                if (!f32out && P.fepi) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        w[j] = fepi_pair(f[2 * j], f[2 * j + 1], cc2, __int_as_float(btw[2 * j]),
                                         __int_as_float(btw[2 * j + 1]), a.vf_lo, a.vf_hi);
                } else if (!f32out && a.v32) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        int c2[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int jj = 2 * j + h;
                            c2[h] = epi32_code(e32w, __float2int_rn(__uint_as_float(f[jj])), btw[jj], (int)((phiw >> jj) & 1u));
                        }
                        w[j] = pack_codes_f16(c2[0], c2[1]);
                    }
                } else if (!f32out) {
                    const Epi64 e64 = make_epi64(a);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        int c2[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int k = cw * 16 + 2 * j + h;
                            const int acc = __float2int_rn(__uint_as_float(f[2 * j + h]));
                            const int32_t b = (a.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                            c2[h] = epi64_code<false>(e64, (long long)acc, b, 0, 0);
                        }
                        w[j] = pack_codes_f16(c2[0], c2[1]);
                    }
                }
            }
            uint32_t fhh[16], fhl[16], flh[16], fll[16];
            if (WIN) {
                const uint32_t abase = lane_base + buf * (uint32_t)(4 * BN) + (uint32_t)(cw * 16);
                tmem_ld16_nw(abase, fhh);
                tmem_ld16_nw(abase + (uint32_t)BN, fhl);
                tmem_ld16_nw(abase + (uint32_t)(2 * BN), flh);
                tmem_ld16_nw(abase + (uint32_t)(3 * BN), fll);
                tmem_wait_ld();
                reg_fence(fhh);
                reg_fence(fhl);
                reg_fence(flh);
                reg_fence(fll);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
            }
            if (WIN && f32out) {
                // the fp32 nearest-even image of v = 2^16 T + Lo (ReLU: 0 when T < 0), scaled by 2^-s
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) {
                    const int2 bt = wtab[cw * 16 + jj];
                    const int mid = __float2int_rn(__uint_as_float(fhl[jj])) + __float2int_rn(__uint_as_float(flh[jj]));
                    const int L = mid * 256 + __float2int_rn(__uint_as_float(fll[jj])) + bt.y;
                    const int T = __float2int_rn(__uint_as_float(fhh[jj])) + bt.x + (L >> 16);
                    const long long v = (a.relu && T < 0) ? 0LL : ((long long)T << 16) + (L & 0xFFFF);
                    w[jj] = __float_as_uint(__ll2float_rn(v) * a.f32_scale);
                }
            }
            // codes: in fp32 first, t = v / 2^sh within P.win_eps; only a value that close to a rounding
            // boundary (about one in a thousand) is decided by the exact 32-bit arithmetic of win_code
#pragma unroll
            for (int j = 0; j < ((WIN && !f32out) ? 8 : 0); ++j) {
                if (P.win_eps > 0.0f) {
                    float tv[2];
                    bool near = false;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int jj = 2 * j + h;
                        float x = fmaf(__uint_as_float(fhh[jj]), P.win_c[0], wtabf[cw * 16 + jj]);
                        x = fmaf(__uint_as_float(fhl[jj]) + __uint_as_float(flh[jj]), P.win_c[1], x);
                        x = fmaf(__uint_as_float(fll[jj]), P.win_c[2], x);
                        x = fminf(fmaxf(x, flo), fhi);
                        const float r = (x + 12582912.0f) - 12582912.0f;
                        near |= fabsf(x - r) > 0.5f - P.win_eps;
                        tv[h] = x;
                    }
                    w[j] = f32_codes_f16x2(tv[0], tv[1]);
                    if (near)
                        w[j] = pack_codes_f16(win_code(fhh[2 * j], fhl[2 * j], flh[2 * j], fll[2 * j], wtab[cw * 16 + 2 * j],
                                                       m, half, mmask, a.relu, lo, hi),
                                              win_code(fhh[2 * j + 1], fhl[2 * j + 1], flh[2 * j + 1], fll[2 * j + 1],
                                                       wtab[cw * 16 + 2 * j + 1], m, half, mmask, a.relu, lo, hi));
                } else {
                    w[j] = pack_codes_f16(win_code(fhh[2 * j], fhl[2 * j], flh[2 * j], fll[2 * j], wtab[cw * 16 + 2 * j], m,
                                                   half, mmask, a.relu, lo, hi),
                                          win_code(fhh[2 * j + 1], fhl[2 * j + 1], flh[2 * j + 1], fll[2 * j + 1],
                                                   wtab[cw * 16 + 2 * j + 1], m, half, mmask, a.relu, lo, hi));
                }
            }
            if (f32out) {
                // fp32 image out: this row's 16 values are 64 contiguous bytes of the output row
                const long long mrow = tile_row(P, t, row);
                if (mrow >= 0) {
                    float* yp = static_cast<float*>(a.y) + mrow * a.K + cw * 16;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (cw * 16 + 4 * q < a.K)
                            *reinterpret_cast<uint4*>(yp + 4 * q) = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                }
                continue;
            }
            const uint32_t sb = u & 1, n = u >> 1;  // staging tile and its use count
            const uint32_t sfull = sb ? stg_full2 : stg_full, sfree = sb ? stg_free2 : stg_free;
            // the store of tile u - 2 (this staging tile) must have read it
            if (n > 0 && !wait_bounded(sfree, (n - 1) & 1, abort, P.status)) {
                ok = false;
                break;
            }
            unsigned char* sbuf = sO + sb * (TC_BM * 128);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int chunk = cw * 2 + q;
                *reinterpret_cast<uint4*>(sbuf + row * 128 + ((chunk ^ (row & 7)) << 4)) =
                    make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(sfull);
        }
    } else if (warp < MMA_WARP) {
        // ============================================================ epilogue
        // Warp w drains TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31 (the quadrant a warp may access) and
        // the 32-column chunks cw * CPW .. cw * CPW + CPW - 1, cw = (w - 4) / 4, of every accumulator.
        const int quad = warp & 3;
        const int cw = (warp - 4) >> 2;
        const int row = quad * 32 + lane;
        const int nbuf = P.nbuf;
        uint32_t gcount = 0;
        bool ok = true;
        // Integer running sums of a tile live in TMEM after the accumulator buffers: columns
        // [nbuf BN, nbuf BN + BN * words), words = 1 (int32) or 2 (int64 as lo / hi column blocks).
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t run_base = (uint32_t)(nbuf * BN);
        uint32_t u = 0;  // tiles written through the staging tiles so far
        const int place = row_in_tile(P, row);
        TileIter T(P, SPLIT ? 0 : blockIdx.x);
        for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
            const int sp = SPLIT ? ut % P.ksplit : 0;
            if (SPLIT) TileIter::split(P, ut / P.ksplit, T.tn, T.iq, T.ip, T.ng);
            const int tn = T.tn;
            // -1: row outside the output (not needed where the TMA store clips)
            const long long m = FE && !DIRECT && P.fast_store ? 0 : row_at(P, T, place, row);
            if (!SPLIT) T.next(P);
            unsigned char* const stg = sO + (NSTG == 2 ? (u & 1) * STG_BYTES : 0);  // this tile's staging tile
            const int g_lo = SPLIT ? P.gs[sp] : 0, g_hi = SPLIT ? P.gs[sp + 1] : P.n_groups;
            for (int gi = g_lo; gi < g_hi; ++gi) {
                const int shift = P.g[gi].shift;
                const bool first = gi == g_lo, last = gi == g_hi - 1;
                const uint32_t buf = nbuf == 2 ? (gcount & 1) : 0;
                const uint32_t par = nbuf == 2 ? ((gcount >> 1) & 1) : (gcount & 1);
                if (!wait_bounded(accfull0 + 8 * buf, par, abort, P.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                // the store of tile u - NSTG must have read this tile's staging tile
                if (STORE_WARP && last && P.fast_store && u >= NSTG &&
                    !wait_bounded(NSTG == 2 && (u & 1) ? stg_free2 : stg_free, (u / NSTG - 1) & 1, abort, P.status)) {
                    ok = false;
                    break;
                }
#pragma unroll 1
                for (int c = 0; c < CPW; ++c) {
                    const int cb = cw * CPW + c;
                    const int k0 = tn * BN + cb * 32;
                    const uint32_t run_col = run_base + cb * 32;
                    if (!WEPI && k0 >= a.K) {  // no channel of this chunk is stored
                        if (c == CPW - 1) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
                        }
                        continue;
                    }
                    if constexpr (!FE) {
                    if (sizeof(ACC) == 8 && P.patch == 3 && P.nacc == 4 && P.fast_store && a.sh >= 1 && a.sh <= 62) {
                        // window mode, two-limb x and w, one-plane codes out: each 16-column half goes
                        // from the four limb accumulators to packed codes before the next is loaded
                        // (keeps the live 64-bit values to 16)
                        const Epi64 e64 = make_epi64(a);
                        const int k0 = tn * BN + cb * 32;
                        const uint32_t abase = lane_base + buf * (uint32_t)(P.nacc * BN) + cb * 32;
                        uint32_t w[16];
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t fhh[16], fhl[16], flh[16], fll[16];
                            tmem_ld16_nw(abase + 16 * hf, fhh);
                            tmem_ld16_nw(abase + (uint32_t)BN + 16 * hf, fhl);
                            tmem_ld16_nw(abase + (uint32_t)(2 * BN) + 16 * hf, flh);
                            tmem_ld16_nw(abase + (uint32_t)(3 * BN) + 16 * hf, fll);
                            tmem_wait_ld();
                            reg_fence(fhh);
                            reg_fence(fhl);
                            reg_fence(flh);
                            reg_fence(fll);
                            if (hf == 1 && c == CPW - 1) {
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
                            }
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                int c2[2];
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const int jj = 2 * j + h;
                                    const int k = k0 + 16 * hf + jj;
                                    const long long v = ((long long)__float2int_rn(__uint_as_float(fhh[jj])) << 16) +
                                                        ((long long)(__float2int_rn(__uint_as_float(fhl[jj])) +
                                                                     __float2int_rn(__uint_as_float(flh[jj])))
                                                         << 8) +
                                                        (long long)__float2int_rn(__uint_as_float(fll[jj]));
                                    const int32_t b = (e64.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                                    c2[h] = epi64_code<SC>(e64, v, b, SC ? scale_code(a, k) : 0,
                                                           SC ? shift_code(a, k) : 0);
                                }
                                w[8 * hf + j] = pack_codes_f16(c2[0], c2[1]);
                            }
                        }
                        unsigned char* half_buf = stg + (cb >> 1) * (TC_BM * 128);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int chunk = (cb & 1) * 4 + q;
                            *reinterpret_cast<uint4*>(half_buf + row * 128 + ((chunk ^ (row & 7)) << 4)) =
                                make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                        }
                        continue;
                    }
                    }
                    if constexpr (FE) {
                        // one exact group: codes straight from the fp32 sums
                        uint32_t f0[16], f1[16], w[16];
                        tmem_ld16_nw(lane_base + buf * BN + cb * 32, f0);
                        tmem_ld16_nw(lane_base + buf * BN + cb * 32 + 16, f1);
                        // the chunk's 32 channel constants, one per lane, to every lane through shared
                        // memory that this warp overwrites with the codes afterwards
                        const int kl = k0 + lane;
                        const bool image = a.out_mode == FXPQ_OUT_F32;
                        const int32_t b = a.has_bias && kl < a.K ? __ldg(a.bias + kl) : 0;
                        float t, ms = 0.0f;  // the channel's constants
                        if constexpr (SC) {
                            const float2 mt = fepi_scale(a, b, scale_code(a, kl), shift_code(a, kl));
                            ms = mt.x;
                            t = mt.y;
                        } else {
                            t = image ? (float)b * a.vi_b : a.has_bias ? fepi_bias(a, b) : 0.0f;
                        }
                        unsigned char* wbuf = sO + (warp - 4) * 2048;                     // DIRECT, fp32 image
                        unsigned char* half_buf = stg + (cb >> 1) * (TC_BM * 128);         // staged tile
                        // four constants 4 q .. 4 q + 3 (8 + q: the second set)
                        auto tab = [&](int q) {
                            return DIRECT || image ? wbuf + 16 * q
                                          : half_buf + (quad * 32 + (q >> 2)) * 128 + ((((cb & 1) * 4 + (q & 3)) ^ (q >> 2)) << 4);
                        };
                        *reinterpret_cast<float*>(tab(lane >> 2) + 4 * (lane & 3)) = t;
                        if constexpr (SC) *reinterpret_cast<float*>(tab(8 + (lane >> 2)) + 4 * (lane & 3)) = ms;
                        __syncwarp();
                        tmem_wait_ld();
                        reg_fence(f0);
                        reg_fence(f1);
                        if (c == CPW - 1) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
                        }
                        if (image) {
                            float v[32];
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const float4 tq = *reinterpret_cast<const float4*>(tab(q));
                                const uint32_t* f = q < 4 ? f0 + 4 * q : f1 + 4 * (q - 4);
                                float4 mq = make_float4(a.vi_c, a.vi_c, a.vi_c, a.vi_c);
                                if constexpr (SC) mq = *reinterpret_cast<const float4*>(tab(8 + q));
                                v[4 * q] = fepi_image(a, __uint_as_float(f[0]), mq.x, tq.x);
                                v[4 * q + 1] = fepi_image(a, __uint_as_float(f[1]), mq.y, tq.y);
                                v[4 * q + 2] = fepi_image(a, __uint_as_float(f[2]), mq.z, tq.z);
                                v[4 * q + 3] = fepi_image(a, __uint_as_float(f[3]), mq.w, tq.w);
                            }
                            __syncwarp();
                            store_f32_direct(a, m, k0, v, wbuf, lane);
                            continue;
                        }
                        const uint64_t cc = f32x2_splat(a.vf_c);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            const float4 tq = *reinterpret_cast<const float4*>(tab(q));
                            const uint32_t* f = q < 4 ? f0 + 4 * q : f1 + 4 * (q - 4);
                            if constexpr (SC) {
                                const float4 mq = *reinterpret_cast<const float4*>(tab(8 + q));
                                w[2 * q] = fepi_scale_pair(a, k0 + 4 * q, f[0], f[1], mq.x, mq.y, tq.x, tq.y);
                                w[2 * q + 1] = fepi_scale_pair(a, k0 + 4 * q + 2, f[2], f[3], mq.z, mq.w, tq.z, tq.w);
                                continue;
                            }
                            w[2 * q] = fepi_pair(f[0], f[1], cc, tq.x, tq.y, a.vf_lo, a.vf_hi);
                            w[2 * q + 1] = fepi_pair(f[2], f[3], cc, tq.z, tq.w, a.vf_lo, a.vf_hi);
                        }
                        __syncwarp();
                        if (DIRECT) {
                            store_codes_direct(a, m, k0, w, wbuf, lane);
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int chunk = (cb & 1) * 4 + q;
                                *reinterpret_cast<uint4*>(half_buf + row * 128 + ((chunk ^ (row & 7)) << 4)) =
                                    make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                            }
                        }
                    } else {
                    // One TMEM round trip per load batch: the fp32 group sums and, after the first group,
                    // the integer running sums are loaded together; the running-sum stores share one
                    // completion wait.
                    ACC acc[32];
                    if (sizeof(ACC) == 8 && P.patch == 3) {
                        // window mode: one accumulator per limb pair (ia, iw), combined with its weight
                        // 2^(8 ((px-1-ia) + (pw-1-iw))); each is an exact integer below 2^24
                        const uint32_t abase = lane_base + buf * (uint32_t)(P.nacc * BN) + cb * 32;
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            if (P.nacc == 4) {
                                // two-limb x and w: the four accumulators share one load round trip;
                                // v = 2^16 S_hh + 2^8 (S_hl + S_lh) + S_ll, the middle pair summed in 32 bits
                                uint32_t fhh[16], fhl[16], flh[16], fll[16];
                                tmem_ld16_nw(abase + 16 * hf, fhh);
                                tmem_ld16_nw(abase + (uint32_t)BN + 16 * hf, fhl);
                                tmem_ld16_nw(abase + (uint32_t)(2 * BN) + 16 * hf, flh);
                                tmem_ld16_nw(abase + (uint32_t)(3 * BN) + 16 * hf, fll);
                                tmem_wait_ld();
                                reg_fence(fhh);
                                reg_fence(fhl);
                                reg_fence(flh);
                                reg_fence(fll);
#pragma unroll
                                for (int j = 0; j < 16; ++j) {
                                    const int hh = __float2int_rn(__uint_as_float(fhh[j]));
                                    const int mid = __float2int_rn(__uint_as_float(fhl[j])) +
                                                    __float2int_rn(__uint_as_float(flh[j]));
                                    const int ll = __float2int_rn(__uint_as_float(fll[j]));
                                    acc[16 * hf + j] = ((ACC)hh << 16) + ((ACC)mid << 8) + (ACC)ll;
                                }
                            } else {
#pragma unroll
                                for (int j = 0; j < 16; ++j) acc[16 * hf + j] = 0;
                                for (int ia = 0; ia < a.px; ++ia)
                                    for (int iw = 0; iw < a.pw; ++iw) {
                                        uint32_t f16[16];
                                        tmem_ld16_nw(abase + (uint32_t)((ia * a.pw + iw) * BN) + 16 * hf, f16);
                                        tmem_wait_ld();
                                        reg_fence(f16);
                                        const int sh = 8 * ((a.px - 1 - ia) + (a.pw - 1 - iw));
#pragma unroll
                                        for (int j = 0; j < 16; ++j)
                                            acc[16 * hf + j] += ((ACC)__float2int_rn(__uint_as_float(f16[j]))) << sh;
                                    }
                            }
                        }
                    } else if (sizeof(ACC) == 8) {
                        // int64 running sums in 16-column halves (lo and hi words in separate column blocks)
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t f16[16], lo[16], hi[16];
                            tmem_ld16_nw(lane_base + buf * BN + cb * 32 + 16 * hf, f16);
                            if (!first) {
                                tmem_ld16_nw(lane_base + run_col + 16 * hf, lo);
                                tmem_ld16_nw(lane_base + run_col + BN + 16 * hf, hi);
                            }
                            tmem_wait_ld();
                            reg_fence(f16);
                            if (!first) {
                                reg_fence(lo);
                                reg_fence(hi);
                            }
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                ACC v = ((ACC)__float2int_rn(__uint_as_float(f16[j]))) << shift;
                                if (!first) v += (ACC)(((unsigned long long)hi[j] << 32) | lo[j]);
                                acc[16 * hf + j] = v;
                            }
                            if (!last) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) {
                                    lo[j] = (uint32_t)(unsigned long long)acc[16 * hf + j];
                                    hi[j] = (uint32_t)((unsigned long long)acc[16 * hf + j] >> 32);
                                }
                                tmem_st16_nw(lane_base + run_col + 16 * hf, lo);
                                tmem_st16_nw(lane_base + run_col + BN + 16 * hf, hi);
                            }
                        }
                        if (!last) tmem_wait_st();
                    } else {
                        // int32 running sums, 16-column halves (keeps the live registers low)
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t f16[16], run[16];
                            tmem_ld16_nw(lane_base + buf * BN + cb * 32 + 16 * hf, f16);
                            if (!first) tmem_ld16_nw(lane_base + run_col + 16 * hf, run);
                            tmem_wait_ld();
                            reg_fence(f16);
                            if (!first) reg_fence(run);
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                ACC v = ((ACC)__float2int_rn(__uint_as_float(f16[j]))) << shift;
                                if (!first) v += (ACC)(int)run[j];
                                acc[16 * hf + j] = v;
                            }
                            if (!last) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) run[j] = (uint32_t)(unsigned long long)acc[16 * hf + j];
                                tmem_st16_nw(lane_base + run_col + 16 * hf, run);
                            }
                        }
                        if (!last) tmem_wait_st();
                    }
                    if (c == CPW - 1) {
                        // every chunk of this warp is out of the accumulator buffer: free it for the
                        // next group's MMAs before the final arithmetic (one arrival per warp: same-address
                        // arrivals of every thread serialise)
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(accempty0 + 8 * buf);
                    }
                    if (!last) continue;
                    if constexpr (SPLIT) {
                        // one share of the reduction: its exact integer sums go to the partial buffer
                        if (m >= 0) {
                            // (16 bytes per store: with one value per store 64 x 4096 outputs of 4096 products took 29 us, 19 so)
                            ACC* dst = static_cast<ACC*>(P.part) + ((long long)sp * a.M + m) * a.K + k0;
                            constexpr int V = 16 / (int)sizeof(ACC);
                            if (a.K % V == 0) {
#pragma unroll
                                for (int j = 0; j < 32; j += V)
                                    if (k0 + j < a.K) {
                                        if constexpr (V == 4)
                                            *reinterpret_cast<int4*>(dst + j) = make_int4((int)acc[j], (int)acc[j + 1], (int)acc[j + 2], (int)acc[j + 3]);
                                        else
                                            *reinterpret_cast<longlong2*>(dst + j) = make_longlong2((long long)acc[j], (long long)acc[j + 1]);
                                    }
                            } else {
#pragma unroll
                                for (int j = 0; j < 32; ++j)
                                    if (k0 + j < a.K) dst[j] = acc[j];
                            }
                        }
                    } else if (P.fast_store) {
                        // 32 one-plane codes -> 4 swizzled 16-byte chunks of this row in the staging buffer
                        // (the epilogue constants are rebuilt here from the parameters rather than kept
                        // live across the tile loop)
                        uint32_t w[16];
                        const Epi32 e32 = make_epi32(a);
                        const Epi64 e64 = make_epi64(a);
                        if (sizeof(ACC) == 4 && !SC && a.v32) {
                            // the chunk's 32 biases by 16-byte loads where they are whole and aligned
                            const bool bvec = e32.has_bias && k0 + 32 <= a.K &&
                                              (reinterpret_cast<uintptr_t>(a.bias) & 15u) == 0;
#pragma unroll
                            for (int j4 = 0; j4 < 8; ++j4) {
                                int bb[4];
                                if (bvec) {
                                    const int4 v4 = __ldg(reinterpret_cast<const int4*>(a.bias + k0) + j4);
                                    bb[0] = v4.x;
                                    bb[1] = v4.y;
                                    bb[2] = v4.z;
                                    bb[3] = v4.w;
                                } else {
#pragma unroll
                                    for (int e = 0; e < 4; ++e) {
                                        const int k = k0 + 4 * j4 + e;
                                        bb[e] = (e32.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                                    }
                                }
                                int c4[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    c4[e] = epi32_code(e32, (int)acc[4 * j4 + e], (bb[e] << e32.bsl) >> e32.bsr,
                                                       min(bb[e] & e32.fmask, 1));
                                w[2 * j4] = pack_codes_f16(c4[0], c4[1]);
                                w[2 * j4 + 1] = pack_codes_f16(c4[2], c4[3]);
                            }
                        } else if (e64.ok) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                int c2[2];
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const int k = k0 + 2 * j + h;
                                    const int32_t b = (e64.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                                    c2[h] = epi64_code<SC>(e64, (long long)acc[2 * j + h], b,
                                                           SC ? scale_code(a, k) : 0, SC ? shift_code(a, k) : 0);
                                }
                                w[j] = pack_codes_f16(c2[0], c2[1]);
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                int c2[2];
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const int k = k0 + 2 * j + h;
                                    const int32_t b = (a.has_bias && k < a.K) ? __ldg(a.bias + k) : 0;
                                    c2[h] = qlayer_code(a, cblock_value<SC>(a, k, (long long)acc[2 * j + h], b));
                                }
                                w[j] = pack_codes_f16(c2[0], c2[1]);
                            }
                        }
                        if (DIRECT) {
                            store_codes_direct(a, m, k0, w, sO + (warp - 4) * 2048, lane);
                            continue;
                        }
                        unsigned char* half_buf = stg + (cb >> 1) * (TC_BM * 128);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int chunk = (cb & 1) * 4 + q;
                            *reinterpret_cast<uint4*>(half_buf + row * 128 + ((chunk ^ (row & 7)) << 4)) =
                                make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
                        }
                    } else {
                        // everything else, through the warp's 2 KiB of the (unused) staging tile
                        ACC v[32];
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = acc[j];
                        epilogue_block32<ACC, SC>(make_epi_block(a), m, k0, v, PK ? nullptr : sO + (warp - 4) * epi_buf_bytes<ACC>(), lane);
                    }
                    }
                }
                ++gcount;
                if (STORE_WARP && last && P.fast_store) {
                    // make the staging writes visible to the async proxy, then hand the tile to the store warp
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(NSTG == 2 && (u & 1) ? stg_full2 : stg_full);
                    ++u;
                }
            }
        }
    } else if (STORE_WARP && warp > MMA_WARP) {
        // ============================================================ tile stores (one thread)
        // Tile u goes out of staging tile u % NSTG once every epilogue warp has written it.  The tile is free
        // again when the store has read it; with two tiles that is waited for with the next store in flight.
        if (lane == 0 && P.fast_store) {
            TileIter T(P, blockIdx.x);
            uint32_t u = 0;
            for (int t = blockIdx.x; t < P.n_tiles; t += gridDim.x, ++u) {
                const uint32_t sb = u % NSTG;
                if (!wait_bounded(sb ? stg_full2 : stg_full, (u / NSTG) & 1, abort, P.status)) break;
                for (int hb = 0; hb < BN / 64; ++hb) {
                    const uint32_t src = smem_u32(sO + sb * STG_BYTES + hb * (TC_BM * 128));
                    if (WEPI || P.patch)
                        tma_store_4d(&P.tmap_y, T.tn * BN + hb * 64, T.iq * P.TW, T.ip * P.TH, T.ng * P.TN, src);
                    else
                        tma_store_2d(&P.tmap_y, T.tn * BN + hb * 64, T.ng * P.rows, src);
                }
                bulk_commit();
                if (NSTG == 1) {
                    bulk_wait_read0();
                    mbar_arrive(stg_free);
                } else if (u >= 1) {
                    bulk_wait_read1();  // the store of tile u - 1 has read the other staging tile
                    mbar_arrive(sb ? stg_free : stg_free2);
                }
                T.next(P);
            }
            bulk_wait0();  // every output store has completed
        }
    } else if (PK && warp > MMA_WARP) {
        // ============================================================ packed-weight converters
        pk_convert_loop<BN, SPLIT>(P, 3 + (warp - MMA_WARP - 1), lane, sP, sB, pkfull0, full0, abort);
    } else if (!WIN && P.patch == 4) {
        // ============================================================ MMA issue, 64-channel window mode
        // Per tile, tap (r, s) and 16-channel step kk: one MMA.  A is window copy s from row r: rows 128
        // bytes apart, the 8-row groups (patch rows, TW = 8) one pattern (1 KiB) apart; B the resident tap
        // block (a B stage's layout).  One barrier round per tile.
        const uint32_t copyb = (uint32_t)P.WH * 1024u;
        uint32_t stage = 0, phase = 0, gcount = 0;
        bool ok = wait_warp(wbar, 0, abort, P.status);
        tc_fence_after();
        for (int t = blockIdx.x; t < P.n_tiles && ok; t += gridDim.x) {
            const uint32_t buf = gcount & 1;
            if (!wait_warp(accempty0 + 8 * buf, ((gcount >> 1) & 1) ^ 1, abort, P.status) ||
                !wait_warp(full0 + 8 * stage, phase, abort, P.status)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t wa = smem_u32(sA) + (uint32_t)P.w64_slot0 + stage * (uint32_t)P.w64_slot_stride;
            const uint32_t d = tmem + buf * BN;
            uint32_t accum = 0;
            for (int r = 0; r < a.R; ++r)
                for (int q = 0; q < a.S; ++q) {
                    const uint64_t ad = make_sdesc(wa + (uint32_t)q * copyb + (uint32_t)r * 1024u);
                    const uint64_t bd = make_sdesc(smem_u32(sA) + (uint32_t)(r * a.S + q) * 8192u);
#pragma unroll
                    for (int kk = 0; kk < TC_BK / 16; ++kk) {
                        tc_mma(d, ad + 2 * kk, bd + 2 * kk, IDESC, accum);
                        accum = 1;
                    }
                }
            tc_commit(empty0 + 8 * stage);
            if (++stage == 2) {
                stage = 0;
                phase ^= 1;
            }
            tc_commit(accfull0 + 8 * buf);
            ++gcount;
        }
        // every MMA issued by this thread has completed once `done` fires
        tc_commit(done_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(done_bar, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
        }
    } else if (!W64 && P.patch == 3) {
        // ============================================================ MMA issue, window mode
        // Per tile and limb pair (ia, iw): R * S2/2 MMAs of K = 16 (two taps of 8 channels).  The A
        // operand of taps (r, 2sp), (r, 2sp + 1) is the window shifted by (r, 2sp) pixels: K-major
        // without swizzle, the two K core matrices one pixel (16 bytes) apart, the 8-row groups (the
        // patch rows, TW = 8) one window row apart.  B is the resident box (iw, r, sp).
        const int np = P.S2 / 2;
        const uint32_t tapb = (uint32_t)(BN * 16);
        // N = pw BN: the B operand of tap pair (r, sp) holds [W_hi | W_lo] (one plane: N = BN); its K
        // core matrices (the two taps) are pw BN 16 bytes apart, its 8-row groups 128 bytes apart
        const uint32_t idesc_w = a.pw == 2 ? make_idesc(TC_BM, 2 * BN) : IDESC;
        uint64_t bdesc[8];
        uint32_t aoff[8];  // A start of tap pair (r, sp) in the window, in 16-byte units
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = i / np, sp = i - r * np;
            bdesc[i] = make_sdesc_noswz(smem_u32(sB) + (uint32_t)(i * 2 * a.pw) * tapb, (uint32_t)a.pw * tapb, 128);
            aoff[i] = (uint32_t)((r * P.WW + 2 * sp) * 16) >> 4;
        }
        uint32_t stage = 0, phase = 0, gcount = 0;
        bool ok = wait_warp(wbar, 0, abort, P.status);
        tc_fence_after();
        for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
            const int t = SPLIT ? ut / P.ksplit : ut, sp = SPLIT ? ut - t * P.ksplit : 0;
            (void)sp;
            const uint32_t buf = gcount & 1;
            if (!wait_warp(accempty0 + 8 * buf, ((gcount >> 1) & 1) ^ 1, abort, P.status) ||
                !wait_warp(full0 + 8 * stage, phase, abort, P.status)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t d0 = tmem + buf * (uint32_t)(P.nacc * BN);
            const uint32_t wa = smem_u32(sA + stage * A_BYTES);
            for (int ia = 0; ia < a.px; ++ia) {
                // accumulators (ia, iw) at columns (ia pw + iw) BN: one MMA of N = pw BN fills the pw of them
                const uint32_t d = d0 + (uint32_t)(ia * a.pw * BN);
                const uint64_t ad0 = make_sdesc_noswz(wa + (uint32_t)(ia * P.win_bytes), 16, (uint32_t)(P.WW * 16));
                const int nt = a.R * np;  // <= 8
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i < nt) tc_mma(d, ad0 + (uint64_t)aoff[i], bdesc[i], idesc_w, i > 0 ? 1u : 0u);
            }
            tc_commit(empty0 + 8 * stage);
            if (++stage == TC_STAGES) {
                stage = 0;
                phase ^= 1;
            }
            tc_commit(accfull0 + 8 * buf);
            ++gcount;
        }
        // every MMA issued by this thread has completed once `done` fires
        tc_commit(done_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(done_bar, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
        }
    } else if (!WEPI) {
        // ============================================================ MMA issue (MMA_WARP, one elected lane)
        // Descriptors of stage 0; a stage or a 16-element k step moves the start-address field
        // (address >> 4, 14 bits) without carry since shared addresses stay below 256 KB.
        // 8-channel patch tiles: no-swizzle A, one 16-element k step = two taps = 4096 bytes
        const bool narrow_a = P.patch == 2;
        const uint64_t adesc0 = narrow_a ? make_sdesc_noswz(smem_u32(sA), 2048, 128) : make_sdesc(smem_u32(sA));
        const uint32_t a_kstep = narrow_a ? 4096u >> 4 : 2u;
        const uint64_t bdesc0 = make_sdesc(smem_u32(sB));
        uint32_t stage = 0, phase = 0, gcount = 0;
        bool ok = true;
        for (int ut = blockIdx.x; ut < (SPLIT ? P.n_units : P.n_tiles) && ok; ut += gridDim.x) {
            const int t = SPLIT ? ut / P.ksplit : ut, sp = SPLIT ? ut - t * P.ksplit : 0;
            (void)sp;
            // (channels past the last tile's rows2 are whatever the stage holds; their sums are never stored)
            const uint32_t idesc = !PK && P.rows2 && t % P.tiles_n == P.tiles_n - 1 ? P.idesc2 : IDESC;
            for (int gi = SPLIT ? P.gs[sp] : 0; gi < (SPLIT ? P.gs[sp + 1] : P.n_groups) && ok; ++gi) {
                const TcGroup g = P.g[gi];
                const uint32_t buf = P.nbuf == 2 ? (gcount & 1) : 0;
                const uint32_t par = P.nbuf == 2 ? ((gcount >> 1) & 1) : (gcount & 1);
                if (!wait_warp(accempty0 + 8 * buf, par ^ 1, abort, P.status)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + buf * BN;
                uint32_t accum = 0;
                // patch 1: a tap's last channel block has ksteps 16-channel steps, the others (and every
                // k-block of the other forms) four
                int cb = P.patch == 1 ? g.kb0 % P.kbt : 0;
                const int cb_last = P.patch == 1 ? P.kbt - 1 : -1;
                const int ksteps = (a.Cp - (P.kbt - 1) * TC_BK + 15) / 16;
                for (int kb = g.kb0; kb < g.kb1; ++kb) {
                    if (!wait_warp(full0 + 8 * stage, phase, abort, P.status)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = adesc0 + (uint64_t)((stage * A_BYTES) >> 4);
                    const uint64_t bd = bdesc0 + (uint64_t)((stage * B_BYTES) >> 4);
                    const int ns = cb == cb_last ? ksteps : TC_BK / 16;
                    if (++cb > cb_last) cb = 0;
#pragma unroll
                    for (int kk = 0; kk < TC_BK / 16; ++kk) {
                        if (kk < ns) tc_mma(d, ad + a_kstep * kk, bd + 2 * kk, idesc, accum);
                        accum = 1;
                    }
                    tc_commit(empty0 + 8 * stage);
                    if (++stage == TC_STAGES) {
                        stage = 0;
                        phase ^= 1;
                    }
                }
                if (!ok) break;
                tc_commit(accfull0 + 8 * buf);
                ++gcount;
            }
        }
        // every MMA issued by this thread has completed once `done` fires
        tc_commit(done_bar);
        const long long t0 = clock64();
        while (!mbar_try_wait(done_bar, 0) && clock64() - t0 < TC_WAIT_CYCLES) {
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
    }
}

// Patch shape of a layer's output: TW x TH pixels of TN images (see patch_shape).
struct PatchShape {
    int TW = 0, TH = 0, TN = 0;
    long long tiles = 0;
};
// What the host chose for a layer, besides its exact groups.
struct TcForm {
    bool rows_geom;   // row tiles by TMA: the im2col matrix is the stored activations
    bool narrow;      // 8 stored channels
    bool use_patch;   // patch tiles of shape ps, else (without rows_geom) gathered row tiles
    bool acc64;       // int64 running sums
    bool pk;          // packed weights are read
    int BN;           // tile width
    PatchShape ps;
};

}  // namespace tc

// The host's choices for a layer on `sms` SMs: P's exact groups (and P.kbt) and f.  path: FXPQ_CONV_PATH or null; has_ws:
// there is scratch for two shares of a split.  False: the tensor-core path cannot keep the sums exact.  Touches no device.
bool choose_form(const ConvArgs& a, const fxpq_conv_desc& d, const char* path, int sms, bool has_ws, tc::TcParams& P,
                 tc::TcForm& f);

// Launches the SC = true kernel for tile width BN (acc64: the 64-bit running-sum variant, BN = 64).
fxpq_status launch_conv_tc_scaled(const tc::TcParams& P, int BN, bool acc64, int grid, cudaStream_t st);

}  // namespace fxpq
