// fxpq_conv_tc.cu -- host side of the tensor-core C-Block (planning, tensor maps, launch) and the
// kernels without a Scale layer; the kernel itself is in fxpq_conv_tc.cuh.
#include <algorithm>
#include <cmath>

#include "fxpq_conv_tc.cuh"

namespace fxpq {

using namespace tc;

namespace {

int g_num_sms = 0;
std::mutex g_tc_mu;

// FXPQ_CONV_PATH picks among exact alternatives so that tests can compare them on the same shapes: "tc" takes patch
// tiles up to four times the gathered form's k-blocks (by default the form that takes less time)
// and space-to-depth at any size, "tc_patch" patch tiles wherever the geometry allows them, "tc_rows" 128-row tiles
// gathered by the producer warps for every layer, "tc_bn128" no 256-column tiles and "tc_bn256" them wherever the layer
// allows (by default the width whose rounds take the fewest cycles), "tc_win64" window mode's two-limb epilogue in
// 64-bit arithmetic, "tc_win32" in 32-bit integers, "tc_nowin" no window mode, "tc_iepi" the one-group layers' epilogue
// in integers, "tc_nos2d" no space-to-depth, "tc_nosplit" no split reduction, "tc_nopack" no packed weights.
bool g_tc_attr_set = false;

// Largest |limb| of a format's codes: the only plane (k <= 8) or the hi / lo limb (k > 8).
long long limb_max(const fxpq_fmt& f, int plane) {
    const long long mx = qmax_of(f), mn = -qmin_of(f);
    if (f.bits <= 8) return mx > mn ? mx : mn;
    if (plane == 1) return 255;
    const long long hmx = mx >> 8, hmn = (mn + 255) >> 8;  // |floor(code / 256)|
    return hmx > hmn ? hmx : hmn;
}

}  // namespace

int num_sms() {
    std::lock_guard<std::mutex> lk(g_tc_mu);
    if (g_num_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

// Patch shape of a layer's output: TW x TH pixels of TN images, at most 128, with the fewest tiles (a 7 x 7 map
// of 128 images takes 49 tiles like its 6272 rows do, not 128).  Only widths and heights that divide the map
// into equal counts matter; among equals the fewest images and the widest rows.
static PatchShape patch_shape(const ConvArgs& a, int max_tn) {
    PatchShape s;
    const long long ideal = (a.M + TC_BM - 1) / TC_BM;
    const int span = (256 - 1) / a.stride + 1;  // a TMA box spans at most 256 input positions
    const int wmax = span < TC_BM ? span : TC_BM;
    // i columns of patches are ceil(Q / i) wide: from the widest that fits, each distinct width with its fewest columns (rows
    // likewise).  Shapes whose padded pixels fill more tiles than the best one has are passed over.  About 1 us for 55 x
    // 55 and 56 x 56 maps, 0.5 for 112 x 112, 3 for 4095 x 4095 (every i and j tried: 3, 1.7 and 870).
    for (int i = (a.Q + wmax - 1) / wmax, tw; i <= a.Q; i = tw > 1 ? (a.Q + tw - 2) / (tw - 1) : a.Q + 1) {
        tw = (a.Q + i - 1) / i;
        const int hmax = TC_BM / tw < span ? TC_BM / tw : span;
        if (s.TW && (long long)a.N * a.P * i > s.tiles * (TC_BM / tw)) continue;
        for (int j = (a.P + hmax - 1) / hmax, th; j <= a.P; j = th > 1 ? (a.P + th - 2) / (th - 1) : a.P + 1) {
            th = (a.P + j - 1) / j;
            if (s.TW && (long long)a.N * (i * tw) * (j * th) > s.tiles * TC_BM) continue;
            int tn = TC_BM / (th * tw);
            if (tn > a.N) tn = a.N;
            if (tn > max_tn) tn = max_tn;
            const long long t = (long long)((a.N + tn - 1) / tn) * j * i;
            if (s.TW == 0 || t < s.tiles || (t == s.tiles && tn < s.TN)) s.TW = tw, s.TH = th, s.TN = tn, s.tiles = t;
            if (s.tiles == ideal && s.TN == 1) return s;
        }
    }
    return s;
}

// Builds the group table over n_kb k-blocks; returns false if the tensor-core path cannot keep the sums exact.
bool plan_tc(const ConvArgs& a, const fxpq_conv_desc& d, TcParams& P, bool& acc64, int n_kb) {
    P.a = a;
    P.RSC = a.R * a.S * a.Cp;
    const int pa = planes_of(d.fmt_x), pw = planes_of(d.fmt_w);
    int ng = 0;
    bool shifted = false;
    for (int ia = 0; ia < pa; ++ia)
        for (int iw = 0; iw < pw; ++iw) {
            const long long bound = limb_max(d.fmt_x, ia) * limb_max(d.fmt_w, iw);
            if (bound == 0) continue;
            const long long kmax = ((1LL << 24) - 1) / bound;  // taps per exact fp32 group
            int kb_per = (int)(kmax / TC_BK);
            // every partial sum of channel o is at most max|x limb| * sum_taps |w[o]| <= max|x| * w_l1:
            // below 2^24 the whole reduction is one exact group
            if (d.w_l1 > 0 && d.w_l1 < (1LL << 24) && pw == 1 && limb_max(d.fmt_x, ia) * d.w_l1 < (1LL << 24))
                kb_per = n_kb;
            if (kb_per < 1) return false;
            const int shift = 8 * ((pa - 1 - ia) + (pw - 1 - iw));
            shifted |= shift > 0;
            for (int kb0 = 0; kb0 < n_kb; kb0 += kb_per) {
                if (ng >= TC_MAX_GROUPS) return false;
                P.g[ng++] = TcGroup{kb0, kb0 + kb_per < n_kb ? kb0 + kb_per : n_kb, ia, iw, shift};
            }
        }
    P.n_groups = ng;
    double total = ldexp(1.0, d.fmt_x.bits - d.fmt_x.is_signed) * ldexp(1.0, d.fmt_w.bits - d.fmt_w.is_signed) *
                   (double)a.R * a.S * a.Cp;
    if (d.w_l1 > 0 && pw == 1)
        total = fmin(total, ldexp(1.0, d.fmt_x.bits - d.fmt_x.is_signed) * (double)d.w_l1);
    acc64 = shifted || total >= ldexp(1.0, 31) - 1.0;
    P.status = status_ptr();
    return ng > 0;
}

// FXPQ_CONV_PATH as `path` (may be null) is one of the names above.
static bool path_is(const char* path, const char* name) { return path && strcmp(path, name) == 0; }

// The host's choices for a layer: P's exact groups and f.  False: the tensor-core path cannot keep the sums exact.
bool choose_form(const ConvArgs& a, const fxpq_conv_desc& d, const char* path, int sms, bool has_ws, TcParams& P, TcForm& f) {
    auto conv_path_is = [path](const char* name) { return path_is(path, name); };
    bool& acc64 = f.acc64 = false;
    const long long row_tiles_est = (a.M + TC_BM - 1) / TC_BM;
    // Layers whose im2col matrix is the stored activations themselves: 1x1 stride-1 convolutions
    // without padding ([M][Cp] per plane) and kernels covering the whole unpadded map (P = Q = 1,
    // FC layers: [N][H W Cp]).  A 128-row A tile is then one 2-D box of [M][R S Cp].
    const bool one_by_one = a.R == 1 && a.S == 1 && a.stride == 1 && a.pad == 0 && a.x_sw == a.Cp;
    const bool whole_map = a.R == a.H && a.S == a.W && a.pad == 0 && a.P == 1 && a.Q == 1;
    const bool rows_geom = f.rows_geom = (one_by_one || whole_map) && a.M > 0 && a.M < (1LL << 31) - TC_BM &&
                           !conv_path_is("tc_rows") && !conv_path_is("tc_patch");
    // Patch tiles or gathered row tiles for every other layer, patches if a TMA box can traverse the stride: a patch takes
    // whole 64-channel blocks per tap, which may be several times the k-blocks of the gathered rows' flattened reduction,
    // each of which takes longer (a 7 x 7 512-channel layer of 128 images 95 us gathered, 31 us as patches); 8-channel
    // stride-1 inputs take boxes of one tap each (narrow)
    const bool narrow = f.narrow = a.Cp == 8;
    PatchShape& ps = f.ps = PatchShape();
    if (!rows_geom && a.P > 0 && a.Q > 0 && a.N > 0 && a.stride <= (narrow ? 1 : 8) && !conv_path_is("tc_rows"))
        ps = patch_shape(a, TC_BM);
    const int kbt = P.kbt = (a.Cp + TC_BK - 1) / TC_BK;
    const int kb_flat = (a.R * a.S * a.Cp + TC_BK - 1) / TC_BK;
    // A layer's time in a form, in us, as fitted to 1734 layers of 1 to 1500 tiles in both (the better one is met but for
    // 0.1 to 1.4% on average over their kinds, at worst 1.4 times): a round of tiles, or of a split's shares, over the SMs
    // costs 2.4 per limb pair that it drains and per k-block, on one SM of few and on one of all, 0.34 to 0.38 gathered,
    // 0.11 to 0.19 as patches and 0.15 to 0.32 where a pixel is not whole 32-byte sectors, whose boxes cost double, more
    // in wider tiles; a split its second kernel.  (By tiles and k-blocks alone the choice was up to 1.7 times off: 16-bit,
    // 3 x 3 / 2 on 13 maps of 75 x 75 x 64, 169 patches against 140 row tiles, 34.4 / 26.7.)
    const bool two_limb = a.px * a.pw > 1, lone = row_tiles_est * ((a.K + 63) / 64) <= sms;
    auto rounds = [&](long long tiles, int bn) { return (double)((tiles * ((a.K + bn - 1) / bn) + sms - 1) / sms); };
    // Tile width: 64 columns for int64 sums and at most 64 output channels, else the width whose whole rounds over the SMs
    // take the fewest cycles.  A k-block costs what its stage takes from L2 at about 80 bytes per cycle and SM (24, 32 and
    // 48 KB: 300, 410 and 615 cycles; the MMAs 228, 256 and 512); a 256-column tile of several exact groups has one
    // accumulator buffer, whose drain is not hidden.
    auto width = [&](long long tiles, bool groups) {
        const double c64 = rounds(tiles, 64) * 300, c128 = rounds(tiles, 128) * 410, c256 = rounds(tiles, 256) * (groups ? 1100 : 615);
        const int bn = c128 <= c64 ? 128 : 64;
        return a.K > 128 && !conv_path_is("tc_bn128") && c256 <= (bn == 128 ? c128 : c64) ? 256 : bn;
    };
    auto form_us = [&](bool patch) {
        const long long tiles = patch ? ps.tiles : row_tiles_est;
        const int bn = two_limb || a.K <= 64 ? 64 : width(tiles, false);
        const double n = (double)tiles * ((a.K + bn - 1) / bn), kb = patch ? a.R * a.S * kbt : kb_flat, pairs = a.px * a.pw;
        const double wide = (bn == 64 ? 300 : bn == 128 ? 410 : 615) / 300.0 - 1.0, outputs = 1e-6 * (double)a.M * a.K;
        auto per_kb = [&](double load) {
            return !patch      ? 0.34 + 0.04 * load + 0.33 * wide
                   : a.Cp % 16 ? 0.15 + 0.17 * load + 0.30 * wide
                               : 0.11 + 0.08 * load + 0.11 * wide;
        };
        double shares = 1.0;
        if (has_ws && bn == 64 && 2.0 * n <= sms) {
            shares = std::floor(std::min({sms / n, (double)TC_MAX_SPLIT, std::max(kb / 4.0, two_limb ? pairs * std::ceil(kb / 8.0) : 0.0)}));
            const bool fp32 = !two_limb && a.py == 1 && a.out_mode != FXPQ_OUT_ACC64;
            if (shares < 2.0 || (fp32 && kb * (1.0 - 1.0 / shares) * per_kb(1.0) < 1.9 + 3.5 * shares * outputs)) shares = 1.0;
        }
        const double n_rounds = std::ceil(n * shares / sms), load = n * shares / (sms * n_rounds);
        const double round = 2.4 * (1.0 + wide) * std::max(1.0, pairs / shares) - 1.0 + per_kb(load) * kb * pairs / shares;
        return (patch ? 3.4 : 4.8) + n_rounds * round + (shares > 1.0 ? 1.5 + 3.5 * shares * outputs : 0.0);
    };
    // Eight-channel patches take the gathered form's k-blocks, a box per tap: one-limb layers 1.1 to 1.4 times faster with
    // up to 40 taps (11 x 11: 17 maps of 46 x 46 33.3 / 20.7; 23 of 28 x 28 23.8 / 12.6), two-limb ones only with few
    // (128 channels, 3 x 3, 1568 tiles: 134 / 140; 64 channels, 7 x 7: 132 / 114) and up to 256 output channels (344
    // channels, 3 x 3, 3198 tiles: 235 / 207).
    // Overlapping pixels (the flat space-to-depth form) are read by patches whatever they cost: a tensor map has the
    // strides that the gather does not look at.
    const bool overlap = a.x_sw != a.Cp;
    const bool any_patch = conv_path_is("tc") || conv_path_is("tc_bn256");
    const bool worth = narrow      ? any_patch || (two_limb ? !lone && a.R * a.S <= 16 && a.K <= 256 : a.R * a.S <= 40)
                       : any_patch ? (double)ps.tiles * a.R * a.S * kbt <= 4.0 * (double)row_tiles_est * kb_flat
                                   : form_us(true) <= form_us(false);
    bool& use_patch = f.use_patch;
    use_patch = ps.TW > 0 && (overlap || conv_path_is("tc_patch") || worth);
    if (overlap && !use_patch && !rows_geom) return false;
    if (use_patch && !narrow && !plan_tc(a, d, P, acc64, a.R * a.S * kbt)) {  // too many groups: gathered, if that has fewer
        if (overlap) return false;
        use_patch = false;
    }
    if (!(use_patch && !narrow) && !plan_tc(a, d, P, acc64, kb_flat)) return false;
    // ... with few row tiles (FC layers at small batches) they take 256-column tiles and a split
    // reduction fills the SMs: the MMA thread's fixed cost per k-block is then hidden, and the weights
    // stream at the memory's rate
    const bool wide_split = rows_geom && !acc64 && !a.has_scale && has_ws && a.K > 128 && !conv_path_is("tc_bn128") &&
                            !conv_path_is("tc_nosplit") && row_tiles_est * ((a.K + 255) / 256) * 2 <= sms &&
                            (kb_flat * a.px * a.pw >= 32 || d.d_wpacked);  // (shorter ones are not split, see below)
    int& BN = f.BN = 64;
    if (acc64 || a.K <= 64)
        BN = 64;
    else if (wide_split || (a.K > 128 && conv_path_is("tc_bn256")))
        BN = 256;
    else
        BN = width(use_patch ? ps.tiles : row_tiles_est, P.n_groups > 1);
    // packed k-bit weights (k <= 8, one plane) are read by the 256-column TMA-row instances of the
    // split (FC) layers, whose weights stream through once; elsewhere every weight tile is expanded
    // once per row tile and the fp16 codes are read instead
    f.pk = d.d_wpacked && d.fmt_w.bits <= 8 && BN == 256 && wide_split && (reinterpret_cast<uintptr_t>(d.d_wpacked) & 15) == 0 &&
           !conv_path_is("tc_nopack");
    return true;
}

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link-time driver dependency).
EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    std::lock_guard<std::mutex> lk(g_tc_mu);
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}
}  // namespace

fxpq_status launch_conv_tc(const ConvArgs& a, const fxpq_conv_desc& d, cudaStream_t st, bool& launched, void* ws,
                           size_t ws_bytes) {
    launched = false;
    // (read once: a search of the environment takes about as long as encoding a tensor map)
    const char* const path = getenv("FXPQ_CONV_PATH");
    auto conv_path_is = [path](const char* name) { return path_is(path, name); };
    TcParams P;
    TcForm f;
    const int sms = num_sms();
    const bool two_shares = ws && ws_bytes / 2 >= (size_t)a.M * a.K * sizeof(int);  // room for a split
    if (!choose_form(a, d, path, sms, two_shares, P, f)) return FXPQ_OK;
    const bool rows_geom = f.rows_geom, narrow = f.narrow, use_patch = f.use_patch, two_limb = a.px * a.pw > 1;
    const PatchShape& ps = f.ps;
    bool acc64 = f.acc64;
    int BN = f.BN;
    P.pk = f.pk;
    P.wpack = static_cast<const uint32_t*>(d.d_wpacked);
    P.wk = d.fmt_w.bits;
    P.wsigned = d.fmt_w.is_signed;
    P.K_pad = (a.K + 255) / 256 * 256;
    // BN = 256 fills TMEM with two accumulator buffers; with several exact groups per tile it keeps one
    // buffer and the integer running sums
    P.nbuf = (BN == 256 && P.n_groups > 1) ? 1 : 2;
    {
        EncodeTiledFn enc = encode_tiled();
        if (!enc) return FXPQ_OK;  // no tensor-map encoder: the CUDA-core kernel runs instead
        const cuuint64_t dims[3] = {(cuuint64_t)P.RSC, (cuuint64_t)a.K, (cuuint64_t)a.pw};
        const cuuint64_t strides[2] = {(cuuint64_t)P.RSC * 2, (cuuint64_t)a.K * P.RSC * 2};
        const cuuint32_t box[3] = {(cuuint32_t)TC_BK, (cuuint32_t)BN, 1};
        const cuuint32_t es[3] = {1, 1, 1};
        if (enc(&P.tmap_w, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(a.w), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return FXPQ_OK;
        P.rows2 = a.K % BN ? (a.K % BN + 7) / 8 * 8 : 0;
        P.idesc2 = make_idesc(TC_BM, (P.rows2 + 15) / 16 * 16);
        if (P.rows2) {
            const cuuint32_t box2[3] = {(cuuint32_t)TC_BK, (cuuint32_t)P.rows2, 1};
            if (enc(&P.tmap_w2, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(a.w), dims, strides, box2, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return FXPQ_OK;
        }
        P.patch = 0;
        P.rows_tma = 0;
        P.rows = TC_BM;
        P.w32 = 0;
        P.wf32 = 0;
        P.win_eps = P.win_c[0] = P.win_c[1] = P.win_c[2] = 0.0f;
        P.nacc = 1;
        P.TH = P.TW = P.TN = P.tiles_p = P.tiles_q = 1;
        // window mode for 8-channel stride-1 layers with at most 64 output channels: 8 x 16 output
        // patches, one input window per tile and limb plane, weights resident in shared memory, one
        // exact fp32 accumulator per limb pair (R * S2 * 8 products each); with several limb pairs, as one
        // pair's sums take the fp32 epilogue of the patch tiles (3 x 3, 64 channels, 8-bit, 6272 tiles: 188 us as
        // windows, 130 as patches; 16-bit, 1568 tiles: 23 / 103)
        {
            const int S2 = (a.S + 1) & ~1;
            const int WW = 8 + S2 - 1, WH = 16 + a.R - 1;
            const int win_bytes = (WW * WH * 16 + 127) / 128 * 128;
            bool ok = two_limb && a.stride == 1 && a.Cp == 8 && a.x_sw == 8 && a.K <= 64 && a.N > 0 && a.R * S2 <= 16 && 8 * WW <= 256 &&
                      WH <= 256 && a.px * win_bytes <= TC_BM * TC_BK * 2 &&
                      a.pw * a.R * (S2 / 2) * 64 * 32 <= tc_stages(64) * 64 * TC_BK * 2 && !conv_path_is("tc_rows") &&
                      !conv_path_is("tc_nowin");
            for (int ia = 0; ok && ia < a.px; ++ia)
                for (int iw = 0; iw < a.pw; ++iw)
                    if ((double)limb_max(d.fmt_x, ia) * limb_max(d.fmt_w, iw) * a.R * S2 * 8 >= 16777216.0) ok = false;
            if (ok) {
                // the input as [planes][N][H][W * 8]: one window row (WW pixels of 8 channels) is a single
                // 16 WW-byte run of the box rather than WW 16-byte rows
                const cuuint64_t xdims[4] = {(cuuint64_t)a.W * 8, (cuuint64_t)a.H, (cuuint64_t)a.N, (cuuint64_t)a.px};
                const cuuint64_t xstrides[3] = {(cuuint64_t)a.W * 16, (cuuint64_t)a.H * a.W * 16, (cuuint64_t)a.x_ps * 2};
                const cuuint32_t xbox[4] = {(cuuint32_t)(8 * WW), (cuuint32_t)WH, 1, 1};
                // weights as {c, out channel, s, r, plane} (strides in that order, not memory order)
                const cuuint64_t wdims[5] = {8, (cuuint64_t)a.K, (cuuint64_t)a.S, (cuuint64_t)a.R, (cuuint64_t)a.pw};
                const cuuint64_t wstrides[4] = {(cuuint64_t)a.R * a.S * 16, 16, (cuuint64_t)a.S * 16,
                                                (cuuint64_t)a.w_ps * 2};
                const cuuint32_t wbox[5] = {8, 64, 1, 1, 1};  // one tap of one plane
                const cuuint32_t es5[5] = {1, 1, 1, 1, 1};
                CUtensorMap mx, mw;
                if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<__half*>(a.x), xdims, xstrides, xbox, es5,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS &&
                    enc(&mw, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<__half*>(a.w), wdims, wstrides, wbox, es5,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
                    P.tmap_x = mx;
                    P.tmap_w = mw;
                    P.patch = 3;
                    P.TW = 8;
                    P.TH = 16;
                    P.tiles_p = (a.P + 15) / 16;
                    P.tiles_q = (a.Q + 7) / 8;
                    P.S2 = S2;
                    P.WW = WW;
                    P.WH = WH;
                    P.win_bytes = win_bytes;
                    P.nacc = a.px * a.pw;
                    P.n_groups = 1;
                    P.g[0] = TcGroup{0, 1, 0, 0, 0};
                    P.nbuf = 2;
                    BN = 64;
                    acc64 = true;  // the int64 instance: its TMEM holds two buffers of the limb accumulators
                    // 32-bit epilogue of two-limb x and w (v = 2^16 T + Lo, see the kernel): every limb
                    // sum covers R * S2 * 8 products; L = 2^8 (S_hl + S_lh) + S_ll + Lo(B') and T must stay
                    // below 2^31, the aligned bias must not be finer than the sums (delta >= 0), and
                    // sh - 16 in [0, 30]; the per-channel bias tables take the last 768 bytes of the B region
                    const bool codes32 = a.out_mode == FXPQ_OUT_CODES && a.py == 1 && a.sh >= 16 && a.sh <= 46;
                    const bool image32 = a.out_mode == FXPQ_OUT_F32 && a.K % 4 == 0;  // the fp32 image
                    if (a.px == 2 && a.pw == 2 && !a.has_scale && a.delta >= 0 && (codes32 || image32) &&
                        a.pw * a.R * (S2 / 2) * 64 * 32 + 768 <= tc_stages(64) * 64 * TC_BK * 2) {
                        const double taps = (double)a.R * S2 * 8;
                        const double hh = (double)limb_max(d.fmt_x, 0) * limb_max(d.fmt_w, 0) * taps;
                        const double hl = (double)limb_max(d.fmt_x, 0) * limb_max(d.fmt_w, 1) * taps;
                        const double lh = (double)limb_max(d.fmt_x, 1) * limb_max(d.fmt_w, 0) * taps;
                        const double ll = (double)limb_max(d.fmt_x, 1) * limb_max(d.fmt_w, 1) * taps;
                        const double bb = a.has_bias ? ldexp(1.0, d.fmt_b.bits - d.fmt_b.is_signed + a.delta) : 0.0;
                        const double Lb = 256.0 * (hl + lh) + ll + 65536.0;
                        const double Tb = hh + bb / 65536.0 + 1.0 + Lb / 65536.0 + 1.0;
                        const bool ok32 = Lb < ldexp(1.0, 31) && Tb < ldexp(1.0, 31) && !conv_path_is("tc_win64");
                        P.w32 = ok32 && codes32;
                        P.wf32 = ok32 && image32;
                        if (P.w32) {
                            // t = hh 2^(16-sh) + B' 2^-sh, + mid 2^(8-sh), + ll 2^-sh: every step is off by at
                            // most 2^-24 of its result, which for a t inside the clip levels (widened by one)
                            // is at most `top`, plus the terms still to come; so are mid and the constant.
                            // Beyond one 64th the exact arithmetic would run too often.
                            const double u = ldexp(1.0, -a.sh), top = (double)(a.hi > -a.lo ? a.hi : -a.lo) + 2.0;
                            const double tm = (hl + lh) * 256.0 * u, tl = ll * u;
                            const double eps = ldexp(1.0, -24) * ((top + tm + tl) + tm + (top + tl) + top + bb * u) * 1.25;
                            for (int i = 0; i < 3; ++i) P.win_c[i] = (float)ldexp(u, 16 - 8 * i);
                            P.win_eps = eps < 1.0 / 64 && !conv_path_is("tc_win32") ? (float)eps : 0.0f;
                        }
                    }
                }
            }
        }
        // 64-channel window mode (W64 instance) for one-plane stride-1 layers with at most 64 output
        // channels, kernels up to 3 x 3, a reduction of one exact group and one-plane codes out (VGG
        // conv1_2): 8 x 16 output patches, the weights resident (one 8 KiB swizzled block per tap), then
        // two window slots of S copies (shifted by 0 .. S - 1 pixels) of TH + R - 1 rows of 8 pixels
        if (P.patch == 0 && BN == 64 && a.K <= 64 && !acc64 && a.stride == 1 && a.Cp == 64 && a.px == 1 &&
            a.pw == 1 && P.n_groups == 1 && a.N > 0 && a.P > 0 && a.Q > 0 && a.R <= 3 && a.S <= 3 &&
            ((a.out_mode == FXPQ_OUT_CODES && a.py == 1 && (a.v32 || (a.sh >= 1 && a.sh <= 62))) ||
             (a.out_mode == FXPQ_OUT_F32 && a.K % 4 == 0)) &&
            !a.has_scale &&
            !conv_path_is("tc_rows") && !conv_path_is("tc_patch") && !conv_path_is("tc_nowin")) {
            const int WH = 16 + a.R - 1;
            const long long slot = (long long)a.S * WH * 1024;
            const long long wb = (long long)a.R * a.S * 8192;
            if (wb + 2 * slot <= TC_W64_SO) {
                const cuuint64_t xdims[4] = {(cuuint64_t)a.Cp, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.N};
                const cuuint64_t xstrides[3] = {(cuuint64_t)a.x_sw * 2, (cuuint64_t)a.x_sh * 2, (cuuint64_t)a.x_sn * 2};
                const cuuint32_t xbox[4] = {64, 8, (cuuint32_t)WH, 1};
                const cuuint32_t es4[4] = {1, 1, 1, 1};
                CUtensorMap mx;
                if (enc(&mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<__half*>(a.x), xdims, xstrides, xbox, es4,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
                    P.tmap_x = mx;  // the weights keep the tiled map above (box {64, 64}: one tap)
                    P.patch = 4;
                    P.TW = 8;
                    P.TH = 16;
                    P.tiles_p = (a.P + 15) / 16;
                    P.tiles_q = (a.Q + 7) / 8;
                    P.WW = 8;
                    P.WH = WH;
                    P.win_bytes = (int)slot;
                    P.w64_slot0 = (int)wb;
                    P.w64_slot_stride = (int)slot;
                    P.nbuf = 2;
                }
            }
        }
        if (P.patch == 0 && rows_geom) {
            const cuuint64_t xdims[3] = {(cuuint64_t)P.RSC, (cuuint64_t)a.M, (cuuint64_t)a.px};
            const cuuint64_t xstrides[2] = {(cuuint64_t)P.RSC * 2, (cuuint64_t)a.x_ps * 2};
            const long long parts = (a.M + TC_BM - 1) / TC_BM;
            const int rows = (int)(((a.M + parts - 1) / parts + 7) / 8 * 8);
            const cuuint32_t xbox[3] = {(cuuint32_t)TC_BK, (cuuint32_t)rows, 1};
            if (enc(&P.tmap_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(a.x), xdims, xstrides, xbox, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
                P.rows_tma = 1;
                P.rows = rows;
            }
        }
        if (P.patch == 0 && !P.rows_tma && use_patch) {
            const cuuint64_t xdims[5] = {(cuuint64_t)a.Cp, (cuuint64_t)a.W, (cuuint64_t)a.H, (cuuint64_t)a.N, (cuuint64_t)a.px};
            const cuuint64_t xstrides[4] = {(cuuint64_t)a.x_sw * 2, (cuuint64_t)a.x_sh * 2, (cuuint64_t)a.x_sn * 2, (cuuint64_t)a.x_ps * 2};
            const cuuint32_t st = (cuuint32_t)a.stride;
            const cuuint32_t xbox[5] = {(cuuint32_t)(narrow ? 8 : TC_BK), (ps.TW - 1) * st + 1, (ps.TH - 1) * st + 1,
                                        (cuuint32_t)ps.TN, 1};
            const cuuint32_t es5[5] = {1, st, st, 1, 1};
            if (enc(&P.tmap_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<__half*>(a.x), xdims, xstrides, xbox, es5,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, narrow ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return FXPQ_OK;  // the groups are in patch order: the CUDA-core kernel runs instead
            P.patch = narrow ? 2 : 1;
            P.TW = ps.TW;
            P.TH = ps.TH;
            P.TN = ps.TN;
            P.tiles_p = (a.P + ps.TH - 1) / ps.TH;
            P.tiles_q = (a.Q + ps.TW - 1) / ps.TW;
        }
        if (!P.rows_tma) P.pk = 0;
        if (P.w32 && !(a.out_mode == FXPQ_OUT_CODES && a.py == 1)) P.w32 = 0;
        if (P.wf32 && a.out_mode != FXPQ_OUT_F32) P.wf32 = 0;
        // one-plane codes: stage the tile in shared memory and write it with TMA stores (not with packed
        // weights, whose staging region holds the packed stages)
        P.fast_store = 0;
        if (a.out_mode == FXPQ_OUT_CODES && a.py == 1 && !P.pk) {
            CUresult r;
            if (P.patch) {
                const cuuint64_t ydims[4] = {(cuuint64_t)a.K, (cuuint64_t)a.Q, (cuuint64_t)a.P, (cuuint64_t)a.N};
                const cuuint64_t ystrides[3] = {(cuuint64_t)a.K * 2, (cuuint64_t)a.Q * a.K * 2,
                                                (cuuint64_t)a.P * a.Q * a.K * 2};
                const cuuint32_t ybox[4] = {64, (cuuint32_t)P.TW, (cuuint32_t)P.TH, (cuuint32_t)P.TN};
                const cuuint32_t es4[4] = {1, 1, 1, 1};
                r = enc(&P.tmap_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, a.y, ydims, ystrides, ybox, es4,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            } else {
                const cuuint64_t ydims[2] = {(cuuint64_t)a.K, (cuuint64_t)a.M};
                const cuuint64_t ystrides[1] = {(cuuint64_t)a.K * 2};
                const cuuint32_t ybox[2] = {64, (cuuint32_t)P.rows};
                r = enc(&P.tmap_y, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, a.y, ydims, ystrides, ybox, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            }
            P.fast_store = r == CUDA_SUCCESS;
        }
        if (!P.fast_store) P.w32 = 0;  // the 32-bit window epilogue writes through the staging tile
    }
    P.tiles_m = P.patch ? (a.N + P.TN - 1) / P.TN * P.tiles_p * P.tiles_q : (int)((a.M + TC_BM - 1) / TC_BM);
    P.tiles_n = (a.K + BN - 1) / BN;
    P.n_tiles = P.tiles_m * P.tiles_n;
    if (P.n_tiles == 0) {
        launched = true;
        return FXPQ_OK;
    }
    // the fp32 epilogue, for a layer of one exact group that is not split
    const bool fp32_epi = ((a.vf && P.fast_store) || (a.vi && a.K % 4 == 0) ||
                           (a.vs && (P.fast_store || (a.out_mode == FXPQ_OUT_F32 && a.K % 4 == 0)))) &&
                          P.n_groups == 1 && P.g[0].shift == 0 && P.patch != 3 && !P.pk && !acc64 && !conv_path_is("tc_iepi");
    // Split reduction for layers whose tiles cannot occupy the SMs (FC layers, small batches) and whose
    // reduction is long: ks units share every tile's k-blocks (share s of every exact group), and their
    // exact integer sums meet in the workspace.
    P.ksplit = 1;
    P.part = nullptr;
    P.gs[0] = 0;
    P.gs[1] = P.n_groups;
    // (64-column tiles and 256-column TMA-row tiles: the instantiations that carry the split; a Scale layer is
    // applied by the second kernel)
    if (P.patch != 3 && P.patch != 4 && (BN == 64 || (BN == 256 && P.rows_tma && !acc64)) && ws &&
        P.n_tiles * 2 <= sms && !conv_path_is("tc_nosplit")) {
        const int ng = P.n_groups;
        int min_len = 1 << 30;
        for (int gi = 0; gi < ng; ++gi) min_len = std::min(min_len, P.g[gi].kb1 - P.g[gi].kb0);
        const size_t share = (size_t)a.M * a.K * (acc64 ? sizeof(long long) : sizeof(int));
        const int cap = std::min(sms / P.n_tiles, (int)std::min<size_t>(ws_bytes / share, TC_MAX_SPLIT));
        // long groups: each share takes a sub-range of every group (at least four k-blocks); many short
        // groups (two-limb layers): each share takes whole groups
        int ks_sub = std::min(cap, std::min(min_len / 4, TC_MAX_GROUPS / ng));
        int ks_whole = std::min(cap, ng);
        // The second kernel costs about 1.9 us and 3.5 per million values and share, 1.6 and 2.5 where it takes a Scale layer's
        // work off the tiles; a k-block of a tile that has its SM to itself 0.19 to 0.38 us (choose_form): a layer with the
        // fp32 epilogue is split if that shortens the chain by more (FC layers' 256-column tiles: by 12 k-blocks).  Other
        // epilogues run once per tile in one kernel take 4 to 8 us, and the second kernel spreads them: split if anything is
        // saved, for one-plane codes (staged, the shorter ones) if that pays for the shares' traffic as well (334 small
        // layers: 0 to 0.5% off the better of both on average, 16% with 24 k-blocks for all; 9 k-blocks to 16-bit codes, 825
        // x 240 outputs, 14.4 us whole, 8.5 split; 16-bit, 8 k-blocks, 20 x 120 int64 sums 15.4 / 7.1; 2 k-blocks, 0.33 M
        // one-plane codes 11.6 / 14.4; 25 k-blocks, 0.54 M codes with the fp32 epilogue 8.9 / 12.0, 18 and 0.1 M 7.0 / 7.4;
        // ResNet-18's Scale layers of one image, where only those of 14 and more saved k-blocks are split, 172 us, none of
        // 14 177, all 179)
        int total = 0;
        for (int gi = 0; gi < ng; ++gi) total += P.g[gi].kb1 - P.g[gi].kb0;
        const double outputs = 1e-6 * (double)a.M * a.K, per_kb = !P.patch && !P.rows_tma ? 0.38 : P.patch && a.Cp % 16 ? 0.31 : 0.19;
        auto pays = [&](int ks) {
            const double saved = total - total / std::max(ks, 1);
            return saved >= (BN == 256      ? (fp32_epi ? 12.0 : 1.0)
                             : fp32_epi     ? (a.has_scale ? 1.6 + 2.5 * ks * outputs : 1.9 + 3.5 * ks * outputs) / per_kb
                             : P.fast_store ? 1.0 + 16.0 * outputs
                                            : 1.0);
        };
        if (!pays(ks_sub)) ks_sub = 1;
        if (!pays(ks_whole)) ks_whole = 1;
        if (ks_sub >= 2 && ks_sub >= ks_whole) {
            TcGroup g0[TC_MAX_GROUPS];
            for (int gi = 0; gi < ng; ++gi) g0[gi] = P.g[gi];
            for (int s = 0; s < ks_sub; ++s) {
                for (int gi = 0; gi < ng; ++gi) {
                    const int len = g0[gi].kb1 - g0[gi].kb0;
                    TcGroup g = g0[gi];
                    g.kb0 = g0[gi].kb0 + (int)((long long)len * s / ks_sub);
                    g.kb1 = g0[gi].kb0 + (int)((long long)len * (s + 1) / ks_sub);
                    P.g[s * ng + gi] = g;
                }
                P.gs[s] = s * ng;
            }
            P.gs[ks_sub] = ks_sub * ng;
            P.ksplit = ks_sub;
        } else if (ks_whole >= 2) {
            for (int s = 0; s <= ks_whole; ++s) P.gs[s] = (int)((long long)ng * s / ks_whole);
            P.ksplit = ks_whole;
        }
        if (P.ksplit > 1) {
            P.part = ws;
            P.fast_store = 0;
        }
    }
    P.n_units = P.n_tiles * P.ksplit;
    P.fepi = fp32_epi && P.ksplit == 1;
    {
        std::lock_guard<std::mutex> lk(g_tc_mu);
        if (!g_tc_attr_set) {
            if (cudaFuncSetAttribute(conv_tc_kernel<64, long long, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<64>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, long long, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<64>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, int, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<64>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, int, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<64>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, int, false, false, false, false, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<64>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<128, int, false, false, false, false, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<128>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<256, int, false, false, false, false, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_bytes<256>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<128, int, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<128>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<256, int, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<256>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<256, int, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<256>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<256, int, false, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<256, true>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<256, int, false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)tc_smem_bytes<256, true>()) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, long long, false, false, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(tc_smem_bytes<64>())) != cudaSuccess ||
                cudaFuncSetAttribute(conv_tc_kernel<64, int, false, false, false, false, true>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem_w64()) != cudaSuccess)
                return FXPQ_ERR_CUDA;
            g_tc_attr_set = true;
        }
    }
    const int grid = P.n_units < sms ? P.n_units : sms;
    TileIter::split(P, grid, P.step_n, P.step_q, P.step_p, P.step_g);
    launched = true;
    if (a.has_scale && P.ksplit == 1) return launch_conv_tc_scaled(P, BN, acc64, grid, st);
    if (P.patch == 3 && (P.w32 || P.wf32))  // window mode, 32-bit two-limb epilogue: its own instance (never split)
        launch_pdl(conv_tc_kernel<64, long long, false, false, false, true>, grid, tc_threads_win(), tc_smem_bytes<64>(), st, P);
    else if (P.patch == 4 && (P.fast_store || a.out_mode == FXPQ_OUT_F32))
        // 64-channel window mode: the instance with its own shared-memory layout and 16 epilogue warps
        launch_pdl(conv_tc_kernel<64, int, false, false, false, false, true>, grid, tc_threads_win(), tc_smem_w64(), st, P);
    else if (P.patch == 4) {
        launched = false;  // no TMA store of the output: the CUDA-core kernel runs instead
        return FXPQ_OK;
    }
    else if (P.pk && P.ksplit > 1)
        launch_pdl(conv_tc_kernel<256, int, false, true, true>, grid, tc_threads_pk(256, true), tc_smem_bytes<256, true>(), st, P);
    else if (P.pk)
        launch_pdl(conv_tc_kernel<256, int, false, false, true>, grid, tc_threads_pk(256, true), tc_smem_bytes<256, true>(), st, P);
    else if (P.ksplit > 1 && BN == 256)
        launch_pdl(conv_tc_kernel<256, int, false, true>, grid, tc_threads(256), tc_smem_bytes<256>(), st, P);
    else if (P.ksplit > 1 && acc64)
        launch_pdl(conv_tc_kernel<64, long long, false, true>, grid, tc_threads(64), tc_smem_bytes<64>(), st, P);
    else if (P.ksplit > 1)
        launch_pdl(conv_tc_kernel<64, int, false, true>, grid, tc_threads(64), tc_smem_bytes<64>(), st, P);
    else if (P.fepi && BN == 64)
        launch_pdl(conv_tc_kernel<64, int, false, false, false, false, false, true>, grid, tc_threads(64), tc_smem_bytes<64>(), st, P);
    else if (P.fepi && BN == 128)
        launch_pdl(conv_tc_kernel<128, int, false, false, false, false, false, true>, grid, tc_threads(128), tc_smem_bytes<128>(), st, P);
    else if (P.fepi)
        launch_pdl(conv_tc_kernel<256, int, false, false, false, false, false, true>, grid, tc_threads(256), tc_smem_bytes<256>(), st, P);
    else if (acc64)
        launch_pdl(conv_tc_kernel<64, long long, false>, grid, tc_threads(64), tc_smem_bytes<64>(), st, P);
    else if (BN == 64)
        launch_pdl(conv_tc_kernel<64, int, false>, grid, tc_threads(64), tc_smem_bytes<64>(), st, P);
    else if (BN == 128)
        launch_pdl(conv_tc_kernel<128, int, false>, grid, tc_threads(128), tc_smem_bytes<128>(), st, P);
    else
        launch_pdl(conv_tc_kernel<256, int, false>, grid, tc_threads(256), tc_smem_bytes<256>(), st, P);
    launched = true;
    const fxpq_status s = after_launch("conv_tc");
    if (s != FXPQ_OK || P.ksplit == 1) return s;
    return launch_splitk_reduce(a, P.part, P.ksplit, acc64, st);
}

}  // namespace fxpq

// ------------------------------------------------------------------------------------------
// Failure detection: the kernels' bounded mbarrier wait, run on a barrier that nothing arrives on.
// ------------------------------------------------------------------------------------------
namespace {
__global__ void wait_selftest_kernel(long long limit, int* status) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    abort_flag = 0;
    const uint32_t b = fxpq::tc::smem_u32(&bar);
    fxpq::tc::mbar_init(b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // phase 0 of the barrier never completes: the wait runs out, latches the status and returns
    fxpq::tc::wait_bounded_for(b, 0, &abort_flag, status, limit);
}
}  // namespace

extern "C" fxpq_status fxpq_selftest_wait_timeout(int64_t limit_cycles, void* stream) {
    if (limit_cycles < 1 || limit_cycles > 100000000LL) return FXPQ_ERR_INVALID_ARG;
    wait_selftest_kernel<<<1, 1, 0, fxpq::as_stream(stream)>>>(limit_cycles, fxpq::status_ptr());
    return fxpq::after_launch("wait_selftest");
}
