// fxpq_conv.cu -- C-Block on integer codes (Sec. IV-B): convolution / FC with exact integer
// accumulation and the fused epilogue (bias alignment, ReLU, FxP-QLayer shift-requantize).
//
// This translation unit holds the CUDA-core implicit-GEMM kernel (exact int32 / int64 MACs),
// used for every shape, and the host entry points.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include "fxpq_common.cuh"
#include "fxpq_conv.cuh"

namespace fxpq {
namespace {

__device__ __forceinline__ int load_code(const __half* __restrict__ t, long long row, int Cp, int planes, int c,
                                         long long plane_stride) {
    return code_get(t, row * Cp + c, planes, plane_stride);
}

constexpr int TM = 64, TN = 64, TK = 16, NT = 256;

template <typename ACC>
__global__ void __launch_bounds__(NT) conv_simt_kernel(ConvArgs a) {
    __shared__ int As[TK][TM + 1];
    __shared__ int Bs[TK][TN + 1];
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const long long M = (long long)a.N * a.P * a.Q;
    const long long m0 = (long long)blockIdx.x * TM;
    const int n0 = blockIdx.y * TN;

    // per-thread loader coordinates: 4 (row, channel) entries of the A and B tiles
    long long pix_n[4];
    int pix_p[4], pix_q[4];
    bool pix_ok[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        int e = tid + NT * i;
        long long m = m0 + (e >> 4);
        pix_ok[i] = m < M;
        long long mm = pix_ok[i] ? m : 0;
        pix_n[i] = mm / ((long long)a.P * a.Q);
        int pq = (int)(mm - pix_n[i] * a.P * a.Q);
        pix_p[i] = pq / a.Q;
        pix_q[i] = pq - pix_p[i] * a.Q;
    }

    ACC acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;

    for (int r = 0; r < a.R; ++r)
        for (int s = 0; s < a.S; ++s)
            for (int c0 = 0; c0 < a.Cp; c0 += TK) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    int e = tid + NT * i;
                    int cc = e & (TK - 1);
                    int row = e >> 4;
                    int c = c0 + cc;
                    int code = 0;
                    int h = pix_p[i] * a.stride + r - a.pad;
                    int w = pix_q[i] * a.stride + s - a.pad;
                    if (pix_ok[i] && c < a.Cp && h >= 0 && h < a.H && w >= 0 && w < a.W)
                        code = load_code(a.x, (pix_n[i] * a.H + h) * a.W + w, a.Cp, a.px, c, a.x_ps);
                    As[cc][row] = code;
                    int k = n0 + row;
                    int wc = 0;
                    if (k < a.K && c < a.Cp)
                        wc = load_code(a.w, ((long long)k * a.R + r) * a.S + s, a.Cp, a.pw, c, a.w_ps);
                    Bs[cc][row] = wc;
                }
                __syncthreads();
#pragma unroll
                for (int cc = 0; cc < TK; ++cc) {
                    int av[4], bv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) av[i] = As[cc][ty * 4 + i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) bv[j] = Bs[cc][tx * 4 + j];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] += (ACC)av[i] * (ACC)bv[j];
                }
                __syncthreads();
            }

#pragma unroll
    for (int i = 0; i < 4; ++i) {
        long long m = m0 + ty * 4 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            int k = n0 + tx * 4 + j;
            if (k < a.K) cblock_epilogue_store(a, m, k, (long long)acc[i][j]);
        }
    }
}

// Codes of a strided 8-channel layer to the space-to-depth form (S2dPlan): blocks [0, xb) one thread per pixel of
// x2 and plane, the rest one thread per 8 weights.  HBM-bound (16 bytes read per pixel and plane, st st C2 / (8 C)
// times less written): 128 224 x 224 images, stride 2, 60 us.
__global__ void __launch_bounds__(256) s2d_kernel(const __half* __restrict__ x, const __half* __restrict__ w, int N, int H,
                                                  int W, int K, int R, int S, int pad, long long x_ps, long long w_ps,
                                                  S2dPlan p, int px, int pw, unsigned xb, uint4* __restrict__ x2,
                                                  uint4* __restrict__ w2) {
    pdl_wait();
    const int c8 = p.C2 / 8;
    if (blockIdx.x < xb) {
        const long long npix = (long long)N * p.H2 * p.W2;
        const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
        if (i >= npix * px) return;
        const int pl = (int)(i / npix);
        const long long pix = i - pl * npix;
        const int n = (int)(pix / (p.H2 * p.W2)), r = (int)(pix - (long long)n * p.H2 * p.W2);
        const int h0 = (r / p.W2) * p.st - pad, w0 = (r % p.W2) * p.st - pad;
        const unsigned short* src = reinterpret_cast<const unsigned short*>(x) + pl * x_ps;
        uint32_t o[4] = {0u, 0u, 0u, 0u};
        int e = 0;  // codes gathered so far
        for (int dy = 0; dy < p.st; ++dy)
            for (int dx = 0; dx < p.st; ++dx) {
                const int h = h0 + dy, ww = w0 + dx;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if ((unsigned)h < (unsigned)H && (unsigned)ww < (unsigned)W)
                    v = __ldg(reinterpret_cast<const uint4*>(src + (((long long)n * H + h) * W + ww) * 8));
                const uint32_t q[4] = {v.x, v.y, v.z, v.w};
                for (int c = 0; c < p.C; ++c, ++e) {
                    const uint32_t code = (q[c >> 1] >> (16 * (c & 1))) & 0xFFFFu;
                    const int s = e & 7;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k == (s >> 1)) o[k] |= code << (16 * (s & 1));
                    if (s == 7) {
                        x2[i * c8 + (e >> 3)] = make_uint4(o[0], o[1], o[2], o[3]);
                        o[0] = o[1] = o[2] = o[3] = 0u;
                    }
                }
            }
        if (e & 7) x2[i * c8 + (e >> 3)] = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
        const long long n8 = (long long)K * p.R2 * p.S2 * c8;
        const long long i = (long long)(blockIdx.x - xb) * 256 + threadIdx.x;
        if (i >= n8 * pw) return;
        const int pl = (int)(i / n8);
        const long long j = i - pl * n8;
        const int g = (int)(j % c8);
        const int s2 = (int)((j / c8) % p.S2), r2 = (int)((j / ((long long)c8 * p.S2)) % p.R2);
        const int k = (int)(j / ((long long)c8 * p.S2 * p.R2));
        uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int e = 8 * g + t, c = e % p.C, d = e / p.C;
            const int r = r2 * p.st + d / p.st, s = s2 * p.st + d % p.st;
            if (d < p.st * p.st && r < R && s < S) {
                const uint32_t v = __half_as_ushort(w[pl * w_ps + (((long long)k * R + r) * S + s) * 8 + c]);
                o[t >> 1] |= v << (16 * (t & 1));
            }
        }
        w2[i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

template <typename ACC>
__global__ void splitk_reduce_kernel(const ConvArgs a, const ACC* __restrict__ part, int ks) {
    pdl_wait();
    const long long total = a.M * a.K;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        long long v = 0;
        for (int s = 0; s < ks; ++s) v += (long long)part[s * total + i];
        cblock_epilogue_store(a, i / a.K, (int)(i % a.K), v);
    }
}

}  // namespace

fxpq_status launch_splitk_reduce(const ConvArgs& a, const void* part, int ks, bool acc64, cudaStream_t st) {
    const long long total = a.M * a.K;
    long long blocks = (total + 255) / 256;
    if (blocks > 152LL * 8) blocks = 152LL * 8;
    if (blocks < 1) blocks = 1;
    if (acc64)
        launch_pdl(splitk_reduce_kernel<long long>, (unsigned)blocks, 256, 0, st, a, static_cast<const long long*>(part), ks);
    else
        launch_pdl(splitk_reduce_kernel<int>, (unsigned)blocks, 256, 0, st, a, static_cast<const int*>(part), ks);
    return after_launch("splitk_reduce");
}

// At most 16 shares of int64 sums, for layers whose M x K outputs are small enough for the split to pay
// (it is taken only when the tiles cannot occupy the SMs); capped at 64 MiB.
size_t conv_split_ws_bytes(long long M, int K) {
    const size_t one = (size_t)M * (size_t)K * sizeof(long long);
    const size_t cap = (size_t)64 << 20;
    if (M <= 0 || K <= 0 || 2 * one > cap) return 0;
    return 16 * one < cap ? 16 * one : cap;
}

S2dPlan s2d_plan(const fxpq_conv_desc& d) {
    S2dPlan p = {};
    if (d.Cp != 8 || d.stride < 2 || d.stride > 4 || d.R < d.stride || d.S < d.stride || d.C < 1 || d.C > 8 || d.N < 1 ||
        d.pad < 0 || d.K < 1)
        return p;
    const long long P = ((long long)d.H + 2 * d.pad - d.R) / d.stride + 1, Q = ((long long)d.W + 2 * d.pad - d.S) / d.stride + 1;
    if (d.H + 2 * d.pad < d.R || d.W + 2 * d.pad < d.S || P > (1 << 24) || Q > (1 << 24)) return p;
    p.st = d.stride;
    p.C = d.C;
    p.R2 = (d.R + d.stride - 1) / d.stride;
    p.S2 = (d.S + d.stride - 1) / d.stride;
    p.C2 = (d.stride * d.stride * d.C + 7) / 8 * 8;
    p.H2 = (int)P + p.R2 - 1;
    p.W2 = (int)Q + p.S2 - 1;
    p.flat = (p.S2 * p.C2 + 63) / 64 < p.S2 * ((p.C2 + 63) / 64);
    p.kb = p.flat ? p.R2 * ((p.S2 * p.C2 + 63) / 64) : p.R2 * p.S2 * ((p.C2 + 63) / 64);
    p.kb_own = (d.R * d.S * 8 + 63) / 64;
    p.x_bytes = ((size_t)d.N * p.H2 * p.W2 * p.C2 * 2 * planes_of(d.fmt_x) + 255) / 256 * 256;
    p.w_bytes = ((size_t)d.K * p.R2 * p.S2 * p.C2 * 2 * planes_of(d.fmt_w) + 255) / 256 * 256;
    p.ok = (long long)p.H2 * p.W2 < (1LL << 31) && (long long)d.N * p.H2 * p.W2 * 2 < (1LL << 31) * 128;
    return p;
}

size_t conv_ws_bytes(const fxpq_conv_desc& d) {
    if (d.N < 1 || d.stride < 1 || d.R < 1 || d.S < 1) return 0;
    const int P = (d.H + 2 * d.pad - d.R) / d.stride + 1, Q = (d.W + 2 * d.pad - d.S) / d.stride + 1;
    if (P < 1 || Q < 1) return 0;
    const S2dPlan p = s2d_plan(d);
    return (p.ok ? p.x_bytes + p.w_bytes : 0) + conv_split_ws_bytes((long long)d.N * P * Q, d.K);
}

// Host-side planning shared by conv and gemm: fills ConvArgs, checks the integer bounds.
fxpq_status plan_conv(const fxpq_conv_desc& d, const void* x, const void* w, const int32_t* bias, void* y,
                      ConvArgs& a, int32_t* out_scale, bool& need64) {
    if (d.N < 0 || d.H < 1 || d.W < 1 || d.C < 1 || d.Cp < d.C || (d.Cp % 8) || d.K < 1 || d.R < 1 || d.S < 1 ||
        d.stride < 1 || d.pad < 0)
        return FXPQ_ERR_INVALID_ARG;
    if (!fmt_ok(d.fmt_x) || !fmt_ok(d.fmt_w)) return FXPQ_ERR_INVALID_ARG;
    if (bias && !fmt_ok(d.fmt_b, 32)) return FXPQ_ERR_INVALID_ARG;
    if (d.out_mode < FXPQ_OUT_CODES || d.out_mode > FXPQ_OUT_F32) return FXPQ_ERR_INVALID_ARG;
    if (d.out_mode == FXPQ_OUT_CODES && (!fmt_ok(d.fmt_y) || (d.K % 8))) return FXPQ_ERR_INVALID_ARG;
    const int P = (d.H + 2 * d.pad - d.R) / d.stride + 1, Q = (d.W + 2 * d.pad - d.S) / d.stride + 1;
    if (P < 1 || Q < 1) return FXPQ_ERR_INVALID_ARG;
    if (d.N > 0 && (!x || !w || !y)) return FXPQ_ERR_INVALID_ARG;
    if (!aligned(x, 16) || !aligned(w, 16) || !aligned(y, 16)) return FXPQ_ERR_INVALID_ARG;
    // |acc| <= max|x code| * max|w code| * R*S*C
    const double ax = ldexp(1.0, d.fmt_x.bits - d.fmt_x.is_signed), aw = ldexp(1.0, d.fmt_w.bits - d.fmt_w.is_signed);
    double bound = ax * aw * (double)d.R * d.S * d.C;
    // with a weight-code L1 bound: |acc| <= max|x code| * max_o sum |w code|
    if (d.w_l1 > 0 && d.fmt_w.bits <= 8 && ax * (double)d.w_l1 < bound) bound = ax * (double)d.w_l1;
    if (d.w_l1 < 0) return FXPQ_ERR_INVALID_ARG;
    if (bound >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
    need64 = bound >= ldexp(1.0, 31) - 1.0;
    a.x = static_cast<const __half*>(x);
    a.w = static_cast<const __half*>(w);
    a.bias = bias;
    a.y = y;
    a.N = d.N, a.H = d.H, a.W = d.W, a.Cp = d.Cp, a.K = d.K, a.R = d.R, a.S = d.S;
    a.stride = d.stride, a.pad = d.pad, a.P = P, a.Q = Q;
    a.M = (long long)d.N * P * Q;
    a.x_ps = (long long)d.N * d.H * d.W * d.Cp;
    a.w_ps = (long long)d.K * d.R * d.S * d.Cp;
    a.x_sw = d.Cp, a.x_sh = (long long)d.W * d.Cp, a.x_sn = (long long)d.H * d.W * d.Cp;
    a.px = planes_of(d.fmt_x);
    a.pw = planes_of(d.fmt_w);
    a.relu = d.relu;
    a.out_mode = d.out_mode;
    int s = d.fmt_x.fl + d.fmt_w.fl;
    a.delta = 0;
    double vbound = bound;
    if (bias) {
        a.delta = s - d.fmt_b.fl;
        const double bb = ldexp(1.0, d.fmt_b.bits - d.fmt_b.is_signed);
        if (a.delta >= 0) {
            if (a.delta > 40 || bb * ldexp(1.0, a.delta) + bound >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
            vbound = bound + bb * ldexp(1.0, a.delta);
        } else {
            if (-a.delta > 40 || bound * ldexp(1.0, -a.delta) + bb >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
            vbound = bound * ldexp(1.0, -a.delta) + bb;
            s = d.fmt_b.fl;
        }
    }
    a.has_scale = d.d_scale != nullptr;
    a.scale = d.d_scale;
    a.shift = d.d_shift;
    a.delta2 = 0;
    if (a.has_scale) {
        // v * aleph1 at scale s + fl_aleph1, then aleph2 aligned like the bias
        if (!d.d_shift || !fmt_ok(d.fmt_scale, 32) || !fmt_ok(d.fmt_shift, 32)) return FXPQ_ERR_INVALID_ARG;
        const double mb = ldexp(1.0, d.fmt_scale.bits - d.fmt_scale.is_signed);
        const double hb = ldexp(1.0, d.fmt_shift.bits - d.fmt_shift.is_signed);
        const double pbound = vbound * mb;
        if (pbound >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
        s += d.fmt_scale.fl;
        a.delta2 = s - d.fmt_shift.fl;
        if (a.delta2 >= 0) {
            if (a.delta2 > 40 || hb * ldexp(1.0, a.delta2) + pbound >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
            vbound = pbound + hb * ldexp(1.0, a.delta2);
        } else {
            if (-a.delta2 > 40 || pbound * ldexp(1.0, -a.delta2) + hb >= ldexp(1.0, 62)) return FXPQ_ERR_RANGE;
            vbound = pbound * ldexp(1.0, -a.delta2) + hb;
            s = d.fmt_shift.fl;
        }
    } else if (d.d_shift) {
        return FXPQ_ERR_INVALID_ARG;
    }
    (void)vbound;
    a.s_out = s;
    a.has_bias = bias != nullptr;
    a.v32 = 0;
    a.vf = 0;
    a.vf_c = a.vf_lo = a.vf_hi = 0.0f;
    a.vi = d.out_mode == FXPQ_OUT_F32 && !a.has_scale && (!bias || d.fmt_b.bits <= 24);
    a.vi_c = ldexpf(1.0f, -(d.fmt_x.fl + d.fmt_w.fl));
    a.vi_b = bias ? ldexpf(1.0f, -d.fmt_b.fl) : 0.0f;
    if (d.out_mode == FXPQ_OUT_CODES) {
        a.sh = s - d.fmt_y.fl;
        if (a.sh > 62) return FXPQ_ERR_RANGE;
        a.lo = qmin_of(d.fmt_y);
        a.hi = qmax_of(d.fmt_y);
        a.py = planes_of(d.fmt_y);
        // 32-bit path: N = acc + aligned integer part of the bias, plus the rounding increment
        // 2^(sh32 - 1), stays below 2^31 in magnitude and the FxP-QLayer is a right shift by 1..30 bits
        // of N (see qlayer_code32)
        const double two31 = ldexp(1.0, 31) - 1.0;
        const double bb = bias ? ldexp(1.0, d.fmt_b.bits - d.fmt_b.is_signed) : 0.0;
        const int s_acc = d.fmt_x.fl + d.fmt_w.fl;
        a.bsh = a.delta;
        a.sh32 = s_acc - d.fmt_y.fl;
        const double nbound = bound + (a.delta >= 0 ? bb * ldexp(1.0, a.delta) : bb * ldexp(1.0, a.delta) + 1.0);
        a.v32 = (!a.has_scale && a.sh32 >= 1 && a.sh32 <= 30 && nbound + ldexp(1.0, a.sh32 - 1) < two31 && a.delta >= -30 &&
                 a.delta <= 30)
                    ? 1
                    : 0;
        // fp32 path (fepi_bias): the aligned bias and the sums below 2^23, or every larger sum clipped
        const double b_al = bb * ldexp(1.0, a.delta), top = (double)(a.hi > -a.lo ? a.hi : -a.lo) + 1.0;
        a.vf = !a.has_scale && a.py == 1 && a.sh32 >= 1 && a.sh32 <= 30 && a.delta >= -30 && a.delta <= 30 &&
               b_al <= ldexp(1.0, 22) && (top * ldexp(1.0, a.sh32) <= ldexp(1.0, 23) || bound + b_al + 1.0 <= ldexp(1.0, 23));
        a.vf_c = ldexpf(1.0f, -a.sh32);
        a.vf_lo = a.relu && a.lo < 0 ? 0.0f : (float)a.lo;
        a.vf_hi = (float)a.hi;
    } else {
        a.sh = 0;
        a.lo = a.hi = 0;
        a.py = 1;
    }
    a.f32_scale = ldexpf(1.0f, -s);
    // Scale layers in fp32 (fepi_scale): the factors' codes exact in fp32, every power of two well inside its range
    a.vs = 0;
    a.vs_m = a.vs_b = a.vs_h = a.vs_eps = 0.0f;
    if (a.has_scale && a.py == 1 && d.out_mode != FXPQ_OUT_ACC64 && d.fmt_scale.bits <= 24 && d.fmt_shift.bits <= 24) {
        const int fy = d.out_mode == FXPQ_OUT_CODES ? d.fmt_y.fl : 0;
        const int em = fy - d.fmt_x.fl - d.fmt_w.fl - d.fmt_scale.fl, eb = bias ? fy - d.fmt_b.fl - d.fmt_scale.fl : 0,
                  eh = fy - d.fmt_shift.fl;
        const bool fits = em >= -90 && em <= 30 && eb >= -90 && eb <= 30 && eh >= -90 && eh <= 30;
        const double mb = ldexp(1.0, d.fmt_scale.bits - d.fmt_scale.is_signed);
        const double tb = (bias ? ldexp(1.0, d.fmt_b.bits - d.fmt_b.is_signed) * mb * ldexp(1.0, eb) : 0.0) +
                          ldexp(1.0, d.fmt_shift.bits - d.fmt_shift.is_signed) * ldexp(1.0, eh);
        a.vs_m = ldexpf(1.0f, em);
        a.vs_b = bias ? ldexpf(1.0f, eb) : 0.0f;
        a.vs_h = ldexpf(1.0f, eh);
        if (d.out_mode == FXPQ_OUT_CODES) {
            // half a unit of the last place of x (inside the clip levels, widened by one) and of t, whose three
            // roundings (with a bias) count, with a margin
            const double top = (double)(a.hi > -a.lo ? a.hi : -a.lo) + 2.0;
            const double eps = ldexp(1.0, -24) * (top + (bias ? 3.0 * tb : 0.0)) * 1.25;
            a.vs = fits && a.sh >= 1 && eps < 1.0 / 64 && (!bias || d.fmt_b.bits <= 24);
            a.vs_eps = (float)eps;
            a.vf_lo = a.relu && a.lo < 0 ? 0.0f : (float)a.lo;
            a.vf_hi = (float)a.hi;
        } else {
            a.vs = fits && !bias;  // t is exact: the fused multiply-add rounds the exact value once
        }
    }
    if (out_scale) *out_scale = s;
    return FXPQ_OK;
}

// The layer's arguments in the space-to-depth form.
ConvArgs s2d_args(const ConvArgs& a, const S2dPlan& p, const __half* x2, const __half* w2) {
    ConvArgs b = a;
    b.x = x2;
    b.w = w2;
    b.H = p.H2;
    b.W = p.flat ? a.Q : p.W2;  // flat: one overlapping pixel of S2 C2 channels per output column
    b.Cp = p.flat ? p.S2 * p.C2 : p.C2;
    b.R = p.R2;
    b.S = p.flat ? 1 : p.S2;
    b.stride = 1;
    b.pad = 0;
    b.x_ps = (long long)a.N * p.H2 * p.W2 * p.C2;
    b.w_ps = (long long)a.K * p.R2 * p.S2 * p.C2;
    b.x_sw = p.C2;
    b.x_sh = (long long)p.W2 * p.C2;
    b.x_sn = (long long)p.H2 * p.W2 * p.C2;
    return b;
}

fxpq_conv_desc s2d_desc(const fxpq_conv_desc& d) {
    fxpq_conv_desc e = d;
    e.d_wpacked = nullptr;
    return e;
}

fxpq_status launch_conv(const ConvArgs& a, const fxpq_conv_desc& d, bool need64, cudaStream_t st, void* ws,
                        size_t ws_bytes, const float* images) {
    const long long M = (long long)a.N * a.P * a.Q;
    if (M == 0) return FXPQ_OK;
    auto codes = [&] {  // a.x, where they are not there yet
        return images ? fxpq_quantize_images(images, a.N, d.C, a.H, a.W, d.fmt_x, a.Cp, const_cast<__half*>(a.x), st) : FXPQ_OK;
    };
    // FXPQ_CONV_PATH=tc_rows / tc_nos2d keep strided 8-channel layers on their own codes, simt keeps every layer off
    // the tensor cores
    const char* const path = getenv("FXPQ_CONV_PATH");
    const bool s2d = !(path && (strcmp(path, "tc_rows") == 0 || strcmp(path, "tc_nos2d") == 0));
    if (!(path && strcmp(path, "simt") == 0)) {
        bool launched = false;
        // A strided 8-channel layer runs in the space-to-depth form when the workspace holds it: its taps are
        // then whole runs of a pixel row, where gathered rows cost about 2600 cycles per 8 taps (ResNet conv1,
        // 7 x 7 / 2 of 128 images, 455 -> 216 us with its copy; AlexNet conv1, 11 x 11 / 4 of 256, 431 -> 336)
        const S2dPlan p = s2d_plan(d);
        // Rewriting the input is a launch of its own: worth it where the gathered form's row tiles take more than one
        // round over the SMs (7 x 7 / 2, 98 tiles: 14.0 us rewritten, 11.5 gathered; 196 tiles: 15.0 / 17.3) and, for
        // codes that are there already, where it saves a quarter of at least three k-blocks (300 layers: with 7 x 7 / 2
        // 0.69 times as long on average, 3 x 3 / 2 0.96 to 1.04; 8 channels, 7 x 7 / 4, 185 tiles 24.1 us rewritten,
        // 13.7 gathered); a chosen alternative takes this form at any size
        const bool worth = (M + 127) / 128 * ((a.K + 63) / 64) > num_sms() && (images || (4 * p.kb <= 3 * p.kb_own && p.kb_own >= 3));
        if (p.ok && (worth || path) && ws && ws_bytes >= p.x_bytes + p.w_bytes && s2d) {
            char* base = static_cast<char*>(ws);
            const bool direct = images && launch_quantize_s2d(images, a.N, a.H, a.W, d.fmt_x, p, a.pad, base, st);
            fxpq_status s = direct ? after_launch("quantize_s2d") : codes();
            if (s != FXPQ_OK) return s;
            if (!direct) images = nullptr;
            const long long npix = direct ? 0 : (long long)a.N * p.H2 * p.W2 * a.px, nw = (long long)a.K * p.R2 * p.S2 * (p.C2 / 8) * a.pw;
            const unsigned xb = (unsigned)((npix + 255) / 256), wb = (unsigned)((nw + 255) / 256);
            launch_pdl(s2d_kernel, xb + wb, 256, 0, st, a.x, a.w, a.N, a.H, a.W, a.K, a.R, a.S, a.pad, a.x_ps, a.w_ps, p, a.px, a.pw,
                                                xb, reinterpret_cast<uint4*>(base), reinterpret_cast<uint4*>(base + p.x_bytes));
            s = after_launch("s2d");
            if (s != FXPQ_OK) return s;
            const ConvArgs b = s2d_args(a, p, reinterpret_cast<const __half*>(base),
                                        reinterpret_cast<const __half*>(base + p.x_bytes));
            const size_t used = p.x_bytes + p.w_bytes;
            s = launch_conv_tc(b, s2d_desc(d), st, launched, ws_bytes > used ? base + used : nullptr, ws_bytes - used);
            if (s != FXPQ_OK || launched) return s;
        }
        fxpq_status s = codes();
        if (s != FXPQ_OK) return s;
        images = nullptr;
        s = launch_conv_tc(a, d, st, launched, ws, ws_bytes);
        if (s != FXPQ_OK || launched) return s;
    }
    const fxpq_status s = codes();
    if (s != FXPQ_OK) return s;
    dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)((a.K + TN - 1) / TN));
    if (need64)
        conv_simt_kernel<long long><<<grid, NT, 0, st>>>(a);
    else
        conv_simt_kernel<int><<<grid, NT, 0, st>>>(a);
    return after_launch("conv_simt");
}

fxpq_status conv_fwd(const fxpq_conv_desc& d, const float* images, const void* d_x, const void* d_w, const int32_t* d_bias, void* d_y,
                     int32_t* h_out_scale, void* d_ws, size_t ws_bytes, void* stream) {
    if (d_ws && !aligned(d_ws, 256)) return FXPQ_ERR_WORKSPACE;
    ConvArgs a;
    bool need64 = false;
    fxpq_status st = plan_conv(d, d_x, d_w, d_bias, d_y, a, h_out_scale, need64);
    if (st != FXPQ_OK) return st;
    return launch_conv(a, d, need64, as_stream(stream), d_ws, d_ws ? ws_bytes : 0, images);
}

}  // namespace fxpq

using namespace fxpq;

extern "C" size_t fxpq_conv_workspace(const fxpq_conv_desc* h_desc) {
    return h_desc ? conv_ws_bytes(*h_desc) : 0;
}

extern "C" fxpq_status fxpq_conv_fwd(const fxpq_conv_desc* h_desc, const void* d_x, const void* d_w,
                                     const int32_t* d_bias, void* d_y, int32_t* h_out_scale, void* d_ws,
                                     size_t ws_bytes, void* stream) {
    if (!h_desc) return FXPQ_ERR_INVALID_ARG;
    return conv_fwd(*h_desc, nullptr, d_x, d_w, d_bias, d_y, h_out_scale, d_ws, ws_bytes, stream);
}

extern "C" fxpq_status fxpq_gemm(const void* d_x, fxpq_fmt fmt_x, const void* d_w, fxpq_fmt fmt_w,
                                 const int32_t* d_bias, fxpq_fmt fmt_b, int32_t M, int32_t N, int32_t Kdim,
                                 int32_t relu, int32_t out_mode, fxpq_fmt fmt_y, void* d_y, int32_t* h_out_scale,
                                 void* d_ws, size_t ws_bytes, void* stream) {
    fxpq_conv_desc d = {};
    d.N = M;
    d.H = d.W = 1;
    d.C = Kdim;
    d.Cp = Kdim;
    d.K = N;
    d.R = d.S = 1;
    d.stride = 1;
    d.pad = 0;
    d.relu = relu;
    d.out_mode = out_mode;
    d.fmt_x = fmt_x;
    d.fmt_w = fmt_w;
    d.fmt_b = fmt_b;
    d.fmt_y = fmt_y;
    d.w_l1 = 0;
    return fxpq_conv_fwd(&d, d_x, d_w, d_bias, d_y, h_out_scale, d_ws, ws_bytes, stream);
}
