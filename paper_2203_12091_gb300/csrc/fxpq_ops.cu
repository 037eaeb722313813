// fxpq_ops.cu -- the non-contraction C-Blocks of the integer-only graph (Sec. IV-A.2):
// MAX-POOL (no FxP-QLayer), Eltwise residual add with FL alignment, global AVG-POOL with the
// reciprocal of the patch size quantized like a parameter.  All HBM-bound, one thread per output.
#include <math.h>

#include "fxpq_common.cuh"

namespace fxpq {
namespace {

struct OutArgs {
    int mode;         // FXPQ_OUT_*
    int sh;           // requant shift (CODES)
    long long lo, hi;
    int py;
    float f32_scale;  // 2^-s
};

// y plane stride for CODES output: y_ps elements
__device__ __forceinline__ void store_out(const OutArgs& o, void* y, long long pix, int Cp, int c, long long v,
                                          long long y_ps) {
    if (o.mode == FXPQ_OUT_CODES) {
        long long q;
        if (o.sh > 0) {
            q = rne_shift(v, o.sh);
        } else {
            const int l = -o.sh;
            const long long lim = 1LL << 20;
            if (l >= 32 || v > lim || v < -lim)
                q = v > 0 ? o.hi : (v < 0 ? o.lo : 0);
            else
                q = v << l;
        }
        q = q < o.lo ? o.lo : (q > o.hi ? o.hi : q);
        code_put(static_cast<__half*>(y), pix * Cp + c, o.py, y_ps, (int)q);
    } else if (o.mode == FXPQ_OUT_ACC64) {
        static_cast<long long*>(y)[pix * Cp + c] = v;
    } else {
        static_cast<float*>(y)[pix * Cp + c] = __ll2float_rn(v) * o.f32_scale;
    }
}

__global__ void maxpool_kernel(const __half* __restrict__ x, int N, int H, int W, int Cp, int planes, int k,
                               int stride, int pad, int P, int Q, __half* __restrict__ y) {
    const long long total = (long long)N * P * Q * Cp;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
        const int c = (int)(i % Cp);
        const long long pix = i / Cp;
        const int q = (int)(pix % Q);
        const int p = (int)((pix / Q) % P);
        const long long n = pix / ((long long)P * Q);
        int best = INT_MIN;
        for (int r = 0; r < k; ++r) {
            const int h = p * stride + r - pad;
            if (h < 0 || h >= H) continue;
            for (int s = 0; s < k; ++s) {
                const int w = q * stride + s - pad;
                if (w < 0 || w >= W) continue;
                best = max(best, code_get(x, ((n * H + h) * W + w) * Cp + c, planes, (long long)N * H * W * Cp));
            }
        }
        code_put(y, pix * Cp + c, planes, total, best);
    }
}

__device__ __forceinline__ uint4 max_f16x8(uint4 a, uint4 b) {
    uint4 o;
    const uint32_t x[4] = {a.x, a.y, a.z, a.w}, y[4] = {b.x, b.y, b.z, b.w};
    uint32_t m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 h = __hmax2(*reinterpret_cast<const __half2*>(&x[i]), *reinterpret_cast<const __half2*>(&y[i]));
        m[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    o.x = m[0], o.y = m[1], o.z = m[2], o.w = m[3];
    return o;
}

// One-plane codes: 8 channels per thread with 16-byte loads and stores.  The codes are exact integers in fp16, so the
// half-precision max is exact.  The loads of a K x K / ST window are all in flight, and its place in the image is found
// by 32-bit divisions (64-bit ones and loads one after the other bounded this kernel: 3 x 3 / 2 on 128 images of 112 x
// 112 x 64, 68 -> 48 us, 38 at the rate of a copy; 2 x 2 / 2 on 64 of 224 x 224 x 64, 97 -> 76 us, 76 at that rate; two
// or four outputs per thread, which share a row, 64 us for the first).  K = 0: any window.
template <int K, int ST>
__global__ void __launch_bounds__(256) maxpool_vec8_kernel(const uint4* __restrict__ x, int N, int H, int W, int C8, int k,
                                                           int stride, int pad, int P, int Q, uint4* __restrict__ y) {
    pdl_wait();
    const uint4 ninf = make_uint4(0xFC00FC00u, 0xFC00FC00u, 0xFC00FC00u, 0xFC00FC00u);
    const unsigned i = blockIdx.x * 256u + threadIdx.x, per = (unsigned)P * Q * C8;
    if (i >= per) return;
    const unsigned c8 = i % C8, t = i / C8, q = t % Q, p = t / Q;
    for (int n = blockIdx.y; n < N; n += gridDim.y) {
        const uint4* xi = x + (long long)n * H * W * C8 + c8;
        uint4 m = ninf;
        if constexpr (K > 0) {
            const int h0 = (int)p * ST - pad, w0 = (int)q * ST - pad;
            uint4 in[K * K];
#pragma unroll
            for (int j = 0; j < K * K; ++j) {
                const int h = h0 + j / K, w = w0 + j % K;
                in[j] = (unsigned)h < (unsigned)H && (unsigned)w < (unsigned)W ? __ldg(xi + (long long)(h * W + w) * C8) : ninf;
            }
#pragma unroll
            for (int j = 0; j < K * K; ++j) m = max_f16x8(m, in[j]);
        } else {
            for (int r = 0; r < k; ++r) {
                const int h = (int)p * stride + r - pad;
                if (h < 0 || h >= H) continue;
                for (int c = 0; c < k; ++c) {
                    const int w = (int)q * stride + c - pad;
                    if (w >= 0 && w < W) m = max_f16x8(m, __ldg(xi + ((long long)h * W + w) * C8));
                }
            }
        }
        y[(long long)n * per + i] = m;
    }
}

// The same for many images of few outputs (up to 64 threads each), as many in a block as it holds: 16384 maps of 2 x 2 x 64,
// 2 x 2 / 2, 9.2 us at one image per block, 2.1 so (3.4 with all outputs in one row and 64-bit divisions); at 72 threads
// per image, or for 128 images, one image per block is faster (1.7 / 2.0 and 1.1 / 1.4).
template <int K, int ST>
__global__ void __launch_bounds__(256) maxpool_few_kernel(const uint4* __restrict__ x, int N, int H, int W, int C8, int k,
                                                          int stride, int pad, int P, int Q, uint4* __restrict__ y) {
    pdl_wait();
    const uint4 ninf = make_uint4(0xFC00FC00u, 0xFC00FC00u, 0xFC00FC00u, 0xFC00FC00u);
    const unsigned per = (unsigned)P * Q * C8, imgs = 256u / per, sub = threadIdx.x / per, i = threadIdx.x - sub * per;
    const long long n = (long long)blockIdx.x * imgs + sub;
    if (sub >= imgs || n >= N) return;
    const unsigned c8 = i % C8, t = i / C8;
    const int h0 = (int)(t / Q) * (K ? ST : stride) - pad, w0 = (int)(t % Q) * (K ? ST : stride) - pad;
    const uint4* xi = x + n * H * W * C8 + c8;
    uint4 m = ninf;
    if constexpr (K > 0) {
        uint4 in[K * K];
#pragma unroll
        for (int j = 0; j < K * K; ++j) {
            const int h = h0 + j / K, w = w0 + j % K;
            in[j] = (unsigned)h < (unsigned)H && (unsigned)w < (unsigned)W ? __ldg(xi + (long long)(h * W + w) * C8) : ninf;
        }
#pragma unroll
        for (int j = 0; j < K * K; ++j) m = max_f16x8(m, in[j]);
    } else {
        for (int r = max(-h0, 0); r < min(k, H - h0); ++r)
            for (int c = max(-w0, 0); c < min(k, W - w0); ++c)
                m = max_f16x8(m, __ldg(xi + ((long long)(h0 + r) * W + (w0 + c)) * C8));
    }
    y[n * per + i] = m;
}

__global__ void eltwise_kernel(const __half* __restrict__ a, int pa, int sa, const __half* __restrict__ b, int pb,
                               int sb, long long npix, int Cp, int relu, OutArgs o, void* y) {
    const long long total = npix * Cp;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
        const int c = (int)(i % Cp);
        const long long pix = i / Cp;
        long long v = ((long long)code_get(a, i, pa, total) << sa) + ((long long)code_get(b, i, pb, total) << sb);
        if (relu && v < 0) v = 0;
        store_out(o, y, pix, Cp, c, v, total);
    }
}

// One-plane operands, 8 codes per thread with 16-byte loads and stores, in fp32: with shifts of at most 15
// bits the aligned sum is an integer below 2^24, so a ca + b cb (ca = 2^(sa - sh), cb = 2^(sb - sh)) is the
// exact multiple of 2^-sh that the FxP-QLayer rounds, clipping first (integer levels: the order is
// immaterial), then adding 1.5 2^23 + 0x6600, which rounds half to even and leaves the fp16 pattern of
// 1536 + code in the low half-word.  HBM-bound: 2^24.6 codes (a 56 x 56 x 64 map of 128 images, 154 MB)
// 101 us with one code per thread in 64-bit integers, 27 us.
struct EltVec {
    float ca, cb;    // operand weights
    float lo, hi;    // clip levels (lo: 0 under a ReLU); fp32 and int64 outputs only take the lower one
    float f32_scale;
};

constexpr int ELT_U = 2;  // 8-code pieces per thread and iteration (their loads are issued together)

template <int MODE>
__global__ void __launch_bounds__(256) eltwise_vec8_kernel(const uint4* __restrict__ a, const uint4* __restrict__ b,
                                                           long long n8, EltVec e, void* __restrict__ y) {
    pdl_wait();
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n8; i0 += ELT_U * step) {
        uint4 va[ELT_U], vb[ELT_U];
#pragma unroll
        for (int u = 0; u < ELT_U; ++u) {
            const long long i = i0 + u * step;
            va[u] = i < n8 ? __ldg(a + i) : make_uint4(0, 0, 0, 0);
            vb[u] = i < n8 ? __ldg(b + i) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < ELT_U; ++u) {
            const long long i = i0 + u * step;
            if (i >= n8) break;
            const uint32_t wa[4] = {va[u].x, va[u].y, va[u].z, va[u].w}, wb[4] = {vb[u].x, vb[u].y, vb[u].z, vb[u].w};
            float v[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 fa = __half22float2(*reinterpret_cast<const __half2*>(&wa[q]));
                const float2 fb = __half22float2(*reinterpret_cast<const __half2*>(&wb[q]));
                v[2 * q] = fmaxf(fmaf(fa.x, e.ca, fb.x * e.cb), e.lo);
                v[2 * q + 1] = fmaxf(fmaf(fa.y, e.ca, fb.y * e.cb), e.lo);
            }
            if constexpr (MODE == FXPQ_OUT_CODES) {
                uint32_t w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    w[q] = f32_codes_f16x2(fminf(v[2 * q], e.hi), fminf(v[2 * q + 1], e.hi));
                static_cast<uint4*>(y)[i] = make_uint4(w[0], w[1], w[2], w[3]);
            } else if constexpr (MODE == FXPQ_OUT_F32) {
                float4* o = static_cast<float4*>(y) + 2 * i;
                o[0] = make_float4(v[0] * e.f32_scale, v[1] * e.f32_scale, v[2] * e.f32_scale, v[3] * e.f32_scale);
                o[1] = make_float4(v[4] * e.f32_scale, v[5] * e.f32_scale, v[6] * e.f32_scale, v[7] * e.f32_scale);
            } else {
                longlong2* o = static_cast<longlong2*>(y) + 4 * i;
#pragma unroll
                for (int q = 0; q < 4; ++q) o[q] = make_longlong2(__float2int_rn(v[2 * q]), __float2int_rn(v[2 * q + 1]));
            }
        }
    }
}

// FxP-QLayer on int64 C-Block values (scale 2^-s): codes (fp16 code tensor), int64 copy, or fp32 image.
__global__ void qlayer_kernel(const long long* __restrict__ v, long long n, OutArgs o, void* y) {
    pdl_wait();
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step)
        store_out(o, y, i, 1, 0, v[i], n);
}

__global__ void avgpool_kernel(const __half* __restrict__ x, int N, int HW, int Cp, int planes, long long recip,
                               OutArgs o, void* y) {
    pdl_wait();
    const long long total = (long long)N * Cp;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
        const int c = (int)(i % Cp);
        const long long n = i / Cp;
        long long s = 0;
        for (int t = 0; t < HW; ++t) s += code_get(x, (n * HW + t) * Cp + c, planes, (long long)N * HW * Cp);
        store_out(o, y, n, Cp, c, s * recip, total);
    }
}

int grid_for(long long work) {
    long long b = (work + 255) / 256;
    if (b < 1) b = 1;
    if (b > 152LL * 32) b = 152LL * 32;
    return (int)b;
}

fxpq_status make_out(int mode, const fxpq_fmt& fy, int s, OutArgs& o, int32_t* h_out_scale) {
    if (mode < FXPQ_OUT_CODES || mode > FXPQ_OUT_F32) return FXPQ_ERR_INVALID_ARG;
    o.mode = mode;
    if (mode == FXPQ_OUT_CODES) {
        if (!fmt_ok(fy)) return FXPQ_ERR_INVALID_ARG;
        o.sh = s - fy.fl;
        if (o.sh > 62) return FXPQ_ERR_RANGE;
        o.lo = qmin_of(fy);
        o.hi = qmax_of(fy);
        o.py = planes_of(fy);
    } else {
        o.sh = 0;
        o.lo = o.hi = 0;
        o.py = 1;
    }
    o.f32_scale = ldexpf(1.0f, -s);
    if (h_out_scale) *h_out_scale = s;
    return FXPQ_OK;
}

}  // namespace
}  // namespace fxpq

using namespace fxpq;

extern "C" fxpq_status fxpq_maxpool(const void* d_x, int32_t N, int32_t H, int32_t W, int32_t Cp, fxpq_fmt fmt,
                                    int32_t k, int32_t stride, int32_t pad, void* d_y, void* stream) {
    if (N < 0 || H < 1 || W < 1 || Cp < 1 || (Cp % 8) || k < 1 || stride < 1 || pad < 0 || pad >= k || !fmt_ok(fmt))
        return FXPQ_ERR_INVALID_ARG;
    const int P = (H + 2 * pad - k) / stride + 1, Q = (W + 2 * pad - k) / stride + 1;
    if (P < 1 || Q < 1) return FXPQ_ERR_INVALID_ARG;
    if (N == 0) return FXPQ_OK;
    if (!d_x || !d_y) return FXPQ_ERR_INVALID_ARG;
    const long long total = (long long)N * P * Q * Cp;
    if (planes_of(fmt) == 1 && aligned(d_x, 16) && aligned(d_y, 16)) {
        const bool two = (k == 2 || k == 3) && stride == 2;
        const long long per = (long long)P * Q * (Cp / 8);
        if (per <= 64 && N >= 1024 && (long long)H * W < (1LL << 31)) {
            auto kernel = two ? (k == 3 ? maxpool_few_kernel<3, 2> : maxpool_few_kernel<2, 2>) : maxpool_few_kernel<0, 0>;
            launch_pdl(kernel, (unsigned)((N + 256 / per - 1) / (256 / per)), 256, 0, as_stream(stream), static_cast<const uint4*>(d_x),
                       N, H, W, Cp / 8, k, stride, pad, P, Q, static_cast<uint4*>(d_y));
            return after_launch("maxpool_few");
        }
        if (per < (1LL << 31) && (long long)H * W < (1LL << 31)) {
            auto kernel = two ? (k == 3 ? maxpool_vec8_kernel<3, 2> : maxpool_vec8_kernel<2, 2>) : maxpool_vec8_kernel<0, 0>;
            launch_pdl(kernel, dim3((unsigned)((per + 255) / 256), (unsigned)(N < 65535 ? N : 65535)), 256, 0, as_stream(stream),
                       static_cast<const uint4*>(d_x), N, H, W, Cp / 8, k, stride, pad, P, Q, static_cast<uint4*>(d_y));
            return after_launch("maxpool_vec8");
        }
    }
    maxpool_kernel<<<grid_for(total), 256, 0, as_stream(stream)>>>(static_cast<const __half*>(d_x), N, H, W, Cp,
                                                                   planes_of(fmt), k, stride, pad, P, Q,
                                                                   static_cast<__half*>(d_y));
    return after_launch("maxpool");
}

extern "C" fxpq_status fxpq_eltwise(const void* d_a, fxpq_fmt fmt_a, const void* d_b, fxpq_fmt fmt_b, int64_t n_pix,
                                    int32_t Cp, int32_t relu, int32_t out_mode, fxpq_fmt fmt_y, void* d_y,
                                    int32_t* h_out_scale, void* stream) {
    if (n_pix < 0 || Cp < 1 || (Cp % 8) || !fmt_ok(fmt_a) || !fmt_ok(fmt_b)) return FXPQ_ERR_INVALID_ARG;
    const int fl = fmt_a.fl > fmt_b.fl ? fmt_a.fl : fmt_b.fl;
    const int sa = fl - fmt_a.fl, sb = fl - fmt_b.fl;
    if (sa > 40 || sb > 40) return FXPQ_ERR_RANGE;
    OutArgs o;
    fxpq_status st = make_out(out_mode, fmt_y, fl, o, h_out_scale);
    if (st != FXPQ_OK) return st;
    if (n_pix == 0) return FXPQ_OK;
    if (!d_a || !d_b || !d_y) return FXPQ_ERR_INVALID_ARG;
    // 16-byte pieces of one-plane codes, sums below 2^24 (the scalar kernel: two planes, coarser alignments)
    if (planes_of(fmt_a) == 1 && planes_of(fmt_b) == 1 && o.py == 1 && sa <= 15 && sb <= 15 && aligned(d_a, 16) &&
        aligned(d_b, 16) && aligned(d_y, 16)) {
        const int sh = out_mode == FXPQ_OUT_CODES ? o.sh : 0;
        const float inf = INFINITY;
        EltVec e{ldexpf(1.0f, sa - sh), ldexpf(1.0f, sb - sh), relu ? 0.0f : -inf, inf, o.f32_scale};
        if (out_mode == FXPQ_OUT_CODES) {
            e.lo = relu && o.lo < 0 ? 0.0f : (float)o.lo;
            e.hi = (float)o.hi;
        }
        const long long n8 = n_pix * Cp / 8;
        const int grid = grid_for((n8 + ELT_U - 1) / ELT_U);
        const uint4 *a = static_cast<const uint4*>(d_a), *b = static_cast<const uint4*>(d_b);
        if (out_mode == FXPQ_OUT_CODES)
            launch_pdl(eltwise_vec8_kernel<FXPQ_OUT_CODES>, grid, 256, 0, as_stream(stream), a, b, n8, e, d_y);
        else if (out_mode == FXPQ_OUT_F32)
            launch_pdl(eltwise_vec8_kernel<FXPQ_OUT_F32>, grid, 256, 0, as_stream(stream), a, b, n8, e, d_y);
        else
            launch_pdl(eltwise_vec8_kernel<FXPQ_OUT_ACC64>, grid, 256, 0, as_stream(stream), a, b, n8, e, d_y);
        return after_launch("eltwise_vec8");
    }
    eltwise_kernel<<<grid_for(n_pix * Cp), 256, 0, as_stream(stream)>>>(
        static_cast<const __half*>(d_a), planes_of(fmt_a), sa, static_cast<const __half*>(d_b), planes_of(fmt_b), sb,
        n_pix, Cp, relu, o, d_y);
    return after_launch("eltwise");
}

extern "C" fxpq_status fxpq_avgpool(const void* d_x, int32_t N, int32_t H, int32_t W, int32_t Cp, fxpq_fmt fmt_x,
                                    int32_t recip_code, fxpq_fmt fmt_recip, int32_t out_mode, fxpq_fmt fmt_y,
                                    void* d_y, int32_t* h_out_scale, void* stream) {
    if (N < 0 || H < 1 || W < 1 || Cp < 1 || (Cp % 8) || !fmt_ok(fmt_x) || !fmt_ok(fmt_recip))
        return FXPQ_ERR_INVALID_ARG;
    if (recip_code < qmin_of(fmt_recip) || recip_code > qmax_of(fmt_recip)) return FXPQ_ERR_INVALID_ARG;
    OutArgs o;
    fxpq_status st = make_out(out_mode, fmt_y, fmt_x.fl + fmt_recip.fl, o, h_out_scale);
    if (st != FXPQ_OK) return st;
    if (N == 0) return FXPQ_OK;
    if (!d_x || !d_y) return FXPQ_ERR_INVALID_ARG;
    launch_pdl(avgpool_kernel, grid_for((long long)N * Cp), 256, 0, as_stream(stream),
        static_cast<const __half*>(d_x), N, H * W, Cp, planes_of(fmt_x), (long long)recip_code, o, d_y);
    return after_launch("avgpool");
}

extern "C" fxpq_status fxpq_qlayer(const int64_t* d_v, int64_t n, int32_t s, int32_t out_mode, fxpq_fmt fmt_y,
                                   void* d_y, void* stream) {
    if (n < 0 || s < -64 || s > 80) return FXPQ_ERR_INVALID_ARG;
    OutArgs o;
    const fxpq_status st = make_out(out_mode, fmt_y, s, o, nullptr);
    if (st != FXPQ_OK) return st;
    if (n == 0) return FXPQ_OK;
    if (!d_v || !d_y) return FXPQ_ERR_INVALID_ARG;
    launch_pdl(qlayer_kernel, grid_for(n), 256, 0, as_stream(stream), reinterpret_cast<const long long*>(d_v), n, o, d_y);
    return after_launch("qlayer");
}

// ---------------------------------------------------------------- BN -> Scale (Sec. IV-A.1)
namespace fxpq {
namespace {

// aleph1 = gamma / r and aleph2 = beta - (gamma * mean) / r with r = sqrt(var + eps), every step one
// correctly rounded fp32 operation (the _rn intrinsics are IEEE round-to-nearest-even, so the
// result does not depend on contraction into fused multiply-adds).
__global__ void bn_to_scale_kernel(const float* __restrict__ g, const float* __restrict__ b,
                                   const float* __restrict__ mu, const float* __restrict__ var, long long n, float eps,
                                   float* __restrict__ a1, float* __restrict__ a2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float r = __fsqrt_rn(__fadd_rn(var[i], eps));
    a1[i] = __fdiv_rn(g[i], r);
    a2[i] = __fsub_rn(b[i], __fdiv_rn(__fmul_rn(g[i], mu[i]), r));
}

}  // namespace
}  // namespace fxpq

extern "C" fxpq_status fxpq_bn_to_scale(const float* d_gamma, const float* d_beta, const float* d_mean,
                                        const float* d_var, int64_t n, float eps, float* d_aleph1, float* d_aleph2,
                                        void* stream) {
    using namespace fxpq;
    if (n < 0 || !(eps >= 0.0f)) return FXPQ_ERR_INVALID_ARG;
    if (n == 0) return FXPQ_OK;
    if (!d_gamma || !d_beta || !d_mean || !d_var || !d_aleph1 || !d_aleph2) return FXPQ_ERR_INVALID_ARG;
    const int T = 256;
    bn_to_scale_kernel<<<(unsigned)((n + T - 1) / T), T, 0, as_stream(stream)>>>(d_gamma, d_beta, d_mean, d_var, n,
                                                                                 eps, d_aleph1, d_aleph2);
    return after_launch("bn_to_scale");
}
