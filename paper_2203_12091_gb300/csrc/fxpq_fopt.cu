// fxpq_fopt.cu -- the forward optimizer's FP32 side (Sec. IV-C, Alg. 1 and its cost F): while one
// data-structure's QPs are searched, every later layer runs in FP32, and the cost needs each
// data-structure's quantization error, range and dispersion and the logits' top-1 ties.
//   conv / max-pool / eltwise / global avg-pool in fp32 (NHWC, true channel counts);
//   code tensors -> fp32 values; fp32 bias + ReLU after an integer contraction;
//   per-data-structure statistics (L of Eq. DSB_QE at one format, min, max, per-sample moments);
//   top-1 tie counts of logits (fp32 or exact int64).
#include <math.h>

#include "fxpq_common.cuh"

namespace fxpq {
namespace {

// ------------------------------------------------------------------ fp32 implicit-GEMM convolution
// x: [N, H, W, C]; w: [K, R*S*C] (KRSC); y: [N, P, Q, K].  Bound by the fp32 FMA rate (128 per cycle and SM).
// A block of 256 threads computes BM output pixels x 64 channels as four groups of 64 threads: every stage of
// 32 reduction steps is split into four slices of 8, one per group, and each thread accumulates (BM / 8) x 8
// outputs over its group's slices, so that small tiles (which occupy the SMs at a few calibration images)
// still read only 4 16-byte pieces of shared memory per 64 FMAs.  The groups' sums are added pairwise at the
// end.  FMAs are issued packed two pixels at a time (fma.rn.f32x2), which leaves issue slots for the loads.
// 24 images (three candidates of 8), ResNet-18: 56 x 56 x 64 177 -> 137 us, 28 x 28 x 128 283 -> 132, 7 x 7 x 512 488 -> 152
// (128 x 64 and 64 x 64 tiles with one accumulator chain before).
constexpr int CF_BN = 64, CF_BK = 32, CF_TAB = 1024;

struct ConvF32Args {
    const float* x;
    const float* w;
    const float* bias;
    float* y;
    int N, H, W, C, K, R, S, stride, pad, P, Q, relu;
    long long M;
    int n_first;  // first output channel of the launch
};

__device__ __forceinline__ unsigned long long f2_pack(float x, float y) {
    unsigned long long v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long v) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}

// VEC: C % 4 == 0 (a float4 of a row stays inside one tap) and 16-byte aligned x and w; otherwise single loads,
// the reduction index decoded through a table in shared memory (up to CF_TAB steps, whose tap rows and columns are below
// CF_TAB too and share a word).  Off: the type of an offset within a window, 64-bit where that spans 2^31 elements (a few
// taps of long rows).
template <int BM, bool VEC, typename Off = int>
__global__ void __launch_bounds__(256, 2) conv_f32_kernel(const ConvF32Args a) {
    pdl_wait();
    constexpr int MT = BM / 8;           // output pixels per thread
    constexpr int AV = BM * CF_BK / 4 / 256;  // float4 of the A stage per thread
    constexpr int BV = CF_BN * CF_BK / 4 / 256;
    // stage: [k][m] and [k][n], 16-byte pieces of row k at piece ^ (k / 4 % 8): the transposing stores of eight
    // lanes with consecutive k / 4 then fall into different banks, and pieces stay whole for the loads
    __shared__ __align__(16) float sa[2][CF_BK][BM];
    __shared__ __align__(16) float sb[2][CF_BK][CF_BN];
    __shared__ Off tab_off[VEC ? 1 : CF_TAB];
    __shared__ int tab_rs[VEC ? 1 : CF_TAB];
    static_assert(CF_TAB <= 32768, "a tap's row and column share a word");
    const int tid = threadIdx.x, grp = tid >> 6, t64 = tid & 63;
    const int tx = t64 & 7, ty = t64 >> 3;
    const long long m0 = (long long)blockIdx.x * BM;
    const int n0 = a.n_first + (int)blockIdx.y * CF_BN;
    const int RSC = a.R * a.S * a.C;
    if (!VEC) {
        for (int k = tid; k < RSC && k < CF_TAB; k += 256) {
            const int c = k % a.C, rs = k / a.C, s = rs % a.S, r = rs / a.S;
            tab_off[k] = ((Off)r * a.W + s) * a.C + c;
            tab_rs[k] = (r << 16) | s;
        }
        __syncthreads();
    }
    // loads: thread t takes k quad t % 8 of rows t / 8, t / 8 + 32, ..
    const int kq = tid & 7, lr = tid >> 3;
    int p0[AV], q0[AV];
    long long xo[AV];
#pragma unroll
    for (int i = 0; i < AV; ++i) {
        const long long m = m0 + lr + 32 * i;
        p0[i] = -(1 << 30);  // rows past the end read zeros
        q0[i] = 0;
        xo[i] = 0;
        if (m < a.M) {
            const long long n = m / ((long long)a.P * a.Q);
            const int rem = (int)(m - n * a.P * a.Q), pp = rem / a.Q, pq = rem - pp * a.Q;
            p0[i] = pp * a.stride - a.pad;
            q0[i] = pq * a.stride - a.pad;
            xo[i] = ((n * a.H + p0[i]) * a.W + q0[i]) * a.C;
        }
    }
    float4 ra[AV], rb[BV];
    // the tap of this thread's k quad, stepped with the stages
    int kc = VEC ? (4 * kq) % a.C : 0, ks = VEC ? (4 * kq) / a.C % a.S : 0, kr = VEC ? (4 * kq) / a.C / a.S : 0;
    auto load = [&](int k0) {
        const int k = k0 + 4 * kq;
        if (VEC) {
            const long long to = ((long long)kr * a.W + ks) * a.C + kc;
#pragma unroll
            for (int i = 0; i < AV; ++i) {
                const int h = p0[i] + kr, w = q0[i] + ks;
                const bool in = k < RSC && (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
                ra[i] = in ? __ldg(reinterpret_cast<const float4*>(a.x + xo[i] + to)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int i = 0; i < BV; ++i) {
                const int o = n0 + lr + 32 * i;
                rb[i] = k < RSC && o < a.K ? __ldg(reinterpret_cast<const float4*>(a.w + (long long)o * RSC + k))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            kc += CF_BK;
            while (kc >= a.C) {
                kc -= a.C;
                if (++ks == a.S) {
                    ks = 0;
                    ++kr;
                }
            }
        } else {
            float va[AV][4], vb[BV][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int kk = k + e;
                int r = 0, s = 0;
                Off off = 0;
                if (kk < CF_TAB && kk < RSC) {
                    off = tab_off[kk];
                    r = tab_rs[kk] >> 16;
                    s = tab_rs[kk] & 0xFFFF;
                } else if (kk < RSC) {
                    const int c = kk % a.C, rs = kk / a.C;
                    s = rs % a.S;
                    r = rs / a.S;
                    off = ((Off)r * a.W + s) * a.C + c;
                }
#pragma unroll
                for (int i = 0; i < AV; ++i) {
                    const int h = p0[i] + r, w = q0[i] + s;
                    const bool in = kk < RSC && (unsigned)h < (unsigned)a.H && (unsigned)w < (unsigned)a.W;
                    va[i][e] = in ? __ldg(a.x + xo[i] + off) : 0.0f;
                }
#pragma unroll
                for (int i = 0; i < BV; ++i) {
                    const int o = n0 + lr + 32 * i;
                    vb[i][e] = kk < RSC && o < a.K ? __ldg(a.w + (long long)o * RSC + kk) : 0.0f;
                }
            }
#pragma unroll
            for (int i = 0; i < AV; ++i) ra[i] = make_float4(va[i][0], va[i][1], va[i][2], va[i][3]);
#pragma unroll
            for (int i = 0; i < BV; ++i) rb[i] = make_float4(vb[i][0], vb[i][1], vb[i][2], vb[i][3]);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int i = 0; i < AV; ++i) {
            const int m = (lr + 32 * i) ^ (kq << 2);
            sa[buf][4 * kq][m] = ra[i].x;
            sa[buf][4 * kq + 1][m] = ra[i].y;
            sa[buf][4 * kq + 2][m] = ra[i].z;
            sa[buf][4 * kq + 3][m] = ra[i].w;
        }
#pragma unroll
        for (int i = 0; i < BV; ++i) {
            const int n = (lr + 32 * i) ^ (kq << 2);
            sb[buf][4 * kq][n] = rb[i].x;
            sb[buf][4 * kq + 1][n] = rb[i].y;
            sb[buf][4 * kq + 2][n] = rb[i].z;
            sb[buf][4 * kq + 3][n] = rb[i].w;
        }
    };
    // pixels 4 ty .. + 3 (and BM / 2 + the same for BM = 64), channels 4 tx .. + 3 and 32 + the same
    unsigned long long acc[MT / 2][8];
#pragma unroll
    for (int i = 0; i < MT / 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < RSC; k0 += CF_BK) {
        const bool more = k0 + CF_BK < RSC;
        if (more) load(k0 + CF_BK);  // next stage's global loads in flight during this stage's FMAs
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            const int k = 8 * grp + kk, x = (2 * grp + (kk >> 2)) & 7;  // k / 4 % 8
            unsigned long long av[MT / 2];
#pragma unroll
            for (int i = 0; i < MT / 4; ++i) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&sa[buf][k][((ty ^ x) << 2) + 32 * i]);
                av[2 * i] = v.x;
                av[2 * i + 1] = v.y;
            }
            float bv[8];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float4 v = *reinterpret_cast<const float4*>(&sb[buf][k][((tx ^ x) << 2) + 32 * j]);
                bv[4 * j] = v.x, bv[4 * j + 1] = v.y, bv[4 * j + 2] = v.z, bv[4 * j + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned long long b2 = f2_pack(bv[j], bv[j]);
#pragma unroll
                for (int i = 0; i < MT / 2; ++i) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(av[i]), "l"(b2));
            }
        }
        if (more) {
            store(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
    // groups 2, 3 onto 0, 1, then 1 onto 0, through the A stage (a group's sums are BM x 64 floats as 16-byte
    // pieces [piece][thread])
    __syncthreads();
    ulonglong2* red = reinterpret_cast<ulonglong2*>(&sa[0][0][0]);
    constexpr int NP = MT * 8 / 4;  // 16-byte pieces per thread
    static_assert(NP * 64 * 16 <= (int)sizeof(sa) && BM <= 64, "one group's sums fit the A stage");
#pragma unroll
    for (int rnd = 0; rnd < 3; ++rnd) {
        const int src = rnd == 0 ? 3 : rnd == 1 ? 2 : 1, dst = rnd == 0 ? 1 : 0;
        if (grp == src)
#pragma unroll
            for (int q = 0; q < NP; ++q) red[q * 64 + t64] = make_ulonglong2(acc[q / 4][2 * (q % 4)], acc[q / 4][2 * (q % 4) + 1]);
        __syncthreads();
        if (grp == dst)
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                const ulonglong2 v = red[q * 64 + t64];
                asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[q / 4][2 * (q % 4)]) : "l"(v.x));
                asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc[q / 4][2 * (q % 4) + 1]) : "l"(v.y));
            }
        __syncthreads();
    }
    if (grp != 0) return;
    const bool v4 = a.K % 4 == 0 && (reinterpret_cast<uintptr_t>(a.y) & 15) == 0;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        const long long mm = m0 + 4 * ty + (i & 3) + (i >> 2) * 32;
        if (mm >= a.M) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float o[4];
            const int oo = n0 + 4 * tx + 32 * h;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 f = f2_unpack(acc[i >> 1][4 * h + j]);
                o[j] = (i & 1) ? f.y : f.x;
                if (a.bias && oo + j < a.K) o[j] += __ldg(a.bias + oo + j);
                if (a.relu) o[j] = fmaxf(o[j], 0.0f);
            }
            if (v4 && oo < a.K)
                *reinterpret_cast<float4*>(a.y + mm * a.K + oo) = make_float4(o[0], o[1], o[2], o[3]);
            else
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (oo + j < a.K) a.y[mm * a.K + oo + j] = o[j];
        }
    }
}

__global__ void maxpool_f32_kernel(const float* __restrict__ x, int N, int H, int W, int C, int k, int stride, int pad,
                                   int P, int Q, float* __restrict__ y) {
    pdl_wait();
    const long long total = (long long)N * P * Q * C;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long pix = i / C;
        const int q = (int)(pix % Q), p = (int)((pix / Q) % P);
        const long long n = pix / ((long long)P * Q);
        float best = -INFINITY;
        for (int r = 0; r < k; ++r) {
            const int h = p * stride + r - pad;
            if (h < 0 || h >= H) continue;
            for (int s = 0; s < k; ++s) {
                const int w = q * stride + s - pad;
                if (w >= 0 && w < W) best = fmaxf(best, x[((n * H + h) * W + w) * C + c]);
            }
        }
        y[i] = best;
    }
}

__global__ void eltwise_f32_kernel(const float* __restrict__ a, const float* __restrict__ b, long long n, int relu,
                                   float* __restrict__ y) {
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float v = a[i] + b[i];
        y[i] = relu ? fmaxf(v, 0.0f) : v;
    }
}

// one thread per (n, c): the mean over H x W (sum in fp32, then divided by H W)
__global__ void avgpool_f32_kernel(const float* __restrict__ x, int N, int HW, int C, float* __restrict__ y) {
    pdl_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)N * C) return;
    const long long n = i / C;
    const int c = (int)(i % C);
    float s = 0.0f;
    for (int p = 0; p < HW; ++p) s += x[(n * HW + p) * C + c];
    y[i] = s / (float)HW;
}

// fp16 code tensor [npix, Cp] (planes) -> fp32 values [npix, C]; the binary quantizer's codes decode
// 0 -> +1, -1 -> -1
__global__ void dequantize_kernel(const __half* __restrict__ codes, long long npix, int Cp, int C, int planes, float scale,
                                  int binary, float* __restrict__ y) {
    pdl_wait();
    const long long total = npix * C;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long pix = i / C;
        const int c = (int)(i - pix * C);
        int code = code_get(codes, pix * Cp + c, planes, npix * Cp);
        if (binary) code = 2 * code + 1;
        y[i] = (float)code * scale;  // exact: |code| < 2^17 and scale a power of two
    }
}

__global__ void bias_relu_f32_kernel(float* __restrict__ y, long long npix, int K, const float* __restrict__ bias,
                                     int relu) {
    const long long total = npix * K;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        float v = y[i];
        if (bias) v += bias[i % K];
        y[i] = relu ? fmaxf(v, 0.0f) : v;
    }
}

__device__ __forceinline__ unsigned ord_key(float x) {
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// ---------------------------------------------------------------- data-structure statistics (batched)
// Items of fxpq_ds_stats_batch, split into work units of DS_CHUNK values of one sample each; the unit
// prefix of each item sits in the kernel parameters.  Three passes: per-unit sums; per-unit sums of
// squared deviations from the sample mean (the mean from the first pass's sums, in unit order), the
// quantization error and the extremes; per-item records from the units in order.  No floating-point
// atomics: every total is formed in a fixed order.
constexpr int DS_MAX_ITEMS = 128;  // items per launch group
constexpr long long DS_CHUNK = 1 << 16;
constexpr int DS_T = 256;

struct DsItemDev {
    const float* x;
    double* out;
    long long nu;
    int n_samples, k, S, fl;
    int chunks;  // units per sample
    int unit0;   // first unit of the item (within its launch group)
};
struct DsBatchDev {
    int n;
    DsItemDev it[DS_MAX_ITEMS];
    int unit_end;  // units of the launch group
};

// Per-unit scratch of one launch group.
struct DsUnit {
    double sum, m2, l2;
    unsigned mn, mx;
};

__device__ __forceinline__ int ds_item_of(const DsBatchDev& B, int u) {
    int lo = 0, hi = B.n - 1;  // last item whose unit0 <= u
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.it[mid].unit0 <= u) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ double ds_block_sum(double v, double* red) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < DS_T / 32; ++i) t += red[i];  // fixed order
    return t;  // valid in thread 0
}

// The sums of these kernels run in triples of fp32: every addition's rounding error is carried into the next
// word (TwoSum), so that a thread's chain keeps about 70 bits, and it meets fp64 once, at the end.  fp64
// arithmetic has 1/64 of the fp32 rate here (two operations per cycle and SM): the twelve operations per
// element of the direct fp64 form were these kernels' time (95 M values of three ResNet-18 candidates: sums
// 555 -> 132 us, deviations 2950 -> 608 us), and its rounding per addition was the larger one.
constexpr int DS_U = 8;  // values per thread and step (their loads are issued together)

__device__ __forceinline__ float two_sum(float a, float b, float& err) {
    const float t = a + b, z = t - a, r = (a - (t - z)) + (b - z);
    err = r;
    return t;
}
struct Sum3 {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    __device__ __forceinline__ void low(float v) {  // v well below the terms of add
        float e;
        b = two_sum(b, v, e);
        c += e;
    }
    __device__ __forceinline__ void add(float v) {
        float e;
        a = two_sum(a, v, e);
        low(e);
    }
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

// f(value) for a unit's values, DS_U per thread and step, consecutive threads in consecutive places.
template <typename F>
__device__ __forceinline__ void ds_walk(const float* __restrict__ xs, long long i0, long long i1, F f) {
    for (long long i = i0 + threadIdx.x; i < i1; i += (long long)DS_U * DS_T) {
        float v[DS_U];
#pragma unroll
        for (int j = 0; j < DS_U; ++j) v[j] = i + (long long)j * DS_T < i1 ? __ldg(xs + i + (long long)j * DS_T) : 0.0f;
#pragma unroll
        for (int j = 0; j < DS_U; ++j)
            if (i + (long long)j * DS_T < i1) f(v[j]);
    }
}

__global__ void __launch_bounds__(DS_T) ds_sum_kernel(const __grid_constant__ DsBatchDev B, DsUnit* units) {
    pdl_wait();
    __shared__ double red[DS_T / 32];
    const int u = blockIdx.x;
    const DsItemDev& it = B.it[ds_item_of(B, u)];
    const int rel = u - it.unit0, s = rel / it.chunks, c = rel % it.chunks;
    const float* xs = it.x + (long long)s * it.nu;
    const long long i0 = (long long)c * DS_CHUNK, i1 = min(i0 + DS_CHUNK, it.nu);
    Sum3 acc;
    double big = 0.0;  // steps with a value of 2^100 or more, whose fp32 sums could overflow
    for (long long i = i0 + threadIdx.x; i < i1; i += (long long)DS_U * DS_T) {
        float v[DS_U], top = 0.0f;
#pragma unroll
        for (int j = 0; j < DS_U; ++j) v[j] = i + (long long)j * DS_T < i1 ? __ldg(xs + i + (long long)j * DS_T) : 0.0f;
#pragma unroll
        for (int j = 0; j < DS_U; ++j) top = fmaxf(top, fabsf(v[j]));
        if (top < 0x1p100f) {
#pragma unroll
            for (int j = 0; j < DS_U; ++j) acc.add(v[j]);
        } else {
#pragma unroll
            for (int j = 0; j < DS_U; ++j) big += (double)v[j];
        }
    }
    const double t = ds_block_sum(acc.value() + big, red);
    if (threadIdx.x == 0) units[u].sum = t;
}

__global__ void __launch_bounds__(DS_T) ds_dev_kernel(const __grid_constant__ DsBatchDev B, DsUnit* units) {
    pdl_wait();
    __shared__ double red[DS_T / 32];
    __shared__ unsigned kmn, kmx;
    const int u = blockIdx.x;
    const DsItemDev& it = B.it[ds_item_of(B, u)];
    const int rel = u - it.unit0, s = rel / it.chunks, c = rel % it.chunks;
    const float* xs = it.x + (long long)s * it.nu;
    const long long i0 = (long long)c * DS_CHUNK, i1 = min(i0 + DS_CHUNK, it.nu);
    // the sample mean from the first pass's unit sums, in unit order
    const int first = it.unit0 + s * it.chunks;
    double sum = 0.0;
    for (int v = 0; v < it.chunks; ++v) sum += units[first + v].sum;
    const double mean = sum / (double)it.nu;
    const double scale = ldexp(1.0, it.fl), inv = ldexp(1.0, -it.fl);
    const double lo = it.S ? -ldexp(1.0, it.k - 1) : 0.0, hi = ldexp(1.0, it.k - it.S) - 1.0;
    const bool binary = it.k == 1 && it.S == 1;
    // In units of 2^-fl (y = x 2^fl), for k <= 16: the code q and r = y - q are exact in fp32 when y is zero or
    // 2^-40 <= |y| < 2^24 (a smaller one's square could leave fp32's range), r^2 and y less the mean (mh + ml + mq)
    // are exact as pairs, but for the last bits of the smaller word.  Other values take the fp64 form.
    const float fscale = (float)scale, flo = (float)lo, fhi = (float)hi;
    const double my = mean * scale;
    const float mh = (float)my, ml = (float)(my - (double)mh), mq = (float)(my - (double)mh - (double)ml);
    const bool narrow = it.k <= 16 && !binary && fabs(my) < 16777216.0 && (my == 0.0 || fabs(my) > 0x1p-40);
    double m2 = 0.0, l2 = 0.0;  // the fp64 form's sums, in units of x
    Sum3 m2y, l2y;              // in units of y
    unsigned mn = 0xFFFFFFFFu, mx = 0u;
    ds_walk(xs, i0, i1, [&](float v) {
        const unsigned key = ord_key(v);
        mn = min(mn, key);
        mx = max(mx, key);
        const float y = v * fscale, ay = fabsf(y);
        if (narrow && (v == 0.0f || (ay < 16777216.0f && ay > 0x1p-40f))) {
            const float q = (fminf(fmaxf(y, flo), fhi) + 12582912.0f) - 12582912.0f;
            // (_rn: products are not contracted into the sums)
            const float r = y - q, p = __fmul_rn(r, r);
            l2y.add(p);
            l2y.low(fmaf(r, r, -p));
            // y - mean = d + e + g, each below half a unit of the last place of the one before; its square
            // d^2 + 2 d e + (2 d g + e^2)
            float e, g;
            float d = two_sum(y, -mh, e);
            e = two_sum(e, -ml, g);
            d = two_sum(d, e, e);
            g -= mq;
            const float w = __fmul_rn(d, d), d2 = 2.0f * d, c = __fmul_rn(d2, e);
            m2y.add(w);
            m2y.low(fmaf(d, d, -w));
            m2y.low(c);
            m2y.c += fmaf(d2, e, -c) + fmaf(d2, g, __fmul_rn(e, e));
        } else {
            const double x = (double)v;
            const double q = binary ? (v < 0.0f ? -inv : inv) : fmin(fmax(nearbyint(x * scale), lo), hi) * inv;
            const double e = x - q, dv = x - mean;
            l2 += e * e;
            m2 += dv * dv;
        }
    });
    l2 += l2y.value() * inv * inv;
    m2 += m2y.value() * inv * inv;
    if (threadIdx.x == 0) {
        kmn = 0xFFFFFFFFu;
        kmx = 0u;
    }
    const double tm2 = ds_block_sum(m2, red);
    const double tl2 = ds_block_sum(l2, red);
    mn = __reduce_min_sync(0xFFFFFFFFu, mn);
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&kmn, mn);
        atomicMax(&kmx, mx);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        units[u].m2 = tm2;
        units[u].l2 = tl2;
        units[u].mn = kmn;
        units[u].mx = kmx;
    }
}

__device__ __forceinline__ float ds_key_value(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// One block per item: its record from its units, a thread per sample adding the sample's units in order, then
// thread 0 the threads' shares of L in order.
constexpr int DF_T = 64;
__global__ void __launch_bounds__(DF_T) ds_finish_kernel(const __grid_constant__ DsBatchDev B, const DsUnit* units) {
    pdl_wait();
    __shared__ double l2s[DF_T];
    __shared__ unsigned kmn, kmx;
    const DsItemDev& it = B.it[blockIdx.x];
    if (threadIdx.x == 0) {
        kmn = 0xFFFFFFFFu;
        kmx = 0u;
    }
    __syncthreads();
    double l2 = 0.0;
    unsigned mn = 0xFFFFFFFFu, mx = 0u;
    for (int s = threadIdx.x; s < it.n_samples; s += DF_T) {
        double sum = 0.0, m2 = 0.0;
        for (int c = 0; c < it.chunks; ++c) {
            const DsUnit& q = units[it.unit0 + s * it.chunks + c];
            sum += q.sum;
            m2 += q.m2;
            l2 += q.l2;
            mn = min(mn, q.mn);
            mx = max(mx, q.mx);
        }
        it.out[3 + 2 * s] = sum / (double)it.nu;
        it.out[4 + 2 * s] = m2;
    }
    l2s[threadIdx.x] = l2;
    atomicMin(&kmn, mn);
    atomicMax(&kmx, mx);
    __syncthreads();
    if (threadIdx.x != 0) return;
    double t = 0.0;
    for (int i = 0; i < DF_T && i < it.n_samples; ++i) t += l2s[i];
    it.out[0] = t;
    it.out[1] = (double)ds_key_value(kmn);
    it.out[2] = (double)ds_key_value(kmx);
}

// ---------------------------------------------------------------- the cost F of Alg. 1
constexpr int COST_MAX_TERMS = 512;
struct CostTermDev {
    long long offset, nu;
    int n_samples, layer;
};
struct CostTerms {
    int n;
    CostTermDev t[COST_MAX_TERMS];
};

// One block per candidate: a thread per term forms its sigma nu (square roots and divisions in fp64, one per
// sample, are the kernel's time), then thread 0 adds the terms in order (a few dozen per network).
__global__ void fopt_cost_kernel(const double* __restrict__ stats, long long cand_stride,
                                 const __grid_constant__ CostTerms T, const int* __restrict__ ties, int N,
                                 int n_classes, double* __restrict__ cost) {
    pdl_wait();
    const int c = blockIdx.x;
    const double* base = stats + (long long)c * cand_stride;
    __shared__ unsigned n_tied, extra;
    __shared__ double snu[COST_MAX_TERMS];  // the terms' sigma nu
    __shared__ double lr[COST_MAX_TERMS];   // and L / R (0 where R = 0)
    if (threadIdx.x == 0) n_tied = extra = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int k = ties[(long long)c * N + i];
        if (k > 1) atomicAdd(&n_tied, 1u);
        atomicAdd(&extra, (unsigned)(k - 1));
    }
    for (int t = threadIdx.x; t < T.n; t += blockDim.x) {
        const CostTermDev& q = T.t[t];
        const double* r = base + q.offset;
        double sig = 0.0;
        for (int s = 0; s < q.n_samples; ++s) sig += sqrt(r[4 + 2 * s] / (double)q.nu);
        snu[t] = sig / q.n_samples * (double)q.nu;
        const double R = r[2] - r[1];
        lr[t] = R == 0.0 ? 0.0 : r[0] / R;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double E = 0.0;
    int t0 = 0;
    while (t0 < T.n) {
        int t1 = t0;
        double den = 0.0, sum = 0.0;
        while (t1 < T.n && T.t[t1].layer == T.t[t0].layer) {  // one layer: sum of sigma nu
            den += snu[t1];
            sum += snu[t1] * lr[t1];
            ++t1;
        }
        if (den > 0.0) E += sum / den;
        t0 = t1;
    }
    const double uc = (double)n_tied / N, mp = (double)extra / ((double)N * n_classes);
    cost[4 * c + 0] = E + uc + mp;
    cost[4 * c + 1] = E;
    cost[4 * c + 2] = uc;
    cost[4 * c + 3] = mp;
}

// one warp per sample: the number of classes whose logit equals the sample's largest
template <typename T>
__global__ void top1_ties_kernel(const T* __restrict__ logits, int N, int C, int32_t* __restrict__ counts) {
    pdl_wait();
    const int n = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (n >= N) return;
    const T* row = logits + (long long)n * C;
    T best = row[0];
    for (int c = lane; c < C; c += 32) best = row[c] > best ? row[c] : best;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const T o = __shfl_xor_sync(0xFFFFFFFFu, best, off);
        best = o > best ? o : best;
    }
    int cnt = 0;
    for (int c = lane; c < C; c += 32) cnt += row[c] == best ? 1 : 0;
    cnt = __reduce_add_sync(0xFFFFFFFFu, (unsigned)cnt);
    if (lane == 0) counts[n] = cnt;
}

__global__ void nchw_to_nhwc_kernel(const float* __restrict__ x, int N, int C, int HW, float* __restrict__ y) {
    const long long total = (long long)N * C * HW;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i % C);
        const long long pix = i / C;  // n * HW + p
        const long long n = pix / HW;
        y[i] = x[(n * C + c) * HW + (pix - n * HW)];
    }
}

int grid_of(long long work) {
    long long b = (work + 255) / 256;
    if (b < 1) b = 1;
    if (b > 152LL * 16) b = 152LL * 16;
    return (int)b;
}

}  // namespace
}  // namespace fxpq

using namespace fxpq;

extern "C" fxpq_status fxpq_conv_f32(const fxpq_conv_f32_desc* h_desc, const float* d_x, const float* d_w,
                                     const float* d_bias, float* d_y, void* stream) {
    if (!h_desc) return FXPQ_ERR_INVALID_ARG;
    const fxpq_conv_f32_desc& d = *h_desc;
    if (d.N < 0 || d.H < 1 || d.W < 1 || d.C < 1 || d.K < 1 || d.R < 1 || d.S < 1 || d.stride < 1 || d.pad < 0)
        return FXPQ_ERR_INVALID_ARG;
    const int P = (d.H + 2 * d.pad - d.R) / d.stride + 1, Q = (d.W + 2 * d.pad - d.S) / d.stride + 1;
    if (P < 1 || Q < 1) return FXPQ_ERR_INVALID_ARG;
    if (d.N > 0 && (!d_x || !d_w || !d_y)) return FXPQ_ERR_INVALID_ARG;
    ConvF32Args a{d_x, d_w, d_bias, d_y, d.N, d.H, d.W, d.C, d.K, d.R, d.S, d.stride, d.pad, P, Q, d.relu ? 1 : 0,
                  (long long)d.N * P * Q};
    if (a.M == 0) return FXPQ_OK;
    const bool vec = d.C % 4 == 0 && aligned(d_x, 16) && aligned(d_w, 16);
    const bool wide = !vec && ((long long)d.R * d.W + d.S) * d.C >= (1LL << 31);
    // 32-pixel tiles for few output pixels (FC layers of a calibration slice), where 64-pixel ones are mostly empty
    const int bm = a.M <= 32 && !wide ? 32 : 64;
    const long long cols = ((long long)d.K + CF_BN - 1) / CF_BN;
    cudaStream_t s = as_stream(stream);
    for (long long c0 = 0; c0 < cols; c0 += 65535) {  // (a grid has at most 65535 rows)
        a.n_first = (int)(c0 * CF_BN);
        const dim3 grid((unsigned)((a.M + bm - 1) / bm), (unsigned)(cols - c0 < 65535 ? cols - c0 : 65535));
        if (wide)
            launch_pdl(conv_f32_kernel<64, false, long long>, grid, 256, 0, s, a);
        else if (bm == 32 && vec)
            launch_pdl(conv_f32_kernel<32, true>, grid, 256, 0, s, a);
        else if (bm == 32)
            launch_pdl(conv_f32_kernel<32, false>, grid, 256, 0, s, a);
        else if (vec)
            launch_pdl(conv_f32_kernel<64, true>, grid, 256, 0, s, a);
        else
            launch_pdl(conv_f32_kernel<64, false>, grid, 256, 0, s, a);
        const fxpq_status st = after_launch("conv_f32");
        if (st != FXPQ_OK) return st;
    }
    return FXPQ_OK;
}

extern "C" fxpq_status fxpq_maxpool_f32(const float* d_x, int32_t N, int32_t H, int32_t W, int32_t C, int32_t k,
                                        int32_t stride, int32_t pad, float* d_y, void* stream) {
    if (N < 0 || H < 1 || W < 1 || C < 1 || k < 1 || stride < 1 || pad < 0 || pad >= k) return FXPQ_ERR_INVALID_ARG;
    const int P = (H + 2 * pad - k) / stride + 1, Q = (W + 2 * pad - k) / stride + 1;
    if (P < 1 || Q < 1 || (N > 0 && (!d_x || !d_y))) return FXPQ_ERR_INVALID_ARG;
    const long long total = (long long)N * P * Q * C;
    if (total == 0) return FXPQ_OK;
    launch_pdl(maxpool_f32_kernel, grid_of(total), 256, 0, as_stream(stream), d_x, N, H, W, C, k, stride, pad, P, Q, d_y);
    return after_launch("maxpool_f32");
}

extern "C" fxpq_status fxpq_eltwise_f32(const float* d_a, const float* d_b, int64_t n, int32_t relu, float* d_y,
                                        void* stream) {
    if (n < 0 || (n > 0 && (!d_a || !d_b || !d_y))) return FXPQ_ERR_INVALID_ARG;
    if (n == 0) return FXPQ_OK;
    launch_pdl(eltwise_f32_kernel, grid_of(n), 256, 0, as_stream(stream), d_a, d_b, n, relu, d_y);
    return after_launch("eltwise_f32");
}

extern "C" fxpq_status fxpq_avgpool_f32(const float* d_x, int32_t N, int32_t H, int32_t W, int32_t C, float* d_y,
                                        void* stream) {
    if (N < 0 || H < 1 || W < 1 || C < 1 || (N > 0 && (!d_x || !d_y))) return FXPQ_ERR_INVALID_ARG;
    const long long total = (long long)N * C;
    if (total == 0) return FXPQ_OK;
    launch_pdl(avgpool_f32_kernel, (unsigned)((total + 255) / 256), 256, 0, as_stream(stream), d_x, N, H * W, C, d_y);
    return after_launch("avgpool_f32");
}

extern "C" fxpq_status fxpq_dequantize(const void* d_codes, int64_t npix, int32_t Cp, int32_t C, fxpq_fmt fmt,
                                       float* d_y, void* stream) {
    if (npix < 0 || C < 1 || Cp < C || !fmt_ok1(fmt) || (npix > 0 && (!d_codes || !d_y))) return FXPQ_ERR_INVALID_ARG;
    if (npix == 0) return FXPQ_OK;
    launch_pdl(dequantize_kernel, grid_of(npix * C), 256, 0, as_stream(stream),
        static_cast<const __half*>(d_codes), npix, Cp, C, planes_of(fmt), ldexpf(1.0f, -fmt.fl),
        fmt.bits == 1 && fmt.is_signed == 1, d_y);
    return after_launch("dequantize");
}

extern "C" fxpq_status fxpq_bias_relu_f32(float* d_y, int64_t npix, int32_t K, const float* d_bias, int32_t relu,
                                          void* stream) {
    if (npix < 0 || K < 1 || (npix > 0 && !d_y)) return FXPQ_ERR_INVALID_ARG;
    if (npix == 0) return FXPQ_OK;
    bias_relu_f32_kernel<<<grid_of(npix * K), 256, 0, as_stream(stream)>>>(d_y, npix, K, d_bias, relu);
    return after_launch("bias_relu_f32");
}

namespace {
// Units of one item (DS_CHUNK values of one sample each), or -1 for an invalid item.
long long ds_units(const fxpq_ds_item& it) {
    if (it.n_samples < 1 || it.n_samples > 65535 || it.nu < 1 || !fxpq::fmt_ok1(it.fmt, 32) || !it.d_x || !it.d_out)
        return -1;
    return (long long)it.n_samples * ((it.nu + DS_CHUNK - 1) / DS_CHUNK);
}
}  // namespace

extern "C" size_t fxpq_ds_stats_batch_workspace(const fxpq_ds_item* h_items, int32_t n_items) {
    if (n_items < 1 || n_items > 4096 || !h_items) return 0;
    long long most = 0;  // the largest launch group's units
    for (int i0 = 0; i0 < n_items; i0 += DS_MAX_ITEMS) {
        long long u = 0;
        for (int i = i0; i < n_items && i < i0 + DS_MAX_ITEMS; ++i) {
            const long long v = ds_units(h_items[i]);
            if (v < 0) return 0;
            u += v;
        }
        most = u > most ? u : most;
    }
    return ((size_t)most * sizeof(DsUnit) + 255) / 256 * 256;
}

extern "C" fxpq_status fxpq_ds_stats_batch(const fxpq_ds_item* h_items, int32_t n_items, void* d_ws, size_t ws_bytes,
                                           void* stream) {
    if (n_items < 1 || n_items > 4096 || !h_items) return FXPQ_ERR_INVALID_ARG;
    for (int i = 0; i < n_items; ++i)
        if (ds_units(h_items[i]) < 0) return FXPQ_ERR_INVALID_ARG;
    const size_t need = fxpq_ds_stats_batch_workspace(h_items, n_items);
    if (!d_ws || ws_bytes < need || !aligned(d_ws, 256)) return FXPQ_ERR_WORKSPACE;
    cudaStream_t s = as_stream(stream);
    DsUnit* units = static_cast<DsUnit*>(d_ws);
    for (int i0 = 0; i0 < n_items; i0 += DS_MAX_ITEMS) {
        DsBatchDev B;
        B.n = 0;
        long long u = 0;
        for (int i = i0; i < n_items && i < i0 + DS_MAX_ITEMS; ++i) {
            const fxpq_ds_item& h = h_items[i];
            DsItemDev& d = B.it[B.n++];
            d.x = h.d_x;
            d.out = h.d_out;
            d.nu = h.nu;
            d.n_samples = h.n_samples;
            d.k = h.fmt.bits;
            d.S = h.fmt.is_signed;
            d.fl = h.fmt.fl;
            d.chunks = (int)((h.nu + DS_CHUNK - 1) / DS_CHUNK);
            d.unit0 = (int)u;
            u += ds_units(h);
        }
        if (u > 0x7FFFFFFFLL) return FXPQ_ERR_INVALID_ARG;
        B.unit_end = (int)u;
        launch_pdl(ds_sum_kernel, (unsigned)u, DS_T, 0, s, B, units);
        fxpq_status st = after_launch("ds_sum");
        if (st != FXPQ_OK) return st;
        launch_pdl(ds_dev_kernel, (unsigned)u, DS_T, 0, s, B, units);
        st = after_launch("ds_dev");
        if (st != FXPQ_OK) return st;
        launch_pdl(ds_finish_kernel, B.n, DF_T, 0, s, B, units);
        st = after_launch("ds_finish");
        if (st != FXPQ_OK) return st;
    }
    return FXPQ_OK;
}

extern "C" fxpq_status fxpq_fopt_cost(const double* d_stats, int64_t cand_stride, const fxpq_cost_term* h_terms,
                                      int32_t n_terms, const int32_t* d_ties, int32_t N, int32_t n_classes,
                                      int32_t n_cand, double* d_cost, void* stream) {
    if (n_terms < 0 || n_terms > COST_MAX_TERMS || (n_terms > 0 && !h_terms) || N < 1 || n_classes < 1 || n_cand < 1 ||
        cand_stride < 0 || !d_stats || !d_ties || !d_cost)
        return FXPQ_ERR_INVALID_ARG;
    CostTerms T;
    T.n = n_terms;
    for (int i = 0; i < n_terms; ++i) {
        const fxpq_cost_term& h = h_terms[i];
        if (h.offset < 0 || h.nu < 1 || h.n_samples < 1) return FXPQ_ERR_INVALID_ARG;
        T.t[i] = CostTermDev{h.offset, h.nu, h.n_samples, h.layer};
    }
    launch_pdl(fopt_cost_kernel, n_cand, 128, 0, as_stream(stream), d_stats, cand_stride, T, d_ties, N, n_classes, d_cost);
    return after_launch("fopt_cost");
}

extern "C" fxpq_status fxpq_top1_ties(const void* d_logits, int32_t is_int64, int32_t N, int32_t C, int32_t* d_counts,
                                      void* stream) {
    if (N < 0 || C < 1 || (N > 0 && (!d_logits || !d_counts))) return FXPQ_ERR_INVALID_ARG;
    if (N == 0) return FXPQ_OK;
    const unsigned blocks = (unsigned)((N + 7) / 8);
    if (is_int64)
        launch_pdl(top1_ties_kernel<long long>, blocks, 256, 0, as_stream(stream), static_cast<const long long*>(d_logits), N, C,
                                                                           d_counts);
    else
        launch_pdl(top1_ties_kernel<float>, blocks, 256, 0, as_stream(stream), static_cast<const float*>(d_logits), N, C,
                                                                       d_counts);
    return after_launch("top1_ties");
}

extern "C" fxpq_status fxpq_nchw_to_nhwc_f32(const float* d_x, int32_t N, int32_t C, int32_t H, int32_t W, float* d_y,
                                             void* stream) {
    if (N < 0 || C < 1 || H < 1 || W < 1 || (N > 0 && (!d_x || !d_y))) return FXPQ_ERR_INVALID_ARG;
    const long long total = (long long)N * C * H * W;
    if (total == 0) return FXPQ_OK;
    nchw_to_nhwc_kernel<<<grid_of(total), 256, 0, as_stream(stream)>>>(d_x, N, C, H * W, d_y);
    return after_launch("nchw_to_nhwc");
}
