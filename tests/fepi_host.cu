// Host-side check of the fp32 epilogue of layers of one exact group: plans each case read from stdin with the library's
// host planner (plan_conv: whether the fp32 forms apply, their constants and error bound) and evaluates, on the CPU, the
// inline functions that the tensor-core kernel uses (fepi_bias, fepi_scale, fepi_image) in the kernel's order of operations.
// tests/test_fepi_host.py compiles it against the library's objects.
//
// Input: as tests/epilogue_host.cu.  Output, one line per case:
//   status  vf code  vs code near  image bits     (NA = -2147483648 where a form does not apply or |acc| >= 2^24)
//   near: the Scale layer's value lies within its error bound of a rounding boundary, where the kernel decides exactly
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "fxpq_conv_tc.cuh"

using namespace fxpq;

int main() {
    long long v[27];
    const long long NA = INT_MIN;
    while (true) {
        int got = 0;
        for (int i = 0; i < 27; ++i) got += scanf("%lld", &v[i]) == 1;
        if (got != 27) break;
        fxpq_conv_desc d = {};
        d.N = 1, d.H = 1, d.W = 1, d.C = (int)v[14], d.Cp = (int)((v[14] + 7) / 8 * 8);
        d.K = 8, d.R = 1, d.S = 1, d.stride = 1, d.pad = 0;
        d.relu = (int)v[12];
        d.fmt_x = fxpq_fmt{(int)v[0], (int)v[1], (int)v[2]};
        d.fmt_w = fxpq_fmt{(int)v[3], (int)v[4], (int)v[5]};
        d.fmt_b = fxpq_fmt{(int)v[6], (int)v[7], (int)v[8]};
        d.fmt_y = fxpq_fmt{(int)v[9], (int)v[10], (int)v[11]};
        d.w_l1 = v[15];
        const bool has_bias = v[13] != 0, has_scale = v[18] != 0;
        static __align__(16) int32_t dummy[16];  // checked for null and alignment only
        if (has_scale) {
            d.fmt_scale = fxpq_fmt{(int)v[19], (int)v[20], (int)v[21]};
            d.fmt_shift = fxpq_fmt{(int)v[22], (int)v[23], (int)v[24]};
            d.d_scale = dummy;
            d.d_shift = dummy;
        }
        const float acc = (float)v[16];
        const bool exact = std::llabs(v[16]) < (1ll << 24);
        const int32_t b = has_bias ? (int32_t)v[17] : 0, m = (int32_t)v[25], h = (int32_t)v[26];
        long long vf = NA, vs = NA, near = 0, image = NA;
        ConvArgs a{};
        int32_t s_out = 0;
        bool need64 = false;
        d.out_mode = FXPQ_OUT_CODES;
        const fxpq_status st = plan_conv(d, dummy, dummy, has_bias ? dummy : nullptr, dummy, a, &s_out, need64);
        if (st == FXPQ_OK && exact && a.vf) {
            const float x = std::fma(acc, a.vf_c, a.has_bias ? fepi_bias(a, b) : 0.0f);
            vf = std::lrint(std::fmin(std::fmax(x, a.vf_lo), a.vf_hi));
        }
        if (st == FXPQ_OK && exact && a.vs) {
            const float2 mt = fepi_scale(a, b, m, h);
            const float x = std::fmin(std::fmax(std::fma(acc, mt.x, mt.y), a.vf_lo), a.vf_hi);
            vs = std::lrint(x);
            near = std::fabs(x - (float)vs) > 0.5f - a.vs_eps;
        }
        d.out_mode = FXPQ_OUT_F32;
        if (plan_conv(d, dummy, dummy, has_bias ? dummy : nullptr, dummy, a, &s_out, need64) == FXPQ_OK && exact && (a.vi || a.vs)) {
            const float2 mt = a.vs ? fepi_scale(a, b, m, h) : make_float2(a.vi_c, (float)b * a.vi_b);
            const float t = std::fma(acc, mt.x, mt.y), f = a.relu ? std::fmax(t, 0.0f) : t;
            uint32_t bits;
            memcpy(&bits, &f, 4);
            image = bits;
        }
        printf("%d %lld %lld %lld %lld\n", (int)st, vf, vs, near, image);
    }
    return 0;
}
