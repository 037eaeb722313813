// Host-side check of the tensor-core path's choices (row tiles, patches, packed weights, space-to-depth) for 152 SMs:
// every layer read from stdin is planned with the library's own host planner (plan_conv, s2d_plan, choose_form), which
// touches no device.  tests/test_form_host.py compiles it against the library's objects.
//
// Input, one layer per line:   N H W C Cp K R S stride pad  xb wb  out_mode packed s2d path ("-": none)
//   s2d 1: the layer in its space-to-depth form (where it has one)
// Output, one line per layer:  status s2d_ok planned  rows_geom narrow use_patch pk BN n_groups  overlap  TW TH TN tiles
//   overlap: the pixels of x overlap, which only a tensor map can read
#include <cstdio>

#include "fxpq_conv_tc.cuh"

using namespace fxpq;
using namespace fxpq::tc;

int main() {
    int v[15];
    char path[32];
    static __align__(16) int32_t dummy[16];  // checked for null and alignment only
    while (true) {
        int got = 0;
        for (int i = 0; i < 15; ++i) got += scanf("%d", &v[i]) == 1;
        if (got != 15 || scanf("%31s", path) != 1) break;
        fxpq_conv_desc d = {};
        d.N = v[0], d.H = v[1], d.W = v[2], d.C = v[3], d.Cp = v[4], d.K = v[5], d.R = v[6], d.S = v[7];
        d.stride = v[8], d.pad = v[9];
        d.fmt_x = fxpq_fmt{v[10], 0, 0}, d.fmt_w = fxpq_fmt{v[11], 1, 4}, d.fmt_y = fxpq_fmt{8, 0, 0};
        d.out_mode = v[12];
        d.d_wpacked = v[13] ? dummy : nullptr;
        ConvArgs a{};
        int32_t s_out = 0;
        bool need64 = false;
        const fxpq_status st = plan_conv(d, dummy, dummy, nullptr, dummy, a, &s_out, need64);
        const S2dPlan p = s2d_plan(d);
        static TcParams P;
        TcForm f = {};
        bool planned = false;
        if (st == FXPQ_OK && (!v[14] || p.ok)) {
            fxpq_conv_desc e = d;
            if (v[14]) {
                a = s2d_args(a, p, a.x, a.w);
                e = s2d_desc(d);
            }
            planned = choose_form(a, e, path[0] == '-' ? nullptr : path, 152, true, P, f);
        }
        printf("%d %d %d  %d %d %d %d %d %d  %d  %d %d %d %lld\n", (int)st, (int)p.ok, (int)planned, (int)f.rows_geom, (int)f.narrow,
               (int)f.use_patch, (int)f.pk, f.BN, P.n_groups, (int)(a.x_sw != a.Cp), f.ps.TW, f.ps.TH, f.ps.TN, f.ps.tiles);
    }
    return 0;
}
