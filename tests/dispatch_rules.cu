// dispatch_rules.cu -- host program of test_dispatch_rules_host.py: reads requests (a rule's name, the
// camera, the cube's dims and a number) and prints 1 or 0 for each, the rule's choice.
#include <cstdio>
#include <cstring>

#include "render_axis.cuh"
#include "render_impl.cuh"
#include "render_roll.cuh"
#include "render_slab.cuh"

using namespace shw;

int main()
{
    char rule[32];
    shw_camera c{};
    int n[3], k;
    auto three = [](float *v) { return std::scanf("%f %f %f", v, v + 1, v + 2) == 3; };
    while (std::scanf("%31s", rule) == 1) {
        if (!three(c.eye) || !three(c.right) || !three(c.up) || !three(c.fwd) ||
            std::scanf("%f %f %d %d %d %d %d %d %d", &c.tan_half_fovy, &c.ortho_half_h, &c.ortho, &c.width, &c.height, n,
                       n + 1, n + 2, &k) != 9)
            return 2;
        bool yes = false;
        const double warps = covered_pixels(c, n[0], n[1], n[2]) / 32.0, rows = warp_rows(c, n[0], n[1], n[2]);
        const double vox = (double)n[0] * n[1] * n[2];
        if (!std::strcmp(rule, "many")) yes = render_raised<SHW_RATIO, SHW_TRILINEAR>(warps, rows, vox);
        if (!std::strcmp(rule, "staged")) yes = slab_pays<SlabGeom<ElemF32>>(c, n[0], n[1], n[2], false);
        if (!std::strcmp(rule, "staged_composite")) yes = slab_pays<SlabGeom<ElemF32>>(c, n[0], n[1], n[2], true);
        if (!std::strcmp(rule, "staged_pair")) yes = slab_pays<SlabGeom<ElemF32Pair>>(c, n[0], n[1], n[2], false);
        if (!std::strcmp(rule, "rows")) yes = axis_rows_pay(k, SHW_TRILINEAR, c, n[2]);
        if (!std::strcmp(rule, "rows_nearest")) yes = axis_rows_pay(k, SHW_NEAREST, c, n[2]);
        const bool tmaps = n[0] % 4 == 0;
        if (!std::strcmp(rule, "taps")) yes = roll_pays<kRollTaps>(c, n, tmaps, k, false, 1.0f);
        if (!std::strcmp(rule, "taps_composite")) yes = roll_pays<kRollTaps>(c, n, tmaps, k, true, 1.0f);
        if (!std::strcmp(rule, "box")) yes = roll_pays<kRollBox>(c, n, tmaps, k, false, 3.0f);
        if (!std::strcmp(rule, "box_composite")) yes = roll_pays<kRollBox>(c, n, tmaps, k, true, 3.0f);
        std::printf("%d\n", yes ? 1 : 0);
    }
    return 0;
}
