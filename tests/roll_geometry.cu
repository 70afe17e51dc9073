// roll_geometry.cu -- host program of test_roll_geometry_host.py: the rolling marcher's staging
// geometry over views that pan across and past a cube, for every reach of the taps.  Prints the
// number of geometries accepted and refused; exits 1 with the first one that breaks an invariant.
#include <cmath>
#include <cstdio>
#include <initializer_list>

#include "render_roll.cuh"

using namespace shw;

// Parallel view along axis `ax` (dir +-1) tilted by `tilt`, panned by `pan` voxels sideways.
static shw_camera view(const int n[3], int ax, float dir, float tilt, int side, float pan, int w, int h, float half)
{
    shw_camera c{};
    const int r = (ax + 1) % 3, u = (ax + 2) % 3, s = side ? u : r;
    const float cs = std::cos(tilt), sn = std::sin(tilt);
    c.fwd[ax] = dir * cs;
    c.fwd[r] = sn;
    c.right[ax] = -dir * sn;
    c.right[r] = cs;
    c.up[u] = 1.0f;
    for (int k = 0; k < 3; ++k) c.eye[k] = 0.5f * (n[k] - 1) - 400.0f * c.fwd[k];
    c.eye[s] += pan;
    c.ortho = 1;
    c.ortho_half_h = half;
    c.width = w;
    c.height = h;
    return c;
}

template <int M>
static void footprint(const TileRays &r, const int n[3], int H, int wa[3], int wb[3])
{
    roll_extent<M>(r, n, H, M == 0 ? kRollXG : 1, wa[M], wb[M]);
}

// The box of every major axis in use holds the footprints of the sampled tiles (as far as the cube
// and a copy's 256 elements go), its planes and slots are as large, and the ring fits the budget.
static bool sound(const shw_camera &cam, const int n[3], int H, int budget, const RollArgs &ra)
{
    int wa[3] = {0, 0, 0}, wb[3] = {0, 0, 0};
    const int on[3] = {1, 1, 1}, tx = ceil_div(cam.width, kSlabTW), ty = ceil_div(cam.height, kSlabTH);
    for (int j = 0; j < 5; ++j)
        for (int i = 0; i < 5; ++i) {
            const TileRays r = roll_rays(cam, (int)((long long)(tx - 1) * i / 4) * kSlabTW,
                                         (int)((long long)(ty - 1) * j / 4) * kSlabTH, on, ra.xbias);
            if (r.major == 0) footprint<0>(r, n, H, wa, wb);
            else if (r.major == 1) footprint<1>(r, n, H, wa, wb);
            else footprint<2>(r, n, H, wa, wb);
        }
    for (int M = 0; M < 3; ++M) {
        const RollGeom &G = ra.geo[M];
        if (!G.on) continue;
        if (G.wa < wa[M] || G.wb < wb[M] || G.wa <= 0 || G.wb <= 0 || G.wa > 256 || G.wb > 256) return false;
        if (G.sb < G.wa || G.plane < G.sb * G.wb || G.slot != G.plane * G.g || G.slot % 32) return false;
        if (G.s < 1 || G.ns < roll_slots(H, G.s, G.g, G.depth) || G.ns > kRollMaxSlots || G.ns * G.g > kRollTable)
            return false;
        if ((long long)G.ns * G.slot * 4 > budget || G.ns * G.slot * 4 > ra.smem_stage) return false;
    }
    return true;
}

int main()
{
    const int cubes[][3] = {{128, 128, 128}, {64, 64, 64}, {65, 130, 67}, {3, 5, 64}, {300, 20, 1}, {1, 1, 1}};
    const int images[][2] = {{256, 256}, {33, 17}};
    const float tilts[] = {0.0f, 0.3f};
    long long accepted = 0, refused = 0;
    for (const auto &n : cubes)
        for (const auto &im : images)
            for (int ax = 0; ax < 3; ++ax)
                for (int side = 0; side < 2; ++side)
                    for (const float tilt : tilts) {
                        // the largest cube pans past its edge in quarter voxels, the others coarsely
                        const bool fine = n[0] == 128 && im[0] == 256 && tilt == 0.0f;
                        for (int q = fine ? 440 : 0; q <= 800; q += fine ? 1 : 37)
                            for (const int H : {0, 1, 2, 4, 9, 14, 16, 24, 32, 64}) {
                                const shw_camera cam = view(n, ax, q & 1 ? 1.0f : -1.0f, tilt, side, 0.25f * q, im[0],
                                                            im[1], 0.5f * (float)n[(ax + 2) % 3]);
                                for (int k = 0; k < 2; ++k) {  // two CTAs per SM, and one
                                    RollArgs ra{};
                                    ra.xbias = k ? 1.0f : 3.0f;
                                    ra.halo = H;
                                    const int budget = (k ? kRollBudget1 : kRollBudget2) - (int)sizeof(RollShared);
                                    if (!roll_geometry(cam, n, H, n[0] % 4 == 0, budget, 4, k ? 1 : 2, ra)) {
                                        ++refused;
                                        continue;
                                    }
                                    ++accepted;
                                    if (!sound(cam, n, H, budget, ra)) {
                                        std::printf("unsound: cube %d x %d x %d, image %d x %d, axis %d, pan %g, reach %d\n",
                                                    n[0], n[1], n[2], im[0], im[1], ax, 0.25 * q, H);
                                        return 1;
                                    }
                                }
                            }
                    }
    std::printf("%lld %lld\n", accepted, refused);
    return 0;
}
