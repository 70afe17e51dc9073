// axis_box.cu -- host program of test_axis_box_host.py: the plane sweep's staged box for pixel
// footprints from a fraction of a voxel to beyond the range of an int.  Exits 1 with the first one
// that is accepted without being sound; prints the number accepted and refused.
#include <cstdio>

#include "render_axis.cuh"

using namespace shw;

int main()
{
    int accepted = 0, refused = 0;
    for (int rows = 0; rows < 2; ++rows)
        for (int nx = 1; nx <= 9; ++nx)
            for (const int mode : {(int)SHW_MIP, (int)SHW_MOMENT1, kMipValue})
                for (double ex = 0.25; ex < 1e40; ex *= 1.37)
                    for (double ey = 0.25; ey < 1e40; ey *= ex < 1e4 ? 1.37 : 19.0) {
                        if (!rows && nx % 4) continue;
                        AxisArgs A{};
                        A.rows = rows;
                        bool fix = false;
                        size_t smem = 0;
                        if (!axis_box(ex, ey, nx, mode, A, fix, smem)) {
                            ++refused;
                            continue;
                        }
                        ++accepted;
                        const long long stride = A.stage_stride, pitch = A.pitch, bw = A.bw, bh = A.bh;
                        const bool ok = bw >= ex && bh >= ey && bw <= 256 && bh <= 256 && bw % 4 == 0 && !(rows && fix) &&
                                        pitch >= bw + (rows ? 10 : 0) && (!rows || (pitch - nx) % 4 == 0) &&
                                        stride >= (fix ? bw : pitch) * bh + (rows ? 16 : 0) && stride % 32 == 0 &&
                                        (long long)smem == axis_stages(mode, fix) * stride * 4 && smem <= (size_t)kAxSmemLimit;
                        if (!ok) {
                            std::printf("unsound: rows %d, nx %d, mode %d, %g x %g voxels: box %lld x %lld, pitch %lld, "
                                        "stride %lld\n", rows, nx, mode, ex, ey, bw, bh, pitch, stride);
                            return 1;
                        }
                    }
    std::printf("%d %d\n", accepted, refused);
    return 0;
}
