// adjoint.cu -- reverse-mode gradient of the compositing render (Algorithm 3 in
// premultiplied form) with respect to the voxels, the 256-entry colour map and the
// opacity scale.
//
// Forward recurrence per ray (k = 0..K-1, K = samples processed):
//   a_k = clamp(s * A_lut(v_hat_k), 0, 1),  C += T_k a_k c_k,  T_{k+1} = T_k (1 - a_k),
//   outputs (C, 1 - T_K).
// Reverse, with gT = dL/dT_{k+1} carried from the end (gT = -dL/dalpha at k = K):
//   dL/da_k   = sum_c gC_c T_k c_k,c  - gT T_k
//   dL/dc_k   = gC T_k a_k
//   dL/dT_k   = gT (1 - a_k) + sum_c gC_c a_k c_k,c
// The transmittance T_k is not stored per sample: the forward kept it every
// `ckpt_interval` samples, and each segment is recomputed from its checkpoint
// into a per-thread array before being walked backwards (memory O(K / interval)
// per ray instead of O(K)).  Clamp kinks pass the gradient on the closed interval.
#include "common.cuh"
#include "ray.cuh"
#include "render_impl.cuh"
#include "sampler.cuh"

namespace shw {

constexpr int kMaxCkptInterval = 64;
constexpr int kBwdThreads = 768;  // one CTA per SM (below)

struct BackwardArgs {
    const float4 *grad_rgba;  // [H][W]
    const int *ckpt_K;        // [H][W]
    const float *ckpt_T;      // [nckpt][H][W]
    float *grad_vol;          // [nz][ny][nx] or null
    float *grad_lut;          // [256][4] or null
    float *grad_scale;        // [1] or null
    const float4 *lut;
    int width, height, nckpt, ckpt_interval, nmax;
    int tiles_x, tiles_y, ctx, cty;  // 8 x 4 pixel tiles; the one at the projected cube centre
    float step, lo, inv_range, opacity_scale;
};

// The voxel gradients of one interpolation cell, kept in registers while a ray's samples stay in
// it (half-voxel steps: about two samples a cell) and added to memory when the ray leaves.
// Clamped indices accumulate on the edge voxel.
template <class Idx>
struct CellGrad {
    int ix = -4, iy = 0, iz = 0;  // the cell (-4: none)
    float g[8];
    __device__ __forceinline__ void flush(float *gv, int nx, int ny, int nz)
    {
        if (ix == -4) return;
        const int x0 = max(ix, 0), dx = min(ix + 1, nx - 1) - x0;
        const int y0 = max(iy, 0), dy = min(iy + 1, ny - 1) - y0;
        const int z0 = max(iz, 0), dz = min(iz + 1, nz - 1) - z0;
        const Idx sy = nx, sz = (Idx)nx * ny;
        float *p = gv + ((Idx)z0 * sz + (Idx)y0 * sy + x0);
        float *py = p + dy * sy, *pz = p + dz * sz, *pyz = pz + dy * sy;
        atomicAdd(p, g[0]);
        atomicAdd(p + dx, g[1]);
        atomicAdd(py, g[2]);
        atomicAdd(py + dx, g[3]);
        atomicAdd(pz, g[4]);
        atomicAdd(pz + dx, g[5]);
        atomicAdd(pyz, g[6]);
        atomicAdd(pyz + dx, g[7]);
    }
    __device__ __forceinline__ void add(float *gv, int nx, int ny, int nz, long long X, long long Y, long long Z, float v)
    {
        const int cx = clampi(fx_cell(X), -1, nx - 1), cy = clampi(fx_cell(Y), -1, ny - 1),
                  cz = clampi(fx_cell(Z), -1, nz - 1);
        const float fx = fx_frac(X), fy = fx_frac(Y), fz = fx_frac(Z);
        if (cx != ix || cy != iy || cz != iz) {
            flush(gv, nx, ny, nz);
            ix = cx;
            iy = cy;
            iz = cz;
#pragma unroll
            for (int c = 0; c < 8; ++c) g[c] = 0.0f;
        }
        const float wx[2] = {1.0f - fx, fx}, wy[2] = {1.0f - fy, fy}, wz[2] = {1.0f - fz, fz};
#pragma unroll
        for (int c = 0; c < 8; ++c) g[c] += v * wx[c & 1] * wy[(c >> 1) & 1] * wz[c >> 2];
    }
};

// Shared memory of a CTA: the colour map, and one set of colour-map sums per warp: entry i's
// sums of (1 - f) dL/dc (its own share of the samples between knots i and i + 1) and of f dL/dc
// (its upper neighbour's share), 8 floats together.
constexpr int kBwdWarps = kBwdThreads / 32, kBwdSums = kLut * 8;
constexpr size_t kBwdSmem = sizeof(float4) * kLut + sizeof(float) * kBwdWarps * kBwdSums;

// Persistent CTAs whose warps take 8 x 4 pixel tiles in turn, centre-out, there and back (warp w
// the w-th of the first round, the w-th last of the second), so that long rays are paired with
// short ones; one ray per thread.  (By index, not from a counter: the call may be captured into
// a graph and replayed.)
//
// What bounds it: the scatter.  A sample adds to 8 voxels (global reductions that nothing waits
// for) and to 8 colour-map sums; as shared-memory float atomics, which are compare-and-swap
// loops on addresses that the rays of a CTA share, the latter took most of the time (256^3 cube,
// 512 x 512: 3.52 ms, 86 % of the shared-memory pipe, half the instructions).  Here every warp
// has its own sums and its lanes add to them in turns: __match_any_sync groups the lanes by
// entry, each lane's rank in its group is its turn, and the turns (the largest group: 3 to 4)
// are plain 16-byte loads, adds and stores.  Lanes of a warp therefore step together.  With that
// 2.68 ms; the voxels of a cell added once per visit and the tiles handed out there and back 1.37 ms:
// the warps then wait on the recomputed fetches and the turns, and at the end on the longest rays (6 of
// 16 cycles an instruction at the last barrier).
// One CTA of 24 warps per SM, not three of 8: the global sums then take 152 additions each, and
// their rounding stays below that of one addition per 16 x 16 pixels.
template <int INTERP, class Idx>
__global__ void __launch_bounds__(kBwdThreads) backward_kernel(SamplerF32<Idx> s, shw_camera cam, BackwardArgs a)
{
    extern __shared__ __align__(16) unsigned char bwd_smem[];
    float4 *lut_s = reinterpret_cast<float4 *>(bwd_smem);
    float *sums = reinterpret_cast<float *>(bwd_smem + sizeof(float4) * kLut);
    __shared__ float gs_s;
    for (int i = threadIdx.x; i < kLut; i += blockDim.x) lut_s[i] = a.lut[i];
    for (int i = threadIdx.x; i < kBwdWarps * kBwdSums; i += blockDim.x) sums[i] = 0.0f;
    if (threadIdx.x == 0) gs_s = 0.0f;
    __syncthreads();
    float4 *mine = reinterpret_cast<float4 *>(sums + (threadIdx.x >> 5) * kBwdSums);
    const int lane = threadIdx.x & 31;
    const long long npix = (long long)a.width * a.height;
    const int I = a.ckpt_interval;
    float vseg[kMaxCkptInterval], Tseg[kMaxCkptInterval];

    float gs_sum = 0.0f, gs_comp = 0.0f;  // the warp's scale gradient (compensated over its tiles)
    const int warps = (int)gridDim.x * kBwdWarps, me = (int)(blockIdx.x + gridDim.x * (threadIdx.x >> 5));
    const int ntiles = a.tiles_x * a.tiles_y;
    for (int round = 0; round * warps < ntiles; ++round) {
        const int t = round * warps + (round & 1 ? warps - 1 - me : me);
        if (t >= ntiles) continue;
        const int rr = t / a.tiles_x, cr = t - rr * a.tiles_x;
        const int px = centre_out(cr, a.ctx, a.tiles_x) * 8 + (lane & 7);
        const int py = centre_out(rr, a.cty, a.tiles_y) * 4 + (lane >> 3);
        const bool inside = px < a.width && py < a.height;
        const long long pix = inside ? (long long)py * a.width + px : 0;
        RayFx r;
        const bool hit = inside && setup_ray(cam, px, py, s.nx, s.ny, s.nz, a.step, r);
        const int K = hit ? max(min(min(a.ckpt_K[pix], r.N), a.nmax), 0) : 0;
        const float4 g = hit ? a.grad_rgba[pix] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float gT = -g.w;  // alpha_out = 1 - T_K
        float gs = 0.0f;
        CellCache cc;
        CellGrad<Idx> cg;
        const int Kw = (int)__reduce_max_sync(0xffffffffu, (unsigned)K);  // the warp's longest ray
        for (int m = Kw > 0 ? (Kw - 1) / I : -1; m >= 0; --m) {
            const int k0 = m * I, n = min(max(K - k0, 0), I), nw = min(Kw - k0, I);
            // recompute the segment forward from its checkpoint
            float T = (n > 0 && m < a.nckpt) ? a.ckpt_T[(long long)m * npix + pix] : 0.0f;
            for (int j = 0; j < n; ++j) {
                const float v = sample<true, INTERP>(s, r.P[0] + (long long)(k0 + j) * r.D[0],
                                                     r.P[1] + (long long)(k0 + j) * r.D[1],
                                                     r.P[2] + (long long)(k0 + j) * r.D[2], cc);
                vseg[j] = v;
                Tseg[j] = T;
                const float vv = isnan(v) ? a.lo : v;
                const float4 c = lut_eval(lut_s, normalise(vv, a.lo, a.inv_range));
                const float al = __saturatef(a.opacity_scale * c.w);
                T = T * (1.0f - al);
            }
            __syncwarp();
            // walk it backwards, the warp's lanes together (a shorter ray joins at its own end)
            for (int j = nw - 1; j >= 0; --j) {
                const bool on = j < n;
                const float v = on ? vseg[j] : a.lo;
                const bool nan = isnan(v);
                const float vv = nan ? a.lo : v;
                const float x = (vv - a.lo) * a.inv_range;
                const float vh = __saturatef(x);
                const float u = vh * 255.0f;
                const int i0 = min(__float2int_rd(u), 254);
                const float f = u - (float)i0;
                const float4 L0 = lut_s[i0], L1 = lut_s[i0 + 1];
                const float4 c = make_float4(lerp(L0.x, L1.x, f), lerp(L0.y, L1.y, f), lerp(L0.z, L1.z, f),
                                             lerp(L0.w, L1.w, f));
                const float alpha = a.opacity_scale * c.w;
                const float al = __saturatef(alpha);
                const float Tk = on ? Tseg[j] : 0.0f;
                const float gc = g.x * c.x + g.y * c.y + g.z * c.z;
                const float ga = gc * Tk - gT * Tk;
                const float wc = Tk * al;
                const float gcr = g.x * wc, gcg = g.y * wc, gcb = g.z * wc;
                if (on) gT = gT * (1.0f - al) + al * gc;
                const float galpha = (on && alpha >= 0.0f && alpha <= 1.0f) ? ga : 0.0f;
                // (an idle lane's c is the map at DATAMIN, which no sample need read: 0 * c.w may be NaN)
                if (on) gs = __fmaf_rn(galpha, c.w, gs);
                const float gca = galpha * a.opacity_scale;
                if (a.grad_lut != nullptr) {
                    // lanes on the same entry take turns (a lane without a sample has an entry of its own)
                    const unsigned same = __match_any_sync(0xffffffffu, on ? i0 : kLut + lane);
                    const int turn = on ? __popc(same & ((1u << lane) - 1u)) : 0;
                    const int turns = __reduce_max_sync(0xffffffffu, turn);
                    const float w0 = 1.0f - f;
                    for (int q = 0; q <= turns; ++q) {
                        if (on && turn == q) {
                            float4 q0 = mine[2 * i0], q1 = mine[2 * i0 + 1];
                            q0.x += w0 * gcr;
                            q0.y += w0 * gcg;
                            q0.z += w0 * gcb;
                            q0.w += w0 * gca;
                            q1.x += f * gcr;
                            q1.y += f * gcg;
                            q1.z += f * gcb;
                            q1.w += f * gca;
                            mine[2 * i0] = q0;
                            mine[2 * i0 + 1] = q1;
                        }
                        __syncwarp();
                    }
                }
                if (a.grad_vol != nullptr && on && !nan) {
                    const float gvh = 255.0f * (gcr * (L1.x - L0.x) + gcg * (L1.y - L0.y) + gcb * (L1.z - L0.z) +
                                                gca * (L1.w - L0.w));
                    const float gv = (x >= 0.0f && x <= 1.0f) ? gvh * a.inv_range : 0.0f;
                    if (gv != 0.0f) {
                        const long long X = r.P[0] + (long long)(k0 + j) * r.D[0];
                        const long long Y = r.P[1] + (long long)(k0 + j) * r.D[1];
                        const long long Z = r.P[2] + (long long)(k0 + j) * r.D[2];
                        if constexpr (INTERP == SHW_NEAREST) {
                            const int xi = clampi(fx_round(X), 0, s.nx - 1), yi = clampi(fx_round(Y), 0, s.ny - 1),
                                      zi = clampi(fx_round(Z), 0, s.nz - 1);
                            atomicAdd(a.grad_vol + ((Idx)zi * s.sz + (Idx)yi * s.sy + xi), gv);
                        } else {
                            cg.add(a.grad_vol, s.nx, s.ny, s.nz, X, Y, Z, gv);
                        }
                    }
                }
            }
        }
        if (INTERP == SHW_TRILINEAR && a.grad_vol != nullptr) cg.flush(a.grad_vol, s.nx, s.ny, s.nz);
        __syncwarp();
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gs += __shfl_xor_sync(0xffffffffu, gs, o);
        const float y = __fsub_rn(gs, gs_comp), z = __fadd_rn(gs_sum, y);
        gs_comp = isfinite(z) ? __fsub_rn(__fsub_rn(z, gs_sum), y) : 0.0f;  // (an infinite sum stays infinite)
        gs_sum = z;
    }
    // the scale gradient: one shared atomic per warp; the colour map's: the warps' sums of an
    // entry's own share and its lower neighbour's upper share; one global atomic per entry per CTA
    if (lane == 0) atomicAdd(&gs_s, gs_sum);
    __syncthreads();
    if (a.grad_lut != nullptr)
        for (int i = threadIdx.x; i < kLut * 4; i += blockDim.x) {
            const int e = i >> 2, ch = i & 3;
            float v = 0.0f;
            for (int w = 0; w < kBwdWarps; ++w) {
                const float *q = sums + w * kBwdSums + 8 * e + ch;
                v += q[0];
                if (e > 0) v += q[-4];
            }
            if (v != 0.0f) atomicAdd(a.grad_lut + i, v);
        }
    if (threadIdx.x == 0 && a.grad_scale != nullptr) atomicAdd(a.grad_scale, gs_s);
}

// One CTA per SM, at most one per tile.
template <int INTERP, class Idx>
static shw_status launch_backward(const SamplerF32<Idx> &s, const shw_camera &cam, const BackwardArgs &a,
                                  cudaStream_t st)
{
    auto kern = backward_kernel<INTERP, Idx>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBwdSmem) != cudaSuccess) {
        cudaGetLastError();
        return SHW_ECUDA;
    }
    const int nsm = sm_count();
    if (nsm <= 0) return SHW_ECUDA;
    const long long tiles = (long long)a.tiles_x * a.tiles_y;
    const unsigned grid = (unsigned)std::max(1LL, std::min((long long)nsm, tiles));
    kern<<<grid, kBwdThreads, kBwdSmem, st>>>(s, cam, a);
    return after_launch();
}

// from api.cu
bool valid_volume(const shw_volume *v);
bool valid_camera(const shw_camera *c);
bool valid_params(const shw_render_params *p, const shw_volume *v);
long long max_samples(const shw_volume *v, float step);
long long ckpt_count(const shw_volume *v, const shw_render_params *p);

}  // namespace shw

using namespace shw;

extern "C" shw_status shw_render_backward(const shw_volume *vol, const shw_camera *cam, const shw_render_params *p,
                                          const float *grad_rgba, const void *ckpt, size_t ckpt_bytes,
                                          float *grad_vol, float *grad_lut, float *grad_scale, void *stream)
{
    NvtxRange nvtx_range("shw_render_backward");
    if (!valid_volume(vol) || !valid_camera(cam) || !valid_params(p, vol)) return SHW_EINVAL;
    if (p->mode != SHW_COMPOSITE || !grad_rgba || !ckpt || !aligned(grad_rgba, 16) || !aligned(ckpt, 4))
        return SHW_EINVAL;
    if (p->ckpt_interval <= 0) return SHW_EINVAL;
    if (p->ckpt_interval > kMaxCkptInterval) return SHW_EUNSUPPORTED;
    if (vol->storage != SHW_F32) return SHW_EUNSUPPORTED;
    if (p->filter != SHW_FILTER_NONE || p->smooth != SHW_SMOOTH_NONE)
        return SHW_EUNSUPPORTED;  // the adjoint has no filter and no smoothing
    if ((grad_vol && !aligned(grad_vol, 4)) || (grad_lut && !aligned(grad_lut, 4)) ||
        (grad_scale && !aligned(grad_scale, 4)))
        return SHW_EINVAL;
    if (ckpt_bytes < shw_ckpt_bytes(vol, cam, p)) return SHW_ENOMEM;
    const long long npix = (long long)cam->width * cam->height;
    BackwardArgs a{};
    a.grad_rgba = reinterpret_cast<const float4 *>(grad_rgba);
    a.ckpt_K = static_cast<const int *>(ckpt);
    a.ckpt_T = reinterpret_cast<const float *>(static_cast<const char *>(ckpt) + npix * 4);
    a.grad_vol = grad_vol;
    a.grad_lut = grad_lut;
    a.grad_scale = grad_scale;
    a.lut = reinterpret_cast<const float4 *>(p->lut);
    a.width = cam->width;
    a.height = cam->height;
    a.nckpt = (int)ckpt_count(vol, p);
    a.ckpt_interval = p->ckpt_interval;
    a.nmax = (int)max_samples(vol, p->step);
    a.step = p->step;
    a.lo = p->lo;
    a.inv_range = 1.0f / (p->hi - p->lo);
    a.opacity_scale = p->opacity_scale;
    a.tiles_x = ceil_div(cam->width, 8);
    a.tiles_y = ceil_div(cam->height, 4);
    float cpx, cpy;
    project_centre(*cam, vol->nx, vol->ny, vol->nz, cpx, cpy);
    a.ctx = (int)fminf(fmaxf(cpx / 8.0f, 0.0f), (float)(a.tiles_x - 1));
    a.cty = (int)fminf(fmaxf(cpy / 4.0f, 0.0f), (float)(a.tiles_y - 1));
    cudaStream_t st = as_stream(stream);
    const float *v = static_cast<const float *>(vol->data);
    // 32-bit voxel offsets below 2^31 voxels
    if ((long long)vol->nx * vol->ny * vol->nz < (1LL << 31)) {
        const SamplerF32<int> s{v, vol->nx, vol->ny, vol->nz, vol->nx, vol->nx * vol->ny};
        return p->interp == SHW_NEAREST ? launch_backward<SHW_NEAREST, int>(s, *cam, a, st)
                                        : launch_backward<SHW_TRILINEAR, int>(s, *cam, a, st);
    }
    const SamplerF32<long long> s{v, vol->nx, vol->ny, vol->nz, (long long)vol->nx, (long long)vol->nx * vol->ny};
    return p->interp == SHW_NEAREST ? launch_backward<SHW_NEAREST, long long>(s, *cam, a, st)
                                    : launch_backward<SHW_TRILINEAR, long long>(s, *cam, a, st);
}
