// render_roll.cuh -- the rolling marcher: in-ray smoothing (Algorithms 8-9) from a ring of
// cube planes in shared memory.
//
// A smoothed sample is up to 25 trilinear fetches around one point.  Gathered from global
// memory (render_impl.cuh) each fetch is 8 loads whose 32 lanes lie in up to 24-32 different
// cache lines, and the L1 pipe bounds the kernel.  Here a CTA owns a 16 x 16 pixel tile and
// its rays advance together along the tile's major axis, a few planes of cells (a step) at a
// time, while one producer warp keeps the planes that the step's samples and taps can touch
// in shared memory:
//   - plane q of the ring holds the cells [oa, oa + wa) x [ob, ob + wb) of that plane, the
//     tile's footprint there widened by the taps' reach; every plane has its own origin, so
//     the window follows oblique rays and a plane is staged once per tile;
//   - a table of plane offsets (pb) turns (plane, a, b) into a shared-memory address;
//   - one tensor copy brings a plane, or one bulk copy per row when the cube's rows are no
//     16-byte multiple: row pitch and plane offset then keep every element's global and
//     shared address equal modulo 16 bytes.  The planes of x-major tiles are strided in
//     memory: the producer warp loads four of them together (16 bytes a row) and transposes
//     them into planes, which costs 4 % of the samples' own shared-memory traffic;
//   - the row pitch follows the view: the 32 rays of a warp cross a plane at about 8 x 4
//     points, and a pitch that puts consecutive rows on consecutive banks keeps them apart.
// Positions, cells, interpolation, the order of the taps and the transfer functions are the
// gather marcher's, so the results are bit-identical to it.  A sample whose cells are not
// all staged (a footprint wider than the ring's planes) reads global memory; staging decides
// the speed, never the result.
//
// What bounds it (512^3 cube, 1000 x 1000 MIP): with 9 taps per axis the shared-memory pipe (88 %
// of its cycles; 104 corner loads a sample at 2.2 wavefronts each, the conflicts of 32
// rays whose cells fall irregularly on 32 banks; 53.9 ms gathered from global memory, 11.5 ms
// here); with the box issue slots and latency (50 % of issue; 5.86 -> 2.32 ms).  On the way: one
// lateral range per step instead of one per cell (4 % of the samples in global memory) 16.8 ms;
// x-major planes as [z][y][4 x] boxes, unspread over the banks (3.9 wavefronts a load) 18.6 ms.
// All three major axes are in one kernel of 96 registers, which spills (208 to 384 bytes stored for
// the taps, 136 to 144 for the box), but not where the samples are: 1 of 1200 instructions of that
// render is a local load or store.
#pragma once

#include "render_slab.cuh"

namespace shw {

enum : int {
    kRollTaps = 0,  // per-axis taps (Algorithm 9)
    kRollBox = 1    // the box along the ray on the sample lattice (Algorithm 8, step 1/2)
};

constexpr int kRollBars = 4;        // headers and barriers: posts in flight
constexpr int kRollTable = 64;      // entries of the plane table (a power of two)
constexpr int kRollMaxSlots = 32;   // one producer lane per slot of a window
constexpr int kRollXG = 4;          // planes per slot of x-major tiles (loaded 16 bytes a row)
constexpr int kRollMinBlocks = 2;
constexpr int kRollBudget2 = 112 * 1024, kRollBudget1 = 226 * 1024;  // bytes of shared memory: two CTAs per SM, one

struct RollHdr {
    int type, tile;
    int major, dir;
    int m0, s_len;  // the step: cells [m0, m0 + s_len) along the major axis
    int pad[2];
};

// Staging geometry of one major axis.
struct RollGeom {
    int on;      // tiles may take this major axis
    int g;       // planes per slot
    int ns;      // slots of the ring
    int s;       // cells per step
    int depth;   // steps staged ahead
    int wa, wb;  // box extents along the lateral axes A and B
    int sb;      // floats between rows along B (along A: 1)
    int plane;   // floats per plane
    int slot;    // floats per slot (g planes)
};

struct RollArgs {
    const float *cube;
    unsigned *ctr, *err;
    int ntiles, polls;
    int halo;       // cells a tap reaches beyond its sample's cell, on each side
    int rows;       // 1: no tensor copies (ragged or unaligned cube): bulk copies of single rows
    int goff;       // rows: floats from the 16-byte boundary below the cube to the cube
    int smem_stage; // bytes of the plane ring
    float xbias;    // (roll_rays)
    int box_mask;   // box: entries of a ray's ring of raw samples, less one (a power of two)
    RollGeom geo[3];
};

// The tensor maps of one plane: y-major, z-major.
struct RollMaps {
    CUtensorMap m[2];
};

// Compositing ends a tile when all its rays have stopped.  dead[t % 4]: how many consumer warps need no
// further step of the CTA's t-th tile, each told once; a hint, so plain shared-memory accesses do.
// (Told at every stage by the tile's number, as the staged marcher does, the taps' compositing took 3
// to 15 % longer, and with any report the other modes, whose rays end with the cube, 1 to 4 %.)
constexpr int kDeadSlots = 4;  // a slot is zeroed when the tiles before the last have been consumed

struct RollShared {
    RollHdr hdr[kRollBars];
    uint64_t full[kRollBars], empty[kRollBars];
    int pb[kRollTable];                   // plane q: stage index of its element (a, b) = (0, 0)
    int oa[kRollTable], ob[kRollTable];   // slot c: origin of its box
    // cell c of a step: the lateral cells [x, x + y) along A and [z, z + w) along B whose
    // corners and taps the planes of its window all hold
    int4 range[kRollTable];
    int dead[kDeadSlots];
    int quit;
    int pad[3];
};

// Lateral axes of major axis M: A (contiguous in the stage) and B.
template <int M>
struct RollAxes {
    static constexpr int A = M == 0 ? 1 : 0;
    static constexpr int B = M == 2 ? 1 : 2;
};

// The major axis: the one the tile's rays advance along fastest, so that lateral slopes stay
// small and the footprint of a plane with them; x only when it is `xbias` times faster than
// the others.
__host__ __device__ __forceinline__ TileRays roll_rays(const shw_camera &c, int px0, int py0, const int on[3],
                                                       float xbias)
{
    TileRays t;
    for (int i = 0; i < 4; ++i)
        corner_ray(c, px0 + (i & 1) * (kSlabTW - 1), py0 + (i >> 1) * (kSlabTH - 1), t.o[i], t.u[i]);
    float best = -1.0f;
    t.major = 2;
    t.dir = 1;
    for (int k = 0; k < 3; ++k) {
        const float s = t.u[0][k] + t.u[1][k] + t.u[2][k] + t.u[3][k], f = fabsf(s) / (k == 0 ? xbias : 1.0f);
        if (on[k] && f > best) {
            best = f;
            t.major = k;
            t.dir = s > 0.0f ? 1 : -1;
        }
    }
    return t;
}

// Lateral positions [lo, hi] on axis AX of the tile's rays between planes m0 and m1.
template <int M, int AX>
__host__ __device__ __forceinline__ void lateral_pos(const TileLines<M> &t, float m0, float m1, float &lo, float &hi)
{
    lo = INFINITY;
    hi = -INFINITY;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float p0 = t.B[i][AX] * m0 + t.A[i][AX], p1 = t.B[i][AX] * m1 + t.A[i][AX];
        lo = fminf(lo, fminf(p0, p1));
        hi = fmaxf(hi, fmaxf(p0, p1));
    }
    const float eps = 0.02f + 1e-5f * fmaxf(fabsf(lo), fabsf(hi));
    lo -= eps;
    hi += eps;
}

// Elements [lo, hi] along axis AX that planes [q0, q1] must hold: the corners of the samples
// next to them widened by the taps' reach H, and the corners of the samples whose taps along
// the major axis reach them; clipped to the cube.
template <int M, int AX>
__host__ __device__ __forceinline__ void plane_extent(const TileLines<M> &t, int q0, int q1, int H, int n, int &lo,
                                                      int &hi)
{
    float l0, h0, l1, h1;
    lateral_pos<M, AX>(t, (float)(q0 - 1), (float)(q1 + 1), l0, h0);
    lateral_pos<M, AX>(t, (float)(q0 - 1 - H), (float)(q1 + 1 + H), l1, h1);
    const float l = fminf(l0 - (float)H, l1), h = fmaxf(h0 + (float)H, h1);
    lo = (int)floorf(fminf(fmaxf(l, 0.0f), (float)n));
    hi = (int)floorf(fmaxf(fminf(h + 1.0f, (float)(n - 1)), -1.0f));
}

// ---- producer -------------------------------------------------------------------------

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// untiled bulk copy: both addresses 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

struct RollRing {
    RollShared &sh;
    const RollArgs &ra;
    int posts = 0, drained = 0;  // posts made; posts known to be consumed by every warp
    __device__ __forceinline__ bool drain_to(int p)
    {
        for (; drained <= p; ++drained)
            if (!slab_wait(&sh.empty[drained % kRollBars], (uint32_t)((drained / kRollBars) & 1), &sh.quit, ra.err,
                           ra.polls))
                return false;
        return true;
    }
    __device__ __forceinline__ bool post_plain(int type, int tile, int seq = 0)
    {
        if (!drain_to(posts - kRollBars)) return false;
        const int st = posts % kRollBars;
        if ((threadIdx.x & 31) == 0) {
            RollHdr h{};
            h.type = type;
            h.tile = tile;
            h.m0 = seq % kDeadSlots;  // (a tile's start: its entry of sh.dead)
            if (type == kStageTile) sh.dead[seq % kDeadSlots] = 0;
            sh.hdr[st] = h;
            mbar_arrive(&sh.full[st]);
        }
        __syncwarp();
        ++posts;
        return true;
    }
};

__device__ __forceinline__ int floor_div(int a, int b)
{
    const int q = a / b;
    return q * b > a ? q - 1 : q;
}

// One row's elements [x, x + len) of the cube (len clipped to the row) from row start index
// `row` into the stage at element index `at` of x: 16-byte pieces by a bulk copy, and at the
// two ends of the whole cube, where a piece would leave it, single elements.  lo, hi: the slot.
__device__ __forceinline__ void roll_row(const RollArgs &ra, float *stage, long long nvox, long long row, int x, int len,
                                         int at, int lo, int hi, uint64_t *bar)
{
    const long long g0 = ra.goff + row + x, g1 = g0 + len;  // floats from the 16-byte boundary
    const float *base = ra.cube - ra.goff;
    long long c0 = g0 & ~3LL, c1 = (g1 + 3) & ~3LL;
    if constexpr (kChecked) {  // whole pieces inside the slot, on 16-byte boundaries there too
        const bool ok = at + (int)(c0 - g0) >= lo && at + (int)(c1 - g0) <= hi && (at + (int)(c0 - g0)) % 4 == 0;
        SHW_CHECK(ok);
        if (!ok) return;
    }
    bool wrote = false;
    if (c0 < ra.goff) {
        c0 += 4;
        for (long long g = g0; g < min(c0, g1); ++g) stage[at + (int)(g - g0)] = __ldg(base + g);
        wrote = true;
    }
    if (c1 > ra.goff + nvox) {
        c1 -= 4;
        for (long long g = max(c1, g0); g < g1; ++g) stage[at + (int)(g - g0)] = __ldg(base + g);
        wrote = true;
    }
    if (c1 > c0) {
        const uint32_t bytes = (uint32_t)(c1 - c0) * 4u;
        mbar_expect_tx(bar, bytes);
        bulk_load(stage + at + (int)(c0 - g0), base + c0, bytes, bar);
    }
    if (wrote) fence_proxy_async();  // a later bulk copy writes the same bytes
}

// Planes q0 .. q0+3 of an x-major tile: every (y, z) row of the box holds four consecutive x,
// loaded together by one lane and written to the four planes.
__device__ __forceinline__ void roll_xplanes(const RollArgs &ra, const RollGeom &G, float *slot, const int n[3], int q0,
                                             int y0, int z0)
{
    constexpr int U = 8;  // loads in flight per lane
    const int lane = threadIdx.x & 31;
    const int wa = min(G.wa, n[1] - y0), total = wa * min(G.wb, n[2] - z0);
    const float inv = 1.0f / (float)wa;
    for (int i0 = lane; i0 < total; i0 += 32 * U) {
        float4 v[U];
        int at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + 32 * u;
            at[u] = -1;
            if (i < total) {
                const int b = (int)(((float)i + 0.5f) * inv), a = i - b * wa;  // (exact: i < 2^16)
                at[u] = b * G.sb + a;
                const float *p = ra.cube + ((size_t)(z0 + b) * n[1] + (y0 + a)) * n[0] + q0;
                if (!ra.rows) {
                    v[u] = __ldg(reinterpret_cast<const float4 *>(p));
                } else {
                    v[u].x = __ldg(p);
                    v[u].y = q0 + 1 < n[0] ? __ldg(p + 1) : 0.0f;
                    v[u].z = q0 + 2 < n[0] ? __ldg(p + 2) : 0.0f;
                    v[u].w = q0 + 3 < n[0] ? __ldg(p + 3) : 0.0f;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (at[u] >= 0) {
                if constexpr (kChecked) {  // inside the plane (the slot holds kRollXG of them)
                    SHW_CHECK(at[u] < G.plane);
                    if (at[u] >= G.plane) continue;
                }
                slot[at[u]] = v[u].x;
                slot[at[u] + G.plane] = v[u].y;
                slot[at[u] + 2 * G.plane] = v[u].z;
                slot[at[u] + 3 * G.plane] = v[u].w;
            }
    }
}

template <int M, bool EARLY>
__device__ __forceinline__ bool roll_produce(const TileRays &r, bool persp, const CUtensorMap *map,
                                             const RenderArgs &a, const RollArgs &ra, int tile, int seq, float *stage,
                                             RollRing &ring)
{
    using AX = RollAxes<M>;
    TileLines<M> L;
    if (!tile_lines<M>(r, L)) return true;  // no steps: the consumers read global memory
    const RollGeom &G = ra.geo[M];
    RollShared &sh = ring.sh;
    const int lane = threadIdx.x & 31, dir = r.dir, H = ra.halo;
    const int n[3] = {a.nx, a.ny, a.nz};
    const int n_m = n[M], n_a = n[AX::A], n_b = n[AX::B];
    const int g = M == 0 ? kRollXG : 1, s = G.s;
    int lo_c = -1, hi_c = n_m - 1;
    if (persp) {  // every sample lies beyond the eye
        const int e = (int)fminf(fmaxf(floorf(r.o[0][M]), -1.0f), (float)n_m);
        if (dir > 0)
            lo_c = max(lo_c, e);
        else
            hi_c = min(hi_c, e);
    }
    // the cells [first, last] at which the tile's rays are inside the cube
    int first = n_m, last = -2;
    for (int c = lo_c; c <= hi_c; c += 32) {
        const int cc = c + lane;
        float al, ah, bl, bh;
        lateral_pos<M, AX::A>(L, (float)cc, (float)(cc + 1), al, ah);
        lateral_pos<M, AX::B>(L, (float)cc, (float)(cc + 1), bl, bh);
        const bool in = cc <= hi_c && ah >= -0.5f && al <= (float)n_a - 0.5f && bh >= -0.5f && bl <= (float)n_b - 0.5f;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (m) {
            first = min(first, c + __ffs(m) - 1);
            last = max(last, c + 31 - __clz(m));
        }
    }
    if (first > last) return true;
    const int before = ring.posts - 2;  // the last post before this tile's start: it may read the ring
    bool fresh = true;
    int have_lo = 0, have_hi = -1;  // slots staged
    for (int m0 = floor_div(dir > 0 ? first : last, s) * s; dir > 0 ? m0 <= last : m0 + s > first; m0 += dir * s) {
        if (EARLY) {  // every ray of the tile has ended
            const int d = *const_cast<const volatile int *>(sh.dead + seq % kDeadSlots);
            if (__shfl_sync(0xffffffffu, d, 0) == kSlabWarps) break;
        }
        const int plo = max(m0 - H, 0), phi = min(m0 + s + H, n_m - 1);
        const int slo = plo / g, shi = phi / g;
        const int c0 = fresh ? slo : (dir > 0 ? have_hi + 1 : slo), c1 = fresh ? shi : (dir > 0 ? shi : have_lo - 1);
        // the slots overwritten now were last read `depth` steps ago (or by the tile before)
        if (!ring.drain_to(max(ring.posts - kRollBars, fresh ? before : ring.posts - 1 - G.depth))) return false;
        const int st = ring.posts % kRollBars;
        uint64_t *bar = &sh.full[st];
        const int cnt = max(c1 - c0 + 1, 0);
        int oa = 0, ob = 0;
        if (lane < cnt) {
            const int c = c0 + lane, q0 = c * g;
            int lo, hi;
            plane_extent<M, AX::A>(L, q0, q0 + g - 1, H, n_a, lo, hi);
            if (hi - lo + 1 > G.wa) lo += (hi - lo + 1 - G.wa) >> 1;
            oa = min(max(lo, 0), n_a - 1);
            if (M != 0 && !ra.rows) oa &= ~3;  // a tensor copy's x start: 16 bytes
            plane_extent<M, AX::B>(L, q0, q0 + g - 1, H, n_b, lo, hi);
            if (hi - lo + 1 > G.wb) lo += (hi - lo + 1 - G.wb) >> 1;
            ob = min(max(lo, 0), n_b - 1);
            sh.oa[c & (kRollTable - 1)] = oa;
            sh.ob[c & (kRollTable - 1)] = ob;
            int pb = (c % G.ns) * G.slot - oa - ob * G.sb;
            if (M != 0 && ra.rows) {
                // equal global and shared addresses modulo 16 bytes (the row pitch agrees already)
                const int want = ra.goff + (M == 2 ? (c * n[1] & 3) * (n[0] & 3) : (c & 3) * (n[0] & 3));
                pb += 4 + ((want - pb) & 3);
            }
#pragma unroll
            for (int j = 0; j < g; ++j) sh.pb[(q0 + j) & (kRollTable - 1)] = pb + j * G.plane;
        }
        __syncwarp();
        if constexpr (M == 0) {
            for (int c = c0; c <= c1; ++c)
                roll_xplanes(ra, G, stage + (c % G.ns) * G.slot, n, c * g, sh.oa[c & (kRollTable - 1)],
                             sh.ob[c & (kRollTable - 1)]);
            fence_proxy_async();  // a later copy may write the same bytes
        } else if (!ra.rows) {
            if (lane < cnt) {
                const int c = c0 + lane;
                float *dst = stage + (size_t)(c % G.ns) * G.slot;
                if (tma_dst_ok(dst, ra.err)) {  // always: slots are 128-byte multiples
                    mbar_expect_tx(bar, (uint32_t)(G.wa * G.wb * 4));
                    if constexpr (M == 1)
                        tma_load_3d(dst, map, oa, c, ob, bar);
                    else
                        tma_load_3d(dst, map, oa, ob, c, bar);
                }
            }
        } else {
            const long long nvox = (long long)n[0] * n[1] * n[2];
            for (int i = lane; i < cnt * G.wb; i += 32) {
                const int c = c0 + i / G.wb, ci = c & (kRollTable - 1);
                const int b = sh.ob[ci] + i % G.wb, x = sh.oa[ci];
                if (b >= n_b) continue;
                const long long row = M == 2 ? ((long long)c * n[1] + b) * n[0] : ((long long)b * n[1] + c) * n[0];
                const int lo = (c % G.ns) * G.slot;
                roll_row(ra, stage, nvox, row, x, min(G.wa, n_a - x), sh.pb[ci] + b * G.sb + x, lo, lo + G.slot, bar);
            }
        }
        if (lane < s) {
            const int cell = m0 + lane;
            const int w0 = max(cell - H, 0) / g, w1 = min(cell + 1 + H, n_m - 1) / g;
            int alo = -1, ahi = n_a - 1, blo = -1, bhi = n_b - 1;
            for (int c = w0; c <= w1; ++c) {
                const int ci = c & (kRollTable - 1), q0 = c * g;
                const bool own = q0 + g - 1 >= cell && q0 <= cell + 1;  // holds the cell's own planes
                const int h = own ? H : 0, x = sh.oa[ci], y = sh.ob[ci];
                if (x > 0) alo = max(alo, x + h);
                if (x + G.wa < n_a) ahi = min(ahi, x + G.wa - 2 - h);
                if (y > 0) blo = max(blo, y + h);
                if (y + G.wb < n_b) bhi = min(bhi, y + G.wb - 2 - h);
            }
            sh.range[cell & (kRollTable - 1)] = make_int4(alo, max(ahi - alo + 1, 0), blo, max(bhi - blo + 1, 0));
        }
        if (lane == 0) {
            RollHdr h;
            h.type = kStageSlab;
            h.tile = tile;
            h.major = M;
            h.dir = dir;
            h.m0 = m0;
            h.s_len = s;
            sh.hdr[st] = h;
        }
        __syncwarp();  // every lane's expected bytes and table entries come before the arrival
        if (lane == 0) mbar_arrive(bar);
        ++ring.posts;
        fresh = false;
        have_lo = slo;
        have_hi = shi;
    }
    return true;
}

template <bool EARLY>
__device__ __forceinline__ void roll_producer(const CUtensorMap *maps, const shw_camera &cam, const RenderArgs &a,
                                              const RollArgs &ra, float *stage, RollShared &sh)
{
    const int lane = threadIdx.x & 31;
    RollRing ring{sh, ra};
    const int on[3] = {ra.geo[0].on, ra.geo[1].on, ra.geo[2].on};
    bool ok = true;
    for (int seq = 0; ok; ++seq) {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(ra.ctr, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= (unsigned)ra.ntiles) {
            ring.post_plain(kStageExit, 0);
            break;
        }
        if (!ring.post_plain(kStageTile, (int)t, seq)) break;
        int tx, ty;
        slab_tile((int)t, a, tx, ty);
        const TileRays r = roll_rays(cam, tx * kSlabTW, ty * kSlabTH, on, ra.xbias);
        const bool persp = !cam.ortho;
        if (r.major == 0)
            ok = roll_produce<0, EARLY>(r, persp, nullptr, a, ra, (int)t, seq, stage, ring);
        else if (r.major == 1)
            ok = roll_produce<1, EARLY>(r, persp, &maps[0], a, ra, (int)t, seq, stage, ring);
        else
            ok = roll_produce<2, EARLY>(r, persp, &maps[1], a, ra, (int)t, seq, stage, ring);
        if (ok) ok = ring.post_plain(kStageTileEnd, (int)t);
    }
    // no exit while a copy into this CTA's shared memory is in flight: wait (bounded) for the
    // last posts
    if (lane == 0) {
        for (int i = max(0, ring.posts - kRollBars); i < ring.posts; ++i)
            for (int it = 0; it < ra.polls && !mbar_try_wait_sleep(&sh.full[i % kRollBars],
                                                                   (uint32_t)((i / kRollBars) & 1), kSlabSleepNs);
                 ++it) {
            }
    }
    __syncwarp();
}

// ---- consumer -------------------------------------------------------------------------

// One axis of a fetch: the two corner indexes and the weight.  CLAMP: indexes clamp to the
// edge voxel (the gather marcher's rule); without it the cell lies inside the cube.
template <bool CLAMP>
__device__ __forceinline__ void roll_axis(long long p, int n, int &i0, int &i1, float &f)
{
    const int c = cell_of<CLAMP>(p, n);
    i0 = CLAMP ? max(c, 0) : c;
    i1 = CLAMP ? min(c + 1, n - 1) : c + 1;
    f = fx_frac(p);
}

// The value at (PA, PB, PM): the trilinear sample, and with TAPS its chain of taps along x,
// then y, then z (smoothed_sample's order and arithmetic), from the staged planes.
template <int M, bool CLAMP, bool TAPS>
__device__ __forceinline__ float roll_value(const float *stage, const int *pbt, int sb, int lim, const int n[3],
                                            const long long P[3], const RenderArgs &a)
{
    using AX = RollAxes<M>;
    constexpr int A = AX::A, B = AX::B;
    int i0[3], i1[3];
    float f[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) roll_axis<CLAMP>(P[k], n[k], i0[k], i1[k], f[k]);
    auto plane = [&](int q) { return pbt[q & (kRollTable - 1)]; };
    // corners c[x + 2 y + 4 z] from plane offsets m0, m1 and in-plane offsets
    auto fetch8 = [&](int m0, int m1, int a0, int a1, int b0, int b1, float fx, float fy, float fz) {
        if constexpr (kChecked) {  // every corner lies in the stage (lim floats)
            const int l0 = min(min(m0, m1) + b0, min(m0, m1) + b1) + a0, l1 = max(m0, m1) + max(b0, b1) + a1;
            const bool ok = l0 >= 0 && l1 < lim;
            SHW_CHECK(ok);
            if (!ok) m0 = m1 = a0 = a1 = b0 = b1 = 0;
        }
        const float *p00 = stage + (m0 + b0), *p01 = stage + (m0 + b1), *p10 = stage + (m1 + b0),
                    *p11 = stage + (m1 + b1);
        float c[8];
#define SHW_C(m, b, x, ptr, off) c[((m) << M) | ((b) << B) | ((x) << A)] = (ptr)[off]
        SHW_C(0, 0, 0, p00, a0);
        SHW_C(0, 0, 1, p00, a1);
        SHW_C(0, 1, 0, p01, a0);
        SHW_C(0, 1, 1, p01, a1);
        SHW_C(1, 0, 0, p10, a0);
        SHW_C(1, 0, 1, p10, a1);
        SHW_C(1, 1, 0, p11, a0);
        SHW_C(1, 1, 1, p11, a1);
#undef SHW_C
        return trilerp(c, fx, fy, fz);
    };
    const int m0 = plane(i0[M]), m1 = plane(i1[M]);
    const int a0 = i0[A], a1 = CLAMP ? i1[A] : a0 + 1;
    const int b0 = i0[B] * sb, b1 = CLAMP ? i1[B] * sb : b0 + sb;
    float v = fetch8(m0, m1, a0, a1, b0, b1, f[0], f[1], f[2]);
    if constexpr (TAPS) {
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            float out = v * a.smooth_c0;
            for (int j = 0; j < a.smooth_n; ++j) {
                const long long off = a.smooth_off[j];
                const float w = a.smooth_w[j];
#pragma unroll
                for (int sgn = 0; sgn < 2; ++sgn) {
                    int t0, t1;
                    float tf;
                    roll_axis<CLAMP>(sgn == 0 ? P[ax] + off : P[ax] - off, n[ax], t0, t1, tf);
                    float t;
                    if (ax == M) {
                        t = fetch8(plane(t0), plane(t1), a0, a1, b0, b1, M == 0 ? tf : f[0], M == 1 ? tf : f[1],
                                   M == 2 ? tf : f[2]);
                    } else if (ax == A) {
                        t = fetch8(m0, m1, t0, CLAMP ? t1 : t0 + 1, b0, b1, A == 0 ? tf : f[0], A == 1 ? tf : f[1], f[2]);
                    } else {
                        const int u0 = t0 * sb, u1 = CLAMP ? t1 * sb : u0 + sb;
                        t = fetch8(m0, m1, a0, a1, u0, u1, f[0], B == 1 ? tf : f[1], B == 2 ? tf : f[2]);
                    }
                    out = __fmaf_rn(t, w, out);
                }
            }
            v = out;
        }
    }
    return v;
}

// The same value from global memory (a sample that the ring does not hold).  Not inlined:
// rare, and its registers would add to the staged path's.
template <bool TAPS, class S>
__device__ __noinline__ float roll_global(const S &s, long long X, long long Y, long long Z, const RenderArgs &a)
{
    CellCache cc;
    if constexpr (TAPS) {
        const long long U[3] = {0, 0, 0};
        return smoothed_sample<SHW_TRILINEAR>(s, X, Y, Z, U, a, cc);
    } else {
        return s.trilinear(X, Y, Z);
    }
}

// One ray's march: its raw samples arrive in order, k = 0 .. N-1 (taps) or, for the box,
// k = -2 arm .. N-1 + 2 arm.
template <int MODE, int KIND>
struct RollMarch {
    using St = typename StateOf<MODE>::type;
    St st;
    long long X, Y, Z;  // position of sample k
    int k, kend;        // next sample, end of the samples
    int ka, kb;         // samples whose cells and taps need no clamping
    int done;           // samples processed
    float s0, s1;       // box: running sums of the classes of the next sample and the one after

    // Take value v of sample k; true if the transfer function stopped the ray.
    __device__ __forceinline__ bool take(const RenderArgs &a, float v, float *ring, int mask)
    {
        if constexpr (KIND == kRollTaps) {
            v = filter_value(isnan(v) ? a.lo : v, a);
            v = isnan(v) ? a.lo : v;  // a NaN sample counts as DATAMIN
            done = k + 1;
            return st.update(v, k);
        } else {
            // march_box_lattice's recurrence (M = 2), its raw samples kept in the ray's ring
            const int arm = a.smooth_n, j = k, c = j - 2 * arm;
            auto at = [&](int i) -> float & { return ring[(i & mask) * (32 * kSlabWarps)]; };
            at(j) = v;
            if (c < 0) return false;
            float t = 0.0f;
            bool direct = (c >> 1) % SHW_BOX_RESUM == 0;
            if (!direct) {
                t = s0 + v - at(j - (4 * arm + 2));
                direct = !isfinite(t);
            }
            if (direct) {  // the definition's order: the sample, then the pairs +-i
                t = at(c);
                for (int i = 1; i <= arm; ++i) {
                    t += at(c + 2 * i);
                    t += at(c - 2 * i);
                }
            }
            s0 = s1;
            s1 = t;
            float w = t * a.smooth_c0;
            w = filter_value(isnan(w) ? a.lo : w, a);
            w = isnan(w) ? a.lo : w;
            done = c + 1;
            return st.update(w, c);
        }
    }
};

// The samples of one ray in the step of h; true if the transfer function stopped the ray.
template <int M, int MODE, int KIND, class S>
__device__ __forceinline__ bool roll_step(const S &s, const RenderArgs &a, RollMarch<MODE, KIND> &q, long long DX,
                                          long long DY, long long DZ, const RollHdr &h, const float *stage,
                                          const RollShared &sh, int sb, int lim, float *ring, int mask)
{
    using AX = RollAxes<M>;
    constexpr bool TAPS = KIND == kRollTaps;
    const int n[3] = {s.nx, s.ny, s.nz};
    for (;;) {
        // samples that need no clamping, as long as the step holds them
        const int kin = min(q.kb, q.kend);
        while (q.k >= q.ka && q.k < kin) {
            const long long P[3] = {q.X, q.Y, q.Z};
            const int cm = fx_cell(P[M]);
            if ((unsigned)(cm - h.m0) >= (unsigned)h.s_len) break;
            const int4 in = sh.range[cm & (kRollTable - 1)];
            if ((unsigned)(fx_cell(P[AX::A]) - in.x) >= (unsigned)in.y ||
                (unsigned)(fx_cell(P[AX::B]) - in.z) >= (unsigned)in.w)
                break;
            const bool stop = q.take(a, roll_value<M, false, TAPS>(stage, sh.pb, sb, lim, n, P, a), ring, mask);
            q.X += DX;
            q.Y += DY;
            q.Z += DZ;
            ++q.k;
            if (stop) return true;
        }
        if (q.k >= q.kend) return false;
        // one sample at the cube's faces, outside the staged boxes, or of a later step
        const long long P[3] = {q.X, q.Y, q.Z};
        const int cm = clampi(fx_cell(P[M]), -1, n[M] - 1), rel = h.dir > 0 ? cm - h.m0 : h.m0 + h.s_len - 1 - cm;
        if (rel >= h.s_len) return false;  // a later step's
        const int ca = clampi(fx_cell(P[AX::A]), -1, n[AX::A] - 1), cb = clampi(fx_cell(P[AX::B]), -1, n[AX::B] - 1);
        const int4 in = sh.range[cm & (kRollTable - 1)];
        float v;
        if (rel >= 0 && (unsigned)(ca - in.x) < (unsigned)in.y && (unsigned)(cb - in.z) < (unsigned)in.w)
            v = roll_value<M, true, TAPS>(stage, sh.pb, sb, lim, n, P, a);
        else
            v = roll_global<TAPS>(s, q.X, q.Y, q.Z, a);
        const bool stop = q.take(a, v, ring, mask);
        q.X += DX;
        q.Y += DY;
        q.Z += DZ;
        ++q.k;
        if (stop) return true;
    }
}

template <int MODE, int KIND, class S>
__device__ __forceinline__ void roll_consumer(const S &s, const shw_camera &cam, const RenderArgs &a,
                                              const RollArgs &ra, const float *stage, RollShared &sh, float *rings)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int lx = (warp & 1) * 8 + (lane & 7), ly = (warp >> 1) * 4 + (lane >> 3);
    volatile int *quit = &sh.quit;
    float *ring = rings + threadIdx.x;
    RollMarch<MODE, KIND> q;
    RayFx r;
    long long pix = 0;
    int N = 0;
    bool has = false, live = false;
    int slot = -1;  // compositing: the tile's entry of sh.dead, -1 once told
    for (int posts = 0;; ++posts) {
        const int si = posts % kRollBars;
        if (!slab_wait(&sh.full[si], (uint32_t)((posts / kRollBars) & 1), quit, ra.err, ra.polls)) return;
        const RollHdr h = sh.hdr[si];
        if (h.type == kStageExit) return;
        if (h.type == kStageTile) {
            int tx, ty;
            slab_tile(h.tile, a, tx, ty);
            const int px = tx * kSlabTW + lx, py = ty * kSlabTH + ly;
            has = px < a.width && py < a.height;
            pix = (long long)py * a.width + px;
            const bool hit = has && !quick_miss(cam, px, py, s.nx, s.ny, s.nz) &&
                             setup_ray(cam, px, py, s.nx, s.ny, s.nz, a.step, r);
            N = hit ? min(r.N, a.nmax) : 0;
            slot = h.m0;
            live = N > 0;
            q.st = typename RollMarch<MODE, KIND>::St{};
            q.done = 0;
            if (live) {
                // samples whose cells lie in [H, n - 2 - H] on every axis
                const int H = ra.halo;
                RayFx in = r;
                for (int k = 0; k < 3; ++k) in.P[k] -= (long long)H << 32;
                interior_range(in, s.nx - 2 * H, s.ny - 2 * H, s.nz - 2 * H, N, q.ka, q.kb);
                init_ray_state<MODE, SHW_TRILINEAR>(q.st, s, a, r, pix, a.lut);
                const int lead = KIND == kRollBox ? 2 * a.smooth_n : 0;  // raw samples before the first
                q.k = -lead;
                q.kend = N + lead;
                q.X = r.P[0] - (long long)lead * r.D[0];
                q.Y = r.P[1] - (long long)lead * r.D[1];
                q.Z = r.P[2] - (long long)lead * r.D[2];
                q.s0 = q.s1 = 0.0f;
            }
        } else if (h.type == kStageSlab) {
            if (live) {
                bool stop;
                if (h.major == 0)
                    stop = roll_step<0, MODE, KIND>(s, a, q, r.D[0], r.D[1], r.D[2], h, stage, sh, ra.geo[0].sb,
                                                    ra.smem_stage / 4, ring, ra.box_mask);
                else if (h.major == 1)
                    stop = roll_step<1, MODE, KIND>(s, a, q, r.D[0], r.D[1], r.D[2], h, stage, sh, ra.geo[1].sb,
                                                    ra.smem_stage / 4, ring, ra.box_mask);
                else
                    stop = roll_step<2, MODE, KIND>(s, a, q, r.D[0], r.D[1], r.D[2], h, stage, sh, ra.geo[2].sb,
                                                    ra.smem_stage / 4, ring, ra.box_mask);
                if (stop) live = false;
            }
        } else if (has) {  // the tile's end
            if (live) {    // samples that no step held
                while (q.k < q.kend) {
                    const float v = roll_global<KIND == kRollTaps>(s, q.X, q.Y, q.Z, a);
                    const bool stop = q.take(a, v, ring, ra.box_mask);
                    q.X += r.D[0];
                    q.Y += r.D[1];
                    q.Z += r.D[2];
                    ++q.k;
                    if (stop) break;
                }
                live = false;
            }
            if (N <= 0) r.P[0] = r.P[1] = r.P[2] = r.D[0] = r.D[1] = r.D[2] = 0;
            emit_ray<MODE, SHW_TRILINEAR>(a, pix, N, r.P, r.D, q.st, q.done);
            has = false;
        }
        __syncwarp();
        if constexpr (is_composite<MODE>)
            if (h.type != kStageTileEnd && slot >= 0 && !__any_sync(0xffffffffu, live && q.k < q.kend)) {
                if (lane == 0) atomicAdd(sh.dead + slot, 1);
                slot = -1;
            }
        if (lane == 0) mbar_arrive(&sh.empty[si]);
    }
}

template <int MODE, int KIND, class S>
__global__ void __launch_bounds__(kSlabThreads, kRollMinBlocks)
    roll_kernel(const __grid_constant__ RollMaps maps, const __grid_constant__ S s,
                const __grid_constant__ shw_camera cam, const __grid_constant__ RenderArgs a,
                const __grid_constant__ RollArgs ra)
{
    extern __shared__ __align__(128) unsigned char roll_smem[];
    float *stage = reinterpret_cast<float *>(roll_smem);
    RollShared &sh = *reinterpret_cast<RollShared *>(roll_smem + ra.smem_stage);
    float *rings = reinterpret_cast<float *>(roll_smem + ra.smem_stage + sizeof(RollShared));
    if (threadIdx.x == 0) {
        for (int i = 0; i < kRollBars; ++i) {
            mbar_init(&sh.full[i], 1);
            mbar_init(&sh.empty[i], kSlabWarps);
        }
        sh.quit = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if ((threadIdx.x >> 5) == kSlabWarps)
        roll_producer<is_composite<MODE>>(maps.m, cam, a, ra, stage, sh);
    else
        roll_consumer<MODE, KIND>(s, cam, a, ra, stage, sh, rings);
}

// ---- host -----------------------------------------------------------------------------

// Largest plane extents of major axis M over sampled tiles and planes.
template <int M>
inline void roll_extent(const TileRays &r, const int n[3], int H, int g, int &wa, int &wb)
{
    using AX = RollAxes<M>;
    TileLines<M> L;
    if (!tile_lines<M>(r, L)) return;
    for (int i = 0; i <= 4; ++i) {
        const int q = (int)((long long)(n[M] - 1) * i / 4) / g * g;
        int al, ah, bl, bh;
        plane_extent<M, AX::A>(L, q, q + g - 1, H, n[AX::A], al, ah);
        plane_extent<M, AX::B>(L, q, q + g - 1, H, n[AX::B], bl, bh);
        if (al > ah || bl > bh) continue;  // the tile passes the cube here
        wa = std::max(wa, ah - al + 1);
        wb = std::max(wb, bh - bl + 1);
    }
}

// Slots that the windows of a step and of the `depth` steps staged ahead of it span, for the
// step start that spans most (steps start at multiples of s, slots at multiples of g).
inline int roll_slots(int H, int s, int g, int depth)
{
    const int back = (H + g - 1) / g + 1;  // (keeps the divisions below on positive numbers)
    int most = 0;
    for (int m = 0; m < s * g; m += s)
        most = std::max(most, (m + s + H + depth * s + back * g) / g - (m - H + back * g) / g + 1);
    return most;
}

// Lateral extent along A of a warp's 8 x 4 pixels where their rays cross one plane (the
// centre tile, at the cube's centre).
template <int M>
inline float roll_warp_extent(const TileRays &r, const int n[3])
{
    TileLines<M> L;
    if (!tile_lines<M>(r, L)) return 8.0f;
    const float m = 0.5f * (float)(n[M] - 1);
    float p[4];
    for (int i = 0; i < 4; ++i) p[i] = L.B[i][RollAxes<M>::A] * m + L.A[i][RollAxes<M>::A];
    return fabsf(p[1] - p[0]) * (7.0f / (kSlabTW - 1)) + fabsf(p[2] - p[0]) * (3.0f / (kSlabTH - 1));
}

// The smallest row pitch >= w, congruent to `mod4` modulo 4, that puts neighbouring rows `ext`
// banks or so apart: the rows of a warp's footprint, ext floats long, then miss each other.
inline int roll_pitch(int w, float ext, int mod4)
{
    auto ok = [&](int p) {
        const int q = (p - mod4) & 31;
        if (ext <= 4.0f) return (q & 7) == 4;
        if (ext <= 8.0f) return (q & 15) == 8;
        return q == 12 || q == 16 || q == 20;
    };
    while (!ok(w)) ++w;
    return w;
}

// The launch's staging geometry: for each major axis that its tiles take, box extents that
// hold the sampled tiles' footprints, the longest step whose window fits the shared memory
// budget.  False when no step fits: the gather marcher then serves the request.
inline bool roll_geometry(const shw_camera &cam, const int n[3], int H, bool tmaps, int budget, int smax, int min_s,
                          RollArgs &ra)
{
    const int on[3] = {1, 1, 1};
    int wa[3] = {0, 0, 0}, wb[3] = {0, 0, 0};
    float ext[3] = {8.0f, 8.0f, 8.0f};
    const int tx = ceil_div(cam.width, kSlabTW), ty = ceil_div(cam.height, kSlabTH);
    for (int j = 0; j < 5; ++j)
        for (int i = 0; i < 5; ++i) {
            const TileRays r = roll_rays(cam, (int)((long long)(tx - 1) * i / 4) * kSlabTW,
                                         (int)((long long)(ty - 1) * j / 4) * kSlabTH, on, ra.xbias);
            const int M = r.major, g = M == 0 ? kRollXG : 1;
            const float was = M == 0   ? (roll_extent<0>(r, n, H, g, wa[0], wb[0]), roll_warp_extent<0>(r, n))
                              : M == 1 ? (roll_extent<1>(r, n, H, g, wa[1], wb[1]), roll_warp_extent<1>(r, n))
                                       : (roll_extent<2>(r, n, H, g, wa[2], wb[2]), roll_warp_extent<2>(r, n));
            if (ext[M] == 8.0f || (i == 2 && j == 2)) ext[M] = was;
        }
    int stage = 0;
    bool any = false;
    for (int M = 0; M < 3; ++M) {
        RollGeom &G = ra.geo[M];
        G = RollGeom{};
        if (wa[M] <= 0 || wb[M] <= 0) continue;  // no sampled tile takes this axis: none will
        const int A = M == 0 ? 1 : 0, B = M == 2 ? 1 : 2;
        G.g = M == 0 ? kRollXG : 1;
        // room for the tiles and planes between the sampled ones (a footprint that the cube clips
        // may be narrower than the taps' reach)
        G.wb = std::min(wb[M] + 2 + std::max(wb[M] - 2 * H, 0) / 10, n[B]);
        G.wa = std::min(wa[M] + 2 + std::max(wa[M] - 2 * H, 0) / 10, n[A]);
        int pad = 0;
        if (M != 0 && tmaps) {
            G.sb = G.wa = roll_pitch(G.wa + 3, ext[M], 0);  // a tensor copy's rows; its x start on 16 bytes
        } else if (M != 0) {
            G.sb = roll_pitch(G.wa + 6, ext[M], (M == 2 ? n[0] : (n[0] & 3) * (n[1] & 3)) & 3);
            pad = 16;
        } else {
            G.sb = roll_pitch(G.wa, ext[M], 0);
        }
        if (G.wa > 256 || G.wb > 256) return false;
        G.plane = (G.sb * G.wb + pad + 31) & ~31;
        G.slot = G.plane * G.g;
        G.depth = 1;
        const int cap = std::min(std::min(kRollMaxSlots, kRollTable / G.g), budget / (G.slot * 4));
        G.s = 0;
        for (int s = 1; s <= smax; ++s)
            if (roll_slots(H, s, G.g, G.depth) <= cap) G.s = s;
        if (G.s < min_s) return false;
        G.ns = roll_slots(H, G.s, G.g, G.depth);
        G.on = 1;
        any = true;
        stage = std::max(stage, G.ns * G.slot * 4);
    }
    ra.smem_stage = (stage + 127) & ~127;
    return any;
}

template <int MODE, int KIND, class S>
shw_status roll_launch_one(const RollMaps &maps, const S &s, const shw_camera &cam, const RenderArgs &a,
                           const RollArgs &ra, size_t smem, cudaStream_t st)
{
    auto kern = roll_kernel<MODE, KIND, S>;
    // The limit is the kernel's, shared by every thread of the process: always the largest ring, so
    // that no concurrent call lowers it between another's setting and launch.  (Residency follows
    // from the launch's own size.)
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRollBudget1) != cudaSuccess) {
        cudaGetLastError();
        return SHW_ECUDA;
    }
    const int nsm = sm_count(), per_sm = smem <= (size_t)kRollBudget2 ? 2 : 1;
    if (nsm <= 0) return SHW_ECUDA;
    const long long grid = std::min<long long>((long long)per_sm * nsm, ra.ntiles);
    kern<<<(unsigned)std::max<long long>(grid, 1), kSlabThreads, smem, st>>>(maps, s, cam, a, ra);
    return after_launch();
}

// Whether the ring pays (else the samples are gathered).  Its hand-overs and halo planes are a fixed
// cost per tile and it keeps one CTA per tile, so it needs tiles that fill the device and
// footprints that are not much wider than the taps' reach; a gather costs least where a warp's rays
// share rows of the cube (y- and z-major views), most in x-major ones and where the cube exceeds the
// second-level cache (from 3 x 10^7 voxels on).  Compositing's gathers stop with the ray, the ring
// with the tile.  From the major axis of the tile at the cube's projected centre, the voxels per
// pixel there, the rows that a gathering warp spans (warp_rows) and the tiles that see the cube.
// Over 2472 renders (32^3 .. 640^3 and oblong cubes, 96^2 .. 1000^2, eleven views and random ones, 3
// to 13 taps, boxes of 3 to 9) the ring took 0.09 to 1.07 of the gather's time in the 472 where this
// takes it, 0.14 to 11 times as long elsewhere (9 taps, 512^3 on
// 1000 x 1000: MIP at yaw 30 24.1 ms gathered, 8.7 staged, at yaw 100 82.6 and 7.9, looking down
// at yaw 20 13.0 and 8.5, compositing 7.1 and 7.4; 129^3 on 128 x 128, MIP along z 0.33 and 0.59).
template <int KIND>
inline bool roll_pays(const shw_camera &cam, const int n[3], bool tmaps, int ntaps, bool composite, float xbias)
{
    const double vox = (double)n[0] * n[1] * n[2], pitch = centre_pitch(cam, n[0], n[1], n[2]);
    const double tiles = covered_pixels(cam, n[0], n[1], n[2]) / (kSlabTW * kSlabTH);
    const double rows = warp_rows(cam, n[0], n[1], n[2]);
    const int least = std::min(n[0], std::min(n[1], n[2]));
    float px, py;
    project_centre(cam, n[0], n[1], n[2], px, py);
    const int on[3] = {1, 1, 1};
    const int major = roll_rays(cam, (int)fminf(fmaxf(px, 0.0f), (float)(cam.width - 1)) / kSlabTW * kSlabTW,
                                (int)fminf(fmaxf(py, 0.0f), (float)(cam.height - 1)) / kSlabTH * kSlabTH, on, xbias)
                          .major;
    const bool big = vox >= 3e7;
    if (KIND == kRollBox) {  // two fetches a sample when gathered: large cubes by tensor copies only
        if (!tmaps || vox < 1e7) return false;
        if (major == 0)
            return composite ? vox >= 2e7 && rows <= 20.0 && pitch <= 2.0 : least >= 80 && rows <= 15.0 && pitch <= 1.6;
        if (composite)
            return least >= 80 && pitch <= 1.25 &&
                   (major == 2 ? tiles >= 450.0 : rows >= 7.0 && rows <= 20.0 && tiles >= 608.0);
        return pitch <= 2.5 && (major == 2 ? vox >= 2e7 : rows >= 6.0 && least >= 80);
    }
    // few taps and row copies need a larger cube; below 64 voxels on an axis most taps clamp
    if (least < 64 || !((tmaps && ntaps >= 2) || vox >= 2e6)) return false;
    if (composite) {
        if (major == 0)
            return (least >= 80 && vox >= 3e6 && tiles >= 30.0 && rows <= 16.0 && pitch <= 1.6) ||
                   (least >= 144 && tiles >= 60.0 && pitch <= 2.5);
        return major == 2 && big && tiles >= 450.0 && pitch <= 2.5;
    }
    if (major == 0)
        return (least >= 152 && pitch <= 2.5) || (vox >= 2e6 && rows <= 14.0 && pitch <= 1.6) ||
               (ntaps >= 2 && rows >= 4.5 && rows <= 16.0 && pitch <= 1.2);
    return (big && pitch <= 2.5 && tiles >= (major == 2 ? 450.0 : 300.0)) ||
           (rows >= 5.0 && pitch <= 1.1 && tiles >= 30.0) || (tiles >= 450.0 && pitch <= 0.5);
}

// In-ray smoothing of a float32 cube through the rolling marcher; SHW_EUNSUPPORTED when it
// does not serve the request.
template <int KIND>
shw_status roll_launch(int mode, const shw_volume &v, const shw_camera &cam, const RenderArgs &a0, cudaStream_t st)
{
    const SamplerF32<int> s{static_cast<const float *>(v.data), v.nx, v.ny, v.nz, v.nx, v.nx * v.ny};
    using S = SamplerF32<int>;
    const int n[3] = {v.nx, v.ny, v.nz};
    RollArgs ra{};
    ra.cube = s.v;
    ra.halo = 0;
    if (KIND == kRollTaps)  // a tap at offset o reaches cells up to ceil(|o|) away
        for (int j = 0; j < a0.smooth_n; ++j) {
            const long long o = a0.smooth_off[j] < 0 ? -a0.smooth_off[j] : a0.smooth_off[j];
            ra.halo = std::max(ra.halo, (int)((o + 0xffffffffLL) >> 32));
        }
    const bool tmaps = v.nx % 4 == 0 && aligned(v.data, 16);
    // Taps: the true major axis (the planes hold the taps' reach on both sides, and only small
    // slopes keep two CTAs on an SM).  The box: x-major planes cost the producer a transposition,
    // so steep y- and z-major ones are taken up to a slope of 3.
    ra.xbias = KIND == kRollTaps ? 1.0f : 3.0f;
    const bool composite = mode == SHW_COMPOSITE || mode == SHW_COMPOSITE_SPECTRAL || mode == SHW_COMPOSITE_RGB;
    if (!debug(SHW_DEBUG_REQUIRE_STAGING) && !roll_pays<KIND>(cam, n, tmaps, a0.smooth_n, composite, ra.xbias))
        return SHW_EUNSUPPORTED;
    ra.rows = !tmaps;
    ra.goff = (int)((reinterpret_cast<uintptr_t>(v.data) >> 2) & 3);
    size_t extra = sizeof(RollShared);
    if (KIND == kRollBox) {
        int len = 1;
        while (len < 4 * a0.smooth_n + 3) len *= 2;
        ra.box_mask = len - 1;
        extra += (size_t)len * 32 * kSlabWarps * 4;
    }
    // two CTAs per SM where a step of at least two cells fits, else one
    const int smax = KIND == kRollTaps ? 4 : 12;
    if (!roll_geometry(cam, n, ra.halo, tmaps, kRollBudget2 - (int)extra, smax, 2, ra) &&
        !roll_geometry(cam, n, ra.halo, tmaps, kRollBudget1 - (int)extra, smax, 1, ra))
        return SHW_EUNSUPPORTED;
    RollMaps maps{};
    if (tmaps) {
        const RollGeom *G = ra.geo;
        if ((G[1].on && !encode_tmap_3d(&maps.m[0], s.v, 4, v.nx, v.ny, v.nz, G[1].wa, 1, G[1].wb)) ||
            (G[2].on && !encode_tmap_3d(&maps.m[1], s.v, 4, v.nx, v.ny, v.nz, G[2].wa, G[2].wb, 1)))
            return SHW_EUNSUPPORTED;
    }
    RenderArgs a = a0;
    a.tiles_x = ceil_div(cam.width, kSlabTW);
    a.tiles_y = ceil_div(cam.height, kSlabTH);
    float cpx, cpy;
    project_centre(cam, v.nx, v.ny, v.nz, cpx, cpy);
    a.ctx = (int)fminf(fmaxf(cpx / kSlabTW, 0.0f), (float)(a.tiles_x - 1));
    a.cty = (int)fminf(fmaxf(cpy / kSlabTH, 0.0f), (float)(a.tiles_y - 1));
    ra.ntiles = a.tiles_x * a.tiles_y;
    ra.err = device_error_word();
    ra.polls = kSlabWaitPolls;
    ra.ctr = work_counter(st);
    if (!ra.ctr) return SHW_ECUDA;
    const size_t smem = (size_t)ra.smem_stage + extra;
    switch (mode) {
    case SHW_MIP:
        // without a channel output only the maximum's value matters
        if (a.index == nullptr) return roll_launch_one<kMipValue, KIND, S>(maps, s, cam, a, ra, smem, st);
        return roll_launch_one<SHW_MIP, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_AVG: return roll_launch_one<SHW_AVG, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_COMPOSITE: return roll_launch_one<SHW_COMPOSITE, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_SPECTRAL: return roll_launch_one<SHW_SPECTRAL, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_MOMENT1: return roll_launch_one<SHW_MOMENT1, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_COMPOSITE_SPECTRAL:
        return roll_launch_one<SHW_COMPOSITE_SPECTRAL, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_MIP_RGB: return roll_launch_one<SHW_MIP_RGB, KIND, S>(maps, s, cam, a, ra, smem, st);
    case SHW_COMPOSITE_RGB: return roll_launch_one<SHW_COMPOSITE_RGB, KIND, S>(maps, s, cam, a, ra, smem, st);
    default: return SHW_EUNSUPPORTED;
    }
}

}  // namespace shw
