// Production render kernels of the batched egocentric rasterizer (sm_100a).
//
// The z-buffer holds one 64-bit key per pixel (in registers or shared memory),
//     key = float_bits(1/z) << 32 | (0xFFFFFF - primitive index) << 8 | class,
// so "nearest fragment wins, exact ties go to the lower index" is an unsigned max that does not
// depend on the order in which primitives arrive; 0 means "no fragment" (background).
//
// A unit of work is a tile: up to 64 x 64 pixels of one view.
//
// cull_kernel.  A warp per tile, or per view of several tiles, finds the primitives and box faces that can touch a pixel
// centre and leaves them as a list per tile in device memory.
//
// render_tile_kernel (pic_tile.cuh).  A warp per tile: set-up, raster and store with the z-buffer in registers.  Tiles whose
// lists overflow are appended to a list in device memory.
//
// cooperative_kernel.  One wave of CTAs walks that list; a whole CTA renders a tile in
// barrier-separated phases with per-round lists (any number of groups, boxes, survivors and
// records): the general path, and the one the others are checked against in the tests.
//
// render_small_kernel (pic_small.cuh).  Calls with few tiles: a CTA of 8 warps takes one tile from culling to store.
//
// coverage_kernel (occlusion counts), colour_kernel (pic_colour.cuh), render_static_kernel (pic_static.cuh).
//
// Cameras (one 64-byte record per view) and per-camera ray / background tables are prepared by
// the set-up kernel, so the prologues are a few loads.
#include <cstddef>

#include "pic_device.cuh"
#include "pic_rows.h"

namespace pic {

constexpr int NTHREADS = 128;
constexpr int NW = NTHREADS / 32;
constexpr int RCAP = 64;          // records (primitives rasterized by a warp) per tile
constexpr int REC = 20;           // words per record (17 used; 16-byte aligned for vector access)
constexpr int GROUP_BATCH = 16;   // groups examined per round
constexpr int LEAFCAP = GROUP_BATCH * GROUP_LEAVES;   // visible leaves per round
constexpr int BOX_ROUND = 64;     // boxes examined per round
constexpr int FACECAP = 6 * BOX_ROUND;
constexpr int SCAP = 128;         // candidates that survive the pixel-box test, per round
constexpr int TINY_MAX_PIXELS = 4;         // pixel centres in the box of a primitive rasterized by its own thread
constexpr int CLASSIFY_MIN_PIXELS = 192;   // pixel boxes at least this large classify cells before rasterizing

struct __align__(16) TileSmem {
    unsigned long long key[TILE * TILE];      // 32 KB, 16-byte chunks XOR-swizzled by row (key_index)
    float4 rec[RCAP * REC / 4];
    uint32_t leaf[LEAFCAP];                   // visible leaves of the round: first primitive << 4 | count
    uint32_t face[FACECAP];                   // box-face items of the round: agent << 3 | face
    uint2 surv[SCAP];                         // candidates whose pixel box holds a pixel centre: (item, box)
    float ray_x[TILE], ray_y[TILE];           // ray coordinates of the tile's pixel columns / rows
    float plane[6][4];                        // tile frustum, ego-relative world space, unit normals: n, offset
    float side[4][4];                         // the four side planes in camera space, unit normals
    Cam cam;
    int n_rec, n_leaf, n_face, n_surv;
    uint32_t touched[2];                      // 8x8 blocks that may hold a fragment (rows 0-3, rows 4-7)
};

static_assert(offsetof(TileSmem, plane) % 16 == 0 && offsetof(TileSmem, side) % 16 == 0, "planes are written with 128-bit stores");

// Keys are stored so that both access patterns spread over all banks.  A 16-byte chunk holds pixels
// (2c, 2c+1) of row y; its low three index bits are XORed with (y & 1) << 2 | (c >> 3).  Raster: a
// 16 x 4 cell is read a row (8 chunks of one 16-pixel column block) per quarter warp.  Store: 32
// consecutive lanes take 32 consecutive 16-pixel segments (two rows x four column blocks per quarter
// warp) and read chunk i of their segment together.
__device__ __forceinline__ int key_index(int x, int y) {
    const int c = x >> 1;
    return (y << 6) | (((c ^ (((y & 1) << 2) | (c >> 3))) << 1) | (x & 1));
}

// Bit mask of the 8x8 blocks touched by a pixel box (inclusive).
__device__ __forceinline__ unsigned long long block_mask(int bx0, int by0, int bx1, int by1) {
    const int c0 = bx0 >> 3, c1 = bx1 >> 3, r0 = by0 >> 3, r1 = by1 >> 3;
    const unsigned long long row = (unsigned long long)(((2u << c1) - (1u << c0)) & 0xffu);
    const unsigned long long rows = (0x0101010101010101ull >> (8 * (7 - (r1 - r0)))) << (8 * r0);
    return row * rows;
}

__device__ __forceinline__ void mark_touched(uint32_t* touched, unsigned long long m) {
    const uint32_t lo = (uint32_t)m, hi = (uint32_t)(m >> 32);
    if (lo & ~touched[0]) atomicOr(&touched[0], lo);
    if (hi & ~touched[1]) atomicOr(&touched[1], hi);
}

// Is the box [lo,hi] (world) possibly inside the tile frustum?  Conservative.
template <class S>
__device__ __forceinline__ bool box_visible(const S& s, const Node& b) {
    const float ax = sub(b.lo[0], s.cam.px), bx = sub(b.hi[0], s.cam.px);
    const float ay = sub(b.lo[1], s.cam.py), by = sub(b.hi[1], s.cam.py);
    const float cx = 0.5f * (ax + bx), cy = 0.5f * (ay + by), cz = 0.5f * (b.lo[2] + b.hi[2]);
    const float hx = 0.5f * (bx - ax), hy = 0.5f * (by - ay), hz = 0.5f * (b.hi[2] - b.lo[2]);
    // rounding of the few float32 operations below, far under any real distance
    const float slack = 1e-3f + 4e-6f * (fabsf(cx) + fabsf(cy) + fabsf(cz) + hx + hy + hz);
    bool vis = true;
#pragma unroll
    for (int p = 0; p < 6; ++p) {
        const float nx = s.plane[p][0], ny = s.plane[p][1], nz = s.plane[p][2], d = s.plane[p][3];
        const float dist = nx * cx + ny * cy + nz * cz + d;
        const float reach = fabsf(nx) * hx + fabsf(ny) * hy + fabsf(nz) * hz;
        vis = vis && (dist + reach >= -slack);
    }
    return vis;
}

template <class S>
__device__ __forceinline__ void put_fragment(S& s, int x, int y, uint32_t wbits, uint32_t key_lo) {
    const unsigned long long k = make_key(wbits, key_lo);
    unsigned long long* addr = &s.key[key_index(x, y)];
    atomicMax(addr, k);
}

// Rasterize a primitive from one thread: loop over its pixel box, atomic max per fragment.
template <class S>
__device__ __forceinline__ int raster_in_thread(S& s, uint32_t* touched, const TileCtx& t, const PrimEq& q, uint32_t key_lo, uint32_t box) {
    const int bx0 = box & 0xff, by0 = (box >> 8) & 0xff, bx1 = (box >> 16) & 0xff, by1 = box >> 24;
    int frags = 0;
    for (int y = by0; y <= by1; ++y) {
        const float ry = s.ray_y[y];
        for (int x = bx0; x <= bx1; ++x) {
            const uint32_t wb = fragment(q, s.ray_x[x], ry, t.w_near, t.w_far);
            if (wb) { put_fragment(s, x, y, wb, key_lo); ++frags; }
        }
    }
    if (frags) mark_touched(touched, block_mask(bx0, by0, bx1, by1));
    return frags;
}

// Plane p of the tile's frustum, ego-relative, and for p >= 2 the same side plane in camera space (see frustum_entry).
template <class S>
__device__ __forceinline__ void tile_planes(S& s, int p, const Cam& c, const TileCtx& t) {
    const float4 e = frustum_plane(p, (float)t.x0 - c.cx, (float)(t.x0 + t.tw) - c.cx, (float)t.y0 - c.cy, (float)(t.y0 + t.th) - c.cy, c.focx, c.focy, t.near_z, t.far_z);
    *reinterpret_cast<float4*>(s.plane[p]) = world_plane(c, rotate_to_world(c, e), e.w);
    if (p >= 2) *reinterpret_cast<float4*>(s.side[p - 2]) = e;
}

// Which faces of another agent's box can reach the tile: 0 if its bounding sphere misses the
// frustum, else the faces that can face the camera (all six near the near plane or inside the box).
template <class S>
__device__ __forceinline__ uint32_t box_faces(const S& s, const Cam& c, const TileCtx& t, const AgentGeom& g) {
    const float hh = 0.5f * g.h;
    const V3 ctr = rotate_to_camera(c, sub(sub(g.x, c.px), c.mwx), sub(sub(g.y, c.py), c.mwy), sub(hh, c.mwz));
    const float rad = sqrtf(g.hl * g.hl + g.hw * g.hw + hh * hh) * 1.0001f + 1e-4f;
    bool vis = (ctr.z + rad >= t.near_z * 0.999f) && (ctr.z - rad <= t.far_z * 1.001f);
#pragma unroll
    for (int p = 0; p < 4; ++p)
        vis = vis && (s.side[p][0] * ctr.x + s.side[p][1] * ctr.y + s.side[p][2] * ctr.z >= -rad);
    if (!vis) return 0u;
    uint32_t faces = 0x3fu;
    if (ctr.z - rad > t.near_z * 1.01f) {
        const float dx = sub(c.mwx, sub(g.x, c.px)), dy = sub(c.mwy, sub(g.y, c.py));
        const float u = g.c * dx + g.s * dy, v = g.c * dy - g.s * dx;
        const float eps = 1e-4f * (1.f + fabsf(dx) + fabsf(dy));
        faces = 0u;
        if (u < -g.hl + eps) faces |= 1u;          // rear
        if (u > g.hl - eps) faces |= 2u;           // front
        if (v < -g.hw + eps) faces |= 4u;          // right
        if (v > g.hw - eps) faces |= 8u;           // left
        if (c.mwz < eps) faces |= 16u;             // bottom
        if (c.mwz > g.h - eps) faces |= 32u;       // top
    }
    return faces;
}

// Work counters of a thread; the production kernel is compiled with NoTally, where they vanish.
struct Tally { int grp, leaf, tested, setup, tiny, recs, fallback, classified, cells, jobs, coop; };
struct NoCount {
    __device__ __forceinline__ NoCount& operator++() { return *this; }
    __device__ __forceinline__ NoCount& operator=(int) { return *this; }
    __device__ __forceinline__ NoCount& operator+=(int) { return *this; }
};
__device__ __forceinline__ int tally_value(int v) { return v; }
__device__ __forceinline__ int tally_value(const NoCount&) { return 0; }
struct NoTally { NoCount grp, leaf, tested, setup, tiny, recs, fallback, classified, cells, jobs, coop; };

// Cooperative kernel, phase 2b body: set a surviving primitive up, rasterize it (tiny) or leave a record.
template <class S, class TL>
__device__ __forceinline__ void setup_prim(S& s, const TileCtx& t, const V3 (&V)[4], bool quad, uint32_t flags,
                                           const V3 Pn, uint32_t key_lo, uint32_t box, int rec_cap, TL& n) {
    PrimEq q;
    if (!prim_equations(V, quad, flags, Pn, q)) return;
    ++n.setup;
    const int bx0 = box & 0xff, by0 = (box >> 8) & 0xff, bx1 = (box >> 16) & 0xff, by1 = box >> 24;
    if ((bx1 - bx0 + 1) * (by1 - by0 + 1) > TINY_MAX_PIXELS) {
        const int slot = atomicAdd(&s.n_rec, 1);
        if (slot < rec_cap) {
            float4* r = &s.rec[slot * (REC / 4)];
            r[0] = make_float4(q.nx[0], q.nx[1], q.nx[2], q.nx[3]);
            r[1] = make_float4(q.ny[0], q.ny[1], q.ny[2], q.ny[3]);
            r[2] = make_float4(q.nz[0], q.nz[1], q.nz[2], q.nz[3]);
            r[3] = make_float4(q.wx, q.wy, q.wz, __uint_as_float(key_lo));
            // the pixel box needs 6 bits per coordinate; the top-left bits ride along
            r[4].x = __uint_as_float((uint32_t)bx0 | ((uint32_t)by0 << 6) | ((uint32_t)bx1 << 12) | ((uint32_t)by1 << 18) | (q.tl << 24));
            ++n.recs;
            return;
        }
        ++n.fallback;          // list full: correct but slow
    } else {
        ++n.tiny;
    }
    raster_in_thread(s, s.touched, t, q, key_lo, box);
}

// Candidate `i` of the round: a primitive of a visible leaf or a box-face item, in camera space.
template <class S>
__device__ __forceinline__ bool fetch_candidate(const S& s, const RenderParams& P, int i, int nl, int e, uint32_t n_map_tris,
                                                V3 (&V)[4], V3& Pn, uint32_t& key_lo, uint32_t& flags, bool want_plane) {
    const Cam& c = s.cam;
    if (i < nl * LEAF_PRIMS) {
        const uint32_t lf = s.leaf[i / LEAF_PRIMS];
        const uint32_t j = i % LEAF_PRIMS;
        if (j >= (lf & 15u)) return false;
        float v[12], vis_cos;
        load_prim(P.prims + (lf >> 4) + j, v, key_lo, flags, vis_cos);
#pragma unroll
        for (int q = 0; q < 4; ++q) V[q] = to_camera(c, v[3 * q], v[3 * q + 1], v[3 * q + 2]);
        if (want_plane) Pn = limit_angular_range(V, plane_normal_world(c, v, flags & 1u), vis_cos);
    } else {
        const uint32_t it = s.face[i - nl * LEAF_PRIMS];
        const int b = (int)(it >> 3), f = (int)(it & 7u);
        const AgentGeom g = P.agents[(size_t)e * P.A + b];
        const uint32_t corners = face_corners(f);
#pragma unroll
        for (int q = 0; q < 4; ++q) V[q] = box_corner(c, g, (corners >> (4 * q)) & 7u);
        key_lo = ((0xFFFFFFu - (n_map_tris + 12u * (uint32_t)b + 2u * (uint32_t)f)) << 8) | agent_box_class(g);
        flags = face_flags(corners);
        if (want_plane) Pn = plane_normal(V, true);
    }
    return true;
}

// The top-left rule "e > 0 || (e == 0 && the edge owns its zeros)" as one comparison e > thr:
// thr is 0 or the smallest negative subnormal -- nothing lies between the two, and neither fma nor
// the comparison flushes subnormals.
__device__ __forceinline__ void edge_thresholds(uint32_t tl, float (&thr)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) thr[e] = __int_as_float(((tl >> e) & 1u) ? (int)0x80000001u : 0);
}

// One 16 x 4 cell at (xx, yy): every lane tests its two pixels and updates their keys with plain
// loads and stores -- the rows of a cell belong to exactly one warp (its bands).  `need`: the edges
// that still have to be tested on this cell (0: the cell is known to be covered and in depth
// range; the range test rides on the edge tests).  Returns whether any lane produced a fragment.
template <class S>
__device__ __forceinline__ bool raster_cell(S& s, const TileCtx& t, const PrimEq& q, const float (&thr)[4], uint32_t key_lo, int xx, int yy,
                                            uint32_t need, int lane) {
    const int x = xx + (lane & 7) * 2, y = yy + (lane >> 3);
    const float rx0 = s.ray_x[x], rx1 = s.ray_x[x + 1], ry = s.ray_y[y];
    const float wt = fm(q.wy, ry, q.wz);
    const float w0 = fm(q.wx, rx0, wt), w1 = fm(q.wx, rx1, wt);
    bool in0 = true, in1 = true;
    if (need) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if ((need >> e) & 1u) {          // warp-uniform: edges known to be positive on the whole cell are skipped
                const float te = fm(q.ny[e], ry, q.nz[e]);
                const float e0 = fm(q.nx[e], rx0, te), e1 = fm(q.nx[e], rx1, te);
                in0 = in0 && (e0 > thr[e]);
                in1 = in1 && (e1 > thr[e]);
            }
        }
        in0 = in0 && (w0 >= t.w_far) && (w0 <= t.w_near);
        in1 = in1 && (w1 >= t.w_far) && (w1 <= t.w_near);
    }
    {
        ulonglong2* kp = reinterpret_cast<ulonglong2*>(&s.key[key_index(x, y)]);
        ulonglong2 kk = *kp;
        const unsigned long long k0 = make_key(__float_as_uint(w0), key_lo), k1 = make_key(__float_as_uint(w1), key_lo);
        const bool up0 = in0 && k0 > kk.x, up1 = in1 && k1 > kk.y;
        if (up0) kk.x = k0;
        if (up1) kk.y = k1;
        if (up0 || up1) *kp = kk;
    }
    return __any_sync(0xffffffffu, in0 || in1);
}

// Cooperative kernel, phase 3: every warp walks all records but rasterizes only the bands (4 pixel rows) it owns --
// band b belongs to warp b % NW -- so keys are updated without atomics and the bands of a large
// primitive are shared out evenly.
template <int NWARPS, class S, class TL>
__device__ __forceinline__ void raster_records(S& s, const float4* rec, uint32_t* touched_out, const TileCtx& t, int n_rec, bool classify, TL& n) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned long long touched = 0ull;     // 8x8 blocks
    for (int p = 0; p < n_rec; ++p) {
        const float4* r = &rec[p * (REC / 4)];
        const uint32_t bw = __float_as_uint(r[4].x);
        const int bx0 = bw & 63, by0 = (bw >> 6) & 63, bx1 = (bw >> 12) & 63, by1 = (bw >> 18) & 63;
        // first band of this warp at or after the box's first band
        const int band0 = by0 >> 2, band1 = by1 >> 2;
        int first = band0 + ((warp - band0) & (NWARPS - 1));
        if (first > band1) continue;
        PrimEq q;
        const float4 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3];
        q.nx[0] = r0.x; q.nx[1] = r0.y; q.nx[2] = r0.z; q.nx[3] = r0.w;
        q.ny[0] = r1.x; q.ny[1] = r1.y; q.ny[2] = r1.z; q.ny[3] = r1.w;
        q.nz[0] = r2.x; q.nz[1] = r2.y; q.nz[2] = r2.z; q.nz[3] = r2.w;
        q.wx = r3.x; q.wy = r3.y; q.wz = r3.z;
        const uint32_t key_lo = __float_as_uint(r3.w);
        q.tl = (bw >> 24) & 15u;
        float thr[4];
        edge_thresholds(q.tl, thr);
        if (classify && (bx1 - bx0 + 1) * (by1 - by0 + 1) >= CLASSIFY_MIN_PIXELS) {
            // (b) lanes 0..15 classify this warp's 16 cells: reject / partly covered / inside
            if (warp == 0) ++n.classified;
            const int band = (lane >> 2) * NWARPS + warp, col = lane & 3;
            const int xa = col * 16, xb = xa + 15, ya = band * 4, yb = ya + 3;
            bool reject = lane >= 16 || xb < bx0 || xa > bx1 || yb < by0 || ya > by1;
            uint32_t need = 0u;
            if (!reject) {
                const float rxa = s.ray_x[xa], rxb = s.ray_x[xb], rya = s.ray_y[ya], ryb = s.ray_y[yb];   // rxa < rxb, rya < ryb
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    // fma is monotone in each argument, so the cell's extreme values are at its corners
                    const float ta = fm(q.ny[e], rya, q.nz[e]), tb = fm(q.ny[e], ryb, q.nz[e]);
                    const float emax = fm(q.nx[e], q.nx[e] >= 0.f ? rxb : rxa, fmaxf(ta, tb));
                    const float emin = fm(q.nx[e], q.nx[e] >= 0.f ? rxa : rxb, fminf(ta, tb));
                    reject = reject || (emax < 0.f);
                    if (!(emin > 0.f)) need |= 1u << e;
                }
                const float wa = fm(q.wy, rya, q.wz), wb = fm(q.wy, ryb, q.wz);
                const float wmax = fm(q.wx, q.wx >= 0.f ? rxb : rxa, fmaxf(wa, wb));
                const float wmin = fm(q.wx, q.wx >= 0.f ? rxa : rxb, fminf(wa, wb));
                reject = reject || (wmax < t.w_far) || (wmin > t.w_near);
                // the depth range test rides on the edge tests: if it is still needed, so is one edge
                if (need == 0u && !((wmin >= t.w_far) && (wmax <= t.w_near))) need = 1u;
            }
            for (unsigned m = __ballot_sync(0xffffffffu, !reject); m; m &= m - 1) {
                const int cell = __ffs(m) - 1;
                const int xx = (cell & 3) * 16, yy = ((cell >> 2) * NWARPS + warp) * 4;
                const uint32_t need_c = __shfl_sync(0xffffffffu, need, cell);
                ++n.cells;
                if (raster_cell(s, t, q, thr, key_lo, xx, yy, need_c, lane)) touched |= 3ull << ((yy >> 3) * 8 + (xx >> 3));
            }
        } else {
            for (int band = first; band <= band1; band += NWARPS)
                for (int xx = bx0 & ~15; xx <= bx1; xx += 16) {
                    ++n.cells;
                    if (raster_cell(s, t, q, thr, key_lo, xx, band * 4, 0xFu, lane)) touched |= 3ull << ((band >> 1) * 8 + (xx >> 3));
                }
        }
    }
    if (lane == 0 && touched) mark_touched(touched_out, touched);
}

// (d) keys -> class / depth images.  `touched`: the 8x8 blocks that may hold a fragment.
template <class S>
__device__ __forceinline__ void store_tile(S& s, const TileCtx& t, const RenderParams& P, size_t view, int k, bool ego_active,
                                           unsigned long long touched, int tid = threadIdx.x, int nthr = NTHREADS,
                                           uint32_t n_map_tris = 0u) {
    const size_t img = (size_t)P.H * P.W;
    uint32_t* occ = P.occlusion ? P.occlusion + view * (size_t)P.A * 2u : nullptr;   // visible-pixel counts of this view
    uint8_t* oc = P.out_class + view * img;
    uint16_t* od = P.out_depth + view * img;
    float* o32 = P.out_depth32 ? P.out_depth32 + view * img : nullptr;
    // (pic_render_static takes outputs of any alignment)
    const bool vec_ok = (P.W % 16 == 0) && o32 == nullptr && ((reinterpret_cast<uintptr_t>(P.out_class) | reinterpret_cast<uintptr_t>(P.out_depth)) & 15u) == 0;
    const int segs_per_row = (t.tw + 15) >> 4;
    const int n_seg = t.th * segs_per_row;
    // consecutive threads take consecutive 16-pixel segments of a row, then the next row: a warp's
    // class stores cover 512 contiguous bytes of a 64-pixel-wide image, its depth stores 1 KB
    for (int seg = tid; seg < n_seg; seg += nthr) {
        const int y = seg / segs_per_row;
        const int xs = (seg - y * segs_per_row) * 16;
        uint32_t bg_cls = P.cls_sky;
        float bg_z = P.far_z;
        if (ego_active) { bg_cls = __ldg(P.rig.bg_cls + (size_t)k * P.H + t.y0 + y); bg_z = __ldg(P.rig.bg_z + (size_t)k * P.H + t.y0 + y); }
        const size_t o = (size_t)(t.y0 + y) * P.W + t.x0 + xs;
        const bool empty = ((touched >> ((y >> 3) * 8 + (xs >> 3))) & 3ull) == 0ull;   // both blocks of the segment
        if (vec_ok && xs + 16 <= t.tw) {
            uint32_t cw[4], dw[8];
            if (empty) {
                const uint32_t c4 = bg_cls * 0x01010101u;
                const __half2 h = __floats2half2_rn(bg_z, bg_z);
                const uint32_t d2 = *reinterpret_cast<const uint32_t*>(&h);
#pragma unroll
                for (int j = 0; j < 4; ++j) cw[j] = c4;
#pragma unroll
                for (int j = 0; j < 8; ++j) dw[j] = d2;
            } else {
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const ulonglong2 kk = *reinterpret_cast<const ulonglong2*>(&s.key[key_index(xs + j, y)]);
                    if (occ) { count_visible(occ, kk.x, n_map_tris); count_visible(occ, kk.y, n_map_tris); }
                    const float z0 = kk.x ? fast_rcp(__uint_as_float((uint32_t)(kk.x >> 32))) : bg_z;
                    const float z1 = kk.y ? fast_rcp(__uint_as_float((uint32_t)(kk.y >> 32))) : bg_z;
                    const uint32_t c0 = kk.x ? (uint32_t)(kk.x & 0xff) : bg_cls, c1 = kk.y ? (uint32_t)(kk.y & 0xff) : bg_cls;
                    const __half2 h = __floats2half2_rn(z0, z1);
                    dw[j >> 1] = *reinterpret_cast<const uint32_t*>(&h);
                    if ((j & 3) == 0) cw[j >> 2] = c0 | (c1 << 8); else cw[j >> 2] |= (c0 << 16) | (c1 << 24);
                }
            }
            *reinterpret_cast<uint4*>(oc + o) = make_uint4(cw[0], cw[1], cw[2], cw[3]);
            *reinterpret_cast<uint4*>(od + o) = make_uint4(dw[0], dw[1], dw[2], dw[3]);
            *reinterpret_cast<uint4*>(od + o + 8) = make_uint4(dw[4], dw[5], dw[6], dw[7]);
        } else {
            for (int j = 0; j < 16 && xs + j < t.tw; ++j) {
                const unsigned long long key = empty ? 0ull : s.key[key_index(xs + j, y)];
                if (occ) count_visible(occ, key, n_map_tris);
                const float z = key ? fast_rcp(__uint_as_float((uint32_t)(key >> 32))) : bg_z;
                oc[o + j] = (uint8_t)(key ? (uint32_t)(key & 0xff) : bg_cls);
                od[o + j] = __half_as_ushort(__float2half_rn(z));
                if (o32) o32[o + j] = z;
            }
        }
    }
}

// One unit of work: a tile of a view.
struct Job {
    int tile, k, a, e;
    size_t view;
    TileCtx t;
};

// Job `id` of the launch: tiles of a view are consecutive, views follow P.view_first.
// (tile_h: rows of a tile, for the kernel that cuts views into lower pieces.)
__device__ __forceinline__ Job decode_job(const RenderParams& P, unsigned id, int tile_h = TILE) {
    const unsigned vrel = divide(id, P.div_tiles);
    const unsigned v = (unsigned)P.view_first + vrel;         // E * A * K < 2^31 (checked by the launcher)
    Job j;
    j.tile = (int)(id - vrel * (unsigned)(P.tiles_x * P.tiles_y));
    j.view = (size_t)v;
    const unsigned va = divide(v, P.div_K);
    j.k = (int)(v - va * (unsigned)P.K);
    j.e = (int)divide(va, P.div_A);
    j.a = (int)(va - (unsigned)j.e * (unsigned)P.A);
    const int ty = (int)divide((unsigned)j.tile, P.div_tiles_x);
    j.t.x0 = (j.tile - ty * P.tiles_x) * TILE; j.t.y0 = ty * tile_h;
    j.t.tw = min(TILE, P.W - j.t.x0); j.t.th = min(tile_h, P.H - j.t.y0);
    j.t.w_near = P.w_near; j.t.w_far = P.w_far; j.t.near_z = P.near_z; j.t.far_z = P.far_z;
    return j;
}

// The job CTA i of a launch takes where the tiles with the horizon of all views come first, then the rows below, the sky last, so that
// the last CTAs to come in are not the ones that take longest.
__device__ __forceinline__ unsigned horizon_first(const RenderParams& P, unsigned i) {
    const unsigned tiles = (unsigned)(P.tiles_x * P.tiles_y), pos = divide(i, P.div_views), view = i - pos * divide(P.n_jobs, P.div_tiles);
    const unsigned t = pos + (unsigned)(P.H / (2 * TILE) * P.tiles_x);
    return view * tiles + (t < tiles ? t : t - tiles);
}

// Ray coordinates of tile column / row i, 0..63.
__device__ __forceinline__ float ray_column(const RenderParams& P, const Job& j, int i) { return __ldg(P.rig.ray_x + (size_t)j.k * ray_stride(P.W) + j.t.x0 + i); }
__device__ __forceinline__ float ray_row(const RenderParams& P, const Job& j, int i) { return __ldg(P.rig.ray_y + (size_t)j.k * ray_stride(P.H) + j.t.y0 + i); }
template <class S>
__device__ __forceinline__ void load_rays(S& s, const RenderParams& P, const Job& j, int i) {
    s.ray_x[i] = ray_column(P, j, i);
    s.ray_y[i] = ray_row(P, j, i);
}

// A whole tile rendered by the CTA in barrier-separated phases with per-round lists: any number of
// groups, boxes, survivors and records.  It serves the tiles that a render kernel's lists cannot hold.
template <class TL, int NT>
__device__ __forceinline__ void cooperative_job(TileSmem& s, const RenderParams& P, unsigned job_id, TL& n) {
    const Job job = decode_job(P, job_id);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool classify = !(P.debug_flags & 1);
    const int rec_cap = (P.debug_flags & 2) ? 2 : RCAP;
    const int k = job.k, a = job.a, e = job.e;
    const size_t view = job.view;
    const TileCtx t = job.t;
    const bool ego_active = P.agents[(size_t)e * P.A + a].active != 0;
    // issued now so that their latency overlaps the prologue: the map of this environment, the
    // group box this lane tests first, and the background of the two rows this thread stores
    const MapInfo mi = P.env_maps[e];
    Node gn0;
    gn0.first = 0; gn0.count = 0;
    if (lane < GROUP_BATCH && mi.group_begin + lane < mi.group_end) gn0 = P.groups[mi.group_begin + lane];

    // ---- prologue: camera, ray tables, frustum planes, cleared keys
    if (threadIdx.x < 7) {
        Cam c;
        load_camera(c, P.cams[view], P.cam[k], P.W, P.H);
        if (threadIdx.x == 6) {
            s.cam = c;
            s.n_rec = 0; s.n_leaf = 0; s.n_face = 0; s.n_surv = 0;
            s.touched[0] = 0u; s.touched[1] = 0u;
        } else {
            tile_planes(s, threadIdx.x, c, t);
        }
    } else if (threadIdx.x >= 64 && threadIdx.x < 64 + TILE) {
        load_rays(s, P, job, threadIdx.x - 64);
    }
#pragma unroll
    for (int i = 0; i < TILE * TILE / 2 / NT; ++i)
        reinterpret_cast<ulonglong2*>(s.key)[i * NT + threadIdx.x] = make_ulonglong2(0ull, 0ull);
    __syncthreads();

    if (ego_active) {
        const Cam& c = s.cam;
        const uint32_t n_groups = mi.group_end - mi.group_begin;
        const int n_rounds = max((int)((n_groups + GROUP_BATCH - 1) / GROUP_BATCH), (P.A + BOX_ROUND - 1) / BOX_ROUND);
        for (int round = 0; round < n_rounds; ++round) {
            // ---- phase 1 (a): hierarchy and boxes of this round
            const uint32_t g0 = mi.group_begin + (uint32_t)round * GROUP_BATCH;
            if (g0 < mi.group_end) {
                const uint32_t g = g0 + lane;
                bool vis = false;
                Node gn;
                if (lane < GROUP_BATCH && g < mi.group_end) { gn = (round == 0) ? gn0 : P.groups[g]; vis = box_visible(s, gn); if (warp == 0) ++n.grp; }
                unsigned gm = __ballot_sync(0xffffffffu, vis);
                // warp w takes the visible groups w, w + NT / 32, ...
                for (int i = 0; gm; gm &= gm - 1, ++i) {
                    if ((i & (NT / 32 - 1)) != warp) continue;
                    const int src = __ffs(gm) - 1;
                    const uint32_t first = __shfl_sync(0xffffffffu, gn.first, src);
                    const uint32_t cnt = __shfl_sync(0xffffffffu, gn.count, src);
                    bool lvis = false;
                    Node lf;
                    if (lane < (int)cnt) { lf = P.leaves[first + lane]; lvis = box_visible(s, lf); ++n.leaf; }
                    const unsigned lm = __ballot_sync(0xffffffffu, lvis);
                    int base = 0;
                    if (lane == 0 && lm) base = atomicAdd(&s.n_leaf, __popc(lm));
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (lvis) s.leaf[base + __popc(lm & ((1u << lane) - 1u))] = (lf.first << 4) | lf.count;
                }
            }
            // boxes are taken from the last thread down: the first warps are busier with the visible groups
            for (int b = round * BOX_ROUND + (NT - 1 - (int)threadIdx.x); b < min(P.A, (round + 1) * BOX_ROUND); b += NT) {
                if (b == a) continue;
                const AgentGeom g = P.agents[(size_t)e * P.A + b];
                if (!g.active) continue;
                uint32_t faces = box_faces(s, c, t, g);
                if (!faces) continue;
                int slot = atomicAdd(&s.n_face, __popc(faces));
                for (; faces; faces &= faces - 1) s.face[slot++] = ((uint32_t)b << 3) | (uint32_t)(__ffs(faces) - 1);
            }
            __syncthreads();
            // ---- phase 2a (a): one thread per candidate: camera space, pixel box; survivors are compacted
            const int nl = s.n_leaf, nf = s.n_face;
            const int n_items = nl * LEAF_PRIMS + nf;
            for (int i0 = 0; i0 < n_items; i0 += NT) {
                const int i = i0 + threadIdx.x;
                V3 V[4], Pn;
                uint32_t key_lo, flags, box = 0;
                bool keep = false;
                if (i < n_items && fetch_candidate(s, P, i, nl, e, mi.n_tris, V, Pn, key_lo, flags, false)) {
                    ++n.tested;
                    keep = pixel_box(c, t, V, box);
                }
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&s.n_surv, __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (keep) {
                    const int slot = base + __popc(m & ((1u << lane) - 1u));
                    if (slot < SCAP) s.surv[slot] = make_uint2((uint32_t)i, box);
                    else {                                                                  // list full (rare)
                        fetch_candidate(s, P, i, nl, e, mi.n_tris, V, Pn, key_lo, flags, true);
                        setup_prim(s, t, V, flags & 1u, flags, Pn, key_lo, box, rec_cap, n);
                    }
                }
            }
            __syncthreads();
            // ---- phase 2b (c): one thread per survivor: edge functions, 1/z plane, tiny raster or record
            const int ns = min(s.n_surv, SCAP);
            for (int j = threadIdx.x; j < ns; j += NT) {
                const uint2 sv = s.surv[j];
                V3 V[4], Pn;
                uint32_t key_lo, flags;
                fetch_candidate(s, P, (int)sv.x, nl, e, mi.n_tris, V, Pn, key_lo, flags, true);
                setup_prim(s, t, V, flags & 1u, flags, Pn, key_lo, sv.y, rec_cap, n);
            }
            __syncthreads();
            if (round + 1 < n_rounds) {
                // the lists are reused by the next round; records are rasterized now if they might overflow
                const int n_rec = min(s.n_rec, rec_cap);
                if (n_rec > rec_cap / 2) raster_records<NT / 32>(s, s.rec, s.touched, t, n_rec, classify, n);
                __syncthreads();
                if (threadIdx.x == 0) { s.n_leaf = 0; s.n_face = 0; s.n_surv = 0; if (n_rec > rec_cap / 2) s.n_rec = 0; }
                __syncthreads();
            }
        }
        // ---- phase 3 (b)+(c): one warp per record
        raster_records<NT / 32>(s, s.rec, s.touched, t, min(s.n_rec, rec_cap), classify, n);
        __syncthreads();
    }
    // ---- phase 4 (d)
    store_tile(s, t, P, view, k, ego_active, ((unsigned long long)s.touched[1] << 32) | s.touched[0], threadIdx.x, NT, mi.n_tris);
    if (threadIdx.x == 0) { ++n.jobs; ++n.coop; }
}

// Adds the CTA's tallies to the optional counters: [0] tiles, [1..9] group tests, leaf tests,
// candidates tested, set up, rasterized by their thread, records, record-list overflows, records
// classified per cell, cells visited, [10] tiles rendered by cooperative_job.
__device__ __forceinline__ void flush_counters(const RenderParams&, const NoTally&) {}
__device__ __forceinline__ void flush_counters(const RenderParams& P, const Tally& n) {
    const int lane = threadIdx.x & 31;
    const int vals[11] = {n.jobs, n.grp, n.leaf, n.tested, n.setup, n.tiny, n.recs, n.fallback, n.classified, n.cells, n.coop};
#pragma unroll
    for (int i = 0; i < 11; ++i) {
        // classified / cells are counted by every lane of a warp alike
        const int v = ((i == 8 || i == 9) && lane != 0) ? 0 : vals[i];
        const int sum = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0 && sum) atomicAdd(&P.counters[i], (unsigned long long)sum);
    }
}

// ---------------------------------------------------------------------------------------------
// Cull kernel, and the render kernels over its survivor lists (see the head of this file).
// ---------------------------------------------------------------------------------------------
constexpr int W_ITEM = 448;        // items of a tile or view tested at a time in the cull kernel
static_assert(W_ITEM >= 32 * LARGE_LEAF_PRIMS && W_ITEM >= 32 * 6, "what a pass over the leaves or the boxes can add fits an empty list");
// Survivor buffer, SURV_STRIDE uint2 per tile: a 16-byte head (number of survivors, or all ones if there are more than
// W_SURV; work counts), then W_SURV entries (id, pixel box).
constexpr int SURV_STRIDE = 256;
constexpr int W_SURV = SURV_STRIDE - 2;
constexpr uint32_t SURV_OVERFLOW = 0xffffffffu;
constexpr uint32_t SURV_FACE = 0x80000000u;   // survivor id: index into grid_prims, or SURV_FACE | agent << 3 | face
constexpr uint32_t REC_TINY = 1u << 28, REC_DEAD = 1u << 29;   // flags in the box word of a record

// A tile's frustum and its footprint on the ground plane.
struct __align__(16) Frustum {
    float plane[6][4];                        // (read as float4: kept first, 16-byte aligned)
    float side[4][4];
    Cam cam;
    float seg[10][6];                         // footprint segments: x, y, dx, dy, 1 / dy, unused
    float pt[5][2];                           // footprint corners (ego-relative xy): apex, four far corners
    int n_seg;                                // segments to look at: 3 for a camera without pitch (the corners coincide in pairs), else 10
};
static_assert(offsetof(Frustum, plane) % 16 == 0 && offsetof(Frustum, side) % 16 == 0, "planes are read with 128-bit loads");

struct __align__(16) FrontLists {
    Frustum f;
    uint32_t item[W_ITEM];                    // survivor ids to be tested
    uint32_t row_base[32];                    // grid rows of a pass that have candidates: first entry of the row's range in grid_prims less the candidates before it
};

// Box test against planes held in registers (see box_visible).
__device__ __forceinline__ bool box_visible_reg(const float4 (&pl)[6], float px, float py, const Node& b) {
    const float ax = sub(b.lo[0], px), bx = sub(b.hi[0], px);
    const float ay = sub(b.lo[1], py), by = sub(b.hi[1], py);
    const float cx = 0.5f * (ax + bx), cy = 0.5f * (ay + by), cz = 0.5f * (b.lo[2] + b.hi[2]);
    const float hx = 0.5f * (bx - ax), hy = 0.5f * (by - ay), hz = 0.5f * (b.hi[2] - b.lo[2]);
    const float slack = 1e-3f + 4e-6f * (fabsf(cx) + fabsf(cy) + fabsf(cz) + hx + hy + hz);
    bool vis = true;
#pragma unroll
    for (int p = 0; p < 6; ++p) {
        const float dist = pl[p].x * cx + pl[p].y * cy + pl[p].z * cz + pl[p].w;
        const float reach = fabsf(pl[p].x) * hx + fabsf(pl[p].y) * hy + fabsf(pl[p].z) * hz;
        vis = vis && (dist + reach >= -slack);
    }
    return vis;
}

__device__ __forceinline__ Node load_node(const Node* p) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    Node nd;
    nd.lo[0] = a.x; nd.lo[1] = a.y; nd.lo[2] = a.z; nd.first = __float_as_uint(a.w);
    nd.hi[0] = b.x; nd.hi[1] = b.y; nd.hi[2] = b.z; nd.count = __float_as_uint(b.w);
    return nd;
}

__device__ __forceinline__ AgentGeom load_agent(const AgentGeom* p) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    AgentGeom g;
    g.x = a.x; g.y = a.y; g.c = a.z; g.s = a.w; g.hl = b.x; g.hw = b.y; g.h = b.z; g.active = __float_as_uint(b.w);
    return g;
}

// Warp-wide append to the survivor list (a slot past the end is not written; the caller checks the total).
__device__ __forceinline__ void append_survivor(uint2* __restrict__ surv, bool keep, uint32_t id, uint32_t box, int& n, int lane) {
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep) { const int slot = n + __popc(m & ((1u << lane) - 1u)); if (slot < W_SURV) surv[slot] = make_uint2(id, box); }
    n += __popc(m);
}

// Pixel box of camera-space vertices in a whole image, inclusive; false: no pixel centre (margin m) can be touched.  Where
// pixel_box gives up because a vertex lies behind or close to the camera, the primitive is cut a little before the near depth --
// nothing nearer is kept -- and what remains is projected, so that a road under the camera reaches only the tiles it is seen in.
//
// The box has to hold every pixel that the edge functions and the 1/z plane, as they are evaluated, let through.  Against the exact
// polygon, with L the largest vertex distance, h the plane's distance from the camera, and focal length f in pixels:
//   1/z is off by 5e-7 L / h of itself: within the 1 % before the near depth while L / h <= 1e4;
//   an edge function carries some 5 roundings of |V| |edge|, which moves its line by shift = 3e-7 f L / h pixels, and the corner
//     of two lines by a few times that (8: down to an angle of a quarter; a thinner tip is narrower than the shift);
//   the cut of an edge is off by 8 roundings of the edge's length, f |edge| / near times that in pixels (twice that is allowed, L
//     being taken as a sum of three components and an edge as 2 L).
// A plane too close to the camera for this (an edge-on one) keeps the whole image as its box.
__device__ __forceinline__ bool view_box(const Cam& c, const TileCtx& t, const V3 (&V)[4], int& bx0, int& by0, int& bx1, int& by1, float m) {
    bool ok = pixel_box_int(c, t, V, bx0, by0, bx1, by1, m);
    if (ok && fminf(fminf(V[0].z, V[1].z), fminf(V[2].z, V[3].z)) < t.near_z * ZPROJ_FRAC) {
        float reach = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) reach = fmaxf(reach, fabsf(V[i].x) + fabsf(V[i].y) + fabsf(V[i].z));
        const V3 n = plane_normal(V, true);                  // (of a triangle too: its third vertex is there twice)
        const float ratio = fast_div(reach * sqrtf(vdot(n, n)), fabsf(vdot(n, V[0])));      // L / h
        const float zc = t.near_z * 0.99f, izc = fast_rcp(zc), f = fmaxf(c.focx, c.focy), shift = 3e-7f * f * ratio;
        if (ratio <= 1e4f && shift <= 0.5f) {
            const float mm = m + 0.25f + 8.f * shift + 2e-6f * f * reach * izc;               // (an edge is at most 2 L)
            float sx0 = 3e38f, sx1 = -3e38f, sy0 = 3e38f, sy1 = -3e38f;
            auto include = [&](float x, float y, float iz) {
                const float sx = fm(c.focx, mul(x, iz), c.cx), sy = fm(c.focy, mul(y, iz), c.cy);
                sx0 = fminf(sx0, sx); sx1 = fmaxf(sx1, sx); sy0 = fminf(sy0, sy); sy1 = fmaxf(sy1, sy);
            };
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const V3 a = V[i], b = V[(i + 1) & 3];
                if (a.z >= zc) include(a.x, a.y, fast_rcp(a.z));
                if ((a.z < zc) != (b.z < zc)) {
                    const float u = fast_div(zc - a.z, b.z - a.z);
                    include(fm(u, b.x - a.x, a.x), fm(u, b.y - a.y, a.y), izc);
                }
            }
            const float fx0 = fmaxf(ceilf(sx0 - 0.5f - mm), 0.f), fx1 = fminf(floorf(sx1 - 0.5f + mm), (float)(t.tw - 1));
            const float fy0 = fmaxf(ceilf(sy0 - 0.5f - mm), 0.f), fy1 = fminf(floorf(sy1 - 0.5f + mm), (float)(t.th - 1));
            ok = fx0 <= fx1 && fy0 <= fy1;
            bx0 = (int)fx0; by0 = (int)fy0; bx1 = (int)fx1; by1 = (int)fy1;
        }
    }
    return ok;
}

// Bit per tile (row-major, at most 32 per view) reached by a pixel box of the image.
__device__ __forceinline__ uint32_t box_tiles(const RenderParams& P, int bx0, int by0, int bx1, int by1) {
    const uint32_t cols = (uint32_t)((2ull << (bx1 / TILE)) - (1ull << (bx0 / TILE)));
    uint32_t tiles = 0u;
    for (int ty = by0 / TILE; ty <= by1 / TILE; ++ty) tiles |= cols << (ty * P.tiles_x);
    return tiles;
}

// Appends each lane's survivor to the lists of the tiles it reaches, with its box cut to the tile.  Lane l keeps the count of tile l.
__device__ __forceinline__ void deal_survivors(uint2* __restrict__ surv, const RenderParams& P, uint32_t tiles, uint32_t id, int bx0, int by0, int bx1, int by1,
                                               int& n, int lane) {
#pragma unroll 1
    for (uint32_t any = __reduce_or_sync(0xffffffffu, tiles); any; any &= any - 1) {
        const int tile = __ffs(any) - 1;
        const bool in = (tiles >> tile) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        const int slot = __shfl_sync(0xffffffffu, n, tile) + __popc(m & ((1u << lane) - 1u));
        if (in && slot < W_SURV) {
            const int ty = (int)divide((unsigned)tile, P.div_tiles_x), x0 = (tile - ty * P.tiles_x) * TILE, y0 = ty * TILE;
            const uint32_t box = (uint32_t)max(bx0 - x0, 0) | ((uint32_t)max(by0 - y0, 0) << 8) | ((uint32_t)min(bx1 - x0, TILE - 1) << 16) | ((uint32_t)min(by1 - y0, TILE - 1) << 24);
            surv[(size_t)tile * SURV_STRIDE + slot] = make_uint2(id, box);
        }
        if (lane == tile) n += __popc(m);
    }
}

// Camera, frustum planes and footprint of a part of a view, by one warp.  `entry`: of lane i < FRUSTUM_ENTRIES the part's entry i in
// camera space.  The same rotation turns the normals of the planes and the corners of the footprint.  The footprint is the convex
// hull of the apex and the four far corners, kept as the segments between them (the hull's edges are among them, the others lie
// inside it).
__device__ __forceinline__ void frustum_setup(Frustum& f, const RenderParams& P, const Job& job, const float4 entry, int lane) {
    if (lane < FRUSTUM_ENTRIES) {
        Cam c;
        load_camera(c, P.cams[job.view], P.cam[job.k], P.W, P.H);
        const V3 v = rotate_to_world(c, entry);
        if (lane < 6) {
            *reinterpret_cast<float4*>(f.plane[lane]) = world_plane(c, v, entry.w);
            if (lane >= 2) *reinterpret_cast<float4*>(f.side[lane - 2]) = entry;
        } else {
            f.pt[lane - 6][0] = c.mwx + v.x;
            f.pt[lane - 6][1] = c.mwy + v.y;
        }
        if (lane == 6) {
            f.cam = c;
            f.n_seg = (c.dx == 0.f && c.dy == 0.f) ? 3 : 10;     // no pitch: corners 1, 3 and 2, 4 have the same x, y
        }
    }
    __syncwarp();
    if (lane < 10) {
        const int i = (int)((0x3221100100ull >> (4 * lane)) & 15u), j = (int)((0x4434443221ull >> (4 * lane)) & 15u);   // (0,1) (0,2) (1,2) (0,3) (0,4) (1,3) (1,4) (2,3) (2,4) (3,4)
        const float px = f.pt[i][0], py = f.pt[i][1], dx = f.pt[j][0] - px, dy = f.pt[j][1] - py;
        f.seg[lane][0] = px; f.seg[lane][1] = py; f.seg[lane][2] = dx; f.seg[lane][3] = dy;
        f.seg[lane][4] = fabsf(dy) > 1e-30f ? fast_rcp(dy) : 0.f; f.seg[lane][5] = 0.f;
    }
    __syncwarp();
}
// Lane i's entry of the frustum of a tile, or (tile = number of tiles) of the whole image.
__device__ __forceinline__ float4 frustum_table(const RenderParams& P, const Job& job, int tile, int lane) {
    const int tiles = P.tiles_x * P.tiles_y;
    return lane < FRUSTUM_ENTRIES ? __ldg(P.rig.frusta + (size_t)((job.k * (tiles + 1) + tile) * FRUSTUM_ENTRIES + lane)) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// The grid rows crossed by the footprint, widened by the map's margin.
struct GridRows {
    int lo, hi;             // (within the grid; hi < lo if the footprint misses it)
    float gx0, gy0;         // the grid's corner, ego-relative
};
__device__ __forceinline__ GridRows grid_rows(const Frustum& f, const MapInfo& mi) {
    GridRows g;
    g.gx0 = sub(mi.gx0, f.cam.px); g.gy0 = sub(mi.gy0, f.cam.py);
    float ylo = f.pt[0][1], yhi = ylo;
#pragma unroll
    for (int k = 1; k < 5; ++k) { ylo = fminf(ylo, f.pt[k][1]); yhi = fmaxf(yhi, f.pt[k][1]); }
    const float fr0 = floorf((ylo - mi.margin - g.gy0) * mi.inv_cell), fr1 = floorf((yhi + mi.margin - g.gy0) * mi.inv_cell);
    clamp_rows(fr0, fr1, mi.ny, g.lo, g.hi);
    return g;
}

// The range of grid_prims under the part of grid row `row` that the widened footprint crosses.  (Rounding: the difference, 1 / dy to an ulp and
// the product put t off by less than 4 x 2^-24 of itself, which moves a crossing by less than 3e-7 of its distance from the segment's
// beginning.  From the apex that is 3e-7 of how far away what is looked for is, where the outermost pixel centres lie half a pixel, 0.5 / f of that
// distance, inside the footprint's sides; a segment between far corners lies 0.1 % beyond the far depth.)
__device__ __forceinline__ void row_range(const Frustum& f, const RenderParams& P, const MapInfo& mi, const GridRows& g, int row, uint32_t& first, uint32_t& cnt) {
    first = 0u; cnt = 0u;
    if (row > g.hi) return;
    const float margin = mi.margin, blo = g.gy0 + (float)row * mi.cell - margin, bhi = blo + mi.cell + 2.f * margin;
    float xlo = 3e38f, xhi = -3e38f;
    const int n_seg = f.n_seg;
#pragma unroll 1
    for (int k = 0; k < n_seg; ++k) {
        const float px = f.seg[k][0], py = f.seg[k][1], dx = f.seg[k][2], dy = f.seg[k][3], idy = f.seg[k][4];
        const float ya = fminf(py, py + dy), yb = fmaxf(py, py + dy);
        if (yb >= blo && ya <= bhi) {
            const float ta = (blo - py) * idy, tb = (bhi - py) * idy;
            const float t0 = idy != 0.f ? fminf(fmaxf(fminf(ta, tb), 0.f), 1.f) : 0.f, t1 = idy != 0.f ? fminf(fmaxf(fmaxf(ta, tb), 0.f), 1.f) : 1.f;
            const float xa = px + t0 * dx, xb = px + t1 * dx;
            xlo = fminf(xlo, fminf(xa, xb)); xhi = fmaxf(xhi, fmaxf(xa, xb));
        }
    }
    if (xlo <= xhi) {
        const float fx0 = floorf((xlo - margin - g.gx0) * mi.inv_cell), fx1 = floorf((xhi + margin - g.gx0) * mi.inv_cell);
        if (fx1 >= 0.f && fx0 <= (float)mi.nx - 1.f) {
            const uint32_t ix0 = (uint32_t)fmaxf(fx0, 0.f), ix1 = (uint32_t)fminf(fx1, (float)mi.nx - 1.f);
            const uint32_t* cs = P.cell_start + mi.cell_begin + (uint32_t)row * mi.nx;
            first = __ldg(cs + ix0);
            cnt = __ldg(cs + ix1 + 1) - first;
        }
    }
}

// Can the primitive inside bound `b` touch a pixel centre of the tile (margin m: see pixel_box)?  Conservative: the
// bound's camera-space box is projected as a whole.  On flat maps this decides most candidates: a lane marking beyond
// some twenty metres projects to a sliver between two rows of pixel centres.
__device__ __forceinline__ bool bound_visible(const Cam& c, const TileCtx& t, const float4 b, const float m) {
    const uint32_t size = __float_as_uint(b.w);
    const float r = __uint_as_float(size & 0xffff0000u), hz = __uint_as_float(size << 16);
    const V3 q = to_camera(c, b.x, b.y, b.z);
    const float cphi = fabsf(c.dz), sphi = fabsf(c.fz_);                       // pitch
    const float rz = cphi * r + sphi * hz, ry = sphi * r + cphi * hz;
    const float z0 = q.z - rz, z1 = q.z + rz;
    bool ok = z1 >= t.near_z * 0.9999f && z0 <= t.far_z * 1.0001f;
    if (z0 >= t.near_z * ZPROJ_FRAC) {                                         // (else a vertex may not project: pixel_box looks closer)
        const float i0 = fast_rcp(z0), i1 = fast_rcp(z1);
        const float xa = q.x - r, xb = q.x + r, ya = q.y - ry, yb = q.y + ry;
        const float mm = m + 0.015625f;                                        // 1/64 pixel for the rounding above
        const float sx0 = fm(c.focx, xa * (xa < 0.f ? i0 : i1), c.cx), sx1 = fm(c.focx, xb * (xb < 0.f ? i1 : i0), c.cx);
        const float sy0 = fm(c.focy, ya * (ya < 0.f ? i0 : i1), c.cy), sy1 = fm(c.focy, yb * (yb < 0.f ? i1 : i0), c.cy);
        const float fx0 = fmaxf(ceilf(sx0 - 0.5f - mm), (float)t.x0), fx1 = fminf(floorf(sx1 - 0.5f + mm), (float)(t.x0 + t.tw - 1));
        const float fy0 = fmaxf(ceilf(sy0 - 0.5f - mm), (float)t.y0), fy1 = fminf(floorf(sy1 - 0.5f + mm), (float)(t.y0 + t.th - 1));
        ok = ok && fx0 <= fx1 && fy0 <= fy1;
    }
    return ok;
}

// Front end of one tile by one warp: fills the survivor list and counts its entries in n_surv (those past the list's end are
// not written; the tile then goes to the cooperative kernel, or shows only the background in a colour image).
//
// Map primitives come from the uniform grid: the footprint of the tile's frustum on the ground
// plane is the convex hull of the apex and the four far corners; for every grid row the footprint
// (widened by the map's margin) crosses, the small primitives of the cells it covers are one
// contiguous range of grid_prims.  The ranges of up to 32 rows are laid end to end and their bounds tested two
// candidates per lane at a time; what remains joins a list of items with the primitives of the visible
// large-primitive leaves (a lane per leaf box against the six frustum planes) and the faces of the other agents' boxes
// (culled as bounding spheres).  The items are then tested a lane each -- camera space, pixel box -- and the survivors
// compacted.  Loads that do not depend on one another are issued together.
//
// Bound by the issue of dependent instructions at 24-32 resident warps: the full test costs some 230 instructions and 64
// bytes a candidate, the bound's some 60 and 16, and four candidates in five die by it.
//
// MULTI: the same for all tiles of a view at once (job.t is the whole image): the survivors' pixel boxes are dealt out to the
// lists of the tiles they reach.  A view of several tiles then pays once for its frustum, grid rows, leaves, agents and
// candidates, instead of once per tile.
//
// ROUNDS: where the large primitives and box faces do not fit the item list, as many as do are tested, and a further call goes on
// from leaf l_done and agent b0; returns whether all is done.  Without it the call gives up there (and returns false).  The
// two are separate code (cull_in_rounds) because what a round has to keep over the tests for the next one costs every view
// registers: 14 880 views of 2 tiles take 131 us without rounds, 137 with them inside, 131 like this; a step of 262 144 views of one
// tile 2 439, 2 557, 2 430.
template <class TL, bool CONS, bool MULTI, bool ROUNDS>
__device__ __forceinline__ bool front_cull(FrontLists& f, uint2* __restrict__ surv, const RenderParams& P, const Job& job,
                                           const MapInfo& mi, uint32_t& l_done, int& b0, int& n_surv, int lane, TL& n) {
    // CONS: conservative pixel boxes -- every pixel whose unit square a primitive touches (antialiased output)
    constexpr float BOX_MARGIN = CONS ? 0.50390625f : 0.00390625f;
    const TileCtx& t = job.t;
    const AgentGeom* env_agents = P.agents + (size_t)job.e * P.A;
    uint32_t l0 = mi.large_begin + l_done;
    Node ln0;
    ln0.first = 0; ln0.count = 0;
    if (l0 + lane < mi.large_end) ln0 = load_node(P.large_leaves + l0 + lane);
    AgentGeom ag0, ag1;
    ag0.active = 0u; ag1.active = 0u;
    if (b0 + lane < P.A) ag0 = load_agent(env_agents + b0 + lane);
    if (b0 + lane + 32 < P.A) ag1 = load_agent(env_agents + b0 + lane + 32);
    Frustum& fr = f.f;
    frustum_setup(fr, P, job, frustum_table(P, job, MULTI ? P.tiles_x * P.tiles_y : job.tile, lane), lane);
    const Cam& c = fr.cam;
    const unsigned below = (1u << lane) - 1u;
    int n_item = 0;                                // (entries are appended in order of lane, so that a call's lists are the same every time)
    // ---- the grid rows crossed by the widened footprint; the first 32 rows' ranges are requested now, the boxes below
    // are tested while the loads are under way
    const GridRows rows = grid_rows(fr, mi);
    uint32_t first, cnt;
    row_range(fr, P, mi, rows, rows.lo + lane, first, cnt);
    // ---- the large primitives' leaves: a lane per leaf box against the six frustum planes
    {
        float4 pl[6];
#pragma unroll
        for (int p = 0; p < 6; ++p) pl[p] = *reinterpret_cast<const float4*>(fr.plane[p]);
        while (l0 < mi.large_end) {
            const bool vis = l0 + lane < mi.large_end && box_visible_reg(pl, c.px, c.py, ln0);
            const unsigned m = __ballot_sync(0xffffffffu, vis);
            const int sum = (int)__reduce_add_sync(0xffffffffu, vis ? ln0.count : 0u);
            if (n_item + sum > W_ITEM) break;
            if (vis) {
                const int slot = n_item + LARGE_LEAF_PRIMS * __popc(m & below);     // (only a map's last leaf may be shorter)
                for (uint32_t k = 0; k < ln0.count; ++k) f.item[slot + k] = ln0.first + k;
            }
            n_item += sum;
            if (l0 + lane < mi.large_end) ++n.leaf;
            l0 += 32;
            if (l0 + lane < mi.large_end) ln0 = load_node(P.large_leaves + l0 + lane);
        }
    }
    // ---- other agents' boxes, a lane each, two passes requested at a time
    const int b_start = b0;
#pragma unroll 1
    for (; l0 >= mi.large_end && b0 < P.A; b0 += 32) {
        const bool second = (b0 - b_start) & 32;
        if (!second && b0 != b_start) {
            ag0.active = 0u; ag1.active = 0u;
            if (b0 + lane < P.A) ag0 = load_agent(env_agents + b0 + lane);
            if (b0 + lane + 32 < P.A) ag1 = load_agent(env_agents + b0 + lane + 32);
        }
        const AgentGeom g = second ? ag1 : ag0;
        uint32_t faces = 0u;
        if (b0 + lane != job.a && g.active) faces = box_faces(fr, c, t, g);
        if (__any_sync(0xffffffffu, faces != 0u)) {
            // (a sum over the lanes below of numbers up to 6, bit by bit)
            const int k = __popc(faces);
            const unsigned m1 = __ballot_sync(0xffffffffu, k & 1), m2 = __ballot_sync(0xffffffffu, k & 2), m4 = __ballot_sync(0xffffffffu, k & 4);
            const int sum = __popc(m1) + 2 * __popc(m2) + 4 * __popc(m4);
            if (n_item + sum > W_ITEM) break;
            int slot = n_item + __popc(m1 & below) + 2 * __popc(m2 & below) + 4 * __popc(m4 & below);
            for (; faces; faces &= faces - 1, ++slot) f.item[slot] = SURV_FACE | ((uint32_t)(b0 + lane) << 3) | (uint32_t)(__ffs(faces) - 1);
            n_item += sum;
        }
    }
    const bool boxes_done = l0 >= mi.large_end && b0 >= P.A;
    if (!ROUNDS && !boxes_done) return false;
    l_done = l0 - mi.large_begin;
    // ---- fill the item list with the candidates of the grid rows (32 rows per pass), test the items, until both are done
    int row = rows.lo, i0 = 0, total = -1, rows_seen = 0;    // total < 0: the ranges of the pass have not been laid out; rows_seen: begun before candidate i0
    uint32_t row_at = 0u;                          // number of candidates before the lane's row (beyond all if it has none)
    bool more = boxes_done && row <= rows.hi;
    if (more && row + lane <= rows.hi) ++n.grp;
#pragma unroll 1
    do {
        while (more && n_item <= W_ITEM - 64) {
            if (total < 0) {
                if (row != rows.lo) {
                    row_range(fr, P, mi, rows, row + lane, first, cnt);
                    if (row + lane <= rows.hi) ++n.grp;
                }
                uint32_t incl = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += up;
                }
                total = (int)__shfl_sync(0xffffffffu, incl, 31);
                __syncwarp();
                const unsigned any = __ballot_sync(0xffffffffu, cnt > 0u);
                row_at = cnt > 0u ? incl - cnt : 0x7fffffffu;
                if (cnt > 0u) f.row_base[__popc(any & below)] = first - row_at;
                __syncwarp();
                i0 = 0;
                rows_seen = 0;
            }
            if (i0 < total) {
                float4 b[2];
                uint32_t id[2] = {0u, 0u};
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int i = i0 + 32 * u + lane;
                    b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    // (the rows that begin at one of these 32 candidates, a bit each: a candidate's row is the number of rows begun so far)
                    const uint32_t at = row_at - (uint32_t)(i0 + 32 * u), starts = __reduce_or_sync(0xffffffffu, at < 32u ? 1u << at : 0u);
                    const int r = rows_seen + __popc(starts & (below | (1u << lane))) - 1;
                    rows_seen += __popc(starts);
                    if (i < total) {
                        id[u] = f.row_base[r] + (uint32_t)i;
                        b[u] = __ldg(reinterpret_cast<const float4*>(P.grid_bounds) + id[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const bool have = i0 + 32 * u + lane < total;
                    const bool keep = have && bound_visible(c, t, b[u], BOX_MARGIN);
                    const unsigned m = __ballot_sync(0xffffffffu, keep);
                    if (keep) f.item[n_item + __popc(m & below)] = id[u];
                    n_item += __popc(m);
                }
                i0 += 64;
            }
            if (i0 >= total) { row += ROW_PASS; total = -1; more = row <= rows.hi; }
        }
        __syncwarp();
#pragma unroll 1
        for (int i = lane; i - lane < n_item; i += 32) {
            uint32_t box = 0, id = 0, tiles = 0;                // tiles: bit per tile of the view that the box reaches
            int bx0 = 0, by0 = 0, bx1 = -1, by1 = -1;
            bool keep = false;
            if (i < n_item) {
                id = f.item[i];
                V3 V[4];
                if (id & SURV_FACE) {
                    const AgentGeom g = load_agent(env_agents + ((id & ~SURV_FACE) >> 3));
                    const uint32_t corners = face_corners((int)(id & 7u));
#pragma unroll
                    for (int q = 0; q < 4; ++q) V[q] = box_corner(c, g, (corners >> (4 * q)) & 7u);
                } else {
                    float v[12];
                    uint32_t key_lo, flags;
                    load_prim(P.grid_prims + id, v, key_lo, flags);
#pragma unroll
                    for (int q = 0; q < 4; ++q) V[q] = to_camera(c, v[3 * q], v[3 * q + 1], v[3 * q + 2]);
                }
                ++n.tested;
                if (MULTI) {
                    if (view_box(c, t, V, bx0, by0, bx1, by1, BOX_MARGIN)) tiles = box_tiles(P, bx0, by0, bx1, by1);
                } else {
                    keep = pixel_box(c, t, V, box, BOX_MARGIN);
                }
            }
            if (MULTI) deal_survivors(surv, P, tiles, id, bx0, by0, bx1, by1, n_surv, lane);
            else append_survivor(surv, keep, id, box, n_surv, lane);
        }
        __syncwarp();
        n_item = 0;
    } while (more);
    return boxes_done;
}

// The views (or tiles) in which more large primitives and box faces are in sight than the item list holds: in rounds, from the
// start.  Returns the number of survivors.
template <class TL, bool CONS, bool MULTI>
__device__ __noinline__ int cull_in_rounds(FrontLists& f, uint2* __restrict__ surv, const RenderParams& P, unsigned id, int lane, TL& n) {
    Job job = decode_job(P, id);
    if (MULTI) { job.t.tw = P.W; job.t.th = P.H; }
    const MapInfo mi = P.env_maps[job.e];
    n.leaf = 0;                                 // (they are looked at again)
    uint32_t l_done = 0;
    int b0 = 0, ns = 0;
#pragma unroll 1
    while (!front_cull<TL, CONS, MULTI, true>(f, surv, P, job, mi, l_done, b0, ns, lane, n)) {}
    return ns;
}

// Survivor `id` in camera space with its plane normal.
__device__ __forceinline__ void fetch_survivor(const Cam& c, const RenderParams& P, uint32_t id, int e, uint32_t n_map_tris,
                                               V3 (&V)[4], V3& Pn, uint32_t& key_lo, uint32_t& flags) {
    if (!(id & SURV_FACE)) {
        float v[12], vis_cos;
        load_prim(P.grid_prims + id, v, key_lo, flags, vis_cos);
#pragma unroll
        for (int q = 0; q < 4; ++q) V[q] = to_camera(c, v[3 * q], v[3 * q + 1], v[3 * q + 2]);
        Pn = limit_angular_range(V, plane_normal_world(c, v, flags & 1u), vis_cos);
    } else {
        const int b = (int)((id & ~SURV_FACE) >> 3), f = (int)(id & 7u);
        const AgentGeom g = P.agents[(size_t)e * P.A + b];
        const uint32_t corners = face_corners(f);
#pragma unroll
        for (int q = 0; q < 4; ++q) V[q] = box_corner(c, g, (corners >> (4 * q)) & 7u);
        key_lo = ((0xFFFFFFu - (n_map_tris + 12u * (uint32_t)b + 2u * (uint32_t)f)) << 8) | agent_box_class(g);
        flags = face_flags(corners);
        Pn = plane_normal(V, true);
    }
}

// A covered pixel's depth lies between the vertices' depths; with a margin far above the rounding
// of the 1/z plane, vertices well inside [near, far] make the per-pixel range test redundant.
__device__ __forceinline__ bool record_in_range(const V3 (&V)[4], const RenderParams& P) {
    const float zlo = fminf(fminf(V[0].z, V[1].z), fminf(V[2].z, V[3].z)), zhi = fmaxf(fmaxf(V[0].z, V[1].z), fmaxf(V[2].z, V[3].z));
    return zlo >= P.near_z * 1.001f && zhi <= P.far_z * 0.999f;
}

// Cull kernel: a warp per tile walks the grid and the other agents' boxes, tests the candidates
// and leaves the tile's survivors (id, pixel box) in device memory: a 16-byte head (count, or -1 if they
// do not fit; with counters, the tile's row / leaf / candidate tests), then the list.  No
// CTA-wide synchronisation.  The lists are small (about 250 bytes per view on the benchmark
// workload) and are read back by the render kernel that follows on the stream.
struct __align__(16) CullSmem {
    FrontLists lists[NW];
};

constexpr int CULL_CTAS = 7;       // CTAs per multiprocessor the cull kernel's registers are bounded for (8 192 agents, a tile per view: 5 256.8, 6 248.7, 7 243.4, 8 245.1 us; views of 8 tiles: 662.5, 659.4, 656.5, 660.5)
// MULTI: a warp per view of several tiles (P.n_jobs counts tiles all the same).
template <class TL, bool CONS, bool MULTI = false>
__global__ void __launch_bounds__(NTHREADS, CULL_CTAS) cull_kernel(const __grid_constant__ RenderParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CullSmem& s = *reinterpret_cast<CullSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned cta = await_previous(blockIdx.x);
    const int tiles = MULTI ? P.tiles_x * P.tiles_y : 1;
    const unsigned id = (cta * (unsigned)NW + warp) * (unsigned)tiles;
    if (id >= P.n_jobs) return;
    TL n = {};
    uint2* blk = P.surv + (size_t)id * SURV_STRIDE;
    int ns = 0;
    if (P.debug_flags & 4) {
        ns = -1;                                // test aid: every tile through cooperative_job
    } else {
        Job job = decode_job(P, id);
        if (MULTI) { job.t.tw = P.W; job.t.th = P.H; }
        const MapInfo mi = P.env_maps[job.e];
        const bool ego_active = P.agents[(size_t)job.e * P.A + job.a].active != 0;
        uint32_t l_done = 0;
        int b0 = 0;
        if (ego_active && !front_cull<TL, CONS, MULTI, false>(s.lists[warp], blk + 2, P, job, mi, l_done, b0, ns, lane, n))
            ns = cull_in_rounds<TL, CONS, MULTI>(s.lists[warp], blk + 2, P, id, lane, n);
        if (ns > W_SURV) ns = -1;               // (MULTI: of the tile of this lane)
    }
    // (the work counts are summed over the warp's lanes; without counters they are constants)
    const uint32_t c_grp = __reduce_add_sync(0xffffffffu, (uint32_t)tally_value(n.grp)), c_leaf = __reduce_add_sync(0xffffffffu, (uint32_t)tally_value(n.leaf)),
                   c_tested = __reduce_add_sync(0xffffffffu, (uint32_t)tally_value(n.tested));
    if (lane < tiles) *reinterpret_cast<uint4*>(blk + (size_t)lane * SURV_STRIDE) = make_uint4((uint32_t)ns, c_grp, c_leaf, c_tested);
    // (only now: blocks of the next kernel that came in earlier would crowd the multiprocessors that still have room
    // instead of spreading over all of them)
    launch_dependents();
}

// The tiles the render kernels left out, a CTA at a time.  (Called from the end of those kernels instead, the same code
// costs them 2 % -- a call bounds their registers -- which is more than a launch that overlaps their last blocks.)
template <class TL>
__global__ void __launch_bounds__(NTHREADS, 5) cooperative_kernel(const __grid_constant__ RenderParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem& cs = *reinterpret_cast<TileSmem*>(smem_raw);
    const unsigned cta = await_previous(blockIdx.x);
    TL n = {};
    const unsigned count = __ldcg(&P.overflow[0]);
    for (unsigned i = cta; i < count; i += gridDim.x) {
        cooperative_job<TL, NTHREADS>(cs, P, __ldcg(&P.overflow[1u + i]), n);
        __syncthreads();
    }
    flush_counters(P, n);
}

cudaError_t configure_small_kernel();

cudaError_t configure_render_kernel() {
    cudaError_t err = configure_small_kernel();
    if (err != cudaSuccess) return err;
    err = cudaFuncSetAttribute(cooperative_kernel<NoTally>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSmem));
    if (err != cudaSuccess) return err;
    return cudaFuncSetAttribute(cooperative_kernel<Tally>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TileSmem));
}

// ---------------------------------------------------------------------------------------------
// Coverage kernel (only with the occlusion option): for every view and every other active agent,
// the pixels at which that agent's box, drawn alone, leaves a kept fragment.  Only coverage counts, so there is no
// z-buffer and no need for tiles: a warp takes a band of 16 rows of a view.  The agents are culled as
// spheres, a lane each; the visible ones' faces are set up four agents at a time, eight lanes per agent of which six have a
// face; then the agents are counted one after the other, four pixels per lane at a time of the box around the agent's faces.  Bound by
// instruction issue.  (A warp per tile that set up and drew one face of one agent after the other took 299 us for 4 096 views
// of 100 x 70 pixels and 64 agents; one pixel per lane at a time instead of four, and the bands in order, 81 us where it now takes 66.)  The arithmetic that decides a pixel is the production kernels' (pic_device.cuh).
// ---------------------------------------------------------------------------------------------
struct __align__(16) CoverWarp {
    float4 edge[4][32], w[32];                // faces of the batch by lane: edge functions with their thresholds, 1/z plane
    Frustum f;
    uint32_t agent[32];                       // visible agents of a pass: agent << 8 | faces to draw
};

__global__ void __launch_bounds__(32) coverage_kernel(const __grid_constant__ RenderParams P, unsigned n_views, int bands, int band_rows) {
    __shared__ CoverWarp s;
    const int lane = threadIdx.x;
    // (the band with the horizon of all views first: all agents in view are in it, and the last warps to come in have little to do)
    const unsigned pos = blockIdx.x / n_views, vrel = blockIdx.x - pos * n_views, band = (pos + (unsigned)(P.H / 2 / band_rows)) % (unsigned)bands;
    const unsigned v = (unsigned)P.view_first + vrel, va = divide(v, P.div_K);
    Job job;
    job.view = v;
    job.k = (int)(v - va * (unsigned)P.K);
    job.e = (int)divide(va, P.div_A);
    job.a = (int)(va - (unsigned)job.e * (unsigned)P.A);
    job.tile = 0;
    TileCtx& t = job.t;
    t.x0 = 0; t.tw = P.W; t.y0 = (int)band * band_rows; t.th = min(band_rows, P.H - t.y0);
    t.w_near = P.w_near; t.w_far = P.w_far; t.near_z = P.near_z; t.far_z = P.far_z;
    const AgentGeom* env_agents = P.agents + (size_t)job.e * P.A;
    if (!env_agents[job.a].active) return;
    const float cx = 0.5f * (float)P.W, cy = 0.5f * (float)P.H;
    frustum_setup(s.f, P, job, frustum_entry(lane, -cx, (float)P.W - cx, (float)t.y0 - cy, (float)(t.y0 + t.th) - cy, P.cam[job.k].fx, P.cam[job.k].fy, t.near_z, t.far_z), lane);
    const Cam& c = s.f.cam;
    const float* ray_x = P.rig.ray_x + (size_t)job.k * ray_stride(P.W);
    const float* ray_y = P.rig.ray_y + (size_t)job.k * ray_stride(P.H) + t.y0;
    uint32_t* occ = P.occlusion + job.view * (size_t)P.A * 2u;
    for (int b0 = 0; b0 < P.A; b0 += 32) {
        uint32_t draw = 0u;
        if (b0 + lane < P.A && b0 + lane != job.a) {
            const AgentGeom g = load_agent(env_agents + b0 + lane);
            if (g.active) draw = box_faces(s.f, c, t, g);             // 0: its bounding sphere misses the frustum
            // (box_faces leaves faces out only where the box lies beyond near; those turned away add no pixel then, unless
            // the facing ones reach beyond far)
            const float reach = sqrtf((g.x - c.px - c.mwx) * (g.x - c.px - c.mwx) + (g.y - c.py - c.mwy) * (g.y - c.py - c.mwy)) + g.hl + g.hw + g.h;
            if (draw && !(reach < t.far_z * 0.99f)) draw = 0x3fu;
        }
        const unsigned m = __ballot_sync(0xffffffffu, draw != 0u);
        const int n_vis = __popc(m);
        if (draw) s.agent[__popc(m & ((1u << lane) - 1u))] = (uint32_t)(b0 + lane) << 8 | draw;
        __syncwarp();
        for (int j0 = 0; j0 < n_vis; j0 += 4) {
            const int j = j0 + (lane >> 3), face = lane & 7;
            int bx0 = 0x7fffffff, by0 = 0x7fffffff, bx1 = -1, by1 = -1;
            bool ok = false;
            if (j < n_vis && ((s.agent[j] >> face) & 1u)) {
                const AgentGeom g = load_agent(env_agents + (s.agent[j] >> 8));
                const uint32_t corners = face_corners(face);
                V3 V[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) V[q] = box_corner(c, g, (corners >> (4 * q)) & 7u);
                int x0, y0, x1, y1;
                PrimEq q;
                ok = pixel_box_int(c, t, V, x0, y0, x1, y1) && prim_equations(V, true, face_flags(corners), plane_normal(V, true), q);
                if (ok) {
                    float thr[4];
                    edge_thresholds(q.tl, thr);
#pragma unroll
                    for (int e = 0; e < 4; ++e) s.edge[e][lane] = make_float4(q.nx[e], q.ny[e], q.nz[e], thr[e]);
                    s.w[lane] = make_float4(q.wx, q.wy, q.wz, 0.f);
                    bx0 = x0; by0 = y0; bx1 = x1; by1 = y1;
                }
            }
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) {                // the box around the agent's faces
                bx0 = min(bx0, __shfl_xor_sync(0xffffffffu, bx0, d)); by0 = min(by0, __shfl_xor_sync(0xffffffffu, by0, d));
                bx1 = max(bx1, __shfl_xor_sync(0xffffffffu, bx1, d)); by1 = max(by1, __shfl_xor_sync(0xffffffffu, by1, d));
            }
            const unsigned valid = __ballot_sync(0xffffffffu, ok);
            __syncwarp();
            for (int i = 0; i < 4; ++i) {
                const unsigned faces = (valid >> (8 * i)) & 0x3fu;
                if (!faces) continue;
                const int x0 = __shfl_sync(0xffffffffu, bx0, 8 * i), y0 = __shfl_sync(0xffffffffu, by0, 8 * i);
                const int w = __shfl_sync(0xffffffffu, bx1, 8 * i) - x0 + 1, h = __shfl_sync(0xffffffffu, by1, 8 * i) - y0 + 1;
                const int dy = 32 / w, dx = 32 - dy * w;     // 32 pixels on, row by row
                int y = lane / w, x = lane - y * w;
                uint32_t cnt = 0u;
                for (; __any_sync(0xffffffffu, y < h); ) {
                    // four pixels per lane at a time: a face is read once for them, and one's latency hides behind the others
                    float rx[4], ry[4];
                    bool have[4], in[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        have[k] = y < h;
                        in[k] = false;
                        rx[k] = have[k] ? __ldg(ray_x + x0 + x) : 0.f;
                        ry[k] = have[k] ? __ldg(ray_y + y0 + y) : 0.f;
                        x += dx; y += dy;
                        if (x >= w) { x -= w; ++y; }
                    }
#pragma unroll 1
                    for (unsigned fm_ = faces; fm_; fm_ &= fm_ - 1) {
                        const int f = 8 * i + __ffs(fm_) - 1;
                        const float4 pw = s.w[f], e0 = s.edge[0][f], e1 = s.edge[1][f], e2 = s.edge[2][f], e3 = s.edge[3][f];
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float wv = fm(pw.x, rx[k], fm(pw.y, ry[k], pw.z));
                            bool cov = wv >= t.w_far;
                            cov = cov & (wv <= t.w_near);
                            cov = cov & (fm(e0.x, rx[k], fm(e0.y, ry[k], e0.z)) > e0.w);
                            cov = cov & (fm(e1.x, rx[k], fm(e1.y, ry[k], e1.z)) > e1.w);
                            cov = cov & (fm(e2.x, rx[k], fm(e2.y, ry[k], e2.z)) > e2.w);
                            cov = cov & (fm(e3.x, rx[k], fm(e3.y, ry[k], e3.z)) > e3.w);
                            in[k] = in[k] | cov;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) cnt += have[k] & in[k] ? 1u : 0u;
                }
                cnt = __reduce_add_sync(0xffffffffu, cnt);
                if (lane == 0 && cnt) atomicAdd(occ + 2 * (s.agent[j0 + i] >> 8) + 1, cnt);
            }
            __syncwarp();
        }
    }
}

// One warp per band of 16 rows: with more, the longest ones -- an agent that fills the image -- are left running alone
// (4 096 views of 100 x 70 pixels, 64 agents, with one pixel per lane: whole views 224 us, 32 rows 128 us, 16 rows in CTAs of one warp 81 us).
static cudaError_t run_coverage(const RenderParams& P, long long n_views, cudaStream_t stream) {
    const int band_rows = 16, bands = (P.H + band_rows - 1) / band_rows;
    if (n_views * bands > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    coverage_kernel<<<(unsigned)(n_views * bands), 32, 0, stream>>>(P, (unsigned)n_views, bands, band_rows);
    return cudaGetLastError();
}

// The cull pass of a call.  Views of several tiles (as many as a warp has lanes) are culled a warp per view while that leaves
// enough warps to hide the latency of each; a view then does the work of its tiles at once, so the line is a number of tiles.
// Measured, time culled per tile / per view at so many views per multiprocessor (class and depth, maps of 5 640 / 1 950 triangles):
//    2 tiles   8: 0.98 / 0.94   10: 1.00 / 0.98   12: 1.00 / 1.01   16: 1.06 / 1.08
//    4 tiles   5: 1.00 / 0.91    6: 0.97 / 0.96    8: 1.07 / 1.09   12: 1.08 / 1.12
//    8 tiles   3: 0.95 / 0.91    4: 1.00 / 1.05    6: 1.07 / 1.14   10: 1.10 / 1.21
//   16 tiles   1: 0.92 / 0.96    2: 1.01 / 1.09    4: 1.12 / 1.19   10: 1.21 / 1.30
//   32 tiles   1: 0.99 / 1.05    2: 1.05 / 1.17    4: 1.15 / 1.28    8: 1.33 / 1.39
// (antialiased colour: the same lines, 0.96 to 1.08).
constexpr int VIEW_CULL_TILES = 28;        // tiles per multiprocessor from which views are culled as a whole
template <class K>
cudaError_t launch_next(K kernel, unsigned grid, size_t smem, cudaStream_t stream, const RenderParams& P, unsigned threads = NTHREADS);
static cudaError_t launch_cull(const RenderParams& P, long long n_views, bool conservative, int sm_count, cudaStream_t stream) {
    const int tiles = P.tiles_x * P.tiles_y;
    if (!P.counters && !(P.debug_flags & 4) && tiles > 1 && tiles <= 32 && n_views * tiles >= VIEW_CULL_TILES * (long long)sm_count)
        return launch_next(conservative ? cull_kernel<NoTally, true, true> : cull_kernel<NoTally, false, true>, (unsigned)((n_views + NW - 1) / NW), sizeof(CullSmem), stream, P);
    const unsigned grid = (P.n_jobs + NW - 1) / NW;
    return launch_next(P.counters ? cull_kernel<Tally, false> : conservative ? cull_kernel<NoTally, true> : cull_kernel<NoTally, false>, grid, sizeof(CullSmem), stream, P);
}

template <bool VEC, bool OCC, bool RGB>
static cudaError_t launch_tiles(const RenderParams& P0, long long n_views, int sm_count, cudaStream_t stream);

// Launches the next kernel of a call: its blocks may be brought in while the last blocks of the kernel before it still
// run (it waits for that kernel itself, see await_previous).
template <class K>
cudaError_t launch_next(K kernel, unsigned grid, size_t smem, cudaStream_t stream, const RenderParams& P, unsigned threads) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P);
}

}  // namespace pic
#include "pic_coverage.cuh"
namespace pic {
#include "pic_tile.cuh"
template <bool VEC, bool OCC, bool RGB>
static cudaError_t launch_tiles(const RenderParams& P0, long long n_views, int sm_count, cudaStream_t stream) {
    RenderParams P = P0;
    P.div_views = fast_div((uint32_t)n_views);
    // (Images whose rows are no groups of four pixels stay in order: neighbouring tiles share 32-byte sectors (1 260 agents x 3 cameras at
    // 159 x 90: 229 us in order, 248 not), but with occlusion counts, which take longer (891 views of 245 x 137: 188 in order, 177 not).
    // A kernel of its own for each order: what the order takes at the start cost the other 1 % in registers.)
    const bool first = (VEC || OCC) && draws_horizon_first(P.H, P.W, P.n_jobs, sm_count);
    return launch_next(first ? render_tile_kernel<NoTally, VEC, OCC, RGB, VEC || OCC> : render_tile_kernel<NoTally, VEC, OCC, RGB, false>, P.n_jobs, 0, stream, P, 32);
}
#include "pic_colour.cuh"
#include "pic_static.cuh"
#include "pic_small.cuh"

size_t render_smem_bytes() { return SMALL_SMEM > sizeof(ColourSmem) ? SMALL_SMEM : sizeof(ColourSmem); }
size_t survivor_bytes_per_tile() { return sizeof(uint2) * SURV_STRIDE; }

cudaError_t launch_render_kernel(const RenderParams& P0, long long n_views, int sm_count, cudaStream_t stream) {
    RenderParams P = P0;
    const long long jobs = n_views * P.tiles_x * P.tiles_y;
    if (jobs > 0x7fffffffLL || (long long)P.E * P.A * P.K > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (jobs <= 0) return cudaSuccess;
    P.n_jobs = (uint32_t)jobs;
    // few tiles: one CTA takes a tile from culling to store.  Measured (a call on 16 agents per environment, both image shapes of the workloads): 64 tiles 37 -> 17 us, 256 tiles 45 -> 14.5, 512 tiles 45 -> 23,
    // and against cull + tile kernel 768 tiles 41.7 -> 31.1, 1 024 tiles 43.5 -> 37.3, 1 280 tiles 44.0 -> 44.9.
    if (jobs <= 8LL * sm_count && !P.counters && !P.occlusion && (P.debug_flags & 15) == 0)
        return launch_next(P.W % 4 == 0 && !P.out_depth32 ? render_small_kernel<true> : render_small_kernel<false>, (unsigned)jobs, SMALL_SMEM, stream, P, SMALL_THREADS);
    // (a) cull: survivors per tile
    cudaError_t err = launch_cull(P, n_views, false, sm_count, stream);
    if (err != cudaSuccess) return err;
    // (b)-(d) set-up, raster, store
    const bool vec = P.W % 4 == 0 && !P.out_depth32;
    err = P.counters    ? launch_next(render_tile_kernel<Tally, false, true>, P.n_jobs, 0, stream, P, 32)
          : P.occlusion ? (vec ? launch_tiles<true, true, false>(P, n_views, sm_count, stream) : launch_tiles<false, true, false>(P, n_views, sm_count, stream))
                        : (vec ? launch_tiles<true, false, false>(P, n_views, sm_count, stream) : launch_tiles<false, false, false>(P, n_views, sm_count, stream));
    if (err != cudaSuccess) return err;
    // the tiles left out (their number is only known on the device): one wave of CTAs walks the list
    const long long wave = (long long)sm_count * 5;
    const unsigned cgrid = (unsigned)(jobs < wave ? jobs : wave);
    err = launch_next(P.counters ? cooperative_kernel<Tally> : cooperative_kernel<NoTally>, cgrid, sizeof(TileSmem), stream, P);
    if (err != cudaSuccess || !P.occlusion) return err;
    return run_coverage(P, n_views, stream);
}

// The coverage pass alone (after the exhaustive kernel, which counts the visible pixels itself).
cudaError_t launch_coverage_kernel(const RenderParams& P0, long long n_views, cudaStream_t stream) {
    return n_views <= 0 || !P0.occlusion ? cudaSuccess : run_coverage(P0, n_views, stream);
}

}  // namespace pic
