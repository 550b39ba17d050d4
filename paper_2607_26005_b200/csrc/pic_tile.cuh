// Render kernel over the cull kernel's survivor lists (included by pic_render.cu, inside namespace pic): set-up, raster
// and store of one tile by one warp, with the z-buffer in registers.
//
// Bound by instruction issue (the images of a step are a seventh of the time at the copy bandwidth), so the split is
// chosen to execute little per pixel.
//   set-up    a lane per survivor.  The pixels of primitives of at most 16 pixel centres are evaluated at once, a lane each
//             whatever the primitive, and leave fragments (pixel, key); the other primitives leave a record (edge functions,
//             1/z plane) -- on the benchmark workload 20 primitives, 33 fragments and 7 records per tile.
//   classify  a tile is 32 cells of 32 x 4 pixels, one per lane: for every record each lane decides whether its cell is
//             outside, partly inside or inside (14 cells hold anything, 28 pairs of record and cell meet, 20 of them partly).
//   raster    cell after cell, four adjacent pixels per lane: the cell's fragments meet in shared memory, then the records of
//             the cell's mask in turn, keeping the largest key per pixel in registers; then conversion and store.  A
//             pixel's key passes through memory only where a cell has fragments, background cells cost their stores, and
//             the warps share nothing, so no barrier holds one back.
// Against the kernel it replaced (four tiles per CTA, keys of 16-row strips in shared memory, records looked at once per
// strip), a step of 65 536 agents x 4 cameras at 64 x 64: 6.2 k instead of 8.0 k warp instructions per tile, 2 430 instead of
// 3 103 us per call.  24 warps per multiprocessor (72 registers): 20 take 3 % longer, 28 1 %.
//
// A tile with more records or fragments than fit is left to the cooperative kernel.
#pragma once

constexpr int TREC = 32;                     // records of a tile: a 32-bit mask
constexpr int TFRAG = 256;                   // fragments of its small primitives
constexpr int SMALL_PIXELS = 16;             // pixel centres in the box of a small primitive (4, 8, 24, 32: within 2 %)
constexpr int TILE_CTAS = 24;                // warps per multiprocessor the registers are bounded for
constexpr int CELL_W = 32, CELL_H = 4;       // pixels of a cell
static_assert((TILE / CELL_W) * (TILE / CELL_H) == 32, "a lane per cell");

template <int N>
struct __align__(16) TileRecords {
    float4 edge[4][N];                       // edge e: E = x rx + y ry + z, covered where E > w (see edge_thresholds)
    float4 w[N];                             // 1/z plane wx, wy, wz; key low word
    __device__ __forceinline__ void write(int slot, const PrimEq& q, uint32_t key_lo) {
        float thr[4];
        edge_thresholds(q.tl, thr);
#pragma unroll
        for (int e = 0; e < 4; ++e) edge[e][slot] = make_float4(q.nx[e], q.ny[e], q.nz[e], thr[e]);
        w[slot] = make_float4(q.wx, q.wy, q.wz, __uint_as_float(key_lo));
    }
};

struct __align__(16) TileWarp {
    TileRecords<TREC> rec;
    union {
        TileRecords<32> small;               // set-up: the small primitives of a pass, by lane
        struct {
            unsigned long long cell_key[CELL_W * CELL_H];   // raster: keys of a cell's fragments
            uint8_t need[TREC][32];          // per record and cell: edges that are not positive on all of it, NEED_RANGE
        };
    };
    unsigned long long frag_key[TFRAG];
    float ray_x[TILE], ray_y[TILE];
    uint32_t cells[TREC];                    // cells that the record's pixel box reaches
    uint16_t frag_px[TFRAG];                 // cell << 7 | pixel of the cell (row << 5 | column)
};
constexpr uint32_t NEED_RANGE = 16u;         // the depth range has to be tested pixel by pixel

// Adds the visible pixels of a cell to the counts of the agents whose boxes won them, one atomic per agent seen.
__device__ __forceinline__ void count_visible_cell(uint32_t* occ, const unsigned long long (&best)[4], uint32_t n_map_tris, int lane) {
    int agent[4];
    bool any = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t index = 0xFFFFFFu - ((uint32_t)best[k] >> 8);
        agent[k] = (best[k] != 0ull && index >= n_map_tris) ? (int)((index - n_map_tris) / 12u) : -1;
        any = any || agent[k] >= 0;
    }
    for (unsigned m = __ballot_sync(0xffffffffu, any); m; m = __ballot_sync(0xffffffffu, any)) {
        const int first = agent[0] >= 0 ? agent[0] : agent[1] >= 0 ? agent[1] : agent[2] >= 0 ? agent[2] : agent[3];
        const int b = __shfl_sync(0xffffffffu, first, __ffs(m) - 1);
        uint32_t cnt = 0u;
        any = false;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (agent[k] == b) { ++cnt; agent[k] = -1; }
            any = any || agent[k] >= 0;
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) atomicAdd(occ + 2 * b, cnt);
    }
}

// best = max(best, key of (w, lo)) where `in`; in float compares, which are fewer instructions than the 64-bit one.
__device__ __forceinline__ void keep_nearer(unsigned long long& best, bool in, float w, uint32_t lo) {
    const uint32_t bh = (uint32_t)(best >> 32), bl = (uint32_t)best;
    const float bw = __uint_as_float(bh);
    const bool up = in & ((w > bw) | ((w == bw) & (lo > bl)));
    best = make_key(up ? __float_as_uint(w) : bh, up ? lo : bl);
}

// Cell << 7 | pixel of the cell (row << 5 | column).
__device__ __forceinline__ uint32_t cell_pixel(int x, int y) { return (uint32_t)((((y >> 2) << 1) | (x >> 5)) << 7 | (y & 3) << 5 | (x & 31)); }

// The pixels of the warp's small primitives -- lane l's is small[l], w x h pixels from (bx0, by0), if `is_small` -- a lane
// each whatever the primitive; `push` gets every lane's result (covered?, 1/z, low key word, pixel).
template <class Push>
__device__ __forceinline__ void small_pixels(const TileRecords<32>& small, const float* ray_x, const float* ray_y, bool is_small, int bx0, int by0, int w, int h,
                                             float w_near, float w_far, int lane, Push push) {
    const int cnt = is_small ? w * h : 0;
    int incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += up;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), before = incl - cnt;
    // x, y of the box and 1024 / w rounded up: (i * inv) >> 10 is i / w for i < 32
    const uint32_t packed = (uint32_t)bx0 | ((uint32_t)by0 << 6) | ((uint32_t)w << 12) | ((uint32_t)((1024 + w - 1) / w) << 18);
    __syncwarp();
#pragma unroll 1
    for (int p0 = 0; p0 < total; p0 += 32) {
        const int p = p0 + lane;
        int own = 0;                                         // the lane whose range holds p: the last with before <= p (and pixels)
#pragma unroll
        for (int st = 16; st; st >>= 1) {
            const int b = __shfl_sync(0xffffffffu, before, own + st);
            if (b <= p) own += st;
        }
        const uint32_t pk = __shfl_sync(0xffffffffu, packed, own);
        const int idx = p - __shfl_sync(0xffffffffu, before, own);
        const int dy = (idx * (int)(pk >> 18)) >> 10, x = (int)(pk & 63u) + idx - dy * (int)((pk >> 12) & 63u), y = (int)((pk >> 6) & 63u) + dy;
        bool in = p < total;
        float wv = 0.f;
        uint32_t lo = 0u;
        if (in) {
            const float rx = ray_x[x], ry = ray_y[y];
            const float4 pw = small.w[own];
            wv = fm(pw.x, rx, fm(pw.y, ry, pw.z));
            lo = __float_as_uint(pw.w);
            in = (wv >= w_far) & (wv <= w_near);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 q4 = small.edge[e][own];
                in = in & (fm(q4.x, rx, fm(q4.y, ry, q4.z)) > q4.w);
            }
        }
        push(in, wv, lo, x, y);
    }
}

// Cells (bit 2 row + column) reached by a pixel box.
__device__ __forceinline__ uint32_t box_cells(uint32_t box) {
    const int bx0 = box & 0xff, by0 = (box >> 8) & 0xff, bx1 = (box >> 16) & 0xff, by1 = box >> 24;
    const uint32_t cols = (bx0 < CELL_W ? 0x55555555u : 0u) | (bx1 >= CELL_W ? 0xaaaaaaaau : 0u);
    const int r0 = by0 >> 2, r1 = by1 >> 2;
    return cols & (0xffffffffu << (2 * r0)) & (0xffffffffu >> (30 - 2 * r1));
}

// Which records reach the lane's cell?  Returns their bits and leaves, per record, what has to be
// tested there pixel by pixel.  An edge function's values on the cell's pixel centres lie within +-h of its value at the
// cell's centre; h is widened by 1e-6 of the terms' sizes, several times what the float32 evaluations can lose, so
// "outside" and "inside" hold for every pixel as it would be evaluated itself.
// (first, step: the records looked at.)
template <class S, class TL>
__device__ __forceinline__ uint32_t classify_records(S& s, int n_rec, bool exact, float w_near, float w_far, int lane, TL& n, int first = 0, int step = 1) {
    const int xa = (lane & 1) * CELL_W, ya = (lane >> 1) * CELL_H;
    const float rxa = s.ray_x[xa], rxb = s.ray_x[xa + CELL_W - 1], rya = s.ray_y[ya], ryb = s.ray_y[ya + CELL_H - 1];
    const float rxc = 0.5f * (rxa + rxb), ryc = 0.5f * (rya + ryb);
    const float hx = 0.5f * (rxb - rxa) + 1e-6f * fmaxf(fabsf(rxa), fabsf(rxb)), hy = 0.5f * (ryb - rya) + 1e-6f * fmaxf(fabsf(rya), fabsf(ryb));
    uint32_t hit = 0u;
#pragma unroll 1
    for (int r = first; r < n_rec; r += step) {
        bool out = !((s.cells[r] >> lane) & 1u);
        uint32_t need = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4 q = s.rec.edge[e][r];
            const float c = fm(q.x, rxc, fm(q.y, ryc, q.z)), h = fm(fabsf(q.x), hx, fm(fabsf(q.y), hy, 1e-6f * fabsf(q.z)));
            out = out || (exact && c < -h);
            if (!(c > h)) need |= 1u << e;
        }
        const float4 w = s.rec.w[r];
        const float c = fm(w.x, rxc, fm(w.y, ryc, w.z)), h = fm(fabsf(w.x), hx, fm(fabsf(w.y), hy, 1e-6f * fabsf(w.z)));
        out = out || (exact && (c + h < w_far || c - h > w_near));
        if (!(c - h >= w_far && c + h <= w_near)) need |= NEED_RANGE;
        if (!exact) need = 15u | NEED_RANGE;
        s.need[r][lane] = (uint8_t)need;
        if (!out) hit |= 1u << r;
        if (lane == 0) ++n.classified;
    }
    return hit;
}

// The records of mask m against the lane's four pixels of cell `cell`.
template <class S>
__device__ __forceinline__ void raster_records_cell(const S& s, uint32_t m, int cell, const float4 rx, float ry, float w_near,
                                                    float w_far, unsigned long long (&best)[4]) {
#pragma unroll 1
    for (; m; m &= m - 1) {
        const int r = __ffs(m) - 1;
        const float4 w = s.rec.w[r];
        const float wt = fm(w.y, ry, w.z);
        const float w0 = fm(w.x, rx.x, wt), w1 = fm(w.x, rx.y, wt), w2 = fm(w.x, rx.z, wt), w3 = fm(w.x, rx.w, wt);
        bool in0 = true, in1 = true, in2 = true, in3 = true;
        if (s.need[r][cell]) {
            // everything at once: a cell that one edge crosses is mostly crossed by two or more, and a branch per edge costs more
            in0 = (w0 >= w_far) & (w0 <= w_near); in1 = (w1 >= w_far) & (w1 <= w_near);
            in2 = (w2 >= w_far) & (w2 <= w_near); in3 = (w3 >= w_far) & (w3 <= w_near);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 q = s.rec.edge[e][r];
                const float t = fm(q.y, ry, q.z);
                in0 = in0 & (fm(q.x, rx.x, t) > q.w); in1 = in1 & (fm(q.x, rx.y, t) > q.w);
                in2 = in2 & (fm(q.x, rx.z, t) > q.w); in3 = in3 & (fm(q.x, rx.w, t) > q.w);
            }
        }
        const uint32_t lo = __float_as_uint(w.w);
        keep_nearer(best[0], in0, w0, lo); keep_nearer(best[1], in1, w1, lo);
        keep_nearer(best[2], in2, w2, lo); keep_nearer(best[3], in3, w3, lo);
    }
}

// The four pixels of a lane -> class and depth images.  VEC: the four pixels exist, 4-pixel groups are aligned, no
// float32 depth image.
template <bool VEC>
__device__ __forceinline__ void store_class_depth(const RenderParams& P, size_t o, const unsigned long long (&best)[4], uint32_t bg_cls, float bg_z, int n_px) {
    float z[4];
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t hi = (uint32_t)(best[k] >> 32);          // (a fragment's 1/z is positive: 0 means none)
        z[k] = hi ? fast_rcp(__uint_as_float(hi)) : bg_z;
        c[k] = hi ? (uint32_t)best[k] : bg_cls;
    }
    const __half2 h0 = __floats2half2_rn(z[0], z[1]), h1 = __floats2half2_rn(z[2], z[3]);
    const uint32_t d0 = *reinterpret_cast<const uint32_t*>(&h0), d1 = *reinterpret_cast<const uint32_t*>(&h1);
    const uint32_t cw = __byte_perm(__byte_perm(c[0], c[1], 0x0040), __byte_perm(c[2], c[3], 0x0040), 0x5410);
    if (VEC) {
        *reinterpret_cast<uint32_t*>(P.out_class + o) = cw;
        *reinterpret_cast<uint2*>(P.out_depth + o) = make_uint2(d0, d1);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < n_px) {
                P.out_class[o + k] = (uint8_t)(cw >> (8 * k));
                P.out_depth[o + k] = (uint16_t)((k < 2 ? d0 : d1) >> (16 * (k & 1)));
                if (P.out_depth32) P.out_depth32[o + k] = z[k];
            }
    }
}

__constant__ float FACE_SHADE[6] = {0.60f, 1.00f, 0.70f, 0.85f, 0.40f, 0.92f};   // rear, front, right, left, bottom, top

// Colour of a key's fragment: its class's, for a box face (primitives from n_map_tris on, two per face) shaded by face
// and depth.
__device__ __forceinline__ uint32_t key_colour(const RenderParams& P, unsigned long long key, uint32_t n_map_tris) {
    const uint32_t pal = __ldg(P.palette + ((uint32_t)key & 0xffu)), index = 0xFFFFFFu - ((uint32_t)key >> 8);
    if (index < n_map_tris) return pal;
    const uint32_t face = ((index - n_map_tris) >> 1) % 6u;
    const float k = FACE_SHADE[face] * (1.f - 0.5f * __fdividef(__fdividef(1.f, __uint_as_float((uint32_t)(key >> 32))) - P.near_z, P.far_z - P.near_z));
    const float r = k * (float)(pal & 0xffu), g = k * (float)((pal >> 8) & 0xffu), b = k * (float)((pal >> 16) & 0xffu);
    return (uint32_t)fminf(r + 0.5f, 255.f) | ((uint32_t)fminf(g + 0.5f, 255.f) << 8) | ((uint32_t)fminf(b + 0.5f, 255.f) << 16);
}

// The four pixels of a lane -> colour image (o: pixel offset).
template <bool VEC>
__device__ __forceinline__ void store_rgb(const RenderParams& P, size_t o, const unsigned long long (&best)[4], uint32_t bg, uint32_t n_map_tris, int n_px) {
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = best[k] ? key_colour(P, best[k], n_map_tris) : bg;
    uint8_t* dst = P.out_rgb + 3 * o;
    if (VEC) {
        uint32_t* d = reinterpret_cast<uint32_t*>(dst);
        d[0] = c[0] | (c[1] << 24); d[1] = (c[1] >> 8) | (c[2] << 16); d[2] = (c[2] >> 16) | (c[3] << 8);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < n_px) { dst[3 * k] = (uint8_t)c[k]; dst[3 * k + 1] = (uint8_t)(c[k] >> 8); dst[3 * k + 2] = (uint8_t)(c[k] >> 16); }
    }
}

// store_background for colours.
__device__ __forceinline__ void store_background_rgb(const RenderParams& P, size_t tile0, const TileCtx& t, bool ego_active, const uint32_t* bg_cls, uint32_t busy, int lane) {
    const bool wide = (P.W & 15) == 0 && (reinterpret_cast<uintptr_t>(P.out_rgb) & 15u) == 0;
    const int x = wide ? (lane & 3) * 16 : (lane & 15) * 4, dy = wide ? 8 : 2;
    if (x >= t.tw) return;
    const uint32_t my_col = busy >> (x / CELL_W), sky = __ldg(P.palette + P.cls_sky);
    for (uint32_t y = wide ? lane >> 2 : lane >> 4; y < (uint32_t)t.th; y += dy) {
        if ((my_col >> ((y >> 2) * 2)) & 1u) continue;
        const uint32_t c = ego_active ? __ldg(P.palette + __ldg(bg_cls + y)) : sky;
        const uint32_t w0 = c | (c << 24), w1 = (c >> 8) | (c << 16), w2 = (c >> 16) | (c << 8);
        uint8_t* dst = P.out_rgb + 3 * (tile0 + (size_t)(y * P.W + x));
        if (wide) {
            uint4* d = reinterpret_cast<uint4*>(dst);
            d[0] = make_uint4(w0, w1, w2, w0); d[1] = make_uint4(w1, w2, w0, w1); d[2] = make_uint4(w2, w0, w1, w2);
        } else {
            uint32_t* d = reinterpret_cast<uint32_t*>(dst);
            d[0] = w0; d[1] = w1; d[2] = w2;
        }
    }
}

// Background of the cells not in `busy`: 16 pixels per lane where rows allow it (128-bit class, two 128-bit depth stores), else 4.
__device__ __forceinline__ void store_background(const RenderParams& P, size_t tile0, const TileCtx& t, bool ego_active, const uint2* bg_fill, uint32_t busy, int lane) {
    const bool wide = (P.W & 15) == 0;                       // (then tiles are whole 16-pixel segments wide)
    const int x = wide ? (lane & 3) * 16 : (lane & 15) * 4, dy = wide ? 8 : 2;
    if (x >= t.tw) return;
    const uint32_t my_col = busy >> (x / CELL_W);            // bit 2 row: is the cell busy
    const uint2 sky = make_uint2(P.cls_sky * 0x01010101u, P.far_z2);
    uint32_t y = wide ? lane >> 2 : lane >> 4;
    size_t o = tile0 + (size_t)(y * P.W + x);
    const size_t step = (size_t)(dy * P.W);
#pragma unroll 2
    for (; y < (uint32_t)t.th; y += dy, o += step) {
        const uint2 b = ego_active ? __ldg(bg_fill + y) : sky;
        if ((my_col >> ((y >> 2) * 2)) & 1u) continue;
        if (wide) {
            *reinterpret_cast<uint4*>(P.out_class + o) = make_uint4(b.x, b.x, b.x, b.x);
            *reinterpret_cast<uint4*>(P.out_depth + o) = make_uint4(b.y, b.y, b.y, b.y);
            *reinterpret_cast<uint4*>(P.out_depth + o + 8) = make_uint4(b.y, b.y, b.y, b.y);
        } else {
            *reinterpret_cast<uint32_t*>(P.out_class + o) = b.x;
            *reinterpret_cast<uint2*>(P.out_depth + o) = make_uint2(b.y, b.y);
        }
    }
}

// VEC: rows of a multiple of four pixels and no float32 depth image.  OCC: with occlusion counts.  RGB: colours instead of
// classes and depths.
template <class TL, bool VEC, bool OCC, bool RGB = false>
__global__ void __launch_bounds__(32, TILE_CTAS) render_tile_kernel(const __grid_constant__ RenderParams P) {
    __shared__ TileWarp s;
    const int lane = threadIdx.x;
    launch_dependents();
    const unsigned id = await_previous(blockIdx.x);
    const uint2* blk = P.surv + (size_t)id * SURV_STRIDE;
    const uint4 head = __ldcg(reinterpret_cast<const uint4*>(blk));
    const uint2 sv0 = __ldcg(blk + 2 + lane);                // (requested with the head; of a shorter list the rest is not looked at)
    const Job job = decode_job(P, id);
    const TileCtx& t = job.t;
    const bool ego_active = __ldg(&P.agents[(size_t)job.e * P.A + job.a].active) != 0u;
    const uint32_t n_map_tris = __ldg(&P.env_maps[job.e].n_tris);
    load_rays(s, P, job, lane);
    load_rays(s, P, job, lane + 32);
    TL n = {};
    // test aids: few records send many tiles to the cooperative kernel
    const int rec_cap = (P.debug_flags & 2) ? 2 : (P.debug_flags & 8) ? 6 : TREC;
    bool fits = head.x != SURV_OVERFLOW;
    const int ns = fits ? (int)head.x : 0;
    int n_rec = 0, n_frag = 0;
    __syncwarp();
    // ---- set-up, a lane per survivor
    if (ns > 0) {
        Cam c;
        load_camera(c, P.cams[job.view], P.cam[job.k], P.W, P.H);
        const unsigned below = (1u << lane) - 1u;
#pragma unroll 1
        for (int i0 = 0; i0 < ns; i0 += 32) {
            const int i = i0 + lane;
            PrimEq q;
            uint32_t key_lo = 0u, box = 0u;
            bool ok = false;
            if (i < ns) {
                const uint2 sv = i0 == 0 ? sv0 : __ldcg(blk + 2 + i);
                V3 V[4], Pn;
                uint32_t flags;
                fetch_survivor(c, P, sv.x, job.e, n_map_tris, V, Pn, key_lo, flags);
                box = sv.y;
                ok = prim_equations(V, flags & 1u, flags, Pn, q);
            }
            const int bx0 = box & 0xff, by0 = (box >> 8) & 0xff, w = (int)((box >> 16) & 0xff) - bx0 + 1, h = (int)(box >> 24) - by0 + 1;
            const bool small = ok && w * h <= SMALL_PIXELS, big = ok && !small;
            if (ok) ++n.setup;
            if (small) { ++n.tiny; s.small.write(lane, q, key_lo); }
            const unsigned mb = __ballot_sync(0xffffffffu, big);
            if (big) {
                ++n.recs;
                const int slot = n_rec + __popc(mb & below);
                if (slot < rec_cap) { s.rec.write(slot, q, key_lo); s.cells[slot] = box_cells(box); }
            }
            n_rec += __popc(mb);
            // ---- the pixels of the small primitives, a lane each whatever the primitive
            small_pixels(s.small, s.ray_x, s.ray_y, small, bx0, by0, w, h, P.w_near, P.w_far, lane, [&](bool in, float wv, uint32_t lo, int x, int y) {
                const unsigned mf = __ballot_sync(0xffffffffu, in);
                const int slot = n_frag + __popc(mf & below);
                if (in && slot < TFRAG) {
                    s.frag_key[slot] = make_key(__float_as_uint(wv), lo);
                    s.frag_px[slot] = (uint16_t)cell_pixel(x, y);
                }
                n_frag += __popc(mf);
            });
            __syncwarp();
        }
        fits = fits && n_rec <= rec_cap && n_frag <= TFRAG;
    }
    if (!fits) {
        // (the cooperative kernel counts the tile again)
        if (lane == 0) P.overflow[1u + atomicAdd(&P.overflow[0], 1u)] = id;
        return;
    }
    if (lane == 0) { n.grp = (int)head.y; n.leaf = (int)head.z; n.tested = (int)head.w; ++n.jobs; }
    // ---- the records of every cell
    const bool exact = !(P.debug_flags & 1);
    const uint32_t hit = classify_records(s, n_rec, exact, P.w_near, P.w_far, lane, n);
    if (n_frag > 0) {
        ulonglong2* ck = reinterpret_cast<ulonglong2*>(s.cell_key);
        ck[lane] = make_ulonglong2(0ull, 0ull); ck[lane + 32] = make_ulonglong2(0ull, 0ull);
    }
    // (the fragment this lane holds; of more than 32, the others are looked at anew in every cell)
    const uint32_t my_frag = lane < n_frag ? s.frag_px[lane] : 0xffffu;
    const unsigned long long my_key = lane < n_frag ? s.frag_key[lane] : 0ull;
    __syncwarp();
    const size_t tile0 = job.view * ((size_t)P.H * P.W) + (size_t)t.y0 * P.W + t.x0;
    const uint32_t* bg_cls = P.rig.bg_cls + (size_t)job.k * P.H + t.y0;
    const float* bg_z = P.rig.bg_z + (size_t)job.k * P.H + t.y0;
    uint32_t* occ = (OCC && P.occlusion) ? P.occlusion + job.view * (size_t)P.A * 2u : nullptr;   // visible-pixel counts of this view
    // cells that hold anything, and those with fragments: only they look for them (64 views of 128 x 256 per environment of a large map,
    // many tiles with more than 32 fragments: 655 us with every busy cell going through the list, 630 with this mask)
    uint32_t busy = __ballot_sync(0xffffffffu, hit != 0u), frag_cells = 0u;
    if (n_frag > 0) {
        frag_cells = lane < n_frag ? 1u << (my_frag >> 7) : 0u;
        for (int f = 32 + lane; f < n_frag; f += 32) frag_cells |= 1u << (s.frag_px[f] >> 7);
        frag_cells = __reduce_or_sync(0xffffffffu, frag_cells);
        busy |= frag_cells;
    }
    // ---- the background of the other cells
    if (VEC && RGB) store_background_rgb(P, tile0, t, ego_active, bg_cls, busy, lane);
    else if (VEC) store_background(P, tile0, t, ego_active, P.rig.bg_fill + (size_t)job.k * P.H + t.y0, busy, lane);
    else busy = 0xffffffffu;
    // ---- cell after cell
    const int px = (lane & 7) * 4, py = lane >> 3;
#pragma unroll 1
    for (; busy; busy &= busy - 1) {
        const int cell = __ffs(busy) - 1;
        const int x = (cell & 1) * CELL_W + px, y = (cell >> 1) * CELL_H + py;
        const uint32_t m = __shfl_sync(0xffffffffu, hit, cell);
        unsigned long long best[4] = {0ull, 0ull, 0ull, 0ull};
        if ((frag_cells >> cell) & 1u) {                     // the cell's fragments meet in shared memory
            if ((int)(my_frag >> 7) == cell) atomicMax(&s.cell_key[my_frag & 127u], my_key);
            for (int f = 32 + lane; f < n_frag; f += 32) {
                const uint32_t fp = s.frag_px[f];
                if ((int)(fp >> 7) == cell) atomicMax(&s.cell_key[fp & 127u], s.frag_key[f]);
            }
            __syncwarp();
            ulonglong2* ck = reinterpret_cast<ulonglong2*>(s.cell_key) + 2 * lane;
            const ulonglong2 a = ck[0], b = ck[1];
            best[0] = a.x; best[1] = a.y; best[2] = b.x; best[3] = b.y;
            ck[0] = make_ulonglong2(0ull, 0ull); ck[1] = make_ulonglong2(0ull, 0ull);
            __syncwarp();
        }
        const float4 rx = *reinterpret_cast<const float4*>(s.ray_x + x);
        const float ry = s.ray_y[y];
        if (lane == 0) n.cells += __popc(m);
        raster_records_cell(s, m, cell, rx, ry, P.w_near, P.w_far, best);
        const bool row_ok = y < t.th;
        const int n_px = row_ok ? t.tw - x : 0;
        if (OCC && occ) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k >= n_px) best[k] = 0ull;
            count_visible_cell(occ, best, n_map_tris, lane);
        }
        if (n_px > 0) {
            uint32_t bc = P.cls_sky;
            float bz = P.far_z;
            if (ego_active) { bc = __ldg(bg_cls + y); if (!RGB) bz = __ldg(bg_z + y); }
            const size_t o = tile0 + (size_t)(y * P.W + x);
            if (RGB) store_rgb<VEC>(P, o, best, __ldg(P.palette + bc), n_map_tris, n_px);
            else store_class_depth<VEC>(P, o, best, bc, bz, n_px);
        }
    }
    flush_counters(P, n);
}
