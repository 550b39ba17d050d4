// Render kernel over the cull kernel's survivor lists (included by pic_render.cu, inside namespace pic): set-up, raster
// and store of one tile by one warp, with the z-buffer in registers.
//
// Bound by instruction issue (the images of a step of 65 536 agents are nearly a quarter of its time at the copy bandwidth), so the split
// is chosen to execute little per pixel.
//   set-up    a lane per survivor.  The pixels of primitives of at most 16 pixel centres are evaluated at once, a lane each
//             whatever the primitive, and leave fragments (pixel, key); the other primitives leave a record (edge functions,
//             1/z plane) -- on the benchmark workload 20 primitives, 33 fragments and 7 records per tile.
//   classify  a tile is 32 cells of 32 x 4 pixels, one per lane: for every record each lane decides whether its cell is
//             outside, partly inside or inside (14 cells hold anything, 27 pairs of record and cell meet, 20 of them partly).
//   raster    cell after cell, four adjacent pixels per lane: the records of the cell's mask in turn, keeping the nearest
//             1/z and key per pixel in registers, then the cell's fragments, which meet in shared memory; then conversion and
//             store.  A pixel's key passes through memory only where a cell has fragments, background cells cost their
//             stores, and the warps share nothing, so no barrier holds one back.
// Against the kernel it replaced (four tiles per CTA, keys of 16-row strips in shared memory, records looked at once per
// strip), a step of 65 536 agents x 4 cameras at 64 x 64: 6.2 k instead of 8.0 k warp instructions per tile, 2 430 instead of
// 3 103 us per call; then 5.0 k and 2 251 us (8 192 agents 243 -> 220, 64 x 64 agents at 128 x 256 655 -> 563) by
//   two edges at a time (packed fma), one predicate carried through a pixel's comparisons, the rare depth-range test in a loop of
//   its own: a pair of record and cell 84 -> 60 instructions;
//   records sorted by index once per tile, so that a tie needs no comparison per pixel (the sort is 85 instructions);
//   columns' ray coordinates kept twice in shared memory, the rows' background in shared memory and in the class register from the
//   start: a cell's own part 122 -> 75;
//   28 warps per multiprocessor (72 registers, 7.3 KB) instead of 24 (80, 8.6 KB): 2 334 -> 2 251; 32 (64, 6.3 KB) take 2 297, with
//   more tiles whose fragments do not fit.
// Measured and left: the smallest of four edges instead of four comparisons (three-operand minimum; edges that own their zeros
// lifted by the smallest subnormal, +1 %), each pair of edges behind its own test (+1 %), warps that stay and draw tiles from a
// counter, the next tile's survivors copied in the meantime (2 333 -> 2 468), two or four warps per CTA (2 440, 2 458), the
// ray tables read only for tiles with survivors (2 371).
//
// A tile with more records or fragments than fit is left to the cooperative kernel.
#pragma once

constexpr int TREC = 32;                     // records of a tile: a 32-bit mask
constexpr int TFRAG = 256;                   // fragments of its small primitives
constexpr int TPOOL = 3328;                  // bytes for both: 32 records and 96 fragments, 256 fragments and 16 records
constexpr int SMALL_PIXELS = 16;             // pixel centres in the box of a small primitive (4, 8, 24, 32: within 2 %, measured with 24 warps and one edge per instruction)
constexpr int TILE_CTAS = 28;                // warps per multiprocessor
constexpr int CELL_W = 32, CELL_H = 4;       // pixels of a cell
static_assert((TILE / CELL_W) * (TILE / CELL_H) == 32, "a lane per cell");

// Two float32 in a register pair; each half is rounded like the scalar operation.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Record of a primitive.  The edges are kept two by two, so that two are evaluated by one instruction.  (80 bytes: 128-bit accesses
// of eight consecutive records meet no bank twice.)
struct __align__(16) TileRecord {
    float4 xy[2];                            // edges 0 and 2, 1 and 3: E = x rx + y ry + z, covered where E > thr (see edge_thresholds): x, x, y, y of a pair
    float4 zt[2];                            //   and z, z, thr, thr
    float4 w;                                // 1/z plane wx, wy, wz; key low word
    __device__ __forceinline__ void write(const PrimEq& q, uint32_t key_lo) {
        float thr[4];
        edge_thresholds(q.tl, thr);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            xy[h] = make_float4(q.nx[h], q.nx[h + 2], q.ny[h], q.ny[h + 2]);
            zt[h] = make_float4(q.nz[h], q.nz[h + 2], thr[h], thr[h + 2]);
        }
        w = make_float4(q.wx, q.wy, q.wz, __uint_as_float(key_lo));
    }
};
// A pair of edges on the row ry (twice): x of both, y ry + z of both, the thresholds.
struct EdgePair { f32x2 x, t; float thr0, thr1; };
__device__ __forceinline__ EdgePair load_edges(const TileRecord& rec, int h, f32x2 ry2) {
    const ulonglong2 xy = *reinterpret_cast<const ulonglong2*>(&rec.xy[h]), zt = *reinterpret_cast<const ulonglong2*>(&rec.zt[h]);
    EdgePair q;
    q.x = xy.x; q.t = fma2(xy.y, ry2, zt.x);
    unpack2(zt.y, q.thr0, q.thr1);
    return q;
}
// `in`, and is the column rx (twice) inside both?  (One predicate carried through the comparisons: joined afterwards they cost an
// instruction each.)
__device__ __forceinline__ bool inside_edges(bool in, const EdgePair& q, f32x2 rx2) {
    float e0, e1;
    unpack2(fma2(q.x, rx2, q.t), e0, e1);
    in = in & (e0 > q.thr0);
    return in & (e1 > q.thr1);
}

struct __align__(16) TileWarp {
    union {                                  // records from the front, fragments' keys from the back: a tile has many of one or the other
        TileRecord rec[TREC];
        unsigned char pool[TPOOL];
    };
    union {
        TileRecord small[32];                // set-up: the small primitives of a pass, by lane
        struct {                             // raster:
            unsigned long long cell_key[CELL_W * CELL_H];   // keys of a cell's fragments
            float2 bg[TILE];                 // background of the rows: depth, and class or colour
        };
    };
    f32x2 ray_xx[TILE];                      // ray coordinates of the columns, twice each, and of the rows
    float ray_y[TILE];
    uint32_t cells[TREC];                    // cells that the record's pixel box reaches
    uint16_t frag_px[TFRAG];                 // cell << 7 | pixel of the cell (row << 5 | column)
    __device__ __forceinline__ unsigned long long& frag_key(int i) { return reinterpret_cast<unsigned long long*>(pool + TPOOL)[-1 - i]; }
};

__device__ __forceinline__ int record_bytes(int n) { return n * (int)sizeof(TileRecord); }

// Records (a bit each) that reach a cell, and those whose edges, or whose depth range, have to be tested there pixel by pixel.
struct CellRecords { uint32_t hit, edges, range; };

// Adds the visible pixels of a cell to the counts of the agents whose boxes won them, one atomic per agent seen.
__device__ __forceinline__ void count_visible_cell(uint32_t* occ, const float (&bw)[4], const uint32_t (&bl)[4], uint32_t n_map_tris, int lane) {
    int agent[4];
    bool any = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t index = 0xFFFFFFu - (bl[k] >> 8);
        agent[k] = (bw[k] > 0.f && index >= n_map_tris) ? (int)((index - n_map_tris) / 12u) : -1;
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

// Cell << 7 | pixel of the cell (row << 5 | column).
__device__ __forceinline__ uint32_t cell_pixel(int x, int y) { return (uint32_t)((((y >> 2) << 1) | (x >> 5)) << 7 | (y & 3) << 5 | (x & 31)); }

// The pixels of the warp's small primitives -- lane l's is small[l], w x h pixels from (bx0, by0), if `is_small` -- a lane
// each whatever the primitive; `push` gets every lane's result (covered?, 1/z, low key word, pixel).
template <class Push>
__device__ __forceinline__ void small_pixels(const TileRecord* small, const f32x2* ray_xx, const float* ray_y, bool is_small, int bx0, int by0, int w, int h,
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
            const f32x2 rx2 = ray_xx[x];
            float rx, rx_again;
            unpack2(rx2, rx, rx_again);
            const float ry = ray_y[y];
            const float4 pw = small[own].w;
            wv = fm(pw.x, rx, fm(pw.y, ry, pw.z));
            lo = __float_as_uint(pw.w);
            const f32x2 ry2 = pack2(ry, ry);
            in = wv >= w_far && wv <= w_near;
            in = inside_edges(inside_edges(in, load_edges(small[own], 0, ry2), rx2), load_edges(small[own], 1, ry2), rx2);
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

template <class S>
__device__ __forceinline__ float ray_at(const S& s, int x) { return reinterpret_cast<const float*>(s.ray_xx + x)[0]; }

// Which records reach the lane's cell, and which of them have to be tested there pixel by pixel?  An edge function's values on
// the cell's pixel centres lie within +-h of its value at the cell's centre; h is widened by 1e-6 of the terms' sizes, several
// times what the float32 evaluations can lose, so "outside" and "inside" hold for every pixel as it would be evaluated itself.
// (first, step: the records looked at.)
template <class S, class TL>
__device__ __forceinline__ CellRecords classify_records(const S& s, int n_rec, bool exact, float w_near, float w_far, int lane, TL& n, int first = 0, int step = 1) {
    const int xa = (lane & 1) * CELL_W, ya = (lane >> 1) * CELL_H;
    const float rxa = ray_at(s, xa), rxb = ray_at(s, xa + CELL_W - 1), rya = s.ray_y[ya], ryb = s.ray_y[ya + CELL_H - 1];
    const float rxc = 0.5f * (rxa + rxb), ryc = 0.5f * (rya + ryb);
    const float hx = 0.5f * (rxb - rxa) + 1e-6f * fmaxf(fabsf(rxa), fabsf(rxb)), hy = 0.5f * (ryb - rya) + 1e-6f * fmaxf(fabsf(rya), fabsf(ryb));
    CellRecords m = {0u, 0u, 0u};
#pragma unroll 1
    for (int r = first; r < n_rec; r += step) {
        bool out = !((s.cells[r] >> lane) & 1u), inside = exact;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 xy = s.rec[r].xy[h], zt = s.rec[r].zt[h];
            const float c0 = fm(xy.x, rxc, fm(xy.z, ryc, zt.x)), h0 = fm(fabsf(xy.x), hx, fm(fabsf(xy.z), hy, 1e-6f * fabsf(zt.x)));
            const float c1 = fm(xy.y, rxc, fm(xy.w, ryc, zt.y)), h1 = fm(fabsf(xy.y), hx, fm(fabsf(xy.w), hy, 1e-6f * fabsf(zt.y)));
            out = out || (exact && (c0 < -h0 || c1 < -h1));
            inside = inside && c0 > h0 && c1 > h1;
        }
        const float4 w = s.rec[r].w;
        const float c = fm(w.x, rxc, fm(w.y, ryc, w.z)), h = fm(fabsf(w.x), hx, fm(fabsf(w.y), hy, 1e-6f * fabsf(w.z)));
        out = out || (exact && (c + h < w_far || c - h > w_near));
        const uint32_t bit = 1u << r;
        if (!out) m.hit |= bit;
        if (!inside) m.edges |= bit;
        if (!out && !(exact && c - h >= w_far && c + h <= w_near)) m.range |= bit;
        if (lane == 0) ++n.classified;
    }
    return m;
}

// The records of a cell against the lane's four pixels (columns rx, row ry), the nearest so far in (bw, bl).  SORTED: the records
// are numbered by primitive index, so that on a tie the one already there stays; else the larger key wins.  RANGE: cell.range is
// looked at (few cells have any; apart because a test per record costs the others).
template <bool SORTED, bool RANGE, class S>
__device__ __forceinline__ void raster_cell_records(const S& s, const CellRecords& cell, int x, float ry, float w_near, float w_far, float (&bw)[4], uint32_t (&bl)[4]) {
    const f32x2 ry2 = pack2(ry, ry);
    f32x2 rx2[4];
    *reinterpret_cast<ulonglong2*>(rx2) = *reinterpret_cast<const ulonglong2*>(s.ray_xx + x);
    *reinterpret_cast<ulonglong2*>(rx2 + 2) = *reinterpret_cast<const ulonglong2*>(s.ray_xx + x + 2);
    float rx[4], rx_again;
#pragma unroll
    for (int k = 0; k < 4; ++k) unpack2(rx2[k], rx[k], rx_again);
#pragma unroll 1
    for (uint32_t m = cell.hit; m; m &= m - 1) {
        const int r = __ffs(m) - 1;
        const uint32_t bit = m & -m;
        const float4 w = s.rec[r].w;
        const float wt = fm(w.y, ry, w.z);
        const uint32_t lo = __float_as_uint(w.w);
        float wv[4];
        bool up[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            wv[k] = fm(w.x, rx[k], wt);
            up[k] = SORTED ? wv[k] > bw[k] : (wv[k] > bw[k]) | ((wv[k] == bw[k]) & (lo > bl[k]));
        }
        if (cell.edges & bit) {
            // everything at once: a cell that one edge crosses is mostly crossed by two or more, and a branch per edge costs more
            const EdgePair q0 = load_edges(s.rec[r], 0, ry2), q1 = load_edges(s.rec[r], 1, ry2);
#pragma unroll
            for (int k = 0; k < 4; ++k) up[k] = inside_edges(inside_edges(up[k], q0, rx2[k]), q1, rx2[k]);
        }
        if (RANGE && (cell.range & bit)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) up[k] = up[k] & (wv[k] >= w_far) & (wv[k] <= w_near);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) { bw[k] = up[k] ? wv[k] : bw[k]; bl[k] = up[k] ? lo : bl[k]; }
    }
}

// The four pixels of a lane -> class and depth images (bl: the background's class where bw is 0).  VEC: the four pixels exist,
// 4-pixel groups are aligned, no float32 depth image.
template <bool VEC>
__device__ __forceinline__ void store_class_depth(const RenderParams& P, size_t o, const float (&bw)[4], const uint32_t (&bl)[4], float bg_z, int n_px) {
    float z[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) z[k] = bw[k] > 0.f ? fast_rcp(bw[k]) : bg_z;     // (a fragment's 1/z is positive)
    const __half2 h0 = __floats2half2_rn(z[0], z[1]), h1 = __floats2half2_rn(z[2], z[3]);
    const uint32_t d0 = *reinterpret_cast<const uint32_t*>(&h0), d1 = *reinterpret_cast<const uint32_t*>(&h1);
    const uint32_t cw = __byte_perm(__byte_perm(bl[0], bl[1], 0x0040), __byte_perm(bl[2], bl[3], 0x0040), 0x5410);
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

// Colour of the fragment (w, key low word): its class's, for a box face (primitives from n_map_tris on, two per face) shaded by face
// and depth.
__device__ __forceinline__ uint32_t key_colour(const RenderParams& P, float w, uint32_t lo, uint32_t n_map_tris) {
    const uint32_t pal = __ldg(P.palette + (lo & 0xffu)), index = 0xFFFFFFu - (lo >> 8);
    if (index < n_map_tris) return pal;
    const uint32_t face = ((index - n_map_tris) >> 1) % 6u;
    const float k = FACE_SHADE[face] * (1.f - 0.5f * fast_div(fast_rcp(w) - P.near_z, P.far_z - P.near_z));
    const float r = k * (float)(pal & 0xffu), g = k * (float)((pal >> 8) & 0xffu), b = k * (float)((pal >> 16) & 0xffu);
    return (uint32_t)fminf(r + 0.5f, 255.f) | ((uint32_t)fminf(g + 0.5f, 255.f) << 8) | ((uint32_t)fminf(b + 0.5f, 255.f) << 16);
}

// The four pixels of a lane -> colour image (o: pixel offset; bl: the background's colour where bw is 0).
template <bool VEC>
__device__ __forceinline__ void store_rgb(const RenderParams& P, size_t o, const float (&bw)[4], const uint32_t (&bl)[4], uint32_t n_map_tris, int n_px) {
    uint32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] = bw[k] > 0.f ? key_colour(P, bw[k], bl[k], n_map_tris) : bl[k];
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

// store_background for colours (bg: colour of the rows).
__device__ __forceinline__ void store_background_rgb(const RenderParams& P, size_t tile0, const TileCtx& t, const float2* bg, uint32_t busy, int lane) {
    const bool wide = (P.W & 15) == 0 && (reinterpret_cast<uintptr_t>(P.out_rgb) & 15u) == 0;
    const int x = wide ? (lane & 3) * 16 : (lane & 15) * 4, dy = wide ? 8 : 2;
    if (x >= t.tw) return;
    const uint32_t my_col = busy >> (x / CELL_W);
    for (uint32_t y = wide ? lane >> 2 : lane >> 4; y < (uint32_t)t.th; y += dy) {
        if ((my_col >> ((y >> 2) * 2)) & 1u) continue;
        const uint32_t c = __float_as_uint(bg[y].y);
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

// Background of the cells not in `busy` (bg: depth and class of the rows): 16 pixels per lane where rows allow it (128-bit class, two 128-bit depth stores), else 4.
__device__ __forceinline__ void store_background(const RenderParams& P, size_t tile0, const TileCtx& t, const float2* bg, uint32_t busy, int lane) {
    const bool wide = (P.W & 15) == 0;                       // (then tiles are whole 16-pixel segments wide)
    const int x = wide ? (lane & 3) * 16 : (lane & 15) * 4, dy = wide ? 8 : 2;
    if (x >= t.tw) return;
    const uint32_t my_col = busy >> (x / CELL_W);            // bit 2 row: is the cell busy
    uint32_t y = wide ? lane >> 2 : lane >> 4;
    size_t o = tile0 + (size_t)(y * P.W + x);
    const size_t step = (size_t)(dy * P.W);
#pragma unroll 2
    for (; y < (uint32_t)t.th; y += dy, o += step) {
        if ((my_col >> ((y >> 2) * 2)) & 1u) continue;
        const __half2 z2 = __float2half2_rn(bg[y].x);
        const uint2 b = make_uint2(__float_as_uint(bg[y].y) * 0x01010101u, *reinterpret_cast<const uint32_t*>(&z2));
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

// Puts the records into the order of their primitive indices (the keys' low words, largest first), a lane per record.
__device__ __forceinline__ void sort_records(TileWarp& s, int n_rec, int lane) {
    const TileRecord r = lane < n_rec ? s.rec[lane] : TileRecord();
    const uint32_t cells = s.cells[lane], key = __float_as_uint(r.w.w);
    int rank = 0;
#pragma unroll 4
    for (int j = 0; j < n_rec; ++j) rank += __shfl_sync(0xffffffffu, key, j) > key ? 1 : 0;
    __syncwarp();
    if (lane < n_rec) {
        s.rec[rank] = r;
        s.cells[rank] = cells;
    }
    __syncwarp();
}

// VEC: rows of a multiple of four pixels and no float32 depth image.  OCC: with occlusion counts.  RGB: colours instead of
// classes and depths.  HORIZON_FIRST: the order of the tiles (see draws_horizon_first).
template <class TL, bool VEC, bool OCC, bool RGB = false, bool HORIZON_FIRST = false>
__global__ void __launch_bounds__(32, TILE_CTAS) render_tile_kernel(const __grid_constant__ RenderParams P) {
    __shared__ TileWarp s;
    const int lane = threadIdx.x;
    launch_dependents();
    const unsigned cta = await_previous(blockIdx.x), id = HORIZON_FIRST ? horizon_first(P, cta) : cta;
    const uint2* blk = P.surv + (size_t)id * SURV_STRIDE;
    const uint4 head = __ldcg(reinterpret_cast<const uint4*>(blk));
    const uint2 sv0 = __ldcg(blk + 2 + lane);                // (requested with the head; of a shorter list the rest is not looked at)
    const Job job = decode_job(P, id);
    const TileCtx& t = job.t;
    const bool ego_active = __ldg(&P.agents[(size_t)job.e * P.A + job.a].active) != 0u;
    const uint32_t n_map_tris = __ldg(&P.env_maps[job.e].n_tris);
#pragma unroll
    for (int i = lane; i < TILE; i += 32) {
        const float rx = ray_column(P, job, i);
        s.ray_xx[i] = pack2(rx, rx);
        s.ray_y[i] = ray_row(P, job, i);
    }
    TL n = {};
    // test aids: few records send many tiles to the cooperative kernel
    const int rec_cap = (P.debug_flags & 2) ? 2 : (P.debug_flags & 8) ? 6 : TREC;
    bool fits = head.x != SURV_OVERFLOW;
    const int ns = fits ? (int)head.x : 0;
    int n_rec = 0, n_frag = 0;
    __syncwarp();
    float2 bg[2];                            // (requested now, put down when the small primitives' records are no longer needed)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int i = lane + 32 * j;
        const size_t at = (size_t)job.k * P.H + t.y0 + i;
        const bool drawn = ego_active && i < t.th;
        if (RGB) bg[j] = make_float2(0.f, __uint_as_float(__ldg(drawn ? P.rig.bg_rgb + at : P.palette + P.cls_sky)));
        else bg[j] = drawn ? make_float2(__ldg(P.rig.bg_z + at), __uint_as_float(__ldg(P.rig.bg_cls + at))) : make_float2(P.far_z, __uint_as_float(P.cls_sky));
    }
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
            if (small) { ++n.tiny; s.small[lane].write(q, key_lo); }
            const unsigned mb = __ballot_sync(0xffffffffu, big);
            if (big) {
                ++n.recs;
                const int slot = n_rec + __popc(mb & below);
                if (slot < rec_cap && record_bytes(slot + 1) + 8 * n_frag <= TPOOL) { s.rec[slot].write(q, key_lo); s.cells[slot] = box_cells(box); }
            }
            n_rec += __popc(mb);
            // ---- the pixels of the small primitives, a lane each whatever the primitive
            small_pixels(s.small, s.ray_xx, s.ray_y, small, bx0, by0, w, h, P.w_near, P.w_far, lane, [&](bool in, float wv, uint32_t lo, int x, int y) {
                const unsigned mf = __ballot_sync(0xffffffffu, in);
                const int slot = n_frag + __popc(mf & below);
                if (in && slot < TFRAG && record_bytes(n_rec) + 8 * (slot + 1) <= TPOOL) {
                    s.frag_key(slot) = make_key(__float_as_uint(wv), lo);
                    s.frag_px[slot] = (uint16_t)cell_pixel(x, y);
                }
                n_frag += __popc(mf);
            });
            __syncwarp();
        }
        fits = fits && n_rec <= rec_cap && n_frag <= TFRAG && record_bytes(n_rec) + 8 * n_frag <= TPOOL;
        if (fits && n_rec > 1) sort_records(s, n_rec, lane);
    }
    if (!fits) {
        // (the cooperative kernel counts the tile again)
        if (lane == 0) P.overflow[1u + atomicAdd(&P.overflow[0], 1u)] = id;
        return;
    }
    if (lane == 0) { n.grp = (int)head.y; n.leaf = (int)head.z; n.tested = (int)head.w; ++n.jobs; }
    // ---- the records of every cell
    const bool exact = !(P.debug_flags & 1);
    const CellRecords mine = classify_records(s, n_rec, exact, P.w_near, P.w_far, lane, n);
    s.bg[lane] = bg[0]; s.bg[lane + 32] = bg[1];
    if (n_frag > 0) {
        ulonglong2* ck = reinterpret_cast<ulonglong2*>(s.cell_key);
        ck[lane] = make_ulonglong2(0ull, 0ull); ck[lane + 32] = make_ulonglong2(0ull, 0ull);
    }
    // (the fragment this lane holds; of more than 32, the others are looked at anew in every cell)
    const uint32_t my_frag = lane < n_frag ? s.frag_px[lane] : 0xffffu;
    const unsigned long long my_key = lane < n_frag ? s.frag_key(lane) : 0ull;
    __syncwarp();
    const size_t tile0 = job.view * ((size_t)P.H * P.W) + (size_t)t.y0 * P.W + t.x0;
    uint32_t* occ = (OCC && P.occlusion) ? P.occlusion + job.view * (size_t)P.A * 2u : nullptr;   // visible-pixel counts of this view
    // cells that hold anything, and those with fragments: only they look for them (views of 128 x 256 pixels of a large map, many
    // tiles with more than 32 fragments: 655 us with every busy cell going through the list, 630 with this mask)
    uint32_t busy = __ballot_sync(0xffffffffu, mine.hit != 0u), frag_cells = 0u;
    if (n_frag > 0) {
        frag_cells = lane < n_frag ? 1u << (my_frag >> 7) : 0u;
        for (int f = 32 + lane; f < n_frag; f += 32) frag_cells |= 1u << (s.frag_px[f] >> 7);
        frag_cells = __reduce_or_sync(0xffffffffu, frag_cells);
        busy |= frag_cells;
    }
    // ---- the background of the other cells
    if (VEC && RGB) store_background_rgb(P, tile0, t, s.bg, busy, lane);
    else if (VEC) store_background(P, tile0, t, s.bg, busy, lane);
    else busy = (t.th > TILE - CELL_H ? 0xffffffffu : (1u << (2 * ((t.th + CELL_H - 1) / CELL_H))) - 1u) & (t.tw > CELL_W ? 0xffffffffu : 0x55555555u);   // the image's cells
    // ---- cell after cell
    const int px = (lane & 7) * 4, py = lane >> 3;
    const size_t lane0 = tile0 + (size_t)(py * P.W + px);
#pragma unroll 1
    for (; busy; busy &= busy - 1) {
        const int cell = __ffs(busy) - 1;
        const int x = (cell & 1) * CELL_W + px, y = (cell >> 1) * CELL_H + py;
        const CellRecords recs = {__shfl_sync(0xffffffffu, mine.hit, cell), __shfl_sync(0xffffffffu, mine.edges, cell), __shfl_sync(0xffffffffu, mine.range, cell)};
        float bw[4] = {0.f, 0.f, 0.f, 0.f};
        const float2 bg = s.bg[y];
        const uint32_t bc = __float_as_uint(bg.y);
        uint32_t bl[4] = {bc, bc, bc, bc};
        if (lane == 0) n.cells += __popc(recs.hit);
        if (recs.range) raster_cell_records<true, true>(s, recs, x, s.ray_y[y], P.w_near, P.w_far, bw, bl);
        else raster_cell_records<true, false>(s, recs, x, s.ray_y[y], P.w_near, P.w_far, bw, bl);
        if ((frag_cells >> cell) & 1u) {                     // the cell's fragments meet in shared memory
            if ((int)(my_frag >> 7) == cell) atomicMax(&s.cell_key[my_frag & 127u], my_key);
            for (int f = 32 + lane; f < n_frag; f += 32) {
                const uint32_t fp = s.frag_px[f];
                if ((int)(fp >> 7) == cell) atomicMax(&s.cell_key[fp & 127u], s.frag_key(f));
            }
            __syncwarp();
            ulonglong2* ck = reinterpret_cast<ulonglong2*>(s.cell_key) + 2 * lane;
            const ulonglong2 a = ck[0], b = ck[1];
            const unsigned long long key[4] = {a.x, a.y, b.x, b.y};
            ck[0] = make_ulonglong2(0ull, 0ull); ck[1] = make_ulonglong2(0ull, 0ull);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (key[k] > (bw[k] > 0.f ? make_key(__float_as_uint(bw[k]), bl[k]) : 0ull)) { bw[k] = __uint_as_float((uint32_t)(key[k] >> 32)); bl[k] = (uint32_t)key[k]; }
        }
        const bool row_ok = y < t.th;
        const int n_px = row_ok ? t.tw - x : 0;
        if (OCC && occ) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k >= n_px) bw[k] = 0.f;
            count_visible_cell(occ, bw, bl, n_map_tris, lane);
        }
        if (n_px > 0) {
            const size_t o = lane0 + (size_t)((cell >> 1) * 4 * P.W + (cell & 1) * CELL_W);
            if (RGB) store_rgb<VEC>(P, o, bw, bl, n_map_tris, n_px);
            else store_class_depth<VEC>(P, o, bw, bl, bg.x, n_px);
        }
    }
    flush_counters(P, n);
}
