// Render kernel of calls with few tiles (included by pic_render.cu, inside namespace pic).
//
// A call of a few views -- one environment stepped interactively, a policy's unit test -- cannot fill the GPU: its time
// is the length of the chain from the first load to the last store of one tile.  Here a CTA of eight warps takes a tile
// through all of it: the warps share the culling (grid rows, large-primitive leaves and agents at the same time, then a
// thread per candidate, which also sets its primitive up), the classification of the records against the tile's 32 cells and
// the cells themselves (render_tile_kernel's, four per warp, interleaved because the crowded ones lie side by side at the
// horizon).  Fragments of small primitives meet in shared memory at once.  Nothing passes through device memory and there is
// one launch instead of three.  One environment of 64 agents, 256 tiles: a strip of eight rows per warp, keys in shared
// memory, took 28.5 us per step; this split takes 18.2 (the horizon's strip was one warp's).  The work per tile is larger than in the
// kernels for many tiles (sparser passes), so this kernel runs only up to some tiles per multiprocessor
// (launch_render_kernel).  A tile with more records than fit is rendered by cooperative_job.
#pragma once

constexpr int SMALL_THREADS = 256;
constexpr int SMALL_WARPS = SMALL_THREADS / 32;
constexpr int SMALL_LARGE = 64, SMALL_FACES = 384;              // visible large-primitive leaves, box-face items

struct __align__(16) SmallSmem {
    unsigned long long key[32][CELL_W * CELL_H];   // keys of the small primitives' fragments, cell by cell
    TileRecord rec[TREC];
    TileRecord small[SMALL_WARPS][32];             // a warp's small primitives, by lane
    f32x2 ray_xx[TILE];                            // see TileWarp
    float ray_y[TILE];
    uint32_t cells[TREC];                          // cells a record's box reaches
    CellRecords recs[32];                          // records that reach a cell
    uint32_t frag_cells;                           // cells with fragments
    Frustum f;
    uint32_t row_first[32], row_off[33];           // grid rows of a pass: first entry of the row's range in grid_prims, and the candidates before the row (all at [32])
    uint32_t lleaf[SMALL_LARGE], face[SMALL_FACES];
    int n_rec, n_leaf, n_face;
};
constexpr size_t SMALL_SMEM = sizeof(SmallSmem) > sizeof(TileSmem) ? sizeof(SmallSmem) : sizeof(TileSmem);

template <bool VEC>
__global__ void __launch_bounds__(SMALL_THREADS, 2) render_small_kernel(const __grid_constant__ RenderParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem& s = *reinterpret_cast<SmallSmem*>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned id = await_previous(blockIdx.x);
    const Job job = decode_job(P, id);
    const TileCtx& t = job.t;
    const MapInfo mi = P.env_maps[job.e];
    const AgentGeom* env_agents = P.agents + (size_t)job.e * P.A;
    const bool ego_active = __ldg(&env_agents[job.a].active) != 0u;
    bool fits = true;
    if (warp == 0) {
        frustum_setup(s.f, P, job, frustum_table(P, job, job.tile, lane), lane);
    } else if (warp == 1) {
        if (lane == 0) { s.n_rec = 0; s.n_leaf = 0; s.n_face = 0; s.frag_cells = 0u; }
        s.recs[lane] = {0u, 0u, 0u};
    } else if (warp < 4) {
        const int i = (int)threadIdx.x - 64;
        const float rx = ray_column(P, job, i);
        s.ray_xx[i] = pack2(rx, rx);
        s.ray_y[i] = ray_row(P, job, i);
    }
    {
        ulonglong2* k2 = reinterpret_cast<ulonglong2*>(s.key);
#pragma unroll
        for (int i = 0; i < TILE * TILE / 2 / SMALL_THREADS; ++i) k2[i * SMALL_THREADS + threadIdx.x] = make_ulonglong2(0ull, 0ull);
    }
    __syncthreads();
    if (ego_active) {
        const Cam& c = s.f.cam;
        const GridRows rows = grid_rows(s.f, mi);
        NoTally n;
        // ---- warp 0: the candidate ranges of the first 32 grid rows; warps 1-3: large leaves; warps 4-7: the other agents
        if (warp >= 4) {
            for (int b = (warp - 4) * 32 + lane; b < P.A; b += 128) {
                const AgentGeom g = load_agent(env_agents + b);
                uint32_t faces = (b != job.a && g.active) ? box_faces(s.f, c, t, g) : 0u;
                if (faces) {
                    int slot = atomicAdd(&s.n_face, __popc(faces));
                    for (; faces; faces &= faces - 1, ++slot)
                        if (slot < SMALL_FACES) s.face[slot] = ((uint32_t)b << 3) | (uint32_t)(__ffs(faces) - 1);
                }
            }
        } else if (warp >= 1) {
            for (uint32_t l = mi.large_begin + (warp - 1) * 32 + lane; l < mi.large_end; l += 96) {
                const Node ln = load_node(P.large_leaves + l);
                if (box_visible(s.f, ln)) {
                    const int slot = atomicAdd(&s.n_leaf, 1);
                    if (slot < SMALL_LARGE) s.lleaf[slot] = (ln.first << 3) | ln.count;
                }
            }
        }
        int n_large = 0, n_face = 0;
        for (int r0 = rows.lo;; r0 += ROW_PASS) {
            if (warp == 0) {
                uint32_t first, cnt;
                row_range(s.f, P, mi, rows, r0 + lane, first, cnt);
                uint32_t incl = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += up;
                }
                s.row_first[lane] = first;
                s.row_off[lane] = incl - cnt;
                if (lane == 31) s.row_off[32] = incl;
            }
            __syncthreads();
            if (r0 == rows.lo) {                     // the boxes' items ride with the first pass
                n_large = s.n_leaf * LARGE_LEAF_PRIMS; n_face = s.n_face;
                if (s.n_leaf > SMALL_LARGE || n_face > SMALL_FACES) { fits = false; break; }
            } else {
                n_large = 0; n_face = 0;
            }
            // ---- a thread per candidate: camera space, pixel box, set-up
            const int n_grid = (int)s.row_off[32], total = n_grid + n_large + n_face;
            for (int i0 = 0; i0 < total; i0 += SMALL_THREADS) {
                const int i = i0 + (int)threadIdx.x;
                uint32_t item = 0u;
                bool have = i < total;
                if (i < n_grid) {
                    int r = 0;
#pragma unroll
                    for (int st = 16; st; st >>= 1)
                        if (s.row_off[r + st] <= (uint32_t)i) r += st;
                    item = s.row_first[r] + ((uint32_t)i - s.row_off[r]);
                } else if (i < n_grid + n_large) {
                    const uint32_t lf = s.lleaf[(i - n_grid) / LARGE_LEAF_PRIMS], j = (uint32_t)(i - n_grid) % LARGE_LEAF_PRIMS;
                    have = j < (lf & 7u);
                    item = (lf >> 3) + j;
                } else if (have) {
                    item = SURV_FACE | s.face[i - n_grid - n_large];
                }
                V3 V[4], Pn;
                uint32_t key_lo = 0u, flags = 0u, box = 0u;
                bool keep = false;
                if (have) {
                    fetch_survivor(c, P, item, job.e, mi.n_tris, V, Pn, key_lo, flags);
                    keep = pixel_box(c, t, V, box);
                }
                PrimEq q;
                const bool ok = keep && prim_equations(V, flags & 1u, flags, Pn, q);
                const int bx0 = box & 0xff, by0 = (box >> 8) & 0xff, w = (int)((box >> 16) & 0xff) - bx0 + 1, h = (int)(box >> 24) - by0 + 1;
                const bool small = ok && w * h <= SMALL_PIXELS, big = ok && !small;
                const unsigned m = __ballot_sync(0xffffffffu, big);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&s.n_rec, __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0);
                const int slot = base + __popc(m & ((1u << lane) - 1u));
                if (big && slot < TREC) { s.rec[slot].write(q, key_lo); s.cells[slot] = box_cells(box); }
                if (__any_sync(0xffffffffu, small)) {
                    if (small) s.small[warp][lane].write(q, key_lo);
                    small_pixels(s.small[warp], s.ray_xx, s.ray_y, small, bx0, by0, w, h, P.w_near, P.w_far, lane, [&](bool in, float wv, uint32_t lo, int x, int y) {
                        if (!in) return;
                        const uint32_t at = cell_pixel(x, y);
                        atomicMax(&s.key[at >> 7][at & 127u], make_key(__float_as_uint(wv), lo));
                        if (!((s.frag_cells >> (at >> 7)) & 1u)) atomicOr(&s.frag_cells, 1u << (at >> 7));
                    });
                    __syncwarp();
                }
            }
            __syncthreads();
            if (!rows_after(r0, rows.hi)) break;
        }
        if (fits) fits = s.n_rec <= TREC;
        if (!fits) {
            __syncthreads();                         // (the job takes over the CTA's shared memory)
            cooperative_job<NoTally, SMALL_THREADS>(*reinterpret_cast<TileSmem*>(smem_raw), P, id, n);
            return;
        }
    }
    // ---- the records of every cell: warp w looks at records w, w + 8, ...
    const int n_rec = ego_active ? s.n_rec : 0;
    if (n_rec > 0) {
        NoTally n;
        const CellRecords mine = classify_records(s, n_rec, true, P.w_near, P.w_far, lane, n, warp, SMALL_WARPS);
        if (mine.hit) {
            atomicOr(&s.recs[lane].hit, mine.hit);
            atomicOr(&s.recs[lane].edges, mine.edges);
            if (mine.range) atomicOr(&s.recs[lane].range, mine.range);
        }
    }
    __syncthreads();
    // ---- cells w, w + 8, ... by warp w: four adjacent pixels per lane
    const uint32_t frag_cells = s.frag_cells;
    const size_t tile0 = job.view * ((size_t)P.H * P.W) + (size_t)t.y0 * P.W + t.x0;
    const int px = (lane & 7) * 4, py = lane >> 3;
#pragma unroll 1
    for (int cell = warp; cell < 32; cell += SMALL_WARPS) {
        const int x = (cell & 1) * CELL_W + px, y = (cell >> 1) * CELL_H + py;
        const int n_px = y < t.th ? t.tw - x : 0;
        uint32_t bc = P.cls_sky;
        float bz = P.far_z;
        if (ego_active && n_px > 0) { bc = __ldg(P.rig.bg_cls + (size_t)job.k * P.H + t.y0 + y); bz = __ldg(P.rig.bg_z + (size_t)job.k * P.H + t.y0 + y); }
        float bw[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t bl[4] = {bc, bc, bc, bc};
        if ((frag_cells >> cell) & 1u) {
            const ulonglong2* ck = reinterpret_cast<const ulonglong2*>(s.key[cell]) + 2 * lane;
            const ulonglong2 a = ck[0], b = ck[1];
            const unsigned long long key[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (key[k]) { bw[k] = __uint_as_float((uint32_t)(key[k] >> 32)); bl[k] = (uint32_t)key[k]; }
        }
        raster_cell_records<false, true>(s, s.recs[cell], x, s.ray_y[y], P.w_near, P.w_far, bw, bl);
        if (n_px > 0) {
            store_class_depth<VEC>(P, tile0 + (size_t)(y * P.W + x), bw, bl, bz, n_px);
        }
    }
}

cudaError_t configure_small_kernel() {
    const cudaError_t err = cudaFuncSetAttribute(render_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM);
    return err != cudaSuccess ? err : cudaFuncSetAttribute(render_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM);
}
