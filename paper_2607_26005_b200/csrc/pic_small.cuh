// Render kernel of calls with few tiles (included by pic_render.cu, inside namespace pic).
//
// A call of a few views -- one environment stepped interactively, a policy's unit test -- cannot fill the GPU: its time
// is the length of the chain from the first load to the last store of one tile.  Here a CTA of eight warps takes a tile
// through all of it: the warps share the culling (grid rows, large-primitive leaves and agents at the same time, then a
// thread per candidate, which also sets its primitive up), and each rasterizes and stores a strip of eight rows.  Nothing
// passes through device memory and there is one launch instead of two (cull, render) or three.  The work per tile is
// larger than in the kernels for many tiles (passes are sparser, every record is looked at in twice as many strips), so
// this kernel runs only while its CTAs are all resident at once (launch_render_kernel).
#pragma once

constexpr int SMALL_THREADS = 256;
constexpr int SMALL_STRIP = TILE / (SMALL_THREADS / 32);        // rows of a strip: one strip per warp
constexpr int SMALL_POOL = 192;                                 // records; a tile with more survivors is rendered by cooperative_job
constexpr int SMALL_LARGE = 64, SMALL_FACES = 384;              // visible large-primitive leaves, box-face items
static_assert(SMALL_STRIP == 8, "strips of 8 rows");

struct __align__(16) SmallSmem {
    unsigned long long key[TILE * TILE];
    RecordPool<SMALL_POOL> pool;
    float ray_x[TILE], ray_y[TILE];
    Frustum f;
    uint32_t row_first[32], row_off[33];       // candidate ranges of the grid rows of a pass (see FrontLists)
    uint32_t lleaf[SMALL_LARGE], face[SMALL_FACES];
    int n_rec, n_leaf, n_face;
};
constexpr size_t SMALL_SMEM = sizeof(SmallSmem) > sizeof(TileSmem) ? sizeof(SmallSmem) : sizeof(TileSmem);

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
        frustum_setup(s.f, P, job, lane);
    } else if (warp == 1) {
        if (lane == 0) { s.n_rec = 0; s.n_leaf = 0; s.n_face = 0; }
    } else if (warp < 4) {
        load_rays(s, P, job, threadIdx.x - 64);
    }
    {
        ulonglong2* k2 = reinterpret_cast<ulonglong2*>(s.key + warp * SMALL_STRIP * TILE);
#pragma unroll
        for (int i = 0; i < SMALL_STRIP * TILE / 2 / 32; ++i) k2[i * 32 + lane] = make_ulonglong2(0ull, 0ull);
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
        for (int r0 = rows.lo;; r0 += 32) {
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
                const unsigned m = __ballot_sync(0xffffffffu, keep);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&s.n_rec, __popc(m));
                base = __shfl_sync(0xffffffffu, base, 0);
                const int slot = base + __popc(m & ((1u << lane) - 1u));
                if (keep && slot < SMALL_POOL) {
                    PrimEq q;
                    if (!prim_equations(V, flags & 1u, flags, Pn, q)) s.pool.box[slot] = REC_DEAD;
                    else write_record(s.pool, slot, q, key_lo, box, (tiny_box(box) ? REC_TINY : 0u) | (record_in_range(V, P) ? REC_INRANGE : 0u));
                }
            }
            __syncthreads();
            if (r0 + 32 > rows.hi) break;
        }
        if (fits) fits = s.n_rec <= SMALL_POOL;
        if (!fits) {
            __syncthreads();                         // (the job takes over the CTA's shared memory)
            cooperative_job<NoTally, SMALL_THREADS>(*reinterpret_cast<TileSmem*>(smem_raw), P, id, n);
            return;
        }
    }
    // ---- a strip of eight rows per warp
    const int ys = warp * SMALL_STRIP;
    if (ys >= t.th) return;
    StripView sv;
    sv.key = s.key + ys * TILE; sv.ray_x = s.ray_x; sv.ray_y = s.ray_y + ys;
    uint32_t touched = 0u;
    if (ego_active) touched = raster_strip<SMALL_STRIP>(sv, s.pool, 0, s.n_rec, ys, P.w_near, P.w_far, lane);
    __syncwarp();
    TileCtx ts = t;
    ts.y0 = t.y0 + ys; ts.th = min(SMALL_STRIP, t.th - ys);
    store_tile(sv, ts, P, job.view, job.k, ego_active, (unsigned long long)touched, false, lane, 32);
}

cudaError_t configure_small_kernel() {
    return cudaFuncSetAttribute(render_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMALL_SMEM);
}
