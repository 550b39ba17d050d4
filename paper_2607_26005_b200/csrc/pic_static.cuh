// Render kernel of pic_render_static (included by pic_render.cu, inside namespace pic): the caller's raw triangles, no
// hierarchy, no memory but the caller's and the library's static scratch.
//
// A CTA takes one tile.  Every triangle and box face is tested against the tile, a thread each (camera space, pixel
// box -- the conservative test of the other kernels); the survivors are compacted, set up a thread each, and rasterized
// like the cooperative kernel's records: a few pixels by their thread, the others cell by cell by the warp that owns the
// rows.  Bound by latency: the batches this call is meant for fill the GPU less than once, so a tile is cut into 32- or
// 16-row pieces (each tests all the items again, which costs less than the wait for the longest tile) while the launch
// would leave multiprocessors idle.  Before, every item visited every pixel: 1 env x 16 agents x 2 cameras at 96 x 128
// with 792 triangles took 1 737 us.
#pragma once

struct StaticParams {
    RenderParams P;              // tiles_y counts pieces of tile_h rows
    const float* tri_xyz;        // dev [N,3,3]
    const uint8_t* tri_class;    // dev [N]
    uint32_t n_tris;
    int32_t tile_h;              // rows of a tile: 64, 32 or 16
};

constexpr int STATIC_RCAP = 128;          // records (and survivors set up) at a time
constexpr int STATIC_SCAP = 256;          // survivors kept before they are set up; a round adds at most NTHREADS

struct __align__(16) StaticSmem {
    unsigned long long key[TILE * TILE];
    float4 rec[STATIC_RCAP * REC / 4];
    uint2 surv[STATIC_SCAP];              // (item, pixel box)
    float ray_x[TILE], ray_y[TILE];
    Cam cam;
    int n_rec, n_surv;
    uint32_t touched[2];
};
static_assert(STATIC_SCAP >= 2 * NTHREADS && STATIC_RCAP <= NTHREADS, "a round's survivors fit; a thread sets up one survivor of a batch");

__device__ __forceinline__ bool lex_less(float ax, float ay, float az, float bx, float by, float bz) {
    if (ax != bx) return ax < bx;
    if (ay != by) return ay < by;
    return az < bz;
}

// Item i of the tile -- triangle i, or face (i - n_tris) of the environment's boxes -- in camera space; false: not drawn.
__device__ __forceinline__ bool static_item(const StaticParams& S, const Cam& c, const Job& job, uint32_t i, bool want_plane, V3 (&V)[4], V3& Pn,
                                            uint32_t& flags, uint32_t& key_lo) {
    if (i < S.n_tris) {
        const float* p = S.tri_xyz + 9 * (size_t)i;
        float v[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) v[j] = __ldg(p + j);
#pragma unroll
        for (int j = 0; j < 3; ++j) V[j] = to_camera(c, v[3 * j], v[3 * j + 1], v[3 * j + 2]);
        V[3] = V[2];
        if (want_plane) {
            const float v12[12] = {v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[6], v[7], v[8]};
            Pn = plane_normal_world(c, v12, false);
            flags = 0u;
            // an edge shared by two triangles is evaluated in the same direction by both
            if (!lex_less(v[0], v[1], v[2], v[3], v[4], v[5])) flags |= 1u << 4;
            if (!lex_less(v[3], v[4], v[5], v[6], v[7], v[8])) flags |= 1u << 5;
            if (!lex_less(v[6], v[7], v[8], v[0], v[1], v[2])) flags |= 1u << 6;
            key_lo = ((0xFFFFFFu - i) << 8) | __ldg(S.tri_class + i);
        }
        return true;
    }
    const uint32_t j = i - S.n_tris;
    const int b = (int)(j / 6u), f = (int)(j % 6u);
    if (b == job.a) return false;
    const AgentGeom g = S.P.agents[(size_t)job.e * S.P.A + b];
    if (!g.active) return false;
    const uint32_t corners = face_corners(f);
#pragma unroll
    for (int q = 0; q < 4; ++q) V[q] = box_corner(c, g, (corners >> (4 * q)) & 7u);
    if (want_plane) {
        flags = face_flags(corners);
        key_lo = ((0xFFFFFFu - (S.n_tris + 12u * (uint32_t)b + 2u * (uint32_t)f)) << 8) | agent_box_class(g);
        Pn = plane_normal(V, true);
    }
    return true;
}

__global__ void __launch_bounds__(NTHREADS, 4) render_static_kernel(const __grid_constant__ StaticParams S) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StaticSmem& s = *reinterpret_cast<StaticSmem*>(smem_raw);
    const RenderParams& P = S.P;
    const int lane = threadIdx.x & 31;
    const Job job = decode_job(P, blockIdx.x, S.tile_h);
    const TileCtx& t = job.t;
    const bool ego_active = P.agents[(size_t)job.e * P.A + job.a].active != 0;
    if (threadIdx.x == 0) {
        load_camera(s.cam, P.cams[job.view], P.cam[job.k], P.W, P.H);
        s.n_rec = 0; s.n_surv = 0;
        s.touched[0] = 0u; s.touched[1] = 0u;
    } else if (threadIdx.x >= 64) {
        load_rays(s, P, job, threadIdx.x - 64);
    }
    for (int i = threadIdx.x; i < TILE * S.tile_h / 2; i += NTHREADS) reinterpret_cast<ulonglong2*>(s.key)[i] = make_ulonglong2(0ull, 0ull);
    __syncthreads();
    if (ego_active) {
        const Cam& c = s.cam;
        NoTally n;
        const uint32_t n_items = S.n_tris + 6u * (uint32_t)P.A;
        int ns = 0;                            // survivors in the list (every thread keeps count)
        for (uint32_t i0 = 0; i0 < n_items; i0 += NTHREADS) {
            // ---- a thread per item: which can touch a pixel centre of the tile?
            const uint32_t i = i0 + threadIdx.x;
            V3 V[4], Pn;
            uint32_t flags, key_lo, box = 0u;
            const bool keep = i < n_items && static_item(S, c, job, i, false, V, Pn, flags, key_lo) && pixel_box(c, t, V, box);
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            int base = 0;
            if (lane == 0 && m) base = atomicAdd(&s.n_surv, __popc(m));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (keep) s.surv[base + __popc(m & ((1u << lane) - 1u))] = make_uint2(i, box);
            ns += __syncthreads_count(keep);
            if (ns + NTHREADS <= STATIC_SCAP && i0 + NTHREADS < n_items) continue;
            // ---- a thread per survivor: edge functions, 1/z plane; then the records, STATIC_RCAP at a time
            for (int j0 = 0; j0 < ns; j0 += STATIC_RCAP) {
                const int j = j0 + (int)threadIdx.x;
                if (j < ns) {
                    const uint2 sv = s.surv[j];
                    static_item(S, c, job, sv.x, true, V, Pn, flags, key_lo);
                    setup_prim(s, t, V, flags & 1u, flags, Pn, key_lo, sv.y, STATIC_RCAP, n);
                }
                __syncthreads();
                raster_records<NW>(s, s.rec, s.touched, t, s.n_rec, true, n);
                __syncthreads();
                if (threadIdx.x == 0) { s.n_rec = 0; s.n_surv = 0; }
                __syncthreads();
            }
            ns = 0;
        }
    }
    store_tile(s, t, P, job.view, job.k, ego_active, ((unsigned long long)s.touched[1] << 32) | s.touched[0]);
}

cudaError_t configure_static_kernel() {
    return cudaFuncSetAttribute(render_static_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StaticSmem));
}

cudaError_t launch_static_kernel(const RenderParams& P, const float* tri_xyz, const uint8_t* tri_class, int n_tris, int sm_count, cudaStream_t stream) {
    StaticParams S;
    S.P = P;
    S.tri_xyz = tri_xyz; S.tri_class = tri_class; S.n_tris = (uint32_t)n_tris;
    S.tile_h = TILE;
    const long long views = (long long)P.E * P.A * P.K * P.tiles_x;
    // (two CTAs per multiprocessor are enough to hide the latency of the tests)
    while (S.tile_h > 16 && views * ((P.H + S.tile_h - 1) / S.tile_h) < 2LL * sm_count) S.tile_h >>= 1;
    S.P.tiles_y = (P.H + S.tile_h - 1) / S.tile_h;
    set_divisors(S.P);
    render_static_kernel<<<(unsigned)(views * S.P.tiles_y), NTHREADS, sizeof(StaticSmem), stream>>>(S);
    return cudaGetLastError();
}
