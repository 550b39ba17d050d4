// Set-up kernel (agents, rig tables), exhaustive cross-check kernel and host-side launchers.
//
// The exhaustive kernel (see pic_exhaustive.cuh) is the cross-check of the production kernels in
// pic_render.cu.
#include "pic_exhaustive.cuh"

namespace pic {

struct RigParams {
    int32_t K, W, H;
    float near_z, far_z;
    uint32_t cls_sky, cls_ground;
    const uint32_t* palette;      // NULL: no colours are rendered
    int32_t tiles_x, tiles;       // of a view
    FastDiv div_tiles_x;
    SetupGrid grid;
    CamConst cam[MAX_CAMS];
};

// ------------------------------------------------------------------------------------------------
// set-up kernel, agents: poses/dims/active -> AgentGeom + one ViewCam per camera (optionally after one
// kinematic-bicycle step of the scene's own state)
// ------------------------------------------------------------------------------------------------
struct AgentArgs {
    int n;
    const float* poses;
    float* state;
    const float* actions;
    const float* dims;
    const uint8_t* active;
    const uint8_t* agent_cls;
    uint32_t default_cls;
    AgentGeom* out;
    ViewCam* cams;
    uint32_t* status;
    float dt, wheelbase, v_max;
};

// One agent: its kinematic step, geometry and camera records.
__device__ __forceinline__ void agent_setup(const AgentArgs& G, const RigParams& R, int i) {
    const float* __restrict__ poses = G.poses;
    const float* __restrict__ actions = G.actions;
    const float* __restrict__ dims = G.dims;
    float* state = G.state;
    const float dt = G.dt, wheelbase = G.wheelbase, v_max = G.v_max;
    const uint8_t* __restrict__ active = G.active;
    uint32_t* status = G.status;
    bool act = active ? active[i] != 0 : true;
    float x, y, th;
    if (state) {                                   // pic_step: update the scene's own state in place
        float v;
        x = state[4 * i]; y = state[4 * i + 1]; th = state[4 * i + 2]; v = state[4 * i + 3];
        if (actions && act) {
            const float acc = actions[2 * i], steer = actions[2 * i + 1];
            float s, c;
            sincosf(th, &s, &c);
            const float nx = fm(mul(v, c), dt, x);
            const float ny = fm(mul(v, s), dt, y);
            const float nth = fm(mul(__fdiv_rn(v, wheelbase), tanf(steer)), dt, th);
            const float nv = fminf(fmaxf(fm(acc, dt, v), 0.f), v_max);
            if (isfinite(acc) && isfinite(steer) && isfinite(nx) && isfinite(ny) && isfinite(nth) && isfinite(nv)) {
                x = nx; y = ny; th = nth; v = nv;
                state[4 * i] = x; state[4 * i + 1] = y; state[4 * i + 2] = th; state[4 * i + 3] = v;
            } else {
                // a non-finite action (or a step that overflows) is flagged, leaves the agent's
                // state as it was and takes the agent out of this step's images
                atomicOr(status, 1u);
                act = false;
            }
        }
    } else {
        x = poses[3 * i]; y = poses[3 * i + 1]; th = poses[3 * i + 2];
    }
    float l = dims[3 * i], w = dims[3 * i + 1], h = dims[3 * i + 2];
    if (!(isfinite(x) && isfinite(y) && isfinite(th) && isfinite(l) && isfinite(w) && isfinite(h))) {
        atomicOr(status, 1u);
        act = false;
        x = y = th = 0.f; l = w = h = 1.f;
    }
    AgentGeom g;
    g.x = x; g.y = y;
    sincosf(th, &g.s, &g.c);
    g.hl = 0.5f * l; g.hw = 0.5f * w; g.h = h;
    g.active = act ? (1u | ((G.agent_cls ? (uint32_t)G.agent_cls[i] : G.default_cls) << 8)) : 0u;
    G.out[i] = g;
    for (int k = 0; k < R.K; ++k) {
        ViewCam vc;
        make_view_cam(vc, g, R.cam[k]);
        float4* dst = reinterpret_cast<float4*>(G.cams + (size_t)i * R.K + k);
        const float4* src = reinterpret_cast<const float4*>(&vc);
        dst[0] = src[0]; dst[1] = src[1]; dst[2] = src[2]; dst[3] = src[3];
    }
}

// Entry i of camera k's tables: the ray coordinate of a pixel column, or that of a pixel row and the row's background.
__device__ __forceinline__ void rig_setup(const RigParams& R, int k, int i, const RigTables& T) {
    const CamConst c = R.cam[k];
    const int nx = ray_stride(R.W), ny = ray_stride(R.H), v = i - nx;
    if (v >= ny) return;
    const bool column = v < 0;
    const float ray = __fdiv_rn(sub(add((float)(column ? i : v), 0.5f), 0.5f * (float)(column ? R.W : R.H)), column ? c.fx : c.fy);
    if (column) {
        const_cast<float*>(T.ray_x)[(size_t)k * nx + i] = ray;
        return;
    }
    const_cast<float*>(T.ray_y)[(size_t)k * ny + v] = ray;
    if (v >= R.H) return;
    uint32_t cls; float z;
    background(c.cphi, c.sphi, c.mz, ray, R.far_z, R.cls_sky, R.cls_ground, cls, z);
    const size_t at = (size_t)k * R.H + v;
    const_cast<float*>(T.bg_z)[at] = z;
    const_cast<uint32_t*>(T.bg_cls)[at] = cls;
    if (R.palette) const_cast<uint32_t*>(T.bg_rgb)[at] = R.palette[cls];
}

// Entry i of the frusta of camera k's tiles and of its whole image.
__device__ __forceinline__ void frusta_setup(const RigParams& R, int k, int i, const RigTables& T) {
    const CamConst c = R.cam[k];
    const float cx = 0.5f * (float)R.W, cy = 0.5f * (float)R.H;
    const int tiles = R.tiles;
    if (i >= (tiles + 1) * FRUSTUM_ENTRIES) return;
    const int t = i / FRUSTUM_ENTRIES, ty = (int)divide((unsigned)t, R.div_tiles_x), x0 = (t - ty * R.tiles_x) * TILE, y0 = ty * TILE;
    const bool whole = t == tiles;
    const_cast<float4*>(T.frusta)[(size_t)k * (tiles + 1) * FRUSTUM_ENTRIES + i] =
        frustum_entry(i % FRUSTUM_ENTRIES, whole ? -cx : (float)x0 - cx, (float)(whole ? R.W : min(x0 + TILE, R.W)) - cx, whole ? -cy : (float)y0 - cy,
                      (float)(whole ? R.H : min(y0 + TILE, R.H)) - cy, c.fx, c.fy, R.near_z, R.far_z);
}

// One launch prepares a call (who does what: setup_item).  Bound by the length of a thread's chain: an entry of the tables or the frusta per
// thread, since a block per camera that goes through them is the longest chain of a call of a few views of many pixels, and the divisions that find
// an entry by numbers fixed per call.  One view, class and depth, a block per camera for both / for the tables / an entry per thread: an empty
// map at 2 160 x 3 840 111 / 21.2 / 18.5 us, a town at 2 160 x 3 840 124 / 35.1 / 31.6 (colours 132 / 43.2 / 39.2), one tile with eight agents
// 8.8 / 9.1 / 8.8 on the GPU alone.
__global__ void __launch_bounds__(SETUP_THREADS) setup_kernel(const __grid_constant__ AgentArgs G, const __grid_constant__ RigParams R,
                                                              const __grid_constant__ RigTables T, uint32_t* overflow) {
    launch_dependents();
    if (overflow && blockIdx.x == 0 && threadIdx.x == 0) overflow[0] = 0u;   // the render kernels' list of left-out tiles starts empty (absent for callers that do not use them)
    const SetupItem it = setup_item(R.grid, (int)blockIdx.x, (int)threadIdx.x);
    if (it.role == SETUP_TABLES) rig_setup(R, it.camera, it.index, T);
    else if (it.role == SETUP_FRUSTA) frusta_setup(R, it.camera, it.index, T);
    else if (it.index < G.n) agent_setup(G, R, it.index);
}

// ------------------------------------------------------------------------------------------------
// exhaustive kernel: the scene's preprocessed primitives through the shared exhaustive tile renderer
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(EXH_THREADS) render_brute_kernel(const __grid_constant__ RenderParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExhaustiveSmem& s = *reinterpret_cast<ExhaustiveSmem*>(smem_raw);
    const unsigned tiles = (unsigned)(P.tiles_x * P.tiles_y);
    const int e = (int)(((size_t)P.view_first + blockIdx.x / tiles) / ((size_t)P.K * P.A));
    const MapInfo mi = P.maps[P.env_map[e]];
    const Prim* prims = P.prims + mi.prim_begin;
    exhaustive_tile(s, P, blockIdx.x, mi.prim_end - mi.prim_begin, mi.n_tris,
                    [prims](uint32_t i, const Cam& c, V3 (&V)[4], V3& Pn, bool& quad, uint32_t& flags, uint32_t& key_lo) {
                        float v[12], vis_cos;
                        load_prim(prims + i, v, key_lo, flags, vis_cos);
                        quad = flags & 1u;
#pragma unroll
                        for (int j = 0; j < 4; ++j) V[j] = to_camera(c, v[3 * j], v[3 * j + 1], v[3 * j + 2]);
                        Pn = limit_angular_range(V, plane_normal_world(c, v, quad), vis_cos);
                    });
}

// ------------------------------------------------------------------------------------------------
// host-side launchers (called from the C ABI)
// ------------------------------------------------------------------------------------------------
size_t render_smem_bytes();                       // pic_render.cu
cudaError_t configure_render_kernel();            // pic_render.cu
cudaError_t launch_render_kernel(const RenderParams& P, long long n_views, int sm_count, cudaStream_t stream);
cudaError_t launch_coverage_kernel(const RenderParams& P, long long n_views, cudaStream_t stream);
cudaError_t configure_colour_kernel();            // pic_colour.cuh (part of pic_render.cu)
cudaError_t launch_colour_kernel(const RenderParams& P, long long n_views, bool antialias, int sm_count, cudaStream_t stream);

size_t max_smem_bytes() { return render_smem_bytes() > sizeof(ExhaustiveSmem) ? render_smem_bytes() : sizeof(ExhaustiveSmem); }

cudaError_t configure_kernels() {
    cudaError_t err = configure_render_kernel();
    if (err != cudaSuccess) return err;
    err = configure_colour_kernel();
    if (err != cudaSuccess) return err;
    return cudaFuncSetAttribute(render_brute_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ExhaustiveSmem));
}

static RigParams rig_params(const RenderParams& P) {
    RigParams R;
    R.K = P.K; R.W = P.W; R.H = P.H; R.near_z = P.near_z; R.far_z = P.far_z; R.cls_sky = P.cls_sky; R.cls_ground = P.cls_ground;
    R.palette = P.out_rgb ? P.palette : nullptr;
    R.tiles_x = P.tiles_x; R.tiles = P.tiles_x * P.tiles_y;
    R.div_tiles_x = P.div_tiles_x;
    for (int k = 0; k < MAX_CAMS; ++k) R.cam[k] = P.cam[k];
    return R;
}

// Per call: rig tables, agents (+ optional bicycle step) and their cameras.
cudaError_t launch_setup(const RenderParams& P, int n_agents, const float* poses, float* state, const float* actions,
                         const float* dims, const uint8_t* active, const uint8_t* agent_cls, AgentGeom* agents_out, ViewCam* cams_out,
                         uint32_t* status, float dt, float wheelbase, float v_max, cudaStream_t stream) {
    RigParams R = rig_params(P);
    AgentArgs G;
    G.n = n_agents; G.poses = poses; G.state = state; G.actions = actions; G.dims = dims; G.active = active;
    G.agent_cls = agent_cls; G.default_cls = P.cls_agent; G.out = agents_out; G.cams = cams_out; G.status = status;
    G.dt = dt; G.wheelbase = wheelbase; G.v_max = v_max;
    R.grid = setup_grid(P.K, P.div_K, P.H, P.W, P.rig.frusta ? R.tiles : 0, n_agents);
    setup_kernel<<<setup_blocks(R.grid), SETUP_THREADS, 0, stream>>>(G, R, P.rig, P.overflow);
    return cudaGetLastError();
}

cudaError_t launch_colour(const RenderParams& P, long long n_views, bool antialias, int sm_count, cudaStream_t stream) {
    return n_views <= 0 ? cudaSuccess : launch_colour_kernel(P, n_views, antialias, sm_count, stream);
}

cudaError_t launch_render(const RenderParams& P, long long n_views, bool brute, int sm_count, cudaStream_t stream) {
    if (n_views <= 0) return cudaSuccess;
    if (!brute) return launch_render_kernel(P, n_views, sm_count, stream);
    const long long blocks = n_views * P.tiles_x * P.tiles_y;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    render_brute_kernel<<<(unsigned)blocks, EXH_THREADS, sizeof(ExhaustiveSmem), stream>>>(P);
    const cudaError_t err = cudaGetLastError();
    return err != cudaSuccess ? err : launch_coverage_kernel(P, n_views, stream);
}

}  // namespace pic
