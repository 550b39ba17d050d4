// pic_render_static: a self-contained render call for hosts that must not allocate device memory.
//
// Everything the ordinary path keeps in buffers obtained with cudaMalloc when a scene is created --
// per-agent geometry, per-view cameras, per-camera ray/background tables, the status word -- lives
// here in ONE file-scope device array of fixed size.  The map is read straight from the caller's
// triangle arrays (no hierarchy is built), so the call needs no scene object at all.
//
// In host code the name of a __device__ array is only a stand-in for the symbol, not an address a
// kernel can use; its device address is looked up with cudaGetSymbolAddress, once per device,
// with that device current, and handed to the kernels as an ordinary pointer.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "../../include/pictura.h"
#include "pic_types.h"

namespace pic {
cudaError_t launch_setup(const RenderParams& P, int n_agents, const float* poses, float* state, const float* actions,
                         const float* dims, const uint8_t* active, const uint8_t* agent_cls, AgentGeom* agents_out, ViewCam* cams_out,
                         uint32_t* status, float dt, float wheelbase, float v_max, cudaStream_t stream);
cudaError_t configure_static_kernel();            // pic_static.cuh (part of pic_render.cu)
cudaError_t launch_static_kernel(const RenderParams& P, const float* tri_xyz, const uint8_t* tri_class, int n_tris, int sm_count, cudaStream_t stream);
void set_last_error(const char* msg);
}  // namespace pic

namespace {

using namespace pic;

constexpr int kMaxAgents = PIC_STATIC_MAX_AGENTS;
constexpr int kMaxViews = PIC_STATIC_MAX_VIEWS;
constexpr int kMaxSide = PIC_STATIC_MAX_SIDE;
constexpr int kMaxDevices = 64;

// scratch layout (bytes)
constexpr size_t kOffAgents = 0;
constexpr size_t kOffCams = kOffAgents + sizeof(AgentGeom) * kMaxAgents;
constexpr size_t kOffTables = kOffCams + sizeof(ViewCam) * kMaxViews;
constexpr size_t kOffStatus = kOffTables + table_bytes(MAX_CAMS, kMaxSide, kMaxSide);
constexpr size_t kScratchBytes = kOffStatus + 256;

// The only device memory this entry point ever uses besides the caller's buffers (about 470 KB,
// held by every device that loads the library until the process exits).
static __device__ __align__(256) unsigned char g_static_scratch[kScratchBytes];

std::mutex g_mutex;
unsigned char* g_scratch_ptr[kMaxDevices] = {};     // device address of g_static_scratch, per device
int g_sm_count[kMaxDevices] = {};

pic_status fail(pic_status st, const char* fmt, ...) {
    char buf[384];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    pic::set_last_error(buf);
    return st;
}

}  // namespace

extern "C" pic_status pic_render_static(const pic_static_desc* d, const float* tri_xyz, const uint8_t* tri_class,
                                        const float* poses, const float* dims, const uint8_t* active,
                                        const pic_camera* rig, uint8_t* out_class, uint16_t* out_depth, void* cuda_stream) {
    if (!d) return fail(PIC_ERR_INVALID_ARG, "desc is NULL");
    if (d->size != sizeof(pic_static_desc)) return fail(PIC_ERR_INVALID_ARG, "desc->size is %u, expected %zu", d->size, sizeof(pic_static_desc));
    if (d->E <= 0 || d->A <= 0 || d->K <= 0 || d->H <= 0 || d->W <= 0 || d->n_tris < 0) return fail(PIC_ERR_SHAPE, "sizes must be positive");
    if (d->K > MAX_CAMS) return fail(PIC_ERR_SHAPE, "at most %d cameras per rig", MAX_CAMS);
    if ((long long)d->E * d->A > kMaxAgents)
        return fail(PIC_ERR_CAPACITY, "pic_render_static holds at most %d agents (E*A), got %lld", kMaxAgents, (long long)d->E * d->A);
    if ((long long)d->E * d->A * d->K > kMaxViews)
        return fail(PIC_ERR_CAPACITY, "pic_render_static holds at most %d views (E*A*K), got %lld", kMaxViews, (long long)d->E * d->A * d->K);
    if (d->H > kMaxSide || d->W > kMaxSide)
        return fail(PIC_ERR_CAPACITY, "pic_render_static renders images up to %d x %d, got %d x %d", kMaxSide, kMaxSide, d->H, d->W);
    if (d->n_tris > PIC_STATIC_MAX_TRIS) return fail(PIC_ERR_CAPACITY, "pic_render_static reads at most %d triangles, got %d", PIC_STATIC_MAX_TRIS, d->n_tris);
    {
        // any primitive may cover every pixel of every view: bound the product, so that a request at all
        // the limits at once cannot occupy the GPU for hours
        const double work = ((double)d->n_tris + 6.0 * d->A) * (double)d->E * d->A * d->K * (double)d->H * d->W;
        if (work > (double)PIC_STATIC_MAX_WORK)
            return fail(PIC_ERR_CAPACITY, "pic_render_static: (n_tris + 6A) * E*A*K*H*W = %.3g primitive-pixel tests, at most %.3g", work,
                        (double)PIC_STATIC_MAX_WORK);
    }
    if (!(d->near_z > 0.f) || !(d->far_z > d->near_z) || !std::isfinite(d->far_z)) return fail(PIC_ERR_INVALID_ARG, "need 0 < near_z < far_z < inf");
    if (!poses || !dims || !rig || !out_class || !out_depth) return fail(PIC_ERR_INVALID_ARG, "a required pointer is NULL");
    if (d->n_tris > 0 && (!tri_xyz || !tri_class)) return fail(PIC_ERR_INVALID_ARG, "triangle arrays are NULL");
    for (int k = 0; k < d->K; ++k) {
        const float vals[7] = {rig[k].mount_x, rig[k].mount_y, rig[k].mount_z, rig[k].yaw, rig[k].pitch, rig[k].fx, rig[k].fy};
        for (float v : vals)
            if (!std::isfinite(v)) return fail(PIC_ERR_INVALID_ARG, "camera %d has a non-finite field", k);
        if (!(rig[k].fx > 0.f) || !(rig[k].fy > 0.f)) return fail(PIC_ERR_INVALID_ARG, "camera %d: focal lengths must be positive", k);
    }
    int dev = -1;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(ce));
    if (dev < 0 || dev >= kMaxDevices) return fail(PIC_ERR_INVALID_ARG, "device ordinal %d not supported", dev);
    unsigned char* scratch = nullptr;
    {
        // once per device, with that device current: the device address of the static array
        std::lock_guard<std::mutex> lock(g_mutex);
        if (!g_scratch_ptr[dev]) {
            void* p = nullptr;
            ce = cudaGetSymbolAddress(&p, g_static_scratch);
            if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(ce));
            ce = pic::configure_static_kernel();
            if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(ce));
            ce = cudaDeviceGetAttribute(&g_sm_count[dev], cudaDevAttrMultiProcessorCount, dev);
            if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "cudaDeviceGetAttribute: %s", cudaGetErrorString(ce));
            g_scratch_ptr[dev] = static_cast<unsigned char*>(p);
        }
        scratch = g_scratch_ptr[dev];
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    RenderParams P;
    memset(&P, 0, sizeof(P));
    P.E = d->E; P.A = d->A; P.K = d->K; P.H = d->H; P.W = d->W;
    P.tiles_x = (d->W + TILE - 1) / TILE; P.tiles_y = (d->H + TILE - 1) / TILE;
    set_divisors(P);
    P.near_z = d->near_z; P.far_z = d->far_z; P.w_near = 1.0f / d->near_z; P.w_far = 1.0f / d->far_z;
    P.cls_agent = d->agent_class; P.cls_sky = d->sky_class; P.cls_ground = d->ground_class;
    AgentGeom* agents = reinterpret_cast<AgentGeom*>(scratch + kOffAgents);
    ViewCam* cams = reinterpret_cast<ViewCam*>(scratch + kOffCams);
    float* tables = reinterpret_cast<float*>(scratch + kOffTables);
    uint32_t* status = reinterpret_cast<uint32_t*>(scratch + kOffStatus);
    P.agents = agents; P.cams = cams;
    P.rig = rig_tables(tables, d->K, d->H, d->W, nullptr);
    P.out_class = out_class; P.out_depth = out_depth;
    for (int k = 0; k < d->K; ++k) {
        CamConst& o = P.cam[k];
        o.mx = rig[k].mount_x; o.my = rig[k].mount_y; o.mz = rig[k].mount_z;
        o.cpsi = (float)std::cos((double)rig[k].yaw); o.spsi = (float)std::sin((double)rig[k].yaw);
        o.cphi = (float)std::cos((double)rig[k].pitch); o.sphi = (float)std::sin((double)rig[k].pitch);
        o.fx = rig[k].fx; o.fy = rig[k].fy;
    }
    // (the status word is sticky across calls, like a scene's: pic_static_status reads and clears it)
    ce = pic::launch_setup(P, d->E * d->A, poses, nullptr, nullptr, dims, active, nullptr, agents, cams, status, 0.f, 1.f, 0.f, stream);
    if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "set-up kernels: %s", cudaGetErrorString(ce));
    ce = pic::launch_static_kernel(P, tri_xyz, tri_class, d->n_tris, g_sm_count[dev], stream);
    if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "render_static_kernel: %s", cudaGetErrorString(ce));
    return PIC_OK;
}

extern "C" pic_status pic_static_status(uint32_t* flags, void* cuda_stream) {
    if (!flags) return fail(PIC_ERR_INVALID_ARG, "flags is NULL");
    *flags = 0u;
    int dev = -1;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(ce));
    if (dev < 0 || dev >= kMaxDevices) return fail(PIC_ERR_INVALID_ARG, "device ordinal %d not supported", dev);
    unsigned char* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        scratch = g_scratch_ptr[dev];
    }
    if (!scratch) return PIC_OK;                  // pic_render_static has not run on this device
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    uint32_t* status = reinterpret_cast<uint32_t*>(scratch + kOffStatus);
    ce = cudaMemcpyAsync(flags, status, sizeof(uint32_t), cudaMemcpyDeviceToHost, stream);
    if (ce == cudaSuccess) ce = cudaMemsetAsync(status, 0, sizeof(uint32_t), stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(stream);
    if (ce != cudaSuccess) return fail(PIC_ERR_CUDA, "reading the status word: %s", cudaGetErrorString(ce));
    return PIC_OK;
}
