// Device/host data layout of the rasterizer library (internal).
#pragma once
#include <stddef.h>
#include <stdint.h>
#include <vector_types.h>

namespace pic {

constexpr int TILE = 64;        // a view is rendered in tiles of up to TILE x TILE pixels
constexpr int MAX_CAMS = 16;    // cameras per rig
constexpr int LEAF_PRIMS = 8;   // primitives per leaf (8 threads per leaf in the cull pass)
constexpr int LONG_LEAF_PRIMS = 8;   // long primitives get leaves of their own so the others' boxes stay tight
constexpr int GROUP_LEAVES = 32;     // leaves per group (one per lane)
constexpr int LARGE_LEAF_PRIMS = 4;  // primitives per leaf of the large-primitive list

// Map primitive in hierarchy order: a triangle, or a planar convex quad fused from two consecutive
// triangles of the input that share an edge (same class).  64 bytes, read as four 128-bit loads.
struct Prim {
    float v[12];        // 4 vertices xyz in perimeter order (triangle: the 4th repeats the 3rd)
    uint32_t key_lo;    // (0xFFFFFF - primitive index) << 8 | class : low half of the z-buffer key
    uint32_t flags;     // bit 0: quad; bits 4..7: edge i runs against its canonical direction
    float vis_cos;      // > 0: drawn only from its front side and within acos(vis_cos) of its normal (triangles only)
    uint32_t pad;
};
static_assert(sizeof(Prim) == 64, "Prim must be 64 bytes");

// Upright cylinder around a primitive of the grid order (same index), 16 bytes: what the cull kernel looks at first.
struct Bound {
    float x, y, z;      // centre
    uint32_t size;      // upper halves of two float32, rounded up: radius << 16 | half height
};
static_assert(sizeof(Bound) == 16, "Bound must be 16 bytes");

// Axis-aligned box of a leaf (over primitives) or a group (over leaves); 32 bytes.
struct Node {
    float lo[3];
    uint32_t first;
    float hi[3];
    uint32_t count;
};
static_assert(sizeof(Node) == 32, "Node must be 32 bytes");

struct MapInfo {
    uint32_t group_begin, group_end;   // range in the groups array
    uint32_t n_tris;                   // triangles of the map as given (box indices start here)
    uint32_t prim_begin;               // first primitive (used by the exhaustive kernel)
    uint32_t prim_end;
    // uniform grid over the map's ground-plane extent (the cull kernel's structure, see pic_bvh.cpp)
    uint32_t cell_begin;               // first entry of this map in the cell-start array (nx * ny + 1 entries)
    uint32_t nx, ny;                   // cells per row, rows
    float gx0, gy0;                    // corner of cell (0, 0)
    float cell, inv_cell;              // cell size, its reciprocal
    float margin;                      // no small primitive reaches farther than this from the centre of its box (xy)
    uint32_t large_begin, large_end;   // range in the large-primitive leaves
    uint32_t pad;
};
static_assert(sizeof(MapInfo) == 64, "MapInfo must be 64 bytes");

// Per-agent geometry written once per render by the set-up kernel; 32 bytes.
struct AgentGeom {
    float x, y;       // box centre on the ground plane
    float c, s;       // cos, sin of the heading
    float hl, hw, h;  // half length, half width, height
    uint32_t active;  // 0: inactive; else 1 | class of the agent's box << 8
};

struct CamConst {
    float mx, my, mz;
    float cpsi, spsi, cphi, sphi;   // cos/sin of the camera yaw and pitch (rounded from double)
    float fx, fy;
};

// Per-view camera written by the set-up kernel: ego position, mount and rotation rows; 64 bytes.
struct ViewCam {
    float px, py;              // ego position
    float mwx, mwy, mwz;       // mount in world axes
    float rx, ry;              // right   (rz = 0)
    float dx, dy, dz;          // down
    float fx, fy, fz;          // forward
    float pad[3];
};
static_assert(sizeof(ViewCam) == 64, "ViewCam must be 64 bytes");

// Per-camera tables shared by all views of a call: ray coordinates of pixel columns / rows, the background (analytic ground plane /
// sky) of every row, and the frusta of the tiles.
struct RigTables {
    const float4* frusta;      // [K][tiles + 1][FRUSTUM_ENTRIES] in camera space (see frustum_entry); the last of a camera's is the whole image's. NULL: not made
    const float* ray_x;        // [K][ray_stride(W)], [K][ray_stride(H)]: beyond the image the same formula goes on, so that a tile that
    const float* ray_y;        //   reaches over the edge reads a monotone table
    const float* bg_z;         // [K][H] background depth
    const uint32_t* bg_cls;    // [K][H] background class
    const uint32_t* bg_rgb;    // [K][H] background colour (calls that render colours)
};

// Division of numbers below 2^31 by a divisor fixed per call (Granlund and Montgomery, "Division by invariant integers
// using multiplication", PLDI 1994): q = (mulhi(n, m) + n) >> s.
struct FastDiv {
    uint32_t m, s;
};
inline FastDiv fast_div(uint32_t d) {
    FastDiv f = {0u, 0u};
    while ((1ull << f.s) < d) ++f.s;
    f.m = (uint32_t)(((1ull << 32) * ((1ull << f.s) - d)) / d + 1ull);
    return f;
}
#ifdef __CUDACC__
__host__ __device__ __forceinline__
#else
inline
#endif
unsigned divide(unsigned n, const FastDiv& f) {
#ifdef __CUDA_ARCH__
    return (__umulhi(n, f.m) + n) >> f.s;      // (written as below the tile kernel takes 0.7 % longer)
#else
    return ((unsigned)(((unsigned long long)n * f.m) >> 32) + n) >> f.s;
#endif
}

struct RenderParams {
    int32_t E, A, K, H, W;
    int32_t tiles_x, tiles_y;
    float near_z, far_z;
    float w_near, w_far;            // 1/near, 1/far: kept range of the reciprocal depth
    uint32_t cls_agent, cls_sky, cls_ground;
    FastDiv div_tiles, div_tiles_x, div_K, div_A;   // by tiles per view, tile columns, cameras, agent slots
    FastDiv div_views;              // by the views of this launch (tile kernel with the horizon first)
    const int32_t* env_map;
    const MapInfo* env_maps;        // [E] the MapInfo of each environment's map (one load instead of two)
    const MapInfo* maps;
    const Node* groups;
    const Node* leaves;
    const Prim* prims;
    const uint32_t* cell_start;     // grid: per map nx * ny + 1 offsets into grid_prims
    const Prim* grid_prims;         // the primitives in grid order: small ones cell by cell (row-major), then the large ones leaf by leaf
    const Bound* grid_bounds;       // bounding cylinder of each of grid_prims
    const Node* large_leaves;       // boxes over up to LARGE_LEAF_PRIMS consecutive large primitives of grid_prims
    const AgentGeom* agents;
    const ViewCam* cams;            // [E*A*K]
    RigTables rig;
    uint8_t* out_class;
    uint16_t* out_depth;
    float* out_depth32;             // optional
    unsigned long long* counters;   // optional [16]
    uint32_t* occlusion;            // optional [E*A*K][A][2]: per view and other agent, visible pixels and pixels its box covers alone
    uint8_t* out_rgb;               // colour output [E*A*K][H][W][3] (colour kernel only)
    const uint32_t* palette;        // [256] RGB of every class, R in the low byte (colour kernels only)
    uint32_t* status;               // the scene's sticky status word
    uint32_t* overflow;             // [1 + tiles of all views]: count, then the tiles left to the cooperative kernel
    uint2* surv;                    // per tile: the cull kernel's survivors (head + list), read by the render kernel
    int32_t debug_flags;            // bit 0: no per-cell trivial accept/reject, bit 1: record lists of 2 entries, bit 2: cooperative kernel only, bit 3: lists of 6
    int32_t tiles_per_cta;          // antialiased colour kernel: 4, or 1
    uint32_t n_jobs;                // tiles to render in this launch (views x tiles per view); set by the launcher
    long long view_first;           // render views [view_first, view_first + gridDim / tiles)
    CamConst cam[MAX_CAMS];
};

// Entries of a ray table for n columns or rows: TILE of them may be read from any that belongs to the image on.  (The tiles of most kernels
// begin at multiples of TILE, those of pic_render_static at multiples of 16 rows, and all read TILE entries.)
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int ray_stride(int n) { return (n + 2 * TILE - 1) / TILE * TILE; }

constexpr int FRUSTUM_ENTRIES = 11;      // six planes, five corners of the footprint
inline size_t frusta_bytes(int K, int H, int W) { return sizeof(float4) * FRUSTUM_ENTRIES * (size_t)K * ((size_t)((W + TILE - 1) / TILE) * (size_t)((H + TILE - 1) / TILE) + 1); }

// What thread t of block b of the set-up kernel does: the first blocks set up an agent per thread (the longest chain: 0.1 us of a small call),
// the next write an entry of a camera's ray and background tables (its columns, then its rows), the others an entry of a camera's frusta.  Entry i of
// the frusta belongs to frustum i / FRUSTUM_ENTRIES of the camera; what lies beyond the entries or the agents is left out by the kernel.
constexpr int SETUP_THREADS = 128;
enum SetupRole { SETUP_TABLES, SETUP_FRUSTA, SETUP_AGENTS };
struct SetupItem { SetupRole role; int camera, index; };
struct SetupGrid { int K, agent_blocks, table_blocks, frusta_blocks; FastDiv div_K; };       // (the cameras take turns, block by block)
inline int setup_parts(long long entries) { return (int)((entries + SETUP_THREADS - 1) / SETUP_THREADS); }
// tiles: of a view, or 0 if no frusta are wanted; n: agents
inline SetupGrid setup_grid(int K, FastDiv div_K, int H, int W, int tiles, int n) {
    return {K, setup_parts(n), K * setup_parts((long long)ray_stride(W) + ray_stride(H)), tiles ? K * setup_parts((tiles + 1LL) * FRUSTUM_ENTRIES) : 0, div_K};
}
#ifdef __CUDACC__
__host__ __device__
#endif
inline SetupItem setup_item(const SetupGrid& G, int b, int t) {
    if (b < G.agent_blocks) return {SETUP_AGENTS, 0, b * SETUP_THREADS + t};
    const int c = b - G.agent_blocks;
    const bool table = c < G.table_blocks;
    const int f = table ? c : c - G.table_blocks;
    const int part = (int)divide((unsigned)f, G.div_K);
    return {table ? SETUP_TABLES : SETUP_FRUSTA, f - part * G.K, part * SETUP_THREADS + t};
}
inline int setup_blocks(const SetupGrid& G) { return G.agent_blocks + G.table_blocks + G.frusta_blocks; }

// Does the tile kernel draw the tiles with the horizon of all views first, then the rows below, the sky last?  A small launch ends with
// whatever its last CTAs meet; a large one, or one whose tiles are all alike, rather keeps neighbouring tiles together, whose stores share
// lines.  So there has to be an order to make -- more than one row of tiles, or a narrower last column, which then comes last -- and few enough
// tiles.  Horizon first / in order, us, agents in platoons, so many tiles per multiprocessor (class and depth; colours; occlusion counts):
//   54 x 96 (2, one narrower)     61: 86 / 92;  95 / 103; 139 / 147    150: 153 / 157; 176 / 183; 254 / 259    259: 237 / 247; 276 / 288; 396 / 405
//   64 x 128 (2 alike)            61: 102 / 100; 118 / 116; 170 / 166   150: 180 / 178; 212 / 210; 303 / 301    259: 287 / 285; 342 / 338; 485 / 482
//   128 x 128 (4)                 59: 82 / 92;  99 / 114; 136 / 148    149: 148 / 157; 186 / 195; 248 / 264    259: 231 / 243; 299 / 307; 387 / 406
//   128 x 256 (8)                 62: 81 / 87; 101 / 106; 142 / 149    152: 128 / 138; 171 / 175; 216 / 226    263: 201 / 209; 269 / 269; 336 / 348
//   216 x 384 (24)                62: 71 / 74;  92 / 93;  110 / 108    150: 107 / 112; 133 / 144; 149 / 159    259: 160 / 159; 201 / 202; 218 / 220
// (At 350 tiles: 0.97 to 1.03 of the time in order.)  One line for all lies at 160; between there and 250 tiles the order in rows gives up to 6 % away.
constexpr int HORIZON_FIRST_TILES = 160;   // tiles per multiprocessor
inline bool draws_horizon_first(int H, int W, long long tiles, int sm_count) {
    return (H > TILE || (W > TILE && W % TILE != 0)) && tiles <= (long long)HORIZON_FIRST_TILES * sm_count;
}

// Layout of the per-camera tables: the frusta, then those of table_bytes bytes.
constexpr size_t table_bytes(int K, int H, int W) { return sizeof(float) * (size_t)K * ((size_t)ray_stride(W) + (size_t)ray_stride(H) + 3 * (size_t)H); }
inline RigTables rig_tables(float* base, int K, int H, int W, float4* frusta) {
    RigTables r;
    r.frusta = frusta;
    r.ray_x = base;
    r.ray_y = r.ray_x + (size_t)K * ray_stride(W);
    r.bg_z = r.ray_y + (size_t)K * ray_stride(H);
    r.bg_cls = reinterpret_cast<const uint32_t*>(r.bg_z + (size_t)K * H);
    r.bg_rgb = r.bg_cls + (size_t)K * H;
    return r;
}
inline void set_divisors(RenderParams& P) {
    P.div_tiles = fast_div((uint32_t)(P.tiles_x * P.tiles_y)); P.div_tiles_x = fast_div((uint32_t)P.tiles_x);
    P.div_K = fast_div((uint32_t)P.K); P.div_A = fast_div((uint32_t)P.A);
}

// Host-side result of the hierarchy build for all maps of a scene.
struct HostHierarchy;
HostHierarchy* build_hierarchy(int num_maps, const int64_t* tri_offset, const float* tri_xyz,
                               const uint8_t* tri_class, const float* tri_vis_cos, int agents_per_env, char* err, int err_len);
void free_hierarchy(HostHierarchy*);
const Prim* hierarchy_prims(const HostHierarchy*, size_t* n);
const Node* hierarchy_leaves(const HostHierarchy*, size_t* n);
const Node* hierarchy_groups(const HostHierarchy*, size_t* n);
const MapInfo* hierarchy_maps(const HostHierarchy*, size_t* n);
const uint32_t* hierarchy_cell_start(const HostHierarchy*, size_t* n);
const Prim* hierarchy_grid_prims(const HostHierarchy*, size_t* n);
const Bound* hierarchy_grid_bounds(const HostHierarchy*, size_t* n);
const Node* hierarchy_large_leaves(const HostHierarchy*, size_t* n);

}  // namespace pic
