// Internal declarations shared by the CUDA translation units of libdn.
#pragma once

#include <cstring>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "dn.h"

namespace dn {

// Gauss abscissae of the 2-point rule mapped to [0,1]: (1 -/+ 1/sqrt(3)) / 2.
#define DN_GA 0.21132486540518711775f
#define DN_GB 0.78867513459481288225f

constexpr int kAlign = 256;

inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

// SMs of the current device (148 where there is none); asked once per thread and device.
inline int sm_count() {
    thread_local int known_dev = -1, known = 0;
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return 148; }
    if (dev == known_dev) return known;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) { (void)cudaGetLastError(); return 148; }
    known_dev = dev; known = n;
    return n;
}

// A launch geometry (and the plan of a whole call) is a pure function of the problem's shape and mode and of the SM count of
// the current device.  The last few that a host thread searched for are remembered, so that a training loop pays the
// search once.
struct GeoKey { int v[12]; };
inline GeoKey geo_key(const dn_problem& p, int sms, int extra = 0) {
    return GeoKey{{p.grid.dim, p.grid.nx, p.grid.ny, (p.grid.dim == 3) ? p.grid.nz : 1, p.batch, (int)p.nu_mode,
                   (p.nu_mode == DN_NU_NODAL) ? 0 : p.kl_modes,     // not read with a stored field
                   p.f != nullptr ? 1 : 0, sms, (int)p.flags, extra, 1}};
}
template <class G, class F>
G memo_geometry(const dn_problem& p, int sms, F search, int extra = 0) {      // one memory per call site (F is its lambda)
    constexpr int kKept = 4;
    thread_local GeoKey key[kKept] = {};               // all zero: equal to no real key (the last entry of one is 1)
    thread_local G geo[kKept] = {};
    thread_local int next = 0;
    const GeoKey k = geo_key(p, sms, extra);
    for (int i = 0; i < kKept; ++i)
        if (memcmp(k.v, key[i].v, sizeof k.v) == 0) return geo[i];
    const int i = next;
    next = (next + 1) % kKept;
    geo[i] = search();
    key[i] = k;
    return geo[i];
}

enum Path { PATH_GENERIC = 0, PATH_TILED2D = 1, PATH_TILED3D = 2, PATH_STRIP2D = 3, PATH_PAIR3D = 4, PATH_ROW2D = 5,
            PATH_STRIP3D = 7,
            PATH_RAGGED2D = 6 };      // 2D rows of any length or alignment (dn_path_name counts them among the any-size ones)

// Where things live inside the caller's workspace (byte offsets, all 256-B aligned).
struct WsLayout {
    size_t partials;      // double [B][nblk][2]  (diffusion part, load part)
    size_t ckl;           // float  [B][m^dim]    KL weights * log2(e) / (1 + i^2 + j^2 (+ k^2))
    size_t cg[3];         // float  [m][gstride[a]] cos(i pi x) at the Gauss abscissae of axis a
    size_t seam;          // float  [B][nseam][nz][nx] contributions across tile seams (tiled 3D kernel)
    int gstride[3];       // padded row length of cg[a] (multiple of 4)
    size_t cn[3];         // float  [m][nstride[a]] cos(i pi x) at the nodes of axis a
    int nstride[3];
    size_t rowpoly;       // float  [B][ny-1][GS] polynomial of the KL exponent along every Gauss row (2D marching kernel)
    size_t zseam;         // float  contributions across the chunk seams of the mirrored-pair 3D kernel
    size_t park;          // float  partial sums the same kernel keeps outside shared memory
    size_t linepoly;      // float  [B][nz-1][ny-1][2 GS] the same along the four Gauss lines of every element row (mirrored-pair 3D kernel)
    int nblk;             // energy partials per sample
    size_t total;
};

// Everything a kernel needs, passed by value.
struct Params {
    int dim, nx, ny, nz, batch;
    int nu_mode, m;
    unsigned flags;
    float f_const, bc_x0, bc_x1;
    float hx, hy, hz;
    const float* u;
    const float* nu;
    const float* f;
    const float* gJ;
    const float* bc0_b;   // per-sample boundary values or NULL (then bc_x0 / bc_x1 hold for every sample)
    const float* bc1_b;
    float* r;             // may be NULL (energy only)
    double* partials;
    const float* ckl;
    const float* cg[3];
    int gstride[3];
    const float* cn[3];   // cosines at the nodes (KL-at-nodes mode)
    int nstride[3];
    int nblk;
    long long nodes;      // per sample
    float* seam;          // tiled 3D: contributions of a tile's top element row to the next tile's first node row
    int nseam;
    float* zseam;         // mirrored-pair 3D: contributions of a chunk's last element plane to the next chunk's first node plane
    float* park;          // mirrored-pair 3D: partial sums of the plane above (nodal modes, nodal forcing)
};

struct Launch {           // tiled-path launch geometry chosen on the host
    int path;
    int nblk;             // blocks (energy partials) per sample
    int chunk;            // rows (2D) or planes (3D) of elements per block
    int variant;          // kernel template variant
};

Launch choose_launch(const dn_problem& p, const float* u, const float* r);
WsLayout make_layout(const dn_problem& p, const Launch& l, bool tight = false);
// dn_energy_grad with the workspace sized for the chosen kernel family only (tight = true).
// What run_tight would answer for a scratch area of ws_bytes, without enqueuing anything or touching the device.
dn_status check_tight(const dn_problem* p, const float* u, const float* r, size_t ws_bytes);
dn_status run_tight(const dn_problem* p, const float* u, const float* gJ, float* J, float* r, void* ws,
                    size_t ws_bytes, void* stream);
// The fused kernel alone, for callers that apply the operator repeatedly: no energy finaliser; the KL tables are
// built only when build_tables is set (they depend on the problem, not on u); *partials / *nblk tell where the
// kernel left its per-block energy pairs (diffusion part, load part), [batch][*nblk][2] doubles.
dn_status run_operator(const dn_problem* p, const float* u, float* r, void* ws, size_t ws_bytes, cudaStream_t s,
                       bool build_tables, const double** partials, int* nblk);
// The parameters of a call that run_operator(p, u, r, ws, ...) made: where its tables are.
Params operator_params(const dn_problem& p, const float* u, float* r, void* ws);

// The solver with one thread-block cluster per sample (dn_multigrid.cu).  mg_blocks: blocks per cluster for `batch` samples at a
// time, 0 where the device can hold no cluster.  mg_solve: samples b0 .. b0 + nb - 1, whose K u - F stands in r; P: parameters of the
// call that left it there; mem: nb times mg_sample_bytes; u, r, relres and iters are the whole batch's.
bool mg_applicable(const dn_problem& p);
size_t mg_sample_bytes(const dn_problem& p);
int mg_blocks(const dn_problem& p, int batch);
cudaError_t mg_solve(const dn_problem& p, const Params& P, int blocks, int b0, int nb, float* mem, float* u, float* r, int max_iters, float rtol,
                     float* relres, int32_t* iters, cudaStream_t s);

// The KL tables alone, laid out as the kernel family chosen for (p, u, r) reads them.  For callers of run_operator
// that apply the operator to several problems sharing one diffusivity: build for the problem whose family needs
// the most (the cosine tables and scaled weights are common to all families).
dn_status build_tables(const dn_problem* p, const float* u, float* r, void* ws, size_t ws_bytes, cudaStream_t s);

// rowpoly (optional, 2D): also writes the per-Gauss-row polynomials the marching kernel reads, rows of rowpoly_stride floats
cudaError_t launch_tables(const Params& P, const float* kl_w, float* ckl, float* const cg[3], float* const cn[3],
                          cudaStream_t s, float* rowpoly = nullptr, int rowpoly_stride = 0,
                          bool rowpoly_nodes = false);   // rowpoly_nodes: one polynomial per node row (KL at the nodes)
cudaError_t launch_generic(const Params& P, cudaStream_t s);
cudaError_t launch_tiled2d(const Params& P, const Launch& l, cudaStream_t s);
cudaError_t launch_tiled3d(const Params& P, const Launch& l, cudaStream_t s);
cudaError_t launch_march2d(const Params& P, int path, const float* rowpoly, cudaStream_t s);
cudaError_t launch_finalize(const double* partials, int nblk, int batch, float* J, cudaStream_t s);
cudaError_t launch_kl_field(const dn_grid& g, int batch, int m, const float* kl_w, float* nu, cudaStream_t s);
cudaError_t launch_apply_bc(const dn_grid& g, int batch, float b0, float b1, int mode, float* field, cudaStream_t s,
                            const float* b0_b = nullptr, const float* b1_b = nullptr);

int generic_blocks_per_sample(long long nodes);
bool tiled2d_applicable(const dn_problem& p);
bool tiled3d_applicable(const dn_problem& p);
// The 2D marching kernel serves three paths: aligned rows that one unit covers (row2d), aligned rows cut into strips
// (strip2d), and rows of any length and alignment (ragged2d).
bool row2d_applicable(const dn_problem& p);
bool strip2d_applicable(const dn_problem& p);
bool march2d_chosen(const dn_problem& p, bool want_r);     // aligned rows: the marching kernel, or the tiled one
Launch march2d_geometry(const dn_problem& p, int path);
size_t march2d_rowpoly_floats(const dn_problem& p);
int march2d_rowpoly_stride(int kl_modes);          // floats per element row of that table
Launch tiled2d_geometry(const dn_problem& p);
Launch tiled3d_geometry(const dn_problem& p);
size_t tiled3d_seam_floats(const dn_problem& p);   // scratch floats the tiled 3D kernel needs for its tile seams
// adds seam[b][s][plane][x] to node row (s + 1) * rows_per_tile of r, for every sample, seam and plane
cudaError_t launch_seam_fixup(float* r, const float* seam, int nx, int ny, int nz, int rows_per_tile, int nseam, int batch,
                              cudaStream_t s);
// Cost of cutting the element rows and planes of a 3D grid into tiles of Ry and chunks of Z, for kernels that march a unit
// (tile, chunk) with one warp or a part of it, `slots` units at a time.  A unit pays, per plane, the finish of its top row,
// and once the filling of its ring and the finish of its last plane.  Full units run in whole waves; what is left over
// at the top of the tiles and chunks runs behind them in the slots that the last wave leaves idle, and what does not fit
// there after it.  Long units also end further apart; flat tiles and short chunks pay seam traffic.  Over 35 problems (24^3
// to 256^3, all diffusivities, with and without nodal forcing, energy alone and with the residual) the cut chosen is 0.9 %
// behind the best one on average, more than 3 % in three of them; counting whole waves of equal units, 1.8 % and in ten.
inline double row3d_cost(int Ry, int Z, int ny, int nz, int batch, long long slots) {
    auto unit = [](int ry, int z) { return z * (ry + 0.5) + 0.4 * ry + 2.0; };
    const int nt = (ny - 1) / Ry, rt = (ny - 1) % Ry, nc = (nz - 1) / Z, rc = (nz - 1) % Z;
    const long long full = (long long)batch * nt * nc, waves = (full + slots - 1) / slots, idle = waves * slots - full;
    const double c = unit(Ry, Z);
    double need = 0.0, late = 0.0, rest = 0.0;          // idle slots asked for, the longest of the small units, all of them
    auto small = [&](int n, int ry, int z) {
        const double d = unit(ry, z);
        need += (double)batch * n / (int)(c / d);
        rest += (double)batch * n * d;
        if (d > late) late = d;
    };
    if (rt) small(nc, rt, Z);
    if (rc) small(nt, Ry, rc);
    if (rt && rc) small(1, rt, rc);
    double span = waves * c;
    if (need > (double)idle) {
        const double after = (rest - idle * c) / slots;
        span += after > late ? after : late;
    }
    return (span + 0.05 * c) * (1.0 + 0.15 / Ry + 0.15 / Z);
}
bool strip3d_applicable(const dn_problem& p, bool want_r);     // aligned 3D rows the scalar kernels are faster for; they read the mirrored-pair kernel's table
Launch strip3d_geometry(const dn_problem& p, bool want_r);
size_t strip3d_seam_floats(const dn_problem& p);
size_t strip3d_zseam_floats(const dn_problem& p);
cudaError_t launch_strip3d(const Params& P, const float* linepoly, cudaStream_t s);
cudaError_t launch_strip3d_seams(const Params& P, float* J, cudaStream_t s);
// Adds the seams a 3D kernel left to r; J: and finishes the energies, in the same launch
cudaError_t launch_seam_fixup3(const Params& P, int Ry, int ntile, int Z, int nchunk, float* J, cudaStream_t s);
// Floats per line of fixed (y, z) in the coefficient table of the 3D kernels: pairs for the powers 0..m, padded to a multiple of 4.
__host__ __device__ constexpr int line_floats(int m) { return (2 * (m + 1) + 3) / 4 * 4; }
// Blocks that write it (LINE_THREADS element rows or node lines each).
constexpr int LINE_THREADS = 128;
inline long long lines3d_blocks(const dn_problem& p) {
    const int off = p.nu_mode == DN_NU_KL_NODAL ? 0 : 1;
    return (long long)p.batch * (p.grid.nz - off) * ((p.grid.ny - off + LINE_THREADS - 1) / LINE_THREADS);
}
// That table; all: and the tables of launch_tables, in the same launch
cudaError_t launch_lines3d(const Params& P, const float* kl_w, float* ckl, float* const cg[3], float* const cn[3], float* lines, bool all, cudaStream_t s);
bool pair3d_applicable(const dn_problem& p);       // 3D rows of at most 257 nodes, any alignment, every option
Launch pair3d_geometry(const dn_problem& p, bool want_r);
size_t pair3d_seam_floats(const dn_problem& p);
size_t pair3d_zseam_floats(const dn_problem& p);
size_t pair3d_park_floats(const dn_problem& p);
size_t pair3d_linepoly_floats(const dn_problem& p);
cudaError_t launch_pair3d(const Params& P, const float* linepoly, cudaStream_t s);
cudaError_t launch_pair3d_seams(const Params& P, float* J, cudaStream_t s);

// Streams and events of one *_host call (created and destroyed inside the call).
struct HostPipe {
    static constexpr int kMaxChunks = 32;
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t start = nullptr, copied[kMaxChunks] = {}, computed[kMaxChunks] = {};
    bool create(int nchunks) {
        if (cudaStreamCreateWithFlags(&in, cudaStreamNonBlocking) != cudaSuccess) return false;
        if (cudaStreamCreateWithFlags(&out, cudaStreamNonBlocking) != cudaSuccess) return false;
        if (cudaEventCreateWithFlags(&start, cudaEventDisableTiming) != cudaSuccess) return false;
        for (int c = 0; c < nchunks; ++c) {
            if (cudaEventCreateWithFlags(&copied[c], cudaEventDisableTiming) != cudaSuccess) return false;
            if (cudaEventCreateWithFlags(&computed[c], cudaEventDisableTiming) != cudaSuccess) return false;
        }
        return true;
    }
    ~HostPipe() {
        for (int c = 0; c < kMaxChunks; ++c) {
            if (copied[c]) cudaEventDestroy(copied[c]);
            if (computed[c]) cudaEventDestroy(computed[c]);
        }
        if (start) cudaEventDestroy(start);
        if (in) cudaStreamDestroy(in);
        if (out) cudaStreamDestroy(out);
    }
};

// Shared memory above the 48 KiB that a kernel may use without asking.  What is allowed is a constant, not what this launch
// needs: a host thread that launches the same kernel for a smaller problem must not take it away from another one between
// its asking and its launch.  reserve: the kernel's static shared memory, at least.
constexpr size_t kMaxBlockShared = 232448;
template <class K>
cudaError_t allow_shared(K kernel, size_t bytes, size_t reserve = 0) {
    return bytes <= 48 * 1024 ? cudaSuccess
                              : cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxBlockShared - reserve));
}

// Launch of a kernel that may start before the kernel ahead of it in the stream has finished (programmatic
// dependent launch): its blocks become resident as the blocks of that kernel retire, and it must not touch anything
// that kernel writes, nor write anything it reads, before dep_wait() has returned.  Hides the launch latency and the
// tail of the kernel ahead.
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

#ifdef __CUDACC__
// dep_wait(): everything the kernels ahead in the stream wrote is complete and visible (a no-op in a kernel that was
// launched the ordinary way).  dep_release(): kernels launched behind this one with launch_dependent may become
// resident from now on (they still wait in dep_wait() for this kernel to finish).
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Work unit su of a 3D march: the full (tile, chunk) pairs first (nt x nc of them per sample), so that the slots the last of
// them leave idle are filled with the smaller units at the top of the tiles and chunks.
__device__ __forceinline__ void row3d_unit(long long su, int batch, int nt, int nc, int ntile, int& b, int& tile, int& chunk) {
    const long long full = (long long)batch * nt * nc;
    const long long i = su < full ? su : su - full;
    const int q = (int)(i / batch);
    b = (int)(i - (long long)q * batch);
    if (su < full) { chunk = q / nt; tile = q - chunk * nt; }
    else if (ntile > nt && q < nc) { chunk = q; tile = nt; }            // the short tile of a full chunk
    else { chunk = nc; tile = q - (ntile > nt ? nc : 0); }              // the short chunk
}

// Sum (d, l) over the block in a fixed order and let thread 0 store the pair.
// Every thread of the block must call this.  blockDim.x * blockDim.y <= 1024.
__device__ __forceinline__ void block_reduce_store(double d, double l, double* slot) {
    __shared__ double sd[32], sl[32];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int nthreads = blockDim.x * blockDim.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d += __shfl_down_sync(0xffffffffu, d, o);
        l += __shfl_down_sync(0xffffffffu, l, o);
    }
    if ((tid & 31) == 0) { sd[tid >> 5] = d; sl[tid >> 5] = l; }
    __syncthreads();
    if (tid == 0) {
        const int nw = (nthreads + 31) >> 5;
        double a = 0.0, b = 0.0;
        for (int w = 0; w < nw; ++w) { a += sd[w]; b += sl[w]; }
        slot[0] = a; slot[1] = b;
    }
}
#endif

}  // namespace dn
