// 3D grids whose rows fit one warp, energy and residual fused or the energy alone, in all three diffusivity modes, with constant or
// nodal forcing, for rows of any length up to 257 nodes and any alignment.
//
// Arithmetic: an element layer between two node planes is two 2D problems and a mass-like one.  With u0, u1 on the planes below and
// above and w = u1 - u0, the field on the Gauss planes s = a, b of the layer is u0 + s w, so the x and y derivatives of a layer are
// those of two bilinear fields; each of them takes the march by edge forces of the 2D kernel (forces of the four edges of an
// element, elements that share an edge add up there first).  The z derivative is w itself, interpolated to the Gauss points
// of the (x, y) plane: rows of w are interpolated in x once for both element rows they belong to, then in y.  What the
// two planes get back, (f_a, f_b), goes to the node planes as f_a + f_b - F and F = a f_a + b f_b.  KL with m = 3: 88 FP32
// lane operations per element and 24 for the exponents, where derivatives at the 12 Gauss lines with their adjoint and the chain
// rule to 8 corners take 137 in all.  The two Gauss planes are the halves of packed f32x2 registers (the coefficient table of
// the KL exponents holds them as pairs already), the two Gauss columns those of the z part.
// The diffusion energy of the fused call is 1/2 sum_i u_i (K u)_i (Euler's identity).
//
// Layout of the work.  A work unit is one sample, one tile of Ry element rows (y) across the whole x extent, one
// chunk of Z element planes (z).  A unit belongs to LW = 4 .. 32 lanes of one warp (a lane owns NX = 4 consecutive nodes of a
// row, 8 on rows of more than 129); a warp with LW < 32 carries 32 / LW units that have nothing to do
// with one another.  No warp ever waits for another one.  A unit marches over its element planes from bottom to top, and inside
// a plane over its element rows.  The node rows stream through a ring of rows in shared memory that belongs to the unit alone:
// row (plane k, row j) of the tile is entry k T + j of a linear sequence (T node rows per plane), entry n lives in slot n mod C, and
// the ring holds the two planes being worked on plus D rows in flight (cp.async, one group per row).
// What a layer leaves for the plane above is parked, a row at a time, until the next layer reads it back: in the output array
// (aligned rows), else in shared memory (KL at the Gauss points, constant forcing) or a scratch array.
// Tiles and chunks do not overlap: the top node row of a tile leaves its sums in a scratch array (seam, [B][ntile-1][nz][nx]),
// the top plane of a chunk in another (zseam, [B][nchunk-1][ny][nx], plus [B][nchunk-1][ntile-1][nx] for the nodes on both
// kinds of seam), and a small kernel adds them to r afterwards.  Every element is computed exactly once.  No atomics; every sum has
// a fixed order.
//
// RG: rows that are not a multiple of the lanes' nodes, or pointers that are not 16-byte aligned: copied and stored word by word,
// elements beyond the grid carry the factor em = 0.  Of 2^k + 1 nodes the last, a Dirichlet node, takes no lane of its own: its
// residual is 0 and its share of the energy is added by the last lane.
#include "dn_internal.cuh"

#ifndef DN_L3_PART
#define DN_L3_PART 0
#endif

namespace dn {

struct L3Geo {
    int Ry, Z;            // element rows per tile, element planes per chunk
    int ntile, nchunk;
    int NX, LW, lwsh;     // nodes per lane, lanes per unit and log2 of it
    int C, RS;            // ring slots (rows) per unit, floats per slot
    int extra;            // RG: node nx-1 takes no lane
    long long units;
};
cudaError_t launch_layer3d_m12(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_layer3d_m34(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_layer3d_m56(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_layer3d_m78(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s);

namespace {

constexpr int L3_WARPS = 4;                       // warps per block (each warp is on its own)
constexpr int L3_D = 3;                           // rows in flight beyond the two planes in use

typedef unsigned long long u64;
struct f2 { u64 v; };                             // two floats
__device__ __forceinline__ f2 mk2(float lo, float hi) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ f2 dup2(float x) { return mk2(x, x); }
__device__ __forceinline__ void un2(const f2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v)); }
__device__ __forceinline__ float lo2(const f2 a) { float l, h; un2(a, l, h); return l; }
__device__ __forceinline__ float hi2(const f2 a) { float l, h; un2(a, l, h); return h; }
__device__ __forceinline__ f2 operator+(const f2 a, const f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator-(const f2 a, const f2 b) { f2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator*(const f2 a, const f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 fma2(const f2 a, const f2 b, const f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r; }
__device__ __forceinline__ f2 shfl_up2(unsigned mask, const f2 a, int width) {
    float l, h;
    un2(a, l, h);
    return mk2(__shfl_up_sync(mask, l, 1, width), __shfl_up_sync(mask, h, 1, width));
}

__device__ __forceinline__ float l3_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void l3_cp16(unsigned d, const float* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void l3_cp16_if(unsigned d, const float* gsrc, int pred) {      // predicated, no branch
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void l3_cp4_if(unsigned d, const float* gsrc, int pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void l3_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void l3_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Floats per Gauss row (q fixed) of an element row in the coefficient table: (plane s = a, s = b) pairs for
// i = 0..M, padded to a multiple of 4.
__host__ __device__ constexpr int l3_gs(int m) { return (2 * (m + 1) + 3) / 4 * 4; }

// Resident blocks per SM the kernel is compiled for.
__host__ __device__ constexpr int l3_minb(int nx, int mode, int m, bool nf, bool eo) { return nx == 8 ? 2 : eo ? 4 : 3; }

// MODE 0 (KG): KL at the Gauss points; 1 (KN): KL at the nodes, then Q1 interpolation; 2 (ND): stored nodal field.
// In the nodal modes a slot of the ring holds the nu row next to the u row: copied from the field (ND), or computed
// from the polynomial of that node line when the row is first used (KN: the table then holds one polynomial per node
// line, every coefficient twice, and travels with the row itself).
// NF: nodal forcing; the f row sits in the slot as well.  The load vector is the mass matrix applied to f, a smoothing along each
// axis: between the two planes first, then along x, then between the rows.
// EO: energy only; nothing is gathered, parked or stored.
// LWC: lanes per unit at compile time (32 or 16), or 0: taken from G.
template <int NX, int M, int MODE, bool NF, bool EO, int LWC, bool RG>
__global__ void __launch_bounds__(L3_WARPS * 32, l3_minb(NX, MODE, M, NF, EO))
layer3d_kernel(const Params P, const float* __restrict__ linepoly, const L3Geo G) {
    extern __shared__ __align__(16) float smem[];
    dep_wait();                                         // the tables of this call are complete
    dep_release();                                      // the fix-up kernel may move in as units finish
    constexpr bool KG = (MODE == 0), KN = (MODE == 1), ND = (MODE == 2);
    constexpr int GS = l3_gs(M);
    constexpr int CF = KG ? 2 * GS : KN ? GS : 0;       // coefficient floats per slot (KG: Gauss rows q = a, b of an element row)
    constexpr int CFQ = CF / 4;                         // ... in 16-byte pieces
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int LW = LWC ? LWC : G.LW, lwsh = (LWC == 32) ? 5 : (LWC == 16) ? 4 : G.lwsh, SUBS = 32 >> lwsh;
    const int sub = lane >> lwsh, lx = lane & (LW - 1);
    const unsigned submask = (LW == 32) ? 0xffffffffu : (((1u << LW) - 1u) << (sub * LW));
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x0 = NX * lx;
    const bool act = x0 < nx;                           // this lane holds nodes of the grid
    const int x0c = (RG || act) ? x0 : nx - NX;         // (aligned rows) lanes beyond the grid load valid memory and store nothing

    // ---- shared by the block: cos(pi x) at the two Gauss columns of each element of a lane, duplicated into both
    // halves of a pair, as float4 (ca, ca, cb, cb) at [element c][lane of the unit]
    float4* cps = reinterpret_cast<float4*>(smem);
    if constexpr (KG) {
        for (int i = threadIdx.x; i < NX * LW; i += L3_WARPS * 32) {
            const int xe = min(NX * (i & (LW - 1)) + (i >> lwsh), nx - 2);        // element index = index of its left node
            const float ca = __ldg(P.cg[0] + 2 * xe), cb = __ldg(P.cg[0] + 2 * xe + 1);
            cps[i] = make_float4(ca, ca, cb, cb);
        }
        __syncthreads();                                // the only block-wide barrier: before the march starts
    }
    const float4* cpl = cps + lx;
    f2 cnp[NX / 2];                                     // KN: cos(pi x) at this lane's nodes, in pairs
    if constexpr (KN) {
#pragma unroll
        for (int h = 0; h < NX / 2; ++h) cnp[h] = mk2(__ldg(P.cn[0] + min(x0 + 2 * h, nx - 1)), __ldg(P.cn[0] + min(x0 + 2 * h + 1, nx - 1)));
    }

    const long long su = ((long long)blockIdx.x * L3_WARPS + warp) * SUBS + sub;
    if (su >= G.units) return;                          // the other units of the warp synchronise among themselves only
    const int C = G.C, RS = G.RS;
    const unsigned RSB = (unsigned)RS * 4u, RINGB = (unsigned)C * RSB;
    constexpr bool SP = RG && KG && !NF && !EO;         // parked in shared memory
    const int PR = NX * LW;                             // floats of a row of the lanes' nodes
    const int per_unit = C * RS + (RG && !EO ? PR : 0) + (SP ? (G.Ry + 1) * PR : 0);
    float* ring = smem + (KG ? 4 * NX * LW : 0) + (size_t)(warp * SUBS + sub) * per_unit;
    float* obuf = ring + C * RS;                        // RG: one finished row on its way out
    float* park = SP ? obuf + PR : P.park + (size_t)su * ((G.Ry + 1) * PR);      // RG: sums of the upper plane, a row per node row
    const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
    const int UROW = NX * LW + 4;                       // floats of a node row in a slot (with the 4 floats of padding)
    const int FOFF = KG ? UROW : 2 * UROW;              // offset of the f row (nodal forcing)
    const int COEF = FOFF + (NF ? UROW : 0);            // offset of the coefficient row inside a slot
    const int H1 = 4 * LW + 4;                          // NX = 8: offset of the second 16 bytes of every lane

    int b, tile, chunk;
    row3d_unit(su, P.batch, (ny - 1) / G.Ry, (nz - 1) / G.Z, G.ntile, b, tile, chunk);
    const int y0 = tile * G.Ry, e1 = min(y0 + G.Ry, ny - 1);     // element rows y0 .. e1-1, node rows y0 .. e1
    const int T = e1 - y0 + 1;
    const bool lasttile = (e1 == ny - 1);               // then node row e1 = ny-1 is this tile's own, else the next tile's
    const int kbeg = chunk * G.Z, ke = min(kbeg + G.Z, nz - 1);
    const int nplanes = ke - kbeg + 1;                  // node planes kbeg .. ke
    const bool lastchunk = (ke == nz - 1);              // then node plane ke = nz-1 is this chunk's own, else the next chunk's

    const bool first_col = (x0 == 0), last_col = act && (x0 + NX == nx);
    const int kl = nx - 1 - x0;                         // RG: node kl of the lane is node nx-1
    const bool extra = RG && !NF && G.extra != 0;       // node nx-1 is the one right of the last lane's
    const float wX = (extra && lx == LW - 1) ? 1.f : 0.f;       // this lane adds its energy
    const size_t plane = (size_t)nx * ny;
    const int xo = RG ? lx : x0c;                       // where this lane's copies and stores of a row start
    float* rb = EO ? nullptr : P.r + (size_t)b * P.nodes + xo;
    float* sb = (EO || lasttile) ? nullptr : P.seam + (((size_t)b * (G.ntile - 1) + tile) * nz) * nx + xo;
    // where the sums of node plane ke go: r, or for a chunk below another the z seam (row y0 of it; and the entry of
    // this tile's seam row among the nodes that lie on both seams)
    float* ztop = EO ? nullptr : lastchunk ? rb + ((size_t)ke * ny + y0) * nx
                               : P.zseam + (((size_t)b * (G.nchunk - 1) + chunk) * ny + y0) * nx + xo;
    float* zstop = (EO || lasttile) ? nullptr
                 : lastchunk ? sb + (size_t)ke * nx
                             : P.zseam + (size_t)P.batch * (G.nchunk - 1) * ny * nx
                               + (((size_t)b * (G.nchunk - 1) + chunk) * (G.ntile - 1) + tile) * nx + xo;

    const bool impose = (P.flags & DN_IMPOSE_BC_ON_LOAD) != 0;
    const bool nomask = (P.flags & DN_NO_MASK) != 0;
    float bc0 = P.bc_x0, bc1 = P.bc_x1;
    if (impose) {
        if (P.bc0_b) bc0 = __ldg(P.bc0_b + b);
        if (P.bc1_b) bc1 = __ldg(P.bc1_b + b);
    }
    // Everything is kept in units of ku: y forces enter times rho, z forces times rz.
    const float W8 = 0.125f * P.hx * P.hy * P.hz;
    const float kx = W8 / (P.hx * P.hx), ky = W8 / (P.hy * P.hy), kz = W8 / (P.hz * P.hz);
    constexpr float UN = EO ? 1.f : KG ? 6.f : 3.f;     // the plane forces are kept times 6 (Gauss sums) or 3 (interpolated nu)
    const float rho = ky / kx, rz = UN * (kz / kx), ku = kx * (1.f / UN);
    const float gs = P.gJ ? __ldg(P.gJ + b) : 1.f;
    const float fw = NF ? 0.f : P.f_const * P.hx * P.hy * P.hz;    // nodal load of an interior node (constant forcing)
    const bool hasf = !NF && (P.f_const != 0.f);
    const float fsabs = P.hx * P.hy * P.hz * (1.f / 216.f);        // NF: scale of the mass matrix ...
    const float fs = fsabs / ku;                                    // ... in units of ku
    // Output scale, share of the nodal load and weight in the load energy of the lane's first / last node (Dirichlet
    // columns: masked, or with DN_NO_MASK carrying half a load); RG: the last column may be any node of a lane, stores look for it.
    const float sc = gs * ku;
    const float sc0 = (!RG && first_col && !nomask) ? 0.f : sc, scL = (!RG && last_col && !nomask) ? 0.f : sc;
    const float lw0 = (!RG && first_col) ? (nomask ? 0.5f : 0.f) : 1.f, lwL = (!RG && last_col) ? (nomask ? 0.5f : 0.f) : 1.f;
    const float wx0 = first_col ? 0.5f : 1.f, wxL = (!RG && last_col) ? 0.5f : 1.f;
    const float lm = (lx == 0) ? 0.f : 1.f;             // nothing arrives from the left in the first lane
    const f2 lm2 = dup2(lm), rho2 = dup2(rho);
    float em[NX];                                       // 0 for elements right of node nx-1
#pragma unroll
    for (int c = 0; c < NX; ++c) em[c] = RG ? (x0 + c < nx - 1 ? 1.f : 0.f) : (c == NX - 1 && (last_col || !act)) ? 0.f : 1.f;

    // ---- the ring.  Entry n = (plane index pk, row index pj) of the unit goes to slot n mod C: the node row and, for
    // pk, pj >= 1, the coefficients of element row (pk-1, pj-1).
    if constexpr (RG) {                                 // words beyond the grid stay zero
        for (int i = lx; i < C * RS / 4; i += LW) reinterpret_cast<float4*>(ring)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        for (int s = lx; s < C; s += LW) {              // the 4 floats right of the last lane's nodes
            float* pad = ring + (size_t)s * RS + 4 * LW;
            *reinterpret_cast<float4*>(pad) = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (!KG) *reinterpret_cast<float4*>(pad + UROW) = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (NF) *reinterpret_cast<float4*>(pad + FOFF) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __syncwarp(submask);
    int pf = 0, pfj = 0, pfk = 0;
    unsigned pfo = 0;                                   // byte offset of the slot the next entry goes to
    const size_t first = (size_t)b * P.nodes + (size_t)kbeg * plane + (size_t)y0 * nx + xo;
    const float* usrc = P.u + first;
    const float* nsrc = ND ? P.nu + first : nullptr;
    const float* fsrc = NF ? P.f + first : nullptr;
    // coefficient piece of this lane.  KG: of element row (pfk-1, pfj-1), so the pointer starts one row and one plane
    // low; KN: of the node line of the entry itself
    const float* csrc = KG ? linepoly + (((size_t)b * (nz - 1) + kbeg) * (ny - 1) + y0) * CF - ((size_t)(ny - 1) + 1) * CF + 4 * lx
                           : linepoly + (((size_t)b * nz + kbeg) * ny + y0) * CF + 4 * lx;
    const long long uwrap = (long long)plane - (long long)T * nx, cwrap = ((long long)(KG ? ny - 1 : ny) - T) * CF;
    const unsigned d0 = ring_s + 16u * lx, d1 = ring_s + 4u * H1 + 16u * lx, dc = ring_s + 4u * COEF + 16u * lx;
    unsigned dw[NX];                                    // RG: where this lane's words lx, lx + LW, ... of a row go, and whether they exist
    int wok[NX];
#pragma unroll
    for (int i = 0; i < NX; ++i) {
        const int w = lx + LW * i;
        dw[i] = ring_s + 4u * (NX == 8 ? ((w & 4) ? H1 : 0) + 4 * (w >> 3) + (w & 3) : w);
        wok[i] = (w < nx) ? 1 : 0;
    }
    const int xok = (extra && lx == 0) ? 1 : 0;
    auto copy_row = [&](const unsigned o, const float* src) {
        if constexpr (RG) {
#pragma unroll
            for (int i = 0; i < NX; ++i) l3_cp4_if(dw[i] + o, src + LW * i, wok[i]);
            l3_cp4_if(ring_s + 16u * LW + o, src + NX * LW, xok);
        } else {
            l3_cp16(d0 + o, src);
            if constexpr (NX == 8) l3_cp16(d1 + o, src + 4);
        }
    };
    auto issue = [&]() {
        if (pfk < nplanes) {                            // uniform in the unit
            copy_row(pfo, usrc);
            if constexpr (ND) copy_row(pfo + 4u * UROW, nsrc);
            if constexpr (NF) copy_row(pfo + 4u * FOFF, fsrc);
            if constexpr (CF > 0) {
                const bool cok = KN || (pfk >= 1 && pfj >= 1);
                l3_cp16_if(dc + pfo, csrc, (cok && lx < CFQ) ? 1 : 0);
                if constexpr (LWC == 0) {
#pragma unroll
                    for (int i = 4; i < CFQ; i += 4)    // (units of 4 or 8 lanes)
                        l3_cp16_if(dc + pfo + 16u * i, csrc + 4 * i, (cok && (i % LW == 0) && lx + i < CFQ) ? 1 : 0);
                }
            }
        }
        l3_commit();                                    // one group per entry, possibly empty
        ++pf; ++pfj; usrc += nx; csrc += CF;
        if constexpr (ND) nsrc += nx;
        if constexpr (NF) fsrc += nx;
        if (pfj == T) {
            pfj = 0; ++pfk; usrc += uwrap; csrc += cwrap;
            if constexpr (ND) nsrc += uwrap;
            if constexpr (NF) fsrc += uwrap;
        }
        pfo += RSB;
        if (pfo == RINGB) pfo = 0;
    };
    for (int i = 0; i < C; ++i) issue();

    auto ldrow = [&](const unsigned off, const int rowoff, float (&v)[NX + 1]) {
        const float* slot = reinterpret_cast<const float*>(reinterpret_cast<const char*>(ring) + off) + rowoff;
        const float4 q = *reinterpret_cast<const float4*>(slot + 4 * lx);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        if constexpr (NX == 8) {
            const float4 q1 = *reinterpret_cast<const float4*>(slot + H1 + 4 * lx);
            v[4] = q1.x; v[5] = q1.y; v[6] = q1.z; v[7] = q1.w;
        }
        v[NX] = slot[4 * (lx + 1)];                     // first node of the next lane, the node without a lane, or the zero pad
    };
    auto impose_on = [&](float (&v)[NX + 1]) {
        if (first_col) v[0] = bc0;
        if constexpr (RG) {
#pragma unroll
            for (int c = 0; c <= NX; ++c) if (c == kl) v[c] = bc1;
        } else {
            if (last_col) v[NX - 1] = bc1;
        }
    };
    // KN: nu at this lane's nodes of the row in a slot, from the polynomial that came with the row, into the slot
    auto nurow = [&](const unsigned off) {
        float* slot = reinterpret_cast<float*>(reinterpret_cast<char*>(ring) + off);
        f2 gg[GS / 2];
        const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(slot + COEF);
#pragma unroll
        for (int i = 0; i < GS / 4; ++i) { const ulonglong2 t = gp[i]; gg[2 * i].v = t.x; gg[2 * i + 1].v = t.y; }
        float nn[NX];
#pragma unroll
        for (int h = 0; h < NX / 2; ++h) {
            f2 e = gg[M];
#pragma unroll
            for (int i = M - 1; i >= 0; --i) e = fma2(e, cnp[h], gg[i]);
            nn[2 * h] = l3_ex2(lo2(e)); nn[2 * h + 1] = l3_ex2(hi2(e));
        }
        *reinterpret_cast<float4*>(slot + UROW + 4 * lx) = make_float4(nn[0], nn[1], nn[2], nn[3]);
        if constexpr (NX == 8) *reinterpret_cast<float4*>(slot + UROW + H1 + 4 * lx) = make_float4(nn[4], nn[5], nn[6], nn[7]);
        if (RG && extra && lx == LW - 1) {              // the node without a lane
            const float c = __ldg(P.cn[0] + nx - 1);
            float e = lo2(gg[M]);
#pragma unroll
            for (int i = M - 1; i >= 0; --i) e = fmaf(e, c, lo2(gg[i]));
            slot[UROW + 4 * LW] = l3_ex2(e);
        }
    };
    auto ld4 = [&](const float* p, float (&v)[NX]) {
#pragma unroll
        for (int h = 0; h < NX / 4; ++h) {
            const float4 q = *reinterpret_cast<const float4*>(p + 4 * h);
            v[4 * h] = q.x; v[4 * h + 1] = q.y; v[4 * h + 2] = q.z; v[4 * h + 3] = q.w;
        }
    };
    auto st4 = [&](float* p, const float (&v)[NX]) {
#pragma unroll
        for (int h = 0; h < NX / 4; ++h)
            *reinterpret_cast<float4*>(p + 4 * h) = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
    };
    // RG: which of the lane's words is a Dirichlet column (stored as zero)
    int iz = -1;
#pragma unroll
    for (int i = 0; i < NX; ++i) if (RG && !nomask && lx + LW * i == nx - 1) iz = i;
    const bool z0 = RG && !nomask && first_col;
    auto store_row = [&](float* dst, const float (&o)[NX]) {       // a finished row (or a seam's)
        if constexpr (RG) {
            __syncwarp(submask);                        // the row before it has left the buffer
            st4(obuf + x0, o);
            __syncwarp(submask);
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                float v = obuf[lx + LW * i];
                if (i == iz || (i == 0 && z0)) v = 0.f;
                if (wok[i]) dst[LW * i] = v;
            }
            if (xok) dst[NX * LW] = 0.f;
        } else if (act) {
            st4(dst, o);
        }
    };
    // the finished row: its scaled sums, masked, its nodal load added
    auto finish = [&](const float (&raw)[NX], const float nlrow, float (&o)[NX]) {
#pragma unroll
        for (int c = 0; c < NX; ++c) {
            const float s = (c == 0) ? sc0 : (c == NX - 1) ? scL : sc;
            const float l = (c == 0) ? lw0 * nlrow : (c == NX - 1) ? lwL * nlrow : nlrow;
            o[c] = fmaf(s, raw[c], l);
            if constexpr (RG) { if (nomask && (x0 + c == 0 || c == kl)) o[c] = fmaf(-0.5f, nlrow, o[c]); }
        }
    };
    auto load_sum = [&](const float (&v)[NX + 1]) {     // sum of a row of u with the weights of the load
        float a = wx0 * v[0];
#pragma unroll
        for (int c = 1; c < NX - 1; ++c) a += v[c];
        a = fmaf(wxL, v[NX - 1], a);
        if constexpr (RG) {
#pragma unroll
            for (int c = 0; c < NX; ++c) if (c == kl) a = fmaf(-0.5f, v[c], a);
            a = fmaf(0.5f * wX, v[NX], a);
        }
        return a;
    };
    auto wrapb = [&](unsigned o) { return o >= RINGB ? o - RINGB : o; };

    const f2 gab = mk2(DN_GA, DN_GB), ga2 = dup2(DN_GA), gb2 = dup2(DN_GB);
    // NF: weights of the smoothing along x (the nodes of the Dirichlet columns have one neighbour)
    const f2 mxl = dup2(first_col ? 0.f : 1.f), mxr = dup2((!RG && last_col) ? 0.f : 1.f);
    f2 mxc[NX];
#pragma unroll
    for (int c = 0; c < NX; ++c) mxc[c] = dup2(((c == 0 && first_col) || (RG ? c == kl : (c == NX - 1 && last_col))) ? 2.f : 4.f);

    double end = 0.0, eld = 0.0;
    unsigned oA = 0;                                    // slot (byte offset) of the lower plane's row at hand
    int n = 0;                                          // ... and its entry index
    const unsigned TB = (unsigned)T * RSB;

    for (int kk = 0; kk + 1 < nplanes; ++kk) {
        const int k = kbeg + kk;                        // element layer k lies between node planes k and k + 1: plane k is
        const bool hascarry = (kk > 0) && (RG || act);  // finished now, with the sums parked one layer before;
        const bool last = (k + 1 == ke);                // those of plane k + 1 are parked (plane ke: finished after the march)
        const float wzlo = (k == 0) ? 0.5f : 1.f;
        const float nllo = -gs * fw * wzlo;
        float enlo = 0.f, ello = 0.f, elnf = 0.f;
        f2 ex = dup2(0.f), ey = dup2(0.f), ez = dup2(0.f);      // EO
        float* rlo = EO ? nullptr : rb + ((size_t)k * ny + y0) * nx;
        float* rup = EO ? nullptr : last ? ztop : rlo + plane;
        float* prow = RG ? park + x0 : nullptr;         // RG: the parked row

        // ---- state of the node row below the element row at hand, on both Gauss planes (s = a, b) ...
        f2 uh[NX + 1], eh[NX], Fh[NX], Gv[NX + 1];      // field, its x differences, minus the pending x forces, pending y forces
        f2 Az[NX], Hz[NX];                              // ... for the z part at both Gauss columns: w interpolated in x, pending forces
        float u0[NX + 1], u1[NX + 1];                   // the field on the two node planes
        f2 nh[NX + 1], hnu[NX], Am[NX];                 // nodal modes: nu, its sums over x-neighbours; nu summed over the planes
        f2 sx[NX], Fs[NX];                              // NF: smoothed forcing, pending loads of (plane k, plane k + 1)
        // reads the row of plane k in slot oP and of plane k + 1 in slot oQ
        auto field = [&](const unsigned oP, const unsigned oQ, float (&c0)[NX + 1], float (&c1)[NX + 1], f2 (&uc)[NX + 1], f2 (&Ac)[NX]) {
            ldrow(oP, 0, c0); ldrow(oQ, 0, c1);
            if (impose) { impose_on(c0); impose_on(c1); }
            float w[NX + 1];
#pragma unroll
            for (int c = 0; c <= NX; ++c) {
                w[c] = c1[c] - c0[c];
                uc[c] = mk2(fmaf(DN_GA, w[c], c0[c]), fmaf(DN_GB, w[c], c0[c]));
            }
#pragma unroll
            for (int c = 0; c < NX; ++c) { const float d = w[c + 1] - w[c]; Ac[c] = mk2(fmaf(DN_GA, d, w[c]), fmaf(DN_GB, d, w[c])); }
        };
        auto nodal = [&](const unsigned oP, const unsigned oQ, f2 (&nc)[NX + 1], f2 (&Ac)[NX]) {
            float c0[NX + 1], c1[NX + 1], m[NX + 1];
            ldrow(oP, UROW, c0); ldrow(oQ, UROW, c1);
#pragma unroll
            for (int c = 0; c <= NX; ++c) {
                const float d = c1[c] - c0[c];
                nc[c] = mk2(fmaf(DN_GA, d, c0[c]), fmaf(DN_GB, d, c0[c]));
                m[c] = c0[c] + c1[c];
            }
#pragma unroll
            for (int c = 0; c < NX; ++c) { const float d = m[c + 1] - m[c]; Ac[c] = mk2(fmaf(DN_GA, d, m[c]), fmaf(DN_GB, d, m[c])); }
        };
        auto smooth = [&](const unsigned oP, const unsigned oQ, f2 (&s)[NX]) {
            float c0[NX + 1], c1[NX + 1];
            ldrow(oP, FOFF, c0); ldrow(oQ, FOFF, c1);
            f2 q[NX + 1];
#pragma unroll
            for (int c = 0; c <= NX; ++c) q[c] = mk2(fmaf(2.f, c0[c], c1[c]), fmaf(2.f, c1[c], c0[c]));
            const f2 ql = shfl_up2(submask, q[NX - 1], LW);       // lane 0: its own value, times mxl = 0
            s[0] = fma2(mxl, ql, fma2(mxc[0], q[0], q[1]));
#pragma unroll
            for (int c = 1; c < NX; ++c) s[c] = fma2(mxc[c], q[c], q[c - 1]) + (c == NX - 1 ? mxr * q[c + 1] : q[c + 1]);
        };

        l3_wait<0>();                                   // everything issued so far has landed ...
        __syncwarp(submask);                            // ... and is visible to the unit
        {
            const unsigned oC = wrapb(oA + TB);
            if constexpr (KN) {                         // a row is new when it is the upper plane's, and in the unit's first plane
                if (kk == 0) nurow(oA);
                nurow(oC);
                __syncwarp(submask);
            }
            field(oA, oC, u0, u1, uh, Az);
            if constexpr (!KG) nodal(oA, oC, nh, Am);
            if constexpr (NF) smooth(oA, oC, sx);
#pragma unroll
            for (int c = 0; c < NX; ++c) {
                eh[c] = uh[c + 1] - uh[c];
                Fh[c] = dup2(0.f); Gv[c] = dup2(0.f); Hz[c] = dup2(0.f);
                if constexpr (!KG) hnu[c] = nh[c] + nh[c + 1];
                if constexpr (NF) Fs[c] = dup2(0.f);
            }
            Gv[NX] = dup2(0.f);
        }

        for (int jj = 0; jj + 1 < T; ++jj) {
            if (jj > 0) { l3_wait<1>(); __syncwarp(submask); }    // all but the last row issued have landed; the rows retired are free
            float cin[NX];
            if constexpr (!EO) {
#pragma unroll
                for (int c = 0; c < NX; ++c) cin[c] = 0.f;
                if (hascarry) ld4(RG ? prow : rlo, cin);          // the sums parked for this row one layer ago
            }
            while (pf < n + C) issue();
            const unsigned oB = wrapb(oA + RSB), oD = wrapb(wrapb(oA + TB) + RSB);
            if constexpr (KN) {
                if (kk == 0) nurow(oB);
                nurow(oD);
                __syncwarp(submask);                    // the node right of a lane's last is the next lane's
            }
            float c0[NX + 1], c1[NX + 1];
            f2 uc[NX + 1], Ac[NX], nc[NX + 1], Mc[NX];
            field(oB, oD, c0, c1, uc, Ac);
            if constexpr (!KG) nodal(oB, oD, nc, Mc);
            f2 ga[GS / 2], gb[GS / 2];                  // Gauss row q = a / b; each entry holds (plane s = a, s = b)
            if constexpr (KG) {
                const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(ring) + oD) + COEF / 4;
#pragma unroll
                for (int i = 0; i < GS / 4; ++i) {
                    const ulonglong2 t0 = gp[i], t1 = gp[GS / 4 + i];
                    ga[2 * i].v = t0.x; ga[2 * i + 1].v = t0.y; gb[2 * i].v = t1.x; gb[2 * i + 1].v = t1.y;
                }
            }

            f2 raw[NX], Fp, gr, F0, g0, sk = uc[0] - uh[0], v0;
            float zw[NX], zr = 0.f;
            if constexpr (!KG) v0 = nh[0] + nc[0];
#pragma unroll
            for (int c = 0; c < NX; ++c) {
                const f2 e1 = uc[c + 1] - uc[c], s1 = uc[c + 1] - uh[c + 1], e0 = eh[c], t = e1 - e0;
                eh[c] = e1;
                const f2 dA = Ac[c] - Az[c], Da = fma2(ga2, dA, Az[c]), Db = fma2(gb2, dA, Az[c]);     // w at Gauss rows q = a, b
                Az[c] = Ac[c];
                f2 Px, nQx, Py, nQy, bt, Ma, Mb;        // (EO: sums of nu on the Gauss rows and columns); nu summed over the planes
                if constexpr (KG) {
                    const ulonglong2 cc = *reinterpret_cast<const ulonglong2*>(cpl + c * LW);
                    f2 ca, cb;
                    ca.v = cc.x; cb.v = cc.y;
                    f2 haa = ga[M], hab = gb[M], hba = ga[M], hbb = gb[M];           // h_{p q}
#pragma unroll
                    for (int i = M - 1; i >= 0; --i) {
                        haa = fma2(haa, ca, ga[i]); hab = fma2(hab, ca, gb[i]);
                        hba = fma2(hba, cb, ga[i]); hbb = fma2(hbb, cb, gb[i]);
                    }
                    const float paa = l3_ex2(lo2(haa)), qaa = l3_ex2(hi2(haa)), pab = l3_ex2(lo2(hab)), qab = l3_ex2(hi2(hab));
                    const float pba = l3_ex2(lo2(hba)), qba = l3_ex2(hi2(hba)), pbb = l3_ex2(lo2(hbb)), qbb = l3_ex2(hi2(hbb));
                    const f2 naa = mk2(paa, qaa), nab = mk2(pab, qab), nba = mk2(pba, qba), nbb = mk2(pbb, qbb);
                    Ma = mk2(paa + qaa, pba + qba); Mb = mk2(pab + qab, pbb + qbb);
                    const f2 Na = naa + nba, Nb = nab + nbb, Mp = naa + nab;
                    if constexpr (EO) {
                        Px = Na; nQx = Nb; Py = Mp; nQy = nba + nbb; bt = t;
                    } else {
                        const f2 S = Na + Nb, aS = dup2(6.f * DN_GA) * S;
                        Px = fma2(dup2(6.f * (DN_GB - DN_GA)), Na, aS); nQx = fma2(dup2(-6.f), S, Px);
                        Py = fma2(dup2(6.f * (DN_GB - DN_GA)), Mp, aS); nQy = fma2(dup2(-6.f), S, Py);
                        bt = S * t;
                    }
                } else {
                    // sums over corners: h0, h1 over the bottom and top edge, v0, v1 over the left and right one
                    const f2 h0 = hnu[c], h1 = nc[c] + nc[c + 1], v1 = nh[c + 1] + nc[c + 1];
                    hnu[c] = h1;
                    const f2 dM = Mc[c] - Am[c];
                    Ma = fma2(ga2, dM, Am[c]); Mb = fma2(gb2, dM, Am[c]);
                    Am[c] = Mc[c];
                    if constexpr (EO) {
                        const f2 dh = h1 - h0, dv = v1 - v0;
                        Px = fma2(ga2, dh, h0); nQx = fma2(gb2, dh, h0);
                        Py = fma2(ga2, dv, v0); nQy = fma2(gb2, dv, v0);
                        bt = t;
                    } else {
                        const f2 S = h0 + h1, nS = dup2(-1.f) * S;
                        Px = S + h0; nQx = nS - h1; Py = S + v0; nQy = nS - v1;
                        bt = (dup2(0.5f) * S) * t;
                    }
                    v0 = v1;
                }
                const bool masked = RG || c == NX - 1;
                if constexpr (EO) {
                    const f2 Dxa = fma2(ga2, t, e0), Dxb = fma2(gb2, t, e0), Dya = fma2(ga2, t, sk), Dyb = fma2(gb2, t, sk);
                    if (masked) {
                        const f2 m2 = dup2(em[c]);
                        ex = fma2(m2, fma2(Px * Dxa, Dxa, (nQx * Dxb) * Dxb), ex);
                        ey = fma2(m2, fma2(Py * Dya, Dya, (nQy * Dyb) * Dyb), ey);
                        ez = fma2(m2, fma2(Ma * Da, Da, (Mb * Db) * Db), ez);
                    } else {
                        ex = fma2(Px * Dxa, Dxa, ex); ex = fma2(nQx * Dxb, Dxb, ex);
                        ey = fma2(Py * Dya, Dya, ey); ey = fma2(nQy * Dyb, Dyb, ey);
                        ez = fma2(Ma * Da, Da, ez); ez = fma2(Mb * Db, Db, ez);
                    }
                } else {
                    // x and y on the two Gauss planes
                    const f2 Fx = fma2(Px, e0, bt) - Fh[c];               // the bottom edge is complete
                    Fh[c] = fma2(nQx, e1, bt);                            // minus what the top edge keeps for the element above
                    const f2 g = fma2(Py, sk, bt);
                    if (c == 0) {
                        F0 = Fx; g0 = g;
                    } else {
                        const f2 Gk = (masked ? dup2(em[c]) * g : g) - gr;
                        const f2 dxf = masked ? fma2(dup2(-em[c]), Fx, Fp) : Fp - Fx;
                        raw[c] = fma2(rho2, Gv[c] - Gk, dxf);
                        Gv[c] = Gk;
                    }
                    gr = fma2(nQy, s1, bt);                               // minus the force of the right edge
                    Fp = Fx;
                    // z: fluxes at the four Gauss columns, back to the two rows and then to the two nodes of this one
                    const f2 Ga = Ma * Da, Gb = Mb * Db, S = Ga + Gb, top = fma2(gb2, Gb, ga2 * Ga), H = Hz[c] + (S - top);
                    Hz[c] = top;
                    float ha, hb;
                    un2(H, ha, hb);
                    const float right = fmaf(DN_GB, hb, DN_GA * ha), left = (ha + hb) - right;
                    zw[c] = masked ? fmaf(em[c], left, zr) : zr + left;
                    zr = right;
                }
                sk = s1;
            }
            f2 sc_[NX];
            if constexpr (NF) smooth(oB, oD, sc_);
            const float wy = (y0 + jj == 0) ? 0.5f : 1.f;
            if constexpr (!EO) {
                // what the lane on the left adds to this lane's first node
                const f2 fl = shfl_up2(submask, Fp, LW), gl = shfl_up2(submask, gr, LW);
                zw[0] = fmaf(lm, __shfl_up_sync(submask, zr, 1, LW), zw[0]);
                const f2 m0 = dup2(em[0]);
                const f2 Gk = (RG ? m0 * g0 : g0) - lm2 * gl;
                raw[0] = fma2(rho2, Gv[0] - Gk, fma2(lm2, fl, RG ? dup2(-em[0]) * F0 : dup2(-1.f) * F0));
                Gv[0] = Gk;
                float lo[NX], up[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    float fa, fb;
                    un2(raw[c], fa, fb);
                    const float F = fmaf(DN_GB, fb, DN_GA * fa);
                    up[c] = fmaf(rz, zw[c], F);
                    lo[c] = (fa + fb) - up[c];          // F and the z force go to one plane, fa + fb less them to the other
                    if constexpr (NF) {
                        const f2 L = Fs[c] + fma2(dup2(2.f), sx[c], sc_[c]);
                        float l0, l1;
                        un2(L, l0, l1);
                        lo[c] = fmaf(-fs, l0, lo[c]); up[c] = fmaf(-fs, l1, up[c]);
                        elnf = fmaf(u0[c], l0, fmaf(u1[c], l1, elnf));
                    }
                    lo[c] += cin[c];
                    enlo = fmaf(u0[c], lo[c], enlo);
                }
                if constexpr (RG && !NF) {              // the node without a lane: its share of the energy, nothing parked
                    const f2 q = fma2(rho2, Gv[NX] + gr, Fp);
                    float fa, fb;
                    un2(q, fa, fb);
                    const float U = fmaf(rz, zr, fmaf(DN_GB, fb, DN_GA * fa));
                    enlo = fmaf(wX, fmaf(u0[NX], (fa + fb) - U, u1[NX] * U), enlo);
                    Gv[NX] = dup2(-1.f) * gr;
                }
                float o[NX];
                finish(lo, nllo * wy, o);
                if constexpr (RG) {
                    st4(prow, up);
                    store_row(rlo, o);
                    prow += PR;
                } else if (act) {
                    st4(rlo, o);
                    st4(rup, up);
                }
                rlo += nx; rup += nx;
            } else if constexpr (NF) {
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    const f2 L = Fs[c] + fma2(dup2(2.f), sx[c], sc_[c]);
                    elnf = fmaf(u0[c], lo2(L), fmaf(u1[c], hi2(L), elnf));
                }
            }
            if (hasf) ello = fmaf(wy, load_sum(u0), ello);
            if constexpr (NF) {
#pragma unroll
                for (int c = 0; c < NX; ++c) { Fs[c] = fma2(dup2(2.f), sc_[c], sx[c]); sx[c] = sc_[c]; }
            }
#pragma unroll
            for (int c = 0; c <= NX; ++c) { uh[c] = uc[c]; u0[c] = c0[c]; u1[c] = c1[c]; if constexpr (!KG) nh[c] = nc[c]; }
            oA = oB; ++n;
        }
        // ---- the top node row e1 of the tile gets nothing more in this layer.  It is this tile's own if it is the
        // top of the domain; else it belongs to the next tile and its sums go to the seam array (no load term: the
        // owner adds it).
        {
            const float wy = lasttile ? 0.5f : 0.f;
            if constexpr (!EO) {
                float* plo = lasttile ? rlo : sb + (size_t)k * nx;
                float* pup = lasttile ? rup : last ? zstop : plo + nx;
                float cin[NX], lo[NX], up[NX], o[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) cin[c] = 0.f;
                if (hascarry) ld4(RG ? prow : plo, cin);
                const f2 fl = shfl_up2(submask, Fh[NX - 1], LW);
                float zl = 0.f, zq[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    float ha, hb;
                    un2(Hz[c], ha, hb);
                    const float right = fmaf(DN_GB, hb, DN_GA * ha), left = (ha + hb) - right;
                    zq[c] = fmaf(em[c], left, zl);
                    zl = right;
                }
                zq[0] = fmaf(lm, __shfl_up_sync(submask, zl, 1, LW), zq[0]);
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    const f2 fprev = (c == 0) ? lm2 * fl : Fh[c - 1];
                    const f2 q = fma2(rho2, Gv[c], fma2(dup2(em[c]), Fh[c], dup2(-1.f) * fprev));
                    float fa, fb;
                    un2(q, fa, fb);
                    up[c] = fmaf(rz, zq[c], fmaf(DN_GB, fb, DN_GA * fa));
                    lo[c] = (fa + fb) - up[c];
                    if constexpr (NF) {
                        float l0, l1;
                        un2(Fs[c], l0, l1);
                        lo[c] = fmaf(-fs, l0, lo[c]); up[c] = fmaf(-fs, l1, up[c]);
                        elnf = fmaf(u0[c], l0, fmaf(u1[c], l1, elnf));
                    }
                    lo[c] += cin[c];
                    enlo = fmaf(u0[c], lo[c], enlo);
                }
                if constexpr (RG && !NF) {
                    const f2 q = fma2(rho2, Gv[NX], dup2(-1.f) * Fh[NX - 1]);
                    float fa, fb;
                    un2(q, fa, fb);
                    const float U = fmaf(rz, zl, fmaf(DN_GB, fb, DN_GA * fa));
                    enlo = fmaf(wX, fmaf(u0[NX], (fa + fb) - U, u1[NX] * U), enlo);
                }
                finish(lo, nllo * wy, o);
                if constexpr (RG) {
                    st4(prow, up);
                    store_row(plo, o);
                } else if (act) {
                    st4(plo, o);
                    st4(pup, up);
                }
            } else if constexpr (NF) {
#pragma unroll
                for (int c = 0; c < NX; ++c) elnf = fmaf(u0[c], lo2(Fs[c]), fmaf(u1[c], hi2(Fs[c]), elnf));
            }
            if (hasf && lasttile) ello = fmaf(wy, load_sum(u0), ello);
            oA = wrapb(oA + RSB); ++n;
        }
        if constexpr (EO) enlo = (lo2(ex) + hi2(ex)) + fmaf(rho, lo2(ey) + hi2(ey), rz * (lo2(ez) + hi2(ez)));
        end += (double)enlo; eld += NF ? (double)elnf : (double)(wzlo * ello);   // per-layer sums go to double
    }
    l3_wait<0>();
    __syncwarp(submask);

    // ---- node plane ke gets nothing more from this chunk: what was parked for it is complete as far as this chunk
    // goes.  Top of the domain: finished into r with its load.  Else the plane is the next chunk's: the scaled, masked
    // sums stay in the z seam (no load term: the owner adds it).  Its rows are still in the ring (entry n is row 0).
    if (!EO || (hasf && lastchunk)) {
        float entop = 0.f, eltop = 0.f;
        const float lf = lastchunk ? 1.f : 0.f;
        float* ptop = ztop;
        float* prow = RG ? park + x0 : nullptr;
        for (int jj = 0; jj < T; ++jj) {
            const bool seamrow = (jj == T - 1) && !lasttile;
            const int j = y0 + jj;
            const float wy = seamrow ? 0.f : (j == 0 || j == ny - 1) ? 0.5f * lf : lf;
            float uT[NX + 1];
            ldrow(oA, 0, uT);
            if (impose) impose_on(uT);
            if constexpr (!EO) {
                float* p = seamrow ? zstop : ptop;
                float part[NX], o[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) part[c] = 0.f;
                if (RG || act) ld4(RG ? prow : p, part);
#pragma unroll
                for (int c = 0; c < NX; ++c) entop = fmaf(uT[c], part[c], entop);
                finish(part, -gs * fw * 0.5f * wy, o);
                store_row(p, o);
                if constexpr (RG) prow += PR;
                ptop += nx;
            }
            eltop = fmaf(wy, load_sum(uT), eltop);
            oA = wrapb(oA + RSB);
        }
        end += (double)entop;
        if constexpr (!NF) eld += (double)(0.5f * eltop);
    }

    // ---- energy partial of this unit: its lanes summed in a fixed order in double
    // NF, fused: `end` holds sum u (K u - F) in units of ku and `eld` sum u F, so that the load part is fsabs * eld and the
    // diffusion part half of (ku * end + load part)
    double l = !act ? 0.0 : NF ? (double)fsabs * eld : hasf ? (double)fw * eld : 0.0;
    double d = !act ? 0.0 : NF && !EO ? 0.5 * ((double)ku * end + l) : 0.5 * (double)ku * end;
    for (int off = LW >> 1; off > 0; off >>= 1) {
        d += __shfl_down_sync(submask, d, off, LW);
        l += __shfl_down_sync(submask, l, off, LW);
    }
    if (lx == 0) {
        double* slot = P.partials + 2 * ((size_t)b * P.nblk + (size_t)chunk * G.ntile + tile);
        slot[0] = d; slot[1] = l;
    }
}

size_t l3_unit_floats(const L3Geo& g, int mode, bool nf, bool eo, bool rg) {
    const size_t row = (size_t)g.NX * g.LW;
    return (size_t)g.C * g.RS + (rg && !eo ? row : 0) + (rg && !eo && mode == 0 && !nf ? (g.Ry + 1) * row : 0);
}

template <int NX, int M, int MODE, bool NF, bool EO, int LWC, bool RG>
cudaError_t launch_l3(const Params& P, const float* linepoly, const L3Geo& g, cudaStream_t s) {
    const int subs = 32 / g.LW;
    const size_t smem = sizeof(float) * (L3_WARPS * subs * l3_unit_floats(g, MODE, NF, EO, RG) + (MODE == 0 ? 4 * NX * g.LW : 0));
    const long long per_block = (long long)L3_WARPS * subs;
    const unsigned blocks = (unsigned)((g.units + per_block - 1) / per_block);
    const cudaError_t e = allow_shared(layer3d_kernel<NX, M, MODE, NF, EO, LWC, RG>, smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(layer3d_kernel<NX, M, MODE, NF, EO, LWC, RG>, dim3(blocks), dim3(L3_WARPS * 32), smem, s, P, linepoly, g);
}

// The lane counts compiled in where they matter: constant forcing.
template <int M, int MODE, bool RG>
cudaError_t launch_l3_rows(const Params& P, const float* linepoly, const L3Geo& g, cudaStream_t s) {
    const bool eo = P.r == nullptr;
    if (g.NX == 8) {
        if (P.f) return eo ? launch_l3<8, M, MODE, true, true, 32, RG>(P, linepoly, g, s) : launch_l3<8, M, MODE, true, false, 32, RG>(P, linepoly, g, s);
        return eo ? launch_l3<8, M, MODE, false, true, 32, RG>(P, linepoly, g, s) : launch_l3<8, M, MODE, false, false, 32, RG>(P, linepoly, g, s);
    }
    if (P.f) return eo ? launch_l3<4, M, MODE, true, true, 0, RG>(P, linepoly, g, s) : launch_l3<4, M, MODE, true, false, 0, RG>(P, linepoly, g, s);
    if (eo) return launch_l3<4, M, MODE, false, true, 0, RG>(P, linepoly, g, s);
    if (g.LW == 32) return launch_l3<4, M, MODE, false, false, 32, RG>(P, linepoly, g, s);
    if (g.LW == 16) return launch_l3<4, M, MODE, false, false, 16, RG>(P, linepoly, g, s);
    return launch_l3<4, M, MODE, false, false, 0, RG>(P, linepoly, g, s);
}
template <int M, int MODE>
cudaError_t launch_l3_mode(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    return ragged ? launch_l3_rows<M, MODE, true>(P, linepoly, g, s) : launch_l3_rows<M, MODE, false>(P, linepoly, g, s);
}
template <int M>
cudaError_t launch_l3_m(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    return (P.nu_mode == DN_NU_KL_NODAL) ? launch_l3_mode<M, 1>(P, linepoly, g, ragged, s) : launch_l3_mode<M, 0>(P, linepoly, g, ragged, s);
}

}  // namespace

#if DN_L3_PART == 1
cudaError_t launch_layer3d_m34(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 3 ? launch_l3_m<3>(P, linepoly, g, ragged, s) : launch_l3_m<4>(P, linepoly, g, ragged, s);
}
#elif DN_L3_PART == 2
cudaError_t launch_layer3d_m56(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 5 ? launch_l3_m<5>(P, linepoly, g, ragged, s) : launch_l3_m<6>(P, linepoly, g, ragged, s);
}
#elif DN_L3_PART == 3
cudaError_t launch_layer3d_m78(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 7 ? launch_l3_m<7>(P, linepoly, g, ragged, s) : launch_l3_m<8>(P, linepoly, g, ragged, s);
}
#else
cudaError_t launch_layer3d_m12(const Params& P, const float* linepoly, const L3Geo& g, bool ragged, cudaStream_t s) {
    if (P.nu_mode == DN_NU_NODAL) return launch_l3_mode<1, 2>(P, linepoly, g, ragged, s);
    return P.m == 1 ? launch_l3_m<1>(P, linepoly, g, ragged, s) : launch_l3_m<2>(P, linepoly, g, ragged, s);
}
#endif

}  // namespace dn
