// Marching kernel for 2D grids: energy and residual fused, in all three diffusivity modes (KL evaluated in the kernel at
// the Gauss points, KL evaluated at the nodes and then interpolated, a stored nodal field), with constant or nodal
// forcing, and its energy-only variant.
//
// Layout of the work.  A work unit is one sample, one chunk of R node rows and one strip of LW * NX node columns; it
// belongs to LW = 8, 16 or 32 lanes of one warp (a lane owns NX = 4 or 8 consecutive nodes); a warp with LW < 32
// carries 32 / LW units that have nothing to do with one another.  Rows that fit a unit are one strip and nothing
// overlaps in x.  Wider rows are cut into strips that overlap by one lane: lane 0 of every strip but the first
// recomputes the NX elements left of the strip only to hand the forces of the last of them to lane 1, and stores
// nothing.  So no warp ever waits for another one: no block-wide barrier, no exchange between units.  A unit marches
// over its element rows from bottom to top.  The node row below lives in registers (values, differences along x,
// pending edge forces); the row above, the node right of the strip and the polynomial of the KL exponent on that element
// row (prepared once per call by the table kernel) arrive through a ring of DEPTH slots in shared memory that belongs to
// the unit alone, filled with cp.async several rows ahead.  The node right of a lane's last one is read from the ring
// (the next lane's first node, the node right of the strip, or a zero pad).  The first element row of a chunk is
// recomputed by the chunk below (1 / R).  No atomics.
//
// Arithmetic of one element, by edges.  With the differences e0, e1 along the bottom and top edge, s0, s1 along the left
// and right edge and t = e1 - e0 = s1 - s0, the forces of the four edges (derivatives of the element energy by the edge
// differences) are
//     bottom  P e0 + B t,   top  Q e1 - B t,   left  P' s0 + B t,   right  Q' s1 - B t      (x in units of kx, y of ky)
// where, for sums N_a, N_b of nu along x on the two Gauss rows and M_a, M_b along y on the two Gauss columns,
//     P = b N_a + a N_b,  Q = a N_a + b N_b,  P' = b M_a + a M_b,  Q' = a M_a + b M_b,  B = (N_a + N_b) / 6,
// a, b = (1 -/+ 1/sqrt 3) / 2 (a + b = 1, a b = 1/6).  N_a + N_b = M_a + M_b = S, so Q = S - P and B serve both axes.
// The two elements that share an edge add up on the edge first, and a node is the difference of its two edges along
// each axis: 10 FP32 operations per element fewer than the derivatives at the Gauss lines, their adjoint and the chain
// rule to four corners (47 instead of 58 with m = 6).  Everything is kept times 6 (Gauss sums) or 3 (interpolated nu),
// which the output scale takes back.  The diffusion energy is 1/2 sum_i u_i (K u)_i (Euler's identity).
//
// KL diffusivity: for a fixed Gauss row (or, KN, node row) the exponent is a polynomial of degree m in c = cos(pi x),
// its two Gauss rows interleaved so that they are evaluated together with packed two-wide FMAs.
//
// RG: rows of any length and pointers of any alignment.  A row is copied word by word (lane l takes the words l, l + LW,
// ... of the strip, so the copies are coalesced for every offset), elements beyond the grid carry the factor em = 0, and
// finished rows pass through one row of shared memory so that the stores are coalesced words as well.  Where exactly one
// node is left over (2^k + 1 nodes: the Dirichlet column x = 1) it takes no lane of its own: it is the node right of the
// strip, its residual is 0 and its share of the energy is added by the last lane.
//
// What bounds it: issue slots and the FP32 pipe in the KL modes (2048^2 x 16, m = 6: 65 instructions and 53 FP32 lane operations
// per element, an instruction issued in 71 % of the cycles, FMA pipe busy 61 %), HBM with a stored field (85 % of the copy
// bandwidth).  Measured against the two kernels it replaces (differences at the Gauss lines, one kernel for rows up to 256
// nodes, one for wide rows):
// 2048^2 x 16 188.2 -> 180.9 us (KL, m = 6), 156 -> 142 us (KL at the nodes); against the any-size kernel, which served
// rows that are not a multiple of 4: 513^2 x 64 2786 -> 68 us.
//
// The file is compiled in four parts side by side (m = 1, 2 and the stored field; 3, 4; 5, 6; 7, 8).
#include "dn_internal.cuh"

#ifndef DN_M2_PART
#define DN_M2_PART 0
#endif

namespace dn {

struct M2Geo {
    int R, nchunk, nstrip;
    int span;             // rows that pass one after the other, over all waves of units
    int NX, LW, lwsh;     // nodes per lane, lanes per unit and log2 of it
    int RS;               // floats per ring slot
    int extra;            // RG: node nx-1 is the node right of the strip
    int blocks;           // resident blocks per SM
    long long units;
};
cudaError_t launch_march2d_m12(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_march2d_m34(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_march2d_m56(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s);
cudaError_t launch_march2d_m78(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s);

namespace {

constexpr int M2_WARPS = 4;                       // warps per block (each warp is on its own)
constexpr int M2_DEPTH = 8;                       // ring slots per unit (DEPTH - 1 rows in flight)
constexpr size_t kM2ThirdOfSm = 70000;            // shared memory of a block of which an SM holds three, not four
__host__ __device__ constexpr int m2_minb(int nx) { return nx == 8 ? 3 : 4; }    // resident blocks per SM: 168 or 128 registers

typedef unsigned long long u64;

__device__ __forceinline__ float m2_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void m2_unpack(u64 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ u64 m2_pack(float lo, float hi) {
    u64 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ u64 m2_fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ void m2_cp16(unsigned d, const float* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void m2_cp16_if(unsigned d, const float* gsrc, int pred) {    // predicated, no branch
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void m2_cp4_if(unsigned d, const float* gsrc, int pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void m2_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void m2_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Floats per row of the coefficient table: pairs for k = 0..M, padded to a multiple of 4.
__host__ __device__ constexpr int m2_gs(int m) { return (2 * (m + 1) + 3) / 4 * 4; }

// MODE 0: KL at the Gauss points; 1 (KN): KL at the nodes, then Q1 interpolation; 2 (ND): stored nodal field
// NF: nodal forcing.  The f row rides in the ring next to the u row; the load vector is the consistent mass matrix
// applied to f, a 3 x 3 stencil that separates into a smoothing along x (neighbours by shuffle) and one along y (the row
// below carried, the row above arriving), with the one-sided weights on the boundary nodes.
// EO: energy only.  The same march, but every element adds its own energy and nothing is gathered or stored.
// LWC: lanes per unit at compile time (32 or 16), or 0: taken from G
template <int NX, int M, int MODE, bool NF, bool EO, int LWC, bool RG>
__global__ void __launch_bounds__(M2_WARPS * 32, m2_minb(NX))
march2d_kernel(const Params P, const float* __restrict__ rowpoly, const M2Geo G) {
    extern __shared__ __align__(16) float smem[];
    dep_wait();                                         // the tables of this call are complete
    dep_release();                                      // the finaliser may move in behind the last units
    static_assert(NX == 4 || (NX == 8 && !RG && !NF), "layouts in use");
    constexpr bool KG = (MODE == 0), KN = (MODE == 1), ND = (MODE == 2);
    constexpr int GS = m2_gs(M);
    constexpr int CFQ = ND ? 0 : GS / 4;                // 16-byte pieces of a coefficient row
    constexpr bool CREG = (NX == 4);                    // KG: cosines in registers, else in a table of the unit
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int LW = LWC ? LWC : G.LW, lwsh = (LWC == 32) ? 5 : (LWC == 16) ? 4 : G.lwsh, SUBS = 32 >> lwsh;
    const int sub = lane >> lwsh, lx = lane & (LW - 1);
    const unsigned submask = (LW == 32) ? 0xffffffffu : (((1u << LW) - 1u) << (sub * LW));
    // KG, 8 nodes per lane (one strip): the cosines of a lane's elements in a table that the block shares, (ca, ca, cb, cb) at
    // [element k][lane].  A unit of 10 rows cannot hide 16 scattered loads per lane of its own (a call on 256 x 64 x 64,
    // m = 1: 11.8 -> 11.4 us, 256^2 x 64 19.6 -> 19.1)
    float4* cps = reinterpret_cast<float4*>(smem);
    if constexpr (KG && !CREG) {
        for (int i = threadIdx.x; i < NX * LW; i += M2_WARPS * 32) {
            const int xe = min(NX * (i & (LW - 1)) + (i >> lwsh), P.nx - 2);      // element index = index of its left node
            const float ca = __ldg(P.cg[0] + 2 * xe), cb = __ldg(P.cg[0] + 2 * xe + 1);
            cps[i] = make_float4(ca, ca, cb, cb);
        }
        __syncthreads();                                // the only block-wide barrier: before the march starts
    }
    const unsigned su = (blockIdx.x * M2_WARPS + warp) * SUBS + sub;      // fewer than 2^32 units of at least 4 nodes fit a GPU
    if (su >= G.units) return;                          // the other units of the warp synchronise among themselves only
    const unsigned nstrip = G.nstrip, sq = su / nstrip;
    const int strip = (int)(su - sq * nstrip);
    const int chunk = (int)(sq / (unsigned)P.batch), b = (int)(sq - (unsigned)chunk * (unsigned)P.batch);

    const int nx = P.nx, ny = P.ny;
    const int xs = strip * (LW - 1) * NX;               // first column of the strip
    const int x0 = xs + NX * lx;
    const bool act = x0 < nx;                           // this lane holds nodes of the grid
    const int x0c = act ? x0 : nx - NX;                 // (aligned rows) lanes beyond the grid load valid memory and store nothing
    const bool owner = act && (lx > 0 || strip == 0);   // lane 0 of a later strip only feeds lane 1
    const bool has_first = (x0 == 0);                   // node 0 is this lane's first node
    const bool has_last = act && (x0 + NX == nx);       // node nx-1 is this lane's last node
    const bool has_halo = (xs + NX * LW < nx);          // the node right of the strip exists
    const bool extra = RG && !NF && G.extra != 0;
    const int n0 = chunk * G.R, n1 = min(n0 + G.R, ny);
    const int jbeg = max(n0 - 1, 0);
    const int jend = min(n1 - 1, ny - 2);               // last element row of this unit (inclusive)

    // ---- shared memory of this unit: the ring, (RG) one row on its way out
    const int RS = G.RS;
    const int per_unit = M2_DEPTH * RS + (RG ? NX * LW : 0);
    float* ring = smem + ((KG && !CREG) ? 4 * NX * LW : 0) + (size_t)(warp * SUBS + sub) * per_unit;
    float* obuf = ring + M2_DEPTH * RS;
    const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
    const int UROW = NX * LW + 4;                       // floats of a node row in a slot (with the pad / the node right of the strip)
    const int FOFF = ND ? 2 * UROW : UROW;              // NF: where the f row starts inside a slot (ND: behind the nu row at UROW)
    const int COEF = FOFF + (NF ? UROW : 0);            // the coefficient row
    const int H1 = 4 * LW + 4;                          // NX = 8: offset of the second 16 bytes of every lane

    const float* ub = P.u + (size_t)b * P.nodes;
    float* rb = EO ? nullptr : P.r + (size_t)b * P.nodes;
    const bool impose = (P.flags & DN_IMPOSE_BC_ON_LOAD) != 0;
    const bool nomask = (P.flags & DN_NO_MASK) != 0;
    float bc0 = P.bc_x0, bc1 = P.bc_x1;
    if (impose) {
        if (P.bc0_b) bc0 = __ldg(P.bc0_b + b);
        if (P.bc1_b) bc1 = __ldg(P.bc1_b + b);
    }
    const float kx = 0.25f * P.hy / P.hx, ky = 0.25f * P.hx / P.hy;
    const float rho = ky / kx;                          // the march works in units of ku; y forces enter times rho
    const float ku = EO ? kx : kx * (KG ? 1.f / 6.f : 1.f / 3.f);
    const float fw = NF ? 0.f : P.f_const * P.hx * P.hy;   // nodal load of an interior node (constant forcing)
    const bool hasf = !NF && (P.f_const != 0.f);
    const float gs = P.gJ ? __ldg(P.gJ + b) : 1.f;

    // Lane constants that make the march branch-free:
    //  lm        0 in lane 0 (nothing arrives from the left), else 1
    //  em        0 for elements right of node nx-1 (they do not exist), else 1: on aligned rows only the last of a lane can be
    //  gsf/gsl, nlf/nll   output scale and nodal load of the lane's first / last node (Dirichlet columns: masked to zero,
    //            or with DN_NO_MASK carrying half the nodal load); wf/wl their weights in the load energy.  With RG the
    //            last column may be any node of a lane: stores and load weights look for it
    const float lm = (lx == 0) ? 0.f : 1.f;
    float em[NX];
#pragma unroll
    for (int k = 0; k < NX; ++k) em[k] = RG ? ((x0 + k < nx - 1) ? 1.f : 0.f) : (k == NX - 1 && has_last) ? 0.f : 1.f;
    const float nl = -gs * fw;
    const float gku = gs * ku;
    const float gm0 = (!RG && has_first && !nomask) ? 0.f : 1.f, gmL = (!RG && has_last && !nomask) ? 0.f : 1.f;
    const float gsf = gku * gm0, gsl = gku * gmL;
    const float nlf = (!RG && has_first) ? (nomask ? 0.5f * nl : 0.f) : nl, nll = (!RG && has_last) ? (nomask ? 0.5f * nl : 0.f) : nl;
    const float wf = has_first ? 0.5f : 1.f, wl = (!RG && has_last) ? 0.5f : 1.f;
    const float wX = (extra && lx == LW - 1) ? 1.f : 0.f;        // this lane adds the energy of the left-over node
    const int kl = RG ? nx - 1 - x0 : -1;               // RG: node kl of the lane is node nx-1 (0 .. NX: it or the one right of it)

    // cos(pi x) at the two Gauss columns of each element, duplicated into both halves of a pair
    u64 cda[CREG ? NX : 1], cdb[CREG ? NX : 1];
    const float4* cpl = cps + lx;
    u64 cnp[NX / 2];                                    // KN: cos(pi x) at this lane's nodes (pairs) and at the node right of them
    float cnh = 0.f;
    if constexpr (KG && CREG) {
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const int xe = min(x0 + k, nx - 2);         // element index = index of its left node
            const float ca = __ldg(P.cg[0] + 2 * xe), cb = __ldg(P.cg[0] + 2 * xe + 1);
            cda[k] = m2_pack(ca, ca); cdb[k] = m2_pack(cb, cb);
        }
    }
    if constexpr (KN) {
        float cn[NX + 1];
#pragma unroll
        for (int k = 0; k <= NX; ++k) cn[k] = __ldg(P.cn[0] + min(x0 + k, nx - 1));
#pragma unroll
        for (int h = 0; h < NX / 2; ++h) cnp[h] = m2_pack(cn[2 * h], cn[2 * h + 1]);
        cnh = cn[NX];
    }

    // ---- the ring: step i = j - jbeg uses slot i % DEPTH, which holds node row j + 1 of u (and nu, f), the node right
    // of the strip behind each row, and the coefficients of element row j (KG) or of node row j + 1 (KN)
    if constexpr (RG) {                                 // words beyond the grid stay zero
        for (int i = lx; i < M2_DEPTH * RS / 4; i += LW) reinterpret_cast<float4*>(ring)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (!has_halo) {
        for (int i = lx; i < M2_DEPTH; i += LW) {       // the pad right of the last lane's nodes
            float* pad = ring + (size_t)i * RS + 4 * LW;
            *reinterpret_cast<float4*>(pad) = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (ND) *reinterpret_cast<float4*>(pad + UROW) = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (NF) *reinterpret_cast<float4*>(pad + FOFF) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __syncwarp(submask);
    int fetch = jbeg;                                   // next element row to fetch
    unsigned pfo = 0;                                   // byte offset of the slot it goes to
    const unsigned RSB = 4u * RS, RINGB = M2_DEPTH * RSB;
    const size_t row1 = (size_t)(jbeg + 1) * nx + (RG ? xs + lx : x0c);
    const float* usrc = ub + row1;
    const float* nsrc = ND ? P.nu + (size_t)b * P.nodes + row1 : nullptr;
    const float* fsrc = NF ? P.f + (size_t)b * P.nodes + row1 : nullptr;
    const bool xcoef = !ND && lx < CFQ, xhalo = !RG && (lx == LW - 1) && has_halo;
    const int xp = (xcoef || xhalo) ? 1 : 0;            // this lane makes a second copy per row
    const float* polyb = rowpoly + (size_t)b * (KN ? ny : ny - 1) * GS;
    const float* xsrc = xcoef ? polyb + (size_t)(KN ? jbeg + 1 : jbeg) * GS + 4 * lx : usrc + NX;
    const int xstep = xcoef ? GS : nx;
    const unsigned d0 = ring_s + (RG ? 4u : 16u) * lx, d1 = ring_s + 4u * H1 + 16u * lx;
    const unsigned dx = ring_s + (xcoef ? 4u * COEF + 16u * lx : 16u * LW);
    int wok[NX];                                        // RG: which of this lane's words exist
    const int hok = (RG && lx == 0 && has_halo) ? 1 : 0;
#pragma unroll
    for (int i = 0; i < NX; ++i) wok[i] = (RG && xs + lx + LW * i < nx) ? 1 : 0;
    auto copy_row = [&](const unsigned d, const float* src) {            // RG: one row, word by word
#pragma unroll
        for (int i = 0; i < NX; ++i) m2_cp4_if(d + 4u * LW * i, src + LW * i, wok[i]);
        m2_cp4_if(d + 4u * LW * NX, src + LW * NX, hok);
    };
    auto issue = [&]() {
        if (fetch <= jend) {                            // uniform in the unit
            if constexpr (RG) {
                copy_row(d0 + pfo, usrc);
                if constexpr (ND) copy_row(d0 + 4u * UROW + pfo, nsrc);
                if constexpr (NF) copy_row(d0 + 4u * FOFF + pfo, fsrc);
                if constexpr (!ND) m2_cp16_if(dx + pfo, xsrc, xp);
            } else {
                m2_cp16(d0 + pfo, usrc);
                if constexpr (NX == 8) m2_cp16(d1 + pfo, usrc + 4);
                m2_cp16_if(dx + pfo, xsrc, xp);
                if constexpr (ND) {
                    m2_cp16(d0 + 4u * UROW + pfo, nsrc);
                    if constexpr (NX == 8) m2_cp16(d1 + 4u * UROW + pfo, nsrc + 4);
                    m2_cp16_if(ring_s + 4u * UROW + 16u * LW + pfo, nsrc + NX, xhalo ? 1 : 0);
                }
                if constexpr (NF) {
                    m2_cp16(d0 + 4u * FOFF + pfo, fsrc);
                    m2_cp16_if(ring_s + 4u * FOFF + 16u * LW + pfo, fsrc + NX, xhalo ? 1 : 0);
                }
            }
        }
        m2_commit();                                    // one group per step, possibly empty
        ++fetch; usrc += nx; xsrc += xstep;
        if constexpr (ND) nsrc += nx;
        if constexpr (NF) fsrc += nx;
        pfo += RSB;
        if (pfo == RINGB) pfo = 0;
    };
#pragma unroll
    for (int d = 0; d < M2_DEPTH - 1; ++d) issue();

    // a node row from global memory (row 0 of the unit only) / from a slot: the lane's NX nodes and the node right of them
    auto ldrow_g = [&](const float* row, float (&v)[NX + 1]) {
#pragma unroll
        for (int k = 0; k <= NX; ++k) v[k] = (x0 + k < nx && (k < NX || lx < LW - 1 || has_halo)) ? __ldg(row + x0 + k) : 0.f;
    };
    auto ldrow_s = [&](const float* slot, float (&v)[NX + 1]) {
        const float4 q = *reinterpret_cast<const float4*>(slot + 4 * lx);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        if constexpr (NX == 8) {
            const float4 q1 = *reinterpret_cast<const float4*>(slot + H1 + 4 * lx);
            v[4] = q1.x; v[5] = q1.y; v[6] = q1.z; v[7] = q1.w;
        }
        v[NX] = slot[4 * (lx + 1)];
    };
    auto impose_on = [&](float (&v)[NX + 1]) {          // aligned rows: the node right of a lane is imposed by its owner's copy only,
        if (has_first) v[0] = bc0;                      // and the element that would read it does not exist
        if constexpr (RG) {
#pragma unroll
            for (int k = 0; k <= NX; ++k) if (k == kl) v[k] = bc1;
        } else {
            if (has_last) v[NX - 1] = bc1;
        }
    };

    // ---- state of the node row below the current element row
    float lo[NX + 1], cu[NX + 1], eh[NX], Fh[NX], Gv[NX + 1];
    ldrow_g(ub + (size_t)jbeg * nx, lo);
    if (impose) impose_on(lo);
#pragma unroll
    for (int k = 0; k < NX; ++k) { eh[k] = lo[k + 1] - lo[k]; Fh[k] = 0.f; Gv[k] = 0.f; }
    Gv[NX] = 0.f;                                       // the left-over node's

    // KN: nu at this lane's nodes and at the node right of them, from the polynomial of that node row
    auto nu_row = [&](const u64 (&gg)[GS / 2], float (&nn)[NX + 1]) {
#pragma unroll
        for (int h = 0; h < NX / 2; ++h) {
            u64 e = gg[M];
#pragma unroll
            for (int i = M - 1; i >= 0; --i) e = m2_fma2(e, cnp[h], gg[i]);
            float e0, e1;
            m2_unpack(e, e0, e1);
            nn[2 * h] = m2_ex2(e0); nn[2 * h + 1] = m2_ex2(e1);
        }
        float gh, dmy;
        m2_unpack(gg[M], gh, dmy);
#pragma unroll
        for (int i = M - 1; i >= 0; --i) { float gi; m2_unpack(gg[i], gi, dmy); gh = fmaf(gh, cnh, gi); }
        nn[NX] = m2_ex2(gh);
    };
    float nlo[NX + 1], hnu[NX];                         // KN, ND: nu on the node row below and its sums over x-neighbours
    if constexpr (ND) ldrow_g(P.nu + (size_t)b * P.nodes + (size_t)jbeg * nx, nlo);
    if constexpr (KN) {
        u64 gg[GS / 2];
        const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(polyb + (size_t)jbeg * GS);
#pragma unroll
        for (int k = 0; k < GS / 4; ++k) { const ulonglong2 t = __ldg(gp + k); gg[2 * k] = t.x; gg[2 * k + 1] = t.y; }
        nu_row(gg, nlo);
    }
    if constexpr (KN || ND) {
#pragma unroll
        for (int k = 0; k < NX; ++k) hnu[k] = nlo[k] + nlo[k + 1];
    }

    // NF: x-smoothed forcing (hx/6) (f[k-1] + 4 f[k] + f[k+1]) of a node row, one-sided on the Dirichlet columns
    const float m6x = P.hx * (1.f / 6.f), m6y = P.hy * (1.f / 6.f);
    const float mxl = has_first ? 0.f : m6x;            // weight of the node left of the lane
    const float mxr = (!RG && has_last) ? 0.f : m6x;    // (RG: beyond the grid f is zero)
    float mxc[NX];                                      // central weights
#pragma unroll
    for (int k = 0; k < NX; ++k) mxc[k] = ((k == 0 && has_first) || (RG ? k == kl : (k == NX - 1 && has_last))) ? 2.f * m6x : 4.f * m6x;
    auto smooth_x = [&](const float (&f)[NX + 1], float (&g)[NX]) {
        const float fleft = __shfl_up_sync(submask, f[NX - 1], 1, LW);   // lane 0: its own value, unused (mxl = 0 or a lane that stores nothing)
        g[0] = fmaf(mxl, fleft, fmaf(mxc[0], f[0], m6x * f[1]));
#pragma unroll
        for (int k = 1; k < NX; ++k) g[k] = fmaf(m6x, f[k - 1], fmaf(mxc[k], f[k], (k == NX - 1 ? mxr : m6x) * f[k + 1]));
    };
    float gf_lo[NX], gf_mid[NX];                        // smoothed f of the row below the current node row, and of that row
#pragma unroll
    for (int k = 0; k < NX; ++k) { gf_lo[k] = 0.f; gf_mid[k] = 0.f; }
    if constexpr (NF) {
        const float* fb = P.f + (size_t)b * P.nodes + (size_t)jbeg * nx;
        float f0[NX + 1];
        ldrow_g(fb, f0);
        smooth_x(f0, gf_mid);
        if (jbeg > 0) {                                 // the row below the unit's first row (uniform)
            ldrow_g(fb - nx, f0);
            smooth_x(f0, gf_lo);
        }
    }
    float en = 0.f, ell = 0.f;                          // sum u (K u) and sum w u of the rows this lane went over
    float* rrow = EO ? nullptr : rb + (size_t)jbeg * nx + (RG ? xs + lx : x0c);
    unsigned rdo = 0;                                   // byte offset of the slot to read
    // RG: which of the lane's words are stored, and which one of them is a Dirichlet column (stored as zero)
    int sok[NX], iz = -1;
#pragma unroll
    for (int i = 0; i < NX; ++i) {
        const int w = lx + LW * i;
        sok[i] = wok[i] && (strip == 0 || w >= NX);
        if (RG && !nomask && (xs + w == nx - 1)) iz = i;
    }
    const bool z0 = RG && !nomask && has_first;         // word 0 of lane 0
    auto store_row = [&](float* dst, const float (&o)[NX]) {
        if constexpr (RG) {
            *reinterpret_cast<float4*>(obuf + 4 * lx) = make_float4(o[0], o[1], o[2], o[3]);
            __syncwarp(submask);
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                float v = obuf[lx + LW * i];
                if (i == iz || (i == 0 && z0)) v = 0.f;
                if (sok[i]) dst[LW * i] = v;
            }
            if (extra && lx == 0) dst[NX * LW] = 0.f;
        } else if (owner) {
#pragma unroll
            for (int h = 0; h < NX / 4; ++h)
                *reinterpret_cast<float4*>(dst + 4 * h) = make_float4(o[4 * h], o[4 * h + 1], o[4 * h + 2], o[4 * h + 3]);
        }
    };
    // load energy of a row (weight wrow: half on the first and last row) with constant forcing
    auto load_energy = [&](const float (&a)[NX + 1], const float wrow) {
        float w = wf * a[0];
#pragma unroll
        for (int k = 1; k < NX - 1; ++k) w += a[k];
        w = fmaf(wl, a[NX - 1], w);
        if constexpr (RG) {
#pragma unroll
            for (int k = 0; k < NX; ++k) if (k == kl) w = fmaf(-0.5f, a[k], w);
            w = fmaf(0.5f * wX, a[NX], w);
        }
        ell = fmaf(wrow, w, ell);
    };
    // the finished row: K u scaled, masked, its nodal load added
    auto finish = [&](const float (&raw)[NX], const float wrow, float (&o)[NX]) {
#pragma unroll
        for (int k = 0; k < NX; ++k)
            o[k] = fmaf((k == 0) ? gsf : (k == NX - 1) ? gsl : gku, raw[k], wrow * ((k == 0) ? nlf : (k == NX - 1) ? nll : nl));
        if constexpr (RG) {
            if (nomask && hasf) {                       // raw residual wanted: half a load on the Dirichlet columns
#pragma unroll
                for (int k = 0; k < NX; ++k) if (x0 + k == 0 || k == kl) o[k] = fmaf(-0.5f * wrow, nl, o[k]);
            }
        }
    };

    // One element row: a holds node row j, c receives node row j + 1.
    auto step = [&](float (&a)[NX + 1], float (&c)[NX + 1], const int j) {
        m2_wait<M2_DEPTH - 2>();                        // this step's slot has landed (for the lanes that copied it)
        __syncwarp(submask);                            // ... is visible to the unit, and the slot read last step is free
        issue();                                        // refill it
        const float* slot = reinterpret_cast<const float*>(reinterpret_cast<const char*>(ring) + rdo);
        rdo += RSB;
        if (rdo == RINGB) rdo = 0;
        ldrow_s(slot, c);
        if (impose) impose_on(c);
        u64 g2[GS / 2];
        if constexpr (!ND) {
            const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(slot + COEF);
#pragma unroll
            for (int k = 0; k < GS / 4; ++k) { const ulonglong2 t = gp[k]; g2[2 * k] = t.x; g2[2 * k + 1] = t.y; }
        }
        float ncur[NX + 1];
        if constexpr (KN) nu_row(g2, ncur);
        if constexpr (ND) ldrow_s(slot + UROW, ncur);

        float Fp = 0.f, gr = 0.f, F0 = 0.f, g0 = 0.f, sk = c[0] - a[0], raw[NX];
        float ex[2] = {0.f, 0.f}, ey[2] = {0.f, 0.f};   // EO: sums over this lane's elements of N D^2 along x and along y
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const float e1 = c[k + 1] - c[k];
            const float s1 = c[k + 1] - a[k + 1];
            const float e0 = eh[k];
            eh[k] = e1;
            const float t = e1 - e0;
            float Px, Qx, Py, Qy, bt;
            if constexpr (KN || ND) {
                // Q1 interpolation of nu to the Gauss points leaves sums over corners: with the sums h0, h1 over the bottom
                // and top edge and v0, v1 over the left and right one, 3 P = S + h0, 3 Q = S + h1, 3 B = S / 2 (same in y)
                const float h0 = hnu[k], h1 = ncur[k] + ncur[k + 1];
                hnu[k] = h1;
                const float v0 = nlo[k] + ncur[k], v1 = nlo[k + 1] + ncur[k + 1];
                if constexpr (EO) {
                    const float dh = h1 - h0, dv = v1 - v0;
                    Px = fmaf(DN_GA, dh, h0); Qx = fmaf(DN_GB, dh, h0);
                    Py = fmaf(DN_GA, dv, v0); Qy = fmaf(DN_GB, dv, v0);
                    bt = 0.f;
                } else {
                    const float S = h0 + h1;
                    Px = S + h0; Qx = S + h1; Py = S + v0; Qy = S + v1;
                    bt = (0.5f * S) * t;
                }
            } else {
                u64 ea = g2[M], eb = g2[M];             // (row a, row b) pairs at column a / column b
                u64 ca, cb;
                if constexpr (CREG) { ca = cda[k]; cb = cdb[k]; }
                else { const ulonglong2 cc = *reinterpret_cast<const ulonglong2*>(cpl + k * LW); ca = cc.x; cb = cc.y; }
#pragma unroll
                for (int i = M - 1; i >= 0; --i) { ea = m2_fma2(ea, ca, g2[i]); eb = m2_fma2(eb, cb, g2[i]); }
                float xaa, xab, xba, xbb;
                m2_unpack(ea, xaa, xab);
                m2_unpack(eb, xba, xbb);
                const float naa = m2_ex2(xaa), nab = m2_ex2(xab), nba = m2_ex2(xba), nbb = m2_ex2(xbb);
                const float Na = naa + nba, Nb = nab + nbb, Ma = naa + nab;
                if constexpr (EO) {
                    Px = Na; Qx = Nb; Py = Ma; Qy = nba + nbb; bt = 0.f;
                } else {
                    const float S = Na + Nb, aS = (6.f * DN_GA) * S;
                    Px = fmaf(6.f * (DN_GB - DN_GA), Na, aS); Qx = fmaf(6.f, S, -Px);
                    Py = fmaf(6.f * (DN_GB - DN_GA), Ma, aS); Qy = fmaf(6.f, S, -Py);
                    bt = S * t;
                }
            }
            if constexpr (EO) {                         // P, Q hold the sums of nu on the Gauss rows / columns here
                const float Dxa = fmaf(DN_GA, t, e0), Dxb = fmaf(DN_GB, t, e0);
                const float Dya = fmaf(DN_GA, t, sk), Dyb = fmaf(DN_GB, t, sk);
                if (RG || k == NX - 1) { Px *= em[k]; Qx *= em[k]; Py *= em[k]; Qy *= em[k]; }
                ex[0] = fmaf(Px * Dxa, Dxa, ex[0]); ex[1] = fmaf(Qx * Dxb, Dxb, ex[1]);
                ey[0] = fmaf(Py * Dya, Dya, ey[0]); ey[1] = fmaf(Qy * Dyb, Dyb, ey[1]);
            } else {
                const float Fx = fmaf(Px, e0, Fh[k] + bt);          // the bottom edge is complete
                Fh[k] = fmaf(Qx, e1, -bt);                          // the top edge waits for the element above
                const float g = fmaf(Py, sk, bt);
                if (k == 0) {
                    F0 = Fx; g0 = g;
                } else {
                    const bool masked = RG || k == NX - 1;
                    const float Gk = masked ? fmaf(em[k], g, gr) : g + gr;
                    const float dxf = masked ? fmaf(-em[k], Fx, Fp) : Fp - Fx;
                    raw[k] = fmaf(rho, Gv[k] - Gk, dxf);
                    Gv[k] = Gk;
                }
                gr = fmaf(Qy, s1, -bt);
                Fp = Fx;
            }
            sk = s1;
        }
        float gf_up[NX];                                // NF: smoothed f of node row j + 1
        if constexpr (NF) {
            float fu[NX + 1];
            ldrow_s(slot + FOFF, fu);
            smooth_x(fu, gf_up);
        }
        if constexpr (!EO) {
            // forces of the element left of this lane's first node
            const float fl = __shfl_up_sync(submask, Fp, 1, LW);
            const float gl = __shfl_up_sync(submask, gr, 1, LW);
            const float Gk = fmaf(gl, lm, RG ? em[0] * g0 : g0);
            raw[0] = fmaf(rho, Gv[0] - Gk, fmaf(fl, lm, RG ? -em[0] * F0 : -F0));
            Gv[0] = Gk;
        }
        if (j >= n0) {                                  // uniform: this unit owns node row j
            if constexpr (EO) {
                en += fmaf(rho, ey[0] + ey[1], ex[0] + ex[1]);      // element row j belongs to the chunk that owns node row j
            } else {
#pragma unroll
                for (int k = 0; k < NX; ++k) en = fmaf(a[k], raw[k], en);      // Euler's identity
                if constexpr (RG && !NF) en = fmaf(a[NX] * wX, fmaf(rho, Gv[NX] - gr, Fp), en);
            }
            float o[NX];
            if constexpr (NF) {
                // load of node row j: the y-smoothing of the three smoothed rows (row 0 has no row below)
                const float wc = (j == 0) ? 2.f * m6y : 4.f * m6y;
#pragma unroll
                for (int k = 0; k < NX; ++k) {
                    const float F = fmaf(m6y, gf_lo[k] + gf_up[k], wc * gf_mid[k]);
                    ell = fmaf(a[k], F, ell);
                    if constexpr (!EO) o[k] = ((k == 0) ? gs * gm0 : (k == NX - 1) ? gs * gmL : gs) * fmaf(ku, raw[k], -F);
                }
            } else {
                const float wrow = (j == 0) ? 0.5f : 1.f;
                if (hasf) load_energy(a, wrow);
                if constexpr (!EO) finish(raw, wrow, o);
            }
            if constexpr (!EO) store_row(rrow, o);
        }
        if constexpr (RG) Gv[NX] = gr;
        if constexpr (!EO) rrow += nx;
        if constexpr (NF) {
#pragma unroll
            for (int k = 0; k < NX; ++k) { gf_lo[k] = gf_mid[k]; gf_mid[k] = gf_up[k]; }
        }
        if constexpr (KN || ND) {
#pragma unroll
            for (int k = 0; k <= NX; ++k) nlo[k] = ncur[k];
        }
    };

    {
        int j = jbeg;
        while (true) {
            step(lo, cu, j);
            if (++j > jend) {
#pragma unroll
                for (int k = 0; k <= NX; ++k) lo[k] = cu[k];
                break;
            }
            step(cu, lo, j);
            if (++j > jend) break;
        }
    }
    m2_wait<0>();

    // ---- the top node row of the grid has no element row above it (lo holds it; its edges are complete)
    if (n1 == ny) {
        float o[NX], raw[NX];
        if constexpr (!EO) {
            const float fl = __shfl_up_sync(submask, Fh[NX - 1], 1, LW);
            raw[0] = fmaf(rho, Gv[0], fmaf(fl, lm, -em[0] * Fh[0]));
#pragma unroll
            for (int k = 1; k < NX; ++k) raw[k] = fmaf(rho, Gv[k], fmaf(-em[k], Fh[k], Fh[k - 1]));
#pragma unroll
            for (int k = 0; k < NX; ++k) en = fmaf(lo[k], raw[k], en);
            if constexpr (RG && !NF) en = fmaf(lo[NX] * wX, fmaf(rho, Gv[NX], Fh[NX - 1]), en);
        }
        if constexpr (NF) {
#pragma unroll
            for (int k = 0; k < NX; ++k) {              // the top row: one-sided in y
                const float F = m6y * fmaf(2.f, gf_mid[k], gf_lo[k]);
                ell = fmaf(lo[k], F, ell);
                if constexpr (!EO) o[k] = ((k == 0) ? gs * gm0 : (k == NX - 1) ? gs * gmL : gs) * fmaf(ku, raw[k], -F);
            }
        } else {
            load_energy(lo, 0.5f);
            if constexpr (!EO) finish(raw, 0.5f, o);
        }
        if constexpr (!EO) {
            if constexpr (RG) __syncwarp(submask);      // the row before it has left the buffer
            store_row(rb + (size_t)(ny - 1) * nx + (RG ? xs + lx : x0c), o);
        }
    }

    // ---- energy partial of this unit: owning lanes summed in a fixed order in double
    double d = owner ? 0.5 * (double)ku * (double)en : 0.0;
    double l = !owner ? 0.0 : NF ? (double)ell : hasf ? (double)fw * (double)ell : 0.0;
    for (int off = LW >> 1; off > 0; off >>= 1) {
        d += __shfl_down_sync(submask, d, off, LW);
        l += __shfl_down_sync(submask, l, off, LW);
    }
    if (lx == 0) {
        double* slot = P.partials + 2 * ((size_t)b * P.nblk + (size_t)chunk * nstrip + strip);
        slot[0] = d; slot[1] = l;
    }
}

template <int NX, int M, int MODE, bool NF, bool EO, int LWC, bool RG>
cudaError_t launch_m2(const Params& P, const float* rowpoly, const M2Geo& g, cudaStream_t s) {
    const int subs = 32 / g.LW;
    const size_t per_unit = (size_t)M2_DEPTH * g.RS + (RG ? NX * g.LW : 0);
    size_t smem = sizeof(float) * (M2_WARPS * subs * per_unit + ((MODE == 0 && NX == 8) ? 4 * NX * g.LW : 0));
    if (g.blocks < m2_minb(NX) && smem < kM2ThirdOfSm) smem = kM2ThirdOfSm;      // keeps the fourth block out
    const long long per_block = (long long)M2_WARPS * subs;
    const unsigned blocks = (unsigned)((g.units + per_block - 1) / per_block);
    const cudaError_t e = allow_shared(march2d_kernel<NX, M, MODE, NF, EO, LWC, RG>, smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(march2d_kernel<NX, M, MODE, NF, EO, LWC, RG>, dim3(blocks), dim3(M2_WARPS * 32), smem, s, P, rowpoly, g);
}

// The lane counts compiled in where they matter (3 to 9 % against taking them from G): fused, constant forcing.
template <int M, int MODE>
cudaError_t launch_m2_mode(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    const bool eo = P.r == nullptr;
    if (ragged) {
        if (P.f) return eo ? launch_m2<4, M, MODE, true, true, 0, true>(P, rowpoly, g, s) : launch_m2<4, M, MODE, true, false, 0, true>(P, rowpoly, g, s);
        if (eo) return launch_m2<4, M, MODE, false, true, 0, true>(P, rowpoly, g, s);
        if (g.LW == 16) return launch_m2<4, M, MODE, false, false, 16, true>(P, rowpoly, g, s);
        return g.LW == 32 ? launch_m2<4, M, MODE, false, false, 32, true>(P, rowpoly, g, s) : launch_m2<4, M, MODE, false, false, 0, true>(P, rowpoly, g, s);
    }
    if (P.f) return eo ? launch_m2<4, M, MODE, true, true, 0, false>(P, rowpoly, g, s) : launch_m2<4, M, MODE, true, false, 0, false>(P, rowpoly, g, s);
    if constexpr (MODE != 2) {
        if (g.NX == 8) return eo ? launch_m2<8, M, MODE, false, true, 32, false>(P, rowpoly, g, s) : launch_m2<8, M, MODE, false, false, 32, false>(P, rowpoly, g, s);
    }
    if (eo) return g.LW == 32 ? launch_m2<4, M, MODE, false, true, 32, false>(P, rowpoly, g, s) : launch_m2<4, M, MODE, false, true, 0, false>(P, rowpoly, g, s);
    if (g.LW == 32) return launch_m2<4, M, MODE, false, false, 32, false>(P, rowpoly, g, s);
    if (g.LW == 16) return launch_m2<4, M, MODE, false, false, 16, false>(P, rowpoly, g, s);
    return launch_m2<4, M, MODE, false, false, 0, false>(P, rowpoly, g, s);
}

template <int M>
cudaError_t launch_m2_m(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    return (P.nu_mode == DN_NU_KL_NODAL) ? launch_m2_mode<M, 1>(P, rowpoly, g, ragged, s) : launch_m2_mode<M, 0>(P, rowpoly, g, ragged, s);
}

}  // namespace

#if DN_M2_PART == 1
cudaError_t launch_march2d_m34(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 3 ? launch_m2_m<3>(P, rowpoly, g, ragged, s) : launch_m2_m<4>(P, rowpoly, g, ragged, s);
}
#elif DN_M2_PART == 2
cudaError_t launch_march2d_m56(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 5 ? launch_m2_m<5>(P, rowpoly, g, ragged, s) : launch_m2_m<6>(P, rowpoly, g, ragged, s);
}
#elif DN_M2_PART == 3
cudaError_t launch_march2d_m78(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    return P.m == 7 ? launch_m2_m<7>(P, rowpoly, g, ragged, s) : launch_m2_m<8>(P, rowpoly, g, ragged, s);
}
#else
cudaError_t launch_march2d_m12(const Params& P, const float* rowpoly, const M2Geo& g, bool ragged, cudaStream_t s) {
    if (P.nu_mode == DN_NU_NODAL) return launch_m2_mode<1, 2>(P, rowpoly, g, ragged, s);
    return P.m == 1 ? launch_m2_m<1>(P, rowpoly, g, ragged, s) : launch_m2_m<2>(P, rowpoly, g, ragged, s);
}

namespace {

// Nodes per lane: 4, except on aligned rows of 129 to 256 nodes that are a multiple of 8, which one warp covers with 8
// (the nodal modes' 8-node rows gain nothing over strips of 4 nodes per lane where two strips cover the row).
int m2_nodes_per_lane(const dn_problem& p, bool ragged) {
    const int nx = p.grid.nx;
    return (!ragged && p.f == nullptr && nx > 128 && nx <= 256 && nx % 8 == 0 && p.nu_mode != DN_NU_NODAL) ? 8 : 4;
}

M2Geo m2_search(const dn_problem& p, bool ragged, int sms) {
    M2Geo g{};
    const int nx = p.grid.nx, ny = p.grid.ny;
    const bool nf = p.f != nullptr, nomask = (p.flags & DN_NO_MASK) != 0;
    g.NX = m2_nodes_per_lane(p, ragged);
    g.LW = 8; g.lwsh = 3;
    const int left = (ragged && !nf && !nomask) ? 1 : 0;         // one node may be left over
    while (g.LW < 32 && g.LW * g.NX + left < nx) { g.LW *= 2; ++g.lwsh; }
    auto strips = [&](int lw) {                                  // a later strip's first lane repeats the last of the one before
        const int cols = lw * g.NX, stride = cols - g.NX;
        return (nx <= cols + left) ? 1 : (nx - cols + stride - 1) / stride + 1;
    };
    // Rows cut into strips: units of 16 lanes where that saves 10 % of the lanes' nodes (512 nodes: 5 strips of 128 columns or 9 of 64,
    // 640 and 576) or, with a stored field, whose extra columns are extra traffic, 15 %; not in small problems, whose units are latency.
    // From 380 problems both ways: 512^2 x 64 KL m = 4 60.3 -> 55.5 us, 513^2 x 64 KL at the nodes 66.0 -> 64.5, 132^2 x 425 stored
    // 33.8 -> 28.0, 144^2 x 1174 stored 76.6 -> 67.4, the energy alone 152^2 x 627 with forcing 65.6 -> 49.7; against 8 % (650 x 701 x 14 KL
    // m = 4 31.9 -> 32.7, 632 x 833 x 35 stored 44.7 -> 46.6), a stored field at 12 % (384 x 120 x 295 37.2 -> 39.5), small ragged
    // problems (393^2 x 7 13.0 -> 13.6, 297 x 93 x 71 stored 13.9 -> 14.7) and aligned ones (720^2 8.0 -> 10.6); but 160^2 x 41 8.9 -> 8.3, and
    // ragged rows where a quarter is saved (129 to 184 nodes: 141^2 x 72 KL at the nodes with forcing 26.1 -> 25.2)
    const bool stored = p.nu_mode == DN_NU_NODAL;
    const int lanes = 100 * 16 * strips(16), keep = (stored && !nf) ? 85 : 90;
    const long long few = (ragged && (stored || lanes > 75 * 32 * strips(32))) ? 1ll << 21 : 1ll << 20;
    if (g.LW == 32 && g.NX == 4 && lanes <= keep * 32 * strips(32) && (long long)p.batch * nx * ny >= few) { g.LW = 16; g.lwsh = 4; }
    const int cols = g.LW * g.NX;
    g.extra = (left && nx == cols + 1) ? 1 : 0;
    g.nstrip = strips(g.LW);
    const int rows = 1 + (p.nu_mode == DN_NU_NODAL ? 1 : 0) + (nf ? 1 : 0);
    g.RS = rows * (cols + 4) + (p.nu_mode == DN_NU_NODAL ? 0 : m2_gs(p.kl_modes));
    // Three fields (stored field and nodal forcing) on wide, tall grids stream better in fewer and longer units, three blocks to an SM:
    // 4096^2 58.3 us with four, 55.4 with three, 2048^2 x 4 56.5 and 54.6, 1536^2 x 7 56.1 and 53.5; 192^2 x 455 62 and 69.
    g.blocks = (p.nu_mode == DN_NU_NODAL && nf && !ragged && nx >= 1024 && ny >= 256) ? 3 : m2_minb(g.NX);
    const long long slots = (long long)sms * g.blocks * M2_WARPS * (32 / g.LW);
    // R from a cost search over waves of units; a unit pays the recomputed row and the filling of its ring (a stored field,
    // 1024^2 x 32: R = 128, one wave, 78.6 us, R = 63 74.3, R = 32 75.4, R = 16 81.1; right behind the kernel that wrote the
    // field, whose write-back long units meet all at once: 86 and 79 us)
    long long best = -1;
    int bestR = 2;
    for (int R = 2; R <= 1024; ++R) {
        if (R > ny && R > 2) break;
        // chunks of R rows, and behind them one of the rows that are left over: those units run in the slots that the
        // last wave of full ones leaves idle, and what does not fit there after it
        const long long nch = (ny + R - 1) / R, rest = ny % R, rows = (long long)p.batch * g.nstrip;
        const long long full = rows * (rest ? nch - 1 : nch), waves = full / slots, over = full % slots;
        long long span = (waves + (over ? 1 : 0)) * (R + 5);
        if (rest) {
            const long long room = over ? (slots - over) * ((R + 5) / (rest + 5)) : 0;
            if (rows > room) span += (rows - room + slots - 1) / slots * (rest + 5);
        }
        // long units also end further apart (3 R; 1024^2 x 32, above), less so where one wave of units of moderate length fills the
        // device: 4096^2 44.4 us with R = 58, 47.8 with R = 29 (KL m = 4 50.2 and 54.5), 513^2 x 64 60.9 with 74, 64.9 with 37
        // (KL at the nodes with imposed faces 67.5 and 67.0); but 128^2 x 1024 with forcing, where one wave is 86 % full, 59.6
        // with R = 64, 55.4 with 32
        const bool one_wave = R <= 96 && rows * nch <= slots && 100 * rows * nch >= 94 * slots;
        const long long cost = 16 * span + (one_wave ? 2 : 3) * R;
        if (best < 0 || cost < best) { best = cost; bestR = R; g.span = (int)span; }
    }
    g.R = bestR;
    g.nchunk = (ny + g.R - 1) / g.R;
    g.units = (long long)p.batch * g.nstrip * g.nchunk;
    return g;
}

M2Geo m2_geometry(const dn_problem& p, bool ragged) {
    const int sms = sm_count();
    return memo_geometry<M2Geo>(p, sms, [&]() { return m2_search(p, ragged, sms); }, ragged ? 1 : 0);
}

}  // namespace

// Aligned rows that one unit covers: at most 128 nodes, or at most 256 in the KL modes (a multiple of 8, so that only
// the last element of the last lane falls outside the grid).  Constant forcing.
bool row2d_applicable(const dn_problem& p) {
    if (!(p.grid.dim == 2 && p.f == nullptr && p.grid.nx % 4 == 0 && p.grid.nx >= 8 && p.grid.nx <= 256 && p.grid.ny >= 2))
        return false;
    if (p.grid.nx <= 128) return true;
    return p.grid.nx % 8 == 0 && p.nu_mode != DN_NU_NODAL;
}

// Aligned rows cut into strips whose lanes are at most 15 % more than the row, or that the tiled kernel cannot serve.
bool strip2d_applicable(const dn_problem& p) {
    if (!(p.grid.dim == 2 && p.grid.nx % 4 == 0 && p.grid.nx >= (p.f ? 8 : 256) && p.grid.ny >= 16)) return false;
    const long long lanes = (long long)((p.grid.nx - 128 + 123) / 124 + 1) * 128;
    return !tiled2d_applicable(p) || 100 * lanes <= 115ll * p.grid.nx || p.f != nullptr;
}

// Which aligned 2D problems the marching kernel takes from the tiled one (which serves constant forcing on rows of at
// most 2048 nodes).  With the residual: all of them (256^2 x 128: 33.2 against 33.2 us KL, 27.3 against 29.0 us with a
// stored field; 1024^2 x 8: 30.3 against 33.3 and 21.7 against 29.0; 384^2 x 56: 34.7 against 45.6 and 23.8 against 39.5).
// Energy only: the tiled kernel keeps 8 nodes in a lane and runs no row twice, so it is ahead where its rows of 256 lanes
// are well filled and the march is short.  The line is drawn by what the march occupies (lanes times rows of all its
// waves, and 6 rows to start) over the lanes of the tiled kernel's rows: KL at 1.26 (384^2 x 227, 1.13: 92.7 against
// 107.4 us; 384^2 x 56, 1.32: 35.1 against 33.2), from 768 nodes on, where the tiled kernel runs best, at 1.16 (896^2 x
// 41, 1.14: 78.6 against 84.6; 1024^2 x 32, 1.28: 78.7 against 72.2); with 8 nodes per lane at 1.33 (m <= 5), KL at the nodes 1.6
// (192^2 x 910, 1.32: 99.5 against 121.2; 192^2 x 227, 1.51: 41.8 against 37.4, at the nodes 28.2 against 33.2; 256^2 x
// 128, 1.68: 35.4 against 27.2 and 24.9 against 23.2); stored field at 1.6 (512^2 x 128, 1.46: 63.7 against 76.1;
// 512^2 x 32, 1.70: 24.1 against 22.5).
bool march2d_chosen(const dn_problem& p, bool want_r) {
    const int nx = p.grid.nx;
    if (!(p.grid.dim == 2 && nx % 4 == 0 && nx >= 8)) return false;
    if (want_r || p.f != nullptr || !tiled2d_applicable(p)) return true;
    const M2Geo g = m2_geometry(p, false);
    const double march = (double)(g.span + 6) * sm_count() * m2_minb(g.NX) * M2_WARPS * 32 * g.NX;
    const double tiled = (double)p.batch * p.grid.ny * (nx <= 128 ? 128 : (nx + 255) / 256 * 256);
    const double line = (p.nu_mode == DN_NU_NODAL) ? 1.6 : (g.NX == 8 && p.nu_mode == DN_NU_KL_NODAL) ? 1.6
                        : (g.NX == 8 && p.kl_modes <= 5) ? 1.33 : nx < 768 ? 1.26 : 1.16;
    return march <= line * tiled;
}

Launch march2d_geometry(const dn_problem& p, int path) {
    const M2Geo g = m2_geometry(p, path == PATH_RAGGED2D);
    Launch l{};
    l.path = path;
    l.nblk = g.nchunk * g.nstrip;
    l.chunk = g.R;
    l.variant = g.nstrip;
    return l;
}

size_t march2d_rowpoly_floats(const dn_problem& p) {
    if (p.grid.dim != 2 || p.nu_mode == DN_NU_NODAL) return 0;   // the stored field needs no table
    return (size_t)p.batch * p.grid.ny * m2_gs(p.kl_modes);      // ny - 1 element rows, or ny node rows (KL at the nodes)
}

int march2d_rowpoly_stride(int kl_modes) { return m2_gs(kl_modes); }

cudaError_t launch_march2d(const Params& P, int path, const float* rowpoly, cudaStream_t s) {
    dn_problem p{};
    p.grid.dim = 2; p.grid.nx = P.nx; p.grid.ny = P.ny; p.grid.nz = 1; p.batch = P.batch;
    p.nu_mode = P.nu_mode; p.kl_modes = P.m; p.f = P.f; p.flags = P.flags;
    const bool ragged = path == PATH_RAGGED2D;
    const M2Geo g = m2_geometry(p, ragged);
    if (P.nu_mode == DN_NU_NODAL || P.m <= 2) return launch_march2d_m12(P, rowpoly, g, ragged, s);
    if (P.m <= 4) return launch_march2d_m34(P, rowpoly, g, ragged, s);
    if (P.m <= 6) return launch_march2d_m56(P, rowpoly, g, ragged, s);
    return launch_march2d_m78(P, rowpoly, g, ragged, s);
}
#endif  // DN_M2_PART

}  // namespace dn
