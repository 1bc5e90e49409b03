// Mirrored-pair kernel for 2D grids: energy and residual fused, constant forcing, and its energy-only variant; rows of any
// length and alignment.  The march, the edge arithmetic and the ring are those of the 2D marching kernel (dn_march2d.cu);
// what differs is that a lane owns 4 columns counted from the left face and the 4 columns mirrored at x = 1/2, as the two
// halves of packed f32x2 registers.
//
// Why pairs.  The element, the Gauss rule, the Dirichlet faces and the gather are symmetric under x -> 1 - x, and
// cos(pi x) only changes sign.  So both sides run the same instructions, two elements per issue slot, the work per row that
// does not depend on its length (ring, coefficients, loop) is shared by 8 nodes, and with KL at the Gauss points the
// polynomial of the exponent splits into E(c^2) + c O(c^2) on the left and E(c^2) - c O(c^2) at the mirrored point: m + 1
// packed operations where two Horner chains take 2 m.
//
// Layout of the work.  A work unit is one sample, one chunk of R node rows and one strip of 4 LW columns of either side;
// it belongs to LW = 8, 16 or 32 lanes of one warp.  A side has (nx + 1) / 2 columns on the left and nx / 2 on the right.
// A side that fits a unit is one strip; wider ones overlap by one lane, whose elements are recomputed to hand
// their forces to the next lane.  With an even number of nodes both sides compute the middle element (each uses its own corner);
// with an odd one the middle node belongs to the left side, and where the columns of a side end exactly before it, it
// takes no lane: the last lane finishes it from both sides.  Rows arrive in the ring already interleaved into pairs
// (4-byte asynchronous copies: coalesced for every row offset, any destination).
//
// @@MEASURED@@
//
// The file is compiled in four parts side by side (m = 1, 2 and the stored field; 3, 4; 5, 6; 7, 8).
#include "dn_internal.cuh"
#include "dn_pair.cuh"

#ifndef DN_P2_PART
#define DN_P2_PART 0
#endif

namespace dn {

struct P2Geo {
    int R, nchunk, nstrip;
    int LW, lwsh;         // lanes per unit and log2 of it
    int RS;               // floats per ring slot
    int extra;            // the middle node is the one right of the last strip
    long long units;
};
cudaError_t launch_pair2d_m12(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s);
cudaError_t launch_pair2d_m34(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s);
cudaError_t launch_pair2d_m56(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s);
cudaError_t launch_pair2d_m78(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s);

namespace {

constexpr int P2_WARPS = 4;                       // warps per block (each warp is on its own)
constexpr int P2_DEPTH = 6;                       // ring slots per unit (DEPTH - 1 rows in flight)
constexpr int P2_MINB = 3;                        // resident blocks per SM: up to 168 registers
constexpr int NX = 4;                             // columns per lane and side

// Floats per row of the coefficient table: (Gauss row a, b) pairs, or each coefficient twice, for k = 0..M, padded to a multiple of 4.
__host__ __device__ constexpr int p2_gs(int m) { return (2 * (m + 1) + 3) / 4 * 4; }

// MODE 0: KL at the Gauss points; 1 (KN): KL at the nodes, then Q1 interpolation; 2 (ND): stored nodal field
// EO: energy only.  The same march, but every element adds its own energy and nothing is gathered or stored.
// LWC: lanes per unit at compile time (32 or 16), or 0: taken from G
// RG: rows that are not a multiple of 8, or an r that is not 16-byte aligned: finished rows pass through one row of shared
// memory and are stored word by word; nodes that belong to the other side are left out.
template <int M, int MODE, bool EO, int LWC, bool RG>
__global__ void __launch_bounds__(P2_WARPS * 32, P2_MINB)
pair2d_kernel(const Params P, const float* __restrict__ rowpoly, const P2Geo G) {
    extern __shared__ __align__(16) float smem[];
    dep_wait();                                         // the tables of this call are complete
    dep_release();                                      // the finaliser may move in behind the last units
    constexpr bool KG = (MODE == 0), KN = (MODE == 1), ND = (MODE == 2);
    constexpr int GS = p2_gs(M);
    constexpr int CFQ = ND ? 0 : GS / 4;                // 16-byte pieces of a coefficient row
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int LW = LWC ? LWC : G.LW, lwsh = (LWC == 32) ? 5 : (LWC == 16) ? 4 : G.lwsh, SUBS = 32 >> lwsh;
    const int sub = lane >> lwsh, lx = lane & (LW - 1);
    const unsigned submask = (LW == 32) ? 0xffffffffu : (((1u << LW) - 1u) << (sub * LW));
    const unsigned su = (blockIdx.x * P2_WARPS + warp) * SUBS + sub;      // fewer than 2^32 units of at least 4 nodes fit a GPU
    if (su >= G.units) return;                          // the other units of the warp synchronise among themselves only
    const unsigned nstrip = G.nstrip, sq = su / nstrip;
    const int strip = (int)(su - sq * nstrip);
    const int chunk = (int)(sq / (unsigned)P.batch), b = (int)(sq - (unsigned)chunk * (unsigned)P.batch);

    const int nx = P.nx, ny = P.ny;
    const int ownL = (nx + 1) / 2, ownR = nx / 2;       // columns of the left and of the mirrored side
    const int xs = strip * (LW - 1) * NX;               // first column of the strip, from either face
    const int x0 = xs + NX * lx;
    const bool act = x0 < ownL && (lx > 0 || strip == 0);      // this lane finishes nodes (lane 0 of a later strip only feeds lane 1)
    const bool first_col = (x0 == 0);                   // its first column is a Dirichlet face on both sides
    const bool lastx = RG && G.extra != 0 && lx == LW - 1 && strip == (int)nstrip - 1;
    const int n0 = chunk * G.R, n1 = min(n0 + G.R, ny);
    const int jbeg = max(n0 - 1, 0);
    const int jend = min(n1 - 1, ny - 2);               // last element row of this unit (inclusive)

    // ---- shared memory of this unit: the ring and (RG) one row on its way out.  A row: pairs of columns 4l, 4l + 1 at 4l, of
    // columns 4l + 2, 4l + 3 at H1 + 4l (conflict-free 128-bit reads), the pair right of the last lane's columns at 4 LW.
    const int RS = G.RS;
    float* ring = smem + (size_t)(warp * SUBS + sub) * (P2_DEPTH * RS + ((RG && !EO) ? 2 * NX * LW : 0));
    float* obuf = ring + P2_DEPTH * RS;
    const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
    const int H1 = 4 * LW + 4, UROW = 2 * H1;
    const int COEF = ND ? 2 * UROW : UROW;              // the coefficient row (ND: none; the nu row sits at UROW)

    const int bn = b / P.rep;                           // whose diffusivity this is
    const float* ub = P.u + (size_t)b * P.nodes;
    float* rb = EO ? nullptr : P.r + (size_t)b * P.nodes;
    const bool impose = (P.flags & DN_IMPOSE_BC_ON_LOAD) != 0;
    const bool nomask = (P.flags & DN_NO_MASK) != 0;
    float bc0 = P.bc_x0, bc1 = P.bc_x1;
    if (impose) {
        if (P.bc0_b) bc0 = __ldg(P.bc0_b + b);
        if (P.bc1_b) bc1 = __ldg(P.bc1_b + b);
    }
    const f2 bcp = mk2(bc0, bc1);
    const float kx = 0.25f * P.hy / P.hx, ky = 0.25f * P.hx / P.hy;
    const f2 rho = dup2(ky / kx);                       // the march works in units of ku; y forces enter times rho
    const float ku = EO ? kx : kx * (KG ? 1.f / 6.f : 1.f / 3.f);
    const float fw = P.f_const * P.hx * P.hy;           // nodal load of an interior node
    const bool hasf = (P.f_const != 0.f);
    const float gs = P.gJ ? __ldg(P.gJ + b) : 1.f;
    // Lane constants that make the march branch-free: lm = 0 in lane 0 (nothing arrives from the left); output scale, nodal
    // load and load-energy weight of the lane's first column (lane 0 of the first strip: the Dirichlet faces, masked to
    // zero, or with DN_NO_MASK carrying half the nodal load)
    const f2 lm = dup2((lx == 0) ? 0.f : 1.f);
    const float nl = -gs * fw, gku = gs * ku;
    const f2 gk2 = dup2(gku), gf2 = dup2((first_col && !nomask) ? 0.f : gku);
    const float nlf = first_col ? (nomask ? 0.5f * nl : 0.f) : nl;
    const f2 wf = dup2(first_col ? 0.5f : 1.f);
    const int kL = ownL - x0, kR = ownR - x0;           // RG: columns of this lane below kL / kR are its own
    auto owned = [&](const int k, const f2 v) {         // v at column k, zero where the node belongs to the other side
        if constexpr (!RG) return v;
        float l, h;
        un2(v, l, h);
        return mk2(k < kL ? l : 0.f, k < kR ? h : 0.f);
    };
    f2 em[EO ? NX : 1];                                 // EO: the elements this lane counts
    if constexpr (EO) {
#pragma unroll
        for (int k = 0; k < NX; ++k) em[k] = mk2(act && x0 + k < nx / 2 ? 1.f : 0.f, act && x0 + k < (nx - 1) / 2 ? 1.f : 0.f);
    }

    // cos(pi x) and its square at the two Gauss columns of each element, duplicated into both halves (KG); (c, -c) at the nodes (KN)
    f2 ca[KG ? NX : 1], cb[KG ? NX : 1], ca2[KG ? NX : 1], cb2[KG ? NX : 1], cn[KN ? NX + 1 : 1];
    if constexpr (KG) {
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const int xe = min(x0 + k, nx - 2);         // element index = index of its left node
            const float va = __ldg(P.cg[0] + 2 * xe), vb = __ldg(P.cg[0] + 2 * xe + 1);
            ca[k] = dup2(va); cb[k] = dup2(vb); ca2[k] = dup2(va * va); cb2[k] = dup2(vb * vb);
        }
    }
    if constexpr (KN) {
#pragma unroll
        for (int k = 0; k <= NX; ++k) {
            const float c = __ldg(P.cn[0] + min(x0 + k, nx - 1));
            cn[k] = mk2(c, -c);
        }
    }

    // ---- the ring: step i = j - jbeg uses slot i % DEPTH, which holds node row j + 1 of u (and nu) and the coefficients of
    // element row j (KG) or of node row j + 1 (KN)
    int fetch = jbeg;                                   // next element row to fetch
    unsigned pfo = 0;                                   // byte offset of the slot it goes to
    const unsigned RSB = 4u * RS, RINGB = P2_DEPTH * RSB;
    const int w0 = xs + lx;                             // this lane copies columns w0, w0 + LW, ... of both sides
    const bool tiny = xs + NX * LW >= nx;               // the strip reaches beyond the far face: columns there repeat it
    const size_t row1 = (size_t)(jbeg + 1) * nx;
    const float* usrc = ub + row1;
    const float* nsrc = ND ? P.nu + (size_t)bn * P.nodes + row1 : nullptr;
    const float* polyb = rowpoly + (size_t)bn * (KN ? ny : ny - 1) * GS;
    const int clx = (lx < CFQ) ? lx : 0;
    const float* csrc = polyb + (size_t)(KN ? jbeg + 1 : jbeg) * GS + 4 * clx;
    const unsigned dw = ring_s + 4u * ((lx >> 2) * 4 + ((lx >> 1) & 1) * H1 + 2 * (lx & 1)), dc = ring_s + 4u * COEF + 16u * clx;
    auto copy_row = [&](const unsigned d, const unsigned dh, const float* src) {
        if (!tiny) {
            const float *l = src + w0, *r = src + (nx - 1 - w0);
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                cp4(d + 4u * LW * i, l + LW * i);
                cp4(d + 4u * LW * i + 4u, r - LW * i);
            }
            cp4_if(dh + 4u * lx, (lx & 1) ? src + (nx - 1 - xs - NX * LW) : src + xs + NX * LW, (lx < 2) ? 1 : 0);
        } else {
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                const int w = min(w0 + LW * i, nx - 1);
                cp4(d + 4u * LW * i, src + w);
                cp4(d + 4u * LW * i + 4u, src + (nx - 1 - w));
            }
            const int w = min(xs + NX * LW, nx - 1);
            cp4_if(dh + 4u * lx, src + ((lx & 1) ? nx - 1 - w : w), (lx < 2) ? 1 : 0);
        }
    };
    auto issue = [&]() {
        if (fetch <= jend) {                            // uniform in the unit
            const unsigned dh = ring_s + 16u * LW + pfo;
            copy_row(dw + pfo, dh, usrc);
            if constexpr (ND) copy_row(dw + 4u * UROW + pfo, dh + 4u * UROW, nsrc);
            else cp16_if(dc + pfo, csrc, (lx < CFQ) ? 1 : 0);           // (8 lanes at least, 5 pieces at most)
        }
        cp_commit();                                    // one group per step, possibly empty
        ++fetch; usrc += nx; csrc += GS;
        if constexpr (ND) nsrc += nx;
        pfo += RSB;
        if (pfo == RINGB) pfo = 0;
    };
#pragma unroll
    for (int d = 0; d < P2_DEPTH - 1; ++d) issue();

    auto col = [&](const float* row, const int w) { const int c = min(w, nx - 1); return mk2(__ldg(row + c), __ldg(row + (nx - 1 - c))); };
    auto ldslot = [&](const float* slot, f2 (&v)[NX + 1]) {
        const ulonglong2 q0 = *reinterpret_cast<const ulonglong2*>(slot + 4 * lx);
        const ulonglong2 q1 = *reinterpret_cast<const ulonglong2*>(slot + H1 + 4 * lx);
        v[0].v = q0.x; v[1].v = q0.y; v[2].v = q1.x; v[3].v = q1.y;
        v[NX].v = *reinterpret_cast<const u64*>(slot + 4 * (lx + 1));
    };
    auto impose_on = [&](f2 (&v)[NX + 1]) {
        if (first_col) v[0] = bcp;
        if constexpr (RG || EO) {                       // a far face within reach: rows of at most 3 nodes need it
#pragma unroll
            for (int k = 0; k <= NX; ++k) if (x0 + k == nx - 1) v[k] = mk2(bc1, bc0);
        }
    };

    // ---- state of the node row below the current element row
    f2 lo[NX + 1], cu[NX + 1], eh[NX], H[EO ? 1 : NX], Gv[EO ? 1 : NX];     // H: minus the pending force of the row's edges along x
    float gx = 0.f;                                     // the middle node without a lane: its Gv
#pragma unroll
    for (int k = 0; k <= NX; ++k) lo[k] = col(ub + (size_t)jbeg * nx, x0 + k);
    if (impose) impose_on(lo);
#pragma unroll
    for (int k = 0; k < NX; ++k) {
        eh[k] = lo[k + 1] - lo[k];
        if constexpr (!EO) { H[k] = dup2(0.f); Gv[k] = dup2(0.f); }
    }

    // KN: nu at this lane's columns and at the ones right of them, from the polynomial of that node row
    auto nu_row = [&](const f2 (&gg)[GS / 2], f2 (&nn)[NX + 1]) {
#pragma unroll
        for (int k = 0; k <= NX; ++k) {
            f2 e = gg[M];
#pragma unroll
            for (int i = M - 1; i >= 0; --i) e = fma2(e, cn[KN ? k : 0], gg[i]);
            float e0, e1;
            un2(e, e0, e1);
            nn[k] = mk2(ex2f(e0), ex2f(e1));
        }
    };
    f2 nlo[NX + 1], hnu[NX];                            // KN, ND: nu on the node row below and its sums over x-neighbours
    if constexpr (ND) {
#pragma unroll
        for (int k = 0; k <= NX; ++k) nlo[k] = col(P.nu + (size_t)bn * P.nodes + (size_t)jbeg * nx, x0 + k);
    }
    if constexpr (KN) {
        f2 gg[GS / 2];
        const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(polyb + (size_t)jbeg * GS);
#pragma unroll
        for (int k = 0; k < GS / 4; ++k) { const ulonglong2 t = __ldg(gp + k); gg[2 * k].v = t.x; gg[2 * k + 1].v = t.y; }
        nu_row(gg, nlo);
    }
    if constexpr (KN || ND) {
#pragma unroll
        for (int k = 0; k < NX; ++k) hnu[k] = nlo[k] + nlo[k + 1];
    }
    f2 en = dup2(0.f);                                  // sum u (K u) of the rows this lane went over
    float ell = 0.f;                                    // sum w u
    float* rrow = EO ? nullptr : rb + (size_t)jbeg * nx;
    unsigned rdo = 0;                                   // byte offset of the slot to read

    auto store_row = [&](float* row, const f2 (&o)[NX]) {
        if constexpr (RG) {
            __syncwarp(submask);                        // the row before it has left the buffer
            ulonglong2 q0, q1;
            q0.x = o[0].v; q0.y = o[1].v; q1.x = o[2].v; q1.y = o[3].v;
            *reinterpret_cast<ulonglong2*>(obuf + 4 * lx) = q0;
            *reinterpret_cast<ulonglong2*>(obuf + 4 * LW + 4 * lx) = q1;
            __syncwarp(submask);
            const float* src = obuf + (lx >> 2) * 4 + ((lx >> 1) & 1) * 4 * LW + 2 * (lx & 1);
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                const int w = w0 + LW * i;
                const bool mine = i > 0 || strip == 0 || lx >= NX;       // lane 0 of a later strip only feeds lane 1
                f2 t;
                t.v = *reinterpret_cast<const u64*>(src + LW * i);
                if (mine && w < ownL) row[w] = lo2(t);
                if (mine && w < ownR) row[nx - 1 - w] = hi2(t);
            }
        } else if (act) {
            float l[NX], r[NX];
#pragma unroll
            for (int k = 0; k < NX; ++k) un2(o[k], l[k], r[k]);
            *reinterpret_cast<float4*>(row + x0) = make_float4(l[0], l[1], l[2], l[3]);
            *reinterpret_cast<float4*>(row + nx - NX - x0) = make_float4(r[3], r[2], r[1], r[0]);
        }
    };
    auto load_energy = [&](const f2 (&a)[NX + 1], const float wrow) {
        f2 w = wf * owned(0, a[0]);
#pragma unroll
        for (int k = 1; k < NX; ++k) w = w + owned(k, a[k]);
        float l, h;
        un2(w, l, h);
        l += h;
        if (RG && lastx) l += lo2(a[NX]);
        ell = fmaf(wrow, l, ell);
    };

    // One element row: a holds node row j, c receives node row j + 1.
    auto step = [&](f2 (&a)[NX + 1], f2 (&c)[NX + 1], const int j) {
        cp_wait<P2_DEPTH - 2>();                        // this step's slot has landed (for the lanes that copied it)
        __syncwarp(submask);                            // ... is visible to the unit, and the slot read last step is free
        issue();                                        // refill it
        const float* slot = reinterpret_cast<const float*>(reinterpret_cast<const char*>(ring) + rdo);
        rdo += RSB;
        if (rdo == RINGB) rdo = 0;
        ldslot(slot, c);
        if (impose) impose_on(c);
        f2 g2[GS / 2];
        if constexpr (!ND) {
            const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(slot + COEF);
#pragma unroll
            for (int k = 0; k < GS / 4; ++k) { const ulonglong2 t = gp[k]; g2[2 * k].v = t.x; g2[2 * k + 1].v = t.y; }
        }
        f2 ncur[NX + 1];
        if constexpr (KN) nu_row(g2, ncur);
        if constexpr (ND) ldslot(slot + UROW, ncur);

        f2 Fp, gn, F0, g0, sk = c[0] - a[0], raw[NX];   // gn: minus the force of the element's right edge
        f2 es = dup2(0.f);                              // EO: sum over this lane's elements of N D^2
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const f2 e1 = c[k + 1] - c[k], s1 = c[k + 1] - a[k + 1], e0 = eh[k];
            eh[k] = e1;
            const f2 t = e1 - e0;
            f2 Px, Qx, Py, Qy, bt;                      // Qx, Qy with the opposite sign (not EO)
            if constexpr (KN || ND) {
                // Q1 interpolation of nu to the Gauss points leaves sums over corners: with the sums h0, h1 over the bottom
                // and top edge and v0, v1 over the left and right one, 3 P = S + h0, 3 Q = S + h1, 3 B = S / 2 (same in y)
                const f2 h0 = hnu[k], h1 = ncur[k] + ncur[k + 1];
                hnu[k] = h1;
                const f2 v0 = nlo[k] + ncur[k], v1 = nlo[k + 1] + ncur[k + 1];
                if constexpr (EO) {
                    const f2 dh = h1 - h0, dv = v1 - v0;
                    Px = fma2(dup2(DN_GA), dh, h0); Qx = fma2(dup2(DN_GB), dh, h0);
                    Py = fma2(dup2(DN_GA), dv, v0); Qy = fma2(dup2(DN_GB), dv, v0);
                    bt = t;
                } else {
                    const f2 S = h0 + h1, Sn = neg2(S);
                    Px = S + h0; Qx = Sn - h1; Py = S + v0; Qy = Sn - v1;
                    bt = (dup2(0.5f) * S) * t;
                }
            } else {
                f2 xl[2], xr[2];                        // (row a, row b) exponents at the two Gauss columns, left and mirrored
                exponents<M>(g2, ca[k], ca2[k], xl[0], xr[0]);
                exponents<M>(g2, cb[k], cb2[k], xl[1], xr[1]);
                f2 n[2][2];                             // nu at (column p, row q)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float la, lb, ra, rbv;
                    un2(xl[p], la, lb); un2(xr[p], ra, rbv);
                    n[p][0] = mk2(ex2f(la), ex2f(ra)); n[p][1] = mk2(ex2f(lb), ex2f(rbv));
                }
                const f2 Na = n[0][0] + n[1][0], Nb = n[0][1] + n[1][1], Ma = n[0][0] + n[0][1];
                if constexpr (EO) {
                    Px = Na; Qx = Nb; Py = Ma; Qy = n[1][0] + n[1][1]; bt = t;
                } else {
                    const f2 S = Na + Nb, aS = dup2(6.f * DN_GA) * S;
                    Px = fma2(dup2(6.f * (DN_GB - DN_GA)), Na, aS); Qx = fma2(dup2(-6.f), S, Px);
                    Py = fma2(dup2(6.f * (DN_GB - DN_GA)), Ma, aS); Qy = fma2(dup2(-6.f), S, Py);
                    bt = S * t;
                }
            }
            if constexpr (EO) {                         // P, Q hold the sums of nu on the Gauss rows / columns here
                const f2 Dxa = fma2(dup2(DN_GA), t, e0), Dxb = fma2(dup2(DN_GB), t, e0);
                const f2 Dya = fma2(dup2(DN_GA), t, sk), Dyb = fma2(dup2(DN_GB), t, sk);
                const f2 ex = fma2(Px * Dxa, Dxa, (Qx * Dxb) * Dxb), ey = fma2(Py * Dya, Dya, (Qy * Dyb) * Dyb);
                es = fma2(em[EO ? k : 0], fma2(rho, ey, ex), es);
            } else {
                const f2 Fx = fma2(Px, e0, bt - H[k]);              // the bottom edge is complete
                H[k] = fma2(Qx, e1, bt);                            // the top edge waits for the element above
                const f2 g = fma2(Py, sk, bt);
                if (k == 0) {
                    F0 = Fx; g0 = g;
                } else {
                    const f2 Gk = g - gn;
                    raw[k] = fma2(rho, Gv[k] - Gk, Fp - Fx);
                    Gv[k] = Gk;
                }
                gn = fma2(Qy, s1, bt);
                Fp = Fx;
            }
            sk = s1;
        }
        float rawx = 0.f;
        if constexpr (!EO) {
            // forces of the element left of this lane's first column
            f2 fl, gl;
            fl.v = __shfl_up_sync(submask, Fp.v, 1, LW);
            gl.v = __shfl_up_sync(submask, gn.v, 1, LW);
            const f2 Gk = fma2(neg2(gl), lm, g0);
            raw[0] = fma2(rho, Gv[0] - Gk, fma2(fl, lm, neg2(F0)));
            Gv[0] = Gk;
            if (RG && lastx) {                          // the middle node: its two elements of this row are the last of either side
                float l, h;
                un2(gn, l, h);
                const float G1 = -(l + h);
                un2(Fp, l, h);
                rawx = fmaf(lo2(rho), gx - G1, l + h);
                gx = G1;
            }
        }
        if (j >= n0) {                                  // uniform: this unit owns node row j
            const float wrow = (j == 0) ? 0.5f : 1.f;
            if (hasf) load_energy(a, wrow);
            if constexpr (EO) {
                en = en + es;                           // element row j belongs to the chunk that owns node row j
            } else {
                f2 o[NX];
#pragma unroll
                for (int k = 0; k < NX; ++k) {
                    en = fma2(owned(k, a[k]), raw[k], en);           // Euler's identity
                    o[k] = fma2(k == 0 ? gf2 : gk2, raw[k], dup2(wrow * (k == 0 ? nlf : nl)));
                }
                store_row(rrow, o);
                if (RG && lastx) {
                    en = fma2(a[NX], mk2(rawx, 0.f), en);
                    rrow[ownL - 1] = fmaf(gku, rawx, wrow * nl);
                }
            }
        }
        if constexpr (!EO) rrow += nx;
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
    cp_wait<0>();

    // ---- the top node row of the grid has no element row above it (lo holds it; its edges are complete)
    if (n1 == ny) {
        load_energy(lo, 0.5f);
        if constexpr (!EO) {
            f2 hl, raw[NX], o[NX];
            hl.v = __shfl_up_sync(submask, H[NX - 1].v, 1, LW);
            raw[0] = fma2(rho, Gv[0], H[0] - hl * lm);
#pragma unroll
            for (int k = 1; k < NX; ++k) raw[k] = fma2(rho, Gv[k], H[k] - H[k - 1]);
#pragma unroll
            for (int k = 0; k < NX; ++k) {
                en = fma2(owned(k, lo[k]), raw[k], en);
                o[k] = fma2(k == 0 ? gf2 : gk2, raw[k], dup2(0.5f * (k == 0 ? nlf : nl)));
            }
            float* row = rb + (size_t)(ny - 1) * nx;
            store_row(row, o);
            if (RG && lastx) {
                float l, h;
                un2(H[NX - 1], l, h);
                const float rawx = fmaf(lo2(rho), gx, -(l + h));
                en = fma2(lo[NX], mk2(rawx, 0.f), en);
                row[ownL - 1] = fmaf(gku, rawx, 0.5f * nl);
            }
        }
    }

    // ---- energy partial of this unit: owning lanes summed in a fixed order in double
    float el, eh2;
    un2(en, el, eh2);
    double d = act ? 0.5 * (double)ku * ((double)el + (double)eh2) : 0.0;
    double l = (act && hasf) ? (double)fw * (double)ell : 0.0;
    for (int off = LW >> 1; off > 0; off >>= 1) {
        d += __shfl_down_sync(submask, d, off, LW);
        l += __shfl_down_sync(submask, l, off, LW);
    }
    if (lx == 0) {
        double* slot = P.partials + 2 * ((size_t)b * P.nblk + (size_t)chunk * nstrip + strip);
        slot[0] = d; slot[1] = l;
    }
}

template <int M, int MODE, bool EO, int LWC, bool RG>
cudaError_t launch_p2(const Params& P, const float* rowpoly, const P2Geo& g, cudaStream_t s) {
    const int subs = 32 / g.LW;
    const size_t smem = sizeof(float) * P2_WARPS * subs * ((size_t)P2_DEPTH * g.RS + ((RG && !EO) ? 2 * NX * g.LW : 0));
    const long long per_block = (long long)P2_WARPS * subs;
    const unsigned blocks = (unsigned)((g.units + per_block - 1) / per_block);
    if (smem > 48 * 1024) {                             // what a kernel may use without asking
        const cudaError_t e = cudaFuncSetAttribute(pair2d_kernel<M, MODE, EO, LWC, RG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_dependent(pair2d_kernel<M, MODE, EO, LWC, RG>, dim3(blocks), dim3(P2_WARPS * 32), smem, s, P, rowpoly, g);
}

// whole: r can be stored 16 bytes at a time
template <int M, int MODE>
cudaError_t launch_p2_mode(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    if (P.r == nullptr) return g.LW == 32 ? launch_p2<M, MODE, true, 32, true>(P, rowpoly, g, s) : launch_p2<M, MODE, true, 0, true>(P, rowpoly, g, s);
    if (whole) {
        if (g.LW == 32) return launch_p2<M, MODE, false, 32, false>(P, rowpoly, g, s);
        if (g.LW == 16) return launch_p2<M, MODE, false, 16, false>(P, rowpoly, g, s);
        return launch_p2<M, MODE, false, 0, false>(P, rowpoly, g, s);
    }
    return g.LW == 32 ? launch_p2<M, MODE, false, 32, true>(P, rowpoly, g, s) : launch_p2<M, MODE, false, 0, true>(P, rowpoly, g, s);
}

template <int M>
cudaError_t launch_p2_m(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    return (P.nu_mode == DN_NU_KL_NODAL) ? launch_p2_mode<M, 1>(P, rowpoly, g, whole, s) : launch_p2_mode<M, 0>(P, rowpoly, g, whole, s);
}

}  // namespace

#if DN_P2_PART == 1
cudaError_t launch_pair2d_m34(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    return P.m == 3 ? launch_p2_m<3>(P, rowpoly, g, whole, s) : launch_p2_m<4>(P, rowpoly, g, whole, s);
}
#elif DN_P2_PART == 2
cudaError_t launch_pair2d_m56(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    return P.m == 5 ? launch_p2_m<5>(P, rowpoly, g, whole, s) : launch_p2_m<6>(P, rowpoly, g, whole, s);
}
#elif DN_P2_PART == 3
cudaError_t launch_pair2d_m78(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    return P.m == 7 ? launch_p2_m<7>(P, rowpoly, g, whole, s) : launch_p2_m<8>(P, rowpoly, g, whole, s);
}
#else
cudaError_t launch_pair2d_m12(const Params& P, const float* rowpoly, const P2Geo& g, bool whole, cudaStream_t s) {
    if (P.nu_mode == DN_NU_NODAL) return launch_p2_mode<1, 2>(P, rowpoly, g, whole, s);
    return P.m == 1 ? launch_p2_m<1>(P, rowpoly, g, whole, s) : launch_p2_m<2>(P, rowpoly, g, whole, s);
}

namespace {

P2Geo p2_search(const dn_problem& p, int sms) {
    P2Geo g{};
    const int nx = p.grid.nx, ny = p.grid.ny, side = (nx + 1) / 2, left = nx & 1;
    g.LW = 8; g.lwsh = 3;
    while (g.LW < 32 && g.LW * NX + left < side) { g.LW *= 2; ++g.lwsh; }
    const int cols = g.LW * NX, stride = cols - NX;
    g.nstrip = (side <= cols + left) ? 1 : (side - left - cols + stride - 1) / stride + 1;
    g.extra = (left && side == cols + (g.nstrip - 1) * stride + 1) ? 1 : 0;
    const int urow = 2 * (4 * g.LW + 4);
    g.RS = (p.nu_mode == DN_NU_NODAL) ? 2 * urow : urow + p2_gs(p.kl_modes);
    const long long slots = (long long)sms * P2_MINB * P2_WARPS * (32 / g.LW);
    // R from a cost search over whole waves of units; a unit pays the recomputed row and the filling of its ring
    long long best = -1;
    int bestR = 2;
    for (int R = 2; R <= 1024; ++R) {
        if (R > ny && R > 2) break;
        const long long nch = (ny + R - 1) / R;
        const long long units = (long long)p.batch * g.nstrip * nch;
        const long long waves = (units + slots - 1) / slots;
        const long long cost = waves * (R + 5) * 1000 + (1000 / R);      // prefer less redundancy on ties
        if (best < 0 || cost < best) { best = cost; bestR = R; }
    }
    g.R = bestR;
    g.nchunk = (ny + g.R - 1) / g.R;
    g.units = (long long)p.batch * g.nstrip * g.nchunk;
    return g;
}

P2Geo p2_geometry(const dn_problem& p) {
    const int sms = sm_count();
    return memo_geometry<P2Geo>(p, sms, [&]() { return p2_search(p, sms); });
}

}  // namespace

Launch pair2d_geometry(const dn_problem& p) {
    const P2Geo g = p2_geometry(p);
    Launch l{};
    l.path = PATH_PAIR2D;
    l.nblk = g.nchunk * g.nstrip;
    l.chunk = g.R;
    l.variant = g.nstrip;
    return l;
}

cudaError_t launch_pair2d(const Params& P, const float* rowpoly, cudaStream_t s) {
    dn_problem p{};
    p.grid.dim = 2; p.grid.nx = P.nx; p.grid.ny = P.ny; p.grid.nz = 1; p.batch = P.batch;
    p.nu_mode = P.nu_mode; p.kl_modes = P.m; p.flags = P.flags;
    const P2Geo g = p2_geometry(p);
    const bool whole = P.nx % 8 == 0 && (reinterpret_cast<uintptr_t>(P.r) & 15u) == 0;
    if (P.nu_mode == DN_NU_NODAL || P.m <= 2) return launch_pair2d_m12(P, rowpoly, g, whole, s);
    if (P.m <= 4) return launch_pair2d_m34(P, rowpoly, g, whole, s);
    if (P.m <= 6) return launch_pair2d_m56(P, rowpoly, g, whole, s);
    return launch_pair2d_m78(P, rowpoly, g, whole, s);
}
#endif  // DN_P2_PART

}  // namespace dn
