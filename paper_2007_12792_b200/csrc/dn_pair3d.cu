// Mirrored-pair kernel for 3D grids whose rows fit one warp (nx <= 257): fused element quadrature, energy reduction,
// node gather, mask and store on hexahedra, without any barrier between warps; rows of any length and any alignment.
//
// Mirrored pairs.  Column w counted from the left face and column w counted from the right face go through the same
// arithmetic: the element, the Gauss rule, the Dirichlet faces and the gather are symmetric under x -> 1 - x, and
// cos(pi x) only changes sign.  So a lane owns 4 consecutive columns w and handles the node (or element) at w from the
// left together with the one at w from the right as the two halves of packed f32x2 registers: every operation of the
// march is a two-wide add / sub / mul / fma.  A packed FMA occupies the FP32 pipe for two cycles but takes one issue slot
// (measured: 2.03 cycles each, the latency of a scalar one), which leaves half the slots to loads, moves and exponentials.
// The scalar kernel before it was bound by issue (72 % of the cycles) at 53 % of the FP32 rate.  With an even number of nodes
// both sides also compute the middle element (each side uses its own corners); with an odd one the middle node belongs to the
// left side.
//
// Layout of the work.  A work unit is one sample, one tile of Ry element rows (y) across the whole x extent, one chunk of
// Z element planes (z).  A unit belongs to LW = 4, 8, 16 or 32 lanes of one warp (8 LW >= nx, or nx = 8 LW + 1: then the
// middle node has no lane and the last lane finishes it); a warp with LW < 32 carries 32 / LW units that have nothing to
// do with one another.  A unit marches over its element planes from bottom to top, and inside a plane over its element
// rows.  The node rows stream through a ring of rows in shared memory that belongs to the unit alone, already interleaved
// into pairs (4-byte asynchronous copies: coalesced for every row offset, any destination): row (plane k, row j) of the
// tile is entry k * T + j of a linear sequence (T node rows per plane), entry n lives in slot n mod C, and the ring holds
// the two planes being worked on plus D rows in flight.  Every node is read from global memory once per unit.
//
// Element (x, j, k) is computed once per side, by the lane that owns node x.  Of its 8 corner contributions those to
// column w + 1 pass to the next element of the lane (to the next lane by shuffle), those to row j + 1 are kept until the
// next row of the same plane, and those to plane k + 1 are parked
// (every lane its own words, no synchronisation): one plane later they are read back, completed and stored to r once.
// They are parked in shared memory where a slot of the ring is one row; with two or three rows in a slot (nodal modes,
// nodal forcing) that would leave room for tiles of 3 or 4 rows only, and they go to a scratch array, in L2 all the time.
//
// Tiles do not overlap in y: the top element row of a tile leaves what it contributes to the first node row of the next
// tile in a scratch array (seam, [B][ntile-1][nz][nx]), and a small fix-up kernel adds those rows to r afterwards.
// Chunks do not overlap in z either: what the last element plane of a chunk contributes to the first node plane of
// the next chunk goes to a second scratch array (zseam, [B][nchunk-1][ny][nx], plus [B][nchunk-1][ntile-1][nx] for the
// nodes that are on a tile seam as well), added by the same fix-up kernel.  No atomics; every sum has a fixed order.
//
// Arithmetic of one element: hierarchical coordinates of the trilinear field (edge differences e, s, w at the low
// corner, second differences txy, txz, tyz, third difference txyz), derivatives at the 4 Gauss lines of each direction,
// sums of nu along each derivative's own axis, the adjoint of the interpolation and the chain rule to the 8 corners.  The
// diffusion energy is taken from the residual by Euler's identity for quadratic forms: 1/2 sum over (node, contribution)
// pairs of u_node times contribution, each pair counted by the unit that computes it.
//
// KL diffusivity at the Gauss points: along a Gauss line (y_q, z_s fixed) the exponent is a polynomial of degree m in
// c = cos(pi x), E(c^2) + c O(c^2) at the left and E(c^2) - c O(c^2) at the mirrored point: m + 1 packed operations for
// two planes and both sides where two Horner chains take 2 m.  A table kernel prepares the coefficients of all four
// lines of every element row of every element plane once per call in double ([B][nz-1][ny-1][2][GS] floats: Gauss row q, then
// coefficient i and Gauss plane s interleaved); they travel through the ring with the node row that completes
// the element row.
//
// What bounds it: two warps per scheduler (244 to 255 registers) do not keep the FP32 pipe full.  256^3 x 4, m = 3: 107
// instructions and 125 FP32 lane operations per element (167 and 134 in the scalar kernel it replaces), the pipe busy in 61 %
// of the cycles, an instruction issued in 50 %, DRAM at 16 %: 428 us with the seams (459 before; 224 at the full FP32 rate).  Rows of
// any length: 129^3 x 8 with a stored field 3339 -> 172 us, which one thread per node served.
#include "dn_internal.cuh"

namespace dn {

namespace {

constexpr int P3_WARPS = 4;                       // warps per block (each warp is on its own)
constexpr int P3_D = 3;                           // rows in flight beyond the two planes in use
constexpr int P3_MINB = 2;                        // resident blocks per SM: up to 255 registers
constexpr int NX = 4;                             // columns per lane and side

typedef unsigned long long u64;

// two floats: the lower one belongs to the left side, the upper one to the mirrored side
struct f2 { u64 v; };
__device__ __forceinline__ f2 mk2(float lo, float hi) { f2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ f2 dup2(float x) { return mk2(x, x); }
__device__ __forceinline__ void un2(const f2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v)); }
__device__ __forceinline__ float lo2(const f2 a) { float l, h; un2(a, l, h); return l; }
__device__ __forceinline__ float hi2(const f2 a) { float l, h; un2(a, l, h); return h; }
__device__ __forceinline__ f2 operator+(const f2 a, const f2 b) { f2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator-(const f2 a, const f2 b) { f2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 operator*(const f2 a, const f2 b) { f2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ f2 fma2(const f2 a, const f2 b, const f2 c) { f2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r; }
__device__ __forceinline__ f2 neg2(const f2 a) { f2 r; r.v = a.v ^ 0x8000000080000000ull; return r; }

__device__ __forceinline__ float p3_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void p3_cp4(unsigned d, const float* gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void p3_cp4_if(unsigned d, const float* gsrc, int pred) {      // predicated, no branch
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void p3_cp16_if(unsigned d, const float* gsrc, int pred) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.cg.shared.global [%0], [%1], 16;\n\t}"
                 ::"r"(d), "l"(gsrc), "r"(pred) : "memory");
}
__device__ __forceinline__ void p3_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void p3_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

}  // namespace

// The file is compiled in four parts side by side: DN_P3_PART 0 (the default) holds everything and the kernels for
// m = 1, 2 and the stored field; parts 1, 2, 3 hold the kernels for m = 3, 4; 5, 6; 7, 8.
#ifndef DN_P3_PART
#define DN_P3_PART 0
#endif

struct P3Geo {
    int Ry, Z;            // element rows per tile, element planes per chunk
    int ntile, nchunk;
    int LW, lwsh;         // lanes per unit and log2 of it
    int C, RS;            // ring slots (rows) per unit, floats per slot
    long long units;
};
cudaError_t launch_pair3d_m12(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s);
cudaError_t launch_pair3d_m34(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s);
cudaError_t launch_pair3d_m56(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s);
cudaError_t launch_pair3d_m78(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s);

namespace {

// nu at the 8 Gauss points of one element pair, index [p][q][s] -> n[4 p + 2 q + s].  g: (plane a, plane b) pairs of the
// coefficients of Gauss row q; c, cc: cos(pi x) of Gauss column p and its square, both halves the same.
template <int M>
__device__ __forceinline__ void p3_exponents(const f2 (&g)[line_floats(M) / 2], const f2 c, const f2 cc, f2& left, f2& right) {
    constexpr int ME = M / 2 * 2, MO = (M - 1) / 2 * 2 + 1;       // highest even and odd power
    f2 E = g[ME], O = g[MO];
#pragma unroll
    for (int i = ME - 2; i >= 0; i -= 2) E = fma2(E, cc, g[i]);
#pragma unroll
    for (int i = MO - 2; i >= 1; i -= 2) O = fma2(O, cc, g[i]);
    left = fma2(O, c, E);
    right = fma2(neg2(O), c, E);
}
template <int M>
__device__ __forceinline__ void p3_nu_gauss(const f2 (&ga)[line_floats(M) / 2], const f2 (&gb)[line_floats(M) / 2], const f2 (&col)[4], f2 (&n)[8]) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            f2 l, r;
            p3_exponents<M>(q ? gb : ga, col[2 * p], col[2 * p + 1], l, r);
            float la, lb, ra, rb;
            un2(l, la, lb); un2(r, ra, rb);
            n[4 * p + 2 * q] = mk2(p3_ex2(la), p3_ex2(ra));
            n[4 * p + 2 * q + 1] = mk2(p3_ex2(lb), p3_ex2(rb));
        }
    }
}

// Sums of nu along each derivative's own axis, from nu at the 8 Gauss points n[4p + 2q + s]:
// Nx[2q + s] = sum_p, Ny[2p + s] = sum_q, Nz[2p + q] = sum_s.
__device__ __forceinline__ void p3_sums_gauss(const f2 (&n)[8], f2 (&Nx)[4], f2 (&Ny)[4], f2 (&Nz)[4]) {
    Nx[0] = n[0] + n[4]; Nx[1] = n[1] + n[5]; Nx[2] = n[2] + n[6]; Nx[3] = n[3] + n[7];
    Ny[0] = n[0] + n[2]; Ny[1] = n[1] + n[3]; Ny[2] = n[4] + n[6]; Ny[3] = n[5] + n[7];
    Nz[0] = n[0] + n[1]; Nz[1] = n[2] + n[3]; Nz[2] = n[4] + n[5]; Nz[3] = n[6] + n[7];
}

// The same sums for a trilinear nu given at the corners.  Summing the interpolant over the two Gauss points of an axis
// leaves the sum of the two corner values along that axis (the weights a and b add up to 1), interpolated in the other
// two.  h00, h10, h01, h11: those edge sums at (first, second) other coordinate = low/high; out[2 i1 + i2] at the
// Gauss abscissae (i1, i2) of the two other axes.
__device__ __forceinline__ void p3_bilerp(const f2 h00, const f2 h10, const f2 h01, const f2 h11, f2 (&out)[4]) {
    const f2 A = dup2(DN_GA), Bq = dup2(DN_GB);
    const f2 d0 = h10 - h00, d1 = h11 - h01;
    const f2 ma0 = fma2(A, d0, h00), mb0 = fma2(Bq, d0, h00);     // first coordinate a / b, second low
    const f2 ma1 = fma2(A, d1, h01), mb1 = fma2(Bq, d1, h01);     // ... second high
    const f2 da = ma1 - ma0, db = mb1 - mb0;
    out[0] = fma2(A, da, ma0); out[1] = fma2(Bq, da, ma0);
    out[2] = fma2(A, db, mb0); out[3] = fma2(Bq, db, mb0);
}

// Nodal forcing: the element mass matrix applied to the 8 corner values of f, by sum factorisation (per axis the
// matrix [[2, 1], [1, 2]]; the factor hx hy hz / 216 is applied by the caller).  f and m are indexed i + 2j + 4k.
__device__ __forceinline__ void p3_mass(const f2 (&f)[8], f2 (&m)[8]) {
    const f2 two = dup2(2.f);
    f2 g[8], h[8];
#pragma unroll
    for (int t = 0; t < 8; t += 2) { g[t] = fma2(two, f[t], f[t + 1]); g[t + 1] = fma2(two, f[t + 1], f[t]); }          // x
#pragma unroll
    for (int t = 0; t < 8; ++t) { if (t & 2) continue; h[t] = fma2(two, g[t], g[t + 2]); h[t + 2] = fma2(two, g[t + 2], g[t]); }   // y
#pragma unroll
    for (int t = 0; t < 4; ++t) { m[t] = fma2(two, h[t], h[t + 4]); m[t + 4] = fma2(two, h[t + 4], h[t]); }               // z
}

// The element pair: from the 12 sums of nu and the 7 hierarchical coordinates of u to the 8 corner contributions
// r[i + 2j + 4k] (i, j, k the x, y, z bits of the corner), all in units of kap = hx hy hz / (8 h^2) on cubic cells (ISO),
// else scaled by kx, ky, kz here.
template <bool ISO>
__device__ __forceinline__ void p3_element(f2 (&Nx)[4], f2 (&Ny)[4], f2 (&Nz)[4], const f2 e0, const f2 s0, const f2 w0,
                                           const f2 txy, const f2 txz, const f2 tyz, const f2 txyz,
                                           const float kx, const float ky, const float kz, f2 (&r)[8]) {
    const f2 a = dup2(DN_GA), bq = dup2(DN_GB);
    if constexpr (!ISO) {
#pragma unroll
        for (int i = 0; i < 4; ++i) { Nx[i] = Nx[i] * dup2(kx); Ny[i] = Ny[i] * dup2(ky); Nz[i] = Nz[i] * dup2(kz); }
    }
    // derivatives at the Gauss lines: d/dx at (eta q, zeta s) = (e + q txy) + s (txz + q txyz), and cyclically
    const f2 Axa = fma2(a, txy, e0), Axb = fma2(bq, txy, e0);
    const f2 Bxa = fma2(a, txyz, txz), Bxb = fma2(bq, txyz, txz);
    const f2 Gx_aa = Nx[0] * fma2(a, Bxa, Axa), Gx_ab = Nx[1] * fma2(bq, Bxa, Axa);        // (q, s)
    const f2 Gx_ba = Nx[2] * fma2(a, Bxb, Axb), Gx_bb = Nx[3] * fma2(bq, Bxb, Axb);
    const f2 Aya = fma2(a, txy, s0), Ayb = fma2(bq, txy, s0);
    const f2 Bya = fma2(a, txyz, tyz), Byb = fma2(bq, txyz, tyz);
    const f2 Gy_aa = Ny[0] * fma2(a, Bya, Aya), Gy_ab = Ny[1] * fma2(bq, Bya, Aya);        // (p, s)
    const f2 Gy_ba = Ny[2] * fma2(a, Byb, Ayb), Gy_bb = Ny[3] * fma2(bq, Byb, Ayb);
    const f2 Aza = fma2(a, txz, w0), Azb = fma2(bq, txz, w0);
    const f2 Gz_aa = Nz[0] * fma2(a, Bya, Aza), Gz_ab = Nz[1] * fma2(bq, Bya, Aza);        // (p, q)
    const f2 Gz_ba = Nz[2] * fma2(a, Byb, Azb), Gz_bb = Nz[3] * fma2(bq, Byb, Azb);
    // Adjoint of the three interpolations: partial derivatives of the element energy.  With b = a + dl the weighted
    // sums over a 2 x 2 set of Gauss lines reduce to its total S, the sum R over the lines whose first index is b, the
    // sum C over those whose second index is b, and the (b, b) entry:
    //   sum i1 G = a S + dl R,   sum i2 G = a S + dl C,   sum i1 i2 G = a^2 S + a dl (R + C) + dl^2 G_bb.
    constexpr float dl = DN_GB - DN_GA;
    const f2 dl2 = dup2(dl);
    const f2 R1x = Gx_ba + Gx_bb, Cx = Gx_ab + Gx_bb, dE = (Gx_aa + Gx_ab) + R1x;
    const f2 R1y = Gy_ba + Gy_bb, Cy = Gy_ab + Gy_bb, dS = (Gy_aa + Gy_ab) + R1y;
    const f2 R1z = Gz_ba + Gz_bb, Cz = Gz_ab + Gz_bb, dW = (Gz_aa + Gz_ab) + R1z;
    const f2 Sxy = dE + dS, Sxz = dE + dW, Syz = dS + dW;
    const f2 P1 = R1x + R1y, P2 = Cx + R1z, P3 = Cy + Cz;
    const f2 dXY = fma2(dl2, P1, a * Sxy);             // txy enters d/dx through q and d/dy through p
    const f2 dXZ = fma2(dl2, P2, a * Sxz);             // txz enters d/dx through s and d/dz through p
    const f2 dYZ = fma2(dl2, P3, a * Syz);             // tyz enters d/dy through s and d/dz through q
    const f2 dXYZ = fma2(dup2(dl * dl), (Gx_bb + Gy_bb) + Gz_bb,
                         fma2(dup2(DN_GA * dl), (P1 + P2) + P3, dup2(DN_GA * DN_GA) * (Sxy + dW)));
    // chain rule to the corners
    const f2 r110 = dXY - dXYZ, r101 = dXZ - dXYZ, r011 = dYZ - dXYZ;
    r[0] = ((r011 - dW) + (dXY - dE)) + (dXZ - dS);
    r[1] = (dE - r110) - dXZ; r[2] = (dS - r110) - dYZ; r[4] = (dW - r101) - dYZ;
    r[3] = r110; r[5] = r101; r[6] = r011; r[7] = dXYZ;
}

// The element pair's diffusion energy, twice over and in the same units: sum over the 12 Gauss lines of N D^2 (the
// derivatives as in p3_element; the residual it returns is the gradient of half this sum).
__device__ __forceinline__ f2 p3_energy(const f2 (&Nx)[4], const f2 (&Ny)[4], const f2 (&Nz)[4], const f2 e0, const f2 s0, const f2 w0,
                                        const f2 txy, const f2 txz, const f2 tyz, const f2 txyz,
                                        const float kx, const float ky, const float kz) {
    const f2 a = dup2(DN_GA), bq = dup2(DN_GB);
    auto quad = [&](const f2 A0, const f2 A1, const f2 B0, const f2 B1, const f2 (&N)[4]) {
        const f2 D0 = fma2(a, B0, A0), D1 = fma2(bq, B0, A0), D2 = fma2(a, B1, A1), D3 = fma2(bq, B1, A1);
        return fma2(N[0] * D0, D0, (N[1] * D1) * D1) + fma2(N[2] * D2, D2, (N[3] * D3) * D3);
    };
    const f2 Bxa = fma2(a, txyz, txz), Bxb = fma2(bq, txyz, txz), Bya = fma2(a, txyz, tyz), Byb = fma2(bq, txyz, tyz);
    const f2 ex = quad(fma2(a, txy, e0), fma2(bq, txy, e0), Bxa, Bxb, Nx);
    const f2 ey = quad(fma2(a, txy, s0), fma2(bq, txy, s0), Bya, Byb, Ny);
    const f2 ez = quad(fma2(a, txz, w0), fma2(bq, txz, w0), Bya, Byb, Nz);
    return fma2(dup2(kx), ex, fma2(dup2(ky), ey, dup2(kz) * ez));
}

// MODE 0: KL at the Gauss points; 1 (KN): KL at the nodes, then Q1 interpolation; 2 (ND): stored nodal field.
// In the nodal modes a slot of the ring holds the nu row next to the u row: copied from the field (ND), or computed
// from the polynomial of that node line when the row is first used (KN: the table then holds one polynomial per node
// line, every coefficient twice, and travels with the row itself).
// NF: nodal forcing.  The f row sits in the slot as well; the load is taken element by element (mass matrix applied
// to the corner values of f) and joins the corner contributions before they are gathered, so it needs no other
// treatment at the boundary of the domain, a tile or a chunk than the stiffness part.
// EO: energy only.  The same march over the same units, but every element adds its own energy (p3_energy) and
// nothing is gathered, parked or stored: no residual, no seams.
// LWC: lanes per unit at compile time (32, 16 or 8), or 0: taken from G.
// ISO: the cells are cubes.
// RG: rows that are not a multiple of 8 or an r that is not 16-byte aligned: finished rows pass through one row of shared
// memory and are stored word by word; nodes that belong to the other side are left out.
template <int M, int MODE, bool NF, bool EO, int LWC, bool ISO, bool RG>
__global__ void __launch_bounds__(P3_WARPS * 32, P3_MINB)
pair3d_kernel(const Params P, const float* __restrict__ linepoly, const P3Geo G) {
    extern __shared__ __align__(16) float smem[];
    dep_wait();                                         // the tables of this call are complete
    dep_release();                                      // the fix-up kernel may move in as units finish
    constexpr bool KG = (MODE == 0), KN = (MODE == 1), ND = (MODE == 2);
    constexpr int GS = line_floats(M);
    constexpr int CF = KG ? 2 * GS : KN ? GS : 0;       // coefficient floats per slot (KG: Gauss rows q = a, b of an element row)
    constexpr int CFQ = CF / 4;                         // ... in 16-byte pieces
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int LW = LWC ? LWC : G.LW, lwsh = (LWC == 32) ? 5 : (LWC == 16) ? 4 : (LWC == 8) ? 3 : G.lwsh, SUBS = 32 >> lwsh;
    const int sub = lane >> lwsh, lx = lane & (LW - 1);
    const unsigned submask = (LW == 32) ? 0xffffffffu : (((1u << LW) - 1u) << (sub * LW));
    const int nx = P.nx, ny = P.ny, nz = P.nz;
    const int x0 = NX * lx;                             // this lane's first column, from either face
    const int ownL = (nx + 1) / 2, ownR = nx / 2;       // columns of the left and of the mirrored side
    const bool act = x0 < ownL;                         // this lane finishes nodes
    const bool first_col = (x0 == 0);                   // its first column is a Dirichlet face on both sides
    const bool extra = RG && nx == 2 * NX * LW + 1;     // the middle node is the one right of the last lane's columns
    const bool lastx = extra && lx == LW - 1;

    // ---- shared by the block: cos(pi x) at the two Gauss columns of each element of a lane and its square, duplicated
    // into both halves of a pair: float4 (c, c, c^2, c^2) at [element c][column][lane of the unit]
    float4* cps = reinterpret_cast<float4*>(smem);
    if constexpr (KG) {
        for (int i = threadIdx.x; i < 2 * NX * LW; i += blockDim.x) {
            const int l = i & (LW - 1), t = i >> lwsh;
            const int xe = min(NX * l + (t >> 1), nx - 2);      // element index = index of its left node
            const float c = __ldg(P.cg[0] + 2 * xe + (t & 1));
            cps[i] = make_float4(c, c, c * c, c * c);
        }
        __syncthreads();                                // the only block-wide barrier: before the march starts
    }
    const float4* cpl = cps + lx;
    f2 cnp[NX + 1];                                     // KN: cos(pi x) at this lane's nodes and at the one right of them
    if constexpr (KN) {
#pragma unroll
        for (int k = 0; k <= NX; ++k) {
            const float c = __ldg(P.cn[0] + min(x0 + k, nx - 1));
            cnp[k] = mk2(c, -c);
        }
    }

    const long long su = ((long long)blockIdx.x * P3_WARPS + warp) * SUBS + sub;
    if (su >= G.units) return;                          // the other units of the warp synchronise among themselves only
    const int C = G.C, RS = G.RS;
    const unsigned RSB = (unsigned)RS * 4u, RINGB = (unsigned)C * RSB;
    constexpr bool GP = !KG || NF;                      // parked in global memory
    const int PR = 2 * NX * LW;                         // floats of a parked row
    const int XW = (G.Ry + 6) / 4 * 4;                  // words for the middle node without a lane: 2 pending, Ry + 1 parked
    const int per_unit = C * RS + (EO ? 0 : XW + (GP ? 0 : (G.Ry + 1) * PR) + (RG ? PR : 0));
    float* ring = smem + (KG ? 8 * NX * LW : 0) + (size_t)(warp * SUBS + sub) * per_unit;
    float* xw = ring + C * RS;
    float* obuf = xw + XW;                              // RG: one finished row on its way out
    // partial sums of the upper plane, one row per node row of the tile
    float* park = GP ? P.park + (size_t)su * ((G.Ry + 1) * PR) : obuf + (RG ? PR : 0);
    const unsigned ring_s = (unsigned)__cvta_generic_to_shared(ring);
    // A row in a slot: the pair of column 4l + k at k * AS + 2l (conflict-free 64-bit reads), so that the pair right of a lane's
    // columns is the next lane's first; behind the last lane's that of column 4 LW.
    const int AS = 2 * LW + 2;
    const int UROW = NX * AS;
    const int FOFF = KG ? UROW : 2 * UROW;              // offset of the f row (nodal forcing)
    const int COEF = FOFF + (NF ? UROW : 0);            // offset of the coefficient row inside a slot

    int b, tile, chunk;
    row3d_unit(su, P.batch, (ny - 1) / G.Ry, (nz - 1) / G.Z, G.ntile, b, tile, chunk);
    const int y0 = tile * G.Ry, e1 = min(y0 + G.Ry, ny - 1);     // element rows y0 .. e1-1, node rows y0 .. e1
    const int T = e1 - y0 + 1;
    const bool lasttile = (e1 == ny - 1);               // then node row e1 = ny-1 is this tile's own, else the next tile's
    const int z0 = chunk * G.Z, ke = min(z0 + G.Z, nz - 1);
    const int kbeg = z0;                                // element planes z0 .. ke-1
    const int nplanes = ke - kbeg + 1;                  // node planes z0 .. ke
    const bool lastchunk = (ke == nz - 1);              // then node plane ke = nz-1 is this chunk's own, else the next chunk's

    const size_t plane = (size_t)nx * ny;
    float* rb = EO ? nullptr : P.r + (size_t)b * P.nodes;
    float* sb = (EO || lasttile) ? nullptr : P.seam + (((size_t)b * (G.ntile - 1) + tile) * nz) * nx;
    // where the sums of node plane ke go: r, or for a chunk below another the z seam (row y0 of it; and the entry of
    // this tile's seam row among the nodes that lie on both seams)
    float* ztop = EO ? nullptr : lastchunk ? rb + ((size_t)ke * ny + y0) * nx
                            : P.zseam + (((size_t)b * (G.nchunk - 1) + chunk) * ny + y0) * nx;
    float* zstop = (EO || lasttile) ? nullptr
                 : lastchunk ? sb + (size_t)ke * nx
                             : P.zseam + (size_t)P.batch * (G.nchunk - 1) * ny * nx
                               + (((size_t)b * (G.nchunk - 1) + chunk) * (G.ntile - 1) + tile) * nx;

    const bool impose = (P.flags & DN_IMPOSE_BC_ON_LOAD) != 0;
    const bool nomask = (P.flags & DN_NO_MASK) != 0;
    float bc0 = P.bc_x0, bc1 = P.bc_x1;
    if (impose) {
        if (P.bc0_b) bc0 = __ldg(P.bc0_b + b);
        if (P.bc1_b) bc1 = __ldg(P.bc1_b + b);
    }
    const float W8 = 0.125f * P.hx * P.hy * P.hz;
    const float kx = W8 / (P.hx * P.hx), ky = W8 / (P.hy * P.hy), kz = W8 / (P.hz * P.hz);
    const float kap = (ISO && !EO) ? kx : 1.f;          // cubic cells: one scale applied at the end
    const float gs = P.gJ ? __ldg(P.gJ + b) : 1.f;
    const float fw = NF ? 0.f : P.f_const * P.hx * P.hy * P.hz;    // nodal load of an interior node (constant forcing)
    const bool hasf = !NF && (P.f_const != 0.f);
    const float fsabs = P.hx * P.hy * P.hz * (1.f / 216.f);        // NF: scale of the element mass matrix ...
    const float fs = fsabs / kap;                                   // ... in the units the corner contributions are kept in
    // Lane constants that keep the finish of a node row branch-free: output scale, share of the nodal load and weight in
    // the load energy of the lane's first column (in lane 0 the Dirichlet faces: masked, or with DN_NO_MASK
    // carrying half a load); em: the elements it counts (energy only, nodal forcing).
    const float sc = gs * kap;
    const f2 sc2 = dup2(sc), sc02 = dup2((first_col && !nomask) ? 0.f : sc);
    const float lw0 = first_col ? (nomask ? 0.5f : 0.f) : 1.f;
    const f2 wx0 = dup2(first_col ? 0.5f : 1.f);
    const f2 lm2 = dup2((lx == 0) ? 0.f : 1.f);         // nothing arrives from the left in the first lane
    f2 em[NX];
#pragma unroll
    for (int k = 0; k < NX; ++k) em[k] = mk2(x0 + k < nx / 2 ? 1.f : 0.f, x0 + k < (nx - 1) / 2 ? 1.f : 0.f);
    const int kL = ownL - x0, kR = ownR - x0;           // RG: columns of this lane below kL / kR are its own
    auto owned = [&](const int k, const f2 u) {         // u at column k, zero where the node belongs to the other side
        if constexpr (!RG) return u;
        float l, h;
        un2(u, l, h);
        return mk2(k < kL ? l : 0.f, k < kR ? h : 0.f);
    };

    // ---- the ring.  Entry n = (plane index pk, row index pj) of the unit goes to slot n mod C: the node row (lane l copies
    // the words l, l + LW, ... of either side) and, for pk, pj >= 1, the coefficients of element row (pk-1, pj-1).
    int pf = 0, pfj = 0, pfk = 0;
    unsigned pfo = 0;                                   // byte offset of the slot the next entry goes to
    const int back = nx - 1 - 2 * lx;                   // from this lane's first word on the left to its first one on the right
    const bool tiny = nx <= NX * LW;                    // the lanes reach beyond the far face (rows of at most 16 nodes)
    const bool reach = nx <= NX * LW + 1;               // ... or the far face itself (17 nodes)
    const size_t first = (size_t)kbeg * plane + (size_t)y0 * nx + lx;
    const float* usrc = P.u + (size_t)b * P.nodes + first;
    // coefficient piece of this lane.  KG: of element row (pfk-1, pfj-1), so the pointer starts one row and one plane
    // low; KN: of the node line of the entry itself
    const int clx = (lx < CFQ) ? lx : 0;
    const float* csrc = KG ? linepoly + (((size_t)b * (nz - 1) + kbeg) * (ny - 1) + y0) * CF - ((size_t)(ny - 1) + 1) * CF + 4 * clx
                           : linepoly + (((size_t)b * nz + kbeg) * ny + y0) * CF + 4 * clx;
    const float* nsrc = ND ? P.nu + (size_t)b * P.nodes + first : nullptr;
    const float* fsrc = NF ? P.f + (size_t)b * P.nodes + first : nullptr;
    const long long uwrap = (long long)plane - (long long)T * nx, cwrap = ((long long)(KG ? ny - 1 : ny) - T) * CF;
    const unsigned dw = ring_s + 4u * ((lx & 3) * AS + 2 * (lx >> 2)), dc = ring_s + 4u * COEF + 16u * clx;
    auto copy_row = [&](const unsigned d, const unsigned dh, const float* src) {
        if (!tiny) {
            const float* back_src = src + back;
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                p3_cp4(d + 2u * LW * i, src + LW * i);
                p3_cp4(d + 2u * LW * i + 4u, back_src - LW * i);
            }
            p3_cp4_if(dh + 4u * lx, (lx & 1) ? src + (nx - 2 - NX * LW) : src + NX * LW, (lx < 2) ? 1 : 0);   // the pair right of the last lane
        } else {                                        // words beyond the far face repeat it (nothing owned depends on them)
            const float* row = src - lx;
            for (int i = 0; i < NX; ++i) {
                const int w = min(lx + LW * i, nx - 1);
                p3_cp4(d + 2u * LW * i, row + w);
                p3_cp4(d + 2u * LW * i + 4u, row + (nx - 1 - w));
            }
            const int w = min(NX * LW, nx - 1);
            p3_cp4_if(dh + 4u * lx, row + ((lx & 1) ? nx - 1 - w : w), (lx < 2) ? 1 : 0);
        }
    };
    auto issue = [&]() {
        if (pfk < nplanes) {                            // uniform in the unit
            const unsigned dh = ring_s + 8u * LW + pfo;
            copy_row(dw + pfo, dh, usrc);
            if constexpr (ND) copy_row(dw + 4u * UROW + pfo, dh + 4u * UROW, nsrc);
            if constexpr (NF) copy_row(dw + 4u * FOFF + pfo, dh + 4u * FOFF, fsrc);
            if constexpr (CF > 0) {
                const int cok = (KN || (pfk >= 1 && pfj >= 1)) ? 1 : 0;
#pragma unroll
                for (int t = 0; t < CFQ; t += 4)        // 4 lanes are the fewest a unit can have
                    if (t == 0 || LW < CFQ) p3_cp16_if(dc + pfo + 16u * t, csrc + 4 * t, (lx + t < CFQ && (t & (LW - 1)) == 0) ? cok : 0);
            }
        }
        p3_commit();                                    // one group per entry, possibly empty
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

    auto ld2 = [](const float* p) { f2 v; v.v = *reinterpret_cast<const u64*>(p); return v; };
    auto st2 = [](float* p, const f2 v) { *reinterpret_cast<u64*>(p) = v.v; };
    // this lane's first pair of a row in a slot (column k: + k * AS; the one right of its columns: + 2)
    auto slotp = [&](const unsigned off, const int rowoff) {
        return reinterpret_cast<const float*>(reinterpret_cast<const char*>(ring) + off) + rowoff + 2 * lx;
    };
    auto ldu = [&](const float* p, const int k) {       // u at column k (0 .. NX) of the lane
        f2 v = ld2(p + (k < NX ? k * AS : 2));
        if (impose) {
            if (k == 0 && first_col) v = mk2(bc0, bc1);
            // the far face and the columns beyond it, which repeat it: nothing owned depends on them, but they enter sums with
            // weight 0, so what the field itself holds there (NaN, say) must not be read
            if constexpr (RG) { if (reach && x0 + k >= nx - 1) v = mk2(bc1, bc0); }
        }
        return v;
    };
    // KN: nu at this lane's nodes of the row in a slot (and at the pair right of the last lane), from the polynomial that
    // came with the row, into the slot
    auto nurow = [&](const unsigned off) {
        float* slot = reinterpret_cast<float*>(reinterpret_cast<char*>(ring) + off);
        f2 gg[GS / 2];
        const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(slot + COEF);
#pragma unroll
        for (int i = 0; i < GS / 4; ++i) { const ulonglong2 t = gp[i]; gg[2 * i].v = t.x; gg[2 * i + 1].v = t.y; }
        f2 nn[NX + 1];
#pragma unroll
        for (int k = 0; k <= NX; ++k) {
            f2 e = gg[M];
#pragma unroll
            for (int i = M - 1; i >= 0; --i) e = fma2(e, cnp[k], gg[i]);
            float e0, e1;
            un2(e, e0, e1);
            nn[k] = mk2(p3_ex2(e0), p3_ex2(e1));
        }
#pragma unroll
        for (int k = 0; k < NX; ++k) st2(slot + UROW + k * AS + 2 * lx, nn[k]);
        if (lx == LW - 1) st2(slot + UROW + 2 * LW, nn[NX]);
    };
    // a finished row of nx floats to global memory
    auto store_row = [&](float* row, const f2 (&o)[NX]) {
        if constexpr (RG) {
            __syncwarp(submask);                        // the row before it has left the buffer
#pragma unroll
            for (int k = 0; k < NX; ++k) st2(obuf + 2 * (LW * k + lx), o[k]);
            __syncwarp(submask);
            const float* src = obuf + 2 * (LW * (lx & 3) + (lx >> 2));
#pragma unroll
            for (int i = 0; i < NX; ++i) {
                const int w = lx + LW * i;
                const f2 t = ld2(src + LW / 2 * i);
                if (w < ownL) row[w] = lo2(t);
                if (w < ownR) row[nx - 1 - w] = hi2(t);
            }
        } else if (act) {
            float l[NX], r[NX];
#pragma unroll
            for (int k = 0; k < NX; ++k) un2(o[k], l[k], r[k]);
            *reinterpret_cast<float4*>(row + x0) = make_float4(l[0], l[1], l[2], l[3]);
            *reinterpret_cast<float4*>(row + nx - NX - x0) = make_float4(r[3], r[2], r[1], r[0]);
        }
    };
    auto wrapb = [&](unsigned o) { return o >= RINGB ? o - RINGB : o; };

    // the load-energy sum of a row: its owned nodes, half weight on the faces; X: the middle node without a lane
    auto row_sum = [&](const float* p) {
        f2 a = wx0 * owned(0, ldu(p, 0));
#pragma unroll
        for (int c = 1; c < NX; ++c) a = a + owned(c, ldu(p, c));
        float l, h;
        un2(a, l, h);
        l += h;
        if (RG && lastx) l += lo2(ldu(p, NX));
        return l;
    };

    if constexpr (!EO) {
        for (int j = 0; j < T; ++j) {
#pragma unroll
            for (int k = 0; k < NX; ++k) st2(park + j * PR + 2 * (LW * k + lx), dup2(0.f));
            if (RG && lastx) xw[2 + j] = 0.f;
        }
    }
    f2 pendL[NX], pendU[NX];                            // what the element row below left for the current node row
    float* pendx = xw;                                  // ... for the middle node without a lane
    double end = 0.0, eld = 0.0;
    unsigned oA = 0;                                    // slot (byte offset) of the lower-plane, lower row of the current element row
    int n = 0;                                          // ... and its entry index
    const unsigned TB = (unsigned)T * RSB;
    for (int kk = 0; kk + 1 < nplanes; ++kk) {
        const int k = kbeg + kk;                        // element plane k lies between node planes k and k + 1: plane k is
        const float wzlo = (k == 0) ? 0.5f : 1.f;       // finished now, with the partial sums parked one step before; the
        const float nllo = -gs * fw * wzlo;             // sums of plane k + 1 are parked (plane ke: finished after the march)
        f2 enlo = dup2(0.f), elnf = dup2(0.f);
        float ello = 0.f;
#pragma unroll
        for (int c = 0; c < NX; ++c) { pendL[c] = dup2(0.f); pendU[c] = dup2(0.f); }
        if (!EO && RG && lastx) { pendx[0] = 0.f; pendx[1] = 0.f; }
        float* rlo = EO ? nullptr : rb + ((size_t)k * ny + y0) * nx;
        float* pk = park + 2 * lx;                      // column k: + 2 LW k
        float* pkx = xw + 2;
        for (int jj = 0; jj + 1 < T; ++jj) {
            p3_wait<0>();                               // everything issued up to the previous step has landed ...
            __syncwarp(submask);                        // ... is visible to the unit, and the rows it retired are free
            while (pf < n + C) issue();
            const unsigned oB = wrapb(oA + RSB), oC = wrapb(oA + TB), oD = wrapb(oC + RSB);
            const float wy = (y0 + jj == 0) ? 0.5f : 1.f;
            const float *pA = slotp(oA, 0), *pB = slotp(oB, 0), *pC = slotp(oC, 0), *pD = slotp(oD, 0);
            f2 ga[GS / 2], gb[GS / 2];                  // Gauss row q = a / b; each entry holds (plane s = a, s = b)
            if constexpr (KN) {
                // rows meet the march at its upper, far corner: a row is new when it is D, and also when it is B in the
                // unit's first plane, C in a plane's first row, A at the very start
                if (kk == 0 && jj == 0) nurow(oA);
                if (kk == 0) nurow(oB);
                if (jj == 0) nurow(oC);
                nurow(oD);
                __syncwarp(submask);                    // the node right of a lane's last is the next lane's
            }
            if constexpr (KG) {
                const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(ring) + oD) + COEF / 4;
#pragma unroll
                for (int i = 0; i < GS / 4; ++i) {
                    const ulonglong2 t0 = gp[i], t1 = gp[GS / 4 + i];
                    ga[2 * i].v = t0.x; ga[2 * i + 1].v = t0.y; gb[2 * i].v = t1.x; gb[2 * i + 1].v = t1.y;
                }
            }
            const float nlrow = nllo * wy;
            f2 olo[NX], cin[NX];
            if constexpr (GP && !EO) {                  // on their way while the elements are computed
#pragma unroll
                for (int c = 0; c < NX; ++c) cin[c] = ld2(pk + 2 * LW * c);
            }
            // Finish of column c of this row on both planes: `lo` / `up` are everything the lane's elements of this row
            // contribute to node (c, j, k) / (c, j, k+1), `lo1` / `up1` what they leave for row j + 1.
            auto node = [&](const int c, const f2 u, const f2 lo, const f2 lo1, const f2 up, const f2 up1) {
                const f2 raw = (lo + pendL[c]) + (GP ? cin[c] : ld2(pk + 2 * LW * c));
                st2(pk + 2 * LW * c, up + pendU[c]);
                pendL[c] = lo1; pendU[c] = up1;
                enlo = fma2(owned(c, u), raw, enlo);
                olo[c] = fma2((c == 0) ? sc02 : sc2, raw, dup2((c == 0) ? lw0 * nlrow : nlrow));
            };
            // ---- the NX element pairs of this lane, from right to left: element c completes column c + 1
            f2 q000, q010, q001, q011;                  // own-corner contributions of the element on the right
            f2 a100, a110, a101, a111;                  // from the last element of the lane on the left
            // column c + 1 of the four node rows (u, nu, f); column c is read as it is needed, to keep registers few
            f2 uA1 = ldu(pA, NX), uB1 = ldu(pB, NX), uC1 = ldu(pC, NX), uD1 = ldu(pD, NX);
            f2 nA1, nB1, nC1, nD1, fA1, fB1, fC1, fD1;
            if constexpr (!KG) { nA1 = ld2(pA + UROW + 2); nB1 = ld2(pB + UROW + 2); nC1 = ld2(pC + UROW + 2); nD1 = ld2(pD + UROW + 2); }
            if constexpr (NF) { fA1 = ld2(pA + FOFF + 2); fB1 = ld2(pB + FOFF + 2); fC1 = ld2(pC + FOFF + 2); fD1 = ld2(pD + FOFF + 2); }
#pragma unroll
            for (int c = NX - 1; c >= 0; --c) {
                const f2 uA = ldu(pA, c), uB = ldu(pB, c), uC = ldu(pC, c), uD = ldu(pD, c);
                const f2 eA = uA1 - uA, eB = uB1 - uB, eC = uC1 - uC, eD = uD1 - uD;
                const f2 slo = uB - uA, sup = uD - uC, w0 = uC - uA;
                const f2 txy = eB - eA, txyu = eD - eC, txz = eC - eA, tyz = sup - slo, txyz = txyu - txy;
                f2 Nx[4], Ny[4], Nz[4], r[8];
                (void)r;
                if constexpr (KG) {
                    f2 nu[8], col[4];
                    const ulonglong2 ca = *reinterpret_cast<const ulonglong2*>(cpl + (2 * c) * LW);
                    const ulonglong2 cb = *reinterpret_cast<const ulonglong2*>(cpl + (2 * c + 1) * LW);
                    col[0].v = ca.x; col[1].v = ca.y; col[2].v = cb.x; col[3].v = cb.y;
                    p3_nu_gauss<M>(ga, gb, col, nu);
                    p3_sums_gauss(nu, Nx, Ny, Nz);
                } else {
                    const int o = UROW + c * AS;
                    const f2 nA = ld2(pA + o), nB = ld2(pB + o), nC = ld2(pC + o), nD = ld2(pD + o);
                    p3_bilerp(nA + nA1, nB + nB1, nC + nC1, nD + nD1, Nx);         // (q, s)
                    p3_bilerp(nA + nB, nA1 + nB1, nC + nD, nC1 + nD1, Ny);         // (p, s)
                    p3_bilerp(nA + nC, nA1 + nC1, nB + nD, nB1 + nD1, Nz);         // (p, q)
                    nA1 = nA; nB1 = nB; nC1 = nC; nD1 = nD;
                }
                f2 fc[8], uc[8];
                if constexpr (NF) {
                    const int o = FOFF + c * AS;
                    const f2 fA = ld2(pA + o), fB = ld2(pB + o), fC = ld2(pC + o), fD = ld2(pD + o);
                    fc[0] = fA; fc[1] = fA1; fc[2] = fB; fc[3] = fB1; fc[4] = fC; fc[5] = fC1; fc[6] = fD; fc[7] = fD1;
                    uc[0] = uA; uc[1] = uA1; uc[2] = uB; uc[3] = uB1; uc[4] = uC; uc[5] = uC1; uc[6] = uD; uc[7] = uD1;
                    fA1 = fA; fB1 = fB; fC1 = fC; fD1 = fD;
                }
                const f2 un = uA1;                      // u of the node that element c completes
                uA1 = uA; uB1 = uB; uC1 = uC; uD1 = uD;
                if constexpr (EO) {
                    enlo = fma2(em[c], p3_energy(Nx, Ny, Nz, eA, slo, w0, txy, txz, tyz, txyz, kx, ky, kz), enlo);
                    if constexpr (NF) {
                        f2 m[8], ef = dup2(0.f);
                        p3_mass(fc, m);
#pragma unroll
                        for (int t = 0; t < 8; ++t) ef = fma2(uc[t], m[t], ef);
                        elnf = fma2(em[c], ef, elnf);
                    }
                    continue;
                }
                p3_element<ISO>(Nx, Ny, Nz, eA, slo, w0, txy, txz, tyz, txyz, kx, ky, kz, r);
                if constexpr (NF) {
                    f2 m[8], e = dup2(0.f);
                    p3_mass(fc, m);
#pragma unroll
                    for (int t = 0; t < 8; ++t) { r[t] = fma2(dup2(-fs), m[t], r[t]); e = fma2(uc[t], m[t], e); }
                    elnf = fma2(em[c], e, elnf);
                }
                if (c == NX - 1) {
                    // the lane's last element: its right-hand corners belong to the next lane
                    a100.v = __shfl_up_sync(submask, r[1].v, 1, LW); a110.v = __shfl_up_sync(submask, r[3].v, 1, LW);
                    a101.v = __shfl_up_sync(submask, r[5].v, 1, LW); a111.v = __shfl_up_sync(submask, r[7].v, 1, LW);
                    if (RG && lastx) {                  // ... or, from both sides, to the middle node
                        float l, h;
                        un2(r[1], l, h);
                        const float raw = ((l + h) + pendx[0]) + *pkx;
                        un2(r[5], l, h); *pkx = (l + h) + pendx[1];
                        un2(r[3], l, h); pendx[0] = l + h;
                        un2(r[7], l, h); pendx[1] = l + h;
                        enlo = fma2(un, mk2(raw, 0.f), enlo);
                        rlo[NX * LW] = fmaf(sc, raw, nlrow);
                    }
                } else {
                    node(c + 1, un, q000 + r[1], q010 + r[3], q001 + r[5], q011 + r[7]);
                }
                q000 = r[0]; q010 = r[2]; q001 = r[4]; q011 = r[6];
            }
            if constexpr (!EO) node(0, uA1, fma2(a100, lm2, q000), fma2(a110, lm2, q010), fma2(a101, lm2, q001), fma2(a111, lm2, q011));
            if (hasf) ello = fmaf(wy, row_sum(pA), ello);
            if constexpr (!EO) {
                store_row(rlo, olo);
                rlo += nx; pk += PR; ++pkx;
            }
            oA = oB; ++n;
        }
        // ---- the top node row e1 of the tile gets nothing more in this plane.  It is this tile's own if it is the
        // top of the domain; else it belongs to the next tile and its sums go to the seam array (no load term: the
        // owner adds it).
        {
            const float* pA = slotp(oA, 0);
            const float wy = lasttile ? 0.5f : 0.f;
            if constexpr (!EO) {
                const float nlrow = nllo * wy;
                f2 olo[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    const f2 raw = pendL[c] + ld2(pk + 2 * LW * c), u = ldu(pA, c);
                    st2(pk + 2 * LW * c, pendU[c]);
                    enlo = fma2(owned(c, u), raw, enlo);
                    olo[c] = fma2((c == 0) ? sc02 : sc2, raw, dup2((c == 0) ? lw0 * nlrow : nlrow));
                }
                float* plo = lasttile ? rlo : sb + (size_t)k * nx;
                store_row(plo, olo);
                if (RG && lastx) {
                    const float raw = pendx[0] + *pkx;
                    enlo = fma2(ldu(pA, NX), mk2(raw, 0.f), enlo);
                    plo[NX * LW] = fmaf(sc, raw, nlrow);
                    *pkx = pendx[1];
                }
            }
            if (hasf) ello = fmaf(wy, row_sum(pA), ello);
            oA = wrapb(oA + RSB); ++n;
        }
        // per-plane sums go to double
        if (act || EO) {
            float l, h;
            un2(enlo, l, h);
            end += (double)l + (double)h;
            if constexpr (NF) { un2(elnf, l, h); eld += (double)l + (double)h; }
            else eld += (double)(wzlo * ello);
        }
    }
    p3_wait<0>();

    // ---- node plane ke gets nothing more from this chunk: what was parked for it is complete as far as this chunk
    // goes.  Top of the domain: finished into r with its load.  Else the plane is the next chunk's: the scaled, masked
    // sums go to the z seam (no load term: the owner adds it).  Its rows are still in the ring (entry n is row 0).
    {
        f2 entop = dup2(0.f);
        float eltop = 0.f;
        const float lf = lastchunk ? 1.f : 0.f;
        float* ptop = ztop;
        const float* pk = park + 2 * lx;
        for (int jj = 0; jj < T; ++jj) {
            const bool seamrow = (jj == T - 1) && !lasttile;
            const int j = y0 + jj;
            const float wy = seamrow ? 0.f : (j == 0 || j == ny - 1) ? 0.5f * lf : lf;
            const float* pT = slotp(oA, 0);
            if constexpr (!EO) {
                float* p = seamrow ? zstop : ptop;
                const float nlrow = -gs * fw * 0.5f * wy;
                f2 o[NX];
#pragma unroll
                for (int c = 0; c < NX; ++c) {
                    const f2 part = ld2(pk + 2 * LW * c), u = ldu(pT, c);
                    entop = fma2(owned(c, u), part, entop);
                    o[c] = fma2((c == 0) ? sc02 : sc2, part, dup2((c == 0) ? lw0 * nlrow : nlrow));
                }
                store_row(p, o);
                if (RG && lastx) {
                    const float raw = xw[2 + jj];
                    entop = fma2(ldu(pT, NX), mk2(raw, 0.f), entop);
                    p[NX * LW] = fmaf(sc, raw, nlrow);
                }
                ptop += nx; pk += PR;
            }
            if constexpr (!NF) eltop = fmaf(wy, row_sum(pT), eltop);
            oA = wrapb(oA + RSB);
        }
        if (act) {
            float l, h;
            un2(entop, l, h);
            end += (double)l + (double)h;
            if constexpr (!NF) eld += (double)(0.5f * eltop);
        }
    }

    // ---- energy partial of this unit: its lanes summed in a fixed order in double
    // NF: `end` holds sum u (K u - F) in units of kap and `eld` sum u_corner (M_e f_e)_corner, so that
    // the load part is fsabs * eld and the diffusion part half of (kap * end + load part)
    // (energy only: `end` is sum u K u itself, with or without nodal forcing)
    double l = NF ? (double)fsabs * eld : (hasf && act) ? (double)fw * eld : 0.0;
    double d = (NF && !EO) ? 0.5 * ((double)kap * end + l) : 0.5 * (double)kap * end;
    for (int off = LW >> 1; off > 0; off >>= 1) {
        d += __shfl_down_sync(submask, d, off, LW);
        l += __shfl_down_sync(submask, l, off, LW);
    }
    if (lx == 0) {
        double* slot = P.partials + 2 * ((size_t)b * P.nblk + (size_t)chunk * G.ntile + tile);
        slot[0] = d; slot[1] = l;
    }
}

constexpr size_t P3_SMEM_SM = 233472;              // shared memory of an SM; a block also reserves 1 KiB
constexpr size_t P3_SMEM_BLOCK = 232448;           // most a block can ask for

int p3_slot_floats(int lw, int mode, int m, bool nf) {
    const int urow = NX * (2 * lw + 2);
    const int rows = (mode == DN_NU_KL_GAUSS ? 1 : 2) + (nf ? 1 : 0);
    return rows * urow + (mode == DN_NU_KL_GAUSS ? 2 * line_floats(m) : mode == DN_NU_KL_NODAL ? line_floats(m) : 0);
}
bool p3_global_park(int mode, bool nf) { return mode != DN_NU_KL_GAUSS || nf; }
// floats of shared memory a unit needs; rg: with the row on its way out
size_t p3_unit_floats(int C, int RS, int Ry, int lw, bool eo, bool gp, bool rg) {
    if (eo) return (size_t)C * RS;
    return (size_t)C * RS + (Ry + 6) / 4 * 4 + (gp ? 0 : (size_t)(Ry + 1) * 2 * NX * lw) + (rg ? 2 * NX * lw : 0);
}

P3Geo geometry3p_search(const dn_problem& p, int sms, bool eo) {
    P3Geo g{};
    const int nx = p.grid.nx, ny = p.grid.ny, nz = p.grid.nz;
    g.LW = 4; g.lwsh = 2;
    while (2 * NX * g.LW + 1 < nx) { g.LW *= 2; ++g.lwsh; }
    const int subs = 32 / g.LW;
    g.RS = p3_slot_floats(g.LW, p.nu_mode, p.kl_modes, p.f != nullptr);
    size_t per_block = (P3_SMEM_SM - (size_t)P3_MINB * 1024) / P3_MINB;
    if (per_block > P3_SMEM_BLOCK) per_block = P3_SMEM_BLOCK;
    if (p.nu_mode == DN_NU_KL_GAUSS) per_block -= sizeof(float) * 8 * NX * g.LW;      // the block's table of cosines
    const size_t per_unit = per_block / (sizeof(float) * P3_WARPS * subs);            // floats
    int ry_max = ny - 1 < 64 ? ny - 1 : 64;
    while (ry_max > 1 && p3_unit_floats(ry_max + 2 + P3_D, g.RS, ry_max, g.LW, eo, p3_global_park(p.nu_mode, p.f != nullptr), true) > per_unit) --ry_max;
    const long long slots = (long long)sms * P3_MINB * P3_WARPS * subs;
    double best = -1.0;
    for (int Ry = 1; Ry <= ry_max; ++Ry) {
        const long long ntile = (ny - 1 + Ry - 1) / Ry;
        for (int Z = 1; Z <= nz - 1; ++Z) {
            const long long nchunk = (nz - 1 + Z - 1) / Z;
            const long long units = (long long)p.batch * ntile * nchunk;
            const double cost = row3d_cost(Ry, Z, ny, nz, p.batch, slots);
            if (best < 0 || cost < best * (1.0 - 1e-9)) {
                best = cost;
                g.Ry = Ry; g.Z = Z; g.ntile = (int)ntile; g.nchunk = (int)nchunk; g.units = units;
            }
        }
    }
    g.C = g.Ry + 2 + P3_D;
    return g;
}

P3Geo geometry3p(const dn_problem& p, bool eo) {
    const int sms = sm_count();
    return memo_geometry<P3Geo>(p, sms, [&]() { return geometry3p_search(p, sms, eo); }, eo ? 1 : 0);
}

template <int M, int MODE, bool NF, bool EO, int LWC, bool ISO, bool RG>
cudaError_t launch_p3(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    const int subs = 32 / g.LW;
    const size_t per_unit = p3_unit_floats(g.C, g.RS, g.Ry, g.LW, EO, MODE != 0 || NF, RG);
    const size_t smem = sizeof(float) * (P3_WARPS * subs * per_unit + (MODE == 0 ? 8 * NX * g.LW : 0));
    const long long per_block = (long long)P3_WARPS * subs;
    const unsigned blocks = (unsigned)((g.units + per_block - 1) / per_block);
    const cudaError_t e = allow_shared(pair3d_kernel<M, MODE, NF, EO, LWC, ISO, RG>, smem);
    if (e != cudaSuccess) return e;
    return launch_dependent(pair3d_kernel<M, MODE, NF, EO, LWC, ISO, RG>, dim3(blocks), dim3(P3_WARPS * 32), smem, s, P, linepoly, g);
}

template <int M, int MODE, bool RG>
cudaError_t launch_p3_fused(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    if (g.LW == 32) return launch_p3<M, MODE, false, false, 32, true, RG>(P, linepoly, g, s);
    if (g.LW == 16) return launch_p3<M, MODE, false, false, 16, true, RG>(P, linepoly, g, s);
    if (g.LW == 8) return launch_p3<M, MODE, false, false, 8, true, RG>(P, linepoly, g, s);
    return launch_p3<M, MODE, false, false, 0, false, true>(P, linepoly, g, s);      // rows of at most 33 nodes
}

template <int M, int MODE, bool NF>
cudaError_t launch_p3_energy(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    if (g.LW == 32) return launch_p3<M, MODE, NF, true, 32, false, true>(P, linepoly, g, s);
    if (g.LW == 16) return launch_p3<M, MODE, NF, true, 16, false, true>(P, linepoly, g, s);
    return launch_p3<M, MODE, NF, true, 0, false, true>(P, linepoly, g, s);
}

// Variants compiled: constant forcing on cubic cells for 8, 16 or 32 lanes and both ways of storing; the rest for
// any lane count and any row.
template <int M, int MODE>
cudaError_t launch_p3_mode(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    const bool iso = P.hx == P.hy && P.hy == P.hz;
    if (P.r == nullptr) return P.f ? launch_p3_energy<M, MODE, true>(P, linepoly, g, s) : launch_p3_energy<M, MODE, false>(P, linepoly, g, s);
    if (P.f) {
        if (iso && g.LW == 32) return launch_p3<M, MODE, true, false, 32, true, true>(P, linepoly, g, s);
        if (iso && g.LW == 16) return launch_p3<M, MODE, true, false, 16, true, true>(P, linepoly, g, s);
        if (iso && g.LW == 8) return launch_p3<M, MODE, true, false, 8, true, true>(P, linepoly, g, s);
        return launch_p3<M, MODE, true, false, 0, false, true>(P, linepoly, g, s);
    }
    const bool whole = P.nx % 8 == 0 && (reinterpret_cast<uintptr_t>(P.r) & 15u) == 0;
    if (!iso) {
        if (whole && g.LW == 32) return launch_p3<M, MODE, false, false, 32, false, false>(P, linepoly, g, s);
        if (whole && g.LW == 16) return launch_p3<M, MODE, false, false, 16, false, false>(P, linepoly, g, s);
        if (whole && g.LW == 8) return launch_p3<M, MODE, false, false, 8, false, false>(P, linepoly, g, s);
        return launch_p3<M, MODE, false, false, 0, false, true>(P, linepoly, g, s);
    }
    return whole ? launch_p3_fused<M, MODE, false>(P, linepoly, g, s) : launch_p3_fused<M, MODE, true>(P, linepoly, g, s);
}

template <int M>
cudaError_t launch_p3_m(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    return (P.nu_mode == DN_NU_KL_NODAL) ? launch_p3_mode<M, 1>(P, linepoly, g, s) : launch_p3_mode<M, 0>(P, linepoly, g, s);
}

}  // namespace

#if DN_P3_PART == 1
cudaError_t launch_pair3d_m34(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    return P.m == 3 ? launch_p3_m<3>(P, linepoly, g, s) : launch_p3_m<4>(P, linepoly, g, s);
}
#elif DN_P3_PART == 2
cudaError_t launch_pair3d_m56(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    return P.m == 5 ? launch_p3_m<5>(P, linepoly, g, s) : launch_p3_m<6>(P, linepoly, g, s);
}
#elif DN_P3_PART == 3
cudaError_t launch_pair3d_m78(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    return P.m == 7 ? launch_p3_m<7>(P, linepoly, g, s) : launch_p3_m<8>(P, linepoly, g, s);
}
#else
cudaError_t launch_pair3d_m12(const Params& P, const float* linepoly, const P3Geo& g, cudaStream_t s) {
    if (P.nu_mode == DN_NU_NODAL) return launch_p3_mode<1, 2>(P, linepoly, g, s);
    return P.m == 1 ? launch_p3_m<1>(P, linepoly, g, s) : launch_p3_m<2>(P, linepoly, g, s);
}

// Rows of at most 257 nodes: a side of 128 columns is 32 lanes, and of 2^k + 1 nodes the middle one needs no lane.
bool pair3d_applicable(const dn_problem& p) {
    return p.grid.dim == 3 && p.grid.nx <= 2 * NX * 32 + 1 && p.grid.nx >= 2 && p.grid.ny >= 2 && p.grid.nz >= 2;
}

Launch pair3d_geometry(const dn_problem& p, bool want_r) {
    const P3Geo g = geometry3p(p, !want_r);
    Launch l{};
    l.path = PATH_PAIR3D;
    l.nblk = g.ntile * g.nchunk;
    l.chunk = g.Z;
    l.variant = g.Ry;
    return l;
}

size_t pair3d_seam_floats(const dn_problem& p) {
    if (!pair3d_applicable(p)) return 0;
    const P3Geo g = geometry3p(p, false);
    return (size_t)p.batch * (g.ntile - 1) * p.grid.nz * p.grid.nx;
}

// the chunk seams: [B][nchunk-1][ny][nx], then [B][nchunk-1][ntile-1][nx] for the nodes on a tile seam as well
size_t pair3d_zseam_floats(const dn_problem& p) {
    if (!pair3d_applicable(p)) return 0;
    const P3Geo g = geometry3p(p, false);
    return (size_t)p.batch * (g.nchunk - 1) * ((size_t)p.grid.ny + (g.ntile - 1)) * p.grid.nx;
}

// partial sums parked in global memory, one row of pairs per node row of every unit
size_t pair3d_park_floats(const dn_problem& p) {
    if (!pair3d_applicable(p) || !p3_global_park(p.nu_mode, p.f != nullptr)) return 0;
    const P3Geo g = geometry3p(p, false);
    return (size_t)g.units * (g.Ry + 1) * 2 * NX * g.LW;
}

// the coefficient table: per element row its four Gauss lines (KL at the Gauss points), or per node line (KL at the nodes)
size_t pair3d_linepoly_floats(const dn_problem& p) {
    if (!pair3d_applicable(p) || p.nu_mode == DN_NU_NODAL) return 0;
    if (p.nu_mode == DN_NU_KL_NODAL) return (size_t)p.batch * p.grid.nz * p.grid.ny * line_floats(p.kl_modes);
    return (size_t)p.batch * (p.grid.nz - 1) * (p.grid.ny - 1) * 2 * line_floats(p.kl_modes);
}

static dn_problem problem_of(const Params& P) {
    dn_problem p{};
    p.grid.dim = 3; p.grid.nx = P.nx; p.grid.ny = P.ny; p.grid.nz = P.nz; p.batch = P.batch;
    p.nu_mode = P.nu_mode; p.kl_modes = P.m; p.f = P.f; p.flags = P.flags;
    return p;
}

cudaError_t launch_pair3d(const Params& P, const float* linepoly, cudaStream_t s) {
    const P3Geo g = geometry3p(problem_of(P), P.r == nullptr);
    if (P.nu_mode == DN_NU_NODAL || P.m <= 2) return launch_pair3d_m12(P, linepoly, g, s);
    if (P.m <= 4) return launch_pair3d_m34(P, linepoly, g, s);
    if (P.m <= 6) return launch_pair3d_m56(P, linepoly, g, s);
    return launch_pair3d_m78(P, linepoly, g, s);
}

cudaError_t launch_pair3d_seams(const Params& P, float* J, cudaStream_t s) {
    const P3Geo g = geometry3p(problem_of(P), false);
    return launch_seam_fixup3(P, g.Ry, g.ntile, g.Z, g.nchunk, J, s);
}
#endif  // DN_P3_PART

}  // namespace dn
