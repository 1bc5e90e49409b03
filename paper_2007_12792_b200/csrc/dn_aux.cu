// Small kernels around the fused loss kernel: cosine / coefficient tables for the KL
// expansion, the nodal KL field, the Dirichlet face overwrite, the energy finaliser.
#include "dn_internal.cuh"

namespace dn {

namespace {

constexpr double kLog2e = 1.4426950408889634074;

struct Reciprocals {                                    // 1 / q for the eigenvalues q = 1 + i^2 + j^2 (+ k^2), log2 e included
    double r[2 + 3 * DN_MAX_KL_MODES * DN_MAX_KL_MODES];
    constexpr Reciprocals() : r() {
        for (int q = 1; q < 2 + 3 * DN_MAX_KL_MODES * DN_MAX_KL_MODES; ++q) r[q] = kLog2e / q;
    }
};
__device__ constexpr Reciprocals klf_inv{};

// ---------------------------------------------------------------------------------------
// Tables for the KL expansion evaluated at Gauss points (DN_NU_KL_GAUSS):
//   ckl[b][i][j]([k]) = w * log2(e) / (1 + i^2 + j^2 (+ k^2))      so that nu = 2^(sum ckl cos cos (cos))
//   cg[a][i-1][p]     = cos(i pi x_p),  x_p = (p/2 + (p odd ? GB : GA)) * h_a,  p < 2 (n_a - 1)
//   cn[a][i-1][n]     = cos(i pi n h_a) at the nodes (DN_NU_KL_NODAL)
// The cosines are evaluated in double (cospi) and rounded once.
// ---------------------------------------------------------------------------------------
struct TableArgs {
    int dim, m, batch;
    int n[3];
    int gstride[3];
    const float* kl_w;
    float* ckl;
    float* cg[3];
    int nstride[3];
    float* cn[3];
    float* rowpoly;       // 2D, optional: polynomial of the KL exponent along every Gauss row, [B][ny-1][rp_gs]
    int rp_gs;
    int rp_nodes;         // 0: the two Gauss rows of every element row, interleaved; 1: every node row, each coefficient twice
};

// exponent(x, y_q) = sum_k poly[k] c^k with c = cos(pi x), for the Gauss row q of element row j of sample b:
// g_i = sum_j ckl[i][j] cos(j pi y_q) are the coefficients in the Chebyshev basis (cos(i pi x) = T_i(c)), converted
// to monomials in double.  The scaled weights and the cosines are rounded to float first, exactly as the tables
// hold them, so every kernel family sees the same numbers.  Entry 2k + q of the row; the two Gauss rows of an
// element row interleave so that they can be evaluated together with two-wide FMAs.  MX >= m is the compiled loop
// bound (the kernel is instantiated for every m; compile-time bounds keep the small arrays in registers).
template <int MX>
__device__ void rowpoly_entry(const TableArgs& A, long long idx) {
    const int m = A.m, ny = A.n[1];
    const int q = (int)(idx & 1);
    const int rows = A.rp_nodes ? ny : ny - 1;
    const long long row = idx >> 1;                    // b * rows + j
    const int j = (int)(row % rows);
    const long long b = row / rows;
    const double ga = 0.5 * (1.0 - 0.57735026918962576451);
    const double gb = 0.5 * (1.0 + 0.57735026918962576451);
    const double y = ((double)j + (q ? gb : ga)) / (double)(ny - 1);
    // cos(jj pi y) from cos(pi y) by the Chebyshev recurrence in double, rounded to float as the cosine tables are
    double cy[MX], g[MX];
    {
        const double c1 = cospi(A.rp_nodes ? (double)j / (double)(ny - 1) : y);
        double tm = 1.0, tc = c1;
#pragma unroll
        for (int jj = 0; jj < MX; ++jj) {
            cy[jj] = (jj < m) ? (double)(float)tc : 0.0;
            const double tn = 2.0 * c1 * tc - tm;
            tm = tc; tc = tn;
        }
    }
    const float* w = A.kl_w + b * m * m;
#pragma unroll
    for (int i = 0; i < MX; ++i) {
        double a = 0.0;
#pragma unroll
        for (int jj = 0; jj < MX; ++jj) {
            if (i < m && jj < m) {
                const double den = 1.0 + (double)((i + 1) * (i + 1)) + (double)((jj + 1) * (jj + 1));
                a += (double)(float)((double)w[i * m + jj] * (kLog2e / den)) * cy[jj];     // the constant folds: no division
            }
        }
        g[i] = a;
    }
    // sum_i g_i T_i(c) in the monomial basis, T_{i+1} = 2 c T_i - T_{i-1}
    double acc[MX + 1], tp[MX + 1], tc[MX + 1];
#pragma unroll
    for (int k = 0; k <= MX; ++k) { acc[k] = 0.0; tp[k] = (k == 0) ? 1.0 : 0.0; tc[k] = (k == 1) ? 1.0 : 0.0; }
#pragma unroll
    for (int i = 1; i <= MX; ++i) {
        if (i > m) break;                              // uniform; the rest of the terms are zero
#pragma unroll
        for (int k = 0; k <= MX; ++k) acc[k] += g[i - 1] * tc[k];
        double tn[MX + 1];
#pragma unroll
        for (int k = 0; k <= MX; ++k) tn[k] = ((k > 0) ? 2.0 * tc[k - 1] : 0.0) - tp[k];
#pragma unroll
        for (int k = 0; k <= MX; ++k) { tp[k] = tc[k]; tc[k] = tn[k]; }
    }
    float* dst = A.rowpoly + row * A.rp_gs + q;
#pragma unroll
    for (int k = 0; k <= MX; ++k) dst[2 * k] = (float)acc[k];
    for (int k = MX + 1; 2 * k + q < A.rp_gs; ++k) dst[2 * k] = 0.f;      // the padding of the row
}

// Entry idx of the tables.
template <int MX>
__device__ void table_entry(const TableArgs& A, long long idx) {
    const int m = A.m;
    long long mpow = 1;
    for (int a = 0; a < A.dim; ++a) mpow *= m;
    const long long ncoef = mpow * A.batch;
    if (idx < ncoef) {
        long long c = idx % mpow;
        int i, j, k = 0;
        if (A.dim == 3) { k = (int)(c % m) + 1; c /= m; }
        j = (int)(c % m) + 1;
        i = (int)(c / m) + 1;
        const double den = 1.0 + (double)i * i + (double)j * j + (double)k * k;
        A.ckl[idx] = (float)((double)A.kl_w[idx] * (kLog2e / den));      // the same product the row polynomials form
        return;
    }
    idx -= ncoef;
    const double ga = 0.5 * (1.0 - 0.57735026918962576451);
    const double gb = 0.5 * (1.0 + 0.57735026918962576451);
    for (int a = 0; a < A.dim; ++a) {
        const long long cnt = (long long)m * A.gstride[a];
        if (idx < cnt) {
            const int i = (int)(idx / A.gstride[a]) + 1;
            int p = (int)(idx % A.gstride[a]);
            const int ng = 2 * (A.n[a] - 1);
            if (p >= ng) p = ng - 1;                      // padding repeats the last abscissa
            const double x = ((double)(p >> 1) + ((p & 1) ? gb : ga)) / (double)(A.n[a] - 1);
            A.cg[a][idx] = (float)cospi((double)i * x);
            return;
        }
        idx -= cnt;
    }
    for (int a = 0; a < A.dim; ++a) {
        const long long cnt = (long long)m * A.nstride[a];
        if (idx < cnt) {
            const int i = (int)(idx / A.nstride[a]) + 1;
            int n = (int)(idx % A.nstride[a]);
            if (n >= A.n[a]) n = A.n[a] - 1;              // padding repeats the last node
            A.cn[a][idx] = (float)cospi((double)i * (double)n / (double)(A.n[a] - 1));
            return;
        }
        idx -= cnt;
    }
    if (A.rowpoly && idx < 2ll * A.batch * (A.n[1] - (A.rp_nodes ? 0 : 1))) rowpoly_entry<MX>(A, idx);
}

template <int MX>
__global__ void tables_kernel(TableArgs A) {
    dep_wait();                                        // whatever ran before in the stream may still read these tables
    dep_release();
    table_entry<MX>(A, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---------------------------------------------------------------------------------------
// 3D: the polynomials (in c = cos(pi x)) of the KL exponent along lines of fixed (y, z), prepared in double from the weights and
// cosines rounded to float, exactly as the tables hold them.
//   NODES false: along the four Gauss lines of every element row, [B][nz-1][ny-1][2 GS] floats: Gauss row q = a, then q = b, each
//   with (plane s = a, plane s = b) pairs for the powers 0..M.
//   NODES true: along every node line, every coefficient twice, so that two nodes share a packed FMA: [B][nz][ny][GS] floats.
// One block per (sample, plane, LINE_THREADS lines) sums the z factor once; a thread then writes what belongs to its element row or
// node line.
// ALL: the kernel also writes the tables (its last blocks), and the blocks of lines work out their cosines and scaled weights
// themselves: small problems, where a launch counts.
// What bounds it: with few blocks the latency of one, so with ALL the four lines of an element row are worked out side by side (255
// registers with 8 modes); with many the warps in flight, so without it one after the other (70 registers in place of 136; the
// call on 17^3 x 1360 m = 8 232 -> 201 us, 24^3 x 300 101 -> 92, 16^3 x 2634 m = 5 247 -> 227; but 24^3 x 1 m = 7 10.2 -> 10.7 so).
// ---------------------------------------------------------------------------------------
template <int M, bool NODES, bool ALL>
__global__ void __launch_bounds__(LINE_THREADS) lines3d_kernel(const TableArgs A, int chunks, int planes, float* __restrict__ out) {
    constexpr int GS = line_floats(M), S = NODES ? 1 : 2;
    __shared__ double h[S][M][M];                       // h[s][i][j] = sum_k ckl[i][j][k] cos(k pi z_s)
    __shared__ double cz[S][M];
    dep_wait();                                         // (ALL: as in tables_kernel) the scaled weights and cosine tables are complete
    dep_release();
    const int t0 = threadIdx.x, chunk = blockIdx.x % chunks, pb = blockIdx.x / chunks, ez = pb % planes, b = pb / planes;
    if (ALL && b >= A.batch) {
        table_entry<1>(A, (long long)(blockIdx.x - chunks * planes * A.batch) * LINE_THREADS + t0);
        return;
    }
    const double ga = 0.5 * (1.0 - 0.57735026918962576451), gb = 0.5 * (1.0 + 0.57735026918962576451);
    if constexpr (ALL) {
        if (t0 < S * M) {
            const int s = t0 / M, k = t0 % M;
            const double z = (NODES ? (double)ez : (double)ez + (s ? gb : ga)) / (double)(A.n[2] - 1);
            cz[s][k] = (double)(float)cospi((double)(k + 1) * z);
        }
        __syncthreads();
    }
    for (int t = t0; t < S * M * M; t += LINE_THREADS) {
        const int s = t / (M * M), ij = t % (M * M), q = 1 + (ij / M + 1) * (ij / M + 1) + (ij % M + 1) * (ij % M + 1);
        const float* w = (ALL ? A.kl_w : A.ckl) + ((long long)b * M * M + ij) * M;
        const float* tz = NODES ? A.cn[2] + ez : A.cg[2] + 2 * ez + s;      // (not ALL) the cosines of the plane
        const int step = NODES ? A.nstride[2] : A.gstride[2];
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < M; ++k)
            acc += ALL ? (double)(float)((double)w[k] * klf_inv.r[q + (k + 1) * (k + 1)]) * cz[s][k] : (double)w[k] * (double)tz[(size_t)k * step];
        h[s][ij / M][ij % M] = acc;
    }
    __syncthreads();
    const int ey = chunk * LINE_THREADS + t0, rows = NODES ? A.n[1] : A.n[1] - 1;
    if (ey >= rows) return;
    float4* dst = reinterpret_cast<float4*>(out + (((size_t)b * planes + ez) * rows + ey) * (S * GS));
#pragma unroll(ALL ? S : 1)
    for (int q = 0; q < S; ++q) {
        float row[GS];
#pragma unroll
        for (int i = 0; i < GS; ++i) row[i] = 0.f;      // the padding of a row stays zero
        double cy[M];
        if constexpr (ALL) {                            // by the Chebyshev recurrence in double, rounded to float as the tables are
            const double c1 = cospi((NODES ? (double)ey : (double)ey + (q ? gb : ga)) / (double)(A.n[1] - 1));
            double tm = 1.0, tc = c1;
#pragma unroll
            for (int j = 0; j < M; ++j) {
                cy[j] = (double)(float)tc;
                const double tn = 2.0 * c1 * tc - tm;
                tm = tc; tc = tn;
            }
        } else {
#pragma unroll
            for (int j = 0; j < M; ++j) cy[j] = (double)(NODES ? A.cn[1][(size_t)j * A.nstride[1] + ey] : A.cg[1][(size_t)j * A.gstride[1] + 2 * ey + q]);
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if constexpr (!ALL) asm volatile("" ::: "memory");         // one line after the other (see above)
            // sum_i g_i T_i(c) in the monomial basis, T_{i+1} = 2 c T_i - T_{i-1}
            double acc[M + 1], tp[M + 1], tc[M + 1];
#pragma unroll
            for (int k = 0; k <= M; ++k) { acc[k] = 0.0; tp[k] = (k == 0) ? 1.0 : 0.0; tc[k] = (k == 1) ? 1.0 : 0.0; }
#pragma unroll
            for (int i = 1; i <= M; ++i) {
                double g = 0.0;
#pragma unroll
                for (int j = 0; j < M; ++j) g += h[s][i - 1][j] * cy[j];
#pragma unroll
                for (int k = 0; k <= i; ++k) acc[k] += g * tc[k];
                double tn[M + 1];
#pragma unroll
                for (int k = 0; k <= M; ++k) tn[k] = ((k > 0) ? 2.0 * tc[k - 1] : 0.0) - tp[k];
#pragma unroll
                for (int k = 0; k <= M; ++k) { tp[k] = tc[k]; tc[k] = tn[k]; }
            }
#pragma unroll
            for (int k = 0; k <= M; ++k) {
                if constexpr (NODES) { row[2 * k] = (float)acc[k]; row[2 * k + 1] = (float)acc[k]; }
                else row[2 * k + s] = (float)acc[k];
            }
        }
#pragma unroll
        for (int i = 0; i < GS / 4; ++i) dst[q * (GS / 4) + i] = make_float4(row[4 * i], row[4 * i + 1], row[4 * i + 2], row[4 * i + 3]);
    }
}

// ---------------------------------------------------------------------------------------
// Energy finaliser: J[b] = sum over block partials (diffusion part) - (load part), summed
// in a fixed order in double, rounded once to float.
// ---------------------------------------------------------------------------------------
constexpr int FIN_THREADS = 256;
__device__ __forceinline__ void finalize_sample(const double* __restrict__ partials, int nblk, float* __restrict__ J, int b) {
    const double* p = partials + 2ll * b * nblk;
    double d = 0.0, l = 0.0;
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) { d += p[2 * i]; l += p[2 * i + 1]; }
    __shared__ double sd[256], sl[256];
    sd[threadIdx.x] = d; sl[threadIdx.x] = l;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) { sd[threadIdx.x] += sd[threadIdx.x + o]; sl[threadIdx.x] += sl[threadIdx.x + o]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) J[b] = (float)(sd[0] - sl[0]);
}
__global__ void __launch_bounds__(FIN_THREADS) finalize_kernel(const double* __restrict__ partials, int nblk, float* __restrict__ J) {
    dep_wait();
    finalize_sample(partials, nblk, J, blockIdx.x);
}

// Adds the seam contributions of a 3D kernel to r (fixed order per node: own sums, tile seam, chunk seam, the entry for nodes on
// both).  First range of threads: the nodes of the tile seam rows (t + 1) Ry on every plane; second range: the nodes of the
// chunk seam planes (c + 1) Z that are not on a tile seam row.  The two ranges touch different nodes.  V: float4 where
// rows and r allow it (nxv = nx / 4 pieces per row), else float.  The first `samples` blocks finish the energies of as many samples
// instead (small problems, where a launch counts).
__device__ __forceinline__ void seam_add(float& v, const float a) { v += a; }
__device__ __forceinline__ void seam_add(float4& v, const float4 a) { v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w; }
struct SeamArgs {
    int nxv, ny, nz, batch, Ry, ntile, Z, nchunk;
    long long nA, nB;
    int samples, nblk;
    const double* partials;
    float* J;
};
template <class V>
__global__ void __launch_bounds__(FIN_THREADS) seam_fixup3_kernel(V* __restrict__ r, const V* __restrict__ yseam, const V* __restrict__ zseam, const SeamArgs A) {
    dep_wait();                                         // the fused kernel has finished
    dep_release();
    if ((int)blockIdx.x < A.samples) { finalize_sample(A.partials, A.nblk, A.J, blockIdx.x); return; }
    const int nxv = A.nxv, ny = A.ny, nz = A.nz, Ry = A.Ry, ntile = A.ntile, Z = A.Z, nchunk = A.nchunk;
    const long long i = (long long)(blockIdx.x - A.samples) * FIN_THREADS + threadIdx.x, nA = A.nA;
    const V* zy = zseam + (size_t)A.batch * (nchunk - 1) * ny * nxv;
    if (i < nA) {
        const int x = (int)(i % nxv);
        long long t = i / nxv;
        const int k = (int)(t % nz); t /= nz;
        const int sm = (int)(t % (ntile - 1));
        const int b = (int)(t / (ntile - 1));
        const int j = (sm + 1) * Ry;
        V* dst = r + (((size_t)b * nz + k) * ny + j) * nxv + x;
        V v = *dst;
        seam_add(v, __ldg(yseam + i));
        if (k % Z == 0 && k > 0 && k < nz - 1) {        // also the first plane of a chunk
            const int c = k / Z - 1;
            seam_add(v, __ldg(zseam + (((size_t)b * (nchunk - 1) + c) * ny + j) * nxv + x));
            seam_add(v, __ldg(zy + (((size_t)b * (nchunk - 1) + c) * (ntile - 1) + sm) * nxv + x));
        }
        *dst = v;
    } else if (i < nA + A.nB) {
        const long long q = i - nA;
        const int x = (int)(q % nxv);
        long long t = q / nxv;
        const int j = (int)(t % ny); t /= ny;
        const int c = (int)(t % (nchunk - 1));
        const int b = (int)(t / (nchunk - 1));
        if (j % Ry == 0 && j > 0 && j < ny - 1) return;  // a tile seam row: done by the first range
        V* dst = r + (((size_t)b * nz + (c + 1) * Z) * ny + j) * nxv + x;
        V v = *dst;
        seam_add(v, __ldg(zseam + q));
        *dst = v;
    }
}

// ---------------------------------------------------------------------------------------
// Nodal KL field.  cos(i pi ix/(n-1)) is taken from cospif after an exact integer
// reduction of the angle to [0, pi/2], so the only rounding is that of k/(n-1).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float cos_node(int i, int ix, int nm1) {
    int k = ix;                                          // angle = pi * k / nm1, k in [0, 2 nm1)
    if (i > 1) {                                         // i <= 8: 32 bits hold i * ix on any axis of fewer than 2^28 nodes
        k = (nm1 < (1 << 28)) ? (int)((unsigned)(i * ix) % (unsigned)(2 * nm1)) : (int)(((long long)i * ix) % (2ll * nm1));
    }
    if (k > nm1) k = 2 * nm1 - k;                        // cos(2 pi - t) = cos t
    float sgn = 1.0f;
    if (2 * k > nm1) { k = nm1 - k; sgn = -1.0f; }       // cos(pi - t) = -cos t
    return sgn * cospif((float)k / (float)nm1);
}

constexpr int KLF_THREADS = 256;
constexpr int KLF_LINES = 64;                           // grid lines (fixed y, z) per block at most; of whole planes twice as many
constexpr int KLF_PLANES = 16;                          // whole planes per block at most

typedef unsigned long long klf_u64;
__device__ __forceinline__ klf_u64 klf_pack2(float lo, float hi) {
    klf_u64 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void klf_unpack2(klf_u64 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ klf_u64 klf_fma2(klf_u64 a, klf_u64 b, klf_u64 c) {
    klf_u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float klf_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The integer coefficients of the Chebyshev polynomials: T_i(c) = sum_k t[i][k] c^k.
struct Chebyshev {
    double t[DN_MAX_KL_MODES + 1][DN_MAX_KL_MODES + 1];
    constexpr Chebyshev() : t() {
        t[0][0] = 1.0; t[1][1] = 1.0;
        for (int i = 2; i <= DN_MAX_KL_MODES; ++i)
            for (int k = 0; k <= DN_MAX_KL_MODES; ++k) t[i][k] = (k > 0 ? 2.0 * t[i - 1][k - 1] : 0.0) - t[i - 2][k];
    }
};
__device__ constexpr Chebyshev klf_cheb{};

struct KlfGeo {
    int lines, ychunks, tx, ty;                         // lines per block, blocks per (x, y) plane and strip, threads per line, lines at a time
    int planes;                                         // PL: whole planes per block
};

// A block owns up to G.lines consecutive lines of one (x, y) plane, or (PL) several whole planes, and a strip of at most
// 4 * KLF_THREADS nodes in x.
// Along a line the exponent is a polynomial of degree m in c = cos(pi x) (cos(i pi x) = T_i(c)).  Its coefficients are
// prepared in double by the whole block, an item per thread and step (cosines of the lines; weights contracted with the
// cosines of the plane; with those of the lines; Chebyshev to monomials), and stored, duplicated, in shared memory, so a
// pair of nodes costs m packed FMAs, two ex2 and half a 128-bit store.  A thread owns 4 nodes of every ty-th line: next
// to one another where rows are aligned (VEC), else tx apart, so that either way the stores of a warp are contiguous.
// Write-bound where lines are long (1024^2 x 32, m = 4: 21.3 us, 6.3 TB/s; 256^3 x 4, m = 3: 39.8 us, 6.7 TB/s); with short
// lines the preparation counts, which is why no item of it is done twice in a block and none divides: 64^3 x 32, m = 6:
// 13.9 us, 55.5 us where a thread prepared a whole line; 128^3 x 8, m = 4: 13.2 and 28.8; 129^3 x 8: 20.5 and 45.2;
// 1024^2 x 32: 21.3 and 29.0.
template <int M, bool VEC, bool PL>
__global__ void __launch_bounds__(KLF_THREADS)
kl_field_kernel(int dim, int nx, int ny, int nz, const float* __restrict__ kl_w, float* __restrict__ nu, const KlfGeo G) {
    constexpr int GS = (2 * (M + 1) + 3) / 4 * 4;       // floats per line: (g_k, g_k) pairs, padded
    constexpr int NL = PL ? 2 * KLF_LINES : KLF_LINES, NP = PL ? KLF_PLANES : 1;
    __shared__ __align__(16) float gam[NL][GS];
    __shared__ __align__(16) float cx[4 * KLF_THREADS];
    __shared__ double cy[KLF_LINES][M], gi[NL][M], A[NP][M][M], cz[NP][M];
    const int tid = threadIdx.x, b = blockIdx.z;
    const int zb = PL ? blockIdx.x : blockIdx.x / G.ychunks, iz = PL ? zb * G.planes : zb;
    const int y0 = PL ? 0 : (blockIdx.x - zb * G.ychunks) * G.lines;
    const int planes = PL ? min(G.planes, nz - iz) : 1, ylines = PL ? ny : min(G.lines, ny - y0), lines = planes * ylines;
    const int row0 = tid / G.tx, col = tid - row0 * G.tx;
    const int x0 = blockIdx.y * (4 * G.tx) + (VEC ? 4 * col : col), xstep = VEC ? 1 : G.tx;
    for (int t = tid; t < 4 * G.tx; t += KLF_THREADS) cx[t] = cos_node(1, min((int)blockIdx.y * (4 * G.tx) + t, nx - 1), nx - 1);
    for (int t = tid; t < ylines * M; t += KLF_THREADS) cy[t / M][t % M] = (double)cos_node(t % M + 1, y0 + t / M, ny - 1);
    if (tid < planes * M) cz[tid / M][tid % M] = (dim == 3) ? (double)cos_node(tid % M + 1, iz + tid / M, nz - 1) : 1.0;
    dep_wait();                                         // up to here nothing but indices: the weights are complete from here on
    dep_release();
    __syncthreads();
    for (int t = tid; t < planes * M * M; t += KLF_THREADS) {
        const int p = PL ? t / (M * M) : 0, ij = t - p * (M * M);
        const int i = ij / M, j = ij % M, q = 1 + (i + 1) * (i + 1) + (j + 1) * (j + 1);
        double a = 0.0;
        if (dim == 3) {
            const float* w = kl_w + ((long long)b * M * M + ij) * M;
#pragma unroll
            for (int k = 0; k < M; ++k) a += (double)__ldg(w + k) * klf_inv.r[q + (k + 1) * (k + 1)] * cz[p][k];
        } else {
            a = (double)__ldg(kl_w + (long long)b * M * M + ij) * klf_inv.r[q];
        }
        A[p][i][j] = a;
        if constexpr (!PL) break;                       // M * M threads have one each
    }
    __syncthreads();
    for (int t = tid; t < lines * M; t += KLF_THREADS) {
        const int l = t / M, i = t % M, p = PL ? l / ylines : 0, y = l - p * ylines;
        double a = 0.0;
#pragma unroll
        for (int j = 0; j < M; ++j) a += A[p][i][j] * cy[y][j];
        gi[l][i] = a;
    }
    __syncthreads();
    for (int t = tid; t < lines * (M + 1); t += KLF_THREADS) {
        const int l = t / (M + 1), k = t % (M + 1);
        double a = 0.0;
#pragma unroll
        for (int i = 0; i < M; ++i) a += gi[l][i] * klf_cheb.t[i + 1][k];
        *reinterpret_cast<float2*>(&gam[l][2 * k]) = make_float2((float)a, (float)a);
    }
    __syncthreads();
    if (row0 >= G.ty || x0 >= nx) return;
    const float* cl = cx + (VEC ? 4 * col : col);
    const klf_u64 c01 = klf_pack2(cl[0], cl[xstep]), c23 = klf_pack2(cl[2 * xstep], cl[3 * xstep]);
    const bool in1 = x0 + xstep < nx, in2 = x0 + 2 * xstep < nx, in3 = x0 + 3 * xstep < nx;
    float* out = nu + (((long long)b * nz + iz) * ny + y0 + row0) * nx + x0;
    const size_t step = (size_t)G.ty * nx;
    for (int row = row0; row < lines; row += G.ty, out += step) {
        klf_u64 g2[GS / 2];
        const ulonglong2* gp = reinterpret_cast<const ulonglong2*>(&gam[row][0]);
#pragma unroll
        for (int k = 0; k < GS / 4; ++k) { const ulonglong2 t = gp[k]; g2[2 * k] = t.x; g2[2 * k + 1] = t.y; }
        klf_u64 e01 = g2[M], e23 = g2[M];
#pragma unroll
        for (int k = M - 1; k >= 0; --k) { e01 = klf_fma2(e01, c01, g2[k]); e23 = klf_fma2(e23, c23, g2[k]); }
        float e0, e1, e2, e3;
        klf_unpack2(e01, e0, e1);
        klf_unpack2(e23, e2, e3);
        if constexpr (VEC) {
            *reinterpret_cast<float4*>(out) = make_float4(klf_ex2(e0), klf_ex2(e1), klf_ex2(e2), klf_ex2(e3));
        } else {
            out[0] = klf_ex2(e0);
            if (in1) out[xstep] = klf_ex2(e1);
            if (in2) out[2 * xstep] = klf_ex2(e2);
            if (in3) out[3 * xstep] = klf_ex2(e3);
        }
    }
}

template <bool VEC, bool PL>
cudaError_t launch_kl_field_m(const dn_grid& g, int nz, int m, const float* kl_w, float* nu, const KlfGeo& G, dim3 grid, cudaStream_t s) {
    const dim3 block(KLF_THREADS);
    switch (m) {
        case 1: return launch_dependent(kl_field_kernel<1, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 2: return launch_dependent(kl_field_kernel<2, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 3: return launch_dependent(kl_field_kernel<3, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 4: return launch_dependent(kl_field_kernel<4, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 5: return launch_dependent(kl_field_kernel<5, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 6: return launch_dependent(kl_field_kernel<6, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 7: return launch_dependent(kl_field_kernel<7, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
        case 8: return launch_dependent(kl_field_kernel<8, VEC, PL>, grid, block, 0, s, g.dim, g.nx, g.ny, nz, kl_w, nu, G);
    }
    return cudaErrorInvalidValue;
}

template <bool VEC>
cudaError_t launch_kl_field_vec(const dn_grid& g, int nz, int batch, int m, const float* kl_w, float* nu, cudaStream_t s) {
    const int quads = (g.nx + 3) / 4, strips = (quads + KLF_THREADS - 1) / KLF_THREADS;
    KlfGeo G{};
    G.tx = (quads + strips - 1) / strips;
    G.ty = KLF_THREADS / G.tx;
    // the more lines, the fewer blocks prepare the same weights; but enough blocks to keep every SM writing (1024^2 x 32 with
    // 64, 32 and 16 lines: 30.5, 23.4 and 21.2 us), and a few lines for each thread (257^2 x 64 with 8 lines, 3 at a time:
    // 9.9 us, with 29: 7.5)
    const long long want = 8ll * sm_count();
    for (int most = KLF_LINES; ; most /= 2) {
        G.ychunks = (g.ny + most - 1) / most;
        G.lines = (g.ny + G.ychunks - 1) / G.ychunks;
        if (most <= 8 * G.ty || most <= 8 || (long long)G.ychunks * nz * strips * batch >= want) break;
    }
    // planes of few lines share a block as long as that leaves a round of blocks (33 x 8 x 33 x 512, m = 1: 43.7 -> 7.9 us, 128 x 3 x
    // 20 x 512, m = 2: 31.7 -> 7.1); fewer blocks than two rounds are faster with a plane each (64 x 8 x 64, m = 8: 2.4 against 6.9)
    const long long blocks = (long long)G.ychunks * nz * strips * batch;
    if (nz > 1 && 2 * g.ny <= 2 * KLF_LINES && blocks >= 2 * want) {
        int most = 2 * KLF_LINES / g.ny;
        if (most > KLF_PLANES) most = KLF_PLANES;
        if (most > blocks / want) most = (int)(blocks / want);
        const int n = (nz + most - 1) / most;
        G.planes = (nz + n - 1) / n;
        G.lines = G.planes * g.ny;
        return launch_kl_field_m<VEC, true>(g, nz, m, kl_w, nu, G, dim3((unsigned)((nz + G.planes - 1) / G.planes), strips, batch), s);
    }
    return launch_kl_field_m<VEC, false>(g, nz, m, kl_w, nu, G, dim3((unsigned)(G.ychunks * nz), strips, batch), s);
}

__global__ void apply_bc_kernel(long long lines, long long lines_per_sample, int nx, float v0, float v1,
                                const float* __restrict__ v0_b, const float* __restrict__ v1_b,
                                float* __restrict__ field) {
    const long long line = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (line >= lines) return;
    if (v0_b) v0 = v0_b[line / lines_per_sample];
    if (v1_b) v1 = v1_b[line / lines_per_sample];
    field[line * nx] = v0;
    field[line * nx + nx - 1] = v1;
}

}  // namespace

static TableArgs table_args(const Params& P, const float* kl_w, float* ckl, float* const cg[3], float* const cn[3], long long& total) {
    TableArgs A{};
    A.dim = P.dim; A.m = P.m; A.batch = P.batch;
    A.n[0] = P.nx; A.n[1] = P.ny; A.n[2] = P.nz;
    total = (long long)P.batch;
    for (int a = 0; a < P.dim; ++a) total *= P.m;
    for (int a = 0; a < 3; ++a) {
        A.gstride[a] = P.gstride[a]; A.cg[a] = cg[a];
        A.nstride[a] = P.nstride[a]; A.cn[a] = cn[a];
        if (a < P.dim) total += (long long)P.m * (P.gstride[a] + P.nstride[a]);
    }
    A.kl_w = kl_w; A.ckl = ckl;
    return A;
}

cudaError_t launch_tables(const Params& P, const float* kl_w, float* ckl, float* const cg[3], float* const cn[3],
                          cudaStream_t s, float* rowpoly, int rowpoly_stride, bool rowpoly_nodes) {
    long long total;
    TableArgs A = table_args(P, kl_w, ckl, cg, cn, total);
    A.rowpoly = (P.dim == 2) ? rowpoly : nullptr; A.rp_gs = rowpoly_stride; A.rp_nodes = rowpoly_nodes ? 1 : 0;
    if (A.rowpoly) total += 2ll * P.batch * (P.ny - (rowpoly_nodes ? 0 : 1));
    const int threads = 128;
    const dim3 grid((unsigned)((total + threads - 1) / threads));
    switch (A.rowpoly ? P.m : DN_MAX_KL_MODES) {       // the loop bound matters to the row polynomials only
        case 1: return launch_dependent(tables_kernel<1>, grid, dim3(threads), 0, s, A);
        case 2: return launch_dependent(tables_kernel<2>, grid, dim3(threads), 0, s, A);
        case 3: return launch_dependent(tables_kernel<3>, grid, dim3(threads), 0, s, A);
        case 4: return launch_dependent(tables_kernel<4>, grid, dim3(threads), 0, s, A);
        case 5: return launch_dependent(tables_kernel<5>, grid, dim3(threads), 0, s, A);
        case 6: return launch_dependent(tables_kernel<6>, grid, dim3(threads), 0, s, A);
        case 7: return launch_dependent(tables_kernel<7>, grid, dim3(threads), 0, s, A);
    }
    return launch_dependent(tables_kernel<DN_MAX_KL_MODES>, grid, dim3(threads), 0, s, A);
}

template <int M, bool NODES, bool ALL>
static cudaError_t launch_lines3d_m(const TableArgs& A, long long total, float* lines, cudaStream_t s) {
    const int chunks = (A.n[1] - (NODES ? 0 : 1) + LINE_THREADS - 1) / LINE_THREADS, planes = A.n[2] - (NODES ? 0 : 1);
    const long long blocks = (long long)chunks * planes * A.batch + (ALL ? (total + LINE_THREADS - 1) / LINE_THREADS : 0);
    return launch_dependent(lines3d_kernel<M, NODES, ALL>, dim3((unsigned)blocks), dim3(LINE_THREADS), 0, s, A, chunks, planes, lines);
}

cudaError_t launch_lines3d(const Params& P, const float* kl_w, float* ckl, float* const cg[3], float* const cn[3], float* lines, bool all, cudaStream_t s) {
    long long total;
    const TableArgs A = table_args(P, kl_w, ckl, cg, cn, total);
    const bool nodes = P.nu_mode == DN_NU_KL_NODAL;
    switch (P.m) {
#define DN_LINES(m) case m: return all ? (nodes ? launch_lines3d_m<m, true, true>(A, total, lines, s) : launch_lines3d_m<m, false, true>(A, total, lines, s)) \
                                       : (nodes ? launch_lines3d_m<m, true, false>(A, total, lines, s) : launch_lines3d_m<m, false, false>(A, total, lines, s));
        DN_LINES(1) DN_LINES(2) DN_LINES(3) DN_LINES(4) DN_LINES(5) DN_LINES(6) DN_LINES(7) DN_LINES(8)
#undef DN_LINES
    }
    return cudaErrorInvalidValue;
}

// the tile and chunk seams of a 3D kernel that leaves them in P.seam and P.zseam, added to P.r; J: and the energies finished
cudaError_t launch_seam_fixup3(const Params& P, int Ry, int ntile, int Z, int nchunk, float* J, cudaStream_t s) {
    const bool vec = P.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(P.r) & 15u) == 0;
    SeamArgs A{};
    A.nxv = vec ? P.nx / 4 : P.nx; A.ny = P.ny; A.nz = P.nz; A.batch = P.batch;
    A.Ry = Ry; A.ntile = ntile; A.Z = Z; A.nchunk = nchunk;
    A.nA = (long long)P.batch * (ntile - 1) * P.nz * A.nxv;
    A.nB = (long long)P.batch * (nchunk - 1) * P.ny * A.nxv;
    A.samples = J ? P.batch : 0; A.nblk = P.nblk; A.partials = P.partials; A.J = J;
    if (A.nA + A.nB + A.samples == 0) return cudaSuccess;
    const dim3 grid((unsigned)(A.samples + (A.nA + A.nB + FIN_THREADS - 1) / FIN_THREADS));
    if (vec)
        return launch_dependent(seam_fixup3_kernel<float4>, grid, dim3(FIN_THREADS), 0, s, reinterpret_cast<float4*>(P.r),
                                reinterpret_cast<const float4*>(P.seam), reinterpret_cast<const float4*>(P.zseam), A);
    return launch_dependent(seam_fixup3_kernel<float>, grid, dim3(FIN_THREADS), 0, s, P.r, (const float*)P.seam, (const float*)P.zseam, A);
}

cudaError_t launch_finalize(const double* partials, int nblk, int batch, float* J, cudaStream_t s) {
    return launch_dependent(finalize_kernel, dim3((unsigned)batch), dim3(FIN_THREADS), 0, s, partials, nblk, J);
}

cudaError_t launch_kl_field(const dn_grid& g, int batch, int m, const float* kl_w, float* nu, cudaStream_t s) {
    const int nz = (g.dim == 3) ? g.nz : 1;
    const bool vec = (g.nx % 4 == 0) && ((reinterpret_cast<uintptr_t>(nu) & 15u) == 0);
    return vec ? launch_kl_field_vec<true>(g, nz, batch, m, kl_w, nu, s) : launch_kl_field_vec<false>(g, nz, batch, m, kl_w, nu, s);
}

cudaError_t launch_apply_bc(const dn_grid& g, int batch, float b0, float b1, int mode, float* field, cudaStream_t s,
                            const float* b0_b, const float* b1_b) {
    const long long per_sample = (long long)g.ny * ((g.dim == 3) ? g.nz : 1);
    const long long lines = (long long)batch * per_sample;
    const int threads = 256;
    apply_bc_kernel<<<(unsigned)((lines + threads - 1) / threads), threads, 0, s>>>(
        lines, per_sample, g.nx, mode == 0 ? b0 : 0.0f, mode == 0 ? b1 : 0.0f, mode == 0 ? b0_b : nullptr,
        mode == 0 ? b1_b : nullptr, field);
    return cudaGetLastError();
}

}  // namespace dn
