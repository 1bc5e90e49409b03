// Matrix-free conjugate gradients on K(nu) u = F with the Dirichlet faces held at their values: the
// "conventional solver" side of the paper's comparison ("Mathematical preliminaries": the PDE is normally
// discretised and solved; the appendix compares the generator's fields with such solutions), built on the
// same fused energy+residual kernel that scores the generator.  Its result u* is the minimiser of the
// energy J, the lower bound of the loss any generator can reach.
//
// Per sample b (all samples advance together, each with its own scalars; Jacobi preconditioner D = diag K):
//     r = F - K u,  z = D^-1 r,  p = z,  rho = r.z
//     repeat:  q = K p;  alpha = rho / p.q;  u += alpha p;  r -= alpha q;  z = D^-1 r;
//              rho' = r.z;  beta = rho' / rho;  p = z + beta p;  rho = rho'
// K p is the fused kernel applied to p with zero forcing and zero boundary values (p vanishes on the
// Dirichlet faces), and p.q = 2 J(p) comes from the energy that kernel computes anyway, so an iteration is
// the fused kernel plus two streaming kernels (update + dot, new direction) and two one-block-per-sample
// scalar kernels.  Dot products are summed in fp64 in a fixed order.  A sample whose residual norm has
// dropped below rtol times its initial value is frozen (alpha = 0); the iteration count is fixed by the
// caller, so nothing is read back and the whole solve is one stream of launches.
//
// Samples that fit the shared memory of a few SMs (2D grids of up to 257 x 257 nodes, 3D grids of up to 49^3) are solved
// by one thread-block cluster each, all iterations in one launch: see cg_cluster_kernel.
#include <type_traits>

#include "dn_internal.cuh"

namespace dn {
namespace {

constexpr int CG_THREADS = 256;
constexpr int CG_VEC = 4;                    // floats per thread per trip
constexpr int CG_BLOCK_NODES = CG_THREADS * CG_VEC * 4;

struct CgScalars {                           // per sample, in the workspace
    double rho, rr0, rr;
    float alpha, beta;
    int active, iters;
};

__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double sa[CG_THREADS / 32], sb[CG_THREADS / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) { sa[threadIdx.x >> 5] = a; sb[threadIdx.x >> 5] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x = 0.0, y = 0.0;
        for (int w = 0; w < CG_THREADS / 32; ++w) { x += sa[w]; y += sb[w]; }
        a = x; b = y;
    }
}

// r = -r (the fused kernel returns K u - F), p = z = dinv r; partial sums of r.z and r.r per block.
__global__ void __launch_bounds__(CG_THREADS) cg_init_kernel(long long nodes, int nblk, float* __restrict__ r,
                                                             const float* __restrict__ dinv, float* __restrict__ p,
                                                             double* __restrict__ partials) {
    const int b = blockIdx.y;
    const long long base = (long long)b * nodes;
    const long long lo = (long long)blockIdx.x * CG_BLOCK_NODES;
    const long long hi = min(lo + (long long)CG_BLOCK_NODES, nodes);
    double s_rz = 0.0, s_rr = 0.0;
    for (long long i = lo + threadIdx.x; i < hi; i += CG_THREADS) {
        const float rv = -r[base + i];
        const float zv = rv * dinv[base + i];
        r[base + i] = rv;
        p[base + i] = zv;
        s_rz += (double)(rv * zv);
        s_rr += (double)(rv * rv);
    }
    block_sum2(s_rz, s_rr);
    if (threadIdx.x == 0) {
        partials[2 * ((long long)b * nblk + blockIdx.x)] = s_rz;
        partials[2 * ((long long)b * nblk + blockIdx.x) + 1] = s_rr;
    }
}

__device__ __forceinline__ void sum_pairs(const double* __restrict__ p, int n, double& a, double& b) {
    double x = 0.0, y = 0.0;
    for (int i = threadIdx.x; i < n; i += CG_THREADS) { x += p[2 * i]; y += p[2 * i + 1]; }
    block_sum2(x, y);
    a = x; b = y;                            // valid in thread 0
}

__global__ void __launch_bounds__(CG_THREADS) cg_start_kernel(const double* __restrict__ partials, int nblk,
                                                              CgScalars* __restrict__ sc) {
    double rz, rr;
    sum_pairs(partials + 2ll * blockIdx.x * nblk, nblk, rz, rr);
    if (threadIdx.x == 0) {
        CgScalars s;
        s.rho = rz; s.rr0 = rr; s.rr = rr; s.alpha = 0.f; s.beta = 0.f; s.iters = 0;
        s.active = (rr > 0.0 && rz > 0.0) ? 1 : 0;
        sc[blockIdx.x] = s;
    }
}

// alpha = rho / p.q with p.q = 2 (diffusion part - load part) of the fused kernel's energy of p.
__global__ void __launch_bounds__(CG_THREADS) cg_alpha_kernel(const double* __restrict__ op_partials, int op_nblk,
                                                              CgScalars* __restrict__ sc) {
    double d, l;
    sum_pairs(op_partials + 2ll * blockIdx.x * op_nblk, op_nblk, d, l);
    if (threadIdx.x == 0) {
        CgScalars& s = sc[blockIdx.x];
        const double pq = 2.0 * (d - l);
        s.alpha = (s.active && pq > 0.0) ? (float)(s.rho / pq) : 0.0f;
        if (!(pq > 0.0)) s.active = 0;
    }
}

// u += alpha p, r -= alpha q; partial sums of r.z (z = dinv r) and r.r.
__global__ void __launch_bounds__(CG_THREADS) cg_update_kernel(long long nodes, int nblk, float* __restrict__ u,
                                                               float* __restrict__ r, const float* __restrict__ p,
                                                               const float* __restrict__ q,
                                                               const float* __restrict__ dinv,
                                                               const CgScalars* __restrict__ sc,
                                                               double* __restrict__ partials) {
    const int b = blockIdx.y;
    const float alpha = sc[b].alpha;
    const long long base = (long long)b * nodes;
    const long long lo = (long long)blockIdx.x * CG_BLOCK_NODES;
    const long long hi = min(lo + (long long)CG_BLOCK_NODES, nodes);
    double s_rz = 0.0, s_rr = 0.0;
    if (alpha != 0.0f) {
        for (long long i = lo + threadIdx.x; i < hi; i += CG_THREADS) {
            const float pv = p[base + i], qv = q[base + i];
            const float rv = fmaf(-alpha, qv, r[base + i]);
            u[base + i] = fmaf(alpha, pv, u[base + i]);
            r[base + i] = rv;
            const float zv = rv * dinv[base + i];
            s_rz += (double)(rv * zv);
            s_rr += (double)(rv * rv);
        }
    }
    block_sum2(s_rz, s_rr);
    if (threadIdx.x == 0) {
        partials[2 * ((long long)b * nblk + blockIdx.x)] = s_rz;
        partials[2 * ((long long)b * nblk + blockIdx.x) + 1] = s_rr;
    }
}

__global__ void __launch_bounds__(CG_THREADS) cg_beta_kernel(const double* __restrict__ partials, int nblk, double rtol2,
                                                             CgScalars* __restrict__ sc) {
    double rz, rr;
    sum_pairs(partials + 2ll * blockIdx.x * nblk, nblk, rz, rr);
    if (threadIdx.x == 0) {
        CgScalars& s = sc[blockIdx.x];
        if (s.active && s.alpha != 0.0f) {
            s.beta = (float)(rz / s.rho);
            s.rho = rz; s.rr = rr; s.iters += 1;
            if (rr <= rtol2 * s.rr0 || !(rz > 0.0)) s.active = 0;
        } else {
            s.active = 0; s.alpha = 0.0f;    // frozen: u and r no longer change
        }
    }
}

// p = dinv r + beta p
__global__ void __launch_bounds__(CG_THREADS) cg_direction_kernel(long long nodes, const float* __restrict__ r,
                                                                  const float* __restrict__ dinv, float* __restrict__ p,
                                                                  const CgScalars* __restrict__ sc) {
    const int b = blockIdx.y;
    if (!sc[b].active) return;
    const float beta = sc[b].beta;
    const long long base = (long long)b * nodes;
    const long long lo = (long long)blockIdx.x * CG_BLOCK_NODES;
    const long long hi = min(lo + (long long)CG_BLOCK_NODES, nodes);
    for (long long i = lo + threadIdx.x; i < hi; i += CG_THREADS)
        p[base + i] = fmaf(beta, p[base + i], r[base + i] * dinv[base + i]);
}

// ---- diagonal of K by probing ------------------------------------------------------------------------
// Nodes whose indices agree modulo 3 on every axis share no element, so the fused kernel applied to the
// indicator of one such colour class returns K_ii at the nodes i of that class: 3^dim applications give the
// whole diagonal.  One block per x-row; only the rows of the class (iy, iz congruent to the colour) do work.
// phase 0: e = 1 on the free nodes of the class in this row, 0 elsewhere in the row (e is zero outside the class rows).
// phase 1: dinv = 1 / (K e) on the free nodes of the class, 0 on its Dirichlet nodes; the row of e is cleared again.
__global__ void __launch_bounds__(CG_THREADS) cg_probe_kernel(int nx, int ny, int nz, int colour, int phase,
                                                              float* __restrict__ e, const float* __restrict__ q,
                                                              float* __restrict__ dinv) {
    const long long row = blockIdx.x;
    const int iy = (int)(row % ny), iz = (int)((row / ny) % nz);
    const int cx = colour % 3, cy = (colour / 3) % 3, cz = colour / 9;
    if (iy % 3 != cy || iz % 3 != cz) return;
    const long long base = row * nx;
    for (int ix = threadIdx.x; ix < nx; ix += CG_THREADS) {
        const bool mine = ix % 3 == cx, face = ix == 0 || ix == nx - 1;
        if (phase == 0) {
            e[base + ix] = (mine && !face) ? 1.0f : 0.0f;
        } else {
            if (mine) dinv[base + ix] = face ? 0.0f : 1.0f / q[base + ix];
            e[base + ix] = 0.0f;
        }
    }
}

__global__ void cg_report_kernel(const CgScalars* __restrict__ sc, int batch, float* __restrict__ relres,
                                 int32_t* __restrict__ iters) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= batch) return;
    if (relres) relres[b] = sc[b].rr0 > 0.0 ? (float)sqrt(sc[b].rr / sc[b].rr0) : 0.0f;
    if (iters) iters[b] = sc[b].iters;
}

// ---- a sample per cluster ---------------------------------------------------------------------------------
// A sample is cut into C slabs of slices (rows in 2D, planes in 3D), one per block of a cluster, and every iteration runs
// inside the cluster: the direction p of a slab and the slices next to it live in shared memory (a block writes its edge
// slices into its neighbours' memory), the dot products are exchanged the same way, and three cluster barriers per iteration
// take the place of five launches.  The operator is the assembled stencil: the couplings K_ij of a node with its forward
// neighbours (4 in 2D, 13 in 3D; the backward ones are those neighbours' own), in difference form,
//     (K p)_i = d_i p_i + sum_j K_ij (p_j - p_i),      d_i = sum over the free nodes j of K_ij  (zero away from the faces),
// so that it loses no more to cancellation than the element form.  The couplings are read off the probing that gives the
// diagonal (no second element routine).  A cluster stops when its sample is frozen; samples do not wait for one another.
// 2D: couplings in shared memory, u, r, q, 1/diag in registers (NPT nodes per thread).  3D: q and r in shared memory, the
// couplings are streamed from L2.  256^2 x 16 nodes, 956 iterations asked for, about 540 needed: 25.2 ms by
// launches per iteration, 4.2 ms here.
// 2D: a thread owns one free column x of a contiguous group of rows and walks up it, so that p and the coupling of the row
// below stay in registers (10 shared-memory reads per node instead of 17); groups of nx - 2 threads, at most CGC_THREADS.
constexpr int CGC_THREADS = 512;             // 2D: up to 128 registers
constexpr int CGC_THREADS3 = 1024;           // 3D: latency of the streamed couplings
constexpr int CGC_PORTABLE = 8;              // blocks per cluster that every device of the architecture can schedule
constexpr int cgc_max(int dim) { return dim == 3 ? 16 : CGC_PORTABLE; }
constexpr size_t CGC_SMEM = kMaxBlockShared;
constexpr int CGC_UREG = 17;                 // rows per thread up to which u stays in registers

struct CgCluster {
    int nx, slice, nslice, C, nf, max_iters; // nodes per slice, slices per sample, blocks per cluster, forward couplings
    int groups;                              // 2D: row groups per block
    long long nodes;
    int off[13];                             // index offset of the forward neighbours
    const float* coef;                       // [B][nf + 2][nodes]: couplings, 1 / diagonal (0 on the faces), d
    float* u;
    const float* r0;                         // K u - F
    double rtol2;
    float* relres;
    int32_t* iters;
};

__device__ __forceinline__ unsigned cgc_remote(const void* local, int rank) {      // the same address in another block's memory
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cgc_store(unsigned remote, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory"); }
__device__ __forceinline__ void cgc_store(unsigned remote, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory"); }
__device__ __forceinline__ void cgc_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// First slice of block `rank`.
__host__ __device__ inline int cgc_first(int nslice, int C, int rank) { return (int)((long long)nslice * rank / C); }

template <int DIM, int NPT>
__global__ void __launch_bounds__(DIM == 2 ? CGC_THREADS : CGC_THREADS3, 1) cg_cluster_kernel(const CgCluster A) {
    extern __shared__ __align__(16) double cgc_smem[];
    constexpr bool REGS = (DIM == 2);
    constexpr bool UREG = REGS && NPT <= CGC_UREG;       // u in registers too, else updated in L2
    constexpr int NF = (DIM == 2) ? 4 : 13, CGC_WARPS = (DIM == 2 ? CGC_THREADS : CGC_THREADS3) / 32;
    const int tid = threadIdx.x, C = A.C, T = blockDim.x, NW = T / 32;
    const int b = blockIdx.x / C, rank = blockIdx.x % C;
    const int s0 = cgc_first(A.nslice, C, rank), s1 = cgc_first(A.nslice, C, rank + 1);
    const int slice = A.slice, n = (s1 - s0) * slice, pad = (A.nx + 4) / 4 * 4;
    double* red = cgc_smem;                              // [3][C][CGC_WARPS]: p.q, r.z, r.r of every warp of the cluster
    float* p = reinterpret_cast<float*>(red + 3 * C * CGC_WARPS) + pad;       // slices s0 - 1 .. s1
    float* pown = p + slice;
    const int plen = n + 2 * slice + 2 * pad;
    float* cs = p + plen - pad;                          // 2D: couplings of slices s0 - 1 .. s1 - 1, then d next to the faces; 3D: q, r
    const int clen = n + slice + 4;
    const long long g0 = (long long)s0 * slice;          // first own node in the sample
    const float* co = A.coef + (long long)b * (NF + 2) * A.nodes;
    float* ug = A.u + (long long)b * A.nodes + g0;
    const float* rg = A.r0 + (long long)b * A.nodes + g0;
    const float* dinv = co + (long long)NF * A.nodes + g0;
    const float* dg = dinv + A.nodes;
    float* qs = cs;
    float* rs = cs + n;

    for (int i = tid; i < plen; i += T) p[i - pad] = 0.f;
    for (int i = tid; i < 3 * C * CGC_WARPS; i += T) red[i] = 0.0;
    if constexpr (REGS) {
        for (int o = 0; o < NF; ++o)
            for (int i = tid; i < clen; i += T) {
                const long long gi = g0 - slice + i - 4;
                cs[o * clen + i] = (gi >= 0 && gi < g0 + n) ? co[(long long)o * A.nodes + gi] : 0.f;
            }
        for (int i = tid; i < 2 * (s1 - s0); i += T) cs[NF * clen + i] = dg[(i >> 1) * A.nx + ((i & 1) ? A.nx - 2 : 1)];
    }
    const float* cw = cs + 4 + slice;                    // 2D: couplings of own node 0
    const float* ds = cs + NF * clen;
    // 2D: this thread's column and rows; first own node and how many
    const int nx = A.nx, grp = REGS ? tid / (nx - 2) : 0, rows = s1 - s0;        // (2D: at least 3 columns)
    const int j0 = REGS && grp < A.groups ? cgc_first(rows, A.groups, grp) : 0;
    const int mine = REGS && grp < A.groups ? cgc_first(rows, A.groups, grp + 1) - j0 : 0;
    const int x = tid - grp * (nx - 2) + 1, l0 = j0 * nx + x;
    const float dsel = (x == 1 || x == nx - 2) ? 1.f : 0.f;        // d is zero elsewhere
    const float* dp = ds + 2 * j0 + (x == nx - 2 && x != 1 ? 1 : 0);

    float ur[UREG ? NPT : 1], rr_[REGS ? NPT : 1], qr[REGS ? NPT : 1], dr[REGS ? NPT : 1];
    // f(k, l): the own nodes l of this thread.  2D: NPT or NPT - 1 rows (or none).
    auto each = [&](auto f) {
        if constexpr (REGS) {
            if (mine > 0) {
                int l = l0, step = nx;
                asm volatile("" : "+r"(l), "+r"(step));  // else every row's address is kept in a register across the solve
#pragma unroll
                for (int k = 0; k < NPT; ++k, l += step) if (k < NPT - 1 || mine == NPT) f(k, l);
            }
        } else {
            for (int l = tid; l < n; l += T) f(0, l);
        }
    };
    // sums of (a, c) over the cluster, in a fixed order: every warp sends its sums to every block, every warp adds them all
    const int lane = tid & 31, warp = tid >> 5;
    auto cluster_sum = [&](double a, double c, auto two, double& sa, double& sc) {
        constexpr bool TWO = decltype(two)::value;       // slots 1 and 2, else slot 0
        const int S = C * CGC_WARPS;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            if (TWO) c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane < C) {
            const unsigned to = cgc_remote(red + (TWO ? S : 0) + rank * CGC_WARPS + warp, lane);
            cgc_store(to, a);
            if (TWO) cgc_store(to + 8u * S, c);
        }
        cgc_barrier();
        sa = 0.0; sc = 0.0;
        for (int i = lane; i < C * CGC_WARPS; i += 32) {
            sa += red[(TWO ? S : 0) + i];
            if (TWO) sc += red[2 * S + i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
            if (TWO) sc += __shfl_xor_sync(0xffffffffu, sc, o);
        }
    };
    const unsigned up = (rank + 1 < C) ? cgc_remote(p, rank + 1) : 0u;                           // its slice s0 - 1
    const unsigned down = (rank > 0) ? cgc_remote(p + (long long)(s0 - cgc_first(A.nslice, C, rank > 0 ? rank - 1 : 0) + 1) * slice, rank - 1) : 0u;   // its slice s1
    auto put_p = [&](int k, int l, float v) {
        pown[l] = v;
        if (REGS ? (k == 0 && j0 == 0 && rank > 0) : (l < slice && rank > 0)) cgc_store(down + 4u * l, v);
        const int e = l - (n - slice);
        if (REGS ? (k >= NPT - 2 && e >= 0 && rank + 1 < C) : (e >= 0 && rank + 1 < C)) cgc_store(up + 4u * e, v);
    };
    using One = std::false_type;
    using Two = std::true_type;

    cgc_barrier();                                       // every block of the cluster runs, its p and red are zeroed
    double rho, rr0, rr;
    {
        double a = 0.0, c = 0.0;
        each([&](int k, int l) {
            const float rv = -rg[l], di = dinv[l], z = rv * di;
            if constexpr (UREG) ur[k] = ug[l];
            if constexpr (REGS) { rr_[k] = rv; dr[k] = di; } else rs[l] = rv;
            put_p(k, l, z);
            a += (double)(rv * z); c += (double)(rv * rv);
        });
        cluster_sum(a, c, Two{}, rho, rr0);              // (its barrier also publishes p)
        rr = rr0;
    }
    int it = 0;
    const bool active = rr0 > 0.0 && rho > 0.0;
    for (int step = 0; active && step < A.max_iters; ++step) {
        double pq = 0.0, dummy;
        if constexpr (REGS) {
            if (mine > 0) {
                // walk up the column: p of the row below, this row and the row above; couplings N, NE, NW of the row below
                int l = l0, up1 = nx;
                asm volatile("" : "+r"(l), "+r"(up1));   // (as above)
                const float *pp = pown + l, *c = cw + l;
                const float *c1 = c + clen, *c2 = c1 + clen, *c3 = c2 + clen, *dk = dp;
                float bl = pp[-up1 - 1], bc = pp[-up1], br = pp[-up1 + 1], ml = pp[-1], mc = pp[0], mr = pp[1];
                float cn = c2[-up1];             // N of the node below
#pragma unroll
                for (int k = 0; k < NPT; ++k) {
                    if (k < NPT - 1 || mine == NPT) {
                        const float al = pp[up1 - 1], ac = pp[up1], ar = pp[up1 + 1];
                        float q = (dsel * *dk) * mc;
                        q = fmaf(c[0], mr - mc, q);                          // E, and W = E of the node on the left
                        q = fmaf(c[-1], ml - mc, q);
                        q = fmaf(c3[-up1 - 1], bl - mc, q);          // SW, S, SE
                        q = fmaf(cn, bc - mc, q);
                        q = fmaf(c1[-up1 + 1], br - mc, q);
                        cn = c2[0];
                        q = fmaf(c1[0], al - mc, q);                       // NW, N, NE
                        q = fmaf(cn, ac - mc, q);
                        q = fmaf(c3[0], ar - mc, q);
                        qr[k] = q;
                        pq += (double)(mc * q);
                        bl = ml; bc = mc; br = mr; ml = al; mc = ac; mr = ar;
                        pp += up1; c += up1; c1 += up1; c2 += up1; c3 += up1; dk += 2;
                    }
                }
            }
        } else {
            each([&](int k, int l) {
                const float pc = pown[l];
                float q = dg[l] * pc;
                const long long g = g0 + l;
#pragma unroll
                for (int o = 0; o < NF; ++o) {
                    const int f = A.off[o];
                    const float* c = co + (long long)o * A.nodes + g;
                    q = fmaf(__ldg(c), pown[l + f] - pc, q);
                    q = fmaf(g >= f ? __ldg(c - f) : 0.f, pown[l - f] - pc, q);
                }
                qs[l] = q;
                pq += (double)(pc * q);
            });
        }
        double s_pq;
        cluster_sum(pq, 0.0, One{}, s_pq, dummy);
        const float alpha = s_pq > 0.0 ? (float)(rho / s_pq) : 0.f;
        if (!(s_pq > 0.0) || alpha == 0.f) break;        // the same in every block
        double a = 0.0, c = 0.0;
        each([&](int k, int l) {
            const float pc = pown[l];
            float rv, z;
            if constexpr (UREG) ur[k] = fmaf(alpha, pc, ur[k]);
            else if constexpr (!REGS) ug[l] = fmaf(alpha, pc, ug[l]);
            if constexpr (REGS) {
                rv = fmaf(-alpha, qr[k], rr_[k]);
                rr_[k] = rv;
                z = rv * dr[k];
            } else {
                rv = fmaf(-alpha, qs[l], rs[l]);
                rs[l] = rv;
                z = rv * __ldg(dinv + l);
            }
            a += (double)(rv * z); c += (double)(rv * rv);
        });
        if constexpr (REGS && !UREG) each([&](int k, int l) { qr[k] = ug[l]; });      // on their way during the exchange
        double rz;
        cluster_sum(a, c, Two{}, rz, rr);
        if constexpr (REGS && !UREG) each([&](int k, int l) { ug[l] = fmaf(alpha, pown[l], qr[k]); });
        ++it;
        const float beta = (float)(rz / rho);
        rho = rz;
        if (rr <= A.rtol2 * rr0 || !(rz > 0.0)) break;
        each([&](int k, int l) {
            const float z = REGS ? rr_[k] * dr[k] : rs[l] * __ldg(dinv + l);
            put_p(k, l, fmaf(beta, pown[l], z));
        });
        cgc_barrier();                                   // p and the slices next to the slab are complete
    }
    if constexpr (UREG) each([&](int k, int l) { ug[l] = ur[k]; });
    if (rank == 0 && tid == 0) {
        if (A.relres) A.relres[b] = rr0 > 0.0 ? (float)sqrt(rr / rr0) : 0.0f;
        if (A.iters) A.iters[b] = it;
    }
}

// Probing for the couplings, `group` colour classes at a time: field b * group + c is the indicator of class first + c on
// the free nodes.
__global__ void __launch_bounds__(CG_THREADS) cg_colours_kernel(int nx, int ny, int nz, int group, int first, long long total, float* __restrict__ e) {
    const long long t = (long long)blockIdx.x * CG_THREADS + threadIdx.x;      // (field, iz, iy, ix)
    if (t >= total) return;
    const int ix = (int)(t % nx), iy = (int)((t / nx) % ny), iz = (int)((t / ((long long)nx * ny)) % nz);
    const int colour = first + (int)((t / ((long long)nx * ny * nz)) % group);
    e[t] = (ix % 3 + 3 * (iy % 3) + 9 * (iz % 3) == colour && ix > 0 && ix < nx - 1) ? 1.0f : 0.0f;
}

// q = K applied to those fields: every node has one node of every class among itself and its neighbours, so q holds all
// its couplings.
__global__ void __launch_bounds__(CG_THREADS) cg_couplings_kernel(int nx, int ny, int nz, int group, int first, int nf, long long total,
                                                                  const float* __restrict__ q, float* __restrict__ coef) {
    const long long t = (long long)blockIdx.x * CG_THREADS + threadIdx.x;      // (b, iz, iy, ix)
    if (t >= total) return;
    const long long nodes = (long long)nx * ny * nz, b = t / nodes, i = t - b * nodes;
    const int ix = (int)(i % nx), iy = (int)((i / nx) % ny), iz = (int)(i / ((long long)nx * ny));
    float* co = coef + b * (nf + 2) * nodes + i;
    const float* qi = q + b * group * nodes + i;
    const bool face = ix == 0 || ix == nx - 1, near = ix == 1 || ix == nx - 2;
    float d = first == 0 ? 0.f : co[(nf + 1) * nodes];
    for (int c = 0; c < group; ++c) d += qi[c * nodes];
    co[(nf + 1) * nodes] = (face || (!near && first + group == (nz > 1 ? 27 : 9))) ? 0.f : d;
    const int own = ix % 3 + 3 * (iy % 3) + 9 * (iz % 3) - first;
    if (own >= 0 && own < group) co[nf * nodes] = face ? 0.f : 1.0f / qi[own * nodes];
    for (int o = 0; o < nf; ++o) {                       // forward neighbours: (1,0,0), (-1..1,1,0), (-1..1,-1..1,1)
        const int dx = o == 0 ? 1 : (o - 1) % 3 - 1, dy = o == 0 ? 0 : o < 4 ? 1 : (o - 4) / 3 - 1, dz = o < 4 ? 0 : 1;
        const int jx = ix + dx, jy = iy + dy, jz = iz + dz;
        const bool free = !face && jx > 0 && jx < nx - 1 && jy >= 0 && jy < ny && jz < nz;
        if (!free) { if (first == 0) co[o * nodes] = 0.f; continue; }
        const int colour = jx % 3 + 3 * (jy % 3) + 9 * (jz % 3) - first;
        if (colour >= 0 && colour < group) co[o * nodes] = qi[colour * nodes];
    }
}

long long nodes_of(const dn_problem& p) { return (long long)p.grid.nx * p.grid.ny * (p.grid.dim == 3 ? p.grid.nz : 1); }
int vec_blocks(long long nodes) { return (int)((nodes + CG_BLOCK_NODES - 1) / CG_BLOCK_NODES); }

// Blocks per cluster for a problem whose samples fit one, else 0.
size_t cgc_smem_bytes(const dn_problem& p, int C) {
    const bool d3 = p.grid.dim == 3;
    const int nslice = d3 ? p.grid.nz : p.grid.ny;
    const long long slice = d3 ? (long long)p.grid.nx * p.grid.ny : p.grid.nx;
    const long long n = (nslice + C - 1) / C * slice, pad = (p.grid.nx + 4) / 4 * 4;
    const long long plen = n + 2 * slice + 2 * pad;
    const long long rest = d3 ? 2 * n : 4 * (n + slice + 4) + 2 * ((nslice + C - 1) / C);
    return sizeof(double) * 3 * C * ((d3 ? CGC_THREADS3 : CGC_THREADS) / 32) + sizeof(float) * (size_t)(plen + rest);
}
constexpr int CGC_NPT = 22;                  // most rows per thread in 2D: 43 rows in two groups
int cgc_groups(int nx, int rows) {           // 0: not solved by clusters (rows of two nodes have no free column to give a thread)
    if (nx < 3 || nx - 2 > CGC_THREADS) return 0;
    int g = CGC_THREADS / (nx - 2);
    return g < 1 ? 0 : g > rows ? rows : g;
}
bool cgc_fits(const dn_problem& p, int C) {
    const bool d3 = p.grid.dim == 3;
    const int nslice = d3 ? p.grid.nz : p.grid.ny;
    if (C > nslice || cgc_smem_bytes(p, C) > CGC_SMEM) return false;
    if (d3) return true;
    const int groups = cgc_groups(p.grid.nx, nslice / C);
    return groups >= 1 && (nslice + C - 1) / C <= CGC_NPT * groups;
}
// Whether the samples of a problem are solved by clusters.  In 3D as long as the couplings of all samples (15 fields: 79 MB at
// most) stay in L2, from where every iteration streams them.  Microseconds per iteration, clusters and launches: 24^3 x 90 33 and
// 44, 32^3 x 40 34 and 43, 48^3 x 11 36 and 43; beyond: 24^3 x 128 60 and 52, 32^3 x 64 72 and 51, 48^3 x 64 228 and 151.
constexpr long long CGC_NODES3 = 5ll << 18;
bool cgc_applicable(const dn_problem& p) {
    if (nodes_of(p) > (1 << 18) || (long long)p.batch * 9 > 65535) return false;
    if (p.grid.dim == 3 && nodes_of(p) * p.batch > CGC_NODES3) return false;
    if (p.grid.dim == 3 && !(pair3d_applicable(p) || (p.flags & DN_FORCE_GENERIC))) return false;
    for (int C = 1; C <= CGC_PORTABLE; ++C) if (cgc_fits(p, C)) return true;
    return false;
}

struct CgLayout {
    size_t r, q, p, dinv, partials, scalars, op, op_bytes, op1, op1_bytes, coef, total;
    int chunk;                               // clusters: samples solved together
};

// One launch sequence per iteration: four fields and two fused-kernel workspaces, one for the operator on directions (no nodal
// forcing, aligned scratch fields) and one for the caller's problem (initial residual), which may take another kernel family
// with another layout.
CgLayout lockstep_layout(const dn_problem& p) {
    CgLayout L{};
    const size_t field = align_up(sizeof(float) * (size_t)p.batch * nodes_of(p));
    size_t off = 0;
    L.r = off; off += field;
    L.q = off; off += field;
    L.p = off; off += field;
    L.dinv = off; off += field;
    L.partials = off; off += align_up(sizeof(double) * 2 * (size_t)p.batch * vec_blocks(nodes_of(p)));
    L.scalars = off; off += align_up(sizeof(CgScalars) * (size_t)p.batch);
    dn_problem pop = p;
    pop.f = nullptr;
    L.op_bytes = dn_workspace_bytes(&pop);
    L.op = off; off += align_up(L.op_bytes);
    L.op1_bytes = dn_workspace_bytes(&p);
    L.op1 = off; off += align_up(L.op1_bytes);
    L.total = off;
    return L;
}

// One cluster per sample: the residual of all samples, and for `chunk` samples at a time the couplings, the probes of nine
// colour classes per sample (all in 2D, a third in 3D), their images and the workspace of the operator on them.  As many
// samples at a time as keep the layout about within that of the launches per iteration, or within CGC_SPARE bytes where
// that is more, in chunks of equal size.
constexpr int CGC_GROUP = 9;
constexpr size_t CGC_SPARE = (size_t)512 << 20;
CgLayout cluster_layout(const dn_problem& p, const CgLayout& lockstep) {
    CgLayout L{};
    const int nc = p.grid.dim == 3 ? 15 : 6;
    const size_t nodes = (size_t)nodes_of(p), limit = lockstep.total > CGC_SPARE ? lockstep.total : CGC_SPARE;
    const size_t fixed = sizeof(float) * nodes * p.batch + lockstep.op_bytes + lockstep.op1_bytes;      // the residual, tables and partial sums
    const size_t fit = limit > fixed ? (limit - fixed) / (sizeof(float) * nodes * (2 * CGC_GROUP + nc)) : 0;
    const int most = fit < 1 ? 1 : fit < (size_t)p.batch ? (int)fit : p.batch, chunks = (p.batch + most - 1) / most;
    L.chunk = (p.batch + chunks - 1) / chunks;
    size_t off = 0;
    L.r = off; off += align_up(sizeof(float) * p.batch * nodes);
    L.op1_bytes = dn_workspace_bytes(&p);
    L.op1 = off; off += align_up(L.op1_bytes);
    L.p = off; off += align_up(sizeof(float) * L.chunk * CGC_GROUP * nodes);
    L.q = off; off += align_up(sizeof(float) * L.chunk * CGC_GROUP * nodes);
    L.coef = off; off += align_up(sizeof(float) * L.chunk * nc * nodes);
    dn_problem probe = p;
    probe.f = nullptr;
    const int last = p.batch - (p.batch - 1) / L.chunk * L.chunk;         // the last chunk's kernels may tile differently
    for (int n : {L.chunk, last}) {
        probe.batch = n * CGC_GROUP;
        const size_t b = operator_bytes(probe, CGC_GROUP);
        if (b > L.op_bytes) L.op_bytes = b;
    }
    L.op = off; off += align_up(L.op_bytes);
    L.total = off;
    return L;
}

struct CgPlan { CgLayout lockstep, clusters; };       // clusters.chunk = 0: not solved that way
CgPlan cg_plan(const dn_problem& p) {
    return memo_geometry<CgPlan>(p, sm_count(), [&]() {
        CgPlan pl{};
        pl.lockstep = lockstep_layout(p);
        if (cgc_applicable(p)) pl.clusters = cluster_layout(p, pl.lockstep);
        return pl;
    });
}

typedef void (*CgcKernel)(const CgCluster);
// The kernel compiled for the rows of a thread (2D).
CgcKernel cgc_kernel(bool d3, int npt) {
    if (d3) return cg_cluster_kernel<3, 1>;
    switch (npt) {
#define CGC_CASE(n) case n: return cg_cluster_kernel<2, n>;
        CGC_CASE(1) CGC_CASE(2) CGC_CASE(3) CGC_CASE(4) CGC_CASE(5) CGC_CASE(6) CGC_CASE(7) CGC_CASE(8) CGC_CASE(9) CGC_CASE(10) CGC_CASE(11)
        CGC_CASE(12) CGC_CASE(13) CGC_CASE(14) CGC_CASE(15) CGC_CASE(16) CGC_CASE(17) CGC_CASE(18) CGC_CASE(19) CGC_CASE(20) CGC_CASE(21) CGC_CASE(22)
#undef CGC_CASE
    }
    return nullptr;
}
struct CgcLaunch {
    CgcKernel kernel;
    int C, groups, threads;
    size_t smem;
    cudaLaunchConfig_t config(int batch, cudaLaunchAttribute* at, cudaStream_t s) const {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(batch * C)); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = (unsigned)C; at->val.clusterDim.y = 1; at->val.clusterDim.z = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        return cfg;
    }
};
// More than 8 blocks per cluster have to be asked for (constants again: see allow_shared).  In 3D, where a block streams its
// couplings, a single sample needs them: 48^3 41 us per iteration with 8 blocks, 24 with 16 (launches per iteration: 30), 44^3
// 35, 21 and 31, 8 x 48^3 41, 36 (10 blocks; 16 do not fit at once) and 39.
cudaError_t cgc_allow(CgcKernel k, bool d3, size_t smem) {
    const cudaError_t e = allow_shared(k, smem);
    return (e != cudaSuccess || !d3) ? e : cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
// Blocks per cluster: from how many clusters the device holds at a time (16 clusters of 8 blocks do not fit a B200, whose
// clusters stay inside a group of SMs: 256^2 x 16 10.3 us per iteration that way, in two waves, 7.4 with 6 blocks) and the work of
// a block.
CgcLaunch cgc_search(const dn_problem& p) {
    const bool d3 = p.grid.dim == 3;
    const int nslice = d3 ? p.grid.nz : p.grid.ny;
    const long long slice = nodes_of(p) / nslice;
    CgcLaunch best{};
    double cost = 0.0;
    for (int C = 1; C <= cgc_max(p.grid.dim); ++C) {
        if (!cgc_fits(p, C)) continue;
        CgcLaunch l{};
        l.C = C;
        l.smem = cgc_smem_bytes(p, C);
        const int most = (nslice + C - 1) / C;           // slices of the largest slab
        l.groups = d3 ? 1 : cgc_groups(p.grid.nx, nslice / C);
        l.threads = d3 ? CGC_THREADS3 : ((p.grid.nx - 2) * l.groups + 31) / 32 * 32;
        l.kernel = cgc_kernel(d3, (most + l.groups - 1) / l.groups);
        if (cgc_allow(l.kernel, d3, l.smem) != cudaSuccess) { (void)cudaGetLastError(); continue; }
        int active = 0;
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = l.config(p.batch, at, nullptr);
        if (cudaOccupancyMaxActiveClusters(&active, l.kernel, &cfg) != cudaSuccess || active < 1) { (void)cudaGetLastError(); continue; }
        const long long waves = (p.batch + active - 1) / active;
        // microseconds per iteration: barriers, and the nodes of a block (3D streams its couplings)
        const double t = (double)waves * ((C > CGC_PORTABLE ? 3.0 : C > 1 ? 2.0 : 1.0) + (double)(most * slice) * (d3 ? 2e-3 : 3e-4));
        if (best.C == 0 || t < cost) { best = l; cost = t; }
    }
    return best;
}

// The launch for `n` samples at a time; C = 0 if the device can hold no cluster (then it is asked again by the next call).
CgcLaunch cgc_launch(const dn_problem& p, int n) {
    dn_problem q = p;
    q.batch = n;
    const CgcLaunch l = memo_geometry<CgcLaunch>(q, sm_count(), [&]() { return cgc_search(q); });
    return l.C ? l : cgc_search(q);
}

// The solve with one cluster per sample, L.chunk samples at a time; r already holds K u - F.  p0: the operator on directions.
dn_status solve_in_clusters(const dn_problem& p0, const CgLayout& L, const CgcLaunch& l, char* base, float* u, int max_iters, float rtol,
                            float* relres, int32_t* iters, cudaStream_t s) {
    const bool d3 = p0.grid.dim == 3;
    const int nx = p0.grid.nx, ny = p0.grid.ny, nz = d3 ? p0.grid.nz : 1, nf = d3 ? 13 : 4, ncol = d3 ? 27 : 9;
    const long long nodes = nodes_of(p0);
    float* e = reinterpret_cast<float*>(base + L.p);
    float* q = reinterpret_cast<float*>(base + L.q);
    float* coef = reinterpret_cast<float*>(base + L.coef);
    size_t mpow = 1;
    for (int a = 0; a < p0.grid.dim; ++a) mpow *= (size_t)p0.kl_modes;
    auto blocks = [](long long n) { return (unsigned)((n + CG_THREADS - 1) / CG_THREADS); };
    for (int b0 = 0; b0 < p0.batch; b0 += L.chunk) {
        const int nb = p0.batch - b0 < L.chunk ? p0.batch - b0 : L.chunk;
        dn_problem probe = p0;
        probe.batch = CGC_GROUP * nb;
        if (p0.nu_mode == DN_NU_NODAL) probe.nu = p0.nu + (size_t)b0 * nodes;
        else probe.kl_w = p0.kl_w + (size_t)b0 * mpow;
        const long long total = nodes * nb;
        for (int first = 0; first < ncol; first += CGC_GROUP) {
            cg_colours_kernel<<<blocks(CGC_GROUP * total), CG_THREADS, 0, s>>>(nx, ny, nz, CGC_GROUP, first, CGC_GROUP * total, e);
            const dn_status st = run_operator(&probe, e, q, base + L.op, L.op_bytes, s, first == 0, nullptr, nullptr, CGC_GROUP);
            if (st != DN_OK) return st;
            cg_couplings_kernel<<<blocks(total), CG_THREADS, 0, s>>>(nx, ny, nz, CGC_GROUP, first, nf, total, q, coef);
        }
        if (cudaGetLastError() != cudaSuccess) return DN_ERR_CUDA;
        CgCluster A{};
        A.nx = nx; A.slice = d3 ? nx * ny : nx; A.nslice = d3 ? nz : ny; A.C = l.C; A.groups = l.groups; A.nf = nf; A.max_iters = max_iters;
        A.nodes = nodes;
        for (int o = 0; o < nf; ++o) {
            const int dx = o == 0 ? 1 : (o - 1) % 3 - 1, dy = o == 0 ? 0 : o < 4 ? 1 : (o - 4) / 3 - 1, dz = o < 4 ? 0 : 1;
            A.off[o] = dx + nx * (dy + ny * dz);
        }
        A.coef = coef; A.u = u + b0 * nodes; A.r0 = reinterpret_cast<const float*>(base + L.r) + b0 * nodes;
        A.rtol2 = (double)rtol * (double)rtol; A.relres = relres ? relres + b0 : nullptr; A.iters = iters ? iters + b0 : nullptr;
        cudaLaunchAttribute at[1];
        const cudaLaunchConfig_t cfg = l.config(nb, at, s);
        cudaError_t err = cgc_allow(l.kernel, d3, l.smem);
        if (err == cudaSuccess) err = cudaLaunchKernelEx(&cfg, l.kernel, A);
        if (err != cudaSuccess) return DN_ERR_CUDA;
    }
    return DN_OK;
}

}  // namespace
}  // namespace dn

using namespace dn;

extern "C" {

size_t dn_cg_workspace_bytes(const dn_problem* p) {
    if (!p || dn_workspace_bytes(p) == 0) return 0;
    const CgPlan pl = cg_plan(*p);                    // where no cluster can be scheduled, the launches per iteration serve after all
    return pl.clusters.total > pl.lockstep.total ? pl.clusters.total : pl.lockstep.total;
}

dn_status dn_cg_solve(const dn_problem* p, float* u, int32_t max_iters, float rtol, float* relres, int32_t* iters,
                      void* ws, size_t ws_bytes, void* stream) {
    if (!p || !u) return DN_ERR_NULL;
    if (dn_workspace_bytes(p) == 0) {        // invalid problem: let the fused path name the reason
        float dummy;
        return dn_energy(p, u, &dummy, nullptr, 0, stream);
    }
    if (max_iters < 0 || !(rtol >= 0.0f)) return DN_ERR_MODE;
    const CgPlan pl = cg_plan(*p);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) % kAlign) != 0 || ws_bytes < pl.lockstep.total || ws_bytes < pl.clusters.total)
        return DN_ERR_WORKSPACE;
    CgcLaunch cl{};
    if (pl.clusters.chunk) cl = cgc_launch(*p, pl.clusters.chunk);
    const CgLayout& L = cl.C ? pl.clusters : pl.lockstep;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(ws);
    float* r = reinterpret_cast<float*>(base + L.r);
    float* q = reinterpret_cast<float*>(base + L.q);
    float* pd = reinterpret_cast<float*>(base + L.p);
    float* dinv = reinterpret_cast<float*>(base + L.dinv);
    double* partials = reinterpret_cast<double*>(base + L.partials);
    CgScalars* sc = reinterpret_cast<CgScalars*>(base + L.scalars);
    void* op_ws = base + L.op;
    const size_t op_bytes = L.op_bytes;
    void* op1_ws = base + L.op1;
    const size_t op1_bytes = L.op1_bytes;
    const long long nodes = nodes_of(*p);
    const int nvb = vec_blocks(nodes);
    const dim3 vgrid((unsigned)nvb, (unsigned)p->batch);

    // Dirichlet faces of u take their values; r = K u - F (masked) with the caller's forcing
    if (launch_apply_bc(p->grid, p->batch, p->bc_x0, p->bc_x1, 0, u, s, p->bc_x0_b, p->bc_x1_b) != cudaSuccess)
        return DN_ERR_CUDA;
    dn_status st = DN_OK;
    dn_problem p1 = *p;
    p1.flags &= ~(DN_NO_MASK | DN_IMPOSE_BC_ON_LOAD);
    // the operator on directions: zero forcing, zero boundary values, same diffusivity
    dn_problem p0 = p1;
    p0.f = nullptr; p0.f_const = 0.0f; p0.bc_x0 = 0.0f; p0.bc_x1 = 0.0f; p0.bc_x0_b = nullptr; p0.bc_x1_b = nullptr;
    // The KL tables are built once per solve for the direction operator (aligned scratch fields, no nodal forcing); the
    // caller's problem is applied once, in a workspace of its own with its own tables (it may take another family).
    st = run_operator(&p1, u, r, op1_ws, op1_bytes, s, true, nullptr, nullptr);
    if (st != DN_OK) return st;
    if (cl.C) return solve_in_clusters(p0, L, cl, base, u, max_iters, rtol, relres, iters, s);
    st = build_tables(&p0, pd, q, op_ws, op_bytes, s);
    if (st != DN_OK) return st;
    {   // Jacobi preconditioner: the diagonal of K, one colour class per application (p and q serve as scratch)
        const int nz = p->grid.dim == 3 ? p->grid.nz : 1;
        const unsigned rows = (unsigned)((long long)p->batch * nz * p->grid.ny);
        const int ncol = p->grid.dim == 3 ? 27 : 9;
        if (cudaMemsetAsync(pd, 0, sizeof(float) * (size_t)nodes * p->batch, s) != cudaSuccess) return DN_ERR_CUDA;
        for (int c = 0; c < ncol; ++c) {
            cg_probe_kernel<<<rows, CG_THREADS, 0, s>>>(p->grid.nx, p->grid.ny, nz, c, 0, pd, nullptr, nullptr);
            st = run_operator(&p0, pd, q, op_ws, op_bytes, s, false, nullptr, nullptr);
            if (st != DN_OK) return st;
            cg_probe_kernel<<<rows, CG_THREADS, 0, s>>>(p->grid.nx, p->grid.ny, nz, c, 1, pd, q, dinv);
        }
        if (cudaGetLastError() != cudaSuccess) return DN_ERR_CUDA;
    }
    cg_init_kernel<<<vgrid, CG_THREADS, 0, s>>>(nodes, nvb, r, dinv, pd, partials);
    cg_start_kernel<<<p->batch, CG_THREADS, 0, s>>>(partials, nvb, sc);
    if (cudaGetLastError() != cudaSuccess) return DN_ERR_CUDA;

    const double rtol2 = (double)rtol * (double)rtol;
    for (int it = 0; it < max_iters; ++it) {
        const double* op_partials = nullptr;
        int op_nblk = 0;
        st = run_operator(&p0, pd, q, op_ws, op_bytes, s, false, &op_partials, &op_nblk);
        if (st != DN_OK) return st;
        cg_alpha_kernel<<<p->batch, CG_THREADS, 0, s>>>(op_partials, op_nblk, sc);
        cg_update_kernel<<<vgrid, CG_THREADS, 0, s>>>(nodes, nvb, u, r, pd, q, dinv, sc, partials);
        cg_beta_kernel<<<p->batch, CG_THREADS, 0, s>>>(partials, nvb, rtol2, sc);
        cg_direction_kernel<<<vgrid, CG_THREADS, 0, s>>>(nodes, r, dinv, pd, sc);
        if (cudaGetLastError() != cudaSuccess) return DN_ERR_CUDA;
    }
    if (relres || iters) {
        cg_report_kernel<<<(p->batch + 127) / 128, 128, 0, s>>>(sc, p->batch, relres, iters);
        if (cudaGetLastError() != cudaSuccess) return DN_ERR_CUDA;
    }
    return DN_OK;
}

}  // extern "C"
