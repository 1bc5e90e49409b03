// Conjugate gradients on K(nu) u = F, preconditioned by one multigrid V-cycle, a sample per thread-block cluster and all its
// iterations in one launch: the solver of samples that fit the shared memory of a few SMs.
//
// The operator is the assembled stencil: the couplings K_ij of a node with its forward neighbours (4 in 2D, 13 in 3D; the
// backward ones are those neighbours' own), in difference form,
//     (K p)_i = d_i p_i + sum_j K_ij (p_j - p_i),      d_i = -(sum of the couplings with Dirichlet nodes),
// so that it loses no more to cancellation than the element form.
//
// Preconditioner.  Level 0 is the grid; an axis is halved by keeping the even nodes (the free ones along x, where the two faces
// hold zeros), and a level halves those axes whose mesh width is at most 1.5 times the smallest one, so stretched cells become
// round first.  Between levels P is linear interpolation and the coarse operators are P^T A P, formed one axis at a time (a
// 3-point rule along that axis for every offset along the others).  Smoother: one Jacobi sweep before and one after, with
// weight MG_THETA / sum_j |a_ij| in place of 1 / a_ii.  By Gershgorin the sweep then contracts for any symmetric positive
// definite stencil, whatever the coefficient, so the cycle is symmetric positive definite.  On square and cubic Q1 cells
// sum_j |a_ij| = 2 a_ii, where the best weight is 8/9 (2D) and 1 (3D); cells stretched by 2 to 8 do best with 1.5 to 1.7:
// iterations to 1e-5 from noise about the solution's profile with 1.65, with 1.5 and with 1.9: 256^2 4, 5, 5; 256 x 32 7, 7, 13; 48 x
// 16 x 16 9, 9, 12 (from a smooth field 1 to 3 more on square cells: 256^2 6 or 7).  Jacobi alone takes 342 to 540, 364 and 101; a
// coefficient that jumps by up to 1e4 from one patch of 8 nodes per axis to the next 8 to 57, with Jacobi 564 (256^2).
//
// What a cluster does.  The nodes of the larger levels are cut into one contiguous range per block.  A pass that applies a stencil
// first stages the vector it applies it to in shared memory, the range and what the stencil reaches beyond it; what a block
// stages beyond its own range it computes itself from what its neighbours published, so a level takes one cluster barrier on
// the way down (its residual) and one on the way up (its corrected field).  The levels below belong to block 0 alone, which
// keeps them in shared memory; in 2D a block keeps the couplings of its range of level 0 there too, where they fit.  Everything
// else lives in L2.  The last level, of at most 512 nodes, takes a Chebyshev iteration, a node per thread.  Dot products are
// exchanged through distributed shared memory and summed in a fixed order.  A cluster stops when its sample is done; samples do not
// wait for one another.
//
// What bounds it: latency.  256^2 x 16 (16 clusters of 6 blocks: of 7 and more not all fit a B200 at once) takes 590 to 612 us, of which
// the cluster kernel 440; one of its 6 or 7 iterations is 140 thousand cycles in some 20 passes that wait for one another: the
// three over level 0 take 75, block 0's two levels 20, the cluster barriers 20.  A pass has 16 warps to hide L2 behind, so a
// thread loads the rows of four nodes (3D: two) before it uses any; that, the last level of 512 nodes in place of levels down to 4, and
// the coarse operators of the shared levels by kernels of their own, with warps enough, took a solve from 1.29 to 0.85 million
// cycles.  Conjugate gradients with the diagonal, in clusters with their couplings in shared memory, took 4240 us; 48^3 x 9 4895,
// now 988; 32^2 x 64 235, now 113.
#include <cmath>

#include "dn_internal.cuh"

namespace dn {
namespace {

constexpr int MG_THREADS = 512, MG_WARPS = MG_THREADS / 32;
constexpr int MG_LEVELS = 24;
constexpr int MG_MOST = 16;                  // blocks per cluster that may be asked for (8 without asking)
constexpr float MG_THETA = 1.65f;
constexpr int mg_alone(int dim) { return dim == 3 ? 512 : 1100; }      // levels of at most this many nodes belong to block 0
constexpr int MG_LAST = MG_THREADS;          // the last level: at most one node per thread
constexpr int MG_STEPS = 48;                 // ... and Chebyshev steps

__host__ __device__ constexpr int mg_nf(int dim) { return dim == 2 ? 4 : 13; }

struct MgLevel {
    int n[3];                                // nodes per axis (n[2] = 1 in 2D); along x the two faces count
    int slice, N, cut;                       // nodes per slice and in all; bit a: axis a is halved towards the next level
    int reach;                               // how far a stencil reaches in the linear index
    float inv0, invs;                        // 1 / n[0], 1 / slice
    // Offsets (floats): nf couplings, diagonal, weight (level 0: d); right-hand side, field, residual.  Levels up to shared_levels
    // have their stencil (K) in the sample's memory, from there on (also) in block 0's shared memory (s); b, x and t go with it
    int K, s, b, x, t;
};
struct MgArgs {
    int C, nlev, shared_levels, max_iters;   // levels 0 .. shared_levels - 1 are worked on by all blocks
    int z, p, q, xs, tmp;                    // offsets: preconditioned residual, direction, K p, field of level shared_levels, scratch
    int v1, v2, hp, k0, tail, smem;          // offsets in shared memory (floats); k0 < 0: couplings of level 0 stay in L2
    long long sample;                        // floats per sample
    float* mem;
    float* u;
    float* r;                                // K u - F at the start
    int steps;                               // of the last level's Chebyshev iteration; its factors
    float momentum[MG_STEPS], gain[MG_STEPS];
    double rtol2;
    float* relres;
    int32_t* iters;
    MgLevel lev[MG_LEVELS];
};

__device__ __forceinline__ unsigned mg_remote(const void* local, int rank) {       // the same address in another block's memory
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(local)), "r"(rank));
    return r;
}
__device__ __forceinline__ void mg_store(unsigned remote, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory"); }
__device__ __forceinline__ void mg_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__host__ __device__ inline int mg_first(int n, int C, int rank) { return (int)((long long)n * rank / C); }   // first of rank's share of n
// n / d for n + 0.5 < 2^20: the quotient is at least 0.5 / d away from the next integer, the rounding less than n / d * 2^-22
__device__ __forceinline__ int mg_div(int n, float inv) { return (int)(((float)n + 0.5f) * inv); }

// Offsets of the couplings: forward neighbours (1,0,0), (-1..1,1,0), (-1..1,-1..1,1).
__host__ __device__ constexpr int mg_dx(int o) { return o == 0 ? 1 : (o - 1) % 3 - 1; }
__host__ __device__ constexpr int mg_dy(int o) { return o == 0 ? 0 : o < 4 ? 1 : (o - 4) / 3 - 1; }
__host__ __device__ constexpr int mg_dz(int o) { return o < 4 ? 0 : 1; }
__host__ __device__ constexpr int mg_which(int dx, int dy, int dz) { return dz ? 4 + 3 * (dy + 1) + dx + 1 : dy ? 2 + dx : 0; }

// Values that other blocks wrote come from L2; SM: block 0's own, in shared memory.
template <bool SM> __device__ __forceinline__ float mg_ld(const float* p) { return SM ? *p : __ldcg(p); }

// a_ij of node i and its neighbour at (dx, dy, dz).  Neighbours beyond the grid: whatever finite number stands there.
template <int DIM, bool SM>
__device__ __forceinline__ float mg_entry(const float* K, int N, int i, int dx, int dy, int dz, int X, int plane) {
    constexpr int NF = mg_nf(DIM);
    if (dx == 0 && dy == 0 && dz == 0) return mg_ld<SM>(K + NF * N + i);
    const bool fwd = dz > 0 || (dz == 0 && (dy > 0 || (dy == 0 && dx > 0)));
    if (fwd) return mg_ld<SM>(K + mg_which(dx, dy, dz) * N + i);
    return mg_ld<SM>(K + mg_which(-dx, -dy, -dz) * N + i + dx + X * dy + plane * dz);
}

// One axis of P^T A P: node i of the coarse stencil (couplings and diagonal).  A coarse node is the even node c of the axis and
// gathers half of its odd neighbours (all of a last odd node that has no even one behind it).
template <int DIM, int AX, bool SM>
__device__ __forceinline__ void mg_halve(const float* src, const int (&n)[3], float* dst, const int (&m)[3], int i) {
    constexpr int NF = mg_nf(DIM);
    const int X = n[0], plane = n[0] * n[1], N = plane * n[2], M = m[0] * m[1] * m[2];
    const int st = AX == 0 ? 1 : AX == 1 ? X : plane;
    int z = DIM == 3 ? i / (m[0] * m[1]) : 0;
    const int ip = i - z * m[0] * m[1];
    int y = ip / m[0], x = ip - y * m[0];
    const bool face = x == 0 || x == m[0] - 1;
    const int pd = AX == 0 ? x : AX == 1 ? y : z, md = m[AX], ns = n[AX], pc = 2 * pd;
    if (AX == 0) x = pc; else if (AX == 1) y = pc; else z = pc;
    if (face) {
        for (int o = 0; o <= NF; ++o) dst[o * M + i] = 0.f;
        return;
    }
    const int c = x + X * y + plane * z;
    const bool left = pc > 0, right = pc + 1 < ns;
    const float wr = (AX != 0 && pc + 1 == ns - 1) ? 1.f : 0.5f;
    const bool next = AX == 0 ? pd + 1 < md - 1 : pd + 1 < md, prev = AX == 0 ? pd > 1 : pd > 0;
    const int cl = left ? c - st : c, cr = right ? c + st : c;
    float out[NF + 1];
#pragma unroll
    for (int o = 0; o <= NF; ++o) {
        const int d0 = o == NF ? 0 : mg_dx(o), d1 = o == NF ? 0 : mg_dy(o), d2 = o == NF ? 0 : mg_dz(o);
        const int da = AX == 0 ? d0 : AX == 1 ? d1 : d2;
        auto a = [&](int node, int along) {
            return mg_entry<DIM, SM>(src, N, node, AX == 0 ? along : d0, AX == 1 ? along : d1, AX == 2 ? along : d2, X, plane);
        };
        if (da == 0) {
            const float vr = wr * (a(c, 1) + a(cr, -1)) + wr * wr * a(cr, 0), vl = 0.5f * (a(c, -1) + a(cl, 1)) + 0.25f * a(cl, 0);
            out[o] = a(c, 0) + (right ? vr : 0.f) + (left ? vl : 0.f);
        } else if (da == 1) {
            const float v = 0.5f * a(c, 1) + 0.25f * a(cr, 0) + 0.5f * a(cr, 1);
            out[o] = next ? v : 0.f;
        } else {
            const float v = 0.5f * a(c, -1) + 0.25f * a(cl, 0) + 0.5f * a(cl, -1);
            out[o] = prev ? v : 0.f;
        }
    }
#pragma unroll
    for (int o = 0; o <= NF; ++o) dst[o * M + i] = out[o];
}

// Weights of the Jacobi sweeps.
template <int DIM, bool SM>
__device__ void mg_weights(float* K, const MgLevel& L, int lo, int hi) {
    constexpr int NF = mg_nf(DIM);
    for (int i = lo + (int)threadIdx.x; i < hi; i += MG_THREADS) {
        float s = fabsf(mg_ld<SM>(K + NF * L.N + i));
#pragma unroll
        for (int o = 0; o < NF; ++o) {
            const int f = mg_dx(o) + L.n[0] * (mg_dy(o) + L.n[1] * mg_dz(o));
            s += fabsf(mg_ld<SM>(K + o * L.N + i));
            if (i >= f) s += fabsf(mg_ld<SM>(K + o * L.N + i - f));
        }
        K[(NF + 1) * L.N + i] = s > 0.f ? MG_THETA / s : 0.f;
    }
}

// A node's row of a stencil, and applied to a vector; v points at the node's value in shared memory.
template <int DIM> struct MgRow { float c, f[mg_nf(DIM)], k[mg_nf(DIM)]; };     // centre, forward, backward
template <int DIM> __device__ __forceinline__ int mg_step(int o, int X, int slice) {
    return DIM == 3 ? mg_dx(o) + X * mg_dy(o) + slice * mg_dz(o) : mg_dx(o) + X * mg_dy(o);
}
template <int DIM>
__device__ __forceinline__ void mg_load(MgRow<DIM>& R, const float* K, int stride, int X, int slice, float centre) {
    R.c = centre;
#pragma unroll
    for (int o = 0; o < mg_nf(DIM); ++o) { R.f[o] = K[o * stride]; R.k[o] = K[o * stride - mg_step<DIM>(o, X, slice)]; }
}
template <int DIM>
__device__ __forceinline__ float mg_apply(const MgRow<DIM>& R, int X, int slice, const float* v) {
    float q = R.c * v[0];
#pragma unroll
    for (int o = 0; o < mg_nf(DIM); ++o) {
        const int f = mg_step<DIM>(o, X, slice);
        q = fmaf(R.f[o], v[f], q);
        q = fmaf(R.k[o], v[-f], q);
    }
    return q;
}
// The same in difference form (the centre is d_i) on node g of level 0.
template <int DIM>
__device__ __forceinline__ float mg_apply_diff(const MgRow<DIM>& R, int X, int slice, const float* v, int g) {
    const float vc = v[0];
    float q = R.c * vc;
#pragma unroll
    for (int o = 0; o < mg_nf(DIM); ++o) {
        const int f = mg_step<DIM>(o, X, slice);
        q = fmaf(R.f[o], v[f] - vc, q);
        q = fmaf(g >= f ? R.k[o] : 0.f, v[-f] - vc, q);
    }
    return q;
}

// What node i of 0 .. n - 1 needs, load(i, .), and what is done with it, use(i, .): B of this thread's nodes at a time, so that
// their loads are under way together (a pass has too few warps to hide L2's latency otherwise).
template <class T, int B, class F, class S>
__device__ __forceinline__ void mg_each(int n, F load, S use) {
    for (int i = threadIdx.x; i < n; i += B * MG_THREADS) {
        T v[B];
#pragma unroll
        for (int k = 0; k < B; ++k) load(min(i + k * MG_THREADS, n - 1), v[k]);
#pragma unroll
        for (int k = 0; k < B; ++k) if (i + k * MG_THREADS < n) use(i + k * MG_THREADS, v[k]);
    }
}

// Right-hand side of level M at node i: the residual t of level L gathered to it.
template <int DIM, bool SM>
__device__ __forceinline__ float mg_gather(const MgLevel& L, const MgLevel& M, const float* t, int i) {
    constexpr int AS = DIM - 1;
    const int s = mg_div(i, M.invs), ip = i - s * M.slice;
    const int y = DIM == 3 ? mg_div(ip, M.inv0) : 0, x = ip - y * M.n[0];
    if (x == 0 || x == M.n[0] - 1) return 0.f;
    // the node and its odd neighbours along each halved axis: steps (0 where there is none) and weights
    struct { int l, r; float wl, wr; } e[3];
    auto axis = [&](int a, int pos, int step) {
        const bool cut = (L.cut >> a) & 1;
        const int f = cut ? 2 * pos : pos;
        const bool hl = cut && f > 0, hr = cut && f + 1 < L.n[a];
        e[a].l = hl ? -step : 0; e[a].wl = hl ? 0.5f : 0.f;
        e[a].r = hr ? step : 0; e[a].wr = !hr ? 0.f : (a > 0 && f + 1 == L.n[a] - 1) ? 1.f : 0.5f;
        return f;
    };
    const float* c = t + axis(0, x, 1);
    if constexpr (DIM == 3) c += axis(1, y, L.n[0]) * L.n[0];
    c += axis(AS, s, L.slice) * L.slice;
    auto row = [&](const float* v) { return fmaf(e[0].wl, mg_ld<SM>(v + e[0].l), fmaf(e[0].wr, mg_ld<SM>(v + e[0].r), mg_ld<SM>(v))); };
    auto plane = [&](const float* v) {
        if constexpr (DIM == 2) return row(v);
        return fmaf(e[1].wl, row(v + e[1].l), fmaf(e[1].wr, row(v + e[1].r), row(v)));
    };
    return fmaf(e[AS].wl, plane(c + e[AS].l), fmaf(e[AS].wr, plane(c + e[AS].r), plane(c)));
}

// The field of level M at node g of level L, by interpolation: the mean of the values at both ends along every axis (the same
// one twice where the node is a coarse one).
template <int DIM> struct MgPull { float v[1 << DIM], scale, w, b; };
template <int DIM, bool SM>
__device__ __forceinline__ void mg_pull(MgPull<DIM>& P, const MgLevel& L, const MgLevel& M, const float* xc, int g) {
    constexpr int AS = DIM - 1;
    const int s = mg_div(g, L.invs), t = g - s * L.slice;
    const int y = DIM == 3 ? mg_div(t, L.inv0) : 0, x = t - y * L.n[0];
    int step[3] = {0, 0, 0};
    const float* c = xc;
    auto axis = [&](int a, int pos, int st) {
        const bool cut = (L.cut >> a) & 1, odd = cut && (pos & 1) && pos + 1 < L.n[a];
        step[a] = odd ? st : 0;
        c += (cut ? pos >> 1 : pos) * st;
    };
    const bool face = x == 0 || x == L.n[0] - 1;
    axis(0, face ? 0 : x, 1);
    if constexpr (DIM == 3) axis(1, y, M.n[0]);
    axis(AS, s, M.slice);
    P.scale = face ? 0.f : 1.f / (1 << DIM);
#pragma unroll
    for (int k = 0; k < (1 << DIM); ++k) {
        const int o = ((k & 1) ? step[0] : 0) + ((k & 2) ? step[1] : 0) + ((k & 4) ? step[2] : 0);
        P.v[k] = mg_ld<SM>(c + o);
    }
}
template <int DIM> __device__ __forceinline__ float mg_mean(const MgPull<DIM>& P) {
    float a = (P.v[0] + P.v[1]) + (P.v[2] + P.v[3]);
    if constexpr (DIM == 3) a += (P.v[4] + P.v[5]) + (P.v[6] + P.v[7]);
    return P.scale * a;
}

// A block's nodes of a level, what of them and beyond them is staged (V[i]: node lo - reach + i), and its stencil.
struct MgRange {
    int lo, hi, stride;
    const float* K;                          // K + g: the couplings of node g
};

template <int DIM> __host__ __device__ constexpr int mg_batch() { return DIM == 2 ? 4 : 2; }      // nodes whose rows a thread loads together

// On the way down: V = weight * right-hand side, then the residual of that first sweep.  rhs(g): the right-hand side of any
// node that is staged; S: nodes staged together.
template <int DIM, bool SM, int S, class R>
__device__ __forceinline__ void mg_down(const MgLevel& L, const MgRange& G, const float* diag, const float* b, float* V, float* t, R rhs) {
    const int base = G.lo - L.reach, X = L.n[0], slice = L.slice;
    const float* w = diag + L.N;
    struct In { float w, b; };
    mg_each<In, S>(G.hi - G.lo + 2 * L.reach, [&](int i, In& a) {
        const int g = min(max(base + i, 0), L.N - 1);
        a.w = w[g]; a.b = rhs(g);
    }, [&](int i, const In& a) { V[i] = (base + i >= 0 && base + i < L.N) ? a.w * a.b : 0.f; });
    __syncthreads();
    struct Row { MgRow<DIM> r; float b; };
    mg_each<Row, mg_batch<DIM>()>(G.hi - G.lo, [&](int i, Row& a) {
        const int g = G.lo + i;
        a.b = mg_ld<SM>(b + g);
        mg_load<DIM>(a.r, G.K + g, G.stride, X, slice, diag[g]);
    }, [&](int i, const Row& a) { t[G.lo + i] = a.b - mg_apply<DIM>(a.r, X, slice, V + L.reach + i); });
}

// On the way up: the first sweep and the correction from level M, then the second sweep.  Returns this thread's share of b.x.
template <int DIM, bool SM, bool SMC>
__device__ __forceinline__ double mg_up(const MgLevel& L, const MgLevel& M, const MgRange& G, const float* diag, const float* b, const float* xc,
                                        float* V, float* x) {
    const int base = G.lo - L.reach, X = L.n[0], slice = L.slice;
    const float* w = diag + L.N;
    mg_each<MgPull<DIM>, 4>(G.hi - G.lo + 2 * L.reach, [&](int i, MgPull<DIM>& a) {
        const int g = min(max(base + i, 0), L.N - 1);
        a.w = w[g]; a.b = mg_ld<SM>(b + g);
        mg_pull<DIM, SMC>(a, L, M, xc, g);
    }, [&](int i, const MgPull<DIM>& a) { V[i] = (base + i >= 0 && base + i < L.N) ? fmaf(a.w, a.b, mg_mean<DIM>(a)) : 0.f; });
    __syncthreads();
    double sum = 0.0;
    struct Row { MgRow<DIM> r; float w, b; };
    mg_each<Row, mg_batch<DIM>()>(G.hi - G.lo, [&](int i, Row& a) {
        const int g = G.lo + i;
        a.w = w[g]; a.b = mg_ld<SM>(b + g);
        mg_load<DIM>(a.r, G.K + g, G.stride, X, slice, diag[g]);
    }, [&](int i, const Row& a) {
        const float* v = V + L.reach + i;
        const float y = fmaf(a.w, a.b - mg_apply<DIM>(a.r, X, slice, v), v[0]);
        x[G.lo + i] = y;
        sum += (double)(a.b * y);
    });
    return sum;
}

template <int DIM>
__global__ void __launch_bounds__(MG_THREADS, 1) mg_cluster_kernel(const __grid_constant__ MgArgs A) {
    extern __shared__ __align__(16) double mg_smem[];
    constexpr int NF = mg_nf(DIM);
    dep_wait();                                          // the stencils of the shared levels and K u - F are complete
    const int tid = threadIdx.x, C = A.C, lane = tid & 31, warp = tid >> 5;
    const int sample = blockIdx.x / C, rank = blockIdx.x % C, SL = A.shared_levels, last = A.nlev - 1;
    float* sm = reinterpret_cast<float*>(mg_smem);
    double* red = mg_smem;                               // [3][C][MG_WARPS]: p.q, r.r, r.z of every warp of the cluster
    float* V1 = sm + A.v1;
    float* V2 = sm + A.v2;
    float* hp = sm + A.hp;                               // the direction on what is staged beyond the range
    const MgLevel& L0 = A.lev[0];
    const int N = L0.N, reach = L0.reach, X0 = L0.n[0], slice0 = L0.slice;
    const int lo = mg_first(N, C, rank), hi = mg_first(N, C, rank + 1), n = hi - lo;      // own nodes
    float* mem = A.mem + A.sample * sample;
    float* u = A.u + (long long)N * sample;
    float* r = A.r + (long long)N * sample;
    float* z = mem + A.z;
    float* p = mem + A.p;
    float* q = mem + A.q;
    const float* K0 = mem + L0.K;
    const float* d0 = K0 + (NF + 2) * N;

    auto all_sync = [&]() { if (C > 1) mg_barrier(); else __syncthreads(); };
    // sum over the cluster, in a fixed order: every warp sends its sum to every block, every warp adds them all.  One slot per
    // use; at least one other barrier lies between two uses of a slot.
    auto cluster_sum = [&](double a, int slot) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        double* mine = red + slot * C * MG_WARPS;
        if (lane < C) mg_store(mg_remote(mine + rank * MG_WARPS + warp, lane), a);
        all_sync();
        double s = 0.0;
        for (int i = lane; i < C * MG_WARPS; i += 32) s += mine[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };

    for (int i = tid; i < A.smem; i += MG_THREADS) sm[i] = 0.f;
    if (rank == 0) {                                     // zeros in front of every stencil in L2
        for (int l = 0; l <= SL; ++l) {
            const int pad = A.lev[l].reach;
            for (int i = tid; i < pad; i += MG_THREADS) mem[A.lev[l].K - pad + i] = 0.f;
        }
    }
    mg_barrier();                                        // every block of the cluster runs, its sums are zeroed
    MgRange G0{lo, hi, N, C == 1 ? sm + L0.s : K0};
    if (A.k0 >= 0) {                                     // the couplings of the range and of what it reaches below it
        G0.stride = n + reach;
        G0.K = sm + A.k0 - (lo - reach);
        for (int o = 0; o < NF; ++o)
            for (int i = tid; i < n + reach; i += MG_THREADS) {
                const int g = lo - reach + i;
                sm[A.k0 + o * G0.stride + i] = g >= 0 ? __ldg(K0 + o * N + g) : 0.f;
            }
    }
    double rr0 = 0.0;
    for (int i = tid; i < n; i += MG_THREADS) {
        const float rv = -r[lo + i];
        r[lo + i] = rv;
        rr0 += (double)(rv * rv);
    }
    rr0 = cluster_sum(rr0, 1);
    double rr = rr0;
    int it = 0;
    if (rr0 > 0.0 && A.max_iters > 0) {
        // ---- weights of the shared levels, and the operators of block 0's levels
        for (int l = 1; l <= SL; ++l) {
            const MgLevel& M = A.lev[l];
            mg_weights<DIM, false>(mem + M.K, M, mg_first(M.N, C, rank), mg_first(M.N, C, rank + 1));
        }
        all_sync();
        if (rank == 0) {
            {
                const MgLevel& L = A.lev[SL];
                for (int i = tid; i < (NF + 2) * L.N; i += MG_THREADS) sm[L.s + i] = __ldcg(mem + L.K + i);
                __syncthreads();
            }
            for (int l = SL; l < last; ++l) {
                const MgLevel& L = A.lev[l];
                const MgLevel& M = A.lev[l + 1];
                int ns[3] = {L.n[0], L.n[1], L.n[2]};
                const float* src = sm + L.s;
                float* tmp = V1;                         // (the staging area is free)
                int left = L.cut;
                while (left) {
                    const int ax = __ffs(left) - 1;
                    left &= left - 1;
                    int nd[3] = {ns[0], ns[1], ns[2]};
                    nd[ax] = M.n[ax];
                    const int size = nd[0] * nd[1] * nd[2];
                    float* dst = left ? tmp + L.reach : sm + M.s;
                    for (int i = tid; i < size; i += MG_THREADS) {
                        if (ax == 0) mg_halve<DIM, 0, true>(src, ns, dst, nd, i);
                        else if (ax == 1) mg_halve<DIM, 1, true>(src, ns, dst, nd, i);
                        else if constexpr (DIM == 3) mg_halve<DIM, 2, true>(src, ns, dst, nd, i);
                    }
                    __syncthreads();
                    tmp += L.reach + (NF + 1) * size;
                    src = dst;
                    ns[ax] = nd[ax];
                }
                mg_weights<DIM, true>(sm + M.s, M, 0, M.N);
                __syncthreads();
            }
        }

        // z = V-cycle applied to r; the share of this thread in r.z
        auto precondition = [&]() {
            double rz = 0.0;
            auto from_r = [&](int g) { return __ldcg(r + g); };
            auto range = [&](int l) {
                const MgLevel& L = A.lev[l];
                return l == 0 ? G0 : MgRange{mg_first(L.N, C, rank), mg_first(L.N, C, rank + 1), L.N, mem + L.K};
            };
            for (int l = 0; l < SL; ++l) {
                const MgLevel& L = A.lev[l];
                const MgRange G = range(l);
                const float* diag = mem + L.K + NF * L.N;
                if (l == 0) {
                    mg_down<DIM, false, 8>(L, G, diag, r, V1, mem + L.t, from_r);
                } else {
                    const MgLevel& U = A.lev[l - 1];
                    float* b = mem + L.b;
                    mg_down<DIM, false, DIM == 2 ? 2 : 1>(L, G, diag, b, V1, mem + L.t, [&](int g) {
                        const float v = mg_gather<DIM, false>(U, L, mem + U.t, g);
                        if (g >= G.lo && g < G.hi) b[g] = v;
                        return v;
                    });
                }
                all_sync();
            }
            if (rank == 0) {
                auto gathered = [&](int l, int g) {      // right-hand side of level l > 0, kept
                    const float v = l == SL ? mg_gather<DIM, false>(A.lev[l - 1], A.lev[l], mem + A.lev[l - 1].t, g)
                                            : mg_gather<DIM, true>(A.lev[l - 1], A.lev[l], V2, g);
                    sm[A.lev[l].b + g] = v;
                    return v;
                };
                for (int l = SL; l < last; ++l) {
                    const MgLevel& L = A.lev[l];
                    const float* K = sm + L.s;
                    const float* diag = K + NF * L.N;
                    const MgRange G{0, L.N, L.N, K};
                    if (l == 0) mg_down<DIM, false, 8>(L, G, diag, r, V1, V2, from_r);
                    else mg_down<DIM, true, DIM == 2 ? 2 : 1>(L, G, diag, sm + L.b, V1, V2, [&](int g) { return gathered(l, g); });
                    __syncthreads();
                }
                {   // the last level, a node per thread: Chebyshev iteration on the Jacobi-weighted operator
                    const MgLevel& L = A.lev[last];
                    const int X = L.n[0], slice = L.slice;
                    const bool on = tid < L.N;
                    const float* K = sm + L.s + (on ? tid : 0);
                    float* V = V1;                       // (two copies: a step reads one and writes the other)
                    const int copy = L.N + 2 * L.reach;
                    const float b = !on ? 0.f : last == 0 ? __ldcg(r + tid) : gathered(last, tid), w = on ? K[(NF + 1) * L.N] : 0.f;
                    for (int i = tid; i < 2 * copy; i += MG_THREADS) V1[i] = 0.f;
                    MgRow<DIM> R;
                    mg_load<DIM>(R, K, L.N, X, slice, K[NF * L.N]);
                    float d = A.gain[0] * (w * b), x = d;
                    __syncthreads();
                    for (int k = 1; k < A.steps; ++k) {
                        if (on) V[L.reach + tid] = x;
                        __syncthreads();
                        d = fmaf(A.momentum[k], d, A.gain[k] * (w * (b - mg_apply<DIM>(R, X, slice, V + L.reach + (on ? tid : 0)))));
                        x += d;
                        V = V == V1 ? V1 + copy : V1;
                    }
                    if (on) (last == 0 ? z : last == SL ? mem + A.xs : sm + L.x)[tid] = x;
                    if (last == 0) rz = (double)(b * x);
                }
                __syncthreads();
                for (int l = last - 1; l >= SL; --l) {
                    const MgLevel& L = A.lev[l];
                    const float* K = sm + L.s;
                    const float* diag = K + NF * L.N;
                    const MgRange G{0, L.N, L.N, K};
                    const float* xc = sm + A.lev[l + 1].x;
                    if (l == 0) rz = mg_up<DIM, false, true>(L, A.lev[1], G, diag, r, xc, V1, z);
                    else mg_up<DIM, true, true>(L, A.lev[l + 1], G, diag, sm + L.b, xc, V1, l == SL ? mem + A.xs : sm + L.x);
                    __syncthreads();
                }
            }
            if (SL > 0) {
                all_sync();
                for (int l = SL - 1; l >= 0; --l) {
                    const MgLevel& L = A.lev[l];
                    const float* diag = mem + L.K + NF * L.N;
                    rz = mg_up<DIM, false, false>(L, A.lev[l + 1], range(l), diag, l == 0 ? r : mem + L.b,
                                                  mem + (l + 1 == SL ? A.xs : A.lev[l + 1].x), V1, l == 0 ? z : mem + L.x);
                    if (l > 0) all_sync();
                }
            }
            return rz;
        };

        double rho = cluster_sum(precondition(), 2);
        float beta = 0.f;
        while (rho > 0.0 && it < A.max_iters) {
            // p = z + beta p on the range and what is staged beyond it; q = K p
            struct In { float z, old; };
            mg_each<In, 8>(n + 2 * reach, [&](int i, In& a) {
                const int g = min(max(lo - reach + i, 0), N - 1);
                a.z = __ldcg(z + g);
                a.old = (i >= reach && i < n + reach) ? p[g] : hp[i < reach ? i : i - n];
            }, [&](int i, const In& a) {
                const int g = lo - reach + i;
                const float v = (g < 0 || g >= N) ? 0.f : it == 0 ? a.z : fmaf(beta, a.old, a.z);
                V1[i] = v;
                if (i >= reach && i < n + reach) p[g] = v;
                else hp[i < reach ? i : i - n] = v;
            });
            __syncthreads();
            double pq = 0.0;
            mg_each<MgRow<DIM>, mg_batch<DIM>()>(n, [&](int i, MgRow<DIM>& a) {
                mg_load<DIM>(a, G0.K + lo + i, G0.stride, X0, slice0, __ldg(d0 + lo + i));
            }, [&](int i, const MgRow<DIM>& a) {
                const float* v = V1 + reach + i;
                const float y = mg_apply_diff<DIM>(a, X0, slice0, v, lo + i);
                q[lo + i] = y;
                pq += (double)(v[0] * y);
            });
            const double s_pq = cluster_sum(pq, 0);
            const float alpha = s_pq > 0.0 ? (float)(rho / s_pq) : 0.f;
            if (!(s_pq > 0.0) || alpha == 0.f) break;    // the same in every block
            double c = 0.0;
            struct Upd { float q, r, u; };
            mg_each<Upd, 8>(n, [&](int i, Upd& a) {
                const int g = lo + i;
                a.q = q[g]; a.r = r[g]; a.u = u[g];
            }, [&](int i, const Upd& a) {
                const int g = lo + i;
                const float rv = fmaf(-alpha, a.q, a.r);
                u[g] = fmaf(alpha, V1[reach + i], a.u);
                r[g] = rv;
                c += (double)(rv * rv);
            });
            rr = cluster_sum(c, 1);                      // (its barrier publishes r)
            ++it;
            if (rr <= A.rtol2 * rr0 || it == A.max_iters) break;
            const double rz = cluster_sum(precondition(), 2);
            beta = (float)(rz / rho);
            rho = rz;
        }
    }
    if (rank == 0 && tid == 0) {
        if (A.relres) A.relres[sample] = rr0 > 0.0 ? (float)sqrt(rr / rr0) : 0.0f;
        if (A.iters) A.iters[sample] = it;
    }
}

// ---- the stencil of level 0 ----------------------------------------------------------------------------------------
constexpr int MG_BLOCK = 128;

// nu at the Gauss points of all elements, [2 (nz - 1)][2 (ny - 1)][2 (nx - 1)] per sample, one block per Gauss line along x.
// nodal: from that field by Q1 interpolation; else the KL expansion from the tables of the call.
template <int DIM>
__global__ void __launch_bounds__(MG_BLOCK) mg_nu_kernel(const Params P, int b0, const float* __restrict__ nodal, float* __restrict__ nuq, long long sample) {
    dep_wait();
    dep_release();
    const int ngx = 2 * (P.nx - 1), ngy = 2 * (P.ny - 1);
    const int gy = blockIdx.x % ngy, gz = blockIdx.x / ngy, b = blockIdx.y;
    float* dst = nuq + b * sample + (long long)blockIdx.x * ngx;
    const float g[2] = {DN_GA, DN_GB};
    if (nodal) {
        const float* f = nodal + (long long)b * P.nodes + ((long long)(gz >> 1) * P.ny + (gy >> 1)) * P.nx;
        const float ty = g[gy & 1], tz = g[gz & 1];
        for (int gx = threadIdx.x; gx < ngx; gx += MG_BLOCK) {
            const float* c = f + (gx >> 1);
            const float tx = g[gx & 1];
            auto row = [&](const float* v) { return fmaf(tx, __ldg(v + 1) - __ldg(v), __ldg(v)); };
            auto plane = [&](const float* v) { const float lo = row(v), hi = row(v + P.nx); return fmaf(ty, hi - lo, lo); };
            float v = plane(c);
            if constexpr (DIM == 3) v = fmaf(tz, plane(c + (long long)P.nx * P.ny) - v, v);
            dst[gx] = v;
        }
        return;
    }
    __shared__ float a[DN_MAX_KL_MODES];                 // coefficients of cos(i pi x) on this line
    const int m = P.m;
    if ((int)threadIdx.x < m) {
        const int i = threadIdx.x;
        float s = 0.f;
        const float* c = P.ckl + (long long)(b0 + b) * m * m * (DIM == 3 ? m : 1);
        for (int j = 0; j < m; ++j) {
            float t;
            if constexpr (DIM == 3) {
                t = 0.f;
                for (int k = 0; k < m; ++k) t = fmaf(c[(i * m + j) * m + k], P.cg[2][k * P.gstride[2] + gz], t);
            } else {
                t = c[i * m + j];
            }
            s = fmaf(t, P.cg[1][j * P.gstride[1] + gy], s);
        }
        a[i] = s;
    }
    __syncthreads();
    for (int gx = threadIdx.x; gx < ngx; gx += MG_BLOCK) {
        float e = 0.f;
        for (int i = 0; i < m; ++i) e = fmaf(a[i], __ldg(P.cg[0] + i * P.gstride[0] + gx), e);
        dst[gx] = exp2f(e);
    }
}

// T[q][j]: W grad N_0 . grad N_j at Gauss point q of an element (bits: x, y, z).  Every other pair of corners (a, a ^ j) is a
// mirror image: T[q ^ a][j].
struct MgTable { float t[8][8]; };

// One thread per node: its row of K from the elements around it.
template <int DIM>
__global__ void __launch_bounds__(MG_BLOCK) mg_assemble_kernel(int nx, int ny, int nz, const __grid_constant__ MgTable T, const float* __restrict__ nuq_all,
                                                               float* __restrict__ mem, int offset, long long sample) {
    constexpr int NF = mg_nf(DIM), Q = 1 << DIM;
    dep_wait();
    dep_release();
    const int N = nx * ny * nz, i = blockIdx.x * MG_BLOCK + threadIdx.x;
    if (i >= N) return;
    const float* nuq = nuq_all + blockIdx.y * sample;
    float* K = mem + blockIdx.y * sample + offset + i;
    const int ix = i % nx, iy = (i / nx) % ny, iz = i / (nx * ny);
    const int ngx = 2 * (nx - 1), ngy = 2 * (ny - 1);
    if (ix == 0 || ix == nx - 1) {
        for (int o = 0; o < NF + 3; ++o) K[o * N] = 0.f;
        return;
    }
    float acc[DIM == 3 ? 27 : 9];
#pragma unroll
    for (int k = 0; k < (DIM == 3 ? 27 : 9); ++k) acc[k] = 0.f;
#pragma unroll
    for (int e = 0; e < Q; ++e) {                        // the element behind (bit 0) or before (bit 1) the node along each axis
        const int ex = ix - 1 + (e & 1), ey = iy - 1 + ((e >> 1) & 1), ez = DIM == 3 ? iz - 1 + (e >> 2) : 0;
        if (ey < 0 || ey >= ny - 1 || (DIM == 3 && (ez < 0 || ez >= nz - 1))) continue;
        const int a = e ^ (Q - 1);                       // this node's corner of it
        const float* v = nuq + ((long long)(2 * ez) * ngy + 2 * ey) * ngx + 2 * ex;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float nu = __ldg(v + (q & 1) + ((q >> 1) & 1) * ngx + (DIM == 3 ? (long long)(q >> 2) * ngy * ngx : 0));
#pragma unroll
            for (int j = 0; j < Q; ++j) {                // corner j: offset j - a along each axis
                const int ox = (j & 1) - (a & 1), oy = ((j >> 1) & 1) - ((a >> 1) & 1), oz = (j >> 2) - (a >> 2);
                const int k = ox + 1 + 3 * (oy + 1) + (DIM == 3 ? 9 * (oz + 1) : 0);
                acc[k] = fmaf(nu, T.t[q ^ a][j ^ a], acc[k]);
            }
        }
    }
    float d = 0.f, s = 0.f;
#pragma unroll
    for (int k = 0; k < (DIM == 3 ? 27 : 9); ++k) {      // couplings with Dirichlet nodes leave the stencil
        const int jx = ix + k % 3 - 1;
        if (jx == 0 || jx == nx - 1) { d -= acc[k]; acc[k] = 0.f; }
        s += fabsf(acc[k]);
    }
    constexpr int mid = DIM == 3 ? 13 : 4;
#pragma unroll
    for (int o = 0; o < NF; ++o) K[o * N] = acc[mid + mg_dx(o) + 3 * mg_dy(o) + 9 * mg_dz(o)];
    K[NF * N] = acc[mid];
    K[(NF + 1) * N] = s > 0.f ? MG_THETA / s : 0.f;
    K[(NF + 2) * N] = d;
}

// One axis of a shared level's coarse operator, one thread per node.
struct MgHalf { int n[3], m[3], size, src, dst; };
template <int DIM, int AX>
__global__ void __launch_bounds__(MG_BLOCK) mg_halve_kernel(const MgHalf H, float* mem, long long sample) {
    dep_wait();
    dep_release();
    const int i = blockIdx.x * MG_BLOCK + threadIdx.x;
    if (i >= H.size) return;
    float* own = mem + blockIdx.y * sample;
    mg_halve<DIM, AX, false>(own + H.src, H.n, own + H.dst, H.m, i);
}

MgTable mg_table(const dn_grid& g) {
    MgTable T{};
    const int dim = g.dim, Q = 1 << dim;
    const double h[3] = {1.0 / (g.nx - 1), 1.0 / (g.ny - 1), dim == 3 ? 1.0 / (g.nz - 1) : 1.0};
    const double ga[2] = {0.5 * (1.0 - 0.57735026918962576451), 0.5 * (1.0 + 0.57735026918962576451)};
    double W = 1.0;
    for (int a = 0; a < dim; ++a) W *= 0.5 * h[a];
    for (int q = 0; q < Q; ++q)
        for (int j = 0; j < Q; ++j) {
            double s = 0.0;
            for (int a = 0; a < dim; ++a) {              // the derivatives along a, times both shape functions along the others
                double t = W / (h[a] * h[a]) * ((j >> a) & 1 ? -1.0 : 1.0);
                for (int k = 0; k < dim; ++k) {
                    const double x = ga[(q >> k) & 1];
                    if (k != a) t *= (1.0 - x) * ((j >> k) & 1 ? x : 1.0 - x);
                }
                s += t;
            }
            T.t[q][j] = (float)s;
        }
    return T;
}

// ---- levels, memory, launch ----------------------------------------------------------------------------------------
// Everything but the pointers.  Returns false where a sample does not fit `C` blocks.
bool mg_arrange(const dn_problem& p, int C, MgArgs& A, size_t& smem) {
    const int dim = p.grid.dim, NF = mg_nf(dim);
    int n[3] = {p.grid.nx, p.grid.ny, dim == 3 ? p.grid.nz : 1};
    double h[3] = {1.0 / (n[0] - 1), 1.0 / (n[1] - 1), dim == 3 ? 1.0 / (n[2] - 1) : 1.0};
    A = MgArgs{};
    A.C = C;
    long long tmp[MG_LEVELS] = {};                       // scratch of halving a level
    for (;;) {
        MgLevel& L = A.lev[A.nlev];
        for (int a = 0; a < 3; ++a) L.n[a] = n[a];
        L.slice = dim == 3 ? n[0] * n[1] : n[0];
        L.N = n[0] * n[1] * n[2];
        L.reach = L.slice + (dim == 3 ? n[0] : 0) + 1;
        L.inv0 = 1.f / (float)n[0];
        L.invs = 1.f / (float)L.slice;
        const int rest[3] = {n[0] - 2, n[1], n[2]};      // what an axis has to halve
        double least = 0.0;
        for (int a = 0; a < dim; ++a) if (rest[a] >= 2 && (least == 0.0 || h[a] < least)) least = h[a];
        ++A.nlev;
        if (least == 0.0 || L.N <= MG_LAST) break;
        if (A.nlev == MG_LEVELS) return false;
        long long part = L.N;
        for (int a = 0; a < dim; ++a) {
            if (rest[a] < 2 || h[a] > 1.5 * least) continue;
            L.cut |= 1 << a;
            part = part / n[a];
            n[a] = a == 0 ? rest[0] / 2 + 2 : (n[a] + 1) / 2;
            h[a] *= 2.0;
            part *= n[a];
            tmp[A.nlev - 1] += L.reach + (NF + 1) * part;
        }
    }
    if (A.lev[A.nlev - 1].N > MG_LAST) return false;     // (an axis of faces only: rows of three columns have one left)
    {   // the last level: the Chebyshev iteration covers what is above half its lowest mode, the one that varies along x alone
        const double lowest = (2.0 - 2.0 * cos(3.14159265358979323846 / (n[0] - 1))) / (h[0] * h[0]);
        double diag = 0.0;
        for (int a = 0; a < dim; ++a) diag += 2.0 * (dim == 3 ? 4.0 / 9.0 : 2.0 / 3.0) / (h[a] * h[a]);
        const double high = MG_THETA, low = fmin(0.5 * MG_THETA * lowest / diag, 0.5 * MG_THETA);
        const double mid = 0.5 * (high + low), half = 0.5 * (high - low), steps = ceil(sqrt(high / low));
        A.steps = steps < MG_STEPS ? (int)steps : MG_STEPS;
        double rho = half / mid;
        A.gain[0] = (float)(1.0 / mid);
        for (int k = 1; k < A.steps; ++k) {
            const double next = 1.0 / (2.0 * mid / half - rho);
            A.momentum[k] = (float)(next * rho);
            A.gain[k] = (float)(2.0 * next / half);
            rho = next;
        }
    }
    const MgLevel& L0 = A.lev[0];
    while (C > 1 && A.shared_levels < A.nlev - 1 && (A.shared_levels == 0 || A.lev[A.shared_levels].N > mg_alone(dim))) ++A.shared_levels;
    const int SL = A.shared_levels;
    // the sample's memory
    long long off = 0, scratch = 1;
    for (int a = 0; a < dim; ++a) scratch *= 2 * (L0.n[a] - 1);      // before the solve it holds nu at the Gauss points
    for (int l = 0; l <= SL; ++l) {
        MgLevel& L = A.lev[l];
        off += L.reach;
        L.K = (int)off; off += (long long)(NF + (l ? 2 : 3)) * L.N;
        if (l < SL) {
            L.t = (int)off; off += L.N;
            if (l) { L.b = (int)off; off += L.N; L.x = (int)off; off += L.N; }
            if (tmp[l] > scratch) scratch = tmp[l];
        }
    }
    A.z = (int)off; off += L0.N;
    A.p = (int)off; off += L0.N;
    A.q = (int)off; off += L0.N;
    A.xs = (int)off; off += A.lev[SL].N;
    A.tmp = (int)off; off += scratch;
    A.sample = (off + 3) / 4 * 4;
    // shared memory: sums, staging, residual of block 0's levels, direction beyond the range, couplings of level 0, block 0's levels
    auto share = [&](long long N) { return (N + C - 1) / C; };
    long long v1 = 0, v2 = 0;
    auto most = [](long long& a, long long b) { if (b > a) a = b; };
    for (int l = 0; l < A.nlev; ++l) {
        const MgLevel& L = A.lev[l];
        most(v1, (l < SL ? share(L.N) : L.N) + 2ll * L.reach);
        if (l >= SL) { most(v1, tmp[l]); most(v2, L.N); }
        if (l + 1 == A.nlev) most(v1, 2 * (L.N + 2ll * L.reach));
    }
    long long at = 2ll * 3 * C * MG_WARPS;
    A.v1 = (int)at; at += v1;
    A.v2 = (int)at; at += v2;
    A.hp = (int)at; at += 2ll * L0.reach;
    for (int l = SL; l < A.nlev; ++l) {
        MgLevel& L = A.lev[l];
        at += L.reach;
        L.s = (int)at; at += (long long)(NF + 2) * L.N;
        if (l) { L.b = (int)at; at += L.N; }
        if (l > SL) { L.x = (int)at; at += L.N; }
    }
    A.k0 = -1;
    const long long k0 = NF * (share(L0.N) + L0.reach);
    if (dim == 2 && C > 1 && sizeof(float) * (at + k0) <= kMaxBlockShared) { A.k0 = (int)at; at += k0; }
    A.smem = (int)at;
    smem = sizeof(float) * (size_t)at;
    return smem <= kMaxBlockShared && C <= L0.N && off < (1ll << 31);
}

typedef void (*MgKernel)(const MgArgs);
MgKernel mg_kernel(int dim) { return dim == 3 ? mg_cluster_kernel<3> : mg_cluster_kernel<2>; }

struct MgLaunch {
    int C;
    size_t smem;
    cudaLaunchConfig_t config(int batch, cudaLaunchAttribute* at, cudaStream_t s) const {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(batch * C)); cfg.blockDim = dim3(MG_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = s;
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = (unsigned)C; at->val.clusterDim.y = 1; at->val.clusterDim.z = 1;
        cfg.attrs = at; cfg.numAttrs = 1;
        return cfg;
    }
};
// What is allowed are constants (see allow_shared); more than 8 blocks per cluster have to be asked for.
cudaError_t mg_allow(MgKernel k, size_t smem) {
    const cudaError_t e = allow_shared(k, smem);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// Blocks per cluster: from how many clusters the device holds at a time and the work of a block.
MgLaunch mg_search(const dn_problem& p) {
    MgLaunch best{};
    double cost = 0.0;
    for (int C = 1; C <= MG_MOST; ++C) {
        MgArgs A;
        MgLaunch l{};
        l.C = C;
        if (!mg_arrange(p, C, A, l.smem)) continue;
        const MgKernel k = mg_kernel(p.grid.dim);
        if (mg_allow(k, l.smem) != cudaSuccess) { (void)cudaGetLastError(); continue; }
        int active = 0;
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = l.config(p.batch, at, nullptr);
        if (cudaOccupancyMaxActiveClusters(&active, k, &cfg) != cudaSuccess || active < 1) { (void)cudaGetLastError(); continue; }
        const long long waves = (p.batch + active - 1) / active;
        // microseconds per iteration: barriers and passes, and the nodes of a block
        const double t = (double)waves * ((C > 1 ? 10.0 + 3.0 * A.shared_levels : 8.0) + (double)A.lev[0].N / C * (p.grid.dim == 3 ? 3e-3 : 8e-4));
        if (best.C == 0 || t < cost) { best = l; cost = t; }
    }
    return best;
}

}  // namespace

// Samples of three columns or more and at most 2^18 nodes that fit sixteen blocks.  Most fit eight, which every device can schedule;
// thin slabs, whose planes are much of a block's share, take more.  Where a device can hold no such cluster the launches per
// iteration serve (mg_blocks).  Solves to 1e-5, clusters and launches, milliseconds: 511^2 0.74 and 43, x 64 7.6 and 274; 2000 x 100 0.94
// and 151; 63^3 1.1 and 9.7, x 64 13.4 and 86; 100 x 100 x 8 (10 blocks) 1.3 and 11, x 64 9.8 and 44; 56 x 192 x 8 1.8 and 20.
bool mg_applicable(const dn_problem& p) {
    const long long nodes = (long long)p.grid.nx * p.grid.ny * (p.grid.dim == 3 ? p.grid.nz : 1);
    if (p.grid.nx < 3 || nodes > (1 << 18)) return false;
    for (int C = 1; C <= MG_MOST; ++C) {
        MgArgs A;
        size_t smem;
        if (mg_arrange(p, C, A, smem)) return true;
    }
    return false;
}

// Bytes per sample; the nodal field of the KL expansion at the nodes stands behind each sample's memory.
size_t mg_sample_bytes(const dn_problem& p) {
    MgArgs A;
    size_t smem;
    long long most = 0;                                  // of any number of blocks
    for (int C = 1; C <= 2; ++C) {                       // (it depends on whether there are several)
        mg_arrange(p, C, A, smem);
        if (A.sample > most) most = A.sample;
    }
    return sizeof(float) * (size_t)(most + (p.nu_mode == DN_NU_KL_NODAL ? (A.lev[0].N + 3) / 4 * 4 : 0));
}

// Blocks per cluster for `batch` samples at a time; 0 where the device can hold no cluster (then it is asked again by the next call).
int mg_blocks(const dn_problem& p, int batch) {
    dn_problem q = p;
    q.batch = batch;
    const MgLaunch l = memo_geometry<MgLaunch>(q, sm_count(), [&]() { return mg_search(q); });
    return l.C ? l.C : mg_search(q).C;
}

// Solves samples b0 .. b0 + nb - 1.  P: parameters of the call that left K u - F in r (its KL tables are read); mem: nb times
// mg_sample_bytes.  u, r, relres and iters are the whole batch's.
cudaError_t mg_solve(const dn_problem& p, const Params& P, int C, int b0, int nb, float* mem, float* u, float* r, int max_iters, float rtol,
                     float* relres, int32_t* iters, cudaStream_t s) {
    const int dim = p.grid.dim;
    MgArgs A;
    MgLaunch l{};
    l.C = C;
    if (!mg_arrange(p, C, A, l.smem)) return cudaErrorInvalidValue;
    const long long nodes = A.lev[0].N;
    const float* nodal = nullptr;
    if (p.nu_mode == DN_NU_NODAL) nodal = p.nu + b0 * nodes;
    if (p.nu_mode == DN_NU_KL_NODAL) {
        size_t mpow = 1;
        for (int a = 0; a < dim; ++a) mpow *= (size_t)p.kl_modes;
        float* field = mem + A.sample * nb;
        const cudaError_t e = launch_kl_field(p.grid, nb, p.kl_modes, p.kl_w + (size_t)b0 * mpow, field, s);
        if (e != cudaSuccess) return e;
        nodal = field;
    }
    const int nz = dim == 3 ? p.grid.nz : 1;
    const dim3 lines((unsigned)(2 * (p.grid.ny - 1) * (dim == 3 ? 2 * (nz - 1) : 1)), (unsigned)nb);
    const dim3 rows((unsigned)((nodes + MG_BLOCK - 1) / MG_BLOCK), (unsigned)nb);
    const MgTable T = mg_table(p.grid);
    float* nuq = mem + A.tmp;
    cudaError_t e = dim == 3 ? launch_dependent(mg_nu_kernel<3>, lines, dim3(MG_BLOCK), 0, s, P, b0, nodal, nuq, A.sample)
                             : launch_dependent(mg_nu_kernel<2>, lines, dim3(MG_BLOCK), 0, s, P, b0, nodal, nuq, A.sample);
    if (e != cudaSuccess) return e;
    e = dim == 3 ? launch_dependent(mg_assemble_kernel<3>, rows, dim3(MG_BLOCK), 0, s, p.grid.nx, p.grid.ny, nz, T, nuq, mem, A.lev[0].K, A.sample)
                 : launch_dependent(mg_assemble_kernel<2>, rows, dim3(MG_BLOCK), 0, s, p.grid.nx, p.grid.ny, 1, T, nuq, mem, A.lev[0].K, A.sample);
    if (e != cudaSuccess) return e;
    for (int lv = 0; lv < A.shared_levels; ++lv) {
        const MgLevel& L = A.lev[lv];
        const MgLevel& M = A.lev[lv + 1];
        MgHalf H{};
        int n[3] = {L.n[0], L.n[1], L.n[2]}, src = L.K, tmp = A.tmp, left = L.cut;
        for (int a = 0; a < dim; ++a) {
            if (!((left >> a) & 1)) continue;
            left &= ~(1 << a);
            H.src = src;
            H.dst = left ? tmp + L.reach : M.K;
            for (int k = 0; k < 3; ++k) H.n[k] = H.m[k] = n[k];
            H.m[a] = n[a] = M.n[a];
            H.size = n[0] * n[1] * n[2];
            const dim3 grid((unsigned)((H.size + MG_BLOCK - 1) / MG_BLOCK), (unsigned)nb);
            if (dim == 2) e = a == 0 ? launch_dependent(mg_halve_kernel<2, 0>, grid, dim3(MG_BLOCK), 0, s, H, mem, A.sample)
                                     : launch_dependent(mg_halve_kernel<2, 1>, grid, dim3(MG_BLOCK), 0, s, H, mem, A.sample);
            else e = a == 0 ? launch_dependent(mg_halve_kernel<3, 0>, grid, dim3(MG_BLOCK), 0, s, H, mem, A.sample)
                   : a == 1 ? launch_dependent(mg_halve_kernel<3, 1>, grid, dim3(MG_BLOCK), 0, s, H, mem, A.sample)
                            : launch_dependent(mg_halve_kernel<3, 2>, grid, dim3(MG_BLOCK), 0, s, H, mem, A.sample);
            if (e != cudaSuccess) return e;
            src = H.dst;
            tmp += L.reach + (mg_nf(dim) + 1) * H.size;
        }
    }
    A.max_iters = max_iters;
    A.mem = mem; A.u = u + b0 * nodes; A.r = r + b0 * nodes;
    A.rtol2 = (double)rtol * (double)rtol;
    A.relres = relres ? relres + b0 : nullptr;
    A.iters = iters ? iters + b0 : nullptr;
    const MgKernel k = mg_kernel(dim);
    e = mg_allow(k, l.smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = l.config(nb, at, s);
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k, A);
}

}  // namespace dn
