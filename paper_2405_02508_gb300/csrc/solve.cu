// solve.cu -- Laplacian preconditioning of vertex updates (Nicolet et al., "Large Steps in Inverse Rendering
// of Geometry", 2021), which the paper uses for all of its mesh optimisations (Sec. 5 and Supp. B, lambda 16).
//
// The vertex positions x [V, 3] are reparameterised as u = M x with M = I + lambda L, L the combinatorial
// Laplacian of the meshes' edge graph (L_ii = number of neighbours of i, L_ij = -1 for every edge ij).  A
// step then needs M x (once, to start) and two solves M y = b per step: the gradient with respect to u,
// M^-1 dL/dx, and the positions x = M^-1 u after the update.  M is symmetric positive definite (its
// eigenvalues are 1 + lambda * those of L, all >= 1), so the solves are conjugate gradients on the device:
// FP32 vectors, dot products of exact products in FP64 or two-float sums (about 48 bits), all three coordinate
// columns as one block-diagonal system, the iteration scalars kept on the device (so a solve can be captured in a graph): one launch that ends once the residual is below
// the tolerance, or, for systems beyond one resident grid, a fixed sequence of launches that become no-ops then.
//
// The CSR edge graph is built once per mesh on the host (mer_laplacian_csr).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "mer.h"

namespace mer {

constexpr int kSolveThreads = 256;

// Device scalars of one solve, at the start of the solve workspace.
struct CgState {
    double rr;      // r . r of the current residual
    double rr_new;  // r . r after the update of this iteration
    double pAp;     // p . M p
    double rr0;     // b . b (the tolerance is relative to it)
    double tol2;    // (rel_tol)^2 * rr0
    int done;       // 1 once rr <= tol2 (later launches return at once)
    int iters;      // iterations run
    int failed;     // 1 if a grid-wide exchange ran out of polls (the solution is then not valid)
    int pad[3];
};

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;  // valid in thread 0
}

// Row i of y = (I + lambda L) x: x_i + lambda (deg_i x_i - sum of the neighbours' x_j).
__device__ __forceinline__ void apply_row(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                          float lambda, const float* __restrict__ x, int64_t i, float y[3]) {
    const int64_t b = row_ptr[i], e = row_ptr[i + 1];
    float sx = 0.f, sy = 0.f, sz = 0.f;
    for (int64_t k = b; k < e; ++k) {
        const int64_t j = col[k];
        sx += x[3 * j];
        sy += x[3 * j + 1];
        sz += x[3 * j + 2];
    }
    const float deg = (float)(e - b);
    const float xi = x[3 * i], yi = x[3 * i + 1], zi = x[3 * i + 2];
    y[0] = xi + lambda * (deg * xi - sx);
    y[1] = yi + lambda * (deg * yi - sy);
    y[2] = zi + lambda * (deg * zi - sz);
}

__global__ void __launch_bounds__(kSolveThreads) k_apply(const int64_t* __restrict__ row_ptr,
                                                         const int32_t* __restrict__ col, int64_t V, float lambda,
                                                         const float* __restrict__ x, float* __restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
    float r[3];
    apply_row(row_ptr, col, lambda, x, i, r);
    y[3 * i] = r[0];
    y[3 * i + 1] = r[1];
    y[3 * i + 2] = r[2];
}

// r = b - M x, p = r; accumulates r . r into st->rr and b . b into st->rr0.
__global__ void __launch_bounds__(kSolveThreads) k_cg_init(const int64_t* __restrict__ row_ptr,
                                                           const int32_t* __restrict__ col, int64_t V, float lambda,
                                                           const float* __restrict__ b, const float* __restrict__ x,
                                                           float* __restrict__ r, float* __restrict__ p,
                                                           CgState* st) {
    __shared__ double sh[kSolveThreads / 32];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double rr = 0.0, bb = 0.0;
    if (i < V) {
        float mx[3];
        apply_row(row_ptr, col, lambda, x, i, mx);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float bi = b[3 * i + c];
            const float ri = bi - mx[c];
            r[3 * i + c] = ri;
            p[3 * i + c] = ri;
            rr += (double)ri * ri;
            bb += (double)bi * bi;
        }
    }
    const double s1 = block_sum(rr, sh);
    __syncthreads();
    const double s2 = block_sum(bb, sh);
    if (threadIdx.x == 0) {
        atomicAdd(&st->rr, s1);
        atomicAdd(&st->rr0, s2);
    }
}

__global__ void k_cg_start(CgState* st, float rel_tol) {
    st->tol2 = (double)rel_tol * rel_tol * st->rr0;
    st->done = st->rr <= st->tol2 ? 1 : 0;
    st->iters = 0;
    st->pAp = 0.0;
    st->rr_new = 0.0;
}

// Ap = M p, pAp = p . Ap
__global__ void __launch_bounds__(kSolveThreads) k_cg_matvec(const int64_t* __restrict__ row_ptr,
                                                             const int32_t* __restrict__ col, int64_t V,
                                                             float lambda, const float* __restrict__ p,
                                                             float* __restrict__ Ap, CgState* st) {
    __shared__ double sh[kSolveThreads / 32];
    if (st->done) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double d = 0.0;
    if (i < V) {
        float y[3];
        apply_row(row_ptr, col, lambda, p, i, y);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Ap[3 * i + c] = y[c];
            d += (double)p[3 * i + c] * y[c];
        }
    }
    const double s = block_sum(d, sh);
    if (threadIdx.x == 0) atomicAdd(&st->pAp, s);
}

// alpha = rr / pAp; x += alpha p; r -= alpha Ap; rr_new = r . r
__global__ void __launch_bounds__(kSolveThreads) k_cg_update(int64_t V, const float* __restrict__ p,
                                                             const float* __restrict__ Ap, float* __restrict__ x,
                                                             float* __restrict__ r, CgState* st) {
    __shared__ double sh[kSolveThreads / 32];
    if (st->done) return;
    const float alpha = st->pAp > 0.0 ? (float)(st->rr / st->pAp) : 0.f;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double d = 0.0;
    if (i < V) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[3 * i + c] += alpha * p[3 * i + c];
            const float ri = r[3 * i + c] - alpha * Ap[3 * i + c];
            r[3 * i + c] = ri;
            d += (double)ri * ri;
        }
    }
    const double s = block_sum(d, sh);
    if (threadIdx.x == 0) atomicAdd(&st->rr_new, s);
}

// beta = rr_new / rr; p = r + beta p  (the scalars are advanced by k_cg_next afterwards)
__global__ void __launch_bounds__(kSolveThreads) k_cg_direction(int64_t V, const float* __restrict__ r,
                                                                float* __restrict__ p, const CgState* st) {
    if (st->done) return;
    const float beta = st->rr > 0.0 ? (float)(st->rr_new / st->rr) : 0.f;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= V) return;
#pragma unroll
    for (int c = 0; c < 3; ++c) p[3 * i + c] = r[3 * i + c] + beta * p[3 * i + c];
}

__global__ void k_cg_next(CgState* st) {
    if (st->done) return;
    st->rr = st->rr_new;
    st->rr_new = 0.0;
    st->pAp = 0.0;
    st->iters += 1;
    if (st->rr <= st->tol2) st->done = 1;
}


// ---- the whole solve in one launch ----
//
// A solve of the sizes meshes have (a head mesh: 65,538 rows) is latency: per iteration 1.6 MB of vectors and 1.8 MB
// of edge graph, all in L2, against four dependent launches.  So while the rows fit the threads of one resident grid,
// the solve is one kernel: a thread keeps its rows of x, r, p, M p and the neighbour ids in registers, r and p also go
// to shared memory for the CTA's own neighbours and to the workspace (16 bytes a row) for the other CTAs', and an
// iteration has two steps that all threads take together, the two dot products.  p_new = r + beta p_old is formed by
// whoever needs it, for the row itself and for every neighbour (the same operation on the same values, so the same
// bits), which removes a third step.
// A step is a sum over the CTA, over the CTAs of its cluster (in shared memory, with the hardware's cluster barrier),
// and over the clusters: the first CTA of each publishes the sum with the step's number and reads the others'.  All
// CTAs reading all CTAs' sums instead cost 5,000 cycles an exchange with 128 of them.
// The first two sums are FP64; those of the iterations are sums of exact products (each split in two floats by an FMA) in
// two-float arithmetic, about 48 bits against FP64's 53, and so are the iteration's two quotients before they are rounded to
// the FP32 factors alpha and beta.  GB300's FP64 pipe issues one warp instruction in 16 cycles, and the 64-bit sums and
// divisions took longer than the exchanges (9 us an iteration of 258 rows, now 2.8).  The vectors are FP32, so the five bits
// are far below what a solve can show: in 576 solves of 258 to 211,602 rows of at most 8 neighbours (lambda 8, 16 and
// 32, rough, smooth and mixed right-hand sides, cold and warm starts) iterations and solutions had the same bits as the
// launch sequence, whose sums are FP64, hence the same errors against a 64-bit solution.
// Measured (lambda 16, residual 1e-6, 79 and 49 iterations): 65,538 rows 3,760 -> 607 us, 642 rows 2,795 -> 155 us.
constexpr int kCgThreads = 512;         // per CTA of the cluster form (one CTA per SM, up to 128 registers a thread)
constexpr int kCgLocalThreads = 1024;   // the single-CTA form
constexpr int kCgNeighbours = 8;        // neighbour ids kept in registers (a closed mesh averages 6)
// Rows with more neighbours than this (the poles of a sphere of meridians, the hub of a fan) are summed by their warp, 32
// neighbours at a time (hub_sums): one thread going through them, each a trip to L2 and back, held up every iteration of the
// whole solve.  A sphere of 64 x 1,024 quads 21,455 us (the launches 12,852), now 1,430; one of 200 x 1,024 22,600 (13,930) and
// 3,550; a fan of 5,000 28,360 (15,620) and 900.  (In the one-CTA form the trip is to shared memory: a fan of 900 478, the
// launches 4,104.)
constexpr int kCgHub = 64;
constexpr unsigned kCgPolls = 1u << 21;  // polls of one exchange (about a second) before the solve gives up
constexpr int kCgCluster = 8;           // CTAs of a cluster
constexpr int kCgMaxClusters = 32;      // one slot per lane of a warp

// An unevaluated sum hi + lo of two floats.
struct F2 {
    float hi, lo;
};

__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {  // Knuth's exact two-sum of the high parts, then renormalised
    const float s = __fadd_rn(a.hi, b.hi);
    const float bb = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    const float t = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    F2 r;
    r.hi = __fadd_rn(s, t);
    r.lo = __fsub_rn(t, __fsub_rn(r.hi, s));
    return r;
}

__device__ __forceinline__ F2 f2_mul_add(float a, float b, F2 c) {  // c + a b, the product exact
    F2 p;
    p.hi = __fmul_rn(a, b);
    p.lo = __fmaf_rn(a, b, -p.hi);
    return f2_add(c, p);
}

// 16-byte row of an exchanged vector, through L2 (other SMs write it).
__device__ __forceinline__ float4 cg_load(const float4* p) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void cg_store(float4* p, float x, float y, float z) {
    asm volatile("st.global.cg.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(0.f) : "memory");
}

// A cluster's published partial sum, a two-float sum or the two halves of a double: each 32-bit part travels with the
// number of its step in one 8-byte word, so a word that carries the step's number carries its value.  Two sets of
// slots alternate: a cluster can write step e + 2 only after every cluster has published e + 1, hence has read step e.
struct __align__(16) CgSlot {
    unsigned long long a, b;
};

struct CgShared {
    double part[kCgLocalThreads / 32];  // F2 or double partial sums of the warps
    uint2 rank[kCgCluster];             // in a cluster's first CTA: the two halves of its CTAs' sums
    float coef;                         // alpha or beta
    int stop;                           // leave the iteration: converged, or an exchange failed
    int failed;
};

__device__ __forceinline__ double sum_add(double a, double b) { return a + b; }
__device__ __forceinline__ F2 sum_add(F2 a, F2 b) { return f2_add(a, b); }
template <typename T>
__device__ __forceinline__ T from_bits(unsigned a, unsigned b);
template <>
__device__ __forceinline__ double from_bits<double>(unsigned a, unsigned b) { return __hiloint2double((int)a, (int)b); }
template <>
__device__ __forceinline__ F2 from_bits<F2>(unsigned a, unsigned b) {
    F2 v;
    v.hi = __uint_as_float(a);
    v.lo = __uint_as_float(b);
    return v;
}
__device__ __forceinline__ void to_bits(double v, unsigned& a, unsigned& b) {
    a = (unsigned)__double2hiint(v);
    b = (unsigned)__double2loint(v);
}
__device__ __forceinline__ void to_bits(F2 v, unsigned& a, unsigned& b) {
    a = __float_as_uint(v.hi);
    b = __float_as_uint(v.lo);
}

template <typename T>
__device__ __forceinline__ T warp_total(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned a, b;
        to_bits(v, a, b);
        a = __shfl_xor_sync(0xffffffffu, a, o);
        b = __shfl_xor_sync(0xffffffffu, b, o);
        v = sum_add(v, from_bits<T>(a, b));
    }
    return v;
}

// The shared-memory address of CTA `rank` of the cluster that corresponds to p here.
__device__ __forceinline__ unsigned peer_shared(const void* p, unsigned rank) {
    unsigned a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

// (Aligned: a warp executes it together, and callers come from code that only some of its lanes ran.)
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sum of v over all threads of the launch, handed to `then` (in one thread of the CTA, or of every cluster: the scalars
// of the iteration, written to S and copied to the cluster's other CTAs); all threads leave after it.  PUBLISH: all
// writes to the exchanged vectors made before the call are visible to every thread after it (without it, only that
// every thread has done its reads).
template <bool CLUSTER, bool PUBLISH, typename T, typename Then>
__device__ __forceinline__ void cg_sum(T v, unsigned step, CgSlot* slots, unsigned max_polls, CgShared& S, Then then) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const T zero = from_bits<T>(0u, 0u);
    T* part = reinterpret_cast<T*>(S.part);
    v = warp_total(v);
    if (lane == 0) part[warp] = v;
    __syncthreads();
    if (warp == 0) v = warp_total(lane < nw ? part[lane] : zero);
    if (!CLUSTER) {
        if (threadIdx.x == 0) then(v);
        __syncthreads();
        return;
    }
    const unsigned rank = blockIdx.x % kCgCluster, cluster = blockIdx.x / kCgCluster, n_clusters = gridDim.x / kCgCluster;
    if (threadIdx.x == 0) {
        unsigned a, b;
        to_bits(v, a, b);
        asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(peer_shared(S.rank + rank, 0u)), "r"(a), "r"(b) : "memory");
    }
    cluster_sync();
    if (rank == 0 && warp == 0) {
        const uint2 w = S.rank[lane % kCgCluster];
        v = warp_total(lane < kCgCluster ? from_bits<T>(w.x, w.y) : zero);
        bool ok = true;
        if (n_clusters > 1) {
            CgSlot* set = slots + (step & 1u) * kCgMaxClusters;
            const unsigned long long tag = (unsigned long long)step << 32;
            if (lane == 0) {
                unsigned a, b;
                to_bits(v, a, b);
                if (PUBLISH) __threadfence();
                asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(set + cluster), "l"(tag | a), "l"(tag | b)
                             : "memory");
            }
            unsigned long long wa = tag, wb = tag;
            for (unsigned polls = 0;; ++polls) {
                if (lane < (int)n_clusters)
                    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];"
                                 : "=l"(wa), "=l"(wb) : "l"(set + lane) : "memory");
                if (__all_sync(0xffffffffu, (unsigned)(wa >> 32) == step && (unsigned)(wb >> 32) == step)) break;
                if (polls >= max_polls) {
                    ok = false;
                    break;
                }
            }
            if (PUBLISH) __threadfence();
            v = warp_total(from_bits<T>((unsigned)wa, (unsigned)wb));
        }
        if (lane == 0) {
            then(v);
            if (!ok) S.stop = S.failed = 1;
        }
        __syncwarp();
        const float coef = S.coef;
        const int stop = S.stop, failed = S.failed;
        if (lane > 0 && lane < kCgCluster) {
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_shared(&S.coef, lane)), "f"(coef) : "memory");
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_shared(&S.stop, lane)), "r"(stop) : "memory");
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_shared(&S.failed, lane)), "r"(failed) : "memory");
        }
    }
    cluster_sync();
}

// Sums over the neighbours beyond kCgNeighbours of the rows of a warp's lanes that have more than kCgHub, each by all the
// lanes of mask m (the first ones of the warp); zero for the other lanes.  Out of line: inlined, its registers cost every
// iteration of every solve 2 to 4 % (now below 1 %; 7 % in the form of four rows a thread, which spills).
__device__ __noinline__ float4 hub_sums(const int32_t* col, int64_t first, int deg, const float4* r, const float4* p, float beta,
                                        unsigned m) {
    const int lane = threadIdx.x & 31, lanes = __popc(m);
    float4 mine = make_float4(0.f, 0.f, 0.f, 0.f);
    for (unsigned hubs = __ballot_sync(m, deg > kCgHub); hubs; hubs &= hubs - 1) {
        const int src = __ffs((int)hubs) - 1;
        const long long f = __shfl_sync(m, (long long)first, src);
        const int n = __shfl_sync(m, deg, src);
        float s[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
        for (int j = kCgNeighbours + lane; j < n; j += lanes) {
            const int q = __ldg(col + f + j);
            const float4 a = cg_load(r + q), o = cg_load(p + q);
            s[0] += a.x + beta * o.x;
            s[1] += a.y + beta * o.y;
            s[2] += a.z + beta * o.z;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float v = __shfl_down_sync(m, s[c], o);
                if (lane + o < lanes) s[c] += v;
            }
            s[c] = __shfl_sync(m, s[c], 0);
        }
        if (lane == src) mine = make_float4(s[0], s[1], s[2], 0.f);
    }
    return mine;
}

// a / b rounded to a float, for two-float a and b > 0: the correctly rounded quotient of the high parts and one
// correction with the exact remainder.
__device__ __forceinline__ float f2_ratio(F2 a, F2 b) {
    const float q = __fdiv_rn(a.hi, b.hi);
    const float rem = __fadd_rn(__fmaf_rn(-q, b.hi, a.hi), __fmaf_rn(-q, b.lo, a.lo));
    return __fadd_rn(q, __fdiv_rn(rem, b.hi));
}

// Up to R rows a thread, `rows` a CTA.  CLUSTER: clusters of kCgCluster CTAs, all resident; otherwise one CTA.
template <int R, bool CLUSTER>
__global__ void __launch_bounds__(CLUSTER ? kCgThreads : kCgLocalThreads, 1)
    k_cg_solve(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col, int V, float lambda,
               const float* __restrict__ b, float* __restrict__ x, float4* r_ws, float4* p_ws, CgSlot* slots, CgState* st,
               int max_iters, float rel_tol, int rows, unsigned max_polls) {
    extern __shared__ float4 sm[];
    __shared__ CgShared S;
    // residual and search direction (two buffers) of the CTA's rows; CLUSTER: also in the workspace, for the other CTAs
    constexpr int kT = CLUSTER ? kCgThreads : kCgLocalThreads;
    constexpr int kN = kT * R;
    const int base = (int)blockIdx.x * rows;
    int row[R], deg[R], nb[R][kCgNeighbours];
    int64_t first[R];
    float xr[R][3], rr_[R][3], pr[R][3], ap[R][3];
    double s_rr = 0.0, s_bb = 0.0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        row[k] = base + k * kT + (int)threadIdx.x;
        const bool in = k * kT + (int)threadIdx.x < rows && row[k] < V;
        if (!in) row[k] = -1;
        const int i = in ? row[k] : 0;
        first[k] = row_ptr[i];
        deg[k] = in ? (int)(row_ptr[i + 1] - first[k]) : 0;
#pragma unroll
        for (int j = 0; j < kCgNeighbours; ++j) {  // a row of this CTA: its complement within the CTA
            const int q = j < deg[k] ? col[first[k] + j] : base;
            nb[k][j] = (unsigned)(q - base) < (unsigned)rows ? ~(q - base) : q;
        }
        float mx[3];
        apply_row(row_ptr, col, lambda, x, i, mx);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float bi = b[3 * (size_t)i + c];
            xr[k][c] = x[3 * (size_t)i + c];
            rr_[k][c] = bi - mx[c];
            pr[k][c] = 0.f;
            if (in) {
                s_rr += (double)rr_[k][c] * rr_[k][c];
                s_bb += (double)bi * bi;
            }
        }
        if (in) {
            sm[i - base] = make_float4(rr_[k][0], rr_[k][1], rr_[k][2], 0.f);
            sm[kN + i - base] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (CLUSTER) {
                cg_store(r_ws + i, rr_[k][0], rr_[k][1], rr_[k][2]);
                cg_store(p_ws + i, 0.f, 0.f, 0.f);
            }
        }
    }
    // Scalars of the solve, kept by the thread that forms them (the same in every cluster): r . r scaled by 2^(-2e), with
    // e from the first residual, so that the two-float products stay far from the ends of the FP32 range.
    double rr0 = 0.0, tol2 = 0.0, unit = 1.0;
    F2 rr = {0.f, 0.f};
    if (threadIdx.x == 0) S.stop = S.failed = 0;
    if (CLUSTER) cluster_sync();  // every CTA of the cluster has started and cleared its words
    unsigned step = 1;
    cg_sum<CLUSTER, true>(s_bb, step++, slots, max_polls, S, [&](double v) { rr0 = v; });
    cg_sum<CLUSTER, false>(s_rr, step++, slots, max_polls, S, [&](double v) {
        const int e = min(max((int)((__double2hiint(v) >> 20) & 0x7ff) - 1023, -240), 240) / 2;
        S.coef = __int_as_float((127 - e) << 23);  // 2^-e
        unit = (double)S.coef * (double)S.coef;
        tol2 = (double)rel_tol * rel_tol * rr0;
        if (v <= tol2) S.stop = 1;
        v *= unit;
        rr.hi = (float)v;
        rr.lo = (float)(v - (double)rr.hi);
    });
    const float scale = S.coef;
    float beta = 0.f;
    int it = 0;
    bool hub = false;  // a lane of the warp has a row for hub_sums
    if (CLUSTER) {
#pragma unroll
        for (int k = 0; k < R; ++k) hub |= deg[k] > kCgHub;
        hub = __any_sync(0xffffffffu, hub);
    }
    while (!S.stop && it < max_iters) {
        // p = r + beta p for the row and its neighbours, M p, p . M p
        const float4 *p_old = p_ws + (size_t)(it & 1) * V, *ps_old = sm + kN + (it & 1) * kN;
        float4 *p_new = p_ws + (size_t)((it + 1) & 1) * V, *ps_new = sm + kN + ((it + 1) & 1) * kN;
        F2 d = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const unsigned have = CLUSTER && hub ? __ballot_sync(0xffffffffu, row[k] >= 0) : 0u;
            if (row[k] < 0) continue;
            float4 nr[kCgNeighbours], np[kCgNeighbours];
#pragma unroll
            for (int j = 0; j < kCgNeighbours; ++j) {  // all gathers in flight together
                const int q = nb[k][j];
                if (!CLUSTER || q < 0) {
                    nr[j] = sm[~q];
                    np[j] = ps_old[~q];
                } else {
                    nr[j] = cg_load(r_ws + q);
                    np[j] = cg_load(p_old + q);
                }
            }
            float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
            for (int j = 0; j < kCgNeighbours; ++j) {
                const float px = nr[j].x + beta * np[j].x, py = nr[j].y + beta * np[j].y, pz = nr[j].z + beta * np[j].z;
                if (j < deg[k]) {
                    sx += px;
                    sy += py;
                    sz += pz;
                }
            }
            int end = deg[k];
            if (CLUSTER && hub) {
                const float4 h = hub_sums(col, first[k], deg[k], r_ws, p_old, beta, have);
                sx += h.x;
                sy += h.y;
                sz += h.z;
                if (end > kCgHub) end = 0;
            }
            for (int j = kCgNeighbours; j < end; ++j) {
                const int q = __ldg(col + first[k] + j);
                const float4 a = CLUSTER ? cg_load(r_ws + q) : sm[q], o = CLUSTER ? cg_load(p_old + q) : ps_old[q];
                sx += a.x + beta * o.x;
                sy += a.y + beta * o.y;
                sz += a.z + beta * o.z;
            }
            const float sum[3] = {sx, sy, sz};
            const float fd = (float)deg[k];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                pr[k][c] = rr_[k][c] + beta * pr[k][c];
                ap[k][c] = pr[k][c] + lambda * (fd * pr[k][c] - sum[c]);
                d = f2_mul_add(scale * pr[k][c], scale * ap[k][c], d);
            }
            ps_new[row[k] - base] = make_float4(pr[k][0], pr[k][1], pr[k][2], 0.f);
            if (CLUSTER) cg_store(p_new + row[k], pr[k][0], pr[k][1], pr[k][2]);
        }
        // p_new is read after the next exchange only, so this one publishes nothing
        cg_sum<CLUSTER, false>(d, step++, slots, max_polls, S, [&](F2 v) { S.coef = v.hi > 0.f ? f2_ratio(rr, v) : 0.f; });
        if (S.stop) break;
        // x += alpha p, r -= alpha M p, r . r
        const float alpha = S.coef;
        d.hi = d.lo = 0.f;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            if (row[k] < 0) continue;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                xr[k][c] += alpha * pr[k][c];
                rr_[k][c] -= alpha * ap[k][c];
                d = f2_mul_add(scale * rr_[k][c], scale * rr_[k][c], d);
            }
            sm[row[k] - base] = make_float4(rr_[k][0], rr_[k][1], rr_[k][2], 0.f);
            if (CLUSTER) cg_store(r_ws + row[k], rr_[k][0], rr_[k][1], rr_[k][2]);
        }
        cg_sum<CLUSTER, true>(d, step++, slots, max_polls, S, [&](F2 v) {
            S.coef = rr.hi > 0.f ? f2_ratio(v, rr) : 0.f;
            rr = v;
            if (((double)v.hi + (double)v.lo) <= tol2 * unit) S.stop = 1;
        });
        beta = S.coef;
        ++it;
    }
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (row[k] < 0) continue;
#pragma unroll
        for (int c = 0; c < 3; ++c)  // a solve that gave up must not pass for one
            x[3 * (size_t)row[k] + c] = S.failed ? __int_as_float(0x7fffffff) : xr[k][c];
    }
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) {
            st->rr = ((double)rr.hi + (double)rr.lo) / unit;
            st->rr0 = rr0;
            st->tol2 = tol2;
            st->done = S.stop;
            st->iters = it;
        }
        if (S.failed) atomicExch(&st->failed, 1);
    }
}

}  // namespace mer

using namespace mer;

namespace {
inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
inline unsigned blocks_for(int64_t V) { return (unsigned)((V + kSolveThreads - 1) / kSolveThreads); }

// Exchange slots of the one-launch form: two sets, one slot per cluster.
constexpr size_t kCgSlotBytes = 2 * kCgMaxClusters * sizeof(CgSlot);

// The solve in one launch with R rows a thread, in one CTA or in clusters; cudaErrorNotSupported if the clusters do not
// all fit on the device at once.
template <int R, bool CLUSTER>
cudaError_t launch_cg(const int64_t* row_ptr, const int32_t* col, int V, float lambda, const float* b, float* x,
                      float4* r, float4* p, CgSlot* slots, CgState* st, int max_iters, float rel_tol, unsigned max_polls,
                      cudaStream_t s) {
    constexpr int kT = CLUSTER ? kCgThreads : kCgLocalThreads;
    constexpr int kBytes = 3 * kT * R * (int)sizeof(float4);
    constexpr int kUnit = CLUSTER ? kCgCluster : 1;
    auto kernel = k_cg_solve<R, CLUSTER>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
    if (e != cudaSuccess) return e;
    const int units = (V + kUnit * kT * R - 1) / (kUnit * kT * R);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)(units * kUnit));
    c.blockDim = dim3(kT);
    c.dynamicSmemBytes = kBytes;
    c.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kUnit;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;  // all CTAs start together or none
    attr[1].val.cooperative = 1;
    c.attrs = attr;
    if (CLUSTER) {
        c.numAttrs = 1;
        int fit = 0;
        if (units > 1) {
            e = cudaOccupancyMaxActiveClusters(&fit, kernel, &c);
            if (e != cudaSuccess) return e;
            if (fit < units) return cudaErrorNotSupported;
            c.numAttrs = 2;
        }
    }
    const int rows = (V + units * kUnit - 1) / (units * kUnit);
    return cudaLaunchKernelEx(&c, kernel, row_ptr, col, V, lambda, b, x, r, p, slots, st, max_iters, rel_tol, rows,
                              max_polls);
}

// The solve as a fixed sequence of launches (the state cleared before).
int solve_launches(const int64_t* row_ptr, const int32_t* col, int64_t V, float lambda, const float* b, float* x,
                   int max_iters, float rel_tol, char* base, cudaStream_t s) {
    CgState* st = reinterpret_cast<CgState*>(base);
    const size_t vec = align256((size_t)V * 3 * sizeof(float));
    float* r = reinterpret_cast<float*>(base + align256(sizeof(CgState)));
    float* p = reinterpret_cast<float*>(base + align256(sizeof(CgState)) + vec);
    float* Ap = reinterpret_cast<float*>(base + align256(sizeof(CgState)) + 2 * vec);
    const unsigned g = blocks_for(V);
    k_cg_init<<<g, kSolveThreads, 0, s>>>(row_ptr, col, V, lambda, b, x, r, p, st);
    k_cg_start<<<1, 1, 0, s>>>(st, rel_tol);
    for (int it = 0; it < max_iters; ++it) {
        k_cg_matvec<<<g, kSolveThreads, 0, s>>>(row_ptr, col, V, lambda, p, Ap, st);
        k_cg_update<<<g, kSolveThreads, 0, s>>>(V, p, Ap, x, r, st);
        k_cg_direction<<<g, kSolveThreads, 0, s>>>(V, r, p, st);
        k_cg_next<<<1, 1, 0, s>>>(st);
    }
    return cudaGetLastError() == cudaSuccess ? MER_OK : MER_ECUDA;
}
}  // namespace

extern "C" int mer_laplacian_csr(const int32_t* tris, int64_t T, int64_t V, int64_t* row_ptr, int32_t* col) {
    if (T < 0 || V < 0 || !row_ptr || (T > 0 && !tris) || V >= (int64_t(1) << 31)) return MER_EINVAL;
    for (int64_t t = 0; t < 3 * T; ++t)
        if (tris[t] < 0 || tris[t] >= V) return MER_ERANGE;
    // directed edge list (both directions of every triangle edge), sorted and deduplicated per row
    std::vector<int64_t> deg(V + 1, 0);
    for (int64_t t = 0; t < T; ++t)
        for (int k = 0; k < 3; ++k) {
            const int a = tris[3 * t + k], b = tris[3 * t + (k + 1) % 3];
            if (a == b) continue;
            deg[a] += 1;
            deg[b] += 1;
        }
    std::vector<int64_t> start(V + 1, 0);
    for (int64_t v = 0; v < V; ++v) start[v + 1] = start[v] + deg[v];
    std::vector<int32_t> nb(start[V]);
    std::vector<int64_t> fill(start.begin(), start.end() - 1);
    for (int64_t t = 0; t < T; ++t)
        for (int k = 0; k < 3; ++k) {
            const int a = tris[3 * t + k], b = tris[3 * t + (k + 1) % 3];
            if (a == b) continue;
            nb[fill[a]++] = b;
            nb[fill[b]++] = a;
        }
    row_ptr[0] = 0;
    for (int64_t v = 0; v < V; ++v) {
        auto first = nb.begin() + start[v], last = nb.begin() + start[v + 1];
        std::sort(first, last);
        const int64_t n = std::unique(first, last) - first;
        if (col) std::copy(first, first + n, col + row_ptr[v]);
        row_ptr[v + 1] = row_ptr[v] + n;
    }
    return MER_OK;
}

extern "C" int mer_precond_apply(const int64_t* row_ptr, const int32_t* col, int64_t V, float lambda,
                                 const float* x, float* y, void* stream) {
    if (V < 0 || !(lambda >= 0.f)) return MER_EINVAL;
    if (V == 0) return MER_OK;
    if (!row_ptr || !col || !x || !y || x == y) return MER_EINVAL;
    k_apply<<<blocks_for(V), kSolveThreads, 0, static_cast<cudaStream_t>(stream)>>>(row_ptr, col, V, lambda, x, y);
    return cudaGetLastError() == cudaSuccess ? MER_OK : MER_ECUDA;
}

extern "C" size_t mer_precond_solve_workspace_size(int64_t V) {
    if (V < 0) return 0;
    return align256(sizeof(CgState)) + kCgSlotBytes + 3 * align256((size_t)V * sizeof(float4));
}

// The solve with its choices open: max_polls of an exchange, and `launches` for the fixed sequence whatever the size.
extern "C" int mer_launch_precond_solve(const int64_t* row_ptr, const int32_t* col, int64_t V, float lambda, const float* b,
                                        float* x, int max_iters, float rel_tol, void* workspace, unsigned max_polls,
                                        int launches, cudaStream_t s) {
    char* base = static_cast<char*>(workspace);
    CgState* st = reinterpret_cast<CgState*>(base);
    if (cudaMemsetAsync(st, 0, align256(sizeof(CgState)) + kCgSlotBytes, s) != cudaSuccess) return MER_ECUDA;
    if (launches) return solve_launches(row_ptr, col, V, lambda, b, x, max_iters, rel_tol, base, s);
    CgSlot* slots = reinterpret_cast<CgSlot*>(base + align256(sizeof(CgState)));
    float4* r4 = reinterpret_cast<float4*>(base + align256(sizeof(CgState)) + kCgSlotBytes);
    float4* p4 = r4 + V;
    // One CTA up to its 1,024 threads (902 rows: 3.9 us an iteration, the same as a cluster; 258 rows: 2.8 against 4.0).
    // One cluster, with two rows a thread where that saves the exchange between clusters (6,402 rows: 5.4 against 6.4 us).
    // Then the fewest rows a thread whose clusters all fit on the device (16 clusters of 8 with one CTA per SM): 32,402
    // rows 6.9 us with one row, 7.9 with two; 65,538 rows 7.8 us with two; 131,046 rows 12.5 us with four, although that
    // form spills, 211,602 rows 13.3 (the launches 52 and 57).  Larger systems, which one grid cannot hold,
    // and devices without room take the launches, 36-60 us an iteration up to 262,146 rows, 91 at 620,946.
    constexpr int64_t kClusterRows = kCgCluster * kCgThreads;
    cudaError_t e = cudaErrorNotSupported;
    if (V <= kCgLocalThreads)
        e = launch_cg<1, false>(row_ptr, col, (int)V, lambda, b, x, r4, p4, slots, st, max_iters, rel_tol, max_polls, s);
    else if (V <= kCgMaxClusters * kClusterRows && (V <= kClusterRows || V > 2 * kClusterRows))
        e = launch_cg<1, true>(row_ptr, col, (int)V, lambda, b, x, r4, p4, slots, st, max_iters, rel_tol, max_polls, s);
    if (e == cudaErrorNotSupported && V <= 2 * kCgMaxClusters * kClusterRows)
        e = launch_cg<2, true>(row_ptr, col, (int)V, lambda, b, x, r4, p4, slots, st, max_iters, rel_tol, max_polls, s);
    if (e == cudaErrorNotSupported && V <= 4 * kCgMaxClusters * kClusterRows)
        e = launch_cg<4, true>(row_ptr, col, (int)V, lambda, b, x, r4, p4, slots, st, max_iters, rel_tol, max_polls, s);
    if (e == cudaErrorNotSupported)
        return solve_launches(row_ptr, col, V, lambda, b, x, max_iters, rel_tol, base, s);
    return e == cudaSuccess ? MER_OK : MER_ECUDA;
}

extern "C" int mer_precond_solve(const int64_t* row_ptr, const int32_t* col, int64_t V, float lambda,
                                 const float* b, float* x, int max_iters, float rel_tol, void* workspace,
                                 size_t workspace_bytes, void* stream) {
    if (V < 0 || !(lambda >= 0.f) || max_iters < 0 || !(rel_tol >= 0.f)) return MER_EINVAL;
    if (V == 0) return MER_OK;
    if (!row_ptr || !col || !b || !x || b == x || !workspace) return MER_EINVAL;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MER_EINVAL;
    if (workspace_bytes < mer_precond_solve_workspace_size(V)) return MER_EINVAL;
    return mer_launch_precond_solve(row_ptr, col, V, lambda, b, x, max_iters, rel_tol, workspace, kCgPolls, 0,
                                    static_cast<cudaStream_t>(stream));
}

extern "C" int mer_precond_solve_info(const void* workspace, int* iters, double* rel_residual, void* stream) {
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return MER_EINVAL;
    CgState st;
    if (cudaMemcpyAsync(&st, workspace, sizeof(CgState), cudaMemcpyDeviceToHost, static_cast<cudaStream_t>(stream)) !=
        cudaSuccess)
        return MER_ECUDA;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return MER_ECUDA;
    if (st.failed) return MER_ECUDA;
    if (iters) *iters = st.iters;
    if (rel_residual) *rel_residual = st.rr0 > 0.0 ? std::sqrt(st.rr / st.rr0) : 0.0;
    return MER_OK;
}
