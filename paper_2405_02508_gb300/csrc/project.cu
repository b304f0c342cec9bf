// project.cu -- vertex transform module (Supp. B) and its backward.
//
// Forward in FP64 with a fixed operation order and correctly rounded intrinsics
// (no contraction into FMA), so the snapped screen positions X = rint(256 x_s)
// are reproducible bit for bit by any IEEE FP64 implementation of the same
// formula.  Backward: the per-view kernel in FP64 (sums over the views in a fixed order); the batched one
// in FP32 with atomics, or, given a workspace, in FP64 with fixed-point sums (bitwise reproducible).
#include <cuda_runtime.h>

#include "launch.cuh"
#include "mer_device.cuh"

namespace mer {

// These kernels are bound by the FP64 pipe (one warp instruction in 16 cycles on an SM), on which conversions count like
// any operation: 2,097,216 vertices of 32 views took 60 of them each, 204 us for 67 MB.  Exact conversions run on the integer
// pipes instead (f2d, i2d), the snap is one FMA, and the batched backward converts a camera once a warp: 173 us, its
// backward 76 -> 42 (each by itself, cold caches).

__device__ __forceinline__ void write_vertex(double xs, double ys, double zeta, bool front, mer_vertex* out,
                                             mer_vertex* out2 = nullptr) {
    mer_vertex r;
    r.X = 0; r.Y = 0; r.rx = 0.f; r.ry = 0.f; r.zeta = 0.f; r.zeta_lo = 0.f; r.flags = 0u; r.pad = 0.f;
    if (front) {
        r.flags = 1u;
        // inside the guard band: |256 xs|, |256 ys| <= 2^29, compared as integers (false for NaN)
        const long long lim = __double_as_longlong(kGuard / 256.0), keep = 0x7fffffffffffffffLL;
        if ((__double_as_longlong(xs) & keep) <= lim && (__double_as_longlong(ys) & keep) <= lim) {
            r.flags |= 2u;
            // rint(256 xs), ties to even: the sum with 1.5 * 2^52 is rounded to a whole number, whose low word is the
            // integer; xs - X/256 in one FMA (the product is exact)
            const double M = 6755399441055744.0;
            const double tx = __fma_rn(xs, 256.0, M), ty = __fma_rn(ys, 256.0, M);
            r.X = __double2loint(tx);
            r.Y = __double2loint(ty);
            r.rx = __double2float_rn(__fma_rn(__dsub_rn(tx, M), -1.0 / 256.0, xs));
            r.ry = __double2float_rn(__fma_rn(__dsub_rn(ty, M), -1.0 / 256.0, ys));
        }
        r.zeta = __double2float_rn(zeta);
        r.zeta_lo = __double2float_rn(__dsub_rn(zeta, f2d(r.zeta)));
    }
    *out = r;
    if (out2) *out2 = r;
}

__device__ __forceinline__ void project_one(const float* __restrict__ w, const mer_camera& c, mer_vertex* out,
                                            mer_vertex* out2 = nullptr) {
    const double x = f2d(w[0]), y = f2d(w[1]), z = f2d(w[2]);
    const double* R = c.R;
    const double Xc = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(R[0], x), __dmul_rn(R[1], y)), __dmul_rn(R[2], z)), c.t[0]);
    const double Yc = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(R[3], x), __dmul_rn(R[4], y)), __dmul_rn(R[5], z)), c.t[1]);
    const double Zc = __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(R[6], x), __dmul_rn(R[7], y)), __dmul_rn(R[8], z)), c.t[2]);
    const bool front = Zc > c.znear;
    double zeta = 0.0, xs = 0.0, ys = 0.0;
    if (front) {
        zeta = __drcp_rn(Zc);
        xs = __dadd_rn(__dmul_rn(__dmul_rn(c.fx, Xc), zeta), c.cx);
        ys = __dadd_rn(__dmul_rn(__dmul_rn(c.fy, Yc), zeta), c.cy);
    }
    write_vertex(xs, ys, zeta, front, out, out2);
}

// out2 (optional): a second copy.  clear (optional): n_clear words set to zero (the raster's tile counts, which the next
// kernel adds to: one launch less).
__global__ void k_project(const float* verts, int V, const mer_camera* cams, int n,
                          mer_vertex* out, mer_vertex* out2, int* clear,
                          long long n_clear) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long k = i; k < n_clear; k += (long long)gridDim.x * blockDim.x) clear[k] = 0;
    if (i >= (long long)V * n) return;
    const int view = (int)(i / V), v = (int)(i % V);
    project_one(verts + 3 * (size_t)v, cams[view], out + i, out2 ? out2 + i : nullptr);
}

__global__ void k_project_batch(const float* verts, const mer_camera* cams,
                                const mer_item* items, int n_items, long long vrecs,
                                mer_vertex* out) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = warp_find_item(items, n_items, i - (threadIdx.x & 31), i, kFieldVrec);
    if (i >= vrecs) return;
    const mer_item m = items[k];
    project_one(verts + 3 * (size_t)(m.vert + (i - m.vrec)), cams[m.cam], out + i);
}

__global__ void k_project_screen(const double* scr, int V, int n, mer_vertex* out) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)V * n) return;
    const double xs = scr[3 * i], ys = scr[3 * i + 1], zeta = scr[3 * i + 2];
    write_vertex(xs, ys, zeta, zeta > 0.0, out + i);
}

// R^T J^T g for one projected vertex, J = d(x_s, y_s, zeta)/d(X_c, Y_c, Z_c)
// = [[fx z, 0, -(x_s-cx) z], [0, fy z, -(y_s-cy) z], [0, 0, -z^2]]; false if the vertex is behind the camera.
// The camera in FP32 but for its centre.
struct CameraF {
    double cx, cy;
    float R[9], fx, fy;
};

__device__ __forceinline__ CameraF camera_f(const mer_camera& c) {
    CameraF f;
    f.cx = c.cx;
    f.cy = c.cy;
#pragma unroll
    for (int i = 0; i < 9; ++i) f.R[i] = (float)c.R[i];
    f.fx = (float)c.fx;
    f.fy = (float)c.fy;
    return f;
}

__device__ __forceinline__ bool world_grad(const mer_vertex& r, const CameraF& c, const double* g3, float out[3]) {
    if ((r.flags & 1u) == 0u) return false;
    const float gx = (float)g3[0], gy = (float)g3[1], gz = (float)g3[2];
    const float z = r.zeta;
    const float xs = (float)__fma_rn(i2d(r.X), 1.0 / 256.0, -c.cx) + r.rx;  // the product is exact
    const float ys = (float)__fma_rn(i2d(r.Y), 1.0 / 256.0, -c.cy) + r.ry;
    const float gX = gx * c.fx * z;
    const float gY = gy * c.fy * z;
    const float gZ = -z * (gx * xs + gy * ys + gz * z);
    out[0] = c.R[0] * gX + c.R[3] * gY + c.R[6] * gZ;
    out[1] = c.R[1] * gX + c.R[4] * gY + c.R[7] * gZ;
    out[2] = c.R[2] * gX + c.R[5] * gY + c.R[8] * gZ;
    return true;
}

// world_grad in FP64 (vertex position from the exact snapped part plus the residual, zeta from its hi + lo
// split).
__device__ __forceinline__ bool world_grad_f64(const mer_vertex& r, const mer_camera& c, const double* g3,
                                               double out[3]) {
    if ((r.flags & 1u) == 0u) return false;
    const double gx = g3[0], gy = g3[1], gz = g3[2];
    const double z = f2d(r.zeta) + f2d(r.zeta_lo);
    const double xs = __fma_rn(i2d(r.X), 1.0 / 256.0, -c.cx) + f2d(r.rx);  // the product is exact
    const double ys = __fma_rn(i2d(r.Y), 1.0 / 256.0, -c.cy) + f2d(r.ry);
    const double gX = gx * c.fx * z;
    const double gY = gy * c.fy * z;
    const double gZ = -z * (gx * xs + gy * ys + gz * z);
    out[0] = c.R[0] * gX + c.R[3] * gY + c.R[6] * gZ;
    out[1] = c.R[1] * gX + c.R[4] * gY + c.R[7] * gZ;
    out[2] = c.R[2] * gX + c.R[5] * gY + c.R[8] * gZ;
    return true;
}

// Batched: one thread per (item, vertex); items sharing a mesh add into the same rows.
__global__ void k_project_backward_batch(const mer_camera* cams, const mer_item* items,
                                         int n_items, long long vrecs, const mer_vertex* vpix,
                                         const double* grad_vpix, float* grad_verts) {
    after_previous();
    __shared__ CameraF s_cam[8];  // of each warp's first item, converted by its lanes together
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    if (i - lane >= vrecs) return;  // a warp past the end: the item found for it may be an empty one, whose camera nothing checks
    const int k = warp_find_item(items, n_items, i - lane, i, kFieldVrec);
    const int first = __shfl_sync(0xffffffffu, k, 0);
    CameraF& cam = s_cam[threadIdx.x >> 5];
    const mer_camera& c = cams[items[first].cam];
    if (lane < 9) cam.R[lane] = (float)c.R[lane];
    if (lane == 9) cam.fx = (float)c.fx;
    if (lane == 10) cam.fy = (float)c.fy;
    if (lane == 11) cam.cx = c.cx;
    if (lane == 12) cam.cy = c.cy;
    __syncwarp();
    if (i >= vrecs) return;
    const mer_item m = items[k];
    float w[3];
    if (!(k == first ? world_grad(vpix[i], cam, grad_vpix + 3 * i, w)
                     : world_grad(vpix[i], camera_f(cams[m.cam]), grad_vpix + 3 * i, w)))
        return;
    float* o = grad_verts + 3 * (size_t)(m.vert + (i - m.vrec));
    atomicAdd(o, w[0]);
    atomicAdd(o + 1, w[1]);
    atomicAdd(o + 2, w[2]);
}

// Batched, reproducible: FP64 products rounded once to fixed point with 52 fractional bits, held as two
// 64-bit words (hi = floor(w 2^20), lo = the remainder in units of 2^-52, in [0, 2^32]), and added with
// integer atomics into acc [mesh rows, 3, 2] (exact, so the order does not matter); k_world_finalize converts.
__global__ void k_project_backward_batch_fixed(const mer_camera* cams, const mer_item* items,
                                               int n_items, long long vrecs, const mer_vertex* vpix,
                                               const double* grad_vpix, unsigned long long* acc,
                                               void* ws) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = warp_find_item(items, n_items, i - (threadIdx.x & 31), i, kFieldVrec);
    if (i >= vrecs) return;
    const mer_item m = items[k];
    double w[3];
    if (!world_grad_f64(vpix[i], cams[m.cam], grad_vpix + 3 * i, w)) return;
    unsigned long long* o = acc + 6 * (size_t)(m.vert + (i - m.vrec));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (!(fabs(w[c]) < 8589934592.0)) {  // 2^33
            set_status(ws, kStatusFixed);
            continue;
        }
        const double h = floor(w[c] * 1048576.0);
        const long long hi = (long long)h;
        const long long lo = __double2ll_rn((w[c] - h * (1.0 / 1048576.0)) * 4503599627370496.0);
        if (hi != 0) atomicAdd(o + 2 * c, (unsigned long long)hi);
        if (lo != 0) atomicAdd(o + 2 * c + 1, (unsigned long long)lo);
    }
}

__global__ void k_world_finalize(const unsigned long long* acc, long long n, float* grad_verts) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const long long lo = (long long)acc[2 * i + 1];
    const long long hi = (long long)acc[2 * i] + (lo >> 32);
    grad_verts[i] += __double2float_rn((double)hi * (1.0 / 1048576.0) + (double)(lo & 0xffffffffll) * (1.0 / 4503599627370496.0));
}

// One thread per vertex, looping over the views: grad_world = sum_views R^T J^T g (FP64).  STORE: overwrite grad_verts (and
// the second copy) instead of adding to it.
template <bool STORE>
__global__ void k_project_backward(int V, const mer_camera* cams, int n,
                                   const mer_vertex* vpix, const double* grad_vpix,
                                   float* grad_verts, float* copy) {
    after_previous();
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int view = 0; view < n; ++view) {
        const size_t k = (size_t)view * V + v;
        double w[3];
        if (!world_grad_f64(vpix[k], cams[view], grad_vpix + 3 * k, w)) continue;
        a0 += w[0];
        a1 += w[1];
        a2 += w[2];
    }
    float* o = grad_verts + 3 * (size_t)v;
    const float g[3] = {(float)a0, (float)a1, (float)a2};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float r = STORE ? g[c] : o[c] + g[c];
        o[c] = r;
        if (copy) copy[3 * (size_t)v + c] = r;
    }
}

}  // namespace mer

using namespace mer;

extern "C" int mer_launch_project(const float* verts, int V, const mer_camera* cams, int n, mer_vertex* vpix,
                                  mer_vertex* copy, int* clear, long long n_clear, cudaStream_t s) {
    const long long N = (long long)V * n;
    if (N == 0) return 0;
    launch_chained(k_project, (unsigned)((N + 255) / 256), 256, s, verts, V, cams, n, vpix, copy, clear, n_clear);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

extern "C" int mer_launch_project_screen(const double* scr, int V, int n, mer_vertex* vpix, cudaStream_t s) {
    const long long N = (long long)V * n;
    if (N == 0) return 0;
    launch_chained(k_project_screen, (unsigned)((N + 255) / 256), 256, s, scr, V, n, vpix);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

extern "C" int mer_launch_project_backward(int V, const mer_camera* cams, int n, const mer_vertex* vpix,
                                           const double* grad_vpix, float* grad_verts, float* copy, int store,
                                           cudaStream_t s) {
    // without views the kernel's sum over them is empty: an overwritten gradient is zero, a copy is what grad_verts holds
    if (V == 0 || (n == 0 && !(grad_verts && (store || copy)))) return 0;
    if (store)
        launch_chained(k_project_backward<true>, (V + 255) / 256, 256, s, V, cams, n, vpix, grad_vpix, grad_verts, copy);
    else
        launch_chained(k_project_backward<false>, (V + 255) / 256, 256, s, V, cams, n, vpix, grad_vpix, grad_verts, copy);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

extern "C" int mer_launch_project_batch(const float* verts, const mer_camera* cams, const mer_item* items, int n_items,
                                        long long vrecs, mer_vertex* vpix, cudaStream_t s) {
    if (vrecs == 0) return 0;
    launch_chained(k_project_batch, (unsigned)((vrecs + 255) / 256), 256, s, verts, cams, items, n_items, vrecs, vpix);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

// ws: null for the FP32 atomic path; else a workspace whose bytes after the 256-byte header hold
// mesh_rows * 3 two-word fixed-point sums (the reproducible FP64 path).
extern "C" int mer_launch_project_backward_batch(const mer_camera* cams, const mer_item* items, int n_items,
                                                 long long vrecs, long long mesh_rows, const mer_vertex* vpix,
                                                 const double* grad_vpix, float* grad_verts, void* ws,
                                                 cudaStream_t s) {
    if (vrecs == 0) return 0;
    if (ws) {
        unsigned long long* acc = reinterpret_cast<unsigned long long*>(static_cast<char*>(ws) + 256);
        if (cudaMemsetAsync(acc, 0, (size_t)mesh_rows * 48, s) != cudaSuccess) return 2;
        launch_chained(k_project_backward_batch_fixed, (unsigned)((vrecs + 255) / 256), 256, s, cams, items, n_items, vrecs,
                                                                                       vpix, grad_vpix, acc, ws);
        const long long n = 3 * mesh_rows;
        if (n > 0) launch_chained(k_world_finalize, (unsigned)((n + 255) / 256), 256, s, acc, n, grad_verts);
        return cudaGetLastError() == cudaSuccess ? 0 : 2;
    }
    launch_chained(k_project_backward_batch, (unsigned)((vrecs + 255) / 256), 256, s, cams, items, n_items, vrecs, vpix,
                                                                             grad_vpix, grad_verts);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}

namespace mer {
__global__ void k_clear(double* a, long long na, float* b, long long nb) {
    after_previous();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < na) a[i] = 0.0;
    if (i < nb) b[i] = 0.f;
}
}  // namespace mer

// Zeroes two gradient arrays in one launch.
extern "C" int mer_launch_clear(double* a, long long na, float* b, long long nb, cudaStream_t s) {
    const long long m = na > nb ? na : nb;
    if (m > 0) launch_chained(k_clear, (unsigned)((m + 255) / 256), 256, s, a, na, b, nb);
    return cudaGetLastError() == cudaSuccess ? 0 : 2;
}
