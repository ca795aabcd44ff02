// pagerank.cu -- PageRank power iteration on the SpMM path (paper Section 4.1).
//
// Update rule (Section 4.1): PR(u) = (1-d)/N + d * sum_{v in B(u)} PR(v)/L(v),
// with B(u) the in-neighbours of u and L(v) the out-degree of v; the rank of
// dangling vertices (L = 0) is spread uniformly, so the ranks keep summing to 1.
// Row v of A lists the out-links of v, so the in-neighbour sum is the product
// with the transposed matrix: y = A^T z with z[v] = x[v] / L(v).
//
// One iteration = the task kernel on A^T (k = 1, float32) + one fused
// elementwise kernel (new ranks, the next z = x' * (1/L), FP64 per-block
// partial sums of the L1 change and of the dangling mass, added in a fixed order
// by its last block).  Iterations 2..iters are one CUDA
// graph; the handle keeps it with the workspace, so a later call with the
// same x, damping and iteration count only launches it.  Ranks are float32;
// every reduction is FP64 and run-to-run deterministic.
#include <vector>

#include "internal.h"

namespace spmm {

constexpr int kPrThreads = 256;
constexpr int kPrUpdateFewer = 4;    // the update runs a quarter of the other passes' blocks: two an SM

// Fixed-order block sum of a double (xor tree inside warps, then warp sums
// added in warp order by thread 0).  Result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[i];
    __syncthreads();
    return s;
}

// inv[v] = 1/L(v) as float (0 marks a dangling vertex, L = 0); x = x0 or 1/N.
__global__ void pr_init_kernel(const int64_t* __restrict__ row_ptr, int64_t n, float* __restrict__ inv,
                               float* __restrict__ x, const float* __restrict__ x0) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t L = row_ptr[i + 1] - row_ptr[i];
        inv[i] = L > 0 ? 1.0f / (float)L : 0.f;
        x[i] = x0 ? x0[i] : (float)(1.0 / (double)n);
    }
}

// One rank update of element i (float32): x' = base + d*y; returns |x' - x|,
// writes z' = x' / L and adds x' to dang for a dangling vertex.
__device__ __forceinline__ float pr_elem(float y, float& x, float inv, float base, float d, float& z, float& dang) {
    const float xn = fmaf(d, y, base);
    const float r = fabsf(xn - x);
    x = xn;
    z = xn * inv;
    if (inv == 0.f) dang += xn;
    return r;
}

// z = x / L (0 where L = 0); per-block partial of the dangling mass.
__global__ void pr_scale_kernel(const float* __restrict__ x, const float* __restrict__ inv, int64_t n,
                                float* __restrict__ z, double* __restrict__ part_dang) {
    __shared__ double sh[32];
    double dang = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float xi = x[i], iv = inv[i];
        z[i] = xi * iv;
        if (iv == 0.f) dang += (double)xi;
    }
    const double s = block_sum(dang, sh);
    if (threadIdx.x == 0) part_dang[blockIdx.x] = s;
}

// A sum of floats as three floats, each holding what the one before rounded
// away (Knuth's two-sum): 72 bits, so no less exact than an FP64 sum, on the
// FP32 units (an FP64 addition and its conversion take 32 times as long here).
// Terms above 2^100, infinities and NaN, which the floats could not carry, are
// added in FP64 (pr_add).
struct FloatSum {
    float s = 0.f, c = 0.f, d = 0.f;
    double big = 0.0;
    static __device__ __forceinline__ float two_sum(float& a, float b) {
        const float t = __fadd_rn(a, b), bb = __fsub_rn(t, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bb)), __fsub_rn(b, bb));
        a = t;
        return e;
    }
    __device__ __forceinline__ void add(float v) { d = __fadd_rn(d, two_sum(c, two_sum(s, v))); }
    __device__ __forceinline__ double value() const { return big + ((double)s + ((double)c + (double)d)); }
};

// r and dg into the two sums.  One test for both, as a branch: a test in each
// sum took 3 us of an iteration on 4.2 M vertices, this one nothing measurable.
__device__ __forceinline__ void pr_add(FloatSum& res, FloatSum& dang, float r, float dg) {
    if (__builtin_expect(r + fabsf(dg) <= 0x1p100f, 1)) {
        res.add(r);
        dang.add(dg);
    } else {
        res.big += (double)r;
        dang.big += (double)dg;
    }
}

// x' = (1-d)/N + d*D/N + d*y, with D the dangling mass of x (scal[0]);
// partials of sum |x' - x| and of the dangling mass of x'; z' = x' / L; the last
// block to finish adds the partials in block order: scal[0] = the dangling mass
// of x', *res_out = sum |x' - x|.  Float4 accesses, two in flight per thread; the
// per-element arithmetic is float32, groups of four are added to per-thread sums
// of 72 bits, those in FP64.  Bound by memory: with FP64 per-thread sums and 8
// blocks an SM the FP64 units took two thirds of its 31.5 us on 4.2 M vertices,
// and the final sum was a launch of its own (6.4 us); now 21.8 us with the sum (608 blocks 23.6,
// 1216 35.2: each block adds its sums in FP64).
__global__ void __launch_bounds__(kPrThreads)
pr_update_kernel(const float* __restrict__ y, float* __restrict__ x, const float* __restrict__ inv, int64_t n, double d,
                 double* __restrict__ scal, float* __restrict__ z, double* __restrict__ part_res,
                 double* __restrict__ part_dang, double* __restrict__ res_out, unsigned int* __restrict__ done) {
    __shared__ double sh[32];
    __shared__ bool last;
    const float base = (float)((1.0 - d) / (double)n + d * __ldcg(scal) / (double)n);
    const float df = (float)d;
    FloatSum res, dang;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool vec = ((((uintptr_t)x) | ((uintptr_t)y) | ((uintptr_t)z) | ((uintptr_t)inv)) & 15) == 0;
    int64_t done_n = 0;
    if (vec) {
        const int64_t n4 = n >> 2;
        auto four = [&](int64_t i, const float4 y4, float4 x4, const float4 v4) {
            float4 z4;
            float dg = 0.f, r = 0.f;
            r += pr_elem(y4.x, x4.x, v4.x, base, df, z4.x, dg);
            r += pr_elem(y4.y, x4.y, v4.y, base, df, z4.y, dg);
            r += pr_elem(y4.z, x4.z, v4.z, base, df, z4.z, dg);
            r += pr_elem(y4.w, x4.w, v4.w, base, df, z4.w, dg);
            reinterpret_cast<float4*>(x)[i] = x4;
            reinterpret_cast<float4*>(z)[i] = z4;
            pr_add(res, dang, r, dg);
        };
        const float4 *y_4 = reinterpret_cast<const float4*>(y), *v_4 = reinterpret_cast<const float4*>(inv);
        const float4* x_4 = reinterpret_cast<const float4*>(x);
        int64_t i = tid;
        for (; i + stride < n4; i += 2 * stride) {
            const float4 ya = y_4[i], xa = x_4[i], va = v_4[i];
            const float4 yb = y_4[i + stride], xb = x_4[i + stride], vb = v_4[i + stride];
            four(i, ya, xa, va);
            four(i + stride, yb, xb, vb);
        }
        if (i < n4) four(i, y_4[i], x_4[i], v_4[i]);
        done_n = n4 << 2;
    }
    for (int64_t i = done_n + tid; i < n; i += stride) {   // tail (or unaligned buffers)
        float xi = x[i], zi, dg = 0.f;
        const float r = pr_elem(y[i], xi, inv[i], base, df, zi, dg);
        x[i] = xi;
        z[i] = zi;
        pr_add(res, dang, r, dg);
    }
    const double s1 = block_sum(res.value(), sh);
    const double s2 = block_sum(dang.value(), sh);
    if (threadIdx.x == 0) {
        part_res[blockIdx.x] = s1;
        part_dang[blockIdx.x] = s2;
        __threadfence();
        last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;   // wraps to zero for the next launch
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
        a += __ldcg(part_dang + i);
        b += __ldcg(part_res + i);
    }
    const double sa = block_sum(a, sh);
    const double sb = block_sum(b, sh);
    if (threadIdx.x == 0) {
        scal[0] = sa;
        *res_out = sb;
    }
}

// scal[0] = sum of the dangling partials of pr_scale_kernel, in block order
__global__ void pr_reduce_kernel(const double* __restrict__ part_dang, int nparts, double* __restrict__ scal) {
    __shared__ double sh[32];
    double a = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) a += part_dang[i];
    const double sa = block_sum(a, sh);
    if (threadIdx.x == 0) scal[0] = sa;
}

}  // namespace spmm

using namespace spmm;

namespace spmm {

void pagerank_release(spmm_mat* A) {
    PrCache& c = A->pr;
    if (c.exec) cudaGraphExecDestroy(c.exec);
    if (c.s) cudaStreamDestroy(c.s);
    cudaFree(c.inv_deg);
    cudaFree(c.z);
    cudaFree(c.y);
    cudaFree(c.part);
    cudaFree(c.scal);
    cudaFree(c.done);
    cudaFree(c.dres);
    cudaFree(c.xr);
    cudaFree(c.x0r);
    c = PrCache{};
}

void pagerank_invalidate(spmm_mat* A) {
    PrCache& c = A->pr;
    if (c.exec) cudaGraphExecDestroy(c.exec);
    c.exec = nullptr;
    c.x = nullptr;
    c.damping = -1.0;
    c.iters = -1;
}

// The workspace of an n-vertex PageRank with room for `iters` residuals.
static cudaError_t pr_reserve(PrCache& c, int64_t n, int32_t iters, int nblk) {
    cudaError_t e = cudaSuccess;
    if (!c.inv_deg) {
        if ((e = cudaMalloc((void**)&c.inv_deg, n * sizeof(float))) != cudaSuccess ||
            (e = cudaMalloc((void**)&c.z, n * sizeof(float))) != cudaSuccess ||
            (e = cudaMalloc((void**)&c.y, n * sizeof(float))) != cudaSuccess ||
            (e = cudaMalloc((void**)&c.part, 2 * (size_t)nblk * sizeof(double))) != cudaSuccess ||
            (e = cudaMalloc((void**)&c.scal, 8 * sizeof(double))) != cudaSuccess ||
            (e = cudaMalloc((void**)&c.done, sizeof(unsigned int))) != cudaSuccess ||
            (e = cudaStreamCreateWithFlags(&c.s, cudaStreamNonBlocking)) != cudaSuccess ||
            (e = cudaMemsetAsync(c.done, 0, sizeof(unsigned int), c.s)) != cudaSuccess)
            return e;
        c.nblk = nblk;
    }
    if (iters > c.dres_cap) {
        cudaFree(c.dres);
        c.dres = nullptr;
        c.dres_cap = 0;
        if ((e = cudaMalloc((void**)&c.dres, (size_t)iters * sizeof(double))) != cudaSuccess) return e;
        c.dres_cap = iters;
        if (c.exec) {                          // its residual pointers are gone
            cudaGraphExecDestroy(c.exec);
            c.exec = nullptr;
            c.iters = -1;
        }
    }
    return e;
}

}  // namespace spmm

extern "C" int spmm_pagerank(spmm_mat_t A, double damping, int32_t iters, float* x, const float* x0,
                             double* residuals, void* stream) {
    if (!A || !x) { set_error("spmm_pagerank: NULL argument"); return SPMM_ERR_ARG; }
    if (A->fwd.n_rows != A->fwd.n_cols || A->fwd.n_rows < 1) {
        set_error("spmm_pagerank: the matrix must be square and non-empty");
        return SPMM_ERR_ARG;
    }
    if (!A->has_tr) { set_error("spmm_pagerank: needs SPMM_WANT_TRANSPOSE at create"); return SPMM_ERR_ARG; }
    if (A->vtype != -1) {
        set_error("spmm_pagerank: PageRank walks the graph pattern; create the handle without values");
        return SPMM_ERR_ARG;
    }
    if (iters < 0 || !(damping >= 0.0 && damping <= 1.0)) {
        set_error("spmm_pagerank: need iters >= 0 and 0 <= damping <= 1");
        return SPMM_ERR_ARG;
    }
    const int64_t n = A->fwd.n_rows;
    cudaStream_t user = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e, "spmm_pagerank: device query");
    PrCache& c = A->pr;
    int rc = SPMM_OK;
    NvtxRange range("spmm_pagerank");
    auto fail = [&](cudaError_t err, const char* what) { rc = cuda_fail(err, what); };
    do {
        if ((e = cudaStreamSynchronize(user)) != cudaSuccess) { fail(e, "spmm_pagerank: stream"); break; }
        if ((e = pr_reserve(c, n, iters, sms * 8)) != cudaSuccess) {
            fail(e, "spmm_pagerank: workspace");
            pagerank_release(A);
            break;
        }
        const int nblk = c.nblk;
        cudaStream_t s = c.s;
        // SPMM_RELABEL: the iterations run on the ranks in the handle's vertex
        // order, in a buffer the handle keeps (so the captured graph stays
        // valid); the start vector comes in and the ranks go out once
        float* const x_user = x;
        if (A->relabel) {
            if (!c.xr && (e = cudaMalloc((void**)&c.xr, (size_t)n * sizeof(float))) != cudaSuccess) {
                fail(e, "spmm_pagerank: relabelled ranks");
                break;
            }
            if (x0) {
                if (!c.x0r && (e = cudaMalloc((void**)&c.x0r, (size_t)n * sizeof(float))) != cudaSuccess) {
                    fail(e, "spmm_pagerank: relabelled start vector");
                    break;
                }
                if ((e = relabel_rows_dev(A, x0, 1, 1, 4, c.x0r, 1, true, s)) != cudaSuccess) {
                    fail(e, "spmm_pagerank: start vector into the handle's order");
                    break;
                }
                x0 = c.x0r;
            }
            x = c.xr;
        }
        // set-up outside the graph: 1/L, the start vector, z and its dangling mass
        pr_init_kernel<<<nblk, kPrThreads, 0, s>>>(A->fwd.row_ptr, n, c.inv_deg, x, x0);
        pr_scale_kernel<<<nblk, kPrThreads, 0, s>>>(x, c.inv_deg, n, c.z, c.part);
        pr_reduce_kernel<<<1, kPrThreads, 0, s>>>(c.part, nblk, c.scal);
        if ((e = cudaGetLastError()) != cudaSuccess) { fail(e, "spmm_pagerank: init"); break; }
        auto update = [&](int32_t t) {
            pr_update_kernel<<<nblk / kPrUpdateFewer, kPrThreads, 0, s>>>(c.y, x, c.inv_deg, n, damping, c.scal, c.z,
                                                                          c.part + nblk, c.part, c.dres + t, c.done);
        };
        if (iters > 0) {
            // the first iteration runs outside the graph, so the task kernel's
            // one-time launch set-up (attributes, occupancy) happens before capture
            if ((rc = apply_dev(A, 1, c.z, 1, 1, SPMM_F32, c.y, 1, s)) != SPMM_OK) break;
            update(0);
            if ((e = cudaGetLastError()) != cudaSuccess) { fail(e, "spmm_pagerank: first iteration"); break; }
        }
        if (iters > 1) {
            // iterations 2..iters: one graph, captured on the first call with
            // this x, damping and iteration count and relaunched after that
            if (!(c.exec && c.x == x && c.damping == damping && c.iters == iters)) {
                if (c.exec) {
                    cudaGraphExecDestroy(c.exec);
                    c.exec = nullptr;
                }
                c.iters = -1;
                if ((e = cudaStreamSynchronize(s)) != cudaSuccess) { fail(e, "spmm_pagerank: first iteration"); break; }
                if ((e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) {
                    fail(e, "spmm_pagerank: capture");
                    break;
                }
                for (int32_t t = 1; t < iters && rc == SPMM_OK; ++t) {
                    rc = apply_dev(A, 1, c.z, 1, 1, SPMM_F32, c.y, 1, s);
                    if (rc != SPMM_OK) break;
                    update(t);
                }
                cudaGraph_t graph = nullptr;
                cudaError_t ec = cudaStreamEndCapture(s, &graph);
                if (rc == SPMM_OK && ec != cudaSuccess) fail(ec, "spmm_pagerank: end capture");
                if (rc == SPMM_OK && (e = cudaGraphInstantiate(&c.exec, graph, 0)) != cudaSuccess) {
                    c.exec = nullptr;
                    fail(e, "spmm_pagerank: instantiate");
                }
                if (graph) cudaGraphDestroy(graph);
                if (rc != SPMM_OK) break;
                c.x = x;
                c.damping = damping;
                c.iters = iters;
            }
            if ((e = cudaGraphLaunch(c.exec, s)) != cudaSuccess) { fail(e, "spmm_pagerank: launch"); break; }
        }
        if (A->relabel && (e = relabel_rows_dev(A, x, 1, 1, 4, x_user, 1, false, s)) != cudaSuccess) {
            fail(e, "spmm_pagerank: ranks into the input order");
            break;
        }
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) { fail(e, "spmm_pagerank: run"); break; }
        int32_t st = 0;
        if ((e = cudaMemcpy(&st, A->status, sizeof(st), cudaMemcpyDeviceToHost)) != cudaSuccess) {
            fail(e, "spmm_pagerank: status");
            break;
        }
        if (st != 0) {
            cudaMemset(A->status, 0, sizeof(int32_t));
            set_error("spmm_pagerank: a device-side staging wait timed out; the ranks are incomplete");
            rc = SPMM_ERR_TIMEOUT;
            break;
        }
        if (residuals && iters > 0 &&
            (e = cudaMemcpy(residuals, c.dres, (size_t)iters * sizeof(double), cudaMemcpyDeviceToHost)) !=
                cudaSuccess) {
            fail(e, "spmm_pagerank: residuals");
            break;
        }
    } while (0);
    return rc;
}
