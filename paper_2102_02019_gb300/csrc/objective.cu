// Pointwise maps and the objectives used with the adjoint: conserved variables
// (rho, rho u, rho v) <-> evolved variables (ln rho, u, v) (Section 7 evolves
// the latter), the domain kinetic energy sum_i 1/2 rho_i |u_i|^2 V_i with node
// volume V_i = s_i^2, and the probe-weighted momentum sum_i rho_i (px_i u_i +
// py_i v_i), with their vector-Jacobian products.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "labfm_internal.cuh"

namespace labfm {
namespace {

template <typename T>
__global__ void k_to_primitive(int64_t N, const T* __restrict__ c, T* __restrict__ q) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const T rho = c[i];
        q[i] = log(rho);
        q[N + i] = c[N + i] / rho;
        q[2 * N + i] = c[2 * N + i] / rho;
    }
}

// cbar = (d primitive / d conserved)^T qbar
template <typename T>
__global__ void k_conserved_vjp(int64_t N, const T* __restrict__ c, const T* __restrict__ qb,
                                T* __restrict__ cb) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const T rho = c[i], mx = c[N + i], my = c[2 * N + i];
        const T ab = qb[i], ub = qb[N + i], vb = qb[2 * N + i];
        const T ir = T(1) / rho;
        cb[i] = ab * ir - (ub * mx + vb * my) * ir * ir;
        cb[N + i] = ub * ir;
        cb[2 * N + i] = vb * ir;
    }
}

// Sums over the nodes in a fixed order (the same result on every call) without scratch
// memory: one cluster of kSumBlocks blocks, each thread summing every kSumBlocks * 1024th
// node, the blocks' sums added by the first one through distributed shared memory.  The
// sum is bound by the FP64 pipe (exp of every node, 2 lanes a clock and an SM), so it runs
// on 16 SMs, the most that can share their memory: 65,536 nodes 432 -> about 17 us.
constexpr int kSumThreads = 1024;
constexpr int kSumBlocks = 16;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

template <class Term>
__device__ void cluster_sum(int64_t N, const Term& term, double* __restrict__ out) {
    namespace cg = cooperative_groups;
    __shared__ double red[kSumThreads / 32];
    __shared__ double block_sum;
    cg::cluster_group cluster = cg::this_cluster();
    double acc = 0.0;
    for (int64_t i = int64_t(blockIdx.x) * kSumThreads + threadIdx.x; i < N; i += int64_t(gridDim.x) * kSumThreads)
        acc += term(i);
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = warp_sum(red[threadIdx.x]);
        if (threadIdx.x == 0) block_sum = acc;
    }
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double v = 0.0;
        if (threadIdx.x < gridDim.x) v = *cluster.map_shared_rank(&block_sum, threadIdx.x);
        v = warp_sum(v);
        if (threadIdx.x == 0) *out = v;
    }
    cluster.sync();  // the other blocks' shared memory stays until it has been read
}

template <typename T>
__global__ void __launch_bounds__(kSumThreads)
    k_kinetic_energy(int64_t N, const T* __restrict__ q, const double* __restrict__ s, double* __restrict__ out) {
    cluster_sum(
        N,
        [&](int64_t i) {
            const double rho = exp(double(q[i])), u = double(q[N + i]), v = double(q[2 * N + i]);
            return 0.5 * rho * (u * u + v * v) * s[i] * s[i];
        },
        out);
}

template <typename T>
__global__ void k_kinetic_energy_grad(int64_t N, const T* __restrict__ q, const double* __restrict__ s,
                                      double scale, T* __restrict__ g) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const double rho = exp(double(q[i])), u = double(q[N + i]), v = double(q[2 * N + i]);
        const double V = s[i] * s[i] * scale;
        g[i] = T(0.5 * rho * (u * u + v * v) * V);
        g[N + i] = T(rho * u * V);
        g[2 * N + i] = T(rho * v * V);
    }
}

template <typename T>
__global__ void __launch_bounds__(kSumThreads)
    k_probe_momentum(int64_t N, const T* __restrict__ q, const double* __restrict__ px,
                     const double* __restrict__ py, double* __restrict__ out) {
    cluster_sum(
        N,
        [&](int64_t i) {
            const double rho = exp(double(q[i]));
            return rho * (px[i] * double(q[N + i]) + py[i] * double(q[2 * N + i]));
        },
        out);
}

template <typename T>
__global__ void k_probe_momentum_grad(int64_t N, const T* __restrict__ q, const double* __restrict__ px,
                                      const double* __restrict__ py, double scale, T* __restrict__ g) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const double rs = exp(double(q[i])) * scale;
        g[i] = T(rs * (px[i] * double(q[N + i]) + py[i] * double(q[2 * N + i])));
        g[N + i] = T(rs * px[i]);
        g[2 * N + i] = T(rs * py[i]);
    }
}

// One cluster launch of a summing kernel: as many blocks as have nodes, at most kSumBlocks.
template <typename... KArgs, typename... Args>
int launch_sum(const char* what, void (*kernel)(KArgs...), int64_t N, cudaStream_t st, Args... args) {
    int blocks = 1;
    while (blocks < kSumBlocks && int64_t(blocks) * kSumThreads < N) blocks *= 2;
    if (blocks > 8)
        LABFM_CUDA_TRY(cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel),
                                            cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(blocks));
    cfg.blockDim = dim3(kSumThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(blocks);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    if (e != cudaSuccess && blocks > 8) {  // no group of 16 SMs that share memory: the portable size
        cudaGetLastError();
        cfg.gridDim.x = attr[0].val.clusterDim.x = 8;
        e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    }
    if (e != cudaSuccess) return cuda_error(e, what);
    return LABFM_OK;
}

int grid_of(int64_t N) { return int(std::min<int64_t>((N + 255) / 256, 65535)); }

int check_n(int64_t N, int dtype) {
    if (N <= 0) return set_error(LABFM_EINVAL, "N must be positive");
    if (dtype != LABFM_F32 && dtype != LABFM_F64) return set_error(LABFM_EINVAL, "unknown dtype");
    return LABFM_OK;
}

}  // namespace
}  // namespace labfm

using namespace labfm;

extern "C" int labfm_conserved_to_primitive(const void* c, void* q, int64_t N, labfm_dtype dtype,
                                            void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!c || !q) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    if (dtype == LABFM_F32)
        k_to_primitive<float><<<grid_of(N), 256, 0, st>>>(N, static_cast<const float*>(c), static_cast<float*>(q));
    else
        k_to_primitive<double><<<grid_of(N), 256, 0, st>>>(N, static_cast<const double*>(c), static_cast<double*>(q));
    LABFM_LAUNCH_CHECK("conversion kernel");
    return LABFM_OK;
}

extern "C" int labfm_conserved_vjp(const void* c, const void* qbar, void* cbar, int64_t N,
                                   labfm_dtype dtype, void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!c || !qbar || !cbar) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    if (dtype == LABFM_F32)
        k_conserved_vjp<float><<<grid_of(N), 256, 0, st>>>(N, static_cast<const float*>(c),
                                                           static_cast<const float*>(qbar), static_cast<float*>(cbar));
    else
        k_conserved_vjp<double><<<grid_of(N), 256, 0, st>>>(N, static_cast<const double*>(c),
                                                            static_cast<const double*>(qbar), static_cast<double*>(cbar));
    LABFM_LAUNCH_CHECK("conversion adjoint kernel");
    return LABFM_OK;
}

extern "C" int labfm_kinetic_energy(const void* q, const double* s, int64_t N, labfm_dtype dtype,
                                    double* ke_out, void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!q || !s || !ke_out) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    const char* what = "kinetic energy kernel";
    return dtype == LABFM_F32 ? launch_sum(what, k_kinetic_energy<float>, N, st, N, static_cast<const float*>(q), s, ke_out)
                              : launch_sum(what, k_kinetic_energy<double>, N, st, N, static_cast<const double*>(q), s, ke_out);
}

extern "C" int labfm_kinetic_energy_grad(const void* q, const double* s, int64_t N,
                                         labfm_dtype dtype, double scale, void* grad_out,
                                         void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!q || !s || !grad_out) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    if (dtype == LABFM_F32)
        k_kinetic_energy_grad<float><<<grid_of(N), 256, 0, st>>>(N, static_cast<const float*>(q), s, scale,
                                                                 static_cast<float*>(grad_out));
    else
        k_kinetic_energy_grad<double><<<grid_of(N), 256, 0, st>>>(N, static_cast<const double*>(q), s, scale,
                                                                  static_cast<double*>(grad_out));
    LABFM_LAUNCH_CHECK("kinetic energy gradient kernel");
    return LABFM_OK;
}

extern "C" int labfm_probe_momentum(const void* q, const double* px, const double* py, int64_t N,
                                    labfm_dtype dtype, double* j_out, void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!q || !px || !py || !j_out) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    const char* what = "probe momentum kernel";
    return dtype == LABFM_F32
               ? launch_sum(what, k_probe_momentum<float>, N, st, N, static_cast<const float*>(q), px, py, j_out)
               : launch_sum(what, k_probe_momentum<double>, N, st, N, static_cast<const double*>(q), px, py, j_out);
}

extern "C" int labfm_probe_momentum_grad(const void* q, const double* px, const double* py, int64_t N,
                                         labfm_dtype dtype, double scale, void* grad_out, void* stream) {
    if (int rc = check_n(N, dtype)) return rc;
    if (!q || !px || !py || !grad_out) return set_error(LABFM_EINVAL, "null pointer argument");
    cudaStream_t st = as_stream(stream);
    if (dtype == LABFM_F32)
        k_probe_momentum_grad<float><<<grid_of(N), 256, 0, st>>>(N, static_cast<const float*>(q), px, py,
                                                                 scale, static_cast<float*>(grad_out));
    else
        k_probe_momentum_grad<double><<<grid_of(N), 256, 0, st>>>(N, static_cast<const double*>(q), px, py,
                                                                  scale, static_cast<double*>(grad_out));
    LABFM_LAUNCH_CHECK("probe momentum gradient kernel");
    return LABFM_OK;
}
