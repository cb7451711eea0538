// F32 stage and filter launches that are bound by the latency of their loads: those of
// plans whose warps (nearly) all fit on the GPU at once.  In k_stage a lane waits, chunk by
// chunk, for a record and then for the states of its four neighbours, and at the end for
// the node's own register and spacing.  Here it loads its first U chunks, which no earlier
// launch writes, before it waits for the previous launch, has the neighbours of all U in
// flight at once, and the node's own values with them.  Same arithmetic in the same order
// as k_stage, k_stage_rec and k_filter_aos: the results are the same bit for bit.
//
// U is as large as the registers allow for one wave (128 U + 40 bytes a lane or so): 4
// chunks up to 8 warps an SM, 3 up to 12, 2 up to 16, then 1.  Per step (64^2 to 200^2
// nodes at 4 lanes; k_stage and k_filter_aos -> these): 64^2 order 4 20.5 -> 12.6 us, order
// 8 36.5 -> 19.8; 90^2 order 8 54.1 -> 21.3; 110^2 order 8 52.1 -> 27.6; 130^2 order 8
// 53.2 -> 34.3; 160^2 order 4 34.4 -> 29.3; 256^2 order 8 129.3 -> 126.4.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gather.cuh"
#include "labfm_internal.cuh"

namespace labfm {
namespace {

// A state written by an earlier launch.  Not a read-only load (__ldg): that one the compiler
// may move above griddepcontrol.wait, since nothing in this kernel writes the buffer, and
// with the columns in registers before the wait it does.
__device__ __forceinline__ float4 ld_state(const Packed<float>* p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Adds a b to a compensated sum as k_stage does after contraction: a b - c rounded once.
// Written out, because the products may end up in another block than the sums here.
__device__ __forceinline__ void add_product(Acc<float, true>& acc, float a, float b) {
    const float y = __fmaf_rn(a, b, -acc.c);
    const float t = __fadd_rn(acc.s, y);
    acc.c = __fsub_rn(__fsub_rn(t, acc.s), y);
    acc.s = t;
}

struct Chunk24 {
    int c[4];
    float wx[4], wy[4], wxx[4], wxy[4], wyy[4];
};

template <int G, int U, bool WALL, bool REC>
__global__ void __launch_bounds__(32)
    k_stage_ahead(PlanView<float> P, const Packed<float>* X_in, const Packed<float>* Q_in, Packed<float>* Q_out,
                  Packed<float>* X_out, double dt, double bk, double ck, Phys<float> ph, D8<float>* Dout) {
    pdl_launch_dependents();
    const int64_t gt = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int64_t node = P.n_lo + gt / G;
    const int gl = int(gt % G);
    const int i = node < P.n_hi ? int(node) : -1;
    int e0 = 0, e1 = 0;
    float is = 0;
    if (i >= 0) {
        e0 = P.row_ptr[i];
        e1 = P.row_ptr[i + 1];
        is = P.inv_s[i];
    }
    int e = e0 + 4 * gl;
    Chunk24 r[U];
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1)
                load_rhs_chunk(P, e + 4 * G * u, r[u].c, r[u].wx, r[u].wy, r[u].wxx, r[u].wxy, r[u].wyy, 0);
    };
    load();
    pdl_wait();  // the per-node time steps too may come from the launches before
    const double dti = P.dt_node && i >= 0 ? P.dt_node[i] : dt;
    const float cb = float(dti * bk), cx = float(dti * ck);
    float ai = 0, ui = 0, vi = 0, qa = 0, qu = 0, qv = 0;
    if (i >= 0) {
        const float4 x = ld_state(X_in + i);
        ai = x.x;
        ui = x.y;
        vi = x.z;
        if (gl == 0 && Q_in != X_in) {
            const float4 q = ld_state(Q_in + i);
            qa = q.x;
            qu = q.y;
            qv = q.z;
        }
    }
    float ax = 0, ay = 0, ux = 0, uy = 0, vx = 0, vy = 0;
    Acc<float, true> uxx, uxy, uyy, vxx, vxy, vyy;
    while (e < e1) {
        float4 nb[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[u][k] = ld_state(X_in + r[u].c[k]);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float da = nb[u][k].x - ai, du = nb[u][k].y - ui, dv = nb[u][k].z - vi;
                    ax = fma(da, r[u].wx[k], ax);
                    ay = fma(da, r[u].wy[k], ay);
                    ux = fma(du, r[u].wx[k], ux);
                    uy = fma(du, r[u].wy[k], uy);
                    vx = fma(dv, r[u].wx[k], vx);
                    vy = fma(dv, r[u].wy[k], vy);
                    add_product(uxx, du, r[u].wxx[k]);
                    add_product(uxy, du, r[u].wxy[k]);
                    add_product(uyy, du, r[u].wyy[k]);
                    add_product(vxx, dv, r[u].wxx[k]);
                    add_product(vxy, dv, r[u].wxy[k]);
                    add_product(vyy, dv, r[u].wyy[k]);
                }
            }
        e += 4 * G * U;
        load();
    }
    float d[12];
    d[0] = group_sum<G>(ax);
    d[1] = group_sum<G>(ay);
    d[2] = group_sum<G>(ux);
    d[3] = group_sum<G>(uy);
    d[7] = group_sum<G>(vx);
    d[8] = group_sum<G>(vy);
    d[4] = group_sum<G>(uxx.s) - group_sum<G>(uxx.c);
    d[5] = group_sum<G>(uxy.s) - group_sum<G>(uxy.c);
    d[6] = group_sum<G>(uyy.s) - group_sum<G>(uyy.c);
    d[9] = group_sum<G>(vxx.s) - group_sum<G>(vxx.c);
    d[10] = group_sum<G>(vxy.s) - group_sum<G>(vxy.c);
    d[11] = group_sum<G>(vyy.s) - group_sum<G>(vyy.c);
    if (i < 0 || gl != 0) return;
    float Ra, Ru, Rv;
    node_rhs<float, true, WALL>(P, i, d, ai, ui, vi, is, ph, Ra, Ru, Rv);
    if (Q_in == X_in) {
        qa = ai;
        qu = ui;
        qv = vi;
    }
    stage_store(i, cb, cx, Ra, Ru, Rv, qa, qu, qv, Q_out, X_out);
    if (REC) {
        float c[8];
        own_coeffs<float, true>(d, is, c);
        d8_store(Dout, i, c);
    }
}

template <int G, int U>
__global__ void __launch_bounds__(32)
    k_filter_ahead(PlanView<float> P, const Packed<float>* in, Packed<float>* out, float* soa) {
    pdl_launch_dependents();
    const int64_t gt = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int64_t node = P.n_lo + gt / G;
    const int gl = int(gt % G);
    const int i = node < P.n_hi ? int(node) : -1;
    int e0 = 0, e1 = 0;
    if (i >= 0) {
        e0 = P.row_ptr[i];
        e1 = P.row_ptr[i + 1];
    }
    int e = e0 + 4 * gl;
    int c[U][4];
    float wf[U][4];
    auto load = [&]() {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1) load_filt_chunk(P, e + 4 * G * u, c[u], wf[u], 0);
    };
    load();
    pdl_wait();
    float ai = 0, ui = 0, vi = 0;
    if (i >= 0) {
        const float4 x = ld_state(in + i);
        ai = x.x;
        ui = x.y;
        vi = x.z;
    }
    Acc<float, true> aa, uu, vv;
    while (e < e1) {
        float4 nb[U][4];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) nb[u][k] = ld_state(in + c[u][k]);
            }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + 4 * G * u < e1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    add_product(aa, nb[u][k].x - ai, wf[u][k]);
                    add_product(uu, nb[u][k].y - ui, wf[u][k]);
                    add_product(vv, nb[u][k].z - vi, wf[u][k]);
                }
            }
        e += 4 * G * U;
        load();
    }
    const float sa = group_sum<G>(aa.s) - group_sum<G>(aa.c);
    const float su = group_sum<G>(uu.s) - group_sum<G>(uu.c);
    const float sv = group_sum<G>(vv.s) - group_sum<G>(vv.c);
    if (i < 0 || gl != 0) return;
    store(out, i, ai + sa, ui + su, vi + sv);
    if (soa) {
        soa[i] = ai + sa;
        soa[P.N + i] = ui + su;
        soa[2 * P.N + i] = vi + sv;
    }
}

int grid_of(int64_t nodes, int g) { return int((nodes * g + 31) / 32); }

int chunks_ahead(int64_t nodes, int g) {
    const int64_t per_sm = (nodes * g / 32 + 151) / 152;
    // 16 and 32 lanes read most rows in one or two chunks a lane
    if (per_sm <= 8 && g <= 8) return 4;
    if (per_sm <= 12 && g <= 8) return 3;
    return per_sm <= 16 ? 2 : 1;
}

template <int G, int U>
cudaError_t stage_u(const labfm_plan* p, const PlanView<float>& v, const Packed<float>* xin, const Packed<float>* qin,
                    Packed<float>* qout, Packed<float>* xout, double dt, double bk, double ck, const Phys<float>& ph,
                    D8<float>* D, cudaStream_t st) {
    auto* kernel = D ? k_stage_ahead<G, U, false, true>
                     : (p->wall_slot ? k_stage_ahead<G, U, true, false> : k_stage_ahead<G, U, false, false>);
    return launch_pdl(p, kernel, grid_of(v.n_hi - v.n_lo, G), 32, st, v, xin, qin, qout, xout, dt, bk, ck, ph, D);
}

template <int G, int U>
cudaError_t filter_u(const labfm_plan* p, const PlanView<float>& v, const Packed<float>* in, Packed<float>* out,
                     float* soa, cudaStream_t st) {
    return launch_pdl(p, k_filter_ahead<G, U>, grid_of(v.n_hi - v.n_lo, G), 32, st, v, in, out, soa);
}

#define LABFM_AHEAD_U(G, U, call)                            \
    if constexpr (G <= 8) {                                  \
        if (u == 4) { constexpr int U = 4; e = call; }       \
        if (u == 3) { constexpr int U = 3; e = call; }       \
    }                                                        \
    if (u == 2) { constexpr int U = 2; e = call; }           \
    if (u == 1) { constexpr int U = 1; e = call; }
#define LABFM_AHEAD_DISPATCH(call)                                                  \
    switch (group) {                                                                \
        case 2: { constexpr int G = 2; LABFM_AHEAD_U(G, U, call) break; }           \
        case 4: { constexpr int G = 4; LABFM_AHEAD_U(G, U, call) break; }           \
        case 8: { constexpr int G = 8; LABFM_AHEAD_U(G, U, call) break; }           \
        case 16: { constexpr int G = 16; LABFM_AHEAD_U(G, U, call) break; }         \
        case 32: { constexpr int G = 32; LABFM_AHEAD_U(G, U, call) break; }         \
        default: return set_error(LABFM_EINVAL, "unsupported group size");          \
    }

}  // namespace

// Up to 56 warps an SM, 68,000 nodes at 4 lanes: there one chunk ahead takes 126.4 us a step
// (256^2, order 8) against k_stage's 129.3; at 360^2 239 against 235.  No L2 prefetch within
// the row: 131.7 with it.
bool ahead_serves(int64_t nodes, int group) { return nodes * group <= int64_t(152) * 56 * 32; }

int ahead_stage(const labfm_plan* p, int64_t n_lo, int64_t n_hi, int group, const void* xin, const void* qin,
                void* qout, void* xout, double dt, double bk, double ck, const labfm_phys& php, void* D,
                cudaStream_t st) {
    if (n_hi <= n_lo) return LABFM_OK;
    const Phys<float> ph{float(php.c2), float(php.mu), float(php.gx), float(php.gy)};
    const PlanView<float> v = view<float>(p, n_lo, n_hi);
    const int u = chunks_ahead(n_hi - n_lo, group);
    cudaError_t e = cudaErrorInvalidValue;
    LABFM_AHEAD_DISPATCH((stage_u<G, U>(p, v, static_cast<const Packed<float>*>(xin), static_cast<const Packed<float>*>(qin),
                                        static_cast<Packed<float>*>(qout), static_cast<Packed<float>*>(xout), dt, bk, ck,
                                        ph, static_cast<D8<float>*>(D), st)));
    if (e != cudaSuccess) return cuda_error(e, "rk stage kernel (chunks ahead)");
    return LABFM_OK;
}

int ahead_filter(const labfm_plan* p, int64_t n_lo, int64_t n_hi, int group, const void* in, void* out, void* soa,
                 cudaStream_t st) {
    if (n_hi <= n_lo) return LABFM_OK;
    const PlanView<float> v = view<float>(p, n_lo, n_hi);
    const int u = chunks_ahead(n_hi - n_lo, group);
    cudaError_t e = cudaErrorInvalidValue;
    LABFM_AHEAD_DISPATCH((filter_u<G, U>(p, v, static_cast<const Packed<float>*>(in), static_cast<Packed<float>*>(out),
                                         static_cast<float*>(soa), st)));
    if (e != cudaSuccess) return cuda_error(e, "filter kernel (chunks ahead)");
    return LABFM_OK;
}

}  // namespace labfm
