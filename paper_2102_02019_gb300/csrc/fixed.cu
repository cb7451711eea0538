// Kernels of F64 plans, whose sums run in fixed point (fixed.cuh): the right-hand
// side, the RK stage (recording or not), the derivative combinations of the adjoint and the
// filter, and the packing of the rows.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "fixed.cuh"
#include "labfm_internal.cuh"

namespace labfm {
namespace {

// Resident warps per SM that the registers allow for.  The right-hand-side kernels come with
// 96 registers (20 warps, a few spills), with 128 (16 warps, none) and, for launches that are
// bound by the latency of one warp, with the next chunk's gathers in flight (157 registers,
// 12 warps): see warps_for.  The filter has 96 (it spills 240 bytes in 72: 262,144 nodes of
// order 8 230 us with 28 warps, 225 with 20).
constexpr int kManyWarps = 20, kFewWarps = 16, kAheadWarps = 12, kFilterWarps = 20;
#define LABFM_FIXED_BOUNDS __launch_bounds__(32 * kFixedWarps, W / kFixedWarps)
#define LABFM_FIXED_FILTER_BOUNDS __launch_bounds__(32 * kFixedWarps, kFilterWarps / kFixedWarps)

// Launched so that they may start when the launch before ends (launch_pdl), with the row
// pointers read before the wait for it, but without an early griddepcontrol.launch_dependents:
// the next launch's blocks, placed beside this one's, crowd some SMs' pipes while others
// idle.  A step of 10,000 nodes of order 6 takes 173 us with it and 108 without, of 40,000
// 268 and 243, a right-hand side of 4,096 nodes of order 4 23.3 and 11.6; a right-hand side
// of 1,073 nodes 14.3 us launched plainly and 11.8 so.  Where the next launch finds idle SMs
// it gives nothing (576 nodes of order 4 55.9 us a step with it, 55.5 without).

template <int W, int G, bool WALL>
__global__ void LABFM_FIXED_BOUNDS k_fixed_rhs(PlanView<double> P, Fields in, double* __restrict__ out,
                                               Phys<double> ph, int passes) {
    fixed_nodes<G, false, W == kAheadWarps>(P, in, passes,
                          [&](int i, double a, double u, double v, const double (&d)[12]) {
                              double Ra, Ru, Rv;
                              node_rhs<double, false, WALL>(P, i, d, a, u, v, 1.0, ph, Ra, Ru, Rv);
                              out[i] = Ra;
                              out[P.N + i] = Ru;
                              out[2 * P.N + i] = Rv;
                          });
}

// REC: also stores the node's derivative combinations (k_stage_rec).
template <int W, int G, bool WALL, bool REC>
__global__ void LABFM_FIXED_BOUNDS k_fixed_stage(PlanView<double> P, const Packed<double>* X_in,
                                                 const Packed<double>* Q_in, Packed<double>* Q_out,
                                                 Packed<double>* X_out, double dt, double bk, double ck,
                                                 Phys<double> ph, D8<double>* Dout, int passes) {
    fixed_nodes<G, false, W == kAheadWarps>(P, State{X_in}, passes,
                          [&](int i, double a, double u, double v, const double (&d)[12]) {
                              stage_epilogue<double, false, WALL>(P, i, 0, d, a, u, v, X_in, Q_in, Q_out, X_out,
                                                                  dt, bk, ck, ph);
                              if (REC) {
                                  double c[8];
                                  own_coeffs<double, false>(d, 1.0, c);
                                  d8_store(Dout, i, c);
                              }
                          });
}

template <int W, int G>
__global__ void LABFM_FIXED_BOUNDS k_fixed_coeffs(PlanView<double> P, const Packed<double>* X, D8<double>* Dout,
                                                  int passes) {
    fixed_nodes<G, false, W == kAheadWarps>(P, State{X}, passes,
                          [&](int i, double, double, double, const double (&d)[12]) {
                              double c[8];
                              own_coeffs<double, false>(d, 1.0, c);
                              d8_store(Dout, i, c);
                          });
}

template <int G>
__global__ void LABFM_FIXED_FILTER_BOUNDS k_fixed_filter(PlanView<double> P, const Packed<double>* in, Packed<double>* out,
                                                  double* soa, int passes) {
    fixed_nodes<G, true, false>(P, State{in}, passes,
                         [&](int i, double a, double u, double v, const double (&s)[3]) {
                             store(out, i, a + s[0], u + s[1], v + s[2]);
                             if (soa) {
                                 soa[i] = a + s[0];
                                 soa[P.N + i] = u + s[1];
                                 soa[2 * P.N + i] = v + s[2];
                             }
                         });
}

template <int G>
__global__ void LABFM_FIXED_FILTER_BOUNDS k_fixed_filter_soa(PlanView<double> P, Fields in, double* __restrict__ out,
                                                      int passes) {
    fixed_nodes<G, true, false>(P, in, passes,
                         [&](int i, double a, double u, double v, const double (&s)[3]) {
                             out[i] = a + s[0];
                             out[P.N + i] = u + s[1];
                             out[2 * P.N + i] = v + s[2];
                         });
}

// ---------------------------------------------------------------- packing

// s_j from how far (in log2, 2^20 units of the high words) the entry's largest weight lies
// below the row's largest of the same operator: 15 within a factor of two, one less for every
// factor of two more.
__device__ __forceinline__ int entry_shift(int below) { return max(min(kMostShift + 1 + (below >> 20), kMostShift), 0); }

// Warp per row: the row's exponents, then its records (columns with s_j, weight words).
__global__ void k_pack_fixed(int64_t N, int64_t nnz, int64_t off, const int32_t* __restrict__ row_ptr,
                             const int32_t* __restrict__ col, const double* __restrict__ w,
                             const double* __restrict__ kappa, const int32_t* __restrict__ prow,
                             char* __restrict__ rb, char* __restrict__ fb, int16_t* __restrict__ wexp, bool shifts) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t il = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; il < N; il += warps) {
        const int64_t i = off + il;
        const int r0 = row_ptr[il], len = row_ptr[il + 1] - r0;
        const int p0 = prow[i], plen = prow[i + 1] - p0;
        const double kap = kappa[il];
        auto weight = [&](int64_t src, int o) { return o < 5 ? w[o * nnz + src] : kap * w[5 * nnz + src]; };
        int top[6];  // largest high word of |w|
        bool odd = false;
#pragma unroll
        for (int o = 0; o < 6; ++o) top[o] = 0;
        for (int e = lane; e < len; e += 32)
#pragma unroll
            for (int o = 0; o < 6; ++o) top[o] = max(top[o], __double2hiint(weight(int64_t(r0) + e, o)) & 0x7fffffff);
#pragma unroll
        for (int o = 0; o < 6; ++o) {
            top[o] = __reduce_max_sync(0xffffffffu, top[o]);
            // not finite, or (but for a zero operator) beyond 2^+-400
            odd |= top[o] >= (1023 + 400) << 20 || (top[o] < (1023 - 400) << 20 && top[o] > 0);
        }
        auto shift_of = [&](const int (&h)[6], int o0, int o1) {
            if (!shifts) return 0;
            int below = -0x7fffffff;
            for (int o = o0; o < o1; ++o)
                if (top[o] > 0) below = max(below, h[o] - top[o]);
            return entry_shift(below);
        };
        int exps[6], least[6], used[6];  // of |w| 2^-s: the largest and the smallest but zero; how many are not zero
        float sum[6];
#pragma unroll
        for (int o = 0; o < 6; ++o) {
            exps[o] = -2000;
            least[o] = 4000;
            used[o] = 0;
            sum[o] = 0.0f;
        }
        for (int e = lane; e < len; e += 32) {
            int h[6];
#pragma unroll
            for (int o = 0; o < 6; ++o) {
                const double v = weight(int64_t(r0) + e, o);
                h[o] = __double2hiint(v) & 0x7fffffff;
                odd |= h[o] == 0 && __double2loint(v) != 0;  // below 2^-1022
            }
            const int sr = shift_of(h, 0, 5), sf = shift_of(h, 5, 6);
#pragma unroll
            for (int o = 0; o < 6; ++o) {
                const int s = o < 5 ? sr : sf;
                exps[o] = max(exps[o], (h[o] >> 20) - s - 1022);
                if (h[o] > 0) {
                    least[o] = min(least[o], (h[o] >> 20) - s - 1022);
                    ++used[o];
                }
                // |w| 2^-s over the power of two above the row's largest |w|
                const int ex = (h[o] >> 20) - (top[o] >> 20) - s + 126;
                if (h[o] > 0 && ex > 0) sum[o] += __int_as_float((ex << 23) | ((h[o] & 0xfffff) << 3));
            }
        }
#pragma unroll
        for (int o = 0; o < 6; ++o) {
            exps[o] = __reduce_max_sync(0xffffffffu, exps[o]);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) sum[o] += __shfl_xor_sync(0xffffffffu, sum[o], d);
            if (top[o] == 0 || odd) {
                exps[o] = 0;
            } else {
                float a = ldexpf(sum[o], (top[o] >> 20) - 1022 - exps[o]);
                while (a > 31.9f) {
                    a *= 0.5f;
                    ++exps[o];
                }
                odd |= exps[o] + 2 - least[o] > kMostAlign;
            }
        }
        // an operator on few of the row's entries (beside a boundary: differences along one line)
        // meets differences that are often small against the others'
        int most = 0;
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            used[o] = __reduce_add_sync(0xffffffffu, used[o]);
            most = max(most, used[o]);
        }
#pragma unroll
        for (int o = 0; o < 5; ++o) odd |= used[o] > 0 && 2 * used[o] < most;
        const bool raw = __any_sync(0xffffffffu, odd);
        if (lane == 0) {
            int4 v;
            v.x = (exps[0] & 0xffff) | (exps[1] << 16);
            v.y = (exps[2] & 0xffff) | (exps[3] << 16);
            v.z = (exps[4] & 0xffff) | (exps[5] << 16);
            v.w = 0;  // the operators that are zero throughout the row
#pragma unroll
            for (int o = 0; o < 6; ++o) v.w |= top[o] == 0 ? 1 << o : 0;
            if (raw) v.w = kRawRow;
            reinterpret_cast<int4*>(wexp)[i] = v;
        }
        for (int e = lane; e < plen; e += 32) {
            const int64_t dst = int64_t(p0) + entry_slot(e, plen);
            uint32_t c = uint32_t(i), sr = 0, sf = 0;
            long long word[6] = {0, 0, 0, 0, 0, 0};
            if (e < len) {
                const int64_t src = int64_t(r0) + e;
                c = uint32_t(off + col[src]);
                double v[6];
                int h[6];
#pragma unroll
                for (int o = 0; o < 6; ++o) {
                    v[o] = weight(src, o);
                    h[o] = __double2hiint(v[o]) & 0x7fffffff;
                }
                if (!raw) {
                    sr = uint32_t(shift_of(h, 0, 5));
                    sf = uint32_t(shift_of(h, 5, 6));
                }
#pragma unroll
                for (int o = 0; o < 6; ++o)
                    word[o] = raw ? __double_as_longlong(v[o]) : weight_word(v[o], exps[o], int(o < 5 ? sr : sf));
            }
            *reinterpret_cast<uint32_t*>(rb + Rec<double>::col_e(dst)) = c | (sr << 28);
            *reinterpret_cast<uint32_t*>(fb + Rec<double>::fcol_e(dst)) = c | (sf << 28);
#pragma unroll
            for (int o = 0; o < 6; ++o) *reinterpret_cast<long long*>((o < 5 ? rb : fb) + fixed_at(dst, o)) = word[o];
        }
    }
}

// ---------------------------------------------------------------- dispatch

// Lanes per node: the plan's, 16 at most.  They do not depend on the number of nodes, so
// that an instance's sums are the same alone and in a batch.
int lanes_for(int group) { return std::min(group, 16); }

// The filter's lanes likewise.  Half of them, a whole chunk a lane where the right-hand side
// gives a chunk to two, would idle less at the rows' ends (262,144 nodes, order 8: 188 us for
// 203), but doubles the serial chain that bounds small plans (4,096 nodes, order 8: 20.6 us
// for 12.9; 1,600, order 6: 13.8 for 9.5).
int filter_lanes_for(int group) { return lanes_for(group); }

// Passes per warp: all the lanes' worth (32 nodes a warp, so that the work after the sums
// runs on 32 lanes: 262,144 nodes of order 8, one pass 511 us, two 465, four 459) where
// that still leaves every SM ten warps, else fewer, so that small node sets spread
// over the chip (40,000 nodes of order 6: one pass 69 us, two 58, four 78).  The filter, which
// has little work after its sums, takes two at most, for the finer waves (122,500 nodes of
// order 10 138 us, with four 164; 262,144 of order 8 221 and 225; 90,000 of order 6 52.5 and
// 51.2).
constexpr int kRhsPasses = 16, kFilterPasses = 2;
int passes_for(int64_t nodes, int g, int most) {
    int passes = std::min(g, most);
    while (passes > 1 && nodes * g / (32 * passes) < int64_t(152) * 10) passes /= 2;
    return passes;
}

int grid_of(int64_t nodes, int g, int passes) {
    const int64_t per = int64_t(passes) * kFixedWarps * (32 / g);
    return int((nodes + per - 1) / per);
}

// Which of the right-hand-side kernels a grid takes.  Where all its warps fit at 12 an SM, a
// launch takes as long as one warp does, and the one that gathers ahead is the fastest (us a
// right-hand side, ahead and with 128 registers: 576 nodes of order 4 10.7 and 12.0, of order
// 8 17.4 and 21.0; 4,096 of order 8 18.0 and 21.7; 25,600 of order 6 35.4 and 39.1; 28,900 of
// order 8 56.3 and 62.8).  Else the one with 128
// registers where it takes no more waves than that with 96 (62,500 nodes of order 8 126 and
// 138; 65,536 of order 4 55 and 60; 122,500 of order 10 304 and 325), since it loses the wave
// otherwise (40,000 of order 6 71 and 58; 90,000 153 and 109; 262,144 of order 8 459 and 433).
// Ahead with 128 registers: 65,536 nodes of order 4 58.
int warps_for(int grid) {
    auto waves = [&](int warps) { return (grid - 1) / (152 * (warps / kFixedWarps)); };
    if (waves(kAheadWarps) == 0) return kAheadWarps;
    return waves(kFewWarps) == waves(kManyWarps) ? kFewWarps : kManyWarps;
}

#define LABFM_FIXED_DISPATCH(g, call)                         \
    switch (g) {                                              \
        case 2: { constexpr int G = 2; call; break; }         \
        case 4: { constexpr int G = 4; call; break; }         \
        case 8: { constexpr int G = 8; call; break; }         \
        case 16: { constexpr int G = 16; call; break; }       \
        default: return set_error(LABFM_EINVAL, "unsupported group size"); \
    }
// kernel<W, G, ...> for the grid's number of warps
#define LABFM_FIXED_LAUNCH(g, grid, kernel, ...)                                               \
    switch (warps_for(grid)) {                                                                 \
        case kAheadWarps: { constexpr int W = kAheadWarps;                                     \
            LABFM_FIXED_DISPATCH(g, (e = launch(kernel<W, G __VA_ARGS__>))); break; }          \
        case kFewWarps: { constexpr int W = kFewWarps;                                         \
            LABFM_FIXED_DISPATCH(g, (e = launch(kernel<W, G __VA_ARGS__>))); break; }          \
        default: { constexpr int W = kManyWarps;                                               \
            LABFM_FIXED_DISPATCH(g, (e = launch(kernel<W, G __VA_ARGS__>))); }                 \
    }
#define LABFM_COMMA ,

Phys<double> phys_of(const labfm_phys& ph) { return Phys<double>{ph.c2, ph.mu, ph.gx, ph.gy}; }

}  // namespace

int fixed_rhs(const labfm_plan* p, const void* fields, void* rhs, const labfm_phys& php, int group, cudaStream_t st) {
    const double* f = static_cast<const double*>(fields);
    const Fields in{f, f + p->N, f + 2 * p->N};
    const int g = lanes_for(group), passes = passes_for(p->N, g, kRhsPasses);
    const int grid = grid_of(p->N, g, passes);
    double* out = static_cast<double*>(rhs);
    auto launch = [&](auto* kernel) {
        return launch_pdl(p, kernel, grid, 32 * kFixedWarps, st, view<double>(p), in, out, phys_of(php), passes);
    };
    cudaError_t e = cudaSuccess;
    if (p->wall_slot) {
        LABFM_FIXED_LAUNCH(g, grid, k_fixed_rhs, LABFM_COMMA true);
    } else {
        LABFM_FIXED_LAUNCH(g, grid, k_fixed_rhs, LABFM_COMMA false);
    }
    if (e != cudaSuccess) return cuda_error(e, "fixed-point rhs kernel");
    return LABFM_OK;
}

int fixed_stage(const labfm_plan* p, int64_t n_lo, int64_t n_hi, int group, const void* xin, const void* qin,
                void* qout, void* xout, double dt, double bk, double ck, const labfm_phys& php, void* D,
                cudaStream_t st) {
    if (n_hi <= n_lo) return LABFM_OK;
    const int g = lanes_for(group), passes = passes_for(n_hi - n_lo, g, kRhsPasses);
    const int grid = grid_of(n_hi - n_lo, g, passes);
    const PlanView<double> v = view<double>(p, n_lo, n_hi);
    auto launch = [&](auto* kernel) {
        return launch_pdl(p, kernel, grid, 32 * kFixedWarps, st, v, static_cast<const Packed<double>*>(xin),
                          static_cast<const Packed<double>*>(qin), static_cast<Packed<double>*>(qout),
                          static_cast<Packed<double>*>(xout), dt, bk, ck, phys_of(php), static_cast<D8<double>*>(D),
                          passes);
    };
    cudaError_t e = cudaSuccess;
    if (D) {
        LABFM_FIXED_LAUNCH(g, grid, k_fixed_stage, LABFM_COMMA false LABFM_COMMA true);
    } else if (p->wall_slot) {
        LABFM_FIXED_LAUNCH(g, grid, k_fixed_stage, LABFM_COMMA true LABFM_COMMA false);
    } else {
        LABFM_FIXED_LAUNCH(g, grid, k_fixed_stage, LABFM_COMMA false LABFM_COMMA false);
    }
    if (e != cudaSuccess) return cuda_error(e, "fixed-point rk stage kernel");
    return LABFM_OK;
}

int fixed_coeffs(const labfm_plan* p, const void* X, void* D, cudaStream_t st) {
    const int g = lanes_for(p->group), passes = passes_for(p->N, g, kRhsPasses);
    const int grid = grid_of(p->N, g, passes);
    cudaError_t e = cudaSuccess;
    LABFM_FIXED_DISPATCH(g, (e = launch_pdl(p, k_fixed_coeffs<kManyWarps, G>, grid, 32 * kFixedWarps, st, view<double>(p),
                                            static_cast<const Packed<double>*>(X), static_cast<D8<double>*>(D), passes)));
    if (e != cudaSuccess) return cuda_error(e, "fixed-point derivative kernel");
    return LABFM_OK;
}

int fixed_filter(const labfm_plan* p, int64_t n_lo, int64_t n_hi, int group, const void* in, void* out, void* soa,
                 cudaStream_t st) {
    if (n_hi <= n_lo) return LABFM_OK;
    const int g = filter_lanes_for(group), passes = passes_for(n_hi - n_lo, g, kFilterPasses);
    const int grid = grid_of(n_hi - n_lo, g, passes);
    const PlanView<double> v = view<double>(p, n_lo, n_hi);
    cudaError_t e = cudaSuccess;
    LABFM_FIXED_DISPATCH(g, (e = launch_pdl(p, k_fixed_filter<G>, grid, 32 * kFixedWarps, st, v, static_cast<const Packed<double>*>(in),
                                            static_cast<Packed<double>*>(out), static_cast<double*>(soa), passes)));
    if (e != cudaSuccess) return cuda_error(e, "fixed-point filter kernel");
    return LABFM_OK;
}

int fixed_filter_soa(const labfm_plan* p, const void* in, void* out, cudaStream_t st) {
    const double* f = static_cast<const double*>(in);
    const Fields src{f, f + p->N, f + 2 * p->N};
    const int g = filter_lanes_for(p->group), passes = passes_for(p->N, g, kFilterPasses);
    const int grid = grid_of(p->N, g, passes);
    cudaError_t e = cudaSuccess;
    LABFM_FIXED_DISPATCH(g, (e = launch_pdl(p, k_fixed_filter_soa<G>, grid, 32 * kFixedWarps, st, view<double>(p), src,
                                            static_cast<double*>(out), passes)));
    if (e != cudaSuccess) return cuda_error(e, "fixed-point filter kernel");
    return LABFM_OK;
}

int fixed_pack(const PlanInput& in, int64_t off, labfm_plan* p, cudaStream_t st) {
    const int gw = int(std::min<int64_t>((in.N * 32 + 255) / 256, 1 << 20));
    k_pack_fixed<<<gw, 256, 0, st>>>(in.N, in.nnz, off, in.row_ptr, in.col, in.w, in.kappa, p->row_ptr,
                                     static_cast<char*>(p->w), static_cast<char*>(p->wf), p->wexp,
                                     col_mask(p->N) < 0x7fffffffu);
    LABFM_LAUNCH_CHECK("fixed-point pack kernel");
    return LABFM_OK;
}

}  // namespace labfm
