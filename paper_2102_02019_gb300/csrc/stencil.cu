// Neighbour search (Section 2 of the paper: the stencil of node i is every node
// j != i with |r_ji| <= 2 h_i) on a uniform cell list, plus the exclusive scan
// used to turn per-row counts into CSR row pointers.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "labfm_internal.cuh"
#include "nvtx.cuh"

namespace labfm {

// ---------------------------------------------------------------- scan

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int64_t kScanTile = int64_t(kScanThreads) * kScanItems;

// Inclusive block scan of one int64 per thread; returns the inclusive prefix
// and writes the block total to *total.
__device__ int64_t block_inclusive_scan(int64_t v, int64_t* warp_sums, int64_t* total) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    for (int off = 1; off < 32; off <<= 1) {
        int64_t n = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += n;
    }
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        int64_t w = lane < nw ? warp_sums[lane] : 0;
        for (int off = 1; off < 32; off <<= 1) {
            int64_t n = __shfl_up_sync(0xffffffffu, w, off);
            if (lane >= off) w += n;
        }
        if (lane < nw) warp_sums[lane] = w;
    }
    __syncthreads();
    int64_t incl = v + (warp > 0 ? warp_sums[warp - 1] : 0);
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return incl;
}

__global__ void k_scan_reduce(const int32_t* __restrict__ in, int64_t n, int64_t* __restrict__ sums) {
    __shared__ int64_t ws[32];
    __shared__ int64_t tot;
    const int64_t base = int64_t(blockIdx.x) * kScanTile + int64_t(threadIdx.x) * kScanItems;
    int64_t local = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t idx = base + k;
        if (idx < n) local += in[idx];
    }
    block_inclusive_scan(local, ws, &tot);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// One block: exclusive scan of the per-tile sums, carried across chunks.
__global__ void k_scan_sums(int64_t* __restrict__ sums, int64_t nb, int64_t* __restrict__ total) {
    __shared__ int64_t ws[32];
    __shared__ int64_t tot;
    int64_t carry = 0;
    for (int64_t c0 = 0; c0 < nb; c0 += blockDim.x) {
        const int64_t idx = c0 + threadIdx.x;
        const int64_t v = idx < nb ? sums[idx] : 0;
        const int64_t incl = block_inclusive_scan(v, ws, &tot);
        if (idx < nb) sums[idx] = carry + incl - v;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void k_scan_apply(const int32_t* in, int32_t* out, int64_t n,
                             const int64_t* __restrict__ sums, const int64_t* __restrict__ total) {
    __shared__ int64_t ws[32];
    const int64_t base = int64_t(blockIdx.x) * kScanTile + int64_t(threadIdx.x) * kScanItems;
    int32_t vals[kScanItems];
    int64_t local = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t idx = base + k;
        vals[k] = idx < n ? in[idx] : 0;
        local += vals[k];
    }
    const int64_t incl = block_inclusive_scan(local, ws, nullptr);
    int64_t run = sums[blockIdx.x] + incl - local;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t idx = base + k;
        if (idx < n) out[idx] = int32_t(run);
        run += vals[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = int32_t(*total);
}

}  // namespace

size_t exclusive_scan_scratch_bytes(int64_t n) {
    const int64_t nb = std::max<int64_t>(1, (n + kScanTile - 1) / kScanTile);
    return size_t(nb) * sizeof(int64_t);
}

int exclusive_scan_i32(const int32_t* in, int32_t* out, int64_t n, int64_t* total_dev,
                       void* scratch, size_t scratch_bytes, cudaStream_t st) {
    const int64_t nb = std::max<int64_t>(1, (n + kScanTile - 1) / kScanTile);
    if (scratch_bytes < size_t(nb) * sizeof(int64_t))
        return set_error(LABFM_EINVAL, "scan scratch too small");
    int64_t* sums = static_cast<int64_t*>(scratch);
    k_scan_reduce<<<unsigned(nb), kScanThreads, 0, st>>>(in, n, sums);
    k_scan_sums<<<1, kScanThreads, 0, st>>>(sums, nb, total_dev);
    k_scan_apply<<<unsigned(nb), kScanThreads, 0, st>>>(in, out, n, sums, total_dev);
    LABFM_LAUNCH_CHECK("exclusive scan");
    return LABFM_OK;
}

// ---------------------------------------------------------------- CSR check

namespace {
__global__ void k_check_row_ptr(const int32_t* __restrict__ rp, int64_t N, int64_t nnz, int* flags) {
    const int64_t gt = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    bool bad = false;
    for (int64_t i = gt; i < N; i += int64_t(gridDim.x) * blockDim.x) bad |= rp[i + 1] < rp[i];
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flags, 4);
    if (gt == 0) {
        if (rp[0] != 0) atomicOr(flags, 1);
        if (nnz >= 0 && int64_t(rp[N]) != nnz) atomicOr(flags, 2);
    }
}

__global__ void k_check_cols(const int32_t* __restrict__ col, int64_t n, int64_t N, int* flags) {
    bool bad = false;
    for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < n; e += int64_t(gridDim.x) * blockDim.x) {
        const int32_t c = col[e];
        bad |= c < 0 || int64_t(c) >= N;
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flags, 8);
}
}  // namespace

int validate_csr(const int32_t* row_ptr, const int32_t* col, int64_t N, int64_t nnz, cudaStream_t st) {
    int* f = nullptr;
    LABFM_CUDA_TRY(cudaMallocAsync(reinterpret_cast<void**>(&f), sizeof(int), st));
    int flags = 0, total = 0;
    cudaError_t e = cudaMemsetAsync(f, 0, sizeof(int), st);
    if (e == cudaSuccess) {
        const int g = int(std::min<int64_t>((N + 255) / 256, 152 * 8));
        k_check_row_ptr<<<g, 256, 0, st>>>(row_ptr, N, nnz, f);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&flags, f, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&total, row_ptr + N, sizeof(int32_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && flags == 0 && total > 0) {
        if (!col) {
            flags = 16;
        } else {
            const int g = int(std::min<int64_t>((int64_t(total) + 255) / 256, 152 * 8));
            k_check_cols<<<g, 256, 0, st>>>(col, total, N, f);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaMemcpyAsync(&flags, f, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        }
    }
    cudaFreeAsync(f, st);
    if (e != cudaSuccess) return cuda_error(e, "checking the CSR");
    if (flags & 1) return set_error(LABFM_EINVAL, "row_ptr[0] is not 0");
    if (flags & 2) return set_error(LABFM_EINVAL, "row_ptr[N] differs from nnz");
    if (flags & 4) return set_error(LABFM_EINVAL, "row_ptr decreases");
    if (flags & 16) return set_error(LABFM_EINVAL, "null col for a non-empty CSR");
    if (flags & 8) return set_error(LABFM_EINVAL, "a column index is outside [0, N)");
    return LABFM_OK;
}

// ---------------------------------------------------------------- cell list

namespace {

struct CellGrid {
    double csx, csy;  // cell sizes
    int ncx, ncy;
    // in units of max(Lx, Ly), for the FP32 tests: box, cells and their inverses, and the
    // slack (in cells) that covers the rounding of a position and a radius
    float Lx, Ly, wx, wy, iwx, iwy, slx, sly;
};

// Head of the search's work buffer: what the kernels hand to one another and to the host.
struct SearchState {
    unsigned long long hmin;  // bit pattern of the smallest h (positive doubles order like their bits)
    int bad;                  // a node outside the box, or an h that is not positive and finite
    int longest;              // entries of the longest row
    int64_t nnz;
    int64_t cell_total;
    CellGrid g;
};

// The work buffer: SearchState, then the arrays below, each 256-byte aligned.  Its size
// depends on N alone, so a caller can allocate it before anything has run.
struct SearchWork {
    SearchState* st;
    int32_t* cell_start;  // max_cells + 1
    int32_t* cell_of;     // N: cell of node i
    int32_t* rank;        // N: place of node i within its cell
    int32_t* node;        // N: nodes in cell order
    float2* pos;          // N: their positions over max(Lx, Ly)
    char* scan;
    size_t scan_bytes;
    int64_t max_cells;
    size_t bytes;
};

SearchWork split_search_work(void* base, int64_t N) {
    SearchWork w{};
    size_t at = 0;
    auto take = [&](size_t bytes) {
        char* p = static_cast<char*>(base) + at;
        at += (bytes + 255) & ~size_t(255);
        return p;
    };
    w.max_cells = std::min<int64_t>(4 * N + 64, (int64_t(1) << 31) - 2);  // cells are numbered in int32
    w.scan_bytes = exclusive_scan_scratch_bytes(w.max_cells);
    w.st = reinterpret_cast<SearchState*>(take(sizeof(SearchState)));
    w.cell_start = reinterpret_cast<int32_t*>(take(size_t(w.max_cells + 1) * 4));
    w.cell_of = reinterpret_cast<int32_t*>(take(size_t(N) * 4));
    w.rank = reinterpret_cast<int32_t*>(take(size_t(N) * 4));
    w.node = reinterpret_cast<int32_t*>(take(size_t(N) * 4));
    w.pos = reinterpret_cast<float2*>(take(size_t(N) * 8));
    w.scan = take(w.scan_bytes);
    w.bytes = at;
    return w;
}

struct Box {
    double Lx, Ly;
    bool px, py;
};

// Smallest h and input validation: a periodic axis takes [0, L), a bounded one [0, L]
// (a wall may lie on the edge of the box).  One atomic per warp: an atomic per node on the
// one word made this 86 us for 65,536 nodes, now 3 us.
__global__ void k_bounds(const double* __restrict__ xy, const double* __restrict__ h, int64_t N, Box b,
                         SearchState* st) {
    unsigned long long lo = ~0ull;
    bool bad = false;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const double x = xy[2 * i], y = xy[2 * i + 1], hi = h[i];
        const bool ok = isfinite(x) && isfinite(y) && isfinite(hi) && hi > 0.0 && x >= 0.0 &&
                        (b.px ? x < b.Lx : x <= b.Lx) && y >= 0.0 && (b.py ? y < b.Ly : y <= b.Ly);
        bad |= !ok;
        const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(hi));
        if (ok && bits < lo) lo = bits;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, lo, off);
        lo = o < lo ? o : lo;
    }
    const bool any = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
        if (any) atomicOr(&st->bad, 1);
        atomicMin(&st->hmin, lo);
    }
}

__global__ void k_search_init(SearchState* st) {
    *st = SearchState{};
    st->hmin = ~0ull;
}

// Cells of about h_min, at most max_cells of them; on the device, so that the whole
// search synchronises once, after its count.
__global__ void k_make_grid(SearchState* st, Box b, int64_t max_cells) {
    CellGrid g{};
    g.csx = b.Lx;
    g.csy = b.Ly;
    g.ncx = g.ncy = 1;
    if (!st->bad) {
        double cs = __longlong_as_double(static_cast<long long>(st->hmin));
        const double cap = double(max_cells);
        if ((b.Lx / cs) * (b.Ly / cs) > cap) cs = sqrt(b.Lx * b.Ly / cap);
        const double nx = fmin(fmax(floor(b.Lx / cs), 1.0), fmin(cap, 1.0e9));
        const double ny = fmin(fmax(floor(b.Ly / cs), 1.0), fmin(cap, 1.0e9));
        g.ncx = int(nx);
        // a box much narrower than a cell has more rows than the area's share of cells
        g.ncy = int(fmin(ny, fmax(floor(cap / nx), 1.0)));
        g.csx = b.Lx / g.ncx;
        g.csy = b.Ly / g.ncy;
    }
    const double inv_L = 1.0 / fmax(b.Lx, b.Ly);
    g.Lx = float(b.Lx * inv_L);
    g.Ly = float(b.Ly * inv_L);
    g.wx = float(g.csx * inv_L);
    g.wy = float(g.csy * inv_L);
    g.iwx = 1.0f / g.wx;
    g.iwy = 1.0f / g.wy;
    g.slx = 1e-4f + 1e-6f * float(g.ncx);
    g.sly = 1e-4f + 1e-6f * float(g.ncy);
    st->g = g;
}

__device__ __forceinline__ int cell_coord(double x, double cs, int nc) {
    int c = int(floor(x / cs));
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__global__ void k_cell_count(const double* __restrict__ xy, int64_t N, const SearchState* __restrict__ st,
                             int32_t* __restrict__ cell_of, int32_t* __restrict__ rank,
                             int32_t* __restrict__ cell_count) {
    const CellGrid g = st->g;
    if (st->bad) return;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int c = cell_coord(xy[2 * i + 1], g.csy, g.ncy) * g.ncx + cell_coord(xy[2 * i], g.csx, g.ncx);
        cell_of[i] = c;
        rank[i] = atomicAdd(cell_count + c, 1);
    }
}

__global__ void k_cell_scatter(const double* __restrict__ xy, int64_t N, const SearchState* __restrict__ st,
                               double inv_L, const int32_t* __restrict__ cell_of, const int32_t* __restrict__ rank,
                               const int32_t* __restrict__ cell_start, int32_t* __restrict__ node,
                               float2* __restrict__ pos) {
    if (st->bad) return;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < N;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int slot = cell_start[cell_of[i]] + rank[i];
        node[slot] = int32_t(i);
        pos[slot] = make_float2(float(xy[2 * i] * inv_L), float(xy[2 * i + 1] * inv_L));
    }
}

// Cells [lo, hi] covering [x - r, x + r] (in cells) along one axis, widened by `slack`
// for the rounding of x and r.  A periodic range may stick out by less than nc cells on
// either side; one that meets itself becomes 0 .. nc - 1 (returns true).
__device__ __forceinline__ bool axis_range(float x, float r, float slack, int nc, bool periodic, int* lo, int* hi) {
    const float big = 2.0f * float(nc) + 2.0f;
    int a = int(fmaxf(floorf(x - r - slack), -big));
    int b = int(fminf(floorf(x + r + slack), big));
    bool all = false;
    if (periodic) {
        all = b - a + 1 >= nc;
        if (all) {
            a = 0;
            b = nc - 1;
        }
    } else {
        a = min(max(a, 0), nc - 1);
        b = max(min(b, nc - 1), 0);
    }
    *lo = a;
    *hi = b;
    return all;
}

constexpr int kSearchWarps = 4;
constexpr int kRowCap = 512;  // longest row that is put in order by the warp that finds it

// Bitonic sort of 32 P keys held P to a lane; sorted element e ends in lane e / P,
// register e % P.  Strides below P stay within a lane.
template <int P>
__device__ __forceinline__ void bitonic_sort(int (&v)[P], int lane) {
#pragma unroll
    for (int k = 2; k <= 32 * P; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= P) {
                const int lj = j / P;
                // k > j >= P: the direction is a bit of the lane
                const bool up = ((lane * P) & k) == 0;
                const bool low = (lane & lj) == 0;
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const int o = __shfl_xor_sync(0xffffffffu, v[p], lj);
                    v[p] = (up == low) ? min(v[p], o) : max(v[p], o);
                }
            } else {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if (p & j) continue;
                    const bool up = k < P ? (p & k) == 0 : ((lane * P) & k) == 0;
                    const int a = v[p], b = v[p | j];
                    if (k < P) {
                        v[p] = up ? min(a, b) : max(a, b);
                        v[p | j] = up ? max(a, b) : min(a, b);
                    } else {
                        const bool swap = (a > b) == up;
                        v[p] = swap ? b : a;
                        v[p | j] = swap ? a : b;
                    }
                }
            }
        }
    }
}

// One pad word per 32, so that the lanes' runs of P sorted keys land in different banks.
__device__ __forceinline__ int padded(int e) { return e + (e >> 5); }

template <int P>
__device__ __forceinline__ void sort_row(int32_t* buf, int n, int lane, int32_t* __restrict__ out) {
    int v[P];
#pragma unroll
    for (int p = 0; p < P; ++p) v[p] = p * 32 + lane < n ? buf[p * 32 + lane] : 0x7fffffff;
    bitonic_sort<P>(v, lane);
    __syncwarp();
#pragma unroll
    for (int p = 0; p < P; ++p) buf[padded(lane * P + p)] = v[p];
    __syncwarp();
    for (int e = lane; e < n; e += 32) out[e] = buf[padded(e)];
    __syncwarp();
}

// The rank of every key among its row.
__device__ __forceinline__ void rank_row(const int32_t* src, int n, int lane, int32_t* __restrict__ out) {
    for (int e = lane; e < n; e += 32) {
        const int v = src[e];
        int rank = 0;
        for (int k = 0; k < n; ++k) rank += src[k] < v;
        out[rank] = v;
    }
    __syncwarp();
}

// The stencils, one warp per node in cell order.  MODE 0 counts, MODE 1 writes each row
// sorted by ascending j, MODE 2 writes it as found (rows longer than kRowCap; a sort
// kernel follows).
//
// A candidate is decided in FP32 on positions over max(Lx, Ly).  Their differences are
// within 2^-22.5 of the exact ones, three times that where the two take different images
// half a box away; so outside a band of 24 * 2^-24 around the radius (and 4e-6 of its
// square, for the FP32 products) the FP32 distance has the same answer as the exact FP64
// test, and inside it, one candidate in a thousand at a million nodes, that test is made.
// The FP64 pipe of this chip runs 2 lanes a clock and an SM, and the test takes ten FP64
// instructions.  Each lane works out one row of cells, narrowed to the chord of the
// circle (20 instead of 25 h^2 searched, of which 12.6 h^2 are stencil); the candidates of
// all rows are then taken 32 at a time, each lane finding its row by bisection of the
// rows' prefix sums; the row is compacted in shared memory and sorted in registers
// (256 keys in about 500 instructions, against 1,550 for ranking 152).  Bound by
// instruction issue.  1.0M nodes of varying h at order 10 (152 entries): the whole search
// 44.1 -> 2.46 ms, against a thread per node testing every candidate in FP64, twice for
// the count and once to fill, and a ranking sort; half of it is the sort.  48 registers
// (10 blocks an SM; with 92 the fill alone took 2.7 ms), and a grid of 16 blocks for each
// that is resident (4: 2.68 ms, one node a warp: 2.72).
template <int MODE>
__global__ void __launch_bounds__(32 * kSearchWarps, 10)
    k_neighbours(const double* __restrict__ xy, const double* __restrict__ h, int64_t N, Box b, double inv_L,
                 SearchState* st, const int32_t* __restrict__ cell_start, const int32_t* __restrict__ node,
                 const float2* __restrict__ pos, int32_t* __restrict__ counts, const int32_t* __restrict__ row_ptr,
                 int32_t* __restrict__ out) {
    __shared__ int32_t s_row[MODE == 1 ? kSearchWarps : 1][MODE == 1 ? kRowCap + kRowCap / 32 : 1];
    if (st->bad) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const CellGrid g = st->g;
    const float Lxf = g.Lx, Lyf = g.Ly;
    constexpr float kBand = 24.0f / 16777216.0f;
    int longest = 0;
    for (int64_t slot = int64_t(blockIdx.x) * kSearchWarps + warp; slot < N;
         slot += int64_t(gridDim.x) * kSearchWarps) {
        const int i = node[slot];
        const float2 c = pos[slot];
        const double two_h = 2.0 * h[i];
        const float r = float(two_h * inv_L);
        const float rin = r - kBand, rout = r + kBand;
        const float in2 = rin > 0.0f ? rin * rin * (1.0f - 4e-6f) : -1.0f;
        const float out2 = rout * rout * (1.0f + 4e-6f);
        const float X = c.x * g.iwx, Y = c.y * g.iwy;
        const int r0 = MODE == 0 ? 0 : row_ptr[i];
        const int room = MODE == 0 ? 0 : row_ptr[i + 1] - r0;  // nothing is written past the counted row
        // whether any candidate can be another image of its node (wide enough for every rounding)
        const bool image_x = b.px && (c.x < rout + 1e-5f || c.x > Lxf - rout - 1e-5f);
        const bool image_y = b.py && (c.y < rout + 1e-5f || c.y > Lyf - rout - 1e-5f);
        int ylo, yhi, cnt = 0;
        const bool all_rows = axis_range(Y, r * g.iwy, g.sly, g.ncy, b.py, &ylo, &yhi);
        for (int y0 = ylo; y0 <= yhi; y0 += 32) {
            // lane -> one row of cells: a run of consecutive slots [s1, s1 + len1), and where
            // the row meets the edge of the box a second one from s2
            const int cy = y0 + lane;
            int s1 = 0, len1 = 0, s2 = 0, len = 0;
            if (cy <= yhi) {
                float half = r * g.iwx;
                if (!all_rows) {
                    const float gap = fmaxf(fmaxf(float(cy) - Y, Y - float(cy + 1)) - g.sly, 0.0f) * g.wy;
                    half = sqrtf(fmaxf(out2 - gap * gap, 0.0f)) * g.iwx;
                }
                int xlo, xhi;
                axis_range(X, half, g.slx, g.ncx, b.px, &xlo, &xhi);
                const int32_t* cs = cell_start + int64_t(cy < 0 ? cy + g.ncy : (cy >= g.ncy ? cy - g.ncy : cy)) * g.ncx;
                if (xlo < 0 || xhi >= g.ncx) {
                    s2 = cs[0];
                    len = cs[(xlo < 0 ? xhi : xhi - g.ncx) + 1] - s2;
                    if (xlo < 0) xlo += g.ncx;
                    xhi = g.ncx - 1;
                }
                s1 = cs[xlo];
                len1 = cs[xhi + 1] - s1;
                len += len1;
            }
            const int rows = min(yhi - y0 + 1, 32);
            int incl = len;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            const int first = s1 - (incl - len);            // candidate t of this row is slot first + t
            const int end1 = incl - len + len1;             // up to here,
            const int wrap = s2 - s1 - len1;                // and from here on first + t + wrap
            const bool wraps = __any_sync(0xffffffffu, len > len1);
            for (int t0 = 0; t0 < total; t0 += 32) {
                const int t = t0 + lane;
                // the row holding candidate t: how many of the rows end at or before t
                int q = 0;
                auto descend = [&](int step) {
                    const int e = __shfl_sync(0xffffffffu, incl, q + step - 1);
                    if (t >= e && t < total) q += step;
                };
                if (rows > 8) {
                    descend(16);
                    descend(8);
                }
                descend(4);
                descend(2);
                descend(1);
                int k = __shfl_sync(0xffffffffu, first, q) + t;
                if (wraps) {
                    const int e = __shfl_sync(0xffffffffu, end1, q), d = __shfl_sync(0xffffffffu, wrap, q);
                    if (t >= e) k += d;
                }
                k = t < total ? k : int(slot);  // past the last candidate the node itself, which is none
                const float2 p = pos[k];
                float dx = p.x - c.x, dy = p.y - c.y;
                if (image_x) dx = dx > 0.5f * Lxf ? dx - Lxf : (dx < -0.5f * Lxf ? dx + Lxf : dx);
                if (image_y) dy = dy > 0.5f * Lyf ? dy - Lyf : (dy < -0.5f * Lyf ? dy + Lyf : dy);
                const float d2 = dx * dx + dy * dy;
                const bool near = d2 < out2 && k != int(slot);
                bool in = near && d2 <= in2;
                if (__any_sync(0xffffffffu, near && !in)) {  // too close to the radius for FP32
                    if (near && !in) {
                        const int64_t j = node[k];
                        const double ex = min_image(__dsub_rn(xy[2 * j], xy[2 * int64_t(i)]), b.Lx, b.px);
                        const double ey = min_image(__dsub_rn(xy[2 * j + 1], xy[2 * int64_t(i) + 1]), b.Ly, b.py);
                        in = __dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)) <= __dmul_rn(two_h, two_h);
                    }
                }
                const unsigned hits = __ballot_sync(0xffffffffu, in);
                if (MODE != 0 && in) {
                    const int at = cnt + __popc(hits & ((1u << lane) - 1u));
                    if (MODE == 1) {
                        if (at < kRowCap) s_row[warp][at] = node[k];
                    } else if (at < room) {
                        out[int64_t(r0) + at] = node[k];
                    }
                }
                cnt += __popc(hits);
            }
        }
        if (MODE == 0) {
            if (lane == 0) counts[i] = cnt;
            longest = max(longest, cnt);
        }
        if (MODE == 1) {
            __syncwarp();
            int32_t* dst = out + r0;
            const int n = min(cnt, min(room, kRowCap));
            if (n <= 64) sort_row<2>(s_row[warp], n, lane, dst);
            else if (n <= 128) sort_row<4>(s_row[warp], n, lane, dst);
            else if (n <= 256) sort_row<8>(s_row[warp], n, lane, dst);
            else rank_row(s_row[warp], n, lane, dst);
        }
    }
    if (MODE == 0 && lane == 0 && longest > st->longest) atomicMax(&st->longest, longest);
}

// Sort each row by ascending j: warp per row, rank of every entry among its row.
constexpr int kSortWarps = 8;

__global__ void k_sort_rows(const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ tmp,
                            int32_t* __restrict__ col, int64_t N) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    for (int64_t i = blockIdx.x * int64_t(kSortWarps) + warp; i < N;
         i += int64_t(gridDim.x) * kSortWarps) {
        const int r0 = row_ptr[i];
        const int n = row_ptr[i + 1] - r0;
        const int32_t* src = tmp + r0;
        rank_row(src, n, lane, col + r0);
    }
}

struct StreamBuffer {  // stream-ordered scratch of one call
    cudaStream_t st;
    void* p = nullptr;
    explicit StreamBuffer(cudaStream_t s) : st(s) {}
    ~StreamBuffer() {
        if (p) cudaFreeAsync(p, st);
    }
};

int check_search_args(const double* xy, const double* h, int64_t N, double Lx, double Ly, const int32_t* row_ptr) {
    if (!xy || !h || !row_ptr) return set_error(LABFM_EINVAL, "null pointer argument");
    if (N <= 0 || N >= (int64_t(1) << 31) - 1) return set_error(LABFM_EINVAL, "N out of range");
    if (!(Lx > 0.0) || !(Ly > 0.0) || !isfinite(Lx) || !isfinite(Ly))
        return set_error(LABFM_EINVAL, "domain size must be positive and finite");
    return LABFM_OK;
}

Box make_box(double Lx, double Ly, uint32_t mask) { return Box{Lx, Ly, (mask & 1u) != 0, (mask & 2u) != 0}; }

int search_grid(int64_t N) { return int(std::min<int64_t>((N + kSearchWarps - 1) / kSearchWarps, 152 * 10 * 16)); }

// Cell list and row counts: row_ptr, nnz and the longest row; synchronises once.
int count_stencils(const double* xy, const double* h, int64_t N, double Lx, double Ly, uint32_t mask,
                   int32_t* row_ptr, void* work, int64_t* nnz_out, int* longest_out, cudaStream_t st) {
    const SearchWork w = split_search_work(work, N);
    const Box b = make_box(Lx, Ly, mask);
    const double inv_L = 1.0 / std::max(Lx, Ly);
    const int nblk = int(std::min<int64_t>((N + 255) / 256, 152 * 8));
    k_search_init<<<1, 1, 0, st>>>(w.st);
    k_bounds<<<nblk, 256, 0, st>>>(xy, h, N, b, w.st);
    k_make_grid<<<1, 1, 0, st>>>(w.st, b, w.max_cells);
    LABFM_CUDA_TRY(cudaMemsetAsync(w.cell_start, 0, size_t(w.max_cells) * sizeof(int32_t), st));
    k_cell_count<<<nblk, 256, 0, st>>>(xy, N, w.st, w.cell_of, w.rank, w.cell_start);
    LABFM_LAUNCH_CHECK("cell count kernel");
    int rc = exclusive_scan_i32(w.cell_start, w.cell_start, w.max_cells, &w.st->cell_total, w.scan, w.scan_bytes, st);
    if (rc) return rc;
    k_cell_scatter<<<nblk, 256, 0, st>>>(xy, N, w.st, inv_L, w.cell_of, w.rank, w.cell_start, w.node, w.pos);
    k_neighbours<0><<<search_grid(N), 32 * kSearchWarps, 0, st>>>(xy, h, N, b, inv_L, w.st, w.cell_start, w.node,
                                                                  w.pos, row_ptr, nullptr, nullptr);
    LABFM_LAUNCH_CHECK("neighbour count kernel");
    if ((rc = exclusive_scan_i32(row_ptr, row_ptr, N, &w.st->nnz, w.scan, w.scan_bytes, st))) return rc;
    SearchState host{};
    LABFM_CUDA_TRY(cudaMemcpyAsync(&host, w.st, sizeof(host), cudaMemcpyDeviceToHost, st));
    LABFM_CUDA_TRY(cudaStreamSynchronize(st));
    if (host.bad)
        return set_error(LABFM_EINVAL,
                         "a node lies outside the box ([0, L) on a periodic axis, [0, L] on a bounded "
                         "one) or has a non-positive or non-finite h");
    *nnz_out = host.nnz;
    *longest_out = host.longest;
    if (host.nnz >= (int64_t(1) << 31))
        return set_error(LABFM_ECAPACITY, "stencil has 2^31 or more entries (int32 CSR)");
    return LABFM_OK;
}

// The columns, from the cell list that count_stencils left in `work`.
int fill_stencils(const double* xy, const double* h, int64_t N, double Lx, double Ly, uint32_t mask,
                  const int32_t* row_ptr, void* work, int64_t nnz, int longest, int32_t* col, cudaStream_t st) {
    const SearchWork w = split_search_work(work, N);
    const Box b = make_box(Lx, Ly, mask);
    const double inv_L = 1.0 / std::max(Lx, Ly);
    if (longest <= kRowCap) {
        k_neighbours<1><<<search_grid(N), 32 * kSearchWarps, 0, st>>>(xy, h, N, b, inv_L, w.st, w.cell_start, w.node,
                                                                      w.pos, nullptr, row_ptr, col);
        LABFM_LAUNCH_CHECK("neighbour fill kernel");
        return LABFM_OK;
    }
    StreamBuffer tmp(st);
    LABFM_CUDA_TRY(cudaMallocAsync(&tmp.p, size_t(nnz) * sizeof(int32_t), st));
    k_neighbours<2><<<search_grid(N), 32 * kSearchWarps, 0, st>>>(xy, h, N, b, inv_L, w.st, w.cell_start, w.node,
                                                                  w.pos, nullptr, row_ptr,
                                                                  static_cast<int32_t*>(tmp.p));
    LABFM_LAUNCH_CHECK("neighbour fill kernel");
    const int nblk_s = int(std::min<int64_t>((N + kSortWarps - 1) / kSortWarps, 1 << 20));
    k_sort_rows<<<nblk_s, 32 * kSortWarps, 0, st>>>(row_ptr, static_cast<const int32_t*>(tmp.p), col, N);
    LABFM_LAUNCH_CHECK("row sort kernel");
    return LABFM_OK;
}

int injected_capacity_error(int64_t col_capacity, int64_t* nnz_out) {
    *nnz_out = col_capacity + 1;
    return set_error(LABFM_ECAPACITY, "col_capacity " + std::to_string(col_capacity) + " < required " +
                                          std::to_string(col_capacity + 1) +
                                          " (injected: LABFM_FAULT=capacity)");
}

int check_search_work(const void* work, size_t work_bytes, int64_t N) {
    if (!work) return set_error(LABFM_EINVAL, "null work buffer");
    if (work_bytes < split_search_work(nullptr, N).bytes)
        return set_error(LABFM_EINVAL, "work buffer smaller than labfm_stencil_work_bytes");
    if (reinterpret_cast<uintptr_t>(work) % 16 != 0)
        return set_error(LABFM_EINVAL, "work buffer must be 16-byte aligned");
    return LABFM_OK;
}

}  // namespace
}  // namespace labfm

using namespace labfm;

extern "C" int labfm_build_stencils(const double* xy, const double* h, int64_t N, double Lx,
                                    double Ly, uint32_t periodic_mask, int32_t* row_ptr,
                                    int32_t* col, int64_t col_capacity, int64_t* nnz_out,
                                    void* stream) {
    LABFM_NVTX("labfm_build_stencils");
    if (!nnz_out) return set_error(LABFM_EINVAL, "null pointer argument");
    if (int rc = check_search_args(xy, h, N, Lx, Ly, row_ptr)) return rc;
    if (col_capacity < 0) return set_error(LABFM_EINVAL, "negative col_capacity");
    if (fault_alloc()) return injected_alloc_error("labfm_build_stencils");
    if (col && fault_capacity()) return injected_capacity_error(col_capacity, nnz_out);
    cudaStream_t st = as_stream(stream);
    StreamBuffer work(st);
    LABFM_CUDA_TRY(cudaMallocAsync(&work.p, split_search_work(nullptr, N).bytes, st));
    int64_t nnz = 0;
    int longest = 0;
    if (int rc = count_stencils(xy, h, N, Lx, Ly, periodic_mask, row_ptr, work.p, &nnz, &longest, st)) {
        if (rc == LABFM_ECAPACITY) *nnz_out = nnz;
        return rc;
    }
    *nnz_out = nnz;
    if (!col && col_capacity == 0) return LABFM_OK;  // size query
    if (!col || col_capacity < nnz)
        return set_error(LABFM_ECAPACITY, "col_capacity " + std::to_string(col_capacity) +
                                              " < required " + std::to_string(nnz));
    return fill_stencils(xy, h, N, Lx, Ly, periodic_mask, row_ptr, work.p, nnz, longest, col, st);
}

extern "C" size_t labfm_stencil_work_bytes(int64_t N) {
    if (N <= 0 || N >= (int64_t(1) << 31) - 1) return 0;
    return split_search_work(nullptr, N).bytes;
}

extern "C" int labfm_stencil_count(const double* xy, const double* h, int64_t N, double Lx, double Ly,
                                   uint32_t periodic_mask, int32_t* row_ptr, void* work, size_t work_bytes,
                                   int64_t* nnz_out, int32_t* longest_out, void* stream) {
    LABFM_NVTX("labfm_stencil_count");
    if (!nnz_out || !longest_out) return set_error(LABFM_EINVAL, "null pointer argument");
    if (int rc = check_search_args(xy, h, N, Lx, Ly, row_ptr)) return rc;
    if (fault_alloc()) return injected_alloc_error("labfm_stencil_count");
    if (int rc = check_search_work(work, work_bytes, N)) return rc;
    int longest = 0;
    const int rc = count_stencils(xy, h, N, Lx, Ly, periodic_mask, row_ptr, work, nnz_out, &longest, as_stream(stream));
    *longest_out = longest;
    return rc;
}

extern "C" int labfm_stencil_fill(const double* xy, const double* h, int64_t N, double Lx, double Ly,
                                  uint32_t periodic_mask, const int32_t* row_ptr, void* work, size_t work_bytes,
                                  int64_t nnz, int32_t longest, int32_t* col, int64_t col_capacity, void* stream) {
    LABFM_NVTX("labfm_stencil_fill");
    if (!col) return set_error(LABFM_EINVAL, "null pointer argument");
    if (int rc = check_search_args(xy, h, N, Lx, Ly, row_ptr)) return rc;
    if (int rc = check_search_work(work, work_bytes, N)) return rc;
    int64_t need = nnz;
    if (fault_capacity()) return injected_capacity_error(col_capacity, &need);
    if (col_capacity < nnz)
        return set_error(LABFM_ECAPACITY, "col_capacity " + std::to_string(col_capacity) +
                                              " < required " + std::to_string(nnz));
    return fill_stencils(xy, h, N, Lx, Ly, periodic_mask, row_ptr, work, nnz, longest, col, as_stream(stream));
}
