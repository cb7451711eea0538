// FP64 gathers in fixed point on the integer pipe.
//
// GB300 runs 2 FP64 lanes a clock and an SM but 64 lanes of 32 x 32 + 64-bit integer
// multiply-add (measured: 2.05 DFMA, 65 IMAD.WIDE), so the sums
// sum_j w_ji (phi_j - phi_i) of an FP64 plan, 12 multiply-adds and 3 subtractions per
// stencil entry, are bound by the FP64 pipe at 0.2 of the memory rate.  Here only the
// differences d = phi_j - phi_i are taken in FP64 (as before, rounded once); the products
// and sums run on integers:
//
//   weights:  w_ji 2^-s_j ~ (w1 2^28 + w0) 2^(E_w - 56), rounded, 0 <= w0 < 2^28,
//     E_w per row and operator;
//   differences:  |d| 2^s_j ~ (d1 2^28 + d0) 2^(E_d - 57), truncated, |d0| <= 2^27,
//     E_d per row and field, raised as larger differences turn up;
//   sum_j w_ji d_j ~ 2^(E_w + E_d - 113 + 28) (2^28 sum w1 d1 + sum (w1 d0 + w0 d1)),
//     two exact 64-bit sums; w0 d0 (below 2^-57 of the bounds, and of either sign) is dropped.
//
// The plan keeps the FP64 weights themselves, bit for bit, in the form that gives these
// digits with five instructions (weight_word): their 53 bits and the shift that aligns
// them to E_w.  The FP64 fallback and the adjoint read them back exactly.
//
// The shift s_j (0 to 15, four bits of the column word) is the same for an entry's weights
// and its difference and cancels.  It is the entry's size: that of its largest weight, against
// the row's largest of the same operator.  So the weights of all entries come to the same
// scale, and a difference counts with the weight that it meets: a large one at the edge of the
// stencil, where the weights are small, takes no bits from the others.
//
// The error of such a sum over n entries is at most (24 + n) 2^-56 2^(E_w + E_d): relative
// to the bounds, where FP64's is relative to sum |w d|.  So the lanes add up the leading bits
// of |w1| |d1| (four entries an instruction) as they go, and a row where that lower bound of
// sum |w d| is below 1/16 of 2^(E_w + E_d) for any operator and field is summed in FP64
// instead.  What is left is within (24 + n) 2^-52 sum |w d| whatever the fields; FP64's own a
// priori bound is n 2^-53 sum |w d|.  Against exact sums, in units of 2^-53 sum |w d|, over
// 3,840 nodes of orders 4, 6, 8 and 10, the operators x, y and xy, FP64 kernels in brackets:
// smooth fields 0.05-0.19 on average and 1.2 at most (0.21-0.40, 2.1), white noise 0.12-0.25
// and 2.3 (0.35-0.47, 3.5), pulses of 4 and 8 spacings 0.05-0.19 and 1.5 (0.20-0.42, 3.0),
// fronts, impulses, log-normal values of sigma 2 and 5, small pulses and rounding noise on a
// uniform stream 0.05-0.73 and 6.9 (0.10-0.99, 7.0).  In no class was the mean above FP64's by
// more than 1.4 %, nor the largest by more than a quarter.  Smooth fields and noise pass on all
// rows, pulses on nine tenths and more, fronts on half.  With shifts of 0 to 3 and 1/8, pulses
// had passed on a fifth, and the Lamb-Oseen vortex, whose tails they are, on a fifth of its
// rows.  A row that fails costs as much again as FP64 kernels would.  Keeping rows whose
// differences are exact in the high digit (rounding noise) in fixed point gave errors of up to
// 10^5.  The sizes take the right-hand side of 262,144 nodes of order 8 from 403 to 434 us (490
// as a high product of every entry).
//
// No overflow: E_w is raised until sum_j |w_ji| 2^-s_j <= 32 2^E_w, so |sum w1 d1| <=
// 2^(5 + 28 + 29) over a whole row; |sum (w1 d0 + w0 d1)| <= 2^60 + n 2^57 over n entries,
// whose carries a lane moves up after every 32.  Rows with a weight that is not finite,
// beyond 2^+-400 at their largest, subnormal or below 2^-500 of their row's largest hold
// plain FP64 weights and are summed in FP64 (kRawRow), each by itself, so that a failed node
// changes no other row; so are rows where an operator uses less than half the entries that
// another does, beside boundaries, most of which would fail the span test.  A row whose differences are not finite or beyond 2^460 is summed in
// FP64 too, so that infinities and NaN come out as they would, and one whose differences of
// a field, with their shifts, all lie below 2^-498 without being all zero.  Beside larger ones, differences below
// 2^-1022 count as zero.  Plans of 2^28 nodes or more need the four bits for their columns:
// there every s_j is 0.
#pragma once

#include "gather.cuh"

namespace labfm {
namespace {

// The column word: the column, and s_j in the four bits above it.
__host__ __device__ __forceinline__ uint32_t col_mask(int64_t N) { return N < (int64_t(1) << 28) ? 0x0fffffffu : 0x7fffffffu; }
constexpr int kMostShift = 15;
constexpr int kRawRow = 64;  // with the zero operators' bits in wexp[8 i + 6]: the row holds FP64 weights
constexpr int kFixedWarps = 2;  // warps a block
constexpr int kFloorT = 80 << 20;           // T of a field until a difference above it turns up
constexpr int kLeastT = 524 << 20;          // smallest bound of the fixed-point sums
constexpr uint32_t kMostT = 1500u << 20;
constexpr uint32_t kLeastSize = 32;         // 1/16 of the bounds' product, in units of 2^-9 of it

__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// Eight 32-bit words of the record stream, past the L1, which keeps the gathered states
// (the 262,144-node order-8 stage 384 -> 369 us against evict-first loads).
__device__ __forceinline__ void ld8i(const void* p, int (&v)[8]) {
    asm("ld.global.nc.L1::no_allocate.L2::256B.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "l"(p));
}

// Exponent field of d, in place (biased, times 2^20).
__device__ __forceinline__ int exponent20(double d) { return __double2hiint(d) & 0x7ff00000; }

// Digits of d for t = T - exponent20(d) - s 2^20 >= 0, T = (E_d - 1) 2^20 (biased): the 53
// significant bits, leading bit at 60, shifted down by t / 2^20; shifts of 64 and more
// give zero, so a zero difference (exponent field 0) does.  The high digit is rounded, the
// low one signed, so that the dropped products w0 d0 have no mean.
__device__ __forceinline__ void digits(double d, int t, int& d1, int& d0, uint32_t& size) {
    const int h = __double2hiint(d), l = __double2loint(d);
    const uint32_t sh = uint32_t(t) >> 20;
    const uint32_t x1 = (__funnelshift_l(uint32_t(l), uint32_t(h), 8) & 0x1fffffffu) | 0x10000000u;
    const uint64_t x = (uint64_t(x1) << 32) | (uint32_t(l) << 8);
    uint32_t top;
    uint64_t low;
    asm("shr.u32 %0, %1, %2;" : "=r"(top) : "r"(x1), "r"(sh));
    asm("shr.u64 %0, %1, %2;" : "=l"(low) : "l"(x), "r"(sh));
    const int sign = (h >> 31) | 1;
    size = top + (uint32_t(low) >> 31);  // |d1|
    d1 = int(size) * sign;
    d0 = (int(uint32_t(low)) >> 4) * sign;
}

// A weight w = M 2^(ex - 52), |M| in [2^52, 2^53), in a row and operator of bound E and at
// an entry of shift s.  With the alignment t = 1 + E + s - ex (2 for the largest weights,
// kMostAlign at most) in the low nine bits of the word and M above them, the digits are
// bits t + 32 and up and bits t + 4 to t + 31 of the word: what lies below is rounded by
// adding its half beforehand, at bit t + 3 (nothing is lost by t < 6).  From kNoDigits on
// the digits are zero: the word is M + 2^53, not negative, which the shifts clear.
constexpr int kNoDigits = 59;
constexpr int kMostAlign = 511;
__device__ __forceinline__ long long weight_word(double w, int E, int s) {
    const long long b = __double_as_longlong(w);
    if ((b << 1) == 0) return 0;
    const int t = 1 + E + s - (int((b >> 52) & 0x7ff) - 1023);
    const long long mag = (b & 0xfffffffffffffll) | (1ll << 52);
    const long long M = b < 0 ? -mag : mag;
    if (t >= kNoDigits) return ((M + (1ll << 53)) << 9) | t;
    return (M * 512 + (t >= 6 ? 1ll << (t + 3) : 0)) | t;
}
__device__ __forceinline__ double word_weight(long long word, int E, int s) {
    const int t = int(word) & 511;
    const long long M = t < kNoDigits ? (word - (t >= 6 ? 1ll << (t + 3) : 0)) >> 9 : (word >> 9) - (1ll << 53);
    if (M == 0) return 0.0;
    const long long mag = M < 0 ? -M : M;
    return __longlong_as_double((M < 0 ? 1ll << 63 : 0) | ((long long)(1 + E + s - t + 1023) << 52) |
                                (mag & 0xfffffffffffffll));
}
// The digits of the word (lo, hi).
__device__ __forceinline__ void weight_digits(int lo, int hi, int& w1, int& w0) {
    const int t = lo & 511;
    long long low;
    asm("shr.s32 %0, %1, %2;" : "=r"(w1) : "r"(hi), "r"(t));
    asm("shr.s64 %0, %1, %2;" : "=l"(low) : "l"((static_cast<long long>(hi) << 32) | uint32_t(lo)), "r"(t));
    w0 = int(uint32_t(low) >> 4);
}

// s += a b, 32 x 32 + 64 bits.  As a carry pair, which the assembler makes one wide
// multiply-add: given as a plain 64-bit sum it regroups the sums of a chunk into products
// and additions (half as many instructions again, and spills).
__device__ __forceinline__ void mad_wide(long long& s, int a, int b) {
    asm("{\n\t.reg .u32 lo, hi;\n\t"
        "mov.b64 {lo, hi}, %0;\n\t"
        "mad.lo.cc.s32 lo, %1, %2, lo;\n\t"
        "madc.hi.s32 hi, %1, %2, hi;\n\t"
        "mov.b64 %0, {lo, hi};\n\t}"
        : "+l"(s)
        : "r"(a), "r"(b));
}
__device__ __forceinline__ void mac(long long& hi, long long& mid, int w1, int w0, int d1, int d0) {
    mad_wide(hi, w1, d1);
    mad_wide(mid, w1, d0);
    mad_wide(mid, w0, d1);
}

// Bytes of x and y (prmt: 0-3 of x, 4-7 of y, + 8 its sign throughout).
template <int SEL>
__device__ __forceinline__ uint32_t bytes_of(uint32_t x, uint32_t y) {
    uint32_t v;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(v) : "r"(x), "r"(y), "n"(SEL));
    return v;
}
// The leading bytes of four digits: 0 to 16 of a weight's magnitude (|w1| <= 2^28, rounded
// down), 0 to 32 of a difference's.
__device__ __forceinline__ uint32_t leading(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    return bytes_of<0x5410>(bytes_of<0x73>(a, b), bytes_of<0x73>(c, d));
}
__device__ __forceinline__ uint32_t magnitudes(uint32_t v) { return v ^ bytes_of<0xba98>(v, v); }

// Non-zero when d is (-0 is zero).
__device__ __forceinline__ uint32_t not_zero(double d) {
    return (uint32_t(__double2hiint(d)) << 1) | uint32_t(__double2loint(d));
}

// Whether a row needs FP64 for the sums of a field with bound T over K operators, the first
// of them `first`: its differences lie below the range of the fixed-point sums without being
// all zero, or span too many bits for an operator that is not zero throughout the row.
template <int K>
__device__ __forceinline__ bool out_of_range(int T, uint32_t seen, const uint32_t* size, int first, int zero_ops) {
    if (T == kFloorT) return seen != 0;
    bool out = T < kLeastT;
#pragma unroll
    for (int k = 0; k < K; ++k) out |= size[k] < kLeastSize && !(zero_ops >> (first + k) & 1);
    return out;
}

template <int STEP, int G>
__device__ __forceinline__ uint32_t group_add(uint32_t v) {
#pragma unroll
    for (int off = G / 2; off >= STEP; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Largest v over the lanes of the group that lie a multiple of STEP apart.
template <int STEP, int G>
__device__ __forceinline__ uint32_t group_max(uint32_t v) {
#pragma unroll
    for (int off = G / 2; off >= STEP; off >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, off));
    return v;
}

// Raises the bound T of one field for the whole lane group when the chunk's largest
// exponent m (over the group) exceeds it (and only then: other rows of the warp do not
// change a row's sums), shifting the K sums taken so far.
template <int K>
__device__ __forceinline__ void raise_bound(uint32_t m, int& T, long long* hi, long long* mid, uint32_t* size,
                                            bool& cold) {
    if (m <= uint32_t(T)) return;
    if (m >= kMostT) {
        cold = true;
        return;
    }
    const int by = min((int(m) - T) >> 20, 63);
    T = int(m);
#pragma unroll
    for (int k = 0; k < K; ++k) {
        hi[k] >>= by;
        mid[k] >>= by;
        size[k] >>= min(by, 31);
    }
}

// Moves the carries of the low sums up, so that a lane can take rows of any length: due
// every kFold chunks (32 entries).
constexpr int kFold = 8;
template <int K>
__device__ __forceinline__ void fold(long long (&hi)[K], long long (&mid)[K]) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
        hi[k] += mid[k] >> 28;
        mid[k] &= 0xfffffffll;
    }
}

__device__ __forceinline__ void load_cols(const double* w, int64_t off, uint32_t (&c)[4]) {
    const int4 v = ld_na(reinterpret_cast<const int4*>(reinterpret_cast<const char*>(w) + off));
    c[0] = uint32_t(v.x);
    c[1] = uint32_t(v.y);
    c[2] = uint32_t(v.z);
    c[3] = uint32_t(v.w);
}

// States that the launch before may write, packed or as three arrays.  Plain loads: read-only
// ones (__ldg) the compiler may move above the wait for that launch.
struct State {
    const Packed<double>* p;
    __device__ __forceinline__ void get(int j, double& x, double& y, double& z) const { unpack_rw(p, j, x, y, z); }
};
struct Fields {
    const double *a, *u, *v;
    __device__ __forceinline__ void get(int j, double& x, double& y, double& z) const {
        x = a[j];
        y = u[j];
        z = v[j];
    }
};

// Where the values of one field lie: node j's at p[j * stride].
struct Column {
    const double* p;
    int stride;
    __device__ __forceinline__ double operator[](int j) const { return p[int64_t(j) * stride]; }
};
__device__ __forceinline__ Column column(const Fields& f, int k) { return {k == 0 ? f.a : (k == 1 ? f.u : f.v), 1}; }
__device__ __forceinline__ Column column(const State& f, int k) {
    return {reinterpret_cast<const double*>(f.p) + k, 4};
}

// The filter's sums of one row over the lanes of its group, kappa w^hyp on three fields.
// hi, mid: this lane's sums; T: the three bounds; zero_ops: the operators (bits) that are zero
// throughout the row; cold (the same in the whole group): the row needs FP64.  Every lane of
// the warp takes the same number of iterations (a lane without a chunk adds zeros).
template <int G, class F>
__device__ __forceinline__ void filter_row(const PlanView<double>& P, const F& fld, int i, int e0, int e1, int gl,
                                           int zero_ops, long long (&hi)[3], long long (&mid)[3], int (&T)[3],
                                           bool& cold) {
    const int trips = __reduce_max_sync(0xffffffffu, (e1 - e0 + 4 * G - 1) / (4 * G));
    const uint32_t mask = col_mask(P.N);
    double own[3];
    fld.get(i, own[0], own[1], own[2]);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        hi[f] = mid[f] = 0;
        T[f] = kFloorT;
    }
    uint32_t seen[3] = {0, 0, 0};  // a difference other than zero
    uint32_t size[3] = {0, 0, 0};  // sum |w1 d1|
    cold = false;
    int e = e0 + 4 * gl;
#pragma unroll 1
    for (int it = 0; it < trips; ++it, e += 4 * G) {
        const bool on = e < e1;
        const int64_t c = on ? e >> 2 : 0;  // past the row: any chunk, with the node's own (zero) differences
        uint32_t cj[4];
        load_cols(P.wf, Rec<double>::fcol(c), cj);
        int w[8];
        ld8i(reinterpret_cast<const char*>(P.wf) + Rec<double>::fw(c), w);
        double d[3][4];
        int s20[4], t[3][4], low = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t cw = on ? cj[k] : uint32_t(i);
            double v[3];
            fld.get(int(cw & mask), v[0], v[1], v[2]);
            s20[k] = int((cw & ~mask) >> 8);
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                d[f][k] = v[f] - own[f];
                seen[f] |= not_zero(d[f][k]);
                t[f][k] = T[f] - exponent20(d[f][k]) - s20[k];
                low |= t[f][k];
            }
        }
        if (__any_sync(0xffffffffu, low < 0)) {
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                uint32_t m = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) m = max(m, uint32_t(exponent20(d[f][k])) + uint32_t(s20[k]));
                raise_bound<1>(group_max<1, G>(m), T[f], hi + f, mid + f, size + f, cold);
#pragma unroll
                for (int k = 0; k < 4; ++k) t[f][k] = T[f] - exponent20(d[f][k]) - s20[k];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) weight_digits(w[2 * k], w[2 * k + 1], w[2 * k], w[2 * k + 1]);
        const uint32_t wm = magnitudes(leading(w[0], w[2], w[4], w[6]));
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            uint32_t u1[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                int d1, d0;
                digits(d[f][k], t[f][k], d1, d0, u1[k]);
                mac(hi[f], mid[f], w[2 * k], w[2 * k + 1], d1, d0);
            }
            size[f] = __dp4a(wm, leading(u1[0], u1[1], u1[2], u1[3]), size[f]);
        }
        if (it % kFold == kFold - 1) fold(hi, mid);
    }
    fold(hi, mid);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        const uint32_t all = group_add<1, G>(size[f]);
        cold |= out_of_range<1>(T[f], seen[f], &all, 5, zero_ops);
    }
    cold = group_max<1, G>(uint32_t(cold)) != 0;
}

// The twelve derivative sums of one row over the lanes of its group, two lanes to a chunk:
// the even one sums x, y, xx, xy, yy of u, the odd one of v, and each x and y of ln rho
// over two of the chunk's four entries.  One lane for all twelve sums needed 128 registers
// (16 warps an SM) and waited for its gathers.  AHEAD: the next chunk's columns and gathers
// are loaded before the current chunk's sums (16 more registers; a launch that fills the chip
// gains nothing).  hi, mid: [ln rho x, y, then five]; T: bounds of ln rho and of the lane's
// own field.
template <int G, bool AHEAD, class F>
__device__ __forceinline__ void rhs_row(const PlanView<double>& P, const F& fld, int i, int e0, int e1, int gl,
                                        int zero_ops, long long (&hi)[7], long long (&mid)[7], int (&T)[2],
                                        bool& cold) {
    const int trips = __reduce_max_sync(0xffffffffu, (e1 - e0 + 2 * G - 1) / (2 * G));
    const uint32_t mask = col_mask(P.N);
    const bool odd = gl & 1;
    const Column fa = column(fld, 0), ff = column(fld, odd ? 2 : 1);
    const double oa = fa[i], of = ff[i];
#pragma unroll
    for (int k = 0; k < 7; ++k) hi[k] = mid[k] = 0;
    uint32_t size[7] = {0, 0, 0, 0, 0, 0, 0};  // sum |w1 d1|
    T[0] = T[1] = kFloorT;
    uint32_t seen[2] = {0, 0};  // a difference other than zero
    cold = false;
    const char* rec = reinterpret_cast<const char*>(P.w);
    int e = e0 + 4 * (gl >> 1);
    // columns of the chunk at entry q; past the row the node itself (zero differences)
    auto columns = [&](int q, uint32_t (&cj)[4]) {
        load_cols(P.w, Rec<double>::col(q < e1 ? q >> 2 : 0), cj);
#pragma unroll
        for (int k = 0; k < 4; ++k) cj[k] = q < e1 ? cj[k] : uint32_t(i);
    };
    auto values = [&](const uint32_t (&cj)[4], double (&g)[6]) {
#pragma unroll
        for (int k = 0; k < 4; ++k) g[k] = ff[int(cj[k] & mask)];
        g[4] = fa[int((odd ? cj[2] : cj[0]) & mask)];
        g[5] = fa[int((odd ? cj[3] : cj[1]) & mask)];
    };
    uint32_t cj[4];
    double g[6];
    if (AHEAD) {
        columns(e, cj);
        values(cj, g);
    }
#pragma unroll 1
    for (int it = 0; it < trips; ++it, e += 2 * G) {
        const int64_t c = e < e1 ? e >> 2 : 0;
        // the chunks of two iterations on into L2, six lines a chunk among its lanes (444 -> 385 us)
        if (e + 4 * G < e1) {
            const char* ahead = rec + Rec<double>::col((e + 4 * G) >> 2);
            constexpr int NR = G < 8 ? G : 8;
#pragma unroll
            for (int l = 0; l < 6; l += NR)
                if (l + (gl & (NR - 1)) < 6)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(ahead + (l + (gl & (NR - 1))) * 128));
        }
        if (!AHEAD) {
            columns(e, cj);
            values(cj, g);
        }
        double d[4], da[2];
        int t[4], ta[2], low = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            d[k] = g[k] - of;
            seen[1] |= not_zero(d[k]);
            t[k] = T[1] - exponent20(d[k]) - int((cj[k] & ~mask) >> 8);
            low |= t[k];
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            da[k] = g[4 + k] - oa;
            seen[0] |= not_zero(da[k]);
            ta[k] = T[0] - exponent20(da[k]) - int(((odd ? cj[k + 2] : cj[k]) & ~mask) >> 8);
            low |= ta[k];
        }
        if (AHEAD) {
            columns(e + 2 * G, cj);
            values(cj, g);
        }
        if (__any_sync(0xffffffffu, low < 0)) {
            const int T0 = T[0], T1 = T[1];
            uint32_t m = 0, ma = 0;  // exponents with their shifts: T - t
#pragma unroll
            for (int k = 0; k < 4; ++k) m = max(m, uint32_t(T1) - uint32_t(t[k]));
#pragma unroll
            for (int k = 0; k < 2; ++k) ma = max(ma, uint32_t(T0) - uint32_t(ta[k]));
            raise_bound<2>(group_max<1, G>(ma), T[0], hi, mid, size, cold);
            raise_bound<5>(group_max<2, G>(m), T[1], hi + 2, mid + 2, size + 2, cold);
#pragma unroll
            for (int k = 0; k < 4; ++k) t[k] += T[1] - T1;
#pragma unroll
            for (int k = 0; k < 2; ++k) ta[k] += T[0] - T0;
        }
        // digits of the differences (entries 0, 2, 1, 3), and their leading bytes for the sizes
        int d1[4], d0[4], a1[2], a0[2];
        uint32_t um, am;
        {
            uint32_t u[4], v[2];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int q = 2 * (k & 1) + (k >> 1);
                digits(d[q], t[q], d1[k], d0[k], u[k]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) digits(da[k], ta[k], a1[k], a0[k], v[k]);
            um = leading(u[0], u[1], u[2], u[3]);
            am = bytes_of<0x7733>(v[0], v[1]) & (odd ? 0xff00ff00u : 0x00ff00ffu);
        }
        uint32_t wm[5];
#pragma unroll
        for (int k = 0; k < 2; ++k) {  // entries k and k + 2
            int w[2][8];
            ld8i(rec + Rec<double>::w(c, k), w[0]);
            ld8i(rec + Rec<double>::w(c, k + 2), w[1]);
#pragma unroll
            for (int o = 0; o < 4; ++o) {
#pragma unroll
                for (int z = 0; z < 2; ++z) {
                    weight_digits(w[z][2 * o], w[z][2 * o + 1], w[z][2 * o], w[z][2 * o + 1]);
                    mac(hi[2 + o], mid[2 + o], w[z][2 * o], w[z][2 * o + 1], d1[2 * k + z], d0[2 * k + z]);
                }
                const uint32_t m = bytes_of<0x73>(w[0][2 * o], w[1][2 * o]);
                wm[o] = k == 0 ? m : bytes_of<0x5410>(wm[o], m);
            }
#pragma unroll
            for (int o = 0; o < 2; ++o)
                mac(hi[o], mid[o], odd ? w[1][2 * o] : w[0][2 * o], odd ? w[1][2 * o + 1] : w[0][2 * o + 1], a1[k], a0[k]);
        }
        {
            int w[8];  // the fifth operator's words of the four entries
            ld8i(rec + Rec<double>::w(c, 4), w);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int q = 2 * (2 * (k & 1) + (k >> 1));
                weight_digits(w[q], w[q + 1], w[q], w[q + 1]);
                mac(hi[6], mid[6], w[q], w[q + 1], d1[k], d0[k]);
            }
            wm[4] = leading(w[0], w[4], w[2], w[6]);
        }
#pragma unroll
        for (int o = 0; o < 5; ++o) {
            wm[o] = magnitudes(wm[o]);
            size[2 + o] = __dp4a(wm[o], um, size[2 + o]);
            if (o < 2) size[o] = __dp4a(wm[o], am, size[o]);
        }
        if (it % kFold == kFold - 1) fold(hi, mid);
    }
    fold(hi, mid);
#pragma unroll
    for (int k = 0; k < 7; ++k) size[k] = k < 2 ? group_add<1, G>(size[k]) : group_add<2, G>(size[k]);
    cold |= out_of_range<2>(T[0], seen[0], size, 0, zero_ops);
    cold |= out_of_range<5>(T[1], seen[1], size + 2, 0, zero_ops);
    cold = group_max<1, G>(uint32_t(cold)) != 0;
}

// Byte offset of the weight word of operator o (5: the filter's kappa w^hyp) at entry e
// in the RHS (o < 5) or filter records.  The five 32-byte segments of a chunk hold its four
// entries' first four operators, entry by entry, then the fifth operator of all four, so
// that a lane needs one entry's words at a time (operator by operator, as the FP64 records
// are, the kernel needed 164 registers).
__host__ __device__ __forceinline__ int64_t fixed_at(int64_t e, int o) {
    if (o == 5) return Rec<double>::fw(e >> 2) + 8 * (e & 3);
    return o < 4 ? Rec<double>::w(e >> 2, int(e & 3)) + 8 * o : Rec<double>::w(e >> 2, 4) + 8 * (e & 3);
}

__device__ __forceinline__ uint32_t fixed_col_word(const PlanView<double>& P, int e, bool filter) {
    const char* at = filter ? reinterpret_cast<const char*>(P.wf) + Rec<double>::fcol_e(e)
                            : reinterpret_cast<const char*>(P.w) + Rec<double>::col_e(e);
    return *reinterpret_cast<const uint32_t*>(at);
}

// Weight of operator o at entry e of row i of an F64 plan.
__device__ __forceinline__ double fixed_weight(const PlanView<double>& P, int i, int e, int o) {
    const char* rec = o == 5 ? reinterpret_cast<const char*>(P.wf) : reinterpret_cast<const char*>(P.w);
    const long long word = *reinterpret_cast<const long long*>(rec + fixed_at(e, o));
    if (P.wexp[int64_t(i) * 8 + 6] & kRawRow) return __longlong_as_double(word);
    return word_weight(word, P.wexp[int64_t(i) * 8 + o], int((fixed_col_word(P, e, o == 5) & ~col_mask(P.N)) >> 28));
}

// The rows that need FP64, by 8 lanes each, four at a time (whatever the lanes of the
// fixed-point sums and however many rows of the warp need it: a row's sums are the same
// beside any others).  slots: the rows, as bits (fixed_nodes, R of them a pass);
// out[k][slot]: the sums' bit patterns.  Such rows come in clusters (all 16 of a warp, beside
// a boundary), and a warp's chain through them is what the launch waits for: the next entry's
// column, values and words are in flight while the current one's products are summed
// (Lamb-Oseen steps of 40,000 nodes, by an entry at a time 421 us, a chunk of four 423, one
// ahead 392).  With 16 and 32 lanes a row, whose sums take more of the FP64 pipe, the step
// takes 445 and 580 us, with 4 as long as with 8 (391).
template <bool FILTER, int R, int K, class F>
__device__ __noinline__ void cold_rows(const int32_t* row_ptr, const char* rec, const int16_t* wexp, F fld,
                                       uint32_t mask, int64_t first, uint32_t slots, long long (*out)[32]) {
    constexpr int KA = FILTER ? 1 : 2, KV = FILTER ? 1 : 5, L = 8;
    const int lane = threadIdx.x & 31, gl = lane % L;
    auto column = [&](int e) {
        return *reinterpret_cast<const uint32_t*>(rec + (FILTER ? Rec<double>::fcol_e(e) : Rec<double>::col_e(e)));
    };
#pragma unroll 1
    while (slots) {
        uint32_t left = slots;
#pragma unroll 1
        for (int k = 0; k < lane / L; ++k) left &= left - 1;
        const int slot = __ffs(left) - 1;  // this group's row, or -1
        const int i = slot < 0 ? 0 : int(first + (slot / R) * (kFixedWarps * R) + slot % R);
        double sum[K];
#pragma unroll
        for (int k = 0; k < K; ++k) sum[k] = 0.0;
        double ai, ui, vi;
        fld.get(i, ai, ui, vi);
        const int4 ev = *reinterpret_cast<const int4*>(wexp + int64_t(i) * 8);
        const int E[6] = {int16_t(ev.x), ev.x >> 16, int16_t(ev.y), ev.y >> 16, int16_t(ev.z), ev.z >> 16};
        const bool raw = ev.w & kRawRow;
        int e = row_ptr[i] + gl;
        const int e1 = slot < 0 ? 0 : row_ptr[i + 1];
        // the next entry's column, values and words are loaded before this one's products
        uint32_t cw = 0, cn = 0;
        double a = ai, u = ui, v = vi;
        long long word[KV], more[KV];
        auto words = [&](int q, long long (&to)[KV]) {
#pragma unroll
            for (int o = 0; o < KV; ++o) to[o] = *reinterpret_cast<const long long*>(rec + fixed_at(q, FILTER ? 5 : o));
        };
        if (e < e1) {
            cw = column(e);
            words(e, word);
            if (e + L < e1) cn = column(e + L);
            fld.get(int(cw & mask), a, u, v);
        }
#pragma unroll 1
        for (; e < e1; e += L) {
            double an = ai, un = ui, vn = vi;
            uint32_t cm = 0;
            if (e + L < e1) {
                words(e + L, more);
                fld.get(int(cn & mask), an, un, vn);
                if (e + 2 * L < e1) cm = column(e + 2 * L);
            }
            const int s = int((cw & ~mask) >> 28);
            a -= ai;
            u -= ui;
            v -= vi;
#pragma unroll
            for (int o = 0; o < KV; ++o) {
                const double w = raw ? __longlong_as_double(word[o]) : word_weight(word[o], E[FILTER ? 5 : o], s);
                if (o < KA) sum[o] = fma(a, w, sum[o]);
                sum[KA + o] = fma(u, w, sum[KA + o]);
                sum[KA + KV + o] = fma(v, w, sum[KA + KV + o]);
                word[o] = more[o];
            }
            cw = cn;
            cn = cm;
            a = an;
            u = un;
            v = vn;
        }
#pragma unroll 1
        for (int off = L / 2; off > 0; off >>= 1) {
#pragma unroll
            for (int k = 0; k < K; ++k) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], off);
        }
        if (slot >= 0 && gl == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) out[k][slot] = __double_as_longlong(sum[k]);
        }
#pragma unroll 1
        for (int k = 0; k < 32 / L; ++k) slots &= slots - 1;
    }
    __syncwarp();
}

// The sums of the block's nodes, epi(node, a, u, v, sums) for each.  A pass takes 32/G nodes
// a warp and kFixedWarps warps' worth of consecutive nodes a block; after the last pass
// lane l of a warp finishes one node of the warp's: the FP64 work after the sums (about 130
// instructions, which cost the pipe the same for one lane as for 32) runs on as many lanes
// as the warp has had nodes.
template <int G, bool FILTER, bool AHEAD, class F, class Epi>
__device__ __forceinline__ void fixed_nodes(const PlanView<double>& P, const F& fld, int passes, const Epi& epi) {
    constexpr int K = FILTER ? 3 : 12, R = 32 / G, LK = FILTER ? 3 : 7, LT = FILTER ? 3 : 2;
    __shared__ long long s_hi[kFixedWarps][K][32];
    __shared__ int s_lo[kFixedWarps][K][32];
    __shared__ int s_T[kFixedWarps][3][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gl = lane % G;
    const int64_t first = P.n_lo + int64_t(blockIdx.x) * passes * (kFixedWarps * R) + warp * R;
    uint32_t cold_slots = 0;  // of this warp's nodes, those to be summed in FP64
#pragma unroll 1
    for (int p = 0; p < passes; ++p) {
        const int64_t node = first + p * (kFixedWarps * R) + lane / G;
        if (node - lane / G >= P.n_hi) break;
        const int i = int(node < P.n_hi ? node : P.n_hi - 1);
        const int zero_ops = P.wexp[int64_t(i) * 8 + 6];
        const bool raw = node < P.n_hi && (zero_ops & kRawRow);
        const int e0 = P.row_ptr[i], e1 = node < P.n_hi && !raw ? P.row_ptr[i + 1] : e0;
        if (p == 0) pdl_wait();  // nothing before it is written by a launch
        long long hi[LK], lo[LK];
        int T[LT];
        bool cold;
        if constexpr (FILTER) filter_row<G>(P, fld, i, e0, e1, gl, zero_ops, hi, lo, T, cold);
        else rhs_row<G, AHEAD>(P, fld, i, e0, e1, gl, zero_ops, hi, lo, T, cold);
        // over the lanes that share a sum: all of them (filter, ln rho), or every second one
#pragma unroll
        for (int k = 0; k < LK; ++k) {
#pragma unroll
            for (int off = G / 2; off >= (FILTER || k < 2 ? 1 : 2); off >>= 1) {
                hi[k] += __shfl_xor_sync(0xffffffffu, hi[k], off);
                lo[k] += __shfl_xor_sync(0xffffffffu, int(lo[k]), off);
            }
        }
        const int slot = p * R + lane / G;
        if (FILTER ? gl == 0 : gl < 2) {
            const int k0 = FILTER ? 0 : (gl ? 7 : 2);  // this lane's own field
#pragma unroll
            for (int k = 0; k < LK; ++k) {
                if (!FILTER && k < 2 && gl) continue;
                const int at = FILTER || k < 2 ? k : k0 + k - 2;
                s_hi[warp][at][slot] = hi[k] + (lo[k] >> 28);
                s_lo[warp][at][slot] = int(lo[k]) & 0xfffffff;
            }
            if (FILTER) {
#pragma unroll
                for (int f = 0; f < LT; ++f) s_T[warp][f][slot] = T[f];
            } else {
                if (!gl) s_T[warp][0][slot] = T[0];
                s_T[warp][1 + gl][slot] = T[1];
            }
        }
        const uint32_t groups = __ballot_sync(0xffffffffu, (cold || raw) && gl == 0);
        if (groups)
            for (int n = 0; n < R; ++n)
                if (groups >> (n * G) & 1) cold_slots |= 1u << (p * R + n);
    }
    __syncwarp();
    if (cold_slots)
        cold_rows<FILTER, R, K>(P.row_ptr, reinterpret_cast<const char*>(FILTER ? P.wf : P.w), P.wexp, fld, col_mask(P.N),
                                first, cold_slots, s_hi[warp]);
    const int64_t node = first + (lane / R) * (kFixedWarps * R) + lane % R;
    const bool mine = lane < passes * R && node < P.n_hi;
    double sum[K];
    if (mine) {
        const bool cold = cold_slots >> lane & 1;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int f = FILTER ? k : (k < 2 ? 0 : (k < 7 ? 1 : 2));
            const int o = FILTER ? 5 : (k < 2 ? k : (k < 7 ? k - 2 : k - 7));
            // E_w + E_d - 113 + 28, E_d = T / 2^20 + 1 - 1023
            const double S = pow2(max(P.wexp[node * 8 + o] + (s_T[warp][f][lane] >> 20) - 1107, -1000));
            sum[k] = fma(double(s_hi[warp][k][lane]), S * 268435456.0, double(s_lo[warp][k][lane]) * S);
            if (cold) sum[k] = __longlong_as_double(s_hi[warp][k][lane]);
        }
    }
    if (mine) {
        double a, u, v;
        fld.get(int(node), a, u, v);
        epi(int(node), a, u, v, sum);
    }
}

}  // namespace
}  // namespace labfm
