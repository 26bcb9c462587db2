// k_dense_fx.cu -- dense gates on complex128 states in block fixed point on the
// integer multipliers.
//
// GB300 runs FP64 at 2 FMAs per SM and clock: a dense k-qubit gate needs
// 4 2^k of them per amplitude, 2 2^k clocks, against about 1.5 clocks for the
// 32 bytes an amplitude moves. The 32 x 32 -> 64 bit integer multiply-add runs
// more than an order of magnitude faster, so the product is formed exactly in
// integers: the reals of one group (2^k amplitudes) share an exponent E and are
// cut into limbs of L bits, the matrix entries share the exponent em, limb
// products are summed in 64-bit integers (no rounding, no overflow: the bounds
// are with the layouts below), and each sum is rounded once to a double.
//
// Three layouts (u = 2^-53, X a group's largest amplitude; dm: the bits by which the
// smallest nonzero entry's exponent lies below the largest's):
//   two limbs   k = 1, 2: 60 and 59 bits, 3 limb products per real product.
//   digits      k = 3 to 5: 61 and 62 bits, on the tensor cores.
//   three limbs k = 1 to 4: 84 bits, 6 limb products per real product (complex
//               products by three real ones, exact in integers).
// The first two hold an amplitude to a fixed share of X, so a sum that sees X only
// through a small entry is less accurate than one that sees it through a large one.
// Their ranges of dm are those in which the worst amplitude of adversarial groups (the
// smallest entries on the large amplitudes) has no larger an error, in u sum |m||x|,
// than a chain of FP64 multiply-adds on the same groups; worst measured here / chain:
//   k = 1, dm 5: 2.5 / 3.0   k = 2, dm 4: 3.7 / 4.8   (k = 2 at 5: 9.5 / 4.8)
//   k = 3, dm 7: 5.3 / 7.1   k = 4, dm 7: 8.9 / 9.9   k = 5, dm 8: 12.0 / 14.2
// Beyond that, up to 8 (k = 5: 11), the digits serve groups in which every row sees a
// large amplitude through a large entry, and (8; k = 5: 9) those whose reals, and then
// all products, they hold exactly. Three limbs: host and kernel check that entries (dm bits) and nonzero
// amplitudes (t bits) lie within t + dm <= 24 bits of their largest, which keeps the
// error of every term below u / 16 of it. Zeros are exact throughout.
//
// What is bounded is the error of an amplitude's modulus. A part far below its
// amplitude carries that error too, unless the matrix keeps the parts apart (below).
//
// A group outside these ranges (also infinities, NaN, values near the limits of
// the exponent) is computed in FP64 in the same kernel, with k_dense's sums in
// k_dense's order.
#include <algorithm>
#include <cmath>
#include <vector>

#include "k_common.cuh"
#include "sv_internal.h"

namespace svk {
namespace {

constexpr int kThreads = 256;
constexpr int kEMin = 300, kEMax = 1800;   // biased exponents of a group's largest real that stay far from the limits

__device__ __forceinline__ uint64_t shr64(uint64_t v, uint32_t s) {   // 0 for s >= 64
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ uint32_t shl32(uint32_t v, uint32_t s) {   // 0 for s >= 32
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }

// the normalised 64-bit magnitude v (top bit at 63 - n of the value before the
// shift) as a double of biased exponent be and the sign of s, rounded to nearest
__device__ __forceinline__ double pack(uint64_t v, int be, int s) {
    const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
    uint64_t m = ((uint64_t)(hi >> 11) << 32) | __funnelshift_r(lo, hi, 11);
    m += (lo >> 10) & 1u;
    const uint32_t h = (uint32_t)(m >> 32) + ((uint32_t)(be - 1) << 20);   // the implicit bit adds one
    return __hiloint2double((int)(h | ((uint32_t)s & 0x80000000u)), (int)(uint32_t)m);
}

// An integer r times 2^sc; the caller's sc keeps the exponent in range. (The hardware conversion
// takes one instruction where normalising by hand takes about twenty: 26-qubit
// one-qubit gate 0.425 -> 0.326 ms.)
__device__ __forceinline__ double scaled(double r, int sc) {
    const int hi = __double2hiint(r);
    return __hiloint2double(hi == 0 ? 0 : hi + (int)((uint32_t)sc << 20), __double2loint(r));
}

// mantissa of x with the implicit bit at bit 63
__device__ __forceinline__ uint64_t mant64(int hi, int lo) {
    return ((uint64_t)(__funnelshift_l((uint32_t)lo, (uint32_t)hi, 11) | 0x80000000u) << 32) | ((uint32_t)lo << 11);
}

// How a matrix mixes real and imaginary parts. In general every output part sees
// both and a group has one scale. A matrix that is real once some rows and columns
// are multiplied by i (real gates, RX) keeps two classes of reals apart: class 0
// holds the real parts of columns whose bit in col is clear and the imaginary parts
// of the others, class 1 the rest, and row j's real part sums the class that its bit
// in row names. Then (SPLIT) each class has a scale of its own, so that small parts
// beside large ones keep their accuracy, as they do in FP64. 26 qubits, with and
// without: 0.34 / 0.32 ms for k = 1, 0.47 / 0.45 for k = 2, 0.87 / 0.79 and 1.04 / 0.91
// for k = 3 and 4, 2.06 / 2.02 for k = 5.
struct Parts {
    uint32_t row, col;
    bool split;
};

// The classes of an amplitude's parts r, i (and back: a row's parts of the two classes' values)
template <typename T>
__device__ __forceinline__ void by_class(uint32_t bits, int l, const T &r, const T &i, T &c0, T &c1) {
    const bool f = ((bits >> l) & 1u) != 0;
    c0 = f ? i : r;
    c1 = f ? r : i;
}

__device__ __forceinline__ bool out_of_range(int E) { return (unsigned)(E - kEMin) > (unsigned)(kEMax - kEMin); }

// ---------------------------------------------------------------------------
// two limbs of 30 bits. x = (x1 2^30 + x0) 2^-P 2^(E - 1022), sign and
// magnitude, P = 60 (k = 1) or 59 (k = 2) bits; m = (m1 2^30 + m0) 2^-PM 2^em
// with |m0| <= 2^29, PM = 60 or 59. Sums over the 2 2^k real products:
//   k = 1: x1 m1 <= 2^60, 4 of them 2^62; x1 m0 + x0 m1 <= 2^59 + 2^60, 4: 2^62.6
//   k = 2: x1 m1 <= 2^58, 8: 2^61;        x1 m0 + x0 m1 <= 2^58 + 2^59, 8: 2^62.6
// The x0 m0 products (below 2^-59 of the full scale, random sign) are dropped.
//
// What bounds it: HBM, with the integer pipes close behind (about 80 ALU and
// 24 / 48 multiply-add instructions per amplitude). 26 qubits (HBM 0.316 ms):
// 0.32 to 0.34 ms for k = 1 (FP64 1.02), 0.44 to 0.46 for k = 2 (FP64 2.03).
// ---------------------------------------------------------------------------
template <int K> struct Fx2 {
    static constexpr int P = 61 - K, PM = 61 - K;
    int m[1 << (2 * K)][4];         // r1, r0, i1, i0
    int em;
    Parts parts;
    double2 f[1 << (2 * K)];        // for groups out of range
};

template <int K, int U, bool SPLIT>
__global__ void __launch_bounds__(kThreads, K == 1 ? 4 : 3)
k_dense_fx2(double2 *__restrict__ sv, uint64_t n_groups, GroupGeom G, Offs<K> O, Fx2<K> M) {
    constexpr int D = 1 << K, P = Fx2<K>::P, PM = Fx2<K>::PM;
    const uint64_t u0 = (uint64_t)blockIdx.x * (kThreads * U) + threadIdx.x;
    double2 v[U][D];
    uint64_t base[U];
    let_next_start();
#pragma unroll
    for (int u = 0; u < U; ++u) base[u] = insert_zeros(u0 + (uint64_t)u * kThreads, G);
    wait_for_previous();
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (u0 + (uint64_t)u * kThreads < n_groups) {
#pragma unroll
            for (int j = 0; j < D; ++j) v[u][j] = sv[base[u] + O.o[j]];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (u0 + (uint64_t)u * kThreads >= n_groups) continue;
        int hi[2 * D], lo[2 * D], top[2] = {0, 0};       // by class; of all reals if not SPLIT
#pragma unroll
        for (int l = 0; l < D; ++l) {
            hi[2 * l] = __double2hiint(v[u][l].x);
            lo[2 * l] = __double2loint(v[u][l].x);
            hi[2 * l + 1] = __double2hiint(v[u][l].y);
            lo[2 * l + 1] = __double2loint(v[u][l].y);
            const int hr = hi[2 * l] & 0x7fffffff, hj = hi[2 * l + 1] & 0x7fffffff;
            if constexpr (SPLIT) {
                int c0, c1;
                by_class(M.parts.col, l, hr, hj, c0, c1);
                top[0] = max(top[0], c0);
                top[1] = max(top[1], c1);
            } else {
                top[0] = max(top[0], max(hr, hj));
            }
        }
        int E[2] = {top[0] >> 20, SPLIT ? top[1] >> 20 : top[0] >> 20};
        if (out_of_range(E[0]) || (SPLIT && out_of_range(E[1]))) {
            // zeros take any scale; what else is out of range goes to FP64
            uint32_t any[2] = {0, 0};
#pragma unroll
            for (int l = 0; l < D; ++l) {
                const uint32_t ar = (uint32_t)(hi[2 * l] & 0x7fffffff) | (uint32_t)lo[2 * l];
                const uint32_t aj = (uint32_t)(hi[2 * l + 1] & 0x7fffffff) | (uint32_t)lo[2 * l + 1];
                if constexpr (SPLIT) {
                    uint32_t c0, c1;
                    by_class(M.parts.col, l, ar, aj, c0, c1);
                    any[0] |= c0;
                    any[1] |= c1;
                } else {
                    any[0] |= ar | aj;
                }
            }
            const bool none = (any[0] | any[1]) == 0;      // most groups of a state near a basis state
            if (none || (any[0] && out_of_range(E[0])) || (SPLIT && any[1] && out_of_range(E[1]))) {
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    double2 acc = make_double2(0.0, 0.0);
                    if (!none) {
#pragma unroll
                        for (int l = 0; l < D; ++l) cmad(acc, M.f[j * D + l], v[u][l]);
                    }
                    sv[base[u] + O.o[j]] = acc;
                }
                continue;
            }
            if constexpr (SPLIT) {
                if (!any[0]) E[0] = kEMin;
                if (!any[1]) E[1] = kEMin;
            }
        }
        int x1[2 * D], x0[2 * D];
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) {
            const int e = (hi[i] >> 20) & 0x7ff;
            const int Ei = SPLIT && (((M.parts.col >> (i / 2)) ^ i) & 1u) ? E[1] : E[0];
            const uint64_t F = shr64(mant64(hi[i], lo[i]), (uint32_t)(64 - P + Ei - e));
            const int sg = (hi[i] >> 31) | 1;
            x1[i] = (int)__funnelshift_r((uint32_t)F, (uint32_t)(F >> 32), 30) * sg;
            x0[i] = (int)((uint32_t)F & 0x3fffffffu) * sg;
        }
        const int sc[2] = {E[0] - 1022 + M.em + 60 - P - PM, E[1] - 1022 + M.em + 60 - P - PM};
        auto out = [&](long long a1, long long a0, int sc) {
            return scaled(__ll2double_rn(a1 + ((a0 + (1ll << 29)) >> 30)), sc);
        };
#pragma unroll
        for (int j = 0; j < D; ++j) {
            long long r1 = 0, r0 = 0, i1 = 0, i0 = 0;
#pragma unroll
            for (int l = 0; l < D; ++l) {
                const int *m = M.m[j * D + l];
                const int a1 = x1[2 * l], a0 = x0[2 * l], b1 = x1[2 * l + 1], b0 = x0[2 * l + 1];
                r1 = mad_wide(a1, m[0], r1);
                r0 = mad_wide(a1, m[1], r0);
                r0 = mad_wide(a0, m[0], r0);
                r1 = mad_wide(-b1, m[2], r1);
                r0 = mad_wide(-b1, m[3], r0);
                r0 = mad_wide(-b0, m[2], r0);
                i1 = mad_wide(a1, m[2], i1);
                i0 = mad_wide(a1, m[3], i0);
                i0 = mad_wide(a0, m[2], i0);
                i1 = mad_wide(b1, m[0], i1);
                i0 = mad_wide(b1, m[1], i0);
                i0 = mad_wide(b0, m[0], i0);
            }
            int sr = sc[0], si = sc[0];
            if constexpr (SPLIT) by_class(M.parts.row, j, sc[0], sc[1], sr, si);
            sv[base[u] + O.o[j]] = make_double2(out(r1, r0, sr), out(i1, i0, si));
        }
    }
}

// ---------------------------------------------------------------------------
// three limbs of L = 28 bits. x: 84 bits, sign and magnitude; m: 83 bits,
// balanced (|m0|, |m1|, |m2| <= 2^27). With xs = xr + xi, ms = mr + mi taken
// limb by limb (below 2^29 and 2^28), T1 = sum mr xr, T2 = sum mi xi,
// T3 = sum ms xs: re = T1 - T2, im = T3 - T1 - T2. Each T is three 64-bit sums,
// of the limb products of weight 2^4L, 2^3L and 2^2L; the last, with three
// products of at most 2^57 per term, holds up to 2^4 terms (2^62.6).
//
// What bounds it: the integer multiply-adds (18 per complex product; one
// thread holds a group of up to 16 amplitudes in limbs, the matrix is
// broadcast from shared memory, 24 bytes per complex product). 26 qubits: 0.79 ms
// for k = 1 (FP64 1.03), 0.99 for k = 2 (2.05), 1.59 for k = 3 (4.08), 2.98 for k = 4 (8.1; four lanes a group or other
// occupancies up to 3.46).
// ---------------------------------------------------------------------------
constexpr int kL = 28;
constexpr int kFx3Threads = 128;

template <int K> struct Fx3 {
    int m[1 << (2 * K)][6];          // r2, r1, r0, i2, i1, i0
    int em;
    int t;                           // nonzero amplitudes (SPLIT: reals of a class) must lie within 2^t of the largest
    Parts parts;
    double2 f[1 << (2 * K)];
};

struct Sum3 {
    long long a2, a1, a0;
};

// a2 2^2L + a1 2^L + a0 as a double; be: biased exponent of 2^63 in units of a2
__device__ __forceinline__ double out3(long long a2, long long a1, long long a0, int be) {
    constexpr uint32_t mask = (1u << kL) - 1u;
    a1 += a0 >> kL;
    a2 += a1 >> kL;
    uint64_t q = ((uint64_t)((uint32_t)a1 & mask) << (64 - kL)) | ((uint64_t)((uint32_t)a0 & mask) << (64 - 2 * kL));
    const int s = (int)(a2 >> 63);
    uint64_t h = (uint64_t)a2;
    if (s) {                          // negate the 128-bit number h.q
        q = 0ull - q;
        h = ~h + (q == 0 ? 1ull : 0ull);
    }
    if (h == 0) {                     // the sum cancelled below one unit of a2
        if (q == 0) return 0.0;
        h = q;
        q = 0;
        be -= 64;
    }
    const int n = __clzll((long long)h);
    const uint64_t v = n == 0 ? h : (h << n) | (q >> (64 - n));
    return pack(v, be - n, s);
}

// A group is shared by S lanes, DL = 2^K / S of its amplitudes each (lane s holds
// members s DL .. s DL + DL - 1): each lane sums its members' share of S rows,
// then hands every other lane its row's partial sums and finishes one row.
template <int K, int S, bool SPLIT>
__global__ void __launch_bounds__(kFx3Threads, 4)
k_dense_fx3(double2 *__restrict__ sv, uint64_t n_groups, GroupGeom G, const __grid_constant__ Offs<K> O,
            const __grid_constant__ Fx3<K> M) {
    constexpr int D = 1 << K, DL = D / S;
    constexpr int RS = (DL * 8 + (S > 1 ? 8 : 0)) * S;   // ints of a row; lanes' parts 8 banks apart
    __shared__ __align__(16) int Ms[D * RS];
    let_next_start();
    for (int i = threadIdx.x; i < D * D * 6; i += kFx3Threads) {
        const int e = i / 6, j = e / D, l = e % D;
        Ms[j * RS + (l / DL) * (RS / S) + (l % DL) * 8 + i % 6] = M.m[e][i % 6];
    }
    __syncthreads();
    const int s = threadIdx.x & (S - 1);
    uint64_t g = ((uint64_t)blockIdx.x * kFx3Threads + threadIdx.x) / S;
    const bool valid = g < n_groups;
    if (!valid) g = 0;                                  // whole warps take part in the exchanges; nothing is stored
    const uint64_t base = insert_zeros(g, G);
    wait_for_previous();
    int x[2 * DL][3];
    constexpr int NC = SPLIT ? 2 : 1;                   // scales
    int E[NC];
    bool slow, zero;
    {
        double2 v[DL];
#pragma unroll
        for (int j = 0; j < DL; ++j) v[j] = sv[base + O.o[s * DL + j]];
        int top[NC];
        uint32_t low[NC], denorm = 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            top[c] = 0;
            low[c] = 0xffffffffu;
        }
#pragma unroll
        for (int l = 0; l < DL; ++l) {
            const int hr = __double2hiint(v[l].x) & 0x7fffffff, hj = __double2hiint(v[l].y) & 0x7fffffff;
            const uint32_t lr = (uint32_t)__double2loint(v[l].x), lj = (uint32_t)__double2loint(v[l].y);
            int a[NC];
            if constexpr (SPLIT) {
                by_class(M.parts.col, s * DL + l, hr, hj, a[0], a[NC - 1]);
                if (hr == 0) denorm |= lr;
                if (hj == 0) denorm |= lj;
            } else {
                a[0] = max(hr, hj);
                if (a[0] == 0) denorm |= lr | lj;
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                top[c] = max(top[c], a[c]);
                low[c] = min(low[c], (uint32_t)a[c] - 1u);   // an exact zero wraps around and does not count
            }
        }
#pragma unroll
        for (int o = 1; o < S; o <<= 1) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                top[c] = max(top[c], __shfl_xor_sync(0xffffffffu, top[c], o));
                low[c] = min(low[c], __shfl_xor_sync(0xffffffffu, low[c], o));
            }
            denorm |= __shfl_xor_sync(0xffffffffu, denorm, o);
        }
        zero = ((uint32_t)(top[0] | top[NC - 1]) | denorm) == 0;   // the product of zeros: the amplitudes stay zero
        slow = denorm != 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            slow = slow || (uint32_t)top[c] - low[c] > ((uint32_t)M.t << 20) || (top[c] != 0 && out_of_range(top[c] >> 20));
            E[c] = top[c] != 0 ? top[c] >> 20 : kEMin;  // zeros take any scale
        }
#pragma unroll
        for (int i = 0; i < 2 * DL; ++i) {
            const double w = (i & 1) ? v[i >> 1].y : v[i >> 1].x;
            const int hi = __double2hiint(w);
            const int Ei = SPLIT && (((M.parts.col >> (s * DL + (i >> 1))) ^ i) & 1u) ? E[NC - 1] : E[0];
            const uint32_t d = (uint32_t)(Ei - ((hi >> 20) & 0x7ff));
            const uint64_t m = mant64(hi, __double2loint(w));
            const uint64_t hl = shr64(m, d);
            const uint32_t r2 = (uint32_t)(hl >> 32), r1 = (uint32_t)hl;
            const uint32_t r0 = d <= 32 ? shl32((uint32_t)m, 32 - d) : (uint32_t)shr64(m, d - 32);
            constexpr uint32_t mask = (1u << kL) - 1u;
            const int sg = (hi >> 31) | 1;
            x[i][0] = (int)(r2 >> (32 - kL)) * sg;
            x[i][1] = (int)(__funnelshift_r(r1, r2, 64 - 2 * kL) & mask) * sg;
            x[i][2] = (int)(__funnelshift_r(r0, r1, 96 - 3 * kL) & mask) * sg;
        }
    }
    if (__any_sync(0xffffffffu, slow)) {
        // lane s computes rows s DL .. s DL + DL - 1 of its group in FP64
        double2 acc[DL];
#pragma unroll
        for (int j = 0; j < DL; ++j) acc[j] = make_double2(0.0, 0.0);
        if (slow) {
#pragma unroll 1
            for (int l = 0; l < D; ++l) {
                const double2 w = sv[base + O.o[l]];
#pragma unroll
                for (int j = 0; j < DL; ++j) cmad(acc[j], M.f[(s * DL + j) * D + l], w);
            }
        }
        __syncwarp();                                   // every lane has read its group before any writes it
        if (slow && valid) {
#pragma unroll
            for (int j = 0; j < DL; ++j) sv[base + O.o[s * DL + j]] = acc[j];
        }
    }
    if (__all_sync(0xffffffffu, slow || zero)) return;
    const bool store = valid && !slow && !zero;
    // weight of a2: 2^(4L - 84 - 83 + E - 1022 + em); its bit 63 has biased exponent
    // that plus 63 + 1023
    const int be[2] = {E[0] + M.em + 64 + 4 * kL - 167, E[NC - 1] + M.em + 64 + 4 * kL - 167};
    // the row loop stays rolled (the unrolled kernel would not fit the instruction cache)
#pragma unroll 1
    for (int j = 0; j < D; j += S) {
        Sum3 re[S], im[S];
#pragma unroll
        for (int r = 0; r < S; ++r) {
            // rounds of nine independent sums: the multiply-adds of one sum are far apart
            Sum3 t1{0, 0, 0}, t2{0, 0, 0}, t3{0, 0, 0};
            const int *mrow = Ms + (j + r) * RS + s * (RS / S);
#pragma unroll
            for (int l = 0; l < DL; ++l) {
                const int4 ma = *reinterpret_cast<const int4 *>(mrow + 8 * l);
                const int2 mb = *reinterpret_cast<const int2 *>(mrow + 8 * l + 4);
                const int *a = x[2 * l], *b = x[2 * l + 1];
                const int c2 = a[0] + b[0], c1 = a[1] + b[1], c0 = a[2] + b[2];
                const int n2 = ma.x + ma.w, n1 = ma.y + mb.x, n0 = ma.z + mb.y;
                t1.a2 = mad_wide(a[0], ma.x, t1.a2);
                t2.a2 = mad_wide(b[0], ma.w, t2.a2);
                t3.a2 = mad_wide(c2, n2, t3.a2);
                t1.a1 = mad_wide(a[0], ma.y, t1.a1);
                t2.a1 = mad_wide(b[0], mb.x, t2.a1);
                t3.a1 = mad_wide(c2, n1, t3.a1);
                t1.a0 = mad_wide(a[0], ma.z, t1.a0);
                t2.a0 = mad_wide(b[0], mb.y, t2.a0);
                t3.a0 = mad_wide(c2, n0, t3.a0);
                t1.a1 = mad_wide(a[1], ma.x, t1.a1);
                t2.a1 = mad_wide(b[1], ma.w, t2.a1);
                t3.a1 = mad_wide(c1, n2, t3.a1);
                t1.a0 = mad_wide(a[1], ma.y, t1.a0);
                t2.a0 = mad_wide(b[1], mb.x, t2.a0);
                t3.a0 = mad_wide(c1, n1, t3.a0);
                t1.a0 = mad_wide(a[2], ma.x, t1.a0);
                t2.a0 = mad_wide(b[2], ma.w, t2.a0);
                t3.a0 = mad_wide(c0, n2, t3.a0);
            }
            re[r] = Sum3{t1.a2 - t2.a2, t1.a1 - t2.a1, t1.a0 - t2.a0};
            im[r] = Sum3{t3.a2 - t1.a2 - t2.a2, t3.a1 - t1.a1 - t2.a1, t3.a0 - t1.a0 - t2.a0};
        }
        // lane s keeps row j + s: at each step half of the rows go to the other lane
#pragma unroll
        for (int o = S / 2; o > 0; o >>= 1) {
            const bool up = (s & o) != 0;
#pragma unroll
            for (int r = 0; r < o; ++r) {
                auto trade = [&](long long &keep, long long &give) {
                    const long long mine = up ? give : keep, send = up ? keep : give;
                    keep = mine + __shfl_xor_sync(0xffffffffu, send, o);
                };
                trade(re[r].a2, re[r + o].a2);
                trade(re[r].a1, re[r + o].a1);
                trade(re[r].a0, re[r + o].a0);
                trade(im[r].a2, im[r + o].a2);
                trade(im[r].a1, im[r + o].a1);
                trade(im[r].a0, im[r + o].a0);
            }
        }
        int br = be[0], bi = be[0];
        if constexpr (SPLIT) by_class(M.parts.row, j + s, be[0], be[1], br, bi);
        const double2 w = make_double2(out3(re[0].a2, re[0].a1, re[0].a0, br), out3(im[0].a2, im[0].a1, im[0].a0, bi));
        if (store) sv[base + O.o[j + s]] = w;
    }
}

// ---------------------------------------------------------------------------
// k = 3, 4, 5 on the tensor cores, for matrices with no zero entry. Fixed point of P
// bits, rounded (truncated, the worst amplitude had twice the error), in ND balanced
// digits of B bits, held as FP16 integers; a group's 2 2^k reals are one column of an mma.sync B operand, the
// matrix (real 2 x 2 blocks) is A, and digit products of equal weight are summed
// by the FP32 accumulators, exactly: |digit| <= 2^(B-1), so a sum of 2 2^k terms
// and up to ND digit pairs stays within 2^24, where every integer is an FP32 number
// (that the accumulation then rounds nothing is not documented: it rests on the tests,
// which have sums of largest digits, and such sums that cancel):
//   k = 3, 4: 7 digits of 9 bits, 2^16 * 32 * 7 = 2^23.8
//   k = 5:    8 digits of 8 bits, 2^14 * 64 * 8 = 2^23
// Products of digits i, j (from the top) with i + j > ND are left out: below
// 2^-65 of the full scale, random in sign.
//
// Why mma.sync: the matrix is 16 to 64 reals wide; a tcgen05 tile (128 rows)
// would be mostly padding, and its operands would have to pass through shared
// memory, where here a lane forms its own fragment registers: lane 4 c + q of
// column c holds members q, q + 4, ... (re and im adjacent), and with re in rows
// 0..7 and im in rows 8..15 of a tile it gets whole output amplitudes back.
// Columns 2 q and 2 q + 1 are groups q and q + 4 of the warp's eight, so that a
// store instruction covers 64 contiguous bytes per member.
//
// What bounds it: conversions to digits and back (about 110 instructions per
// amplitude; ALU 46 %, FP64 25 % busy at k = 4) and the MMAs (53 %), which the 16 to
// 24 warps of an SM overlap in part; the 32 bytes an amplitude moves are a third to a
// half of the time. 26 qubits: 0.79 ms for k = 3, 0.91 for k = 4, 2.0 for k = 5 (FP64
// 4.08, 8.1, 14.0; three limbs 1.59 and 2.98). Three blocks per SM at k = 4: 1.01.
// ---------------------------------------------------------------------------
constexpr int kFxtThreads = 256;
constexpr int kLarge = 2;                     // an amplitude within 2^kLarge of its group's largest is large

template <int K> struct FxtCfg {
    static constexpr int D = 1 << K, ND = K <= 4 ? 7 : 8, B = K <= 4 ? 9 : 8;
    static constexpr int P = K <= 4 ? 61 : 62;
    static constexpr int blocks = K == 3 ? 3 : K == 4 ? 2 : 1;   // resident per SM
    static constexpr int TM = D / 8;             // 16-row tiles of A, and 16-deep steps
    static constexpr size_t smem = sizeof(uint4) * 32 * TM * TM * ND;
};

template <int K> struct Fxt {
    long long m[1 << (2 * K)][2];   // round(2^(P - em) re, im)
    double2 f[1 << (2 * K)];        // for groups out of range
    int em;
    int exact;                      // 0: every group may be computed so. Else groups whose reals lie within 2^exact
                                    // are held exactly (negative: none), and the others need every row to see
                                    // a large amplitude through an entry outside its
    uint32_t small[1 << K];         // the small entries of each row
    Parts parts;
};

// digit i (from the top) of the offset fixed-point numbers r, j as two FP16 integers;
// HALF: of numbers with one more bit, which is dropped
template <int ND, int B, int HALF = 0>
__device__ __forceinline__ uint32_t digits(uint64_t r, uint64_t j, int i) {
    const int sh = B * (ND - 1 - i) + HALF;
    const uint32_t a = (uint32_t)(r >> sh), b = (uint32_t)(j >> sh);
    constexpr uint32_t mask = ((1u << B) - 1u) * 0x00010001u;
    uint32_t p = (__byte_perm(a, b, 0x5410) & mask) | 0x64006400u;        // 1024 + digit + 2^(B-1)
    const uint32_t off = (0x6400u + (1u << (B - 1))) * 0x00010001u;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(p) : "r"(p), "r"(off));
    return p;
}

template <int ND, int B> __device__ __forceinline__ constexpr uint64_t digit_offset() {
    uint64_t o = 0;
    for (int i = 0; i < ND; ++i) o = (o << B) + (1ull << (B - 1));
    return o;
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

template <int K, bool SPLIT>
__global__ void __launch_bounds__(kFxtThreads, FxtCfg<K>::blocks)
k_dense_fxt(double2 *__restrict__ sv, uint64_t n_groups, GroupGeom G, const __grid_constant__ Offs<K> O,
            const Fxt<K> *__restrict__ Mg, const __grid_constant__ Fxt<(K <= 4 ? K : 1)> Mp) {
    using Cfg = FxtCfg<K>;
    constexpr int D = Cfg::D, ND = Cfg::ND, B = Cfg::B, P = Cfg::P, TM = Cfg::TM, NA = D / 4;
    constexpr int NL = ND + 1;                        // levels: digit pairs i + j = 0 .. ND
    constexpr int HALF = ND * B < 64 ? 1 : 0;
    constexpr uint64_t off = digit_offset<ND, B>();
    extern __shared__ __align__(16) uint4 As[];       // [mt][ks][digit][lane]
    const int lane = threadIdx.x & 31, q = lane & 3, c = lane >> 2;
    const long long(*M)[2] = K <= 4 ? reinterpret_cast<const long long(*)[2]>(Mp.m) : Mg->m;
    const double2 *Mf = K <= 4 ? reinterpret_cast<const double2 *>(Mp.f) : Mg->f;
    let_next_start();
    if constexpr (K > 4) wait_for_previous();          // the matrix is in the workspace
    const int em = K <= 4 ? Mp.em : Mg->em, exact = K <= 4 ? Mp.exact : Mg->exact;
    const uint32_t *small = K <= 4 ? Mp.small : Mg->small;
    const uint32_t prow = K <= 4 ? Mp.parts.row : Mg->parts.row, pcol = K <= 4 ? Mp.parts.col : Mg->parts.col;
    // A's fragments: lane 4 r + q holds rows r (re of member r) and r + 8 (its im),
    // members q (registers x, y) and q + 4 (z, w) of the step
    for (int i = threadIdx.x; i < TM * TM * 32; i += kFxtThreads) {
        const int ln = i & 31, ks = (i >> 5) % TM, mt = (i >> 5) / TM;
        const int row = mt * 8 + (ln >> 2), col = ks * 8 + (ln & 3);
        const uint64_t r0 = off + (uint64_t)M[row * D + col][0], j0 = off + (uint64_t)M[row * D + col][1];
        const uint64_t n0 = off - (uint64_t)M[row * D + col][1];
        const uint64_t r1 = off + (uint64_t)M[row * D + col + 4][0], j1 = off + (uint64_t)M[row * D + col + 4][1];
        const uint64_t n1 = off - (uint64_t)M[row * D + col + 4][1];
#pragma unroll
        for (int d = 0; d < ND; ++d)
            As[((mt * TM + ks) * ND + d) * 32 + ln] = make_uint4(digits<ND, B>(r0, n0, d), digits<ND, B>(j0, r0, d),
                                                                 digits<ND, B>(r1, n1, d), digits<ND, B>(j1, r1, d));
    }
    __syncthreads();
    const int gcol = (c >> 1) + 4 * (c & 1);           // this lane's group of the eight as a B column
    const uint64_t n_tiles = (n_groups + 7) / 8;
    const uint64_t step = (uint64_t)gridDim.x * (kFxtThreads / 32);
    uint64_t t = (uint64_t)blockIdx.x * (kFxtThreads / 32) + (threadIdx.x >> 5);
    // a tile's amplitudes are loaded while the one before is computed
    double2 v[NA];
    uint64_t next = 0;
    auto load = [&](uint64_t tile) {
        const uint64_t g = tile * 8 + gcol;
        next = insert_zeros(g < n_groups ? g : 0, G);
#pragma unroll
        for (int i = 0; i < NA; ++i) v[i] = sv[next + O.o[4 * i + q]];
    };
    if constexpr (K <= 4) wait_for_previous();
    if (t < n_tiles) load(t);
    for (; t < n_tiles; t += step) {
        const bool valid = t * 8 + gcol < n_groups;
        const uint64_t base = next;
        uint32_t b[NA][ND];
        constexpr int NC = SPLIT ? 2 : 1;               // scales
        int E[NC];
        bool slow, zero;
        {
            int top[NC];
            uint32_t any = 0;                           // low words (SPLIT: of reals whose upper word is zero)
#pragma unroll
            for (int c = 0; c < NC; ++c) top[c] = 0;
            auto upper = [&](int i, int (&a)[NC]) {     // an amplitude's magnitude, or its classes'
                const int hr = __double2hiint(v[i].x) & 0x7fffffff, hj = __double2hiint(v[i].y) & 0x7fffffff;
                if constexpr (SPLIT) by_class(pcol, 4 * i + q, hr, hj, a[0], a[NC - 1]);
                else a[0] = max(hr, hj);
            };
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                int a[NC];
                upper(i, a);
#pragma unroll
                for (int c = 0; c < NC; ++c) top[c] = max(top[c], a[c]);
                if (!SPLIT || (__double2hiint(v[i].x) & 0x7fffffff) == 0) any |= (uint32_t)__double2loint(v[i].x);
                if (!SPLIT || (__double2hiint(v[i].y) & 0x7fffffff) == 0) any |= (uint32_t)__double2loint(v[i].y);
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
                for (int c = 0; c < NC; ++c) top[c] = max(top[c], __shfl_xor_sync(0xffffffffu, top[c], o));
                any |= __shfl_xor_sync(0xffffffffu, any, o);
            }
            zero = ((uint32_t)(top[0] | top[NC - 1]) | any) == 0;
            slow = SPLIT && any != 0;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                slow = slow || ((SPLIT ? top[c] != 0 : !zero) && out_of_range(top[c] >> 20));
                E[c] = top[c] != 0 ? top[c] >> 20 : kEMin;   // zeros take any scale
            }
            if (exact) {
                // a row all of whose large amplitudes (or reals of a class) meet small entries, in a
                // group that is not held exactly
                uint32_t large[NC], low[NC], lost = 0;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    large[c] = 0;
                    low[c] = 0xffffffffu;
                }
#pragma unroll
                for (int i = 0; i < NA; ++i) {
                    int a[NC];
                    upper(i, a);
                    const uint32_t r = (uint32_t)(__double2hiint(v[i].x) & 0x7fffffff) - 1u;   // zeros wrap around
                    const uint32_t j = (uint32_t)(__double2hiint(v[i].y) & 0x7fffffff) - 1u;
                    uint32_t l[NC];
                    if constexpr (SPLIT) by_class(pcol, 4 * i + q, r, j, l[0], l[NC - 1]);
                    else l[0] = min(r, j);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        low[c] = min(low[c], l[c]);
                        if (a[c] + (kLarge << 20) >= top[c]) large[c] |= 1u << (4 * i + q);
                    }
                }
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        low[c] = min(low[c], __shfl_xor_sync(0xffffffffu, low[c], o));
                        large[c] |= __shfl_xor_sync(0xffffffffu, large[c], o);
                    }
                }
                for (int row = q; row < D; row += 4) {
                    const uint32_t s = small[row];
#pragma unroll
                    for (int c = 0; c < NC; ++c) lost |= (large[c] & ~s) == 0 ? 1u << c : 0u;
                }
                lost |= __shfl_xor_sync(0xffffffffu, lost, 1);
                lost |= __shfl_xor_sync(0xffffffffu, lost, 2);
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    slow = slow || (top[c] != 0 && ((lost >> c) & 1u) &&
                                    (exact < 0 || (uint32_t)top[c] - low[c] > (uint32_t)exact << 20));
            }
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                // off +- the magnitude, F half units of 2^-P, rounded to whole ones (truncated,
                // the error doubles). With a bit to spare (HALF) the half units go along, and the
                // shift in digits() drops them: downwards, so a positive number first gets another
                auto fixed = [&](double w, int e) {
                    const int hi = __double2hiint(w);
                    const uint64_t F = shr64(mant64(hi, __double2loint(w)), (uint32_t)(63 - P + e - ((hi >> 20) & 0x7ff)));
                    if constexpr (HALF) return hi < 0 ? 2 * off - F : 2 * off + 1 + F;
                    else return hi < 0 ? off - ((F + 1) >> 1) : off + ((F + 1) >> 1);
                };
                int er = E[0], ej = E[0];
                if constexpr (SPLIT) by_class(pcol, 4 * i + q, E[0], E[NC - 1], er, ej);
                const uint64_t fr = fixed(v[i].x, er), fj = fixed(v[i].y, ej);
#pragma unroll
                for (int d = 0; d < ND; ++d) b[i][d] = digits<ND, B, HALF>(fr, fj, d);
            }
        }
        bool store = valid && !slow && !zero;
        if (__any_sync(0xffffffffu, slow)) {
            // a group outside the range: lane q computes rows q NA .. q NA + NA - 1 in FP64
            double2 acc[NA];
#pragma unroll
            for (int j = 0; j < NA; ++j) acc[j] = make_double2(0.0, 0.0);
            if (slow) {
#pragma unroll 1
                for (int l = 0; l < D; ++l) {
                    const double2 w = sv[base + O.o[l]];
#pragma unroll
                    for (int j = 0; j < NA; ++j) cmad(acc[j], Mf[(q * NA + j) * D + l], w);
                }
            }
            __syncwarp();                               // every lane has read its group before any writes it
            if (slow && valid) {
#pragma unroll
                for (int j = 0; j < NA; ++j) sv[base + O.o[q * NA + j]] = acc[j];
            }
        }
        if (t + step < n_tiles) load(t + step);
        // what the output lanes need of columns 2 q and 2 q + 1
        uint64_t ob[2];
        int sc[2][NC];
        bool st[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int from = 4 * (2 * q + h);
            ob[h] = __shfl_sync(0xffffffffu, base, from);
#pragma unroll
            for (int c = 0; c < NC; ++c) sc[h][c] = __shfl_sync(0xffffffffu, E[c], from) - 1022 + em - 2 * P + B * (ND - 2);
            st[h] = __shfl_sync(0xffffffffu, (int)store, from) != 0;
        }
#pragma unroll 1
        for (int mt = 0; mt < TM; ++mt) {
            float a[NL][4];
#pragma unroll
            for (int p = 0; p < NL; ++p)
#pragma unroll
                for (int e = 0; e < 4; ++e) a[p][e] = 0.f;
#pragma unroll
            for (int ks = 0; ks < TM; ++ks) {
#pragma unroll
                for (int i = 0; i < ND; ++i) {
                    const uint4 f = As[((mt * TM + ks) * ND + i) * 32 + lane];
#pragma unroll
                    for (int j = 0; j < ND && i + j < NL; ++j) mma16816(a[i + j], f, b[2 * ks][j], b[2 * ks + 1][j]);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                auto out = [&](int e, int shift) {
                    int w[NL];
#pragma unroll
                    for (int p = 0; p < NL; ++p) w[p] = __float2int_rn(a[p][e]);     // exact: |a| <= 2^24
                    // level p weighs 2^(B (ND - p)) units of the last one; the sum is hi 2^S + lo
                    constexpr int S = B * (NL - 4);
                    const long long hi = (long long)(w[0] * (1 << B) + w[1]) * (1 << (2 * B)) + (long long)w[2] * (1 << B) + w[3];
                    long long lo = (long long)w[4] * (1 << (2 * B)) + (long long)w[5] * (1 << B) + w[6];
#pragma unroll
                    for (int p = 7; p < NL; ++p) lo = lo * (1 << B) + w[p];
                    // 62 bits of it are rounded to the double's 53 (the FP64 pipe, which also
                    // converts, is the scarce one: two conversions and a fused multiply-add
                    // per real kept it 75 % busy)
                    const int h1 = (int)(hi >> 32);
                    const int cut = max(0, S + 2 - __clz(h1 ^ (h1 >> 31)));
                    return scaled(__ll2double_rn((hi << (S - cut)) + (lo >> cut)), shift + cut);
                };
                int sr = sc[h][0], si = sc[h][0];
                if constexpr (SPLIT) by_class(prow, mt * 8 + c, sc[h][0], sc[h][NC - 1], sr, si);
                const double2 w = make_double2(out(h, sr), out(2 + h, si));
                if (st[h]) sv[ob[h] + O.o[mt * 8 + c]] = w;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct MatRange {
    bool finite, zeros;   // all entries finite; some entry exactly zero
    int em;               // largest real below 2^em
    int dm;               // smallest nonzero entry (its larger real) at least 2^(em - 1 - dm)
};

MatRange range_of(const double *mat, int entries) {
    MatRange r{true, false, -5000, 0};
    int lo = 5000;
    for (int i = 0; i < entries; ++i) {
        const double a = std::fmax(std::fabs(mat[2 * i]), std::fabs(mat[2 * i + 1]));
        if (!std::isfinite(mat[2 * i]) || !std::isfinite(mat[2 * i + 1])) r.finite = false;
        if (a == 0.0) {
            r.zeros = true;
            continue;
        }
        int e;
        std::frexp(a, &e);
        if (e > r.em) r.em = e;
        if (e < lo) lo = e;
    }
    r.dm = r.em - lo;
    return r;
}

// row by row, the entries below 2^(em - 1 - bits); returns how many a row has at most
int small_entries(const double *mat, int k, int em, int bits, uint32_t *rows) {
    const int D = 1 << k;
    const double line = std::ldexp(1.0, em - 1 - bits);
    int most = 0;
    for (int j = 0; j < D; ++j) {
        rows[j] = 0;
        for (int l = 0; l < D; ++l) {
            const double *m = mat + 2 * (j * D + l);
            if (std::fmax(std::fabs(m[0]), std::fabs(m[1])) < line) rows[j] |= 1u << l;
        }
        most = std::max(most, __builtin_popcount(rows[j]));
    }
    return most;
}

// round(v 2^(bits - em)) for |v| < 2^em
__int128 to_fixed(double v, int em, int bits) {
    int e;
    const double f = std::frexp(std::fabs(v), &e);
    const __int128 m = (__int128)std::llrint(std::scalbn(f, 53));   // exact: 53 bits
    const int sh = bits - 53 + (e - em);
    __int128 r;
    if (sh >= 0) r = m << sh;
    else if (sh > -54) r = (m + ((__int128)1 << (-sh - 1))) >> -sh;
    else r = 0;
    return v < 0 ? -r : r;
}

// the lowest limb of v, balanced; v becomes the rest
int take_limb(__int128 &v, int bits) {
    const __int128 half = (__int128)1 << (bits - 1);
    __int128 lo = v & (((__int128)1 << bits) - 1);
    if (lo >= half) lo -= (__int128)1 << bits;
    v = (v - lo) >> bits;
    return (int)lo;
}

// Real up to factors i of rows and columns? (Entries without an imaginary part join a
// row and a column of equal factors, entries without a real part of different ones.)
Parts parts_of(const double *mat, int k) {
    const int D = 1 << k;
    int row[32], col[32];
    for (int j = 0; j < D; ++j) row[j] = col[j] = -1;
    auto kind = [&](int j, int l) {                  // -1: zero, 0 real, 1 imaginary, 2 both
        const bool r = mat[2 * (j * D + l)] != 0.0, i = mat[2 * (j * D + l) + 1] != 0.0;
        return r ? (i ? 2 : 0) : (i ? 1 : -1);
    };
    for (int j = 0; j < D; ++j) {
        if (row[j] >= 0) continue;
        row[j] = 0;
        int todo[64], n = 0;                         // rows 0 .. 31, columns 32 .. 63
        todo[n++] = j;
        while (n > 0) {
            const int at = todo[--n];
            for (int o = 0; o < D; ++o) {
                const int t = at < 32 ? kind(at, o) : kind(o, at - 32);
                if (t < 0) continue;
                if (t == 2) return Parts{0, 0, false};
                int &mine = at < 32 ? row[at] : col[at - 32], &other = at < 32 ? col[o] : row[o];
                if (other < 0) {
                    other = mine ^ t;
                    todo[n++] = at < 32 ? 32 + o : o;
                } else if (other != (mine ^ t)) {
                    return Parts{0, 0, false};
                }
            }
        }
    }
    Parts p{0, 0, true};
    for (int j = 0; j < D; ++j) {
        p.row |= (uint32_t)(row[j] == 1) << j;
        p.col |= (uint32_t)(col[j] == 1) << j;
    }
    return p;
}

template <int K> void offsets(const int *tpos, Offs<K> &O) {
    for (int j = 0; j < (1 << K); ++j) {
        uint64_t o = 0;
        for (int t = 0; t < K; ++t)
            if ((j >> t) & 1) o |= 1ull << tpos[t];
        O.o[j] = o;
    }
}

template <int K>
cudaError_t run_fx2(const LaunchCtx &L, void *sv, uint64_t n_groups, const GroupGeom &G, const int *tpos,
                    const double *mat, int em) {
    constexpr int U = K == 1 ? 4 : 2;
    Offs<K> O;
    offsets<K>(tpos, O);
    Fx2<K> M;
    M.em = em;
    M.parts = parts_of(mat, K);
    for (int i = 0; i < (1 << (2 * K)); ++i) {
        for (int c = 0; c < 2; ++c) {
            __int128 v = to_fixed(mat[2 * i + c], em, Fx2<K>::PM);
            M.m[i][2 * c + 1] = take_limb(v, 30);
            M.m[i][2 * c] = (int)v;
        }
        M.f[i] = make_double2(mat[2 * i], mat[2 * i + 1]);
    }
    const uint64_t per = (uint64_t)kThreads * U;
    ++*L.launches;
    return launch_dependent(M.parts.split ? k_dense_fx2<K, U, true> : k_dense_fx2<K, U, false>,
                            (unsigned)((n_groups + per - 1) / per), kThreads, 0, L.stream,
                            reinterpret_cast<double2 *>(sv), n_groups, G, O, M);
}

template <int K>
cudaError_t run_fx3(const LaunchCtx &L, void *sv, uint64_t n_groups, const GroupGeom &G, const int *tpos,
                    const double *mat, const MatRange &r) {
    Offs<K> O;
    offsets<K>(tpos, O);
    Fx3<K> M;
    M.em = r.em;
    M.t = 24 - r.dm;
    M.parts = parts_of(mat, K);
    for (int i = 0; i < (1 << (2 * K)); ++i) {
        for (int c = 0; c < 2; ++c) {
            __int128 v = to_fixed(mat[2 * i + c], r.em, 3 * kL - 1);
            M.m[i][3 * c + 2] = take_limb(v, kL);
            M.m[i][3 * c + 1] = take_limb(v, kL);
            M.m[i][3 * c] = (int)v;
        }
        M.f[i] = make_double2(mat[2 * i], mat[2 * i + 1]);
    }
    constexpr int S = K >= 4 ? 2 : 1;
    ++*L.launches;
    return launch_dependent(M.parts.split ? k_dense_fx3<K, S, true> : k_dense_fx3<K, S, false>,
                            (unsigned)((n_groups * S + kFx3Threads - 1) / kFx3Threads), kFx3Threads, 0, L.stream,
                            reinterpret_cast<double2 *>(sv), n_groups, G, O, M);
}

template <int K>
cudaError_t run_fxt(const LaunchCtx &L, void *sv, uint64_t n_groups, const GroupGeom &G, const int *tpos,
                    const double *mat, const MatRange &r, int exact, const uint32_t *small, void *d_mat) {
    using Cfg = FxtCfg<K>;
    Offs<K> O;
    offsets<K>(tpos, O);
    const Parts parts = parts_of(mat, K);
    auto fill = [&](auto &M) {
        M.em = r.em;
        M.exact = exact;
        std::copy(small, small + Cfg::D, M.small);
        M.parts = parts;
        for (int i = 0; i < (1 << (2 * K)); ++i) {
            for (int c = 0; c < 2; ++c) M.m[i][c] = (long long)to_fixed(mat[2 * i + c], r.em, Cfg::P);
            M.f[i] = make_double2(mat[2 * i], mat[2 * i + 1]);
        }
    };
    auto kern = parts.split ? k_dense_fxt<K, true> : k_dense_fxt<K, false>;
    cudaError_t e = cudaSuccess;
    if constexpr (Cfg::smem > 48 * 1024) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem);
        if (e != cudaSuccess) return e;
    }
    constexpr uint64_t groups_per_block = 8 * (kFxtThreads / 32);
    uint64_t grid = (n_groups + groups_per_block - 1) / groups_per_block;
    const uint64_t most = (uint64_t)L.num_sms * Cfg::blocks;
    if (grid > most) grid = most;
    ++*L.launches;
    double2 *psi = reinterpret_cast<double2 *>(sv);
    if constexpr (K <= 4) {
        Fxt<K> M;
        fill(M);
        return launch_dependent(kern, (unsigned)grid, kFxtThreads, Cfg::smem, L.stream, psi, n_groups, G, O, nullptr, M);
    } else {
        std::vector<Fxt<K>> hm(1);
        fill(hm[0]);
        e = cudaMemcpyAsync(d_mat, hm.data(), sizeof(Fxt<K>), cudaMemcpyHostToDevice, L.stream);
        if (e != cudaSuccess) return e;
        return launch_dependent(kern, (unsigned)grid, kFxtThreads, Cfg::smem, L.stream, psi, n_groups, G, O,
                                reinterpret_cast<const Fxt<K> *>(d_mat), Fxt<1>{});
    }
}

}  // namespace

bool try_dense_fx(const LaunchCtx &L, void *sv, int n, const GroupGeom &G, const int *tpos, int k, const double *mat,
                  void *d_mat, cudaError_t &e) {
    if (k > 5) return false;
    const MatRange r = range_of(mat, 1 << (2 * k));
    if (!r.finite || r.em < -100 || r.em > 100) return false;
    // The lines are where each layout's error reaches FP64's (above), not where the times
    // cross: the first that may run is the fastest. 26 qubits, ms: two limbs 0.32 / 0.45
    // (k = 1, 2), digits 0.79 / 0.91 / 2.0 (k = 3, 4, 5), three limbs 0.79 / 0.99 / 1.59 /
    // 2.98 (k = 1 to 4), FP64 1.03 / 2.05 / 4.08 / 8.1 / 14.0. k = 6 stays in FP64.
    const uint64_t n_groups = 1ull << (n - G.ns);
    if (k <= 2 && !r.zeros && r.dm <= (k == 1 ? 5 : 4)) {
        e = k == 1 ? run_fx2<1>(L, sv, n_groups, G, tpos, mat, r.em) : run_fx2<2>(L, sv, n_groups, G, tpos, mat, r.em);
        return true;
    }
    if (k >= 3 && !r.zeros && r.dm <= (k == 5 ? 11 : 8)) {
        const int sure = k == 5 ? 8 : 7, spare = k == 5 ? 9 : 8;     // spare: bits beyond a double's 53
        uint32_t small[32] = {0};
        int exact = 0;
        bool ok = true;
        if (r.dm > sure) {
            exact = r.dm <= spare ? spare : -1;
            ok = small_entries(mat, k, r.em, sure - kLarge, small) <= 3 * (1 << k) / 4;
        }
        if (ok) {
            e = k == 3   ? run_fxt<3>(L, sv, n_groups, G, tpos, mat, r, exact, small, d_mat)
                : k == 4 ? run_fxt<4>(L, sv, n_groups, G, tpos, mat, r, exact, small, d_mat)
                         : run_fxt<5>(L, sv, n_groups, G, tpos, mat, r, exact, small, d_mat);
            return true;
        }
    }
    if (k > 4 || r.dm > 16) return false;
    switch (k) {
    case 1: e = run_fx3<1>(L, sv, n_groups, G, tpos, mat, r); break;
    case 2: e = run_fx3<2>(L, sv, n_groups, G, tpos, mat, r); break;
    case 3: e = run_fx3<3>(L, sv, n_groups, G, tpos, mat, r); break;
    default: e = run_fx3<4>(L, sv, n_groups, G, tpos, mat, r); break;
    }
    return true;
}

}  // namespace svk
