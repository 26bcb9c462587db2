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
// Two layouts:
//   two limbs   k = 1, 2: 3 limb products per real product. Errors are below
//               about 2^-58 X max|m| 2^k, X the group's largest amplitude, so
//               the host uses it where every entry is within 2^6 (k = 1) or 2^5
//               (k = 2) of the largest: then every output holds a term
//               |m||x| >= 2^-6 max|m| X, and the error stays below the FP64
//               kernel's own bound 2^-53 sum |m||x| whatever the data.
//   three limbs 6 limb products per real product (complex products by three
//               real ones, exact in integers): about 84 bits. The host and the
//               kernel check that entries (dm bits) and nonzero amplitudes (t
//               bits) lie within t + dm <= 24 bits of their largest, which again
//               bounds the error by that of FP64 term by term; zeros are exact.
// A group outside these ranges (also infinities, NaN, values near the limits of
// the exponent) is computed in FP64 in the same kernel, with k_dense's sums in
// k_dense's order.
#include <cmath>
#include <cstring>

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

// mantissa of x with the implicit bit at bit 63
__device__ __forceinline__ uint64_t mant64(int hi, int lo) {
    return ((uint64_t)(__funnelshift_l((uint32_t)lo, (uint32_t)hi, 11) | 0x80000000u) << 32) | ((uint32_t)lo << 11);
}

// ---------------------------------------------------------------------------
// two limbs of 30 bits. x = (x1 2^30 + x0) 2^-P 2^(E - 1022), sign and
// magnitude, P = 60 (k = 1) or 59 (k = 2) bits; m = (m1 2^30 + m0) 2^-PM 2^em
// with |m0| <= 2^29, PM = 60 or 59. Sums over the 2 2^k real products:
//   k = 1: x1 m1 <= 2^60, 4 of them 2^62; x1 m0 + x0 m1 <= 2^59 + 2^60, 4: 2^62.6
//   k = 2: x1 m1 <= 2^58, 8: 2^61;        x1 m0 + x0 m1 <= 2^58 + 2^59, 8: 2^62.6
// The x0 m0 products (below 2^-59 of the full scale, random sign) are dropped.
//
// What bounds it: HBM, with the integer pipes close behind (about 80 ALU and
// 24 / 48 multiply-add instructions per amplitude).
// ---------------------------------------------------------------------------
template <int K> struct Fx2 {
    static constexpr int P = 61 - K, PM = 61 - K;
    int m[1 << (2 * K)][4];         // r1, r0, i1, i0
    int em;
    double2 f[1 << (2 * K)];        // for groups out of range
};

template <int K, int U>
__global__ void __launch_bounds__(kThreads)
k_dense_fx2(double2 *__restrict__ sv, uint64_t n_groups, GroupGeom G, Offs<K> O, Fx2<K> M) {
    constexpr int D = 1 << K, P = Fx2<K>::P, PM = Fx2<K>::PM;
    const uint64_t u0 = (uint64_t)blockIdx.x * (kThreads * U) + threadIdx.x;
    double2 v[U][D];
    uint64_t base[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        base[u] = insert_zeros(u0 + (uint64_t)u * kThreads, G);
        if (u0 + (uint64_t)u * kThreads < n_groups) {
#pragma unroll
            for (int j = 0; j < D; ++j) v[u][j] = sv[base[u] + O.o[j]];
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (u0 + (uint64_t)u * kThreads >= n_groups) continue;
        int hi[2 * D], lo[2 * D], top = 0;
#pragma unroll
        for (int l = 0; l < D; ++l) {
            hi[2 * l] = __double2hiint(v[u][l].x);
            lo[2 * l] = __double2loint(v[u][l].x);
            hi[2 * l + 1] = __double2hiint(v[u][l].y);
            lo[2 * l + 1] = __double2loint(v[u][l].y);
            top = max(top, max(hi[2 * l] & 0x7fffffff, hi[2 * l + 1] & 0x7fffffff));
        }
        const int E = top >> 20;
        if ((unsigned)(E - kEMin) > (unsigned)(kEMax - kEMin)) {
            uint32_t any = 0;
#pragma unroll
            for (int i = 0; i < 2 * D; ++i) any |= (uint32_t)(hi[i] & 0x7fffffff) | (uint32_t)lo[i];
#pragma unroll
            for (int j = 0; j < D; ++j) {
                double2 acc = make_double2(0.0, 0.0);
                if (any) {
#pragma unroll
                    for (int l = 0; l < D; ++l) cmad(acc, M.f[j * D + l], v[u][l]);
                }
                sv[base[u] + O.o[j]] = acc;
            }
            continue;
        }
        int x1[2 * D], x0[2 * D];
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) {
            const int e = (hi[i] >> 20) & 0x7ff;
            const uint64_t F = shr64(mant64(hi[i], lo[i]), (uint32_t)(64 - P + E - e));
            const int sg = (hi[i] >> 31) | 1;
            x1[i] = (int)__funnelshift_r((uint32_t)F, (uint32_t)(F >> 32), 30) * sg;
            x0[i] = (int)((uint32_t)F & 0x3fffffffu) * sg;
        }
        const int be = E + M.em + 64 + 60 - P - PM;
        auto out = [&](long long a1, long long a0) {
            const long long r = a1 + ((a0 + (1ll << 29)) >> 30);
            const int s = (int)(r >> 63);
            const uint64_t a = ((uint64_t)r ^ (uint64_t)(long long)s) - (uint64_t)(long long)s;
            const int n = __clzll((long long)a);
            return a == 0 ? 0.0 : pack(a << n, be - n, s);
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
            sv[base[u] + O.o[j]] = make_double2(out(r1, r0), out(i1, i0));
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
// broadcast from shared memory, 24 bytes per complex product).
// ---------------------------------------------------------------------------
constexpr int kL = 28;

template <int K> struct Fx3 {
    int m[1 << (2 * K)][6];          // r2, r1, r0, i2, i1, i0
    int em;
    int t;                           // nonzero amplitudes must lie within 2^t of the largest
    double2 f[1 << (2 * K)];
};

struct Sum3 {
    long long a2, a1, a0;
};

__device__ __forceinline__ void mul3(Sum3 &s, int x2, int x1, int x0, int m2, int m1, int m0) {
    s.a2 = mad_wide(x2, m2, s.a2);
    s.a1 = mad_wide(x2, m1, s.a1);
    s.a1 = mad_wide(x1, m2, s.a1);
    s.a0 = mad_wide(x2, m0, s.a0);
    s.a0 = mad_wide(x1, m1, s.a0);
    s.a0 = mad_wide(x0, m2, s.a0);
}

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

template <int K>
__global__ void __launch_bounds__(kThreads)
k_dense_fx3(double2 *__restrict__ sv, uint64_t n_groups, GroupGeom G, const __grid_constant__ Offs<K> O,
            const __grid_constant__ Fx3<K> M) {
    constexpr int D = 1 << K;
    __shared__ __align__(16) int Ms[D * D][8];
    for (int i = threadIdx.x; i < D * D * 6; i += kThreads) Ms[i / 6][i % 6] = M.m[i / 6][i % 6];
    __syncthreads();
    const uint64_t g = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
    if (g >= n_groups) return;
    const uint64_t base = insert_zeros(g, G);
    int x[2 * D][3];
    int E;
    bool slow;
    {
        double2 v[D];
#pragma unroll
        for (int j = 0; j < D; ++j) v[j] = sv[base + O.o[j]];
        int top = 0;
        uint32_t low = 0xffffffffu, denorm = 0, any = 0;
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const int hr = __double2hiint(v[l].x) & 0x7fffffff, hj = __double2hiint(v[l].y) & 0x7fffffff;
            const uint32_t lw = (uint32_t)__double2loint(v[l].x) | (uint32_t)__double2loint(v[l].y);
            const int a = max(hr, hj);
            top = max(top, a);
            low = min(low, (uint32_t)a - 1u);          // an exact zero wraps around and does not count
            if (a == 0) denorm |= lw;
        }
        any = (uint32_t)top | denorm;
        E = top >> 20;
        slow = (unsigned)(E - kEMin) > (unsigned)(kEMax - kEMin) || denorm != 0 ||
               (uint32_t)top - low > ((uint32_t)M.t << 20);
        if (any == 0) return;                           // the product of zeros: the amplitudes stay zero
        if (!slow) {
#pragma unroll
            for (int i = 0; i < 2 * D; ++i) {
                const double w = (i & 1) ? v[i >> 1].y : v[i >> 1].x;
                const int hi = __double2hiint(w);
                const uint32_t d = (uint32_t)(E - ((hi >> 20) & 0x7ff));
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
    }
    if (slow) {
        double2 acc[D];
#pragma unroll
        for (int j = 0; j < D; ++j) acc[j] = make_double2(0.0, 0.0);
#pragma unroll 1
        for (int l = 0; l < D; ++l) {
            const double2 w = sv[base + O.o[l]];
#pragma unroll
            for (int j = 0; j < D; ++j) cmad(acc[j], M.f[j * D + l], w);
        }
#pragma unroll
        for (int j = 0; j < D; ++j) sv[base + O.o[j]] = acc[j];
        return;
    }
    // weight of a2: 2^(4L - 84 - 83 + E - 1022 + em); its bit 63 has biased exponent
    // that plus 63 + 1023
    const int be = E + M.em + 64 + 4 * kL - 167;
    // the row loop stays rolled (the unrolled kernel would not fit the instruction cache)
#pragma unroll 1
    for (int j = 0; j < D; ++j) {
        Sum3 t1{0, 0, 0}, t2{0, 0, 0}, t3{0, 0, 0};
        const int(*mrow)[8] = &Ms[j * D];
#pragma unroll
        for (int l = 0; l < D; ++l) {
            const int4 ma = *reinterpret_cast<const int4 *>(mrow[l]);
            const int2 mb = *reinterpret_cast<const int2 *>(mrow[l] + 4);
            const int *a = x[2 * l], *b = x[2 * l + 1];
            mul3(t1, a[0], a[1], a[2], ma.x, ma.y, ma.z);
            mul3(t2, b[0], b[1], b[2], ma.w, mb.x, mb.y);
            mul3(t3, a[0] + b[0], a[1] + b[1], a[2] + b[2], ma.x + ma.w, ma.y + mb.x, ma.z + mb.y);
        }
        const double re = out3(t1.a2 - t2.a2, t1.a1 - t2.a1, t1.a0 - t2.a0, be);
        const double im = out3(t3.a2 - t1.a2 - t2.a2, t3.a1 - t1.a1 - t2.a1, t3.a0 - t1.a0 - t2.a0, be);
        sv[base + O.o[j]] = make_double2(re, im);
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
    for (int i = 0; i < (1 << (2 * K)); ++i) {
        for (int c = 0; c < 2; ++c) {
            __int128 v = to_fixed(mat[2 * i + c], em, Fx2<K>::PM);
            M.m[i][2 * c + 1] = take_limb(v, 30);
            M.m[i][2 * c] = (int)v;
        }
        M.f[i] = make_double2(mat[2 * i], mat[2 * i + 1]);
    }
    const uint64_t per = (uint64_t)kThreads * U;
    k_dense_fx2<K, U><<<(unsigned)((n_groups + per - 1) / per), kThreads, 0, L.stream>>>(
        reinterpret_cast<double2 *>(sv), n_groups, G, O, M);
    ++*L.launches;
    return cudaGetLastError();
}

template <int K>
cudaError_t run_fx3(const LaunchCtx &L, void *sv, uint64_t n_groups, const GroupGeom &G, const int *tpos,
                    const double *mat, const MatRange &r) {
    Offs<K> O;
    offsets<K>(tpos, O);
    Fx3<K> M;
    M.em = r.em;
    M.t = 24 - r.dm;
    for (int i = 0; i < (1 << (2 * K)); ++i) {
        for (int c = 0; c < 2; ++c) {
            __int128 v = to_fixed(mat[2 * i + c], r.em, 3 * kL - 1);
            M.m[i][3 * c + 2] = take_limb(v, kL);
            M.m[i][3 * c + 1] = take_limb(v, kL);
            M.m[i][3 * c] = (int)v;
        }
        M.f[i] = make_double2(mat[2 * i], mat[2 * i + 1]);
    }
    k_dense_fx3<K><<<(unsigned)((n_groups + kThreads - 1) / kThreads), kThreads, 0, L.stream>>>(
        reinterpret_cast<double2 *>(sv), n_groups, G, O, M);
    ++*L.launches;
    return cudaGetLastError();
}

}  // namespace

bool try_dense_fx(const LaunchCtx &L, void *sv, int n, const GroupGeom &G, const int *tpos, int k, const double *mat,
                  cudaError_t &e) {
    if (k > 4) return false;
    const MatRange r = range_of(mat, 1 << (2 * k));
    if (!r.finite || r.em < -100 || r.em > 100) return false;
    const uint64_t n_groups = 1ull << (n - G.ns);
    if (k <= 2 && !r.zeros && r.dm <= (k == 1 ? 6 : 5)) {
        e = k == 1 ? run_fx2<1>(L, sv, n_groups, G, tpos, mat, r.em) : run_fx2<2>(L, sv, n_groups, G, tpos, mat, r.em);
        return true;
    }
    if (r.dm > 16) return false;
    switch (k) {
    case 1: e = run_fx3<1>(L, sv, n_groups, G, tpos, mat, r); break;
    case 2: e = run_fx3<2>(L, sv, n_groups, G, tpos, mat, r); break;
    case 3: e = run_fx3<3>(L, sv, n_groups, G, tpos, mat, r); break;
    default: e = run_fx3<4>(L, sv, n_groups, G, tpos, mat, r); break;
    }
    return true;
}

}  // namespace svk
