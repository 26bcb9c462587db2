// k_pauli.cu -- Pauli-string expectation values (Table I, "Expectation").
//
// For P = prod of Paulis, with x = mask of X/Y sites, z = mask of Z/Y sites and
// nY = number of Y sites,
//   P|i> = i^{nY} (-1)^{popcount(i & z)} |i ^ x>,
//   <psi|P|psi> = sum_i i^{nY} (-1)^{popcount(i & z)} psi_i conj(psi_{i^x}),
// which is real because P is Hermitian. With w_i = psi_i conj(psi_{i^x}) each
// unordered pair {i, i ^ x} gives twice +-Re(w_i) (nY even) or +-Im(w_i) (nY
// odd); x = 0 gives |psi_i|^2 once per amplitude. The host folds i^{nY} and the
// factor 2 into a sign and scale per string.
//
// One pass serves many strings. The strings' x masks span a space V of index
// offsets; a thread loads one whole coset i ^ V (2^R units of 16 bytes) and has
// every pair of every mask of V in registers, so a pass over the state serves
// all strings whose mask lies in V -- up to R independent masks and their
// products, the x = 0 strings, and for complex64 bit 0, which every unit
// spans -- where one pass per mask read the state once for each. The signs
// (-1)^{popcount(i & z)} of a coset's pairs are a product of one sign per basis
// vector of V, so a string's sum over the coset is a binary tree of fused
// multiply-adds with those signs, times the coset's own sign.
//
// What bounds it: HBM (one read of the state per pass) in complex64 with R = 4:
// 24 fermionic terms with 8 masks on 28 qubits are two passes, 0.78 ms (one pass a
// mask: 4.0 ms). complex128 is bound by FP64 (2 per pair and mask, 1 per pair and string).
//
// Precision. Terms are formed in the state's precision. For complex64 a
// string's terms of one coset (at most 16 pairs, or 32 squares) are added in
// FP32 along the tree, so that sum carries a relative rounding error of at most
// 6 u (u = 2^-24) of the sum of its terms' magnitudes (8 u for up to 8 terms in
// sequence before); the sums are accumulated per thread in FP32 with
// compensation (about 2 u) and added in FP64 across threads and blocks. Since
// sum_i |w_i| <= <psi|psi> and a pair's term carries a factor 2, the absolute
// error of a complex64 expectation value is at most about 1.2e-6 <psi|psi>
// (typically far less). complex128 uses FP64 throughout. Block partials are
// reduced by a second kernel in a fixed order, so results are bitwise
// reproducible for a given launch shape.
#include <algorithm>
#include <vector>

#include "sv_internal.h"

namespace svk {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxS = 16;     // strings of a pass (their running sums live in shared memory)
constexpr int kMaxR = 4;      // basis vectors of a pass

template <typename R> struct Amp;
template <> struct Amp<float> { using T = float2; static constexpr int V = 2, vb = 1; };
template <> struct Amp<double> { using T = double2; static constexpr int V = 1, vb = 0; };

__device__ __forceinline__ float fmar(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmar(double a, double b, double c) { return __fma_rn(a, b, c); }

// Strings that share a mask and a part (Re or Im): one set of pair terms.
struct PauliSet {
    int xi;               // the mask's coordinates: bit 0 of complex64, then the basis vectors
    int im;
    int begin, end;       // strings
};

template <typename R> struct PauliPassK {
    int piv[kMaxR];                       // pivot bits of the basis, ascending (unit index)
    uint64_t comb[1 << kMaxR];            // XOR of the basis vectors of every subset (unit index)
    int n_sets, n_str;
    PauliSet set[kMaxS];
    uint64_t z[kMaxS];
    R sg[kMaxS][kMaxR + 1];               // tree signs, in the order of the terms' index bits
};

struct FinishK {
    double scale[kMaxS];
    int slot[kMaxS];
};

// sum of t[i] times the product of sg[b] over the set bits b of i
template <typename R, int N> __device__ __forceinline__ R tree(const R (&t)[N], const R *sg) {
    if constexpr (N == 1) {
        return t[0];
    } else {
        R u[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) u[i] = fmar(t[2 * i + 1], sg[0], t[2 * i]);
        return tree<R, N / 2>(u, sg + 1);
    }
}

constexpr __host__ __device__ int top_bit(int x) { return x <= 1 ? 0 : 1 + top_bit(x >> 1); }

// terms of the pairs {j, j ^ X}, j without X's highest bit, in ascending order
template <int X, bool IM, typename R, typename C, int NA>
__device__ __forceinline__ void pair_terms(const C (&a)[NA], R (&t)[NA / 2]) {
    constexpr int hb = top_bit(X), low = (1 << hb) - 1;
#pragma unroll
    for (int p = 0; p < NA / 2; ++p) {
        const C &u = a[((p & ~low) << 1) | (p & low)], &v = a[(((p & ~low) << 1) | (p & low)) ^ X];
        t[p] = IM ? fmar(u.y, v.x, -(u.x * v.y)) : fmar(u.x, v.x, u.y * v.y);
    }
}

__device__ __forceinline__ void opaque(float2 &a) { asm volatile("" : "+f"(a.x), "+f"(a.y)); }
__device__ __forceinline__ void opaque(double2 &a) { asm volatile("" : "+d"(a.x), "+d"(a.y)); }

// running sums: compensated (Neumaier) FP32 for complex64, where GB300's FP64
// rate would hold the pass back, FP64 for complex128
__device__ __forceinline__ void add_to(float2 &s, float x) {
    const float t = s.x + x;
    s.y += fabsf(s.x) >= fabsf(x) ? (s.x - t) + x : (x - t) + s.x;
    s.x = t;
}
__device__ __forceinline__ void add_to(double &s, double x) { s += x; }
__device__ __forceinline__ double total(const float2 &s) { return (double)s.x + (double)s.y; }
__device__ __forceinline__ double total(double s) { return s; }

// The set's terms, then `use` on them: the mask is uniform, so one leaf runs,
// with every register index a constant.
template <typename R, int LO, int HI, typename C, int NA, typename F>
__device__ __forceinline__ void each_set(int x, const C (&a)[NA], F use, int im) {
    if constexpr (HI - LO > 1) {
        constexpr int mid = (LO + HI) / 2;
        if (x < mid) each_set<R, LO, mid>(x, a, use, im);
        else each_set<R, mid, HI>(x, a, use, im);
    } else if constexpr (LO == 0) {
        R t[NA];
#pragma unroll
        for (int j = 0; j < NA; ++j) t[j] = fmar(a[j].x, a[j].x, a[j].y * a[j].y);
        use(t);
    } else {
        R t[NA / 2];
        if (im) {
            pair_terms<LO, true>(a, t);
            use(t);
        } else {
            pair_terms<LO, false>(a, t);
            use(t);
        }
    }
}

template <typename R> struct Run;
template <> struct Run<float> { using T = float2; };
template <> struct Run<double> { using T = double; };

template <typename R, int RB>
__global__ void __launch_bounds__(kThreads, RB == 4 ? 2 : 3)
k_pauli(const typename Amp<R>::T *__restrict__ sv, uint64_t n_cosets, const __grid_constant__ PauliPassK<R> P,
        double *__restrict__ partials) {
    using C = typename Amp<R>::T;
    using Acc = typename Run<R>::T;
    constexpr int V = Amp<R>::V, NU = 1 << RB, NA = NU * V;
    __shared__ Acc run[kMaxS][kThreads];
    for (int s = 0; s < P.n_str; ++s) run[s][threadIdx.x] = Acc{};
    const uint64_t stride = (uint64_t)gridDim.x * kThreads;
    for (uint64_t w = (uint64_t)blockIdx.x * kThreads + threadIdx.x; w < n_cosets; w += stride) {
        uint64_t u = w;
#pragma unroll
        for (int i = 0; i < RB; ++i) {
            const uint64_t lo = u & ((1ull << P.piv[i]) - 1ull);
            u = ((u ^ lo) << 1) | lo;
        }
        C a[NA];
#pragma unroll
        for (int j = 0; j < NU; ++j) {
            if constexpr (V == 2) {
                const float4 f = reinterpret_cast<const float4 *>(sv)[u ^ P.comb[j]];
                a[2 * j] = C{f.x, f.y};
                a[2 * j + 1] = C{f.z, f.w};
            } else {
                a[j] = sv[u ^ P.comb[j]];
            }
        }
        const uint64_t amp = u * V;
        for (int m = 0; m < P.n_sets; ++m) {
            // the terms of every mask are invariant in this loop; without this the compiler
            // forms all of them before it, far beyond the registers
#pragma unroll
            for (int j = 0; j < NA; ++j) opaque(a[j]);
            each_set<R, 0, NA>(P.set[m].xi, a, [&](auto &t) {
                for (int s = P.set[m].begin; s < P.set[m].end; ++s) {
                    const R x = tree(t, P.sg[s]);
                    const uint64_t b = amp & P.z[s];
                    add_to(run[s][threadIdx.x], (__popc((uint32_t)b ^ (uint32_t)(b >> 32)) & 1) ? -x : x);
                }
            }, P.set[m].im);
        }
    }
    __shared__ double red[kThreads / 32][kMaxS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int s = 0; s < P.n_str; ++s) {
        double x = total(run[s][threadIdx.x]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[warp][s] = x;
    }
    __syncthreads();
    if (threadIdx.x < P.n_str) {
        double acc = 0.0;
        for (int k = 0; k < kThreads / 32; ++k) acc += red[k][threadIdx.x];
        partials[(size_t)blockIdx.x * kMaxS + threadIdx.x] = acc;
    }
}

// out[slot[s]] = scale[s] times the blocks' sums of string s in a fixed order; one block per string
__global__ void __launch_bounds__(kThreads)
k_pauli_finish(const double *__restrict__ partials, int nblocks, const __grid_constant__ FinishK F, double *__restrict__ out) {
    __shared__ double red[kThreads / 32];
    const int s = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double x = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kThreads) x += partials[(size_t)b * kMaxS + s];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) red[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        double acc = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) acc += red[w];
        out[F.slot[s]] = F.scale[s] * acc;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int high_bit(uint64_t v) { return 63 - __builtin_clzll(v); }

// A fully reduced basis: each vector's highest bit (its pivot) is in no other vector,
// so a member's coordinates are its pivot bits. High pivots leave the low index
// bits to consecutive threads (contiguous reads).
struct Basis {
    std::vector<uint64_t> v;
    uint64_t reduce(uint64_t x) const {
        for (uint64_t b : v)
            if ((x >> high_bit(b)) & 1u) x ^= b;
        return x;
    }
    bool insert(uint64_t x) {
        x = reduce(x);
        if (x == 0) return false;
        for (uint64_t &b : v)
            if ((b >> high_bit(x)) & 1u) b ^= x;
        v.push_back(x);
        return true;
    }
};

template <typename R, int RB>
cudaError_t run_pass(const LaunchCtx &L, const void *sv, uint64_t n_units, const PauliPassK<R> &P, const FinishK &F,
                     double *d_partials, int max_blocks, double *d_out) {
    const uint64_t n_cosets = n_units >> RB;
    uint64_t grid = (n_cosets + kThreads - 1) / kThreads;
    grid = std::min<uint64_t>(grid, std::min<uint64_t>((uint64_t)L.num_sms * (RB == 4 ? 2 : 3), (uint64_t)max_blocks));
    k_pauli<R, RB><<<(unsigned)grid, kThreads, 0, L.stream>>>(reinterpret_cast<const typename Amp<R>::T *>(sv), n_cosets,
                                                              P, d_partials);
    ++*L.launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_pauli_finish<<<(unsigned)P.n_str, kThreads, 0, L.stream>>>(d_partials, (int)grid, F, d_out);
    ++*L.launches;
    return cudaGetLastError();
}

template <typename R>
cudaError_t pauli_terms(const LaunchCtx &L, const void *sv, int n, const PauliTerm *terms, int count,
                        double *d_partials, int max_blocks, double *d_out) {
    constexpr int vb = Amp<R>::vb;
    const int ub = n - vb;                                     // unit-index bits
    const uint64_t n_units = 1ull << ub;
    const int rmax = std::min(ub, sizeof(R) == 4 ? 4 : 3);
    // masks with X/Y sites first: the strings of Z and I fit into any pass
    std::vector<int> left(count);
    for (int i = 0; i < count; ++i) left[i] = i;
    std::stable_sort(left.begin(), left.end(), [&](int a, int b) { return (terms[a].x >> vb) > (terms[b].x >> vb); });
    while (!left.empty()) {
        Basis B;
        std::vector<int> take, keep;
        for (int i : left) {
            const uint64_t x = terms[i].x >> vb;
            bool in = (int)take.size() < kMaxS;
            if (in && B.reduce(x) != 0) {
                in = (int)B.v.size() < rmax;
                if (in) B.insert(x);
            }
            (in ? take : keep).push_back(i);
        }
        left = keep;
        // three vectors at least (loads in flight): free index bits from the top
        const int rb = (int)B.v.size() > 3 ? 4 : std::min(rmax, 3);
        for (int q = ub - 1; (int)B.v.size() < rb; --q) B.insert(1ull << q);
        std::sort(B.v.begin(), B.v.end(), [](uint64_t a, uint64_t b) { return high_bit(a) < high_bit(b); });
        PauliPassK<R> P{};
        FinishK F{};
        for (int i = 0; i < rb; ++i) P.piv[i] = high_bit(B.v[i]);
        for (int j = 0; j < (1 << rb); ++j)
            for (int i = 0; i < rb; ++i)
                if ((j >> i) & 1) P.comb[j] ^= B.v[i];
        auto coords = [&](uint64_t x) {
            int c = vb ? (int)(x & 1u) : 0;
            for (int i = 0; i < rb; ++i) c |= (int)((x >> (P.piv[i] + vb)) & 1u) << (i + vb);
            return c;
        };
        auto key = [&](int i) { return 2 * coords(terms[i].x) + (terms[i].ny & 1); };
        std::stable_sort(take.begin(), take.end(), [&](int a, int b) { return key(a) < key(b); });
        for (int i : take) {
            const PauliTerm &t = terms[i];
            const int s = P.n_str++, c = coords(t.x), im = t.ny & 1;
            if (P.n_sets == 0 || P.set[P.n_sets - 1].xi != c || P.set[P.n_sets - 1].im != im)
                P.set[P.n_sets++] = PauliSet{c, im, s, s};
            P.set[P.n_sets - 1].end = s + 1;
            P.z[s] = t.z;
            int b = 0;
            for (int k = 0; k < rb + vb; ++k) {
                if (c != 0 && k == high_bit((uint64_t)c)) continue;          // the bit that pairs the partners
                const uint64_t off = k < vb ? 1ull : B.v[k - vb] << vb;
                P.sg[s][b++] = __builtin_popcountll(off & t.z) & 1 ? R(-1) : R(1);
            }
            // Re(i^{nY} s w): +Re w, -Im w, -Re w, +Im w for nY = 0, 1, 2, 3 (mod 4)
            const int r = t.ny & 3;
            F.scale[s] = ((r == 1 || r == 2) ? -1.0 : 1.0) * (c == 0 ? 1.0 : 2.0);
            F.slot[s] = i;
        }
        cudaError_t e = cudaErrorInvalidValue;
        if (rb == 0) e = run_pass<R, 0>(L, sv, n_units, P, F, d_partials, max_blocks, d_out);
        if (rb == 1) e = run_pass<R, 1>(L, sv, n_units, P, F, d_partials, max_blocks, d_out);
        if (rb == 2) e = run_pass<R, 2>(L, sv, n_units, P, F, d_partials, max_blocks, d_out);
        if (rb == 3) e = run_pass<R, 3>(L, sv, n_units, P, F, d_partials, max_blocks, d_out);
        if constexpr (sizeof(R) == 4)
            if (rb == 4) e = run_pass<R, 4>(L, sv, n_units, P, F, d_partials, max_blocks, d_out);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_pauli(const LaunchCtx &L, sv_dtype_t dt, const void *sv, int n, const PauliTerm *terms, int count,
                         double *d_partials, int n_partials, double *d_out) {
    if (n < 1) return cudaErrorInvalidValue;
    return dt == SV_C64 ? pauli_terms<float>(L, sv, n, terms, count, d_partials, n_partials / kMaxS, d_out)
                        : pauli_terms<double>(L, sv, n, terms, count, d_partials, n_partials / kMaxS, d_out);
}

}  // namespace svk
