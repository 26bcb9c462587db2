// k_reduce.cu -- reductions over the state vector: parity probabilities of a
// Z-product-basis measurement and its collapse (Table I, "Measurement"), the
// norm, the sampler and <Z_q> of every qubit. (Pauli strings: k_pauli.cu.)
//
// Terms are formed in the state's precision; complex64 sums are FP32 over a few
// terms and FP64 beyond, complex128 uses FP64 throughout. Block partials are
// reduced by a second kernel in a fixed order, so results are bitwise
// reproducible for a given launch shape.
#include "sv_internal.h"

namespace svk {
namespace {

constexpr int kThreads = 256;
constexpr int kIlp = 4;     // work items loaded before any is consumed
constexpr int kRun = 1;     // loop iterations summed in FP32 before an FP64 add

template <typename R> struct CT;
template <> struct CT<float> { using T = float2; static constexpr int V = 2; };
template <> struct CT<double> { using T = double2; static constexpr int V = 1; };

// V consecutive amplitudes starting at unit index u (16-byte load either way)
template <typename R>
__device__ __forceinline__ void load_unit(const typename CT<R>::T *sv, uint64_t u, typename CT<R>::T (&a)[CT<R>::V]) {
    if constexpr (CT<R>::V == 2) {
        const float4 f = reinterpret_cast<const float4 *>(sv)[u];
        a[0] = float2{f.x, f.y};
        a[1] = float2{f.z, f.w};
    } else {
        a[0] = sv[u];
    }
}

template <int S>
__device__ __forceinline__ void block_reduce_store(double (&v)[S], int nS, double *out) {
    __shared__ double red[kThreads / 32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        double x = v[s];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[warp][s] = x;
    }
    __syncthreads();
    if (threadIdx.x < nS) {
        double acc = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) acc += red[w][threadIdx.x];
        out[threadIdx.x] = acc;
    }
}

// partials[b * 8 + s] summed over b in a fixed order
__global__ void __launch_bounds__(kThreads)
k_finish(const double *__restrict__ partials, int nblocks, int S, double *__restrict__ out) {
    __shared__ double red[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int s = 0; s < S; ++s) {
        double x = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += kThreads) x += partials[(size_t)b * 8 + s];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[warp] = x;
        __syncthreads();
        if (threadIdx.x == 0) {
            double acc = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) acc += red[w];
            out[s] = acc;
        }
        __syncthreads();
    }
}

template <typename R>
__global__ void __launch_bounds__(kThreads)
k_parity(const typename CT<R>::T *__restrict__ sv, uint64_t n_units, uint64_t mask, double *__restrict__ partials) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V;
    double tot[2] = {0.0, 0.0};
    R run[2] = {R(0), R(0)};
    const uint64_t stride = (uint64_t)gridDim.x * kThreads * kIlp;
    int iter = 0;
    for (uint64_t u0 = (uint64_t)blockIdx.x * kThreads * kIlp + threadIdx.x; u0 < n_units; u0 += stride) {
        C A[kIlp][V];
#pragma unroll
        for (int q = 0; q < kIlp; ++q)
            if (u0 + (uint64_t)q * kThreads < n_units) load_unit<R>(sv, u0 + (uint64_t)q * kThreads, A[q]);
#pragma unroll
        for (int q = 0; q < kIlp; ++q) {
            const uint64_t u = u0 + (uint64_t)q * kThreads;
            if (u >= n_units) continue;
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const R p = A[q][e].x * A[q][e].x + A[q][e].y * A[q][e].y;
                if (__popcll((u * V + e) & mask) & 1) run[1] += p; else run[0] += p;
            }
        }
        if (++iter == kRun) {
            tot[0] += (double)run[0];
            tot[1] += (double)run[1];
            run[0] = run[1] = R(0);
            iter = 0;
        }
    }
    tot[0] += (double)run[0];
    tot[1] += (double)run[1];
    block_reduce_store<2>(tot, 2, partials + (size_t)blockIdx.x * 8);
}

// A unit whose amplitudes are all dropped is written without being read: 1.5
// instead of 2 passes' bytes where the mask's lowest bit is 9
// (27 qubits, two qubits measured: 0.304 -> 0.235 ms).
template <typename R>
__global__ void __launch_bounds__(kThreads)
k_collapse(typename CT<R>::T *__restrict__ sv, uint64_t n_units, uint64_t mask, int parity, R scale) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V;
    const uint64_t u = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
    if (u >= n_units) return;
    const int par = (int)(__popcll((u * V) & mask) & 1);
    bool keep[V], any = false;
#pragma unroll
    for (int e = 0; e < V; ++e) {
        keep[e] = (par ^ (e & (int)mask & 1)) == parity;
        any |= keep[e];
    }
    C A[V];
#pragma unroll
    for (int e = 0; e < V; ++e) A[e] = C{R(0), R(0)};
    if (any) load_unit<R>(sv, u, A);
#pragma unroll
    for (int e = 0; e < V; ++e) {
        A[e].x = keep[e] ? A[e].x * scale : R(0);
        A[e].y = keep[e] ? A[e].y * scale : R(0);
    }
    if constexpr (V == 2) {
        reinterpret_cast<float4 *>(sv)[u] = make_float4(A[0].x, A[0].y, A[1].x, A[1].y);
    } else {
        sv[u] = A[0];
    }
}

template <typename R>
__global__ void k_set_one(typename CT<R>::T *sv, uint64_t index) {
    sv[index] = typename CT<R>::T{R(1), R(0)};
}

inline int reduce_grid(const LaunchCtx &L, uint64_t work, int max_blocks) {
    uint64_t b = (work + (uint64_t)kThreads * kIlp - 1) / ((uint64_t)kThreads * kIlp);
    uint64_t cap = (uint64_t)L.num_sms * 8;
    if (cap > (uint64_t)max_blocks) cap = (uint64_t)max_blocks;
    if (b > cap) b = cap;
    return (int)(b == 0 ? 1 : b);
}

template <typename R>
cudaError_t parity_t(const LaunchCtx &L, const void *sv, int n, uint64_t mask, double *d_partials, int maxb,
                     double *d_out) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V;
    const uint64_t n_units = (1ull << n) / V;
    const int grid = reduce_grid(L, n_units, maxb);
    k_parity<R><<<grid, kThreads, 0, L.stream>>>(reinterpret_cast<const C *>(sv), n_units, mask, d_partials);
    ++*L.launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_finish<<<1, kThreads, 0, L.stream>>>(d_partials, grid, 2, d_out);
    ++*L.launches;
    return cudaGetLastError();
}

template <typename R>
cudaError_t collapse_t(const LaunchCtx &L, void *sv, int n, uint64_t mask, int parity, double scale) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V;
    const uint64_t n_units = (1ull << n) / V;
    const uint64_t grid = (n_units + kThreads - 1) / kThreads;
    k_collapse<R><<<(unsigned)grid, kThreads, 0, L.stream>>>(reinterpret_cast<C *>(sv), n_units, mask, parity,
                                                             (R)scale);
    ++*L.launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sampler (Table I, "Sampler"): measurement outcomes without collapse. The
// state is cut into segments of 2^seg_log amplitudes; their probabilities are
// summed (FP32 runs of 16 terms, FP64 beyond, fixed order), the segment sums
// are scanned into a cumulative distribution by one block in a fixed order,
// and each sample -- one warp -- binary-searches the segment and scans it for
// the first index whose cumulative probability exceeds r * total.
// ---------------------------------------------------------------------------

// What bounds it: HBM (one read of the state). A thread's 16 loads are issued
// before their terms are added (27 qubits, complex64: one load at a time 0.690
// ms, 1.6 TB/s).
template <typename R>
__global__ void __launch_bounds__(kThreads)
k_seg_sums(const typename CT<R>::T *__restrict__ sv, int seg_log, uint64_t n_seg, double *__restrict__ seg) {
    using C = typename CT<R>::T;
    __shared__ double red[kThreads / 32];
    const uint64_t S = 1ull << seg_log;
    constexpr int kAhead = sizeof(R) == 4 ? 16 : 8;     // 128 bytes in flight
    for (uint64_t g = blockIdx.x; g < n_seg; g += gridDim.x) {
        const C *src = sv + g * S + threadIdx.x;
        double acc = 0.0;
        R run = R(0);
        if (S >= 16ull * kThreads) {
            for (uint64_t i = 0; i < S; i += 16ull * kThreads) {
#pragma unroll
                for (int h = 0; h < 16; h += kAhead) {
                    C a[kAhead];
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) a[k] = src[i + (uint64_t)(h + k) * kThreads];
#pragma unroll
                    for (int k = 0; k < kAhead; ++k) run += a[k].x * a[k].x + a[k].y * a[k].y;
                }
                acc += (double)run;
                run = R(0);
            }
        } else {                                         // at most 16 terms
            for (uint64_t i = threadIdx.x; i < S; i += kThreads) {
                const C a = sv[g * S + i];
                run += a.x * a.x + a.y * a.y;
            }
        }
        acc += (double)run;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) t += red[w];
            seg[g] = t;
        }
        __syncthreads();
    }
}

// Inclusive scan of seg[0 .. n) in place, one block of 1024 threads, fixed
// order. Latency-bound: loads go eight at a time ahead of the additions.
__global__ void __launch_bounds__(1024) k_scan(double *__restrict__ seg, uint64_t n) {
    __shared__ double part[1024];
    const uint64_t per = (n + 1023) / 1024;
    const uint64_t b = threadIdx.x * per, e = (b + per < n) ? b + per : n;
    auto each8 = [&](auto use) {
        for (uint64_t i = b; i < e; i += 8) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = i + k < e ? seg[i + k] : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (i + k < e) use(i + k, v[k]);
        }
    };
    double run = 0.0;
    each8([&](uint64_t i, double v) {
        run += v;
        seg[i] = run;
    });
    part[threadIdx.x] = run;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < 1024; i += 8) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = part[i + k];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                part[i + k] = t;
                t += v[k];
            }
        }
    }
    __syncthreads();
    const double off = part[threadIdx.x];
    each8([&](uint64_t i, double v) { seg[i] = v + off; });
}

// |a|^2 of up to kLane consecutive amplitudes to about FP64's accuracy: for
// complex64 as an FP32 pair (exact products by fused multiply-adds, exact
// additions after Knuth), because FP64 runs at 2 operations per SM and clock.
struct PairSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float h = x * x, l = __fmaf_rn(x, x, -h);
        const float t = s + h, z = t - s;
        c += ((s - (t - z)) + (h - z)) + l;
        s = t;
    }
};
__device__ __forceinline__ double prob(const float2 &a) { return (double)a.x * (double)a.x + (double)a.y * (double)a.y; }
__device__ __forceinline__ double prob(const double2 &a) { return a.x * a.x + a.y * a.y; }

constexpr int kLane = 16;

// One warp per sample. A lane sums 16 consecutive amplitudes, a warp scan over
// the 32 lanes' sums finds the lane that holds the outcome, and a second scan
// its amplitude: one scan per 512 amplitudes and one more, where a scan per 32
// amplitudes was bound by FP64 and by the latency of its serial loads (20000
// samples of a 27-qubit state: 1.21 ms).
template <typename R>
__global__ void __launch_bounds__(kThreads)
k_sample(const typename CT<R>::T *__restrict__ sv, int seg_log, uint64_t n_seg, const double *__restrict__ seg,
         const double *__restrict__ rands, int n_samples, long long *__restrict__ out) {
    using C = typename CT<R>::T;
    const int lane = threadIdx.x & 31;
    const int sidx = (int)((blockIdx.x * (uint64_t)kThreads + threadIdx.x) >> 5);
    if (sidx >= n_samples) return;
    const double total = seg[n_seg - 1];
    const double target = rands[sidx] * total;
    uint64_t lo = 0, hi = n_seg - 1;            // first segment with cum > target
    while (lo < hi) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (seg[mid] > target) hi = mid; else lo = mid + 1;
    }
    const double before = lo > 0 ? seg[lo - 1] : 0.0;
    const double want = target - before;
    const uint64_t S = 1ull << seg_log, base = lo * S;
    auto scan = [&](double x) {                 // inclusive
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        return x;
    };
    // the amplitudes c .. c + 15 of the segment: the first whose cumulative sum (from `sum`
    // on) passes `limit`, else the last one that is not zero
    auto locate = [&](uint64_t c, double sum, double limit) {
        const double p = lane < kLane && c + lane < S ? prob(sv[base + c + lane]) : 0.0;
        const double inc = scan(p);
        const unsigned hit = __ballot_sync(0xffffffffu, sum + inc > limit && p > 0.0);
        const unsigned nz = __ballot_sync(0xffffffffu, p > 0.0);
        return (long long)(base + c + (hit ? __ffs(hit) - 1 : nz ? 31 - __clz(nz) : 0));
    };
    double running = 0.0;
    uint64_t last = 0;                          // the last lane's run that is not all zero
    for (uint64_t c = 0; c < S; c += 32 * kLane) {
        const uint64_t at = c + (uint64_t)lane * kLane;
        double p = 0.0;
        if (at + kLane <= S) {
            if constexpr (sizeof(R) == 4) {
                float4 v[kLane / 2];
#pragma unroll
                for (int k = 0; k < kLane / 2; ++k) v[k] = reinterpret_cast<const float4 *>(sv + base + at)[k];
                PairSum q;
#pragma unroll
                for (int k = 0; k < kLane / 2; ++k) {
                    q.add(v[k].x);
                    q.add(v[k].y);
                    q.add(v[k].z);
                    q.add(v[k].w);
                }
                p = (double)q.s + (double)q.c;
            } else {
#pragma unroll
                for (int k = 0; k < kLane; ++k) p += prob(sv[base + at + k]);
            }
        } else {
            for (uint64_t k = at; k < S && k < at + kLane; ++k) p += prob(sv[base + k]);
        }
        const double inc = scan(p);
        double excl = __shfl_up_sync(0xffffffffu, inc, 1);
        if (lane == 0) excl = 0.0;
        const unsigned hit = __ballot_sync(0xffffffffu, running + inc > want && p > 0.0);
        if (hit) {
            const int L = __ffs(hit) - 1;
            const long long i = locate(c + (uint64_t)L * kLane, running + __shfl_sync(0xffffffffu, excl, L), want);
            if (lane == 0) out[sidx] = i;
            return;
        }
        const unsigned nz = __ballot_sync(0xffffffffu, p > 0.0);
        if (nz) last = c + (uint64_t)(31 - __clz(nz)) * kLane;
        running += __shfl_sync(0xffffffffu, inc, 31);
    }
    // rounding left the target past the segment's own sum: its last nonzero amplitude
    const long long i = locate(last, 0.0, 1e300);
    if (lane == 0) out[sidx] = i;
}

template <typename R>
cudaError_t sample_t(const LaunchCtx &L, const void *sv, int n, const double *d_r, int ns, double *d_seg,
                     long long *d_out) {
    using C = typename CT<R>::T;
    int seg_log = n - 20 > 12 ? n - 20 : 12;
    if (seg_log > n) seg_log = n;
    const uint64_t n_seg = 1ull << (n - seg_log);
    uint64_t grid = n_seg;
    const uint64_t cap = (uint64_t)L.num_sms * 8;
    if (grid > cap) grid = cap;
    k_seg_sums<R><<<(unsigned)grid, kThreads, 0, L.stream>>>(reinterpret_cast<const C *>(sv), seg_log, n_seg, d_seg);
    ++*L.launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_scan<<<1, 1024, 0, L.stream>>>(d_seg, n_seg);
    ++*L.launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const uint64_t blocks = ((uint64_t)ns * 32 + kThreads - 1) / kThreads;
    k_sample<R><<<(unsigned)blocks, kThreads, 0, L.stream>>>(reinterpret_cast<const C *>(sv), seg_log, n_seg, d_seg,
                                                             d_r, ns, d_out);
    ++*L.launches;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// <Z_q> for every qubit in one pass: with p_i = |psi_i|^2 and S_q the sum of
// p_i over indices with bit q set, <Z_q> = sum_i p_i - 2 S_q. A block owns an
// aligned range of 16-byte units; from the lowest, the unit index's bits are
// the lane, the warp, one of 8 loads, the iteration, and the block. Bits inside
// a thread (the pair of a complex64 unit, the loads, the iterations) have a
// partial sum each, lane and warp bits select whole thread totals, and block
// bits are left to k_zall_finish, which takes one block per qubit. FP32 for
// complex64 over at most 4 iterations of 16 amplitudes (a tree over the 16),
// FP64 beyond; fixed order.
//
// What bounds it: HBM; 128 bytes per thread are in flight (27 qubits, complex64:
// 0.318 ms with 64 strided bytes in flight, and 0.087 ms for the finish in one
// block).
// ---------------------------------------------------------------------------
constexpr int kZMax = 40;
constexpr int kZIn = 2;       // iterations summed in the state's precision: 2^kZIn
constexpr int kZOuter = 20;   // most iteration bits beyond those
constexpr int kZFew = 6;      // the same for states whose blocks take at most 2^8 iterations

template <typename R, int MO>
__global__ void __launch_bounds__(kThreads)
k_zall(const typename CT<R>::T *__restrict__ sv, uint64_t n_units, int mj, double *__restrict__ partials) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V, vb = V == 2 ? 1 : 0;
    const int t = threadIdx.x;
    const uint64_t u0 = ((uint64_t)blockIdx.x << (11 + mj)) + t;
    const int inner = mj < kZIn ? 1 << mj : 1 << kZIn, mo = mj < kZIn ? 0 : mj - kZIn;
    double dT = 0.0, dE = 0.0, dL[3] = {0.0, 0.0, 0.0}, dI[kZIn] = {0.0}, dO[MO > 0 ? MO : 1];
#pragma unroll
    for (int q = 0; q < MO; ++q) dO[q] = 0.0;
    for (uint32_t j = 0; j < (1u << mo); ++j) {
        R fT = R(0), fE = R(0), fL[3] = {R(0), R(0), R(0)}, fI[kZIn] = {R(0)};
        for (int i = 0; i < inner; ++i) {
            const uint64_t u = u0 + ((uint64_t)((j << kZIn) + i) << 11);
            C a[8][V];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (u + k * kThreads < n_units) {
                    load_unit<R>(sv, u + k * kThreads, a[k]);
                } else {
#pragma unroll
                    for (int e = 0; e < V; ++e) a[k][e] = C{R(0), R(0)};
                }
            }
            R p[8], h[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                p[k] = a[k][0].x * a[k][0].x + a[k][0].y * a[k][0].y;
                if constexpr (V == 2) {
                    h[k] = a[k][V - 1].x * a[k][V - 1].x + a[k][V - 1].y * a[k][V - 1].y;
                    p[k] += h[k];
                }
            }
            const R p23 = p[2] + p[3], p67 = p[6] + p[7], hi = (p[4] + p[5]) + p67;
            const R tot = ((p[0] + p[1]) + p23) + hi;
            fT += tot;
            if constexpr (V == 2) fE += ((h[0] + h[1]) + (h[2] + h[3])) + ((h[4] + h[5]) + (h[6] + h[7]));
            fL[0] += (p[1] + p[3]) + (p[5] + p[7]);
            fL[1] += p23 + p67;
            fL[2] += hi;
#pragma unroll
            for (int q = 0; q < kZIn; ++q)
                if ((i >> q) & 1) fI[q] += tot;
        }
        dT += (double)fT;
        dE += (double)fE;
#pragma unroll
        for (int q = 0; q < 3; ++q) dL[q] += (double)fL[q];
#pragma unroll
        for (int q = 0; q < kZIn; ++q) dI[q] += (double)fI[q];
#pragma unroll
        for (int q = 0; q < MO; ++q)
            if (q < mo && ((j >> q) & 1u)) dO[q] += (double)fT;
    }
    // block sums in a fixed order: value 0 is the total, value 1 + q the sum over bit q of
    // the block's amplitude index; each warp reduces with shuffles, then thread v adds
    // the warps' results in warp order
    constexpr int kV = 1 + vb + 5 + 3 + 3 + kZIn + MO;
    __shared__ double wred[kThreads / 32][kV];
    const int lane = t & 31, warp = t >> 5;
    const int nv = 1 + vb + 11 + mj;
    auto warp_put = [&](double x, int v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) wred[warp][v] = x;
    };
    // the total and the lane bits in one reduction: merging over bit b, the upper half's
    // total becomes that bit's sum
    double tot = dT, lb[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const double other = __shfl_xor_sync(0xffffffffu, tot, 1 << b);
#pragma unroll
        for (int c = 0; c < b; ++c) lb[c] += __shfl_xor_sync(0xffffffffu, lb[c], 1 << b);
        lb[b] = (lane >> b) & 1 ? tot : other;
        tot += other;
    }
    if (lane == 0) {
        wred[warp][0] = tot;
#pragma unroll
        for (int b = 0; b < 5; ++b) wred[warp][1 + vb + b] = lb[b];
#pragma unroll
        for (int b = 0; b < 3; ++b) wred[warp][1 + vb + 5 + b] = (warp >> b) & 1 ? tot : 0.0;
    }
    if constexpr (V == 2) warp_put(dE, 1);
#pragma unroll
    for (int q = 0; q < 3; ++q) warp_put(dL[q], 1 + vb + 8 + q);
#pragma unroll
    for (int q = 0; q < kZIn; ++q)
        if (q < mj) warp_put(dI[q], 1 + vb + 11 + q);
#pragma unroll
    for (int q = 0; q < MO; ++q)
        if (q < mo) warp_put(dO[q], 1 + vb + 11 + kZIn + q);
    __syncthreads();
    if (t < nv) {
        double acc = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) acc += wred[w][t];
        partials[(size_t)t * gridDim.x + blockIdx.x] = acc;
    }
}

// block q < n: out[q] = total - 2 S_q; block n: out[n] = total. in_bits: qubits inside a k_zall block.
__global__ void __launch_bounds__(kThreads)
k_zall_finish(const double *__restrict__ partials, int nblocks, int in_bits, int n, double *__restrict__ out) {
    __shared__ double red[2][kThreads / 32];
    const int q = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double tt = 0.0, a = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kThreads) {
        const double x = partials[b];
        tt += x;
        if (q < in_bits) a += partials[(size_t)(1 + q) * nblocks + b];
        else if ((b >> (q - in_bits)) & 1) a += x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tt += __shfl_xor_sync(0xffffffffu, tt, o);
        a += __shfl_xor_sync(0xffffffffu, a, o);
    }
    if (lane == 0) {
        red[0][warp] = tt;
        red[1][warp] = a;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        tt = a = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) {
            tt += red[0][w];
            a += red[1][w];
        }
        out[q] = q < n ? tt - 2.0 * a : tt;
    }
}

template <typename R>
cudaError_t zall_t(const LaunchCtx &L, const void *sv, int n, double *d_partials, int maxb, double *d_out) {
    using C = typename CT<R>::T;
    constexpr int V = CT<R>::V, vb = V == 2 ? 1 : 0;
    const int ub = n - vb;
    // up to 512 blocks (complex128, whose sums are bound by FP64: 1024) of at least one
    // iteration (2^11 units): all resident, and the closing reductions are few (27 / 28
    // qubits, with the copy of the results: 512 blocks 0.227 / 0.376 ms, 1024 0.246 /
    // 0.397, 2048 0.271 / 0.431)
    constexpr int zb = V == 2 ? 9 : 10;
    const int mj = ub > 11 + zb ? ub - 11 - zb : 0;
    const uint64_t n_units = 1ull << ub;
    const uint64_t blocks = ub > 11 ? n_units >> (11 + mj) : 1;
    if (mj > kZIn + kZOuter || blocks * (uint64_t)(1 + vb + 11 + mj) > (uint64_t)maxb * 8) return cudaErrorInvalidValue;
    // the sums of the outer iteration bits take two registers each
    auto kern = mj <= kZIn + kZFew ? k_zall<R, kZFew> : k_zall<R, kZOuter>;
    kern<<<(unsigned)blocks, kThreads, 0, L.stream>>>(reinterpret_cast<const C *>(sv), n_units, mj, d_partials);
    ++*L.launches;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_zall_finish<<<(unsigned)(n + 1), kThreads, 0, L.stream>>>(d_partials, (int)blocks, vb + 11 + mj, n, d_out);
    ++*L.launches;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_parity(const LaunchCtx &L, sv_dtype_t dt, const void *sv, int n, uint64_t mask,
                          double *d_partials, int max_partial_blocks, double *d_out) {
    if (n < 1) return cudaErrorInvalidValue;
    return dt == SV_C64 ? parity_t<float>(L, sv, n, mask, d_partials, max_partial_blocks, d_out)
                        : parity_t<double>(L, sv, n, mask, d_partials, max_partial_blocks, d_out);
}

cudaError_t launch_collapse(const LaunchCtx &L, sv_dtype_t dt, void *sv, int n, uint64_t mask, int parity,
                            double scale) {
    if (n < 1) return cudaErrorInvalidValue;
    return dt == SV_C64 ? collapse_t<float>(L, sv, n, mask, parity, scale)
                        : collapse_t<double>(L, sv, n, mask, parity, scale);
}

cudaError_t launch_sample(const LaunchCtx &L, sv_dtype_t dt, const void *sv, int n, const double *d_r, int n_samples,
                          double *d_seg, long long *d_out) {
    if (n < 1 || n_samples < 1) return cudaErrorInvalidValue;
    return dt == SV_C64 ? sample_t<float>(L, sv, n, d_r, n_samples, d_seg, d_out)
                        : sample_t<double>(L, sv, n, d_r, n_samples, d_seg, d_out);
}

cudaError_t launch_zall(const LaunchCtx &L, sv_dtype_t dt, const void *sv, int n, double *d_partials,
                        int max_partial_blocks, double *d_out) {
    if (n < 3 || n > kZMax) return cudaErrorInvalidValue;
    return dt == SV_C64 ? zall_t<float>(L, sv, n, d_partials, max_partial_blocks, d_out)
                        : zall_t<double>(L, sv, n, d_partials, max_partial_blocks, d_out);
}

cudaError_t launch_set_basis(const LaunchCtx &L, sv_dtype_t dt, void *sv, int n, uint64_t index) {
    const size_t bytes = (size_t(1) << n) * (dt == SV_C64 ? 8 : 16);
    cudaError_t e = cudaMemsetAsync(sv, 0, bytes, L.stream);
    if (e != cudaSuccess) return e;
    if (dt == SV_C64)
        k_set_one<float><<<1, 1, 0, L.stream>>>(reinterpret_cast<float2 *>(sv), index);
    else
        k_set_one<double><<<1, 1, 0, L.stream>>>(reinterpret_cast<double2 *>(sv), index);
    ++*L.launches;
    return cudaGetLastError();
}

}  // namespace svk
