// k_tc_x3.cu -- dense gates on 5 and 6 targets of a complex64 state at FP32's
// accuracy on the 5th-generation tensor cores (tcgen05, TMEM accumulators).
//
// On CUDA cores these gates are bound by the FP32 pipe (128 / 256 FMAs per
// amplitude against 16 bytes moved; k_gate.cu). Here both operands are cut into
// BF16 digits and the product is the sum of digit products:
//   state: x = hi + mid + two more. With X a power of two above the largest of the
//     real (or of the imaginary) parts of the column, hi is x rounded to a multiple
//     of X 2^-7, mid the rest rounded to a multiple of X 2^-15, and what is left is
//     rounded to BF16 twice (|x - sum| < X 2^-34). A column is one group of 64
//     amplitudes; its real and imaginary parts are operand rows of their own, so
//     neither other groups nor, under a real matrix, the other parts enter the error;
//   matrix row (real or imaginary parts): four digits in the same way, below 2^-34 of
//     the row's largest.
// hi times hi is summed in an accumulator of its own: all its terms are
// multiples of one unit and the sum stays below 2^20 of them, so it is exact
// whatever rounding the tensor core's FP32 accumulation does (a truncating sum
// of the whole product would shrink the norm by a constant per gate). The other
// products (digits i, j from the top with i + j <= 4: 12 kinds) are at most 2^-7 of
// the first, go into a second accumulator smallest first, and the two are added
// with one rounding. Error per gate: see the rule in tc_x3_ok(). Three state digits and nine products (0.98 to 1.00 ms a gate on
// 28 qubits) kept 25 bits below X: where one amplitude dominates a group the small
// outputs then had up to 700 u sum |m||x|.
//
// The pipeline is k_tc6_raw's (k_tc.cu): the 64 members of a group are the
// contraction, the state tile is the MN-major B operand, its rows are re and im
// of 64 columns; 2 copy warps (cp.async into the stage, arriving on `landed`),
// 8 convert warps (digits in place: a 1 KiB atom of 8 members x 32 floats
// becomes its hi and mid atoms, the other two go to one of two 32 KiB buffers that
// the products give back), one MMA thread, 8 epilogue warps that add the
// accumulators, combine the Re and Im rows, stage the result where the tile came
// from and store it. Tiles are 64 columns (32 KiB), in four stages. The matrix is in
// TMEM, beside the accumulators, because the shared-memory port is what the roles
// share. The twelve small kinds of two tiles have an accumulator each, so the next
// tile's can run while the epilogue reads this one (with one: 1.46 ms a gate, 1.11 so).
//
// A 5-target gate takes one more qubit as the top member bit with an identity:
// the block-diagonal product keeps its halves apart, and each half of a column
// has its own X.
//
// What bounds it: the conversion and the tensor pipe, each close to the 4800 clocks of
// a tile of 64 columns (the convert warps wait in 15 % of them, the thread that issues
// the 52 MMAs in 4 %, the pipe is active in 3430; with 10 or 11 products for matrices
// that need no more, a gate was no faster); HBM needs 3000. 28 qubits, one gate: 1.10 to 1.12 ms for k = 6 (k_dense6 3.30) and
// 1.05 to 1.10 ms for k = 5 (k_dense5 1.38); 1.16 and 1.10 ms with qubit 0 a target
// (3.24 and 1.34). N = 64 MMAs (half-tile accumulators) take as long as N = 128 ones;
// digits by 4 convert warps instead of 8 that hold their atoms in registers, the matrix
// in shared memory and ragged tiles were each slower.
#include <cuda_bf16.h>

#include <cmath>

#include "sv_internal.h"
#include "tc_common.cuh"

namespace svk {
namespace {

constexpr int kNT = 64;                       // columns per tile (MMA N = 2 * kNT reals)
constexpr int kStages = 4;
constexpr int kDigA = 4;
constexpr int kADigit = 128 * 64 * 2;         // one digit of A: 128 rows x 64 BF16
constexpr int kA = kDigA * kADigit;
constexpr int kRaw = 64 * 2 * kNT * 4;        // a tile: 64 members x 128 floats, then its first two digits
constexpr int kLow = kRaw;                    // its last two digits, laid out alike
constexpr int kLows = 2;                      // buffers of those, held from the conversion to the end of the products
constexpr int kCopyWarps = 2, kConvWarps = 8, kEpiWarps = 8;
constexpr int kProdWarps = kCopyWarps + kConvWarps;
constexpr int kMmaWarp = kProdWarps + kEpiWarps;
constexpr int kThreads = (kMmaWarp + 1) * 32;
constexpr int kAccCols = 3 * 2 * kNT;         // hi hi, and the rest of two tiles in turn, 128 columns each
constexpr int kACols = kDigA * 32;            // A in TMEM: row m in lane m, two BF16 per column
constexpr int kTmemCols = 512;                // A, then the accumulators
static_assert(kACols + kAccCols <= kTmemCols, "TMEM");

struct Ctl {
    unsigned long long landed[kStages], full[kStages], empty[kStages], low_free[kLows], acc_full, acc_empty, xch[4], done;
    // non-finite columns of a stage: half of the members, column block; bit c: column c of the block's 16
    unsigned bad[kStages][2][4];
    uint32_t share[2][4][2][16];              // maxima of a column block's halves, two tiles in turn
    unsigned tmem_base;
    int abort;
};
constexpr int kGuard = 2048;                  // unused bytes after the last buffer
constexpr int kSmem = kStages * kRaw + kLows * kLow + kGuard + (int)sizeof(Ctl);
static_assert(kSmem <= 227 * 1024, "dynamic shared memory of the kernel exceeds the per-block limit");

// MN-major operand descriptor of BF16 atoms (8 members x 32 columns, 64-byte
// swizzle): column atoms `lbo` bytes apart, member groups `sbo` bytes apart
__device__ __forceinline__ uint64_t sdesc_b(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;
    d |= (uint64_t)(sbo >> 4) << 32;
    d |= 1ull << 46;
    d |= 4ull << 61;
    return d;
}

// D = F32, A = B = BF16, A K-major, B MN-major (bit 16), N = 128, M = 128
constexpr uint32_t kIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)((2 * kNT) >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// A from TMEM
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(kIdesc), "r"(acc)
        : "memory");
}

__device__ __forceinline__ uint32_t bf16x2(float a, float b) {   // a in the low half
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ float bf16_part(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
        "r"(r[30]), "r"(r[31])
        : "memory");
}

// 16 columns of each of two accumulators, one wait
__device__ __forceinline__ void tmem_ld16x2(uint32_t a0, uint32_t a1, float (&v)[16], float (&w)[16]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(a0), "r"(a1)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        v[i] = __uint_as_float(r[i]);
        w[i] = __uint_as_float(r[16 + i]);
    }
}

// One lane's 8 floats of an atom (two 16-byte chunks); with T0 the rows' halves traded
// as split_atom in k_tc.cu does, so that each row holds its own member.
template <bool T0>
__device__ __forceinline__ void load8(uint32_t addr, int r, float (&x)[8]) {
    // odd rows read their second chunk first: eight lanes (two rows) then cover all banks
    const uint32_t odd = (uint32_t)(r & 1) << 4;
    float y[8];
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(y[0]), "=f"(y[1]), "=f"(y[2]), "=f"(y[3]) : "r"(addr + odd));
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(y[4]), "=f"(y[5]), "=f"(y[6]), "=f"(y[7]) : "r"(addr + (odd ^ 16u)));
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = odd ? y[k ^ 4] : y[k];
    if constexpr (T0) {
        const bool even = (r & 1) == 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float *c = x + 4 * h;
            const float s0 = __shfl_xor_sync(0xffffffffu, even ? c[2] : c[0], 5);
            const float s1 = __shfl_xor_sync(0xffffffffu, even ? c[3] : c[1], 5);
            if (even) {
                c[2] = s0;
                c[3] = s1;
            } else {
                c[0] = s0;
                c[1] = s1;
            }
        }
    }
}

// Half of a column block (32 floats x 32 members, 4 atoms 1 KiB apart) of a landed
// stage into its digits, by one warp, the atoms held in registers. A lane's chunks
// are columns 4 lu .. 4 lu + 3 of row r; lanes with the same lu (lane ^ 5, ^ 10,
// ^ 16) hold the other rows. The real and the imaginary parts of every column have
// a scale each, common to all members (the two warps of a block trade their maxima
// through `share` and the block's barrier), or to the members of one half (halves).
template <bool T0>
__device__ __forceinline__ bool convert_half(uint32_t atoms, uint32_t low_atoms, int lane, int half, int halves,
                                             volatile uint32_t (*share)[16], uint32_t xch, uint32_t parity, unsigned *bad,
                                             volatile int *abort_flag, int *d_err) {
    const int r = lane >> 2, u = lane & 3, lu = u ^ (r & 3);
    const uint32_t src = (uint32_t)(r * 128 + u * 32), dst = (uint32_t)(r * 64 + ((lu ^ ((r >> 1) & 3)) << 4));
    float x[4][8];
    uint32_t top[4] = {0, 0, 0, 0};                      // per column: the upper 16 bits of its largest real and imaginary part
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        load8<T0>(atoms + (uint32_t)(g * 1024) + src, r, x[g]);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            top[c] = __vmaxu2(top[c], __byte_perm(__float_as_uint(x[g][2 * c]), __float_as_uint(x[g][2 * c + 1]), 0x7632) &
                                          0x7fff7fffu);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        top[c] = __vmaxu2(top[c], __shfl_xor_sync(0xffffffffu, top[c], 5));
        top[c] = __vmaxu2(top[c], __shfl_xor_sync(0xffffffffu, top[c], 10));
        top[c] = __vmaxu2(top[c], __shfl_xor_sync(0xffffffffu, top[c], 16));
    }
    if (!halves) {
        if (lane < 4) {                                  // row 0: lu = lane
#pragma unroll
            for (int c = 0; c < 4; ++c) share[half][4 * lane + c] = top[c];
        }
        mbar_arrive(xch);
        if (!mbar_wait(xch, parity, abort_flag, d_err)) return false;
#pragma unroll
        for (int c = 0; c < 4; ++c) top[c] = __vmaxu2(top[c], share[half ^ 1][4 * lu + c]);
    }
    float c1[8];                                         // unit X 2^-7; X 2^-15 is 2^-8 of it
    bool in = true;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        // X = 2^(e - 126); adding and taking away 1.5 2^23 units rounds to a multiple of a unit
        const uint32_t t = (k & 1) ? top[k >> 1] >> 16 : top[k >> 1] & 0xffffu, e = t >> 7;
        const bool ok = (e >= 40 && e <= 230) || t == 0;
        in = in && ok;
        c1[k] = ok ? __uint_as_float((((t == 0 ? 40u : e) + 17u) << 23) | 0x400000u) : 0.f;
    }
    auto second = [](float a) { return __uint_as_float(__float_as_uint(a) - (8u << 23)); };
    if (lane == 0) *bad = 0;
    const bool all_in = __all_sync(0xffffffffu, in);
    unsigned nf = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        float hi[8], mid[8], rest[8];
        uint32_t d[4][4];
        if (all_in) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                hi[k] = __fsub_rn(__fadd_rn(x[g][k], c1[k]), c1[k]);
                rest[k] = __fsub_rn(x[g][k], hi[k]);
                const float c2 = second(c1[k]);
                mid[k] = __fsub_rn(__fadd_rn(rest[k], c2), c2);
                rest[k] = __fsub_rn(rest[k], mid[k]);
            }
        } else {
            // columns beyond the range of the scales: digits by rounding to BF16 (their
            // sums are then rounded by the accumulation); non-finite values are left out
            // and their columns marked
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float v = x[g][k];
                if ((__float_as_uint(v) & 0x7f800000u) == 0x7f800000u) {
                    nf |= 1u << (4 * lu + (k >> 1));
                    v = 0.f;
                }
                const float a = c1[k], b = second(a);
                hi[k] = a != 0.f ? __fsub_rn(__fadd_rn(v, a), a) : bf16_part(v);
                rest[k] = __fsub_rn(v, hi[k]);
                mid[k] = a != 0.f ? __fsub_rn(__fadd_rn(rest[k], b), b) : bf16_part(rest[k]);
                rest[k] = __fsub_rn(rest[k], mid[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // hi and mid are BF16 numbers: their upper halves
            d[0][k] = __byte_perm(__float_as_uint(hi[2 * k]), __float_as_uint(hi[2 * k + 1]), 0x7632);
            d[1][k] = __byte_perm(__float_as_uint(mid[2 * k]), __float_as_uint(mid[2 * k + 1]), 0x7632);
            d[2][k] = bf16x2(rest[2 * k], rest[2 * k + 1]);
            d[3][k] = bf16x2(__fsub_rn(rest[2 * k], __uint_as_float(d[2][k] << 16)),
                             __fsub_rn(rest[2 * k + 1], __uint_as_float(d[2][k] & 0xffff0000u)));
        }
        // (every lane has read all four atoms before the shuffles above)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t o = (i < 2 ? atoms : low_atoms) + (uint32_t)(g * 1024 + (i & 1) * 512) + dst;
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(o), "r"(d[i][0]), "r"(d[i][1]), "r"(d[i][2]), "r"(d[i][3])
                         : "memory");
        }
    }
    if (nf) atomicOr(bad, nf);
    return true;
}

// Copy and store orders as in k_tc.cu: PLAIN (qubit 0 free, lowest target 4 or
// more), MAPPED (the table order, qubit 0 free), T0 (qubit 0 a target).
enum Mode { PLAIN = 0, MAPPED = 1, T0M = 2 };

// halves: the members' top bit is the extra qubit of a 5-target gate (columns of the
// two halves are apart; a non-finite value spoils its half only)
template <int MODE>
__global__ void __launch_bounds__(kThreads, 1)
k_tc_x3(float2 *__restrict__ sv, const __grid_constant__ TcGeom G, const __grid_constant__ RawMap R,
        const uint4 *__restrict__ a_img, int *__restrict__ d_err, int halves) {
    constexpr bool TABLE = MODE != PLAIN, T0 = MODE == T0M;
    extern __shared__ __align__(1024) unsigned char smem_dyn[];
    if (smem_u32(smem_dyn) & 1023u) {
        if (threadIdx.x == 0) atomicExch(d_err, kErrSmemAlign);
        return;
    }
    Ctl &S = *reinterpret_cast<Ctl *>(smem_dyn + kStages * kRaw + kLows * kLow + kGuard);
    const uint32_t sB0 = smem_u32(smem_dyn), sLow0 = sB0 + (uint32_t)(kStages * kRaw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    volatile int *abort_flag = &S.abort;

    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) {
            mbar_init(smem_u32(&S.landed[i]), kCopyWarps * 32);
            mbar_init(smem_u32(&S.full[i]), kConvWarps * 32);
            mbar_init(smem_u32(&S.empty[i]), kEpiWarps * 32);
        }
        for (int i = 0; i < kLows; ++i) mbar_init(smem_u32(&S.low_free[i]), 1);
        mbar_init(smem_u32(&S.acc_full), 1);
        mbar_init(smem_u32(&S.acc_empty), kEpiWarps * 32);
        for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&S.xch[i]), 64);
        mbar_init(smem_u32(&S.done), 1);
        S.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_base;
    const uint64_t ntl = G.n_tiles;
    if (warp >= kProdWarps && warp < kProdWarps + 4) {
        // A into TMEM: this warp's lane quarter (rows 32 (warp & 3) ..), digit by digit
        const int q = warp & 3;
        for (int d = 0; d < kDigA; ++d) {
            uint32_t r[32];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 v = a_img[(d * 128 + 32 * q + lane) * 8 + c];
                r[4 * c] = v.x;
                r[4 * c + 1] = v.y;
                r[4 * c + 2] = v.z;
                r[4 * c + 3] = v.w;
            }
            tmem_st32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(d * 32), r);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp < kCopyWarps) {
        // ---------------- copy ----------------
        const int tid = threadIdx.x;
        int i = 0;
        const uint64_t ta = TABLE ? R.cthr_addr[tid] : 0;
        const uint32_t tsm = TABLE ? R.cthr_sm[tid] : 0;
        const int c0 = tid & 31, lb = tid >> 5;          // PLAIN: amplitude pair, member bit 0
        const uint64_t pc = TABLE ? 0 : col_base((uint64_t)(2 * c0), G);
        for (uint64_t t = blockIdx.x; t < ntl; t += gridDim.x, ++i) {
            const int s = i % kStages, n = i / kStages;
            if (n >= 1 && !mbar_wait(smem_u32(&S.empty[s]), (n - 1) & 1, abort_flag, d_err)) break;
            const uint64_t tb = col_base(t * kNT, G);
            const uint32_t sb = sB0 + (uint32_t)(s * kRaw);
            if constexpr (TABLE) {
#pragma unroll 16
                for (int k = 0; k < 32; ++k) cp_async16(sb + (tsm ^ R.cit_sm[k]), sv + (tb | ta | R.cit_addr[k]), 16u);
            } else {
#pragma unroll 16
                for (int k = 0; k < 32; ++k) {
                    const int l = 2 * k + lb;
                    cp_async16(sb + mn_chunk(l, c0), sv + (tb | pc | G.off[l]), 16u);
                }
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&S.landed[s])) : "memory");
        }
        // every copy this thread issued has landed before the CTA may exit
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else if (warp < kProdWarps) {
        // ---------------- convert: column block cb of the tile ----------------
        const int cb = (warp - kCopyWarps) >> 1, half = (warp - kCopyWarps) & 1;
        int i = 0;
        for (uint64_t t = blockIdx.x; t < ntl; t += gridDim.x, ++i) {
            const int s = i % kStages;
            if (!mbar_wait(smem_u32(&S.landed[s]), (i / kStages) & 1, abort_flag, d_err)) break;
            const int low = i % kLows;                   // its products of kLows tiles ago are done
            if (i >= kLows && !mbar_wait(smem_u32(&S.low_free[low]), (i / kLows - 1) & 1, abort_flag, d_err)) break;
            const uint32_t part = (uint32_t)(cb * 8192 + half * 4096);
            if (!convert_half<T0>(sB0 + (uint32_t)(s * kRaw) + part, sLow0 + (uint32_t)(low * kLow) + part, lane, half,
                                  halves, S.share[i & 1][cb], smem_u32(&S.xch[cb]), (uint32_t)(i & 1),
                                  &S.bad[s][half][cb], abort_flag, d_err))
                break;
            fence_proxy_async();
            mbar_arrive(smem_u32(&S.full[s]));
        }
    } else if (warp == kMmaWarp) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            int i = 0;
            for (uint64_t t = blockIdx.x; t < ntl; t += gridDim.x, ++i) {
                const int s = i % kStages;
                if (!mbar_wait(smem_u32(&S.full[s]), (i / kStages) & 1, abort_flag, d_err)) break;
                tc_fence_after();
                const uint32_t d0 = tmem + kACols, d1 = d0 + (uint32_t)(2 * kNT * (1 + (i & 1)));
                const uint32_t b = sB0 + (uint32_t)(s * kRaw);
                // K = 64 members in 4 steps of 16: A 8 columns per step, B two member groups.
                // The descriptors of a tile differ in their start address only (bits 0-13, in
                // units of 16 bytes); one thread issues everything, so each is one addition
                const uint64_t bd = sdesc_b(b, 8192u, 1024u), bl = sdesc_b(sLow0 + (uint32_t)(i % kLows * kLow), 8192u, 1024u);
                auto step = [&](uint32_t d, int da, int db, int ks, uint32_t acc) {
                    mma_bf16(d, tmem + (uint32_t)(da * 32 + ks * 8),
                             (db < 2 ? bd : bl) + (uint64_t)((ks * 2048 + (db & 1) * 512) >> 4), acc);
                };
                // the smaller products first. Their accumulator was read two tiles ago (the wait
                // below, one tile ago); the epilogue may still read the tile before
                constexpr int pa[12] = {3, 2, 1, 3, 2, 1, 0, 2, 1, 0, 1, 0}, pb[12] = {1, 2, 3, 0, 1, 2, 3, 0, 1, 2, 0, 1};
#pragma unroll
                for (int p = 0; p < 12; ++p)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks) step(d1, pa[p], pb[p], ks, p + ks);
                mma_commit(smem_u32(&S.low_free[i % kLows]));
                if (i >= 1 && !mbar_wait(smem_u32(&S.acc_empty), (i - 1) & 1, abort_flag, d_err)) break;
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) step(d0, 0, 0, ks, ks);
                mma_commit(smem_u32(&S.acc_full));
            }
            mma_commit(smem_u32(&S.done));
            const long long t0 = clock64();
            bool drained;
            while (!(drained = mbar_try(smem_u32(&S.done), 0)) && clock64() - t0 < kWaitCycles) {
            }
            if (!drained) {
                *abort_flag = 1;
                atomicExch(d_err, kErrTimeout);
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ----------------
        // warp: TMEM lane quarter q (members 16q .. 16q + 15, Re rows then Im rows),
        // column half hh (amplitudes 32 hh .. 32 hh + 31 of the tile)
        const int q = warp & 3, hh = (warp - kProdWarps) >> 2;
        const int e = lane >> 4, j = 16 * q + (lane & 15);
        const uint64_t wa = TABLE ? G.off[16 * q] | col_base((uint64_t)(32 * hh), G) | R.sl_addr[lane] : 0;
        const uint32_t wsm = TABLE ? out_chunk(16 * q, 16 * hh) ^ R.sl_sm[lane] : 0;
        const int cst = 16 * hh + (lane & 15), lb = lane >> 4;               // PLAIN: pair, member bit 0
        const uint64_t pst = TABLE ? 0 : col_base((uint64_t)(2 * cst), G);
        int i = 0;
        for (uint64_t t = blockIdx.x; t < ntl; t += gridDim.x, ++i) {
            const int s = i % kStages;
            if (!mbar_wait(smem_u32(&S.acc_full), i & 1, abort_flag, d_err)) break;
            tc_fence_after();
            const uint32_t sb = sB0 + (uint32_t)(s * kRaw);
            const uint64_t tb = col_base(t * kNT, G);
#pragma unroll 1
            for (int cc = 0; cc < 4; ++cc) {
                float v[16], w[16];
                const uint32_t ad = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(kACols + hh * kNT + cc * 16);
                tmem_ld16x2(ad, ad + (uint32_t)(2 * kNT * (1 + (i & 1))), v, w);
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] += w[k];
                const int blk = 2 * hh + (cc >> 1);
                unsigned bad = S.bad[s][0][blk] | S.bad[s][1][blk];
                if (bad && halves) bad = S.bad[s][q >> 1][blk];
                // v[2u + f] = row product for amplitude 32 hh + 8 cc + u, component f. Of each
                // four amplitudes 4g .. 4g+3 the Re lane finishes the first two, the Im lane
                // the last two; each sends the partner the four products it needs.
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    float r[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        r[k] = __shfl_xor_sync(0xffffffffu, e ? v[8 * g + k] : v[8 * g + 4 + k], 16);
                    float4 o;
                    if (e == 0) {
                        o = make_float4(v[8 * g] - r[1], v[8 * g + 1] + r[0], v[8 * g + 2] - r[3], v[8 * g + 3] + r[2]);
                    } else {
                        o = make_float4(r[0] - v[8 * g + 5], r[1] + v[8 * g + 4], r[2] - v[8 * g + 7],
                                        r[3] + v[8 * g + 6]);
                    }
                    if (bad) {                           // a non-finite amplitude: its group is not a number
                        const unsigned b2 = bad >> (8 * (cc & 1) + 4 * g + 2 * e);
                        const float nan = __uint_as_float(0x7fffffffu);
                        if (b2 & 1u) o.x = o.y = nan;
                        if (b2 & 2u) o.z = o.w = nan;
                    }
                    if constexpr (T0) {
                        // back to memory order: member rows j, j ^ 1 trade halves
                        const bool even = (lane & 1) == 0;
                        const float s0 = __shfl_xor_sync(0xffffffffu, even ? o.z : o.x, 1);
                        const float s1 = __shfl_xor_sync(0xffffffffu, even ? o.w : o.y, 1);
                        o = even ? make_float4(o.x, o.y, s0, s1) : make_float4(s0, s1, o.z, o.w);
                    }
                    const int c = 16 * hh + 4 * cc + 2 * g + e;
                    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(sb + out_chunk(j, c)), "f"(o.x),
                                 "f"(o.y), "f"(o.z), "f"(o.w)
                                 : "memory");
                }
            }
            tc_fence_before();
            mbar_arrive(smem_u32(&S.acc_empty));
            __syncwarp();
#pragma unroll 4
            for (int r = 0; r < 8; ++r) {
                float4 o;
                const int l = 16 * q + 2 * r + lb;
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                             : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w)
                             : "r"(sb + (TABLE ? wsm ^ R.sr_sm[r] : out_chunk(l, cst))));
                *reinterpret_cast<float4 *>(sv + (TABLE ? tb | wa | R.sr_addr[r] : tb | pst | G.off[l])) = o;
            }
            mbar_arrive(smem_u32(&S.empty[s]));
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// A image: digit d at d * kADigit, row m = 32q + r holds Re G[16q + r % 16][.] (r <
// 16) or Im G[16q + r % 16][.] (r >= 16), 64 members of 2 bytes.
// With 5 targets the two halves of the members hold the same matrix.
std::vector<uint16_t> build_image(const double *g, int k) {
    const int D = 1 << k;
    std::vector<uint16_t> img(kA / 2, 0);
    for (int m = 0; m < 128; ++m) {
        const int j = 16 * (m >> 5) + (m & 15), part = (m >> 4) & 1;
        double t[64], top = 0;
        for (int l = 0; l < D; ++l) {
            t[l] = g[2 * ((j & (D - 1)) * D + l) + part];
            top = std::fmax(top, std::fabs(t[l]));
        }
        if (top == 0.0) continue;
        int e;
        std::frexp(top, &e);                             // top < 2^e
        const double scale = std::ldexp(1.0, 7 - e);
        for (int l = 0; l < D; ++l) t[l] *= scale;       // now in units of the first digit
        for (int d = 0; d < kDigA; ++d) {
            // multiples of 2^(e - 7) and 2^(e - 15), then twice what is left, in BF16
            const float unit = std::ldexp(1.0f, e - 7 - 8 * std::min(d, 2));
            uint16_t *out = &img[(size_t)(d * 128 + m) * 64 + (j & ~(D - 1))];
            constexpr double kRound = 6755399441055744.0;   // 1.5 2^52: adding it rounds to an integer
            for (int l = 0; l < D; ++l) {
                const double v = d < 2 ? (t[l] + kRound) - kRound : bf16_to_float(host_bf16((float)t[l]));
                out[l] = host_bf16((float)v * unit);
                t[l] = (t[l] - v) * (d < 2 ? 256.0 : 1.0);
            }
        }
    }
    return img;
}

template <int MODE>
cudaError_t run(const LaunchCtx &L, float2 *sv, const TcGeom &G, const RawMap &R, const uint4 *d_a, int *d_err, int halves) {
    cudaError_t e = cudaFuncSetAttribute(k_tc_x3<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    uint64_t grid = (uint64_t)L.num_sms;
    if (grid > G.n_tiles) grid = G.n_tiles;
    k_tc_x3<MODE><<<(unsigned)grid, kThreads, kSmem, L.stream>>>(sv, G, R, d_a, d_err, halves);
    ++*L.launches;
    return cudaGetLastError();
}

}  // namespace

// Large states only: a gate's matrix takes the host 22 / 43 us to cut and upload
// (k = 5 / 6). Gates in a row, us each, here and by k_dense5 / k_dense6: k = 5 on 22
// qubits 42 / 39, 23 58 / 58, 24 90 / 107; k = 6 on 21 qubits 59 / 53, 22 60 / 82,
// 23 62 / 130.
//
// The digits leave out about 2^-34 of a row's largest entry and of a group's largest
// part per product. An output whose row meets the one large amplitude of its group with
// a small entry feels this first, so every entry has to be within 2^11 of the largest of
// its row (and zeros stay with the FP32 kernels). There the worst amplitude of such
// groups has 0.84 of the error of a chain of 2 2^k FP32 multiply-adds on the same groups
// (7.4 against 8.8 u sum |m||x| in a model of the digits; at 2^10 0.49, at 2^12 1.7); a
// chain's worst elsewhere is 22 u, where the digits have 2. Of random unitaries 99 % are
// within the line. Random unitaries and states on 23 qubits, relative L2 error against 64
// bits: one gate 3.7e-8 where the FP32 chains have 1.5e-7 (k = 5 and 6), fifty gates 2.6e-7
// against 1.04e-6; no drift of the norm.
bool tc_x3_ok(int n, int k, const double *mat) {
    if (n < (k == 5 ? 23 : 22) || k < 5 || k > 6) return false;
    const int D = 1 << k;
    for (int r = 0; r < D; ++r) {
        double lo = HUGE_VAL, hi = 0.0;
        for (int c = 0; c < D; ++c) {
            const double *m = mat + 2 * (r * D + c), a = m[0] * m[0] + m[1] * m[1];
            lo = std::fmin(lo, a);
            hi = std::fmax(hi, a);
            if (!std::isfinite(a)) return false;
        }
        if (lo * 0x1p22 < hi || lo < 0x1p-120 || hi > 0x1p120) return false;
    }
    return true;
}

cudaError_t launch_tc_x3(const LaunchCtx &L, void *sv, int n, const int *tpos, int k, const double *mat, void *d_a,
                         int *d_err) {
    TcGeom G{};
    int mpos[6];
    for (int i = 0; i < k; ++i) mpos[i] = tpos[i];
    if (k == 5) {                                        // the highest qubit that is no target
        int extra = n - 1;
        for (int i = 4; i >= 0 && tpos[i] == extra; --i) --extra;
        mpos[5] = extra;
    }
    for (int i = 0; i < 6; ++i) G.pos[i] = mpos[i];
    std::sort(G.pos, G.pos + 6);
    for (int j = 0; j < 64; ++j) {
        uint64_t o = 0;
        for (int t = 0; t < 6; ++t)
            if ((j >> t) & 1) o |= 1ull << mpos[t];
        G.off[j] = o;
    }
    G.n_cols = 1ull << (n - 6);
    G.n_tiles = G.n_cols / kNT;                          // whole tiles: n >= 12
    const std::vector<uint16_t> img = build_image(mat, k);
    cudaError_t e = cudaMemcpyAsync(d_a, img.data(), kA, cudaMemcpyHostToDevice, L.stream);
    if (e != cudaSuccess) return e;
    float2 *s = reinterpret_cast<float2 *>(sv);
    const uint4 *a = reinterpret_cast<const uint4 *>(d_a);
    const bool t0 = mpos[0] == 0, plain = G.pos[0] >= 4;
    const RawMap R = plain ? RawMap{} : build_raw_map(G.pos, mpos, t0, 5, 16);
    if (t0) return run<T0M>(L, s, G, R, a, d_err, k == 5);
    if (plain) return run<PLAIN>(L, s, G, R, a, d_err, k == 5);
    return run<MAPPED>(L, s, G, R, a, d_err, k == 5);
}

}  // namespace svk
