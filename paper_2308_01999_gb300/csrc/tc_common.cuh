// tc_common.cuh -- what the tensor-core kernels share: mbarriers with bounded
// waits, operand descriptors, TMEM loads, the tile geometry and the order in
// which a tile's 16-byte chunks are copied.
#pragma once

#include <algorithm>
#include <cstring>
#include <vector>

#include "sv_internal.h"

namespace svk {

constexpr long long kWaitCycles = 4000000000ll;   // ~2 s at 2 GHz
constexpr int kErrTimeout = 0x7c01;
constexpr int kErrSmemAlign = 0x7c02;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t a) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(a) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: false on timeout or when another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, volatile int *abort_flag, int *d_err,
                                          long long budget = kWaitCycles) {
    const long long t0 = clock64();
    for (unsigned n = 1; !mbar_try(a, parity); ++n) {
        if (n & 7u) continue;                 // the abort flag is shared memory too: not on every try
        if (*abort_flag) return false;
        if (clock64() - t0 > budget) {
            *abort_flag = 1;
            atomicExch(d_err, kErrTimeout);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor (tcgen05): start address, leading byte offset
// (unused for swizzled K-major, set to 16 B), stride byte offset 1024 B (eight
// 128-byte rows), descriptor version 1, 128-byte swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(16u >> 4) << 16;
    d |= (uint64_t)(1024u >> 4) << 32;
    d |= 1ull << 46;
    d |= 2ull << 61;
    return d;
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

struct TcGeom {
    int pos[6];          // target positions, ascending
    uint64_t off[64];    // member offsets
    uint64_t n_cols;     // 2^(n-6)
    uint64_t n_tiles;
};

__device__ __forceinline__ uint64_t col_base(uint64_t c, const TcGeom &G) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const uint64_t lo = c & ((1ull << G.pos[i]) - 1ull);
        c = ((c ^ lo) << 1) | lo;
    }
    return c;
}

// byte offset of the 16-byte chunk holding floats 4c .. 4c+3 of member row l
// (c = amplitude pair, 0..63) in a stage: atom (c / 8, l / 8); inside it rows of
// 128 bytes (32 floats of one member) whose four 32-byte units are permuted by
// the row index mod 4
__device__ __forceinline__ uint32_t mn_chunk(int l, int c) {
    return (uint32_t)((c >> 3) * 8192 + (l >> 3) * 1024 + (l & 7) * 128 + ((((c & 7) >> 1) ^ (l & 3)) << 5) +
                      ((c & 1) << 4));
}

// Where the epilogue stages chunk c of row l: mn_chunk with rows 4 .. 7 of an atom in
// the other 16-byte half of their 32-byte unit, so that the eight rows that eight
// lanes write fall on all banks
__device__ __forceinline__ uint32_t out_chunk(int l, int c) { return mn_chunk(l, c) ^ (uint32_t)((l & 4) << 2); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

// Which chunk of the tile each copy (and store) moves is set by the host
// (RawMap): with qubit 0 free a chunk is amplitudes (2p, 2p + 1) of member row l
// (2 x 6 index bits: the member's bits sit at the target positions, the pair's at
// non-target positions 1..6); with qubit 0 a target (T0) it is members 2m, 2m + 1
// of one column c (5 member-pair bits at target positions 1..5, 7 column bits at
// the non-target positions), landed in row 2m + (c & 1) of pair c / 2 and turned
// into member rows by the convert stage. The index bits are ordered by the
// address position they set (the three lowest lane bits chosen among the low
// ones so that eight consecutive lanes hit eight different 16-byte bank groups
// of shared memory); the five first vary across the lanes of a warp, the next
// one across the two copy warps, the rest across a thread's copies.
// Both the amplitude address and the operand offset (mn_chunk is linear over
// XOR) are OR / XOR of per-bit contributions, so a thread combines one
// per-thread and one per-copy table entry.
struct RawMap {
    uint64_t cthr_addr[64], cit_addr[64];   // copy: amplitude offset, thread part / copy part
    uint32_t cthr_sm[64], cit_sm[64];       // copy: operand byte offset in a stage
    uint32_t cthr_col[64], cit_col[64];     // copy: first column of the chunk (ragged tiles)
    uint64_t sl_addr[32], sr_addr[16];      // store: lane part / iteration part (one epilogue warp)
    uint32_t sl_sm[32], sr_sm[16];
    uint32_t sl_col[32], sr_col[16];
};

// ---------------- host ----------------
inline uint16_t host_bf16(float x) {
    // round to nearest even
    uint32_t u;
    std::memcpy(&u, &x, 4);
    if ((u & 0x7f800000u) == 0x7f800000u) return (uint16_t)(u >> 16);
    const uint32_t lsb = (u >> 16) & 1u;
    u += 0x7fffu + lsb;
    return (uint16_t)(u >> 16);
}

inline float bf16_to_float(uint16_t h) {
    const uint32_t u = (uint32_t)h << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}

inline size_t host_sw128(int kb, int r, int chunk) {
    return (size_t)kb * (128 * 128) + (size_t)(r >> 3) * 1024 + (size_t)(r & 7) * 128 + (size_t)((chunk ^ (r & 7)) << 4);
}

// operand byte offset of row l, amplitude pair c in a stage (the host twin of mn_chunk)
inline uint32_t host_mn_chunk(int l, int c) {
    return (uint32_t)((c >> 3) * 8192 + (l >> 3) * 1024 + (l & 7) * 128 + ((((c & 7) >> 1) ^ (l & 3)) << 5) +
                      ((c & 1) << 4));
}

// The address-ordered chunk mapping of the raw-operand kernel for targets tpos on
// an n-qubit state (see RawMap): member bit i at mpos[i], tpos the same positions
// ascending, tiles of 2^(pair_bits + 1) columns; store_row4 is added (XOR) to the
// store side's operand offset of row bit 2. Each index bit of a chunk has an amplitude
// address bit, an operand offset and a column contribution; the bits are sorted
// by address bit and dealt out to lanes first.
inline RawMap build_raw_map(const int *tpos, const int *mpos, bool t0, int pair_bits, uint32_t store_row4 = 0) {
    std::vector<int> npos;                       // non-target positions, ascending; past n for tiny states
    for (int q = 0, t = 0; (int)npos.size() < 8; ++q) {
        if (t < 6 && q == tpos[t]) {
            ++t;
            continue;
        }
        npos.push_back(q);
    }
    struct Bit { int apos; uint64_t addr; uint32_t sm; uint32_t col; };
    auto member_bit = [&](int i) {      // member index bit i (row bit i with qubit 0 free)
        return Bit{mpos[i], 1ull << mpos[i], host_mn_chunk(1 << i, 0), 0u};
    };
    std::vector<Bit> copy, store;
    if (!t0) {
        for (int i = 0; i < pair_bits; ++i)     // pair bit i: column bit i + 1
            copy.push_back(Bit{npos[i + 1], 1ull << npos[i + 1], host_mn_chunk(0, 1 << i), 2u << i});
        for (int i = 0; i < 6; ++i) copy.push_back(member_bit(i));
        for (int i = 0; i < pair_bits - 1; ++i)
            store.push_back(Bit{npos[i + 1], 1ull << npos[i + 1], host_mn_chunk(0, 1 << i), 2u << i});
        for (int i = 0; i < 4; ++i) store.push_back(member_bit(i));
        store[pair_bits - 1 + 2].sm ^= store_row4;
    } else {
        // member-pair bit i (member bit i + 1, row bit i + 1); column bit 0 selects the
        // row of the pair, column bit i >= 1 is pair bit i - 1
        auto pair_bit = [&](int i) {
            return Bit{mpos[i + 1], 1ull << mpos[i + 1], host_mn_chunk(2 << i, 0), 0u};
        };
        auto col_bit = [&](int i) {
            return Bit{npos[i], 1ull << npos[i], i == 0 ? host_mn_chunk(1, 0) : host_mn_chunk(0, 1 << (i - 1)), 1u << i};
        };
        for (int i = 0; i < 5; ++i) copy.push_back(pair_bit(i));
        for (int i = 0; i < pair_bits + 1; ++i) copy.push_back(col_bit(i));
        for (int i = 0; i < 3; ++i) store.push_back(pair_bit(i));
        store[1].sm ^= store_row4;
        for (int i = 0; i < pair_bits; ++i) store.push_back(col_bit(i));
    }
    // Address order, except that lanes 0-2 (the eight lanes of one shared-memory
    // wavefront of 16-byte accesses) take the lowest bits whose operand offsets
    // fall in independent 16-byte bank groups, so that those accesses never
    // conflict; the other bits follow in address order.
    auto order = [](std::vector<Bit> &bits) {
        std::sort(bits.begin(), bits.end(), [](const Bit &a, const Bit &b) { return a.apos < b.apos; });
        std::vector<Bit> out;
        std::vector<char> used(bits.size(), 0);
        uint32_t span = 1;                        // bank groups reachable: bit set of a subspace of GF(2)^3
        for (size_t i = 0; i < bits.size() && out.size() < 3; ++i) {
            const uint32_t g = (bits[i].sm >> 4) & 7u;
            if ((span >> g) & 1u) continue;       // g is 0 or already in the span
            uint32_t next = span;
            for (uint32_t v = 0; v < 8; ++v)
                if ((span >> v) & 1u) next |= 1u << (v ^ g);
            span = next;
            out.push_back(bits[i]);
            used[i] = 1;
        }
        for (size_t i = 0; i < bits.size(); ++i)
            if (!used[i]) out.push_back(bits[i]);
        bits = out;
    };
    if (!t0 && mpos[0] >= 3) {
        // qubits 0-2 free: pair bits across the lanes (each instruction 32 consecutive
        // amplitude pairs of one member), member bits across a thread's copies -- the
        // order that measured fastest there (10.8 ms per 32-qubit block against 11.4
        // in address order); the bits are already in that order
    } else {
        order(copy);
        order(store);
    }
    RawMap R{};
    auto fill = [](const std::vector<Bit> &bits, int first, int count, uint64_t *addr, uint32_t *sm, uint32_t *col) {
        for (int v = 0; v < (1 << count); ++v) {
            uint64_t a = 0;
            uint32_t m = 0, c = 0;
            for (int b = 0; b < count; ++b)
                if ((v >> b) & 1) {
                    a |= bits[first + b].addr;
                    m ^= bits[first + b].sm;
                    c |= bits[first + b].col;
                }
            addr[v] = a;
            sm[v] = m;
            col[v] = c;
        }
    };
    fill(copy, 0, 6, R.cthr_addr, R.cthr_sm, R.cthr_col);
    fill(copy, 6, pair_bits, R.cit_addr, R.cit_sm, R.cit_col);
    fill(store, 0, 5, R.sl_addr, R.sl_sm, R.sl_col);
    fill(store, 5, pair_bits - 2, R.sr_addr, R.sr_sm, R.sr_col);
    return R;
}

}  // namespace svk
