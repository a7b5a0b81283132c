// Device code of the integer linear layer (I-Parakeet, Sec. 2.2, Eqs. 6-7)
// for sm_103a: Y = requant(X W^T + bias) with one dyadic multiplier per
// output channel.  Integer arithmetic only: no floating-point type and no
// division by a run-time value.
//
// What bounds it: the integer MMA pipe (mma.sync m16n8k32 s8, about 65 cycles
// each on an SM sub-partition) and the dp4a pipe (two cycles a warp), which
// work at the same time and reach 157 and 159 TOPS alone, 289 together.  So
// a CTA is four MMA warps and four dp4a warps, one of each on every
// sub-partition, and two CTAs share an SM (128 registers a thread), so that
// one computes while the other starts or finishes a tile.
//
// One CTA computes one tile of Y, in one of four shapes that the host picks by
// the size of the problem (64 x 128 down to 32 x 32 frames x channels).  The K
// axis streams in stages of 128 bytes: TMA lands the X rows and W rows of a
// stage with the 128-byte swizzle.  The warps form groups that each cover the
// whole tile, and a group takes one stage of K at a time on its pipe (as many
// groups as the tile is small: a 32 x 32 tile runs eight, so that even one
// tile per SM keeps both pipes of all sub-partitions busy).  The groups'
// partial sums meet in shared memory, where all eight warps requantise them:
// add the int32 bias, multiply by m[n] in int64, shift right by 31 + s[n] with
// rounding, clamp to [-127, 127], and apply the minimax integer Swish, the
// gated unit or the residual addition; four channels per lane, row-major
// [B][T][N] or head-split [G][B][N/G/128][T][128].  With a row-major X the
// frames of all utterances form one axis of B T rows; with a head-split X a
// tile stays inside one utterance.
//
// Measured (1024 -> 4096 with Swish): 125 frames 24.9 -> 8.2 us, 12000 frames
// 460 -> 425 us; 4096 -> 1024 with the residual: 125 frames 87.6 -> 8.7 us,
// 1332 frames 87.9 -> 55.3 us, 12000 frames 431 -> 405 us (before: one
// persistent CTA of 17 warps per SM over 128 x 128 tiles, the channels of a
// tile split between the pipes: a short batch filled 8 to 32 of the SMs, and
// every lane computed the address of each of its shared loads).
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "ip_ptx.cuh"

namespace ipl {

using namespace ipk;

constexpr int THREADS = 256;            // four MMA warps and four dp4a warps
constexpr int BK = 128;                 // K bytes per stage
constexpr int MAX_SLOTS = 24;           // stages of the largest ring

__host__ __device__ constexpr int lg2(int x) { return x <= 1 ? 0 : 1 + lg2(x >> 1); }

// Shape of one CTA's work.  A unit is what one warp accumulates: 2048
// outputs (64 x 32 or 32 x 64; 64 per lane) or, for the smallest tile, 1024.
// The warps whose units cover the tile once form a group; the groups share
// the K stages, so a group's accumulators are partial sums over its stages,
// added through shared memory at the end.
template <int TM_, int TN_>
struct Shape {
    static constexpr int TM = TM_, TN = TN_;      // frames x channels
    static constexpr int OUT = TM * TN;
    static constexpr int UNIT = OUT >= 2048 ? 2048 : 1024;
    static constexpr int WPG = OUT >> lg2(UNIT);  // warps per group
    static constexpr int NG = 8 >> lg2(WPG);      // groups, half of them on each pipe
    static constexpr int MU_M = UNIT == 1024 ? 32 : (TM >= 64 ? 64 : 32);   // MMA unit
    static constexpr int MU_N = UNIT >> lg2(MU_M);
    static constexpr int DU_M = 32;                                         // dp4a unit
    static constexpr int DU_N = UNIT >> lg2(DU_M);
    static constexpr int A_BYTES = TM * BK;
    static constexpr int STAGE = (TM + TN) * BK;
    static constexpr int LPR = TN >> 2;           // epilogue: lanes per row (four channels each)
    static constexpr int RPW = 32 >> lg2(LPR);    // rows a warp finishes at a time
    static constexpr int ROUNDS = TM >> lg2(8 * RPW);
    static constexpr int CONSTS = 0;              // bias, multiplier, shift of the TN channels
    static constexpr int LUT = CONSTS + 3 * 4 * TN;
    static constexpr int BARS = LUT + 256;
    static constexpr int SLOT_INFO = BARS + 8 * MAX_SLOTS;   // per slot: uses issued, warps done
    static constexpr int RING = (SLOT_INFO + 8 * MAX_SLOTS + 1023) & ~1023;
    // shared memory of a CTA with pg stages per group (+ alignment of the base)
    static constexpr int smem(int pg) { return RING + pg * NG * STAGE + 1024; }
    static constexpr int AREAS = NG >> 1;         // areas of partial sums: one per pair of groups
    static_assert(WPG <= 4 && NG >= 2, "groups");
    static_assert((STAGE & 1023) == 0 && (A_BYTES & 1023) == 0, "128-byte swizzle");
};

constexpr int LAYOUT_ROWS = 0;
constexpr int LAYOUT_HEADS = 1;
constexpr int ERR_PARAM = 16;           // a multiplier, shift or bias out of its domain


struct LinearParams {
    const int32_t *bias;      // [N] or nullptr
    const int32_t *m;         // [N]
    const int32_t *s;         // [N]
    int8_t *y;
    int B, T, K, N;
    int ntn;                  // channel tiles
    int tpu;                  // frame tiles per utterance (head-split X)
    unsigned long long magic_ntn, magic_T, magic_tpu;   // exact division constants
    int heads_per_group;      // N / G / 128 (head-split output)
    int y_layout;
    int x_layout;
    int epi;                  // EPI_*
    int pg;                   // ring stages per group
    int *err;
    long long timeout_cycles;
    // minimax Swish of the requantised output (Eqs. 12-13), EPI_SWISH / EPI_GLU
    int sw_qc, sw_qone, sw_m, sw_e;
    // residual addition of the output to res (Eqs. 1-4), EPI_RES
    const int8_t *res;        // [B][T][N], row-major like the output
    int res_mx, res_my, res_s;
};

struct Tile {
    int n0;        // first channel
    int b, t0;     // utterance and frame of the first row (head-split X)
    int m0;        // flat row of the first row (b T + t0)
};

template <class C>
__device__ __forceinline__ Tile tile_of(unsigned idx, const LinearParams &p) {
    Tile L;
    const unsigned mt = udiv_magic(idx, p.magic_ntn);
    L.n0 = static_cast<int>(idx - mt * static_cast<unsigned>(p.ntn)) * C::TN;
    if (p.x_layout == LAYOUT_ROWS) {
        L.m0 = static_cast<int>(mt) * C::TM;
        L.b = L.t0 = 0;
    } else {
        L.b = static_cast<int>(udiv_magic(mt, p.magic_tpu));
        L.t0 = (static_cast<int>(mt) - L.b * p.tpu) * C::TM;
        L.m0 = L.b * p.T + L.t0;
    }
    return L;
}

// Integer Swish of one int8 value z on the grid S_z (Eqs. 12-13): the
// clipped parabola L = q_one - (min(|z|, q_c) - q_c)^2 is |tanh(z S_z / 2)|
// on the grid S_t, t = q_one + sgn(z) L is 1 + tanh, and z t is requantised
// onto the output grid.  |z t| < 2^31 since t <= 2 q_one < 2^24.
__device__ __forceinline__ int swish_i8(int z, const LinearParams &p) {
    const int a = z < 0 ? -z : z;
    const int dc = (a < p.sw_qc ? a : p.sw_qc) - p.sw_qc;
    const int L = p.sw_qone - dc * dc;
    const int t = z > 0 ? p.sw_qone + L : (z < 0 ? p.sw_qone - L : p.sw_qone);
    const long long v = static_cast<long long>(p.sw_m) * (z * t) + (1ll << (p.sw_e - 1));
    return clamp127(v >> p.sw_e);
}

// Gated linear unit of Eq. 5 on two requantised int8 values: a sigma(b)
// with sigma(b) = (1 + tanh(b/2)) / 2 and the minimax tanh on b's grid;
// |a t| < 2^31 (t <= 2 q_one < 2^24).
__device__ __forceinline__ int glu_i8(int a, int b, const LinearParams &p) {
    const int mag = b < 0 ? -b : b;
    const int dc = (mag < p.sw_qc ? mag : p.sw_qc) - p.sw_qc;
    const int L = p.sw_qone - dc * dc;
    const int t = b > 0 ? p.sw_qone + L : (b < 0 ? p.sw_qone - L : p.sw_qone);
    const long long v = static_cast<long long>(p.sw_m) * (a * t) + (1ll << (p.sw_e - 1));
    return clamp127(v >> p.sw_e);
}

constexpr int EPI_PLAIN = 0;   // requantised int8
constexpr int EPI_SWISH = 1;   // + minimax Swish
constexpr int EPI_GLU = 2;     // interleaved pairs (a_c, b_c) -> a_c sigma(b_c)
constexpr int EPI_RES = 3;     // requantised int8, then the residual addition to res

// Eq. 7 for one accumulator (with its bias): max(round(m acc / 2^(31 + s)), -127)
// with rnd = 2^(30 + s); the callers clamp at 127 (a saturating pack).
// |acc| < 2^30 + 2^29 (a bias below 2^30 and 32768 products of at most 2^14), so
// |m acc| < 3 2^60, and the rounding term adds 2^(30 + s), up to 2^61: the sum stays
// below 5 2^60, and its quotient by 2^(31 + s) is a 32-bit value for every s, but
// the one by 2^31 alone only for s = 0.  HI (s >= 1): the high word and a shift by
// sh = s - 1; else a 64-bit shift by sh = 31 + s.
template <bool HI>
__device__ __forceinline__ int requant(int acc, int cm, int sh, long long rnd) {
    const long long v = static_cast<long long>(cm) * acc + rnd;
    return max(HI ? static_cast<int>(v >> 32) >> sh : static_cast<int>(v >> sh), -127);
}

// One stage of a dp4a unit: lane (rg, cg) of RG row and CG channel groups
// (RG CG = 32) accumulates the rows rg + RG i and the channels cg + CG j.  All
// lanes take the same 16-byte k chunk at a time: chunk c of row r sits at
// 128 r + 16 (c ^ (r & 7)), so the lanes of a quarter-warp load phase read
// either one address or distinct bank groups, and since r & 7 takes one value
// per lane (two where RG or CG is 4) the sixteen loads of a chunk need three
// addresses and immediate offsets.  (With lanes on consecutive rows and
// channels every load had an address of its own to compute: 128 TOPS for the
// loop alone against 143 now, 243 against 263 beside the MMA warps.)  The
// loads run ahead: the next W chunk during the current one's products, the
// next X chunks behind the last use of the current ones.
template <int RI, int CG>
__device__ __forceinline__ void dp4a_stage(int (&acc)[RI][8], uint32_t at, uint32_t bt, int rg,
                                           int cg) {
    constexpr int RG = 32 >> lg2(CG);
    uint32_t a0 = (at + rg * 128) | (static_cast<uint32_t>(rg) << 4), a1 = a0 ^ (RG == 4 ? 64u : 0u);
    uint32_t b0 = (bt + cg * 128) | (static_cast<uint32_t>(cg) << 4), b1 = b0 ^ (CG == 4 ? 64u : 0u);
    uint4 a[RI], b;
#pragma unroll
    for (int i = 0; i < RI; ++i) a[i] = lds128(((i & 1) ? a1 : a0) + i * (RG * 128));
    b = lds128(b0);
#pragma unroll 1
    for (uint32_t c = 0; c < 128; c += 16) {
        const uint32_t d = c ^ ((c + 16) & 127);   // to the next chunk (the first again after the last)
        const uint32_t a0n = a0 ^ d, a1n = a1 ^ d, b0n = b0 ^ d;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint4 bn = j < 7 ? lds128(((j & 1) ? b0 : b1) + (j + 1) * (CG * 128)) : lds128(b0n);
#pragma unroll
            for (int i = 0; i < RI; ++i) {
                acc[i][j] = __dp4a(static_cast<int>(a[i].x), static_cast<int>(b.x), acc[i][j]);
                acc[i][j] = __dp4a(static_cast<int>(a[i].y), static_cast<int>(b.y), acc[i][j]);
                acc[i][j] = __dp4a(static_cast<int>(a[i].z), static_cast<int>(b.z), acc[i][j]);
                acc[i][j] = __dp4a(static_cast<int>(a[i].w), static_cast<int>(b.w), acc[i][j]);
                if (j == 7) a[i] = lds128(((i & 1) ? a1n : a0n) + i * (RG * 128));
            }
            b = bn;
        }
        a0 = a0n;
        a1 = a1n;
        b0 = b0n;
        b1 ^= d;
    }
}

// One stage of an MMA unit of MI m16 x NI n8 tiles.
template <int MI, int NI>
__device__ __forceinline__ void mma_stage(int (&acc)[MI][NI][4], uint32_t at, uint32_t bt, int lane) {
    const int lm_row = lane & 7, lm_mat = lane >> 3;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        uint32_t af[MI][4], bf[NI][2];
#pragma unroll
        for (int i = 0; i < MI; ++i)
            ldsm_x4(at + swz(16 * i + (lm_mat & 1) * 8 + lm_row, 2 * ks + (lm_mat >> 1)), af[i][0],
                    af[i][1], af[i][2], af[i][3]);
#pragma unroll
        for (int j = 0; j < NI; j += 2)
            ldsm_x4(bt + swz(8 * j + (lm_mat >> 1) * 8 + lm_row, 2 * ks + (lm_mat & 1)), bf[j][0],
                    bf[j][1], bf[j + 1][0], bf[j + 1][1]);
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j) mma_s8s8(acc[i][j], af[i], bf[j][0], bf[j][1]);
    }
}

// Wrapping increment of a shared-memory counter (0 .. limit), ordered with
// the accesses before and after it; returns the old value.
__device__ __forceinline__ uint32_t atom_inc(uint32_t addr, uint32_t limit) {
    uint32_t old;
    asm volatile("atom.acq_rel.cta.shared.inc.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(limit) : "memory");
    return old;
}

// Adds v to a word of shared memory.
__device__ __forceinline__ void red_add(uint32_t addr, int v) {
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <int V> struct IntConst {
    static constexpr int value = V;
};

// Word of tile element (row, col) in a group's partial sums: the channel
// index XORed with the row, so that the fragment stores of an MMA warp (four
// rows per phase) fall on distinct banks.
template <int TN>
__device__ __forceinline__ uint32_t part_at(int row, int col) {
    return static_cast<uint32_t>(row * TN + (col ^ ((row & 3) << 3))) * 4u;
}

template <int TM, int TN>
__global__ void __launch_bounds__(THREADS, 2)
    linear_i8_kernel(const __grid_constant__ CUtensorMap tm_x,
                     const __grid_constant__ CUtensorMap tm_w, const LinearParams prm) {
    using C = Shape<TM, TN>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int kt = prm.K / BK;     // BK is a power of two: a shift

    const uint32_t base = smem_u32(smem), ring = base + C::RING;
    auto full_bar = [&](int s) { return base + C::BARS + 8u * s; };
    volatile int *issued = reinterpret_cast<int *>(smem + C::SLOT_INFO);
    const uint32_t done = base + C::SLOT_INFO + 4 * MAX_SLOTS;   // per slot: warps done with its stage
    const uint8_t *swish_lut = smem + C::LUT;
    const int slots = C::NG * prm.pg;

    pdl_launch_dependents();
    if (threadIdx.x < slots) {
        mbar_init(full_bar(threadIdx.x), 1);
        sts32(done + 4u * threadIdx.x, 0u);
        issued[threadIdx.x] = -1;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    const Tile L = tile_of<C>(blockIdx.x, prm);
    __syncthreads();
    pdl_wait();   // the grid before this one on the stream: complete, memory visible

    // Warps 0-3 run the integer MMA pipe, 4-7 the dp4a pipe (one of each on
    // every SM sub-partition).  The MMA groups take the first half of the stages
    // of K in turn, the dp4a groups the second, each through its own pg slots of
    // the ring (g, g + NG, ...); the last of a group's warps to finish a stage
    // refills its slot.  What a warp does between two stages adds to the time in
    // full (three more shared loads there: 5 %), so the split is fixed: with stages
    // claimed from a counter, and an end mark to read in each slot, 321.8 us against
    // 316.7 (12000 x 1024 -> 3072), 408.7 against 405.0 (12000 x 4096 -> 1024), 3.80
    // against 3.60 (125 x 1024 -> 1024).  The halves are equal: at K = 4096 17 of 32
    // stages on the MMA pipe take 412.5 us, 18 take 427.
    const bool on_mma = warp < 4;
    const int gi = C::WPG == 1 ? (warp & 3) : (C::WPG == 2 ? (warp & 3) >> 1 : 0);
    const int u = (warp & 3) & (C::WPG - 1);
    const int grp = 2 * gi + (on_mma ? 0 : 1);
    const int mma_kt = (kt + 1) >> 1, pairs = C::NG / 2;
    const int begin = (on_mma ? 0 : mma_kt) + gi, last = on_mma ? mma_kt : kt;
    const int ahead = prm.pg * pairs;   // stages of the pipe between two uses of a slot
    auto issue = [&](int it, int slot, int use) {
        const uint32_t st = ring + slot * C::STAGE;
        issued[slot] = use;
        mbar_expect_tx(full_bar(slot), C::STAGE);
        if (prm.x_layout == LAYOUT_ROWS)
            tma_load_2d(st, &tm_x, it * BK, L.m0, full_bar(slot));
        else
            tma_load_4d(st, &tm_x, 0, L.t0, it, L.b, full_bar(slot));
        tma_load_2d(st + C::A_BYTES, &tm_w, it * BK, L.n0, full_bar(slot));
    };
    if (u == 0 && lane == 0)
        for (int it = begin, slot = grp; slot < slots && it < last; it += pairs, slot += C::NG) issue(it, slot, 0);

    // while the first stages land: the channel constants (clipped into their
    // domain) and the Swish of every int8 input, entry at the byte value of z
    int32_t *cst = reinterpret_cast<int32_t *>(smem + C::CONSTS);
    if (threadIdx.x < TN) {
        const int n = L.n0 + threadIdx.x;
        int bi = prm.bias != nullptr ? __ldg(prm.bias + n) : 0;
        int mi = __ldg(prm.m + n);
        int si = __ldg(prm.s + n);
        if (mi < 0 || si < 0 || si > 31 || bi >= (1 << 30) || bi <= -(1 << 30)) {
            atomicOr(prm.err, ERR_PARAM);
            mi = mi < 0 ? 0 : mi;
            si = si < 0 ? 0 : (si > 31 ? 31 : si);
            bi = 0;
        }
        cst[threadIdx.x] = bi;
        cst[TN + threadIdx.x] = mi;
        cst[2 * TN + threadIdx.x] = si;
    }
    if (prm.epi == EPI_SWISH)
        smem[C::LUT + threadIdx.x] = static_cast<uint8_t>(
            swish_i8(static_cast<int>(static_cast<int8_t>(static_cast<uint8_t>(threadIdx.x))), prm));

    bool ok = true;
    auto run_stages = [&](auto &&compute) {
        for (int it = begin, slot = grp, use = 0; it < last; it += pairs) {
            if (!warp_wait(full_bar(slot), use & 1, prm.timeout_cycles)) {
                if (lane == 0) atomicOr(prm.err, 1);
                ok = false;
                return;
            }
            compute(ring + slot * C::STAGE);
            const bool refill = it + ahead < last;
            // Without a refill the fence can go: 1332 x 4096 -> 1024 57.0 -> 56.8 us; the
            // largest shape runs 0.5 % faster with it always there.
            if (refill || C::NG == 2) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0 && refill && (C::WPG == 1 || atom_inc(done + 4u * slot, C::WPG - 1) == C::WPG - 1))
                    issue(it + ahead, slot, use + 1);
            }
            slot += C::NG;
            if (slot >= slots) {
                slot = grp;
                ++use;
            }
        }
    };

    // Partial sums of the groups, written over the ring once every warp has read
    // its last stage: the MMA groups store theirs and the dp4a groups add to them
    // (one group each), so that the epilogue reads half as many words.  With an
    // area per group: 324.4 -> 321.7 us (12000 x 1024 -> 3072), 59.1 -> 58.2 (1332 x
    // 4096 -> 1024), 8.67 -> 8.44 (125 x 1024 -> 4096).
    auto all_done = [&]() -> bool {
        if (__syncthreads_or(ok ? 0 : 1) == 0) return true;
        if (threadIdx.x == 0)   // let the copies in flight land before the CTA exits
            for (int s = 0; s < slots; ++s)
                if (issued[s] >= 0) mbar_wait(full_bar(s), issued[s] & 1, 2000000000ll);
        return false;
    };
    const uint32_t part = ring + gi * (C::OUT * 4);
    if (on_mma) {
        constexpr int MI = C::MU_M >> 4, NI = C::MU_N >> 3;
        constexpr int UL = lg2(TM) - lg2(C::MU_M);   // units along the frames: 1 << UL
        const int r0 = C::MU_M * (u & ((1 << UL) - 1)), c0 = C::MU_N * (u >> UL);
        int acc[MI][NI][4];
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0;
        run_stages([&](uint32_t st) {
            mma_stage<MI, NI>(acc, st + r0 * 128, st + C::A_BYTES + c0 * 128, lane);
        });
        if (!all_done()) return;
        const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j)
#pragma unroll
                for (int rr = 0; rr < 2; ++rr)
                    sts64(part + part_at<TN>(r0 + 16 * i + g + 8 * rr, c0 + 8 * j + 2 * t4),
                          acc[i][j][2 * rr], acc[i][j][2 * rr + 1]);
        __syncthreads();
    } else {
        constexpr int CG = C::DU_N >> 3, RI = C::DU_M >> lg2(32 >> lg2(CG));
        constexpr int UL = lg2(TM) - lg2(C::DU_M);
        const int rg = lane >> lg2(CG), cg = lane & (CG - 1);
        const int r0 = C::DU_M * (u & ((1 << UL) - 1)), c0 = C::DU_N * (u >> UL);
        int acc[RI][8];
#pragma unroll
        for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0;
        run_stages([&](uint32_t st) {
            dp4a_stage<RI, CG>(acc, st + r0 * 128, st + C::A_BYTES + c0 * 128, rg, cg);
        });
        if (!all_done()) return;
        __syncthreads();   // the MMA warps' sums are there
#pragma unroll
        for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t at = part + part_at<TN>(r0 + rg + (32 >> lg2(CG)) * i, c0 + cg + CG * j);
                red_add(at, acc[i][j]);
            }
    }

    // ------------------------------------------------------------ epilogue
    // Lane: four consecutive channels, rows rl, rl + 8 RPW, ...; the loads of
    // the residual operand go out before the partial sums are awaited.
    const int cl = 4 * (lane & (C::LPR - 1)), rl = C::RPW * warp + (lane >> lg2(C::LPR));
    const int col = L.n0 + cl, flat0 = L.m0 + rl;
    const int frames = prm.x_layout == LAYOUT_ROWS ? prm.B * prm.T : (L.b + 1) * prm.T;
    const bool glu = prm.epi == EPI_GLU;
    constexpr int STEP = 8 * C::RPW;
    // Row-major Y [B][T][width] (width N, N / 2 behind the gated unit), or
    // head-split Y [G][B][N / G / 128][T][128]: frame t of utterance b.
    const long long width = glu ? prm.N >> 1 : prm.N;
    long long off = static_cast<long long>(flat0) * width + (glu ? col >> 1 : col);
    const bool heads = prm.y_layout == LAYOUT_HEADS;
    int t = 0;
    if (heads) {
        int hh = L.n0 >> 7, gg = 0;
        while (hh >= prm.heads_per_group) {   // at most G - 1 steps
            hh -= prm.heads_per_group;
            ++gg;
        }
        const int b = static_cast<int>(udiv_magic(static_cast<unsigned>(flat0), prm.magic_T));
        t = flat0 - b * prm.T;
        off = ((((static_cast<long long>(gg) * prm.B + b) * prm.heads_per_group + hh) * prm.T + t) << 7) +
              (col & 127);
    }
    uint32_t xr[C::ROUNDS];
    if (prm.epi == EPI_RES) {
#pragma unroll
        for (int q = 0; q < C::ROUNDS; ++q)
            if (flat0 + STEP * q < frames)
                xr[q] = *reinterpret_cast<const uint32_t *>(prm.res + off + STEP * q * width);
    }
    __syncthreads();
    int cb[4], cm[4], cs[4];
    long long rnd[4];
    {
        const uint4 vb = lds128(base + C::CONSTS + 4 * cl);
        const uint4 vm = lds128(base + C::CONSTS + 4 * (TN + cl));
        const uint4 vs = lds128(base + C::CONSTS + 4 * (2 * TN + cl));
        cb[0] = static_cast<int>(vb.x), cb[1] = static_cast<int>(vb.y), cb[2] = static_cast<int>(vb.z), cb[3] = static_cast<int>(vb.w);
        cm[0] = static_cast<int>(vm.x), cm[1] = static_cast<int>(vm.y), cm[2] = static_cast<int>(vm.z), cm[3] = static_cast<int>(vm.w);
        cs[0] = static_cast<int>(vs.x), cs[1] = static_cast<int>(vs.y), cs[2] = static_cast<int>(vs.z), cs[3] = static_cast<int>(vs.w);
#pragma unroll
        for (int e = 0; e < 4; ++e) rnd[e] = 1ll << (30 + cs[e]);
    }
    // One loop per epilogue, shift form and layout, chosen once per tile: the
    // epilogue's instructions take issue slots from the other CTA's dp4a warps
    // (of 331 us at 1024 -> 3072, 12000 frames, 20 us went with it; 324 us with
    // the choices out of the loop and the shift below).  HI: every channel of the
    // warp has s >= 1, and the quotient by 2^(31 + s) is the high word >> (s - 1).
    auto rows = [&](auto epi_tag, auto hi_tag, auto heads_tag) {
        constexpr int EPI = decltype(epi_tag)::value;
        constexpr bool HI = decltype(hi_tag)::value != 0, HEADS = decltype(heads_tag)::value != 0;
        int8_t *dst = prm.y + off;
        int sh[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) sh[e] = HI ? cs[e] - 1 : cs[e] + 31;
#pragma unroll
        for (int q = 0; q < C::ROUNDS; ++q) {
            if (flat0 + STEP * q >= frames) break;
            int a[4] = {cb[0], cb[1], cb[2], cb[3]};
#pragma unroll
            for (int g = 0; g < C::AREAS; ++g) {
                const uint4 v = lds128(ring + g * (C::OUT * 4) + part_at<TN>(rl + STEP * q, cl));
                a[0] += static_cast<int>(v.x);
                a[1] += static_cast<int>(v.y);
                a[2] += static_cast<int>(v.z);
                a[3] += static_cast<int>(v.w);
            }
            int z[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) z[e] = requant<HI>(a[e], cm[e], sh[e], rnd[e]);
            if (EPI == EPI_GLU) {
                // channels (a_c, b_c) interleaved: two gated outputs
                const uint32_t w = (static_cast<uint32_t>(glu_i8(min(z[0], 127), min(z[1], 127), prm)) & 0xffu) |
                                   ((static_cast<uint32_t>(glu_i8(min(z[2], 127), min(z[3], 127), prm)) & 0xffu) << 8);
                *reinterpret_cast<uint16_t *>(dst) = static_cast<uint16_t>(w);
            } else {
                uint32_t w = pack_sat4(z[0], z[1], z[2], z[3]);
                if (EPI == EPI_SWISH)
                    w = swish_lut[w & 0xffu] | (swish_lut[(w >> 8) & 0xffu] << 8) |
                        (swish_lut[(w >> 16) & 0xffu] << 16) | (static_cast<uint32_t>(swish_lut[w >> 24]) << 24);
                else if (EPI == EPI_RES)
                    w = residual4(xr[q], w, prm.res_mx, prm.res_my, prm.res_s);
                *reinterpret_cast<uint32_t *>(dst) = w;
            }
            if (HEADS) {
                dst += STEP << 7;
                for (t += STEP; t >= prm.T; t -= prm.T)   // into the next utterance
                    dst += static_cast<long long>(prm.heads_per_group - 1) * prm.T << 7;
            } else {
                dst += STEP * width;
            }
        }
    };
    const bool hi = __all_sync(0xffffffffu, cs[0] > 0 && cs[1] > 0 && cs[2] > 0 && cs[3] > 0) != 0;
    auto by_shift = [&](auto epi_tag, auto heads_tag) {
        if (hi) rows(epi_tag, IntConst<1>(), heads_tag);
        else rows(epi_tag, IntConst<0>(), heads_tag);
    };
    if (heads) by_shift(IntConst<EPI_PLAIN>(), IntConst<1>());
    else if (prm.epi == EPI_PLAIN) by_shift(IntConst<EPI_PLAIN>(), IntConst<0>());
    else if (prm.epi == EPI_SWISH) by_shift(IntConst<EPI_SWISH>(), IntConst<0>());
    else if (prm.epi == EPI_GLU) by_shift(IntConst<EPI_GLU>(), IntConst<0>());
    else by_shift(IntConst<EPI_RES>(), IntConst<0>());
}

}  // namespace ipl
