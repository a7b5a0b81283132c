// Device code of the remaining integer parts of the I-Parakeet Conformer
// block for sm_103a (Sec. 2.1 Eqs. 1-5, Sec. 2.2, Sec. 3.2, Sec. 3.3):
// residual additions, and the ConvBlock's depthwise convolution with folded
// BatchNorm onto the INT16 grid followed by the minimax Swish.  Integer
// arithmetic only: no floating-point type, no division by a run-time value.
#pragma once

#include <stdint.h>

#include "ip_ptx.cuh"

namespace ipb {

using namespace ipk;

constexpr int RES_THREADS = 256;
constexpr int DW_THREADS = 256;      // one thread per channel of a 256-channel block
constexpr int DW_FRAMES = 32;        // frames per CTA
constexpr int DW_KMAX = 15;          // largest (odd) kernel
constexpr int ERR_PARAM = 16;

struct ResidualParams {
    const int8_t *x, *y;
    int8_t *z;
    long long n;
    int m_x, m_y, s;
};


__global__ void __launch_bounds__(RES_THREADS) residual_i8_kernel(const ResidualParams p) {
    pdl_launch_dependents();
    pdl_wait();   // the grid before this one on the stream: complete, memory visible
    const long long nv = p.n >> 4;   // 16-byte vectors
    const long long stride = static_cast<long long>(gridDim.x) * RES_THREADS;
    for (long long i = static_cast<long long>(blockIdx.x) * RES_THREADS + threadIdx.x; i < nv;
         i += stride) {
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(p.x) + i);
        const uint4 b = __ldcs(reinterpret_cast<const uint4 *>(p.y) + i);
        __stcs(reinterpret_cast<uint4 *>(p.z) + i,
               make_uint4(residual4(a.x, b.x, p.m_x, p.m_y, p.s), residual4(a.y, b.y, p.m_x, p.m_y, p.s),
                          residual4(a.z, b.z, p.m_x, p.m_y, p.s), residual4(a.w, b.w, p.m_x, p.m_y, p.s)));
    }
    // the tail of n (fewer than 16 bytes)
    const long long tail = nv << 4;
    const long long k = tail + static_cast<long long>(blockIdx.x) * RES_THREADS + threadIdx.x;
    if (k < p.n && k < tail + 16)
        p.z[k] = static_cast<int8_t>(residual_one(p.x[k], p.y[k], p.m_x, p.m_y, p.s));
}

struct DwParams {
    const int8_t *x;          // [B][T][C]
    const int8_t *w;          // [C][K]
    const int32_t *bias;      // [C]
    const int32_t *m, *s;     // [C], onto the INT16 grid
    int8_t *y;                // [B][T][C]
    int B, T, C, K;
    int sw_qc, sw_m, sw_s;    // Swish of the INT16 value onto int8
    long long sw_qone;
    int sw_form;              // DW_FAST, DW_WIDE or DW_FULL: the form of dw_out the constants fit
    int *err;
    // four-channels-per-thread kernel: CTA (j, cb) takes channel block cb
    // and the frames [j per, (j + 1) per) of the B T frames in (b, t) order
    uint32_t frames_per_cta;
    unsigned long long t_magic;   // udiv_magic constant of T
};

// Swish of one INT16 value z (Eqs. 12-13 on the grid of z): t = q_one +
// sgn(z) (q_one - D^2) < 2^32, P = z t with |P| < 2^47, and round(m P /
// 2^(31+s)) with m P up to 78 bits, exactly: P = P_hi 2^31 + P_lo with
// 0 <= P_lo < 2^31, so floor((m P + 2^(30+s)) / 2^(31+s)) =
// floor((m P_hi + floor((m P_lo + 2^(30+s)) / 2^31)) / 2^s).
__device__ __forceinline__ int swish16(int z, const DwParams &p) {
    const long long a = z < 0 ? -z : z;
    const long long dc = (a < p.sw_qc ? a : p.sw_qc) - p.sw_qc;
    const long long L = p.sw_qone - dc * dc;
    const long long t = z > 0 ? p.sw_qone + L : (z < 0 ? p.sw_qone - L : p.sw_qone);
    const long long P = static_cast<long long>(z) * t;
    const long long phi = P >> 31;                       // floor(P / 2^31)
    const long long plo = P & 0x7fffffffll;
    const long long m = p.sw_m;
    const long long q1 = m * phi + ((m * plo + (1ll << (30 + p.sw_s))) >> 31);
    const long long r = q1 >> p.sw_s;
    return r > 127 ? 127 : (r < -127 ? -127 : static_cast<int>(r));
}

// Depthwise convolution over time (zero padding at both ends of each
// utterance), per-channel requantisation onto INT16 (folded BatchNorm), and
// the Swish onto int8.  Thread: one channel; CTA: 256 channels x DW_FRAMES
// frames of one utterance, a sliding window of the K input frames in
// registers (K, odd, a compile-time constant: no unused taps).
template <int K>
__global__ void __launch_bounds__(DW_THREADS) dwconv_swish_kernel(const DwParams p) {
    pdl_launch_dependents();
    pdl_wait();   // the grid before this one on the stream: complete, memory visible
    const int c = blockIdx.x * DW_THREADS + threadIdx.x;
    const int t0 = blockIdx.y * DW_FRAMES;
    const int b = blockIdx.z;
    if (c >= p.C) return;
    constexpr int half = K >> 1;
    int w[K];
#pragma unroll
    for (int k = 0; k < K; ++k) w[k] = p.w[static_cast<size_t>(c) * K + k];
    int bias = p.bias[c], mm = p.m[c], ss = p.s[c];
    if (mm < 0 || ss < 0 || ss > 31 || bias >= (1 << 30) || bias <= -(1 << 30)) {
        atomicOr(p.err, ERR_PARAM);
        mm = mm < 0 ? 0 : mm;
        ss = ss < 0 ? 0 : (ss > 31 ? 31 : ss);
        bias = 0;
    }
    const int8_t *xb = p.x + static_cast<size_t>(b) * p.T * p.C + c;
    int8_t *yb = p.y + static_cast<size_t>(b) * p.T * p.C + c;
    // window[k] holds x[t + k - half] for the current output frame t
    int win[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int tt = t0 + k - half;
        win[k] = (tt >= 0 && tt < p.T) ? xb[static_cast<size_t>(tt) * p.C] : 0;
    }
    const int tend = t0 + DW_FRAMES < p.T ? t0 + DW_FRAMES : p.T;
    for (int t = t0; t < tend; ++t) {
        int acc = bias;
#pragma unroll
        for (int k = 0; k < K; ++k) acc += w[k] * win[k];   // |acc| < 2^30 + 2^18
        // onto INT16: round(m acc / 2^(31+s)); |m acc| < 2^62 + 2^50
        const long long v = static_cast<long long>(mm) * acc + (1ll << (30 + ss));
        const long long h = v >> (31 + ss);
        const int z16 = static_cast<int>(h > 32767 ? 32767 : (h < -32767 ? -32767 : h));
        yb[static_cast<size_t>(t) * p.C] = static_cast<int8_t>(swish16(z16, p));
        // slide the window by one frame
#pragma unroll
        for (int k = 0; k < K - 1; ++k) win[k] = win[k + 1];
        const int tn = t + 1 + (K - 1) - half;   // frame entering at slot K - 1
        win[K - 1] = (tn < p.T) ? xb[static_cast<size_t>(tn) * p.C] : 0;
    }
}

// ---- four channels per thread ----------------------------------------------
// The same computation for C a multiple of 4 (and 4-byte aligned x, y, w):
// a thread takes the four channels of one 32-bit word of a frame.  Four
// frame words are byte-transposed into four channel words (four
// consecutive frames of one channel each), so that one dp4a covers four
// taps: output frame t of channel c is the sum over q of dp4a(the four
// frames t - K/2 + 4q .. + 3, taps 4q .. 4q + 3), the frame words taken at
// any byte offset by a funnel shift of two neighbouring channel words.
// What bounds it: instruction issue, and most of all the pipe of the integer
// multiplies (every multiply, dp4a, shift, permute and pack takes two cycles of a
// pipe per warp, additions and minima one).  So the two quotients are taken at word
// boundaries on signed products, a thread makes four frames at a time (eight kept
// more registers and fewer warps: 21.6 us), and up to ten CTAs of 64 threads share an
// SM (96 registers; some shorter grids get more, launch_dw4).  With one form of arithmetic for
// all constants, eight frames at a time and no bound on the registers: 12000 x 1024, K
// = 9 22.8 us, now 19.5; K = 15: 25.3, 22.0; 12000 x 512, K = 5: 15.0, 10.6; 1332 x 1024,
// K = 9: 6.4, 4.9; 400 x 4096, K = 13: 5.7, 5.3; 125 x 1024, K = 9: 3.5, 2.7.
constexpr int DW4_THREADS = 64;      // 256 channels per CTA

struct Swish16K {
    int q_c;
    uint32_t two_qone, m;
    int s;
    unsigned long long h;            // 2^(30+s)
};

// Eq. 7 onto the INT16 grid, then the Swish of that INT16 value onto int8
// (Eqs. 12-13), for one channel: acc the convolution sum with bias, m the
// channel's multiplier, h2 = 2^(31 + s).  z = clamp(floor((m acc + h2 / 2) / 2^(31 +
// s))) and the Swish product is U = z t, |U| < 2^47, with t = 2 q_one - D^2 for z > 0,
// D^2 for z < 0 (D = max(q_c - |z|, 0)).  m_sw U has up to 78 bits.  The forms
// differ in what fits a word; the host picks one by the Swish constants
// (swish16_form), and the clamp of the output at 127 is the pack's.
//
// DW_FAST and DW_WIDE work on signed products: with U = u_hi 2^32 + u_lo (u_hi signed,
// u_lo not), floor(m_sw U / 2^32) is X = m_sw u_hi + floor((m_sw u_lo + h_sw) / 2^32),
// |X| < 2^46, and signs need no case of their own.  X shifted by s_sw - 1 >= 16 fits
// a word, and no negative output is below -127.
// DW_FAST, the usual constants (an INT16 range from 5.7 on, and |bias| of the
// thread's channels at most DW_BIAS): 2 acc is a 32-bit value, so that the first
// quotient is a high word shifted by s; t fits a signed word; and z < -32767 needs
// no clamp, since D = 0 from -q_c on.
// DW_WIDE (a range of 4.02, the least that q_one < 2^31 allows, to 5.7, or any
// bias): a 64-bit shift gives the first quotient (a 32-bit value for every shift,
// since |acc| < 2^30 + 2^18), z is clamped on both sides, and t is unsigned.
// DW_FULL, any other constants of the domain, in sign and magnitude with 32 x 32 ->
// 64-bit products: for n = [v < 0], A = |v| and h = 2^(e-1), floor((m v + h) / 2^e) =
// (1 - 2n) floor((m A + h - n) / 2^e), because floor((h - X) / 2h) = -floor((X + h -
// 1) / 2h); m_sw U is split at bit 31.
// 12000 x 1024, K = 9: FAST 20.1 us, WIDE 22.8, FULL 22.7.  Quotients and clamps of
// signed values in 64 bits for all that is not FAST took 30.2.
constexpr int DW_FAST = 0, DW_WIDE = 1, DW_FULL = 2;
constexpr int DW_BIAS = (1 << 30) - (1 << 20);   // + 128 128 K < 2^30

template <int FORM>
__device__ __forceinline__ int dw_out(int acc, int m, int s, long long h2, const Swish16K &sw) {
    if (FORM == DW_FULL) {
        const uint32_t n = acc < 0 ? 1u : 0u;
        const uint32_t A = acc < 0 ? 0u - static_cast<uint32_t>(acc) : static_cast<uint32_t>(acc);
        const unsigned long long w = static_cast<unsigned long long>(static_cast<uint32_t>(m)) * A +
                                     (static_cast<unsigned long long>(h2 >> 1) - n);   // < 2^63
        const uint32_t a = min(static_cast<uint32_t>(w >> (31 + s)), 32767u);
        const uint32_t q_c = static_cast<uint32_t>(sw.q_c), dc = q_c - min(a, q_c);
        const uint32_t d2 = dc * dc;                          // <= q_c^2 <= q_one < 2^31
        const uint32_t tt = n ? d2 : sw.two_qone - d2;
        const unsigned long long U = static_cast<unsigned long long>(a) * tt;
        const uint32_t ulo = static_cast<uint32_t>(U) & 0x7fffffffu;
        const uint32_t uhi = __funnelshift_r(static_cast<uint32_t>(U), static_cast<uint32_t>(U >> 32), 31);
        const unsigned long long w2 = static_cast<unsigned long long>(sw.m) * ulo + (sw.h - n);
        const uint32_t f = __funnelshift_r(static_cast<uint32_t>(w2), static_cast<uint32_t>(w2 >> 32), 31);
        const unsigned long long X = static_cast<unsigned long long>(sw.m) * uhi + f;   // < 2^48
        const uint32_t xlo = __funnelshift_r(static_cast<uint32_t>(X), static_cast<uint32_t>(X >> 32), sw.s);
        const uint32_t xhi = static_cast<uint32_t>(X >> 32) >> sw.s;
        const uint32_t r = xhi != 0u ? 127u : min(xlo, 127u);
        return static_cast<int>(n ? 0u - r : r);
    }
    int z;
    if (FORM == DW_FAST) {
        const long long w = static_cast<long long>(m) * (2 * acc) + h2;   // < 2^62 + 2^62
        z = min(static_cast<int>(w >> 32) >> s, 32767);
    } else {
        const long long w = static_cast<long long>(m) * acc + (h2 >> 1);
        z = max(min(static_cast<int>(w >> (31 + s)), 32767), -32767);
    }
    const int dc = max(sw.q_c - abs(z), 0);
    const int d2 = dc * dc;                               // <= q_c^2 <= q_one < 2^31
    const uint32_t tt = z > 0 ? sw.two_qone - static_cast<uint32_t>(d2) : static_cast<uint32_t>(d2);
    long long U;
    if (FORM == DW_FAST)
        U = static_cast<long long>(z) * static_cast<int>(tt);
    else   // the unsigned product is 2^32 t above z t for z < 0
        U = static_cast<long long>(static_cast<unsigned long long>(static_cast<uint32_t>(z)) * tt -
                                   (static_cast<unsigned long long>(z < 0 ? tt : 0u) << 32));
    const unsigned long long t = static_cast<unsigned long long>(sw.m) * static_cast<uint32_t>(U) + sw.h;
    const long long X = static_cast<long long>(sw.m) * static_cast<int>(U >> 32) + static_cast<uint32_t>(t >> 32);
    return static_cast<int>(__funnelshift_r(static_cast<uint32_t>(X), static_cast<uint32_t>(X >> 32), sw.s - 1));
}

// Byte transpose of a 4x4 block: y_c = [x0.b_c, x1.b_c, x2.b_c, x3.b_c].
__device__ __forceinline__ void dw_transpose4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                              uint32_t (&y)[4]) {
    const uint32_t t0 = __byte_perm(x0, x1, 0x5140);   // x0.b0 x1.b0 x0.b1 x1.b1
    const uint32_t t1 = __byte_perm(x0, x1, 0x7362);   // x0.b2 x1.b2 x0.b3 x1.b3
    const uint32_t t2 = __byte_perm(x2, x3, 0x5140);
    const uint32_t t3 = __byte_perm(x2, x3, 0x7362);
    y[0] = __byte_perm(t0, t2, 0x5410);
    y[1] = __byte_perm(t0, t2, 0x7632);
    y[2] = __byte_perm(t1, t3, 0x5410);
    y[3] = __byte_perm(t1, t3, 0x7632);
}

// Output frames [ts, te) of one utterance for the thread's four channels.
// Frames are taken in blocks of four from p0 = ts - K/2 (frames outside
// [0, T) read as zero): block u holds frames p0 + 4u .. p0 + 4u + 3, as one
// channel word per channel.  Output frame ts + 4v + i reads the stream at
// offsets 4v + i .. 4v + i + K - 1, i.e. the words of blocks v .. v + Q
// shifted by i bytes.  A step makes one block of four outputs; the frame words
// of the next step's new block are loaded before this step's arithmetic, so
// their latency hides behind it.
template <int K, int FORM>
__device__ __forceinline__ void dw4_segment(const DwParams &p, const uint32_t *xb, uint32_t *yb,
                                            int cw, int ts, int te, const uint32_t (&wq)[4][(K + 3) / 4],
                                            const int (&mq)[4], const int (&sq)[4],
                                            const int (&bq)[4], const long long (&hq)[4],
                                            const Swish16K &sw) {
    constexpr int Q = (K + 3) / 4;    // weight words (taps in fours)
    const int T = p.T;
    const int p0 = ts - (K >> 1);
    auto load_block = [&](int u, uint32_t (&xw)[4]) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int tt = p0 + 4 * u + r;
            xw[r] = (tt >= 0 && tt < T) ? __ldg(xb + static_cast<size_t>(tt) * cw) : 0u;
        }
    };
    uint32_t A[Q + 1][4];   // A[u][j]: channel j of block v + u for step v
    uint32_t nx[4];         // frame words of the next step's new block
#pragma unroll
    for (int u = 0; u < Q; ++u) {
        load_block(u, nx);
        dw_transpose4(nx[0], nx[1], nx[2], nx[3], A[u]);
    }
    load_block(Q, nx);
    const int nsteps = (te - ts + 3) / 4;
#pragma unroll 1
    for (int v = 0; v < nsteps; ++v) {
        dw_transpose4(nx[0], nx[1], nx[2], nx[3], A[Q]);
        if (v + 1 < nsteps) load_block(v + 1 + Q, nx);
        int o[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                int acc = bq[j];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const uint32_t win = i == 0 ? A[q][j] : __funnelshift_r(A[q][j], A[q + 1][j], 8 * i);
                    acc = __dp4a(static_cast<int>(win), static_cast<int>(wq[j][q]), acc);
                }
                o[i][j] = dw_out<FORM>(acc, mq[j], sq[j], hq[j], sw);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = ts + 4 * v + i;
            if (t < te) yb[static_cast<size_t>(t) * cw] = pack_sat4(o[i][0], o[i][1], o[i][2], o[i][3]);
        }
#pragma unroll
        for (int u = 0; u < Q; ++u)
#pragma unroll
            for (int j = 0; j < 4; ++j) A[u][j] = A[u + 1][j];
    }
}

// Thread: channels 4 c4 .. 4 c4 + 3 of channel block blockIdx.y (256
// channels); CTA: a contiguous run of frames_per_cta of the B T frames,
// split at utterance boundaries (the zero padding of each utterance).  The
// grid holds one CTA per resident slot, so there is no partial second wave.
template <int K, int FORM, int CTAS>
__global__ void __launch_bounds__(DW4_THREADS, CTAS) dwconv_swish_x4_kernel(const DwParams p) {
    pdl_launch_dependents();
    pdl_wait();   // the grid before this one on the stream: complete, memory visible
    constexpr int Q = (K + 3) / 4;
    const int cw = p.C >> 2;                               // words per frame
    const int c4 = blockIdx.y * DW4_THREADS + threadIdx.x;
    if (c4 >= cw) return;
    // weights: wq[j][q] = taps 4q .. 4q + 3 of channel 4 c4 + j (zero past
    // K), from the 4 K consecutive bytes of the four channels in w
    uint32_t wq[4][Q];
    {
        const uint32_t *wp = reinterpret_cast<const uint32_t *>(p.w) + static_cast<size_t>(c4) * K;
        uint32_t raw[K];
#pragma unroll
        for (int i = 0; i < K; ++i) raw[i] = __ldg(wp + i);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                uint32_t v = 0;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int k = 4 * q + r;
                    if (k < K) {
                        const int i = j * K + k;   // byte i of the four channels' taps
                        v |= ((raw[i >> 2] >> (8 * (i & 3))) & 0xffu) << (8 * r);
                    }
                }
                wq[j][q] = v;
            }
    }
    int mq[4], sq[4], bq[4];
    long long hq[4];
    bool fast = FORM == DW_FAST;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = 4 * c4 + j;
        int bias = p.bias[c], mm = p.m[c], ss = p.s[c];
        if (mm < 0 || ss < 0 || ss > 31 || bias >= (1 << 30) || bias <= -(1 << 30)) {
            atomicOr(p.err, ERR_PARAM);
            mm = mm < 0 ? 0 : mm;
            ss = ss < 0 ? 0 : (ss > 31 ? 31 : ss);
            bias = 0;
        }
        mq[j] = mm;
        sq[j] = ss;
        bq[j] = bias;
        hq[j] = 1ll << (31 + ss);
        fast &= bias <= DW_BIAS && bias >= -DW_BIAS;
    }
    Swish16K sw;
    sw.q_c = p.sw_qc;
    sw.two_qone = static_cast<uint32_t>(2 * p.sw_qone);
    sw.m = static_cast<uint32_t>(p.sw_m);
    sw.s = p.sw_s;
    sw.h = 1ull << (30 + p.sw_s);
    const uint32_t nframes = static_cast<uint32_t>(p.B) * static_cast<uint32_t>(p.T);   // < 2^31
    uint32_t f = blockIdx.x * p.frames_per_cta;
    const uint32_t fend = min(nframes, f + p.frames_per_cta);
    while (f < fend) {
        const uint32_t b = udiv_magic(f, p.t_magic);
        const int ts = static_cast<int>(f - b * static_cast<uint32_t>(p.T));
        const int te = min(p.T, ts + static_cast<int>(fend - f));
        const size_t base = static_cast<size_t>(b) * p.T * cw + c4;
        const uint32_t *xb = reinterpret_cast<const uint32_t *>(p.x) + base;
        uint32_t *yb = reinterpret_cast<uint32_t *>(p.y) + base;
        if (FORM == DW_FULL)
            dw4_segment<K, DW_FULL>(p, xb, yb, cw, ts, te, wq, mq, sq, bq, hq, sw);
        else if (fast)
            dw4_segment<K, DW_FAST>(p, xb, yb, cw, ts, te, wq, mq, sq, bq, hq, sw);
        else
            dw4_segment<K, DW_WIDE>(p, xb, yb, cw, ts, te, wq, mq, sq, bq, hq, sw);
        f += static_cast<uint32_t>(te - ts);
    }
}

}  // namespace ipb
