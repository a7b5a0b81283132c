// Host side of the integer linear layer of the C ABI (include/ip_mhsa.h):
// argument validation, TMA tensor maps and the launch.  Device code:
// ip_linear_kernels.cuh.
#include "ip_mhsa.h"
#include "ip_linear_kernels.cuh"
#include "ip_host_util.h"

#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// int8 tensor map of `rank` dimensions (innermost first; byte strides of
// dimensions 1..rank-1) with a box of 128 x rows (x 1 ...), 128-byte swizzle;
// elements outside the tensor read as zero.
bool make_map(CUtensorMap *m, const void *base, int rank, const cuuint64_t *dims,
              const cuuint64_t *strides, unsigned rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint32_t box[4] = {128, rows, 1, 1};
    const cuuint32_t estride[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT8, rank, const_cast<void *>(base), dims, strides,
              box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

std::mutex g_mu;
int g_smem_set[64] = {0};
int g_sms[64] = {0};

int sm_count() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_sms[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        g_sms[dev] = n;
    }
    return g_sms[dev];
}

using LinearKernel = void (*)(const CUtensorMap, const CUtensorMap, const ipl::LinearParams);

// The kernel's tile shapes, and what a launch of n tiles costs with each (ns): with
// one tile per SM or less `one + one_r r + one_k kt`, else `base + w (wave + wave_r
// r + wave_k kt)`, where kt = K / 128, r is kt rounded up to the shape's groups of
// warps (they take a stage each at a time: 125 x 128 -> 1024 in 32 x 64 tiles takes as
// long as 125 x 1024 -> 1024, 5.2 and 5.7 us), and w = ceil(n / SMs) (two CTAs share
// an SM, so a wave of one tile per SM takes half of what a pair does).  Fitted on
// GB300 to sweeps of M = 1 .. 12000 frames over N = 128 .. 16384 and eighteen K from
// 128 to 8192 with all four shapes timed at each point, and 400 added to `one`: such a
// CTA holds all of an SM's shared memory, so that the launches before and after
// it cannot share the SM (without it the block of one 10 s utterance takes 95.5
// us for 90.3, and ties fall on the slower side).  On the swept points the choice is
// 0.1 % slower than the best of the four in the mean, 30 % at most (one frame, K = N =
// 8192: 35 us for 27).  A large tile costs the least per output, a small one fills the
// SMs: at K = 1024, N = 4096 64 x 128 tiles take 13.9 us at M = 30, 32 x 32 ones 3.7
// us, and at M = 12000 425 us against 624 us.  A model without r, fitted at K = 1024
// and more, took too small a tile where K is short or no multiple of 1024: 500 x 256 ->
// 8192 22.5 us for 15.2, 333 x 512 -> 16384 53.5 for 35.4, 500 x 1152 -> 4096 35.4 for 27.1.
struct Variant {
    LinearKernel fn;
    int tm, tn;
    int pg1, pg2;         // ring stages per group with one and with two CTAs on an SM
    int smem1, smem2;
    int one, one_r, one_k, base, wave, wave_r, wave_k;
    int groups;
};
template <int TM, int TN, int PG1, int PG2>
constexpr Variant variant(int one, int one_r, int one_k, int base, int wave, int wave_r, int wave_k) {
    static_assert(PG1 * ipl::Shape<TM, TN>::NG <= ipl::MAX_SLOTS, "slots");
    static_assert(TM * TN * 4 <= PG2 * ipl::Shape<TM, TN>::STAGE, "the partial sums reuse the ring");
    return {ipl::linear_i8_kernel<TM, TN>, TM, TN, PG1, PG2, ipl::Shape<TM, TN>::smem(PG1),
            ipl::Shape<TM, TN>::smem(PG2), one, one_r, one_k, base, wave, wave_r, wave_k,
            ipl::Shape<TM, TN>::NG};
}
const Variant VARIANTS[] = {
    variant<64, 128, 4, 2>(3430, 1143, 309, 3117, 579, 611, 628),
    variant<64, 64, 3, 1>(3118, 624, 120, 3042, 402, 443, 203),
    variant<32, 64, 2, 1>(3057, 327, 49, 3129, 433, 185, 131),
    variant<32, 32, 3, 1>(2641, 181, 32, 2289, 503, 90, 79),
};

int ensure_smem() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return IP_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_mu);
    if (g_smem_set[dev]) return IP_OK;
    for (const Variant &v : VARIANTS)
        if (cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, v.smem1) !=
            cudaSuccess)
            return IP_ERR_CUDA;
    g_smem_set[dev] = 1;
    return IP_OK;
}

// Frame tiles of the variant.
long long frame_tiles(const Variant &v, int x_layout, int B, int T) {
    return x_layout == IP_LAYOUT_ROWS ? (static_cast<long long>(B) * T + v.tm - 1) / v.tm
                                      : static_cast<long long>(B) * ((T + v.tm - 1) / v.tm);
}

// Tiles of the variant.
long long tiles_of(const Variant &v, int x_layout, int B, int T, int N) {
    return frame_tiles(v, x_layout, B, T) * (N / v.tn);
}

const Variant &choose_variant(int x_layout, int B, int T, int K, int N, int nsm) {
    const Variant *best = VARIANTS;
    long long least = -1;
    for (const Variant &v : VARIANTS) {
        const long long n = tiles_of(v, x_layout, B, T, N), kt = K / ipl::BK;
        const long long w = (n + nsm - 1) / nsm;
        const long long r = (kt + v.groups - 1) / v.groups * v.groups;
        const long long ns = w <= 1 ? v.one + v.one_r * r + v.one_k * kt
                                    : v.base + w * (v.wave + v.wave_r * r + v.wave_k * kt);
        if (least < 0 || ns < least) {
            least = ns;
            best = &v;
        }
    }
    return *best;
}

int check_swish(const ip_swish_params *p) {
    if (p->q_c < 1 || p->q_c >= (1 << 15) || p->q_one < 1 || p->q_one >= (1 << 23) ||
        static_cast<long long>(p->q_one) < static_cast<long long>(p->q_c) * p->q_c ||
        p->m < 0 || p->s < 0 || p->s > 31)
        return IP_ERR_PARAM;
    return IP_OK;
}

// Residual operand of the RES epilogue: the tensor added and its constants.
struct ResidualArg {
    const int8_t *x;
    int32_t m_x, m_y, s;
};

int linear_launch(const int8_t *x, int x_layout, const int8_t *w, const int32_t *bias,
                  const int32_t *m, const int32_t *s, const ip_swish_params *sw, int epi, int B,
                  int T, int K, int N, int G, int8_t *y, int y_layout, void *workspace,
                  size_t workspace_bytes, ip_stream_t stream, const ResidualArg *res = nullptr) {
    if ((x_layout != IP_LAYOUT_ROWS && x_layout != IP_LAYOUT_HEADS) ||
        (y_layout != IP_LAYOUT_ROWS && y_layout != IP_LAYOUT_HEADS))
        return IP_ERR_PARAM;
    if (B < 0 || B > IP_MAX_B || T < 1 || G < 1) return IP_ERR_SHAPE;
    if (static_cast<long long>(B) * T > IP_LINEAR_MAX_FRAMES) return IP_ERR_SHAPE;
    if (K < 128 || K > IP_LINEAR_MAX_K || K % 128 != 0) return IP_ERR_SHAPE;
    if (N < 128 || N > IP_LINEAR_MAX_N || N % 128 != 0) return IP_ERR_SHAPE;
    if (y_layout == IP_LAYOUT_HEADS && N % (128 * G) != 0) return IP_ERR_SHAPE;
    if (y_layout == IP_LAYOUT_ROWS && G != 1) return IP_ERR_SHAPE;
    if (B == 0) return IP_OK;
    if (!x || !w || !m || !s || !y || !workspace) return IP_ERR_NULL;
    if (!aligned(x, 16) || !aligned(w, 16) || !aligned(y, 16) || !aligned(m, 4) ||
        !aligned(s, 4) || (bias && !aligned(bias, 4)) || !aligned(workspace, 256))
        return IP_ERR_ALIGN;
    if (workspace_bytes < 256) return IP_ERR_WORKSPACE;

    const int nsm = sm_count();
    if (nsm <= 0) return IP_ERR_CUDA;
    const Variant &var = choose_variant(x_layout, B, T, K, N, nsm);
    const long long ntiles = tiles_of(var, x_layout, B, T, N);
    if (ntiles > 0x7fffffffll) return IP_ERR_SHAPE;

    CUtensorMap tm_x, tm_w;
    const cuuint64_t kk = static_cast<cuuint64_t>(K), tt = static_cast<cuuint64_t>(T);
    bool okm;
    if (x_layout == IP_LAYOUT_ROWS) {
        // all frames of all utterances as one axis of B T rows
        const cuuint64_t dims[2] = {kk, tt * static_cast<cuuint64_t>(B)};
        const cuuint64_t strides[1] = {kk};
        okm = make_map(&tm_x, x, 2, dims, strides, var.tm);
    } else {
        const cuuint64_t dims[4] = {128, tt, kk / 128, static_cast<cuuint64_t>(B)};
        const cuuint64_t strides[3] = {128, tt * 128, tt * kk};
        okm = make_map(&tm_x, x, 4, dims, strides, var.tm);
    }
    const cuuint64_t wdims[2] = {kk, static_cast<cuuint64_t>(N)};
    const cuuint64_t wstrides[1] = {kk};
    if (!okm || !make_map(&tm_w, w, 2, wdims, wstrides, var.tn)) return IP_ERR_CUDA;
    int rc = ensure_smem();
    if (rc != IP_OK) return rc;

    ipl::LinearParams prm;
    prm.bias = bias;
    prm.m = m;
    prm.s = s;
    prm.y = y;
    prm.B = B;
    prm.T = T;
    prm.K = K;
    prm.N = N;
    prm.heads_per_group = N / G / 128;
    prm.y_layout = y_layout;
    prm.x_layout = x_layout;
    prm.err = static_cast<int *>(workspace);
    prm.timeout_cycles = 4000000000ll;
    // with a CTA or less per SM the ring takes the whole shared memory
    const bool one = ntiles <= nsm;
    prm.pg = one ? var.pg1 : var.pg2;
    prm.epi = epi;
    prm.ntn = N / var.tn;
    prm.tpu = (T + var.tm - 1) / var.tm;
    prm.magic_ntn = iph::div_magic(prm.ntn);
    prm.magic_T = iph::div_magic(T);
    prm.magic_tpu = iph::div_magic(prm.tpu);
    prm.sw_qc = sw ? sw->q_c : 0;
    prm.sw_qone = sw ? sw->q_one : 0;
    prm.sw_m = sw ? sw->m : 0;
    prm.sw_e = sw ? 31 + sw->s : 0;
    prm.res = res ? res->x : nullptr;
    prm.res_mx = res ? res->m_x : 0;
    prm.res_my = res ? res->m_y : 0;
    prm.res_s = res ? res->s : 0;
    const cudaError_t lrc =
        iph::launch_pdl(var.fn, dim3(static_cast<unsigned>(ntiles)), dim3(ipl::THREADS), one ? var.smem1 : var.smem2,
                        reinterpret_cast<cudaStream_t>(stream), tm_x, tm_w, prm);
    if (lrc != cudaSuccess || cudaGetLastError() != cudaSuccess) return IP_ERR_CUDA;
    return IP_OK;
}

}  // namespace

extern "C" {

int ip_linear_i8(const int8_t *x, int x_layout, const int8_t *w, const int32_t *bias,
                 const int32_t *m, const int32_t *s, int B, int T, int K, int N, int G,
                 int8_t *y, int y_layout, void *workspace, size_t workspace_bytes,
                 ip_stream_t stream) {
    return linear_launch(x, x_layout, w, bias, m, s, nullptr, ipl::EPI_PLAIN, B, T, K, N, G, y,
                         y_layout, workspace, workspace_bytes, stream);
}

int ip_linear_swish_i8(const int8_t *x, const int8_t *w, const int32_t *bias, const int32_t *m,
                       const int32_t *s, const ip_swish_params *sw, int B, int T, int K, int N,
                       int8_t *y, void *workspace, size_t workspace_bytes, ip_stream_t stream) {
    if (!sw) return IP_ERR_NULL;
    const int rc = check_swish(sw);
    if (rc != IP_OK) return rc;
    return linear_launch(x, IP_LAYOUT_ROWS, w, bias, m, s, sw, ipl::EPI_SWISH, B, T, K, N, 1, y,
                         IP_LAYOUT_ROWS, workspace, workspace_bytes, stream);
}

int ip_linear_glu_i8(const int8_t *x, const int8_t *w, const int32_t *bias, const int32_t *m,
                     const int32_t *s, const ip_swish_params *glu, int B, int T, int K, int N,
                     int8_t *y, void *workspace, size_t workspace_bytes, ip_stream_t stream) {
    if (!glu) return IP_ERR_NULL;
    const int rc = check_swish(glu);
    if (rc != IP_OK) return rc;
    return linear_launch(x, IP_LAYOUT_ROWS, w, bias, m, s, glu, ipl::EPI_GLU, B, T, K, N, 1, y,
                         IP_LAYOUT_ROWS, workspace, workspace_bytes, stream);
}

int ip_linear_residual_i8(const int8_t *x, const int8_t *w, const int32_t *bias,
                          const int32_t *m, const int32_t *s, const int8_t *res, int32_t m_x,
                          int32_t m_y, int32_t s_r, int B, int T, int K, int N, int8_t *y,
                          void *workspace, size_t workspace_bytes, ip_stream_t stream) {
    if (m_x < 0 || m_y < 0 || s_r < 0 || s_r > 31) return IP_ERR_PARAM;
    if (B > 0 && !res) return IP_ERR_NULL;
    if (res && !aligned(res, 16)) return IP_ERR_ALIGN;
    if (res && y && res != y && B > 0 && T > 0 && N > 0) {
        // in place (res == y) is fine: every element is read by the thread
        // that then writes it; a partial overlap would race across CTAs
        const uintptr_t a = reinterpret_cast<uintptr_t>(res), b = reinterpret_cast<uintptr_t>(y);
        const uintptr_t n = static_cast<uintptr_t>(B) * static_cast<uintptr_t>(T) *
                            static_cast<uintptr_t>(N);
        if (a < b + n && b < a + n) return IP_ERR_PARAM;
    }
    const ResidualArg ra{res, m_x, m_y, s_r};
    return linear_launch(x, IP_LAYOUT_ROWS, w, bias, m, s, nullptr, ipl::EPI_RES, B, T, K, N, 1, y,
                         IP_LAYOUT_ROWS, workspace, workspace_bytes, stream, &ra);
}

int ip_linear_constants(double S_x, const double *S_w, const double *S_y, int N, int32_t *m,
                        int32_t *s) {
    if (!S_w || !S_y || !m || !s) return IP_ERR_NULL;
    if (N < 1 || !(S_x > 0.0) || !std::isfinite(S_x)) return IP_ERR_PARAM;
    for (int n = 0; n < N; ++n)   // every channel valid before any output is written
        if (!(S_w[n] > 0.0) || !std::isfinite(S_w[n]) || !(S_y[n] > 0.0) || !std::isfinite(S_y[n]))
            return IP_ERR_PARAM;
    for (int n = 0; n < N; ++n) {
        int32_t mm = 0, ss = 0;
        if (ip_dyadic_multiplier(S_x * S_w[n] / S_y[n], &mm, &ss) != IP_OK) return IP_ERR_PARAM;
    }
    for (int n = 0; n < N; ++n)
        ip_dyadic_multiplier(S_x * S_w[n] / S_y[n], &m[n], &s[n]);
    return IP_OK;
}

int ip_swish_params_from_scales(double S_z, double S_y, ip_swish_params *out) {
    if (!out) return IP_ERR_NULL;
    if (!(S_z > 0.0) || !(S_y > 0.0) || !std::isfinite(S_z) || !std::isfinite(S_y))
        return IP_ERR_PARAM;
    const double a = IP_SWISH_A, c = IP_SWISH_C;
    const double s_t = -a * (S_z / 2.0) * (S_z / 2.0);
    const double qc = std::floor(2.0 * c / S_z + 0.5);
    const double qone = std::floor(1.0 / s_t + 0.5);
    if (qc < 1.0 || qc >= 32768.0 || qone < 1.0 || qone >= 8388608.0) return IP_ERR_PARAM;
    ip_swish_params p;
    p.q_c = static_cast<int32_t>(qc);
    p.q_one = static_cast<int32_t>(qone);
    const int rc = ip_dyadic_multiplier(S_z * s_t / (2.0 * S_y), &p.m, &p.s);
    if (rc != IP_OK) return rc;
    if (check_swish(&p) != IP_OK) return IP_ERR_PARAM;
    *out = p;
    return IP_OK;
}

}  // extern "C"
