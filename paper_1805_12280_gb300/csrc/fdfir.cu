// Full-length frequency-domain FIR (Eq. 2): y_z = IFFT_P(FFT_P(x) . FFT_P(h_z)) with P >= n + K - 1
// a power of two, then |y_z|^2 for i < n -- the "naive" FD-FIR that the paper weighs against
// overlap-save (Sec. 3.2.1, Table 1), kept to measure that choice on this GPU.
//
// P-point transforms in four steps, P = P1 * P2 with P1 = 2048 and P2 in {1024, 2048, 4096}:
//   n = P2 n1 + n2,  k = k1 + P1 k2,
//   X[k1 + P1 k2] = sum_n2 W_P2^{n2 k2} W_P^{n2 k1} sum_n1 x[P2 n1 + n2] W_P1^{n1 k1}.
// Column pass: the P1-point FFTs over n1 (stride P2), four columns per block staged in shared
// memory, then the twiddle W_P^{n2 k1}; row pass: the P2-point FFTs over n2 (contiguous).
// Spectra stay in the register-slot orders of the two in-block FFTs (row r = j*NT1 + t holds
// k1 of slot j of thread t; likewise the columns): the product needs only the same order for x
// and h, and the inverse runs the passes backwards to natural order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <new>

#include "fdas_internal.cuh"
#include "fft_regs.cuh"
#include "ols_common.cuh"
#include "ptx.cuh"

namespace fdas {

namespace fd {
constexpr int P1 = 2048, NT1 = P1 / 16, TB = 4, TBP = TB + 1;   // tile rows padded to 5 values
constexpr size_t col_smem_bytes()
{
    return sizeof(float2) * ((size_t)P1 * TBP + P1 + 16 * (NT1 + 1));
}
constexpr int CT_INV = 4;   // columns per block of the inverse column pass
constexpr size_t col_inv_smem_bytes() { return sizeof(float2) * (16 * (NT1 + 1) + 8) * CT_INV; }
template <int P2>
constexpr size_t row_inv_smem_bytes() { return sizeof(float2) * 16 * (P2 / 16 + 1); }
template <int P2>
constexpr size_t row_smem_bytes()
{
    return sizeof(float2) * ((size_t)P2 + 16 * (P2 / 16 + 1));
}

// The 2 M launches of a call overlap (programmatic dependent launch): every block lets the next
// launch start as soon as all blocks of this one run, and waits for the launch before it only
// where it touches the scratch B that the two passes hand back and forth.  A block of launch i
// passes its wait before it ends, so the end of a launch implies the end of all before it.
// 85 templates of 2^23 points: 5896 us without the overlap, 5046 with it (gaps and last waves).

// exp(dir * 2 pi i e / P), e < P <= 2^23 (the argument 2e/P is exact in FP32)
__device__ __forceinline__ float2 twiddle_p(int e, float two_over_p, float dir)
{
    float s, c;
    sincospif(dir * (float)e * two_over_p, &s, &c);
    return make_float2(c, s);
}
}  // namespace fd

// Column pass, forward: columns n2 = blockIdx.x * TB + t of in[P2 n1 + n2] (zero at and beyond
// len) -> A[r][n2] = scale * W_P^{n2 k1} * FFT_P1 over n1, row r = j*NT1 + t for slot j of t.
template <int P2>
__global__ void __launch_bounds__(fd::NT1) fdfir_col_fwd(const float2 *__restrict__ in, int64_t len,
                                                        const float2 *__restrict__ tw1, float2 *__restrict__ A,
                                                        float scale)
{
    using namespace fd;
    extern __shared__ float2 fd_smem[];
    float2 *tile = fd_smem, *e1 = tile + (size_t)P1 * TBP, *e2 = e1 + P1;
    const int tid = threadIdx.x, n2_0 = blockIdx.x * TB;
    constexpr float two_over_p = 2.0f / ((float)P1 * (float)P2);
    for (int idx = tid; idx < P1 * TB; idx += NT1) {
        const int n1 = idx / TB, t = idx % TB;
        const int64_t e = (int64_t)P2 * n1 + n2_0 + t;
        tile[n1 * TBP + t] = e < len ? in[e] : make_float2(0.f, 0.f);
    }
    for (int t = 0; t < TB; ++t) {
        __syncthreads();   // tile loaded; the previous column's exchanges are read
#pragma unroll
        for (int m = 0; m < 16; ++m) e1[m * NT1 + tid] = tile[(m * NT1 + tid) * TBP + t];
        __syncthreads();
        float2 v[16], X[16];
        forward_fft<P1>(e1, e2, tw1, v, X);
        const int n2 = n2_0 + t;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int k1 = freq_of_slot(P1, tid, j);
            const float2 w = twiddle_p(n2 * k1, two_over_p, -1.f);   // n2 k1 < 2^23
            const float2 y = cmul(X[j], w);
            tile[(j * NT1 + tid) * TBP + t] = make_float2(scale * y.x, scale * y.y);
        }
    }
    __syncthreads();
    for (int idx = tid; idx < P1 * TB; idx += NT1) {
        const int r = idx / TB, t = idx % TB;
        A[(size_t)r * P2 + n2_0 + t] = tile[r * TBP + t];
    }
}

// Row pass, forward, in place: row blockIdx.x of A (natural order over n2) -> its P2-point
// spectrum, column c = j*NT2 + t for slot j of thread t.
template <int P2>
__global__ void __launch_bounds__(P2 / 16) fdfir_row_fwd(float2 *__restrict__ A, const float2 *__restrict__ tw2)
{
    constexpr int NT2 = P2 / 16;
    extern __shared__ float2 fd_smem[];
    float2 *e1 = fd_smem, *e2 = e1 + P2;
    const int tid = threadIdx.x;
    float2 *row = A + (size_t)blockIdx.x * P2;
#pragma unroll
    for (int m = 0; m < 16; ++m) e1[m * NT2 + tid] = row[m * NT2 + tid];
    __syncthreads();
    float2 v[16], X[16];
    forward_fft<P2>(e1, e2, tw2, v, X);   // every read of the row precedes its barriers
#pragma unroll
    for (int j = 0; j < 16; ++j) row[j * NT2 + tid] = X[j];
}

// Inverse L-point FFT (unnormalised) of CT independent transforms by L/16 threads each, thread
// (t, column) from the C distribution the forward transform leaves to natural order, v[a] =
// y[a NT + t].  Passes C', B', A' with the twiddles of B' and A' folded into the butterflies
// (dft_twiddled: 16 factors read per thread instead of 31 twiddles); both exchanges go through
// `ex` (16 (NT + 1) CT values, the columns side by side), free on entry, with a barrier between
// the reads of the first and the stores of the second: half the shared memory, so that twice as
// many blocks share an SM.
template <int L, int CT>
__device__ __forceinline__ void inverse_fft_folded(float2 (&v)[16], float2 *ex, const float2 *__restrict__ tw, int t, int col)
{
    using Gm = Geo<L>;
    constexpr int NT = Gm::NT, Q = Gm::Q, R = Gm::R, GB = Gm::GB, GC = Gm::GC, LD = NT + 1, MASK = L - 1;
    const int k1 = t & 15, hi = t >> 4;
    dft<R, 1, 1, 0>(v);
    if constexpr (GC == 2) dft<R, 1, 1, R>(v);
#pragma unroll
    for (int g = 0; g < GC; ++g)
#pragma unroll
        for (int c = 0; c < R; ++c) ex[(k1 + 16 * (hi + (NT / 16) * g) + 16 * Q * c) * CT + col] = v[g * R + c];
    float2 w[8];
#pragma unroll
    for (int g = 0; g < GB; ++g)
        twiddle_factors<Q>(L, 16 * (hi + (NT / 16) * g), [&](int i, int e) { w[g * (Q / 2) + i] = cconj(__ldg(&tw[e & MASK])); });
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GB; ++g) {
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) v[g * Q + k2] = ex[(k1 + 16 * k2 + 16 * Q * (hi + (NT / 16) * g)) * CT + col];
        dft_twiddled<Q>(v + g * Q, w + g * (Q / 2));
    }
    twiddle_factors<16>(L, t, [&](int i, int e) { w[i] = cconj(__ldg(&tw[e & MASK])); });
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GB; ++g)
#pragma unroll
        for (int b = 0; b < Q; ++b) ex[((b * R + hi + (NT / 16) * g) + LD * k1) * CT + col] = v[g * Q + b];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = ex[(t + LD * k) * CT + col];
    dft_twiddled<16>(v, w);
}

// Row pass, inverse, with the product: B[r][n2] = IFFT_P2 over k2 of X[r][.] * H[r][.].
// Bound by memory latency (X from L2, H streamed from DRAM, B written): 32 us per 2^23-point
// template against 50 us with two exchange buffers and 31 twiddle loads per thread.  X and B together
// (134 MB) do not fit L2, and a cyclic walk of X would miss always (read from DRAM whole for every
// template); templates walk the rows up and down in turn, so that what the last one read last is
// read first, and what is read or written once (H, the plane, B in the column pass) is marked
// streaming: 5054 -> 4901 us for 85 templates.
template <int P2>
__global__ void __launch_bounds__(P2 / 16) fdfir_row_inv(const float2 *__restrict__ X, const float2 *__restrict__ H,
                                                         float2 *__restrict__ B, const float2 *__restrict__ tw2, bool up)
{
    constexpr int NT2 = P2 / 16;
    extern __shared__ float2 fd_smem[];
    const int tid = threadIdx.x;
    const size_t off = (size_t)(up ? blockIdx.x : gridDim.x - 1 - blockIdx.x) * P2 + tid;
    float2 v[16];
    launch_dependents();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = cmul(__ldg(&X[off + j * NT2]), __ldcs(&H[off + j * NT2]));
    inverse_fft_folded<P2, 1>(v, fd_smem, tw2, tid, 0);
    wait_prerequisites();   // the column pass of the previous template has read B
#pragma unroll
    for (int a = 0; a < 16; ++a) B[off + a * NT2] = v[a];
}

// Column pass, inverse, with the power: out[P2 n1 + n2] = |IFFT_P1 over k1 of
// W_P^{-n2 k1} B[r(k1)][n2]|^2 for P2 n1 + n2 < n.
//
// CT columns at once: thread (t, column) with the column in the low bits of the thread index, so
// that a row's CT values are read straight into registers as one contiguous run, all 16 loads of
// a thread in flight, and the exchanges (values of the CT columns side by side, one buffer used
// twice) are free of bank conflicts.  The twiddle of slot (g, k3) is a base per g times a step
// per k3: two sincospif per thread and 8 per column.
template <int P2, int CT>
__global__ void __launch_bounds__(fd::NT1 *CT, 2) fdfir_col_inv(const float2 *__restrict__ B, const float2 *__restrict__ tw1,
                                                               float *__restrict__ out, int64_t n)
{
    using namespace fd;
    constexpr int R = Geo<P1>::R, NT = NT1, LD = NT + 1;
    static_assert(R == 8, "slots (g, k3) of the 2048-point transform");
    constexpr float two_over_p = 2.0f / ((float)P1 * (float)P2);
    extern __shared__ float2 fd_smem[];
    float2 *ex = fd_smem, *step = fd_smem + (size_t)16 * LD * CT;
    const int col = threadIdx.x % CT, t = threadIdx.x / CT, k1 = t & 15, hi = t >> 4;
    const int n2 = blockIdx.x * CT + col;
    launch_dependents();
    if (t < 8) step[t * CT + col] = twiddle_p(n2 * 256 * t, two_over_p, 1.f);   // n2 k1 < 2^23
    const float2 base0 = twiddle_p(n2 * (k1 + 16 * hi), two_over_p, 1.f);
    const float2 base1 = twiddle_p(n2 * (k1 + 16 * (hi + NT / 16)), two_over_p, 1.f);
    wait_prerequisites();   // the row pass has written B
    float2 v[16];
    const float2 *src = B + (size_t)t * P2 + n2;
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __ldcs(src + (size_t)j * NT * P2);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < R; ++c) {
        const float2 s = step[c * CT + col];
        v[c] = cmul(v[c], c == 0 ? base0 : cmul(base0, s));
        v[R + c] = cmul(v[R + c], c == 0 ? base1 : cmul(base1, s));
    }
    inverse_fft_folded<P1, CT>(v, ex, tw1, t, col);
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        const int64_t i = (int64_t)P2 * (a * NT + t) + n2;
        if (i < n) __stcs(&out[i], cabs2(v[a]));
    }
}

template <int P2>
static cudaError_t fdfir_attrs()
{
    static bool done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(fdfir_col_fwd<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)fd::col_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fdfir_col_inv<P2, fd::CT_INV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fd::col_inv_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fdfir_row_fwd<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fd::row_smem_bytes<P2>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fdfir_row_inv<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fd::row_inv_smem_bytes<P2>());
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

// Forward P-point transform of in[0, len) (zero-padded) into A, times scale.
template <int P2>
static cudaError_t fdfir_forward_l(const float2 *in, int64_t len, const float2 *tw1, const float2 *tw2, float2 *A,
                                   float scale, cudaStream_t s)
{
    cudaError_t e = fdfir_attrs<P2>();
    if (e != cudaSuccess) return e;
    fdfir_col_fwd<P2><<<P2 / fd::TB, fd::NT1, fd::col_smem_bytes(), s>>>(in, len, tw1, A, scale);
    fdfir_row_fwd<P2><<<fd::P1, P2 / 16, fd::row_smem_bytes<P2>(), s>>>(A, tw2);
    return cudaGetLastError();
}

// Inverse transform of X . H into the power row out[0, n).
template <int P2>
static cudaError_t fdfir_inverse_l(const float2 *X, const float2 *H, float2 *B, const float2 *tw1, const float2 *tw2,
                                   float *out, int64_t n, bool first, bool up, cudaStream_t s)
{
    cudaError_t e = fdfir_attrs<P2>();
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(fd::P1);
    cfg.blockDim = dim3(P2 / 16);
    cfg.dynamicSmemBytes = fd::row_inv_smem_bytes<P2>();
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = first ? 0 : 1;   // the first row pass follows the transform that writes X
    if ((e = cudaLaunchKernelEx(&cfg, fdfir_row_inv<P2>, X, H, B, tw2, up)) != cudaSuccess) return e;
    cfg.gridDim = dim3(P2 / fd::CT_INV);
    cfg.blockDim = dim3(fd::NT1 * fd::CT_INV);
    cfg.dynamicSmemBytes = fd::col_inv_smem_bytes();
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fdfir_col_inv<P2, fd::CT_INV>, (const float2 *)B, tw1, out, n);
}

cudaError_t fdfir_forward(int P2, const float2 *in, int64_t len, const float2 *tw1, const float2 *tw2, float2 *A,
                          float scale, cudaStream_t s)
{
    switch (P2) {
    case 1024: return fdfir_forward_l<1024>(in, len, tw1, tw2, A, scale, s);
    case 2048: return fdfir_forward_l<2048>(in, len, tw1, tw2, A, scale, s);
    case 4096: return fdfir_forward_l<4096>(in, len, tw1, tw2, A, scale, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t fdfir_inverse(int P2, const float2 *X, const float2 *H, float2 *B, const float2 *tw1, const float2 *tw2,
                          float *out, int64_t n, bool first, bool up, cudaStream_t s)
{
    switch (P2) {
    case 1024: return fdfir_inverse_l<1024>(X, H, B, tw1, tw2, out, n, first, up, s);
    case 2048: return fdfir_inverse_l<2048>(X, H, B, tw1, tw2, out, n, first, up, s);
    case 4096: return fdfir_inverse_l<4096>(X, H, B, tw1, tw2, out, n, first, up, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fdas

// ---- C ABI -------------------------------------------------------------------------------

struct fdas_fdfir_s {
    int device = -1;
    int64_t n_max = 0, P = 0;
    int M = 0, K = 0, P2 = 0;
    float2 *d_H = nullptr;      // [M][P] template spectra / P (slot orders of the two passes)
    float2 *d_X = nullptr;      // [P] input spectrum
    float2 *d_B = nullptr;      // [P] row-pass output of the inverse
    float2 *d_tw1 = nullptr;    // [P1] W_P1, FP32 from FP64
    float2 *d_tw2 = nullptr;    // [P2] W_P2
    double2 *d_tw64 = nullptr;  // FP64 twiddle scratch
};

namespace {

void fdfir_free(fdas_fdfir f)
{
    if (!f) return;
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(f->device);
    cudaFree(f->d_H);
    cudaFree(f->d_X);
    cudaFree(f->d_B);
    cudaFree(f->d_tw1);
    cudaFree(f->d_tw2);
    cudaFree(f->d_tw64);
    if (prev >= 0) cudaSetDevice(prev);
    delete f;
}

int fdfir_cuda(cudaError_t e, const char *what)
{
    char buf[256];
    snprintf(buf, sizeof buf, "%s: %s (%s)", what, cudaGetErrorString(e), cudaGetErrorName(e));
    return fdas::set_error(e == cudaErrorMemoryAllocation ? FDAS_ERR_OOM : FDAS_ERR_CUDA, buf);
}

}  // namespace

extern "C" {

int fdas_fdfir_create(fdas_fdfir *out, int64_t n_max, const void *templates, int M, int K)
{
    if (!out) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null output handle");
    *out = nullptr;
    if (!templates) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null templates");
    if (M < 1 || K < 1) return fdas::set_error(FDAS_ERR_INVALID_ARG, "n_templates and tpl_len must be >= 1");
    if (n_max < 1) return fdas::set_error(FDAS_ERR_INVALID_ARG, "n_max must be >= 1");
    int64_t P = int64_t(1) << 21;
    while (P < n_max + K - 1) P <<= 1;
    if (P > (int64_t(1) << 23)) return fdas::set_error(FDAS_ERR_INVALID_ARG, "n_max + tpl_len - 1 exceeds 2^23");
    fdas_fdfir f = new (std::nothrow) fdas_fdfir_s;
    if (!f) return fdas::set_error(FDAS_ERR_OOM, "host allocation");
    if (cudaGetDevice(&f->device) != cudaSuccess) {
        delete f;
        return fdas::set_error(FDAS_ERR_CUDA, "no current CUDA device");
    }
    f->n_max = n_max;
    f->P = P;
    f->M = M;
    f->K = K;
    f->P2 = (int)(P / fdas::fd::P1);
    cudaError_t e;
    float2 *d_h = nullptr;
    const size_t h_bytes = sizeof(float2) * (size_t)M * K;
    int rc = FDAS_OK;
    if ((e = cudaMalloc(&f->d_H, sizeof(float2) * (size_t)M * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc spectra");
    else if ((e = cudaMalloc(&f->d_X, sizeof(float2) * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc input spectrum");
    else if ((e = cudaMalloc(&f->d_B, sizeof(float2) * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc scratch");
    else if ((e = cudaMalloc(&f->d_tw1, sizeof(float2) * fdas::fd::P1)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&f->d_tw2, sizeof(float2) * f->P2)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&f->d_tw64, sizeof(double2) * std::max(fdas::fd::P1, f->P2))) != cudaSuccess)
        rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&d_h, h_bytes)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc template staging");
    else if ((e = cudaMemcpy(d_h, templates, h_bytes, cudaMemcpyHostToDevice)) != cudaSuccess) rc = fdfir_cuda(e, "copy templates");
    else if ((e = fdas::launch_twiddles(fdas::fd::P1, f->d_tw64, f->d_tw1, nullptr)) != cudaSuccess) rc = fdfir_cuda(e, "twiddles");
    else if ((e = fdas::launch_twiddles(f->P2, f->d_tw64, f->d_tw2, nullptr)) != cudaSuccess) rc = fdfir_cuda(e, "twiddles");
    for (int z = 0; rc == FDAS_OK && z < M; ++z) {
        e = fdas::fdfir_forward(f->P2, d_h + (size_t)z * K, K, f->d_tw1, f->d_tw2, f->d_H + (size_t)z * P,
                                1.0f / (float)P, nullptr);
        if (e != cudaSuccess) rc = fdfir_cuda(e, "template transforms");
    }
    if (rc == FDAS_OK && (e = cudaDeviceSynchronize()) != cudaSuccess) rc = fdfir_cuda(e, "plan-time kernels");
    cudaFree(d_h);
    if (rc != FDAS_OK) {
        fdfir_free(f);
        return rc;
    }
    *out = f;
    return FDAS_OK;
}

int fdas_fdfir_length(fdas_fdfir f, int64_t *P)
{
    if (!f || !P) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null argument");
    *P = f->P;
    return FDAS_OK;
}

int fdas_fdfir_convolve(fdas_fdfir f, const void *in, int64_t n, float *out, void *stream)
{
    if (!f) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null plan");
    if (!in || !out) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null input or output pointer");
    if (n < 1 || n > f->n_max) return fdas::set_error(FDAS_ERR_INVALID_ARG, "n outside [1, n_max]");
    if (reinterpret_cast<uintptr_t>(in) % 8 || reinterpret_cast<uintptr_t>(out) % 4)
        return fdas::set_error(FDAS_ERR_INVALID_ARG, "misaligned input or output pointer");
    const uintptr_t i0 = reinterpret_cast<uintptr_t>(in), i1 = i0 + (uintptr_t)n * 8;
    const uintptr_t o0 = reinterpret_cast<uintptr_t>(out), o1 = o0 + (uintptr_t)n * 4 * (uintptr_t)f->M;
    if (i0 < o1 && o0 < i1) return fdas::set_error(FDAS_ERR_INVALID_ARG, "input and output overlap");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != f->device && cudaSetDevice(f->device) != cudaSuccess)
        return fdas::set_error(FDAS_ERR_CUDA, "cannot select plan device");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = fdas::fdfir_forward(f->P2, static_cast<const float2 *>(in), n, f->d_tw1, f->d_tw2, f->d_X, 1.0f, s);
    for (int z = 0; e == cudaSuccess && z < f->M; ++z)
        e = fdas::fdfir_inverse(f->P2, f->d_X, f->d_H + (size_t)z * f->P, f->d_B, f->d_tw1, f->d_tw2,
                                out + (size_t)z * n, n, z == 0, z % 2 == 0, s);
    if (prev >= 0 && prev != f->device) cudaSetDevice(prev);
    if (e != cudaSuccess) return fdfir_cuda(e, "full-length FD-FIR launch");
    return FDAS_OK;
}

int fdas_fdfir_destroy(fdas_fdfir f)
{
    if (!f) return fdas::set_error(FDAS_ERR_INVALID_ARG, "null plan");
    fdfir_free(f);
    return FDAS_OK;
}

}  // extern "C"
