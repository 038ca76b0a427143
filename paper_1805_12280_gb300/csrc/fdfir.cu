// Full-length frequency-domain FIR (Eq. 2): y_z = IFFT_P(FFT_P(x) . FFT_P(h_z)) with P >= n + K - 1
// a power of two, then |y_z|^2 for i < n -- the "naive" FD-FIR that the paper weighs against
// overlap-save (Sec. 3.2.1, Table 1), kept to measure that choice on this GPU.
//
// P-point transforms in four steps, P = P1 * P2 with P1 = 1024 and P2 in {2048, 4096, 8192}:
//   n = P2 n1 + n2,  k = k1 + P1 k2,
//   X[k1 + P1 k2] = sum_n2 W_P2^{n2 k2} W_P^{n2 k1} sum_n1 x[P2 n1 + n2] W_P1^{n1 k1}.
// Column pass: the P1-point FFTs over n1 (stride P2), eight columns per block, then the twiddle
// W_P^{n2 k1}; row pass: the P2-point FFTs over n2 (contiguous; 8192 points as two in-block
// transforms of 4096 joined by one more butterfly).  Spectra stay in the register-slot orders of
// the in-block FFTs (row r = j*NT1 + t holds k1 of slot j of thread t; likewise the columns): the
// product needs only the same order for x and h, and the inverse runs the passes backwards to
// natural order.
//
// Why 1024 x P2: a block's piece of a row is 8 values (64 bytes).  With 2048-point columns four
// fit a block, and their 32-byte pieces (8 cache lines per request of a warp) cost the load/store
// pipe as much as both exchanges of the transform.  85 templates, largest array of P = 2^21 / 2^22, and
// 2^22 points at P = 2^23: 1048 / 2260 / 4470 us (4117 / 8237 / 14316 in the form before: columns of
// 2048 points one after another in a block, the two passes in launches that did not overlap).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <new>
#include <type_traits>

#include "fdas_internal.cuh"
#include "fft_regs.cuh"
#include "ols_common.cuh"
#include "ptx.cuh"

namespace fdas {

namespace fd {
constexpr int P1 = 1024, NT1 = P1 / 16;
constexpr int CT = 8, NT_INV = NT1 * CT;   // columns and threads per block
constexpr int row_halves(int P2) { return P2 > 4096 ? 2 : 1; }
// points and threads of one in-block row transform
constexpr int row_points(int P2) { return P2 / row_halves(P2); }
constexpr int row_threads(int P2) { return row_points(P2) / 16; }
template <int P2>
constexpr size_t row_smem_bytes()
{
    return sizeof(float2) * row_halves(P2) * 16 * (row_threads(P2) + 1);
}
constexpr size_t col_smem_bytes() { return sizeof(float2) * (16 * (NT1 + 1) + 8) * CT; }
template <int P2>
constexpr size_t inv_smem_bytes()
{
    constexpr size_t col = col_smem_bytes();
    constexpr size_t row = sizeof(float2) * 16 * (row_threads(P2) + 1) * (NT_INV / row_threads(P2));
    return col > row ? col : row;
}

// The M + 1 inverse launches of a call overlap (programmatic dependent launch): every block lets
// the next launch start as soon as all blocks of this one run, and waits for the launch before it
// only where it touches the scratch B that the passes hand on.  A block of launch i passes its wait
// before it ends, so the end of a launch implies the end of all before it.

// exp(dir * 2 pi i e / P), e < P <= 2^23 (the argument 2e/P is exact in FP32)
__device__ __forceinline__ float2 twiddle_p(int e, float two_over_p, float dir)
{
    float s, c;
    sincospif(dir * (float)e * two_over_p, &s, &c);
    return make_float2(c, s);
}
}  // namespace fd

// Forward L-point FFT of CT independent transforms by L/16 threads each, thread (t, column) from
// natural order, v[j] = x[j NT + t], to the C distribution (freq_of_slot); NH = 2 and s = 1: at the
// frequencies k + 1/2.  Computed as the conjugate of the inverse of the conjugate, so that passes B
// and C take the folded butterflies: what depends on c alone of pass B's twiddle W^{(b R + c) k1}
// is left to pass C, whose factors become W^{k1 + 16 k2}.  tw: W_{NH L}; ex as in
// inverse_fft_folded.
template <int L, int CT, int NH = 1>
__device__ __forceinline__ void forward_fft_folded(float2 (&v)[16], float2 *ex, const float2 *__restrict__ tw, int t, int col,
                                                   int s = 0)
{
    using Gm = Geo<L>;
    constexpr int NT = Gm::NT, Q = Gm::Q, R = Gm::R, GB = Gm::GB, GC = Gm::GC, LD = NT + 1, T = NH * L;
    const int k1 = t & 15, hi = t >> 4;
    float2 w[8];
    auto factors = [&](auto n, int e, int at) {
        twiddle_factors<n()>(T, e, [&](int i, int x) { w[at + i] = cconj(__ldg(&tw[x & (T - 1)])); });
    };
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = cconj(v[j]);
    if (NH == 2 && s) {
        factors(std::integral_constant<int, 16>{}, T / 32, 0);
        dft_twiddled<16>(v, w);
    } else {
        dft<16, 1>(v);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) ex[(t + LD * k) * CT + col] = v[k];
#pragma unroll
    for (int g = 0; g < GB; ++g) factors(std::integral_constant<int, Q>{}, R * (NH * k1 + s), g * (Q / 2));
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GB; ++g) {
#pragma unroll
        for (int b = 0; b < Q; ++b) v[g * Q + b] = ex[(b * R + hi + (NT / 16) * g + LD * k1) * CT + col];
        dft_twiddled<Q>(v + g * Q, w + g * (Q / 2));
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GB; ++g)
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) ex[(k1 + 16 * k2 + 16 * Q * (hi + (NT / 16) * g)) * CT + col] = v[g * Q + k2];
#pragma unroll
    for (int g = 0; g < GC; ++g)
        factors(std::integral_constant<int, R>{}, NH * (k1 + 16 * (hi + (NT / 16) * g)) + s, g * (R / 2));
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GC; ++g) {
#pragma unroll
        for (int c = 0; c < R; ++c) v[g * R + c] = ex[(k1 + 16 * (hi + (NT / 16) * g) + 16 * Q * c) * CT + col];
        dft_twiddled<R>(v + g * R, w + g * (R / 2));
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = cconj(v[j]);
}

// Column pass, forward: columns n2 = blockIdx.x * CT + col of in[P2 n1 + n2] (zero at and beyond
// len) -> A[r][n2] = scale * W_P^{n2 k1} * FFT_P1 over n1, row r = j*NT1 + t for slot j of t.
// Thread (t, column) as in the inverse pass.
template <int P2>
__global__ void __launch_bounds__(fd::NT_INV, 2) fdfir_col_fwd(const float2 *__restrict__ in, int64_t len,
                                                              const float2 *__restrict__ tw1, float2 *__restrict__ A,
                                                              float scale)
{
    using namespace fd;
    constexpr float two_over_p = 2.0f / ((float)P1 * (float)P2);
    extern __shared__ float2 fd_smem[];
    const int col = threadIdx.x % CT, t = threadIdx.x / CT, n2 = blockIdx.x * CT + col;
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int64_t i = (int64_t)P2 * (j * NT1 + t) + n2;
        v[j] = i < len ? in[i] : make_float2(0.f, 0.f);
    }
    forward_fft_folded<P1, CT>(v, fd_smem, tw1, t, col);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const float2 y = cmul(v[j], twiddle_p(n2 * freq_of_slot(P1, t, j), two_over_p, -1.f));   // n2 k1 < 2^23
        A[(size_t)(j * NT1 + t) * P2 + n2] = make_float2(scale * y.x, scale * y.y);
    }
}

// Row pass, forward, in place: row blockIdx.x of A (natural order over n2) -> its P2-point
// spectrum, column c = j*NT2 + t for slot j of thread t; 8192 points: the even and the odd
// frequencies, each from 4096 sums or differences by its own threads (threadIdx.y).
template <int P2>
__global__ void __launch_bounds__(P2 / 16) fdfir_row_fwd(float2 *__restrict__ A, const float2 *__restrict__ tw)
{
    constexpr int PR = fd::row_points(P2), NT2 = fd::row_threads(P2), NH = fd::row_halves(P2);
    extern __shared__ float2 fd_smem[];
    const int tid = threadIdx.x, h = NH == 2 ? threadIdx.y : 0;
    float2 *row = A + (size_t)blockIdx.x * P2, v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        v[m] = row[m * NT2 + tid];
        if constexpr (NH == 2) {
            const float2 y = row[m * NT2 + tid + PR];
            v[m] = h ? make_float2(v[m].x - y.x, v[m].y - y.y) : make_float2(v[m].x + y.x, v[m].y + y.y);
        }
    }
    // every read of the row precedes its barriers
    forward_fft_folded<PR, 1, NH>(v, fd_smem + (size_t)h * 16 * (NT2 + 1), tw, tid, 0, h);
#pragma unroll
    for (int j = 0; j < 16; ++j) row[h * PR + j * NT2 + tid] = v[j];
}

// tw[L + i L/16 + t]: the factors of the last pass, twiddle_factors<16>(L, t), after the table W_L.
__global__ void fdfir_factors(int L, float2 *tw)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < L / 16) twiddle_factors<16>(L, t, [&](int i, int e) { tw[L + i * (L / 16) + t] = cconj(tw[e & (L - 1)]); });
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
    if constexpr (CT == 1) {   // 32 t per warp: 40 lines from W_L, 16 from the table
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = __ldg(&tw[L + i * NT + t]);
    } else {
        twiddle_factors<16>(L, t, [&](int i, int e) { w[i] = cconj(__ldg(&tw[e & MASK])); });
    }
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

// Row pass, inverse, with the product: B[r][n2] = IFFT_P2 over k2 of X[r][.] * H[r][.]; unit: the
// rows of one block.  X and the two B (201 MB at P = 2^23) do not fit L2, and a cyclic walk of X
// would miss always; templates walk the rows up and down in turn, so that what the last one read
// last is read first (one direction, largest array of P = 2^22: 2300 us against 2256), and what is
// used once is marked streaming: H always, X where it would push B out (2^23: 4471 us, 4628 if not; at
// 2^21, where it stays, 1048 against 1091 with the mark).
template <int P2>
__device__ __forceinline__ void row_inv(const float2 *__restrict__ X, const float2 *__restrict__ H, float2 *__restrict__ B,
                                        const float2 *__restrict__ tw2, const float2 *__restrict__ twr, int unit, float2 *smem)
{
    constexpr int PR = fd::row_points(P2), NT2 = fd::row_threads(P2), G = fd::NT_INV / NT2;
    const int t = threadIdx.x % NT2, g = threadIdx.x / NT2;
    const size_t off = (size_t)(unit * G + g) * PR + t;
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = cmul((P2 > 4096 ? __ldcs(&X[off + j * NT2]) : __ldg(&X[off + j * NT2])), __ldcs(&H[off + j * NT2]));
    inverse_fft_folded<PR, 1>(v, smem + (size_t)g * 16 * (NT2 + 1), tw2, t, 0);
    if constexpr (fd::row_halves(P2) == 1) {
        wait_prerequisites();   // the columns that read this B are done
#pragma unroll
        for (int a = 0; a < 16; ++a) B[off + a * NT2] = v[a];
    } else {
        // y[n2] = e[n2] + W_P2^-n2 o[n2], y[n2 + PR] = e - W o, of the transforms e of the even and
        // o of the odd frequencies: the two groups of threads trade halves of theirs
        static_assert(G == 2, "one row per block");
        float2 u[8];
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 8; ++a) smem[g * (PR / 2) + a * NT2 + t] = g ? v[a] : v[8 + a];
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 8; ++a) u[a] = smem[(1 - g) * (PR / 2) + a * NT2 + t];
        wait_prerequisites();
        float2 *row = B + (size_t)unit * P2 + g * (PR / 2) + t;
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            float2 e = g ? u[a] : v[a], o = g ? v[8 + a] : u[a];
            const float2 w = __ldg(&twr[g * (PR / 2) + a * NT2 + t]);
            bfly_w(e, o, w.x, -w.y);
            row[a * NT2] = e;
            row[a * NT2 + PR] = o;
        }
    }
}

// Column pass, inverse, with the power: out[P2 n1 + n2] = |IFFT_P1 over k1 of
// W_P^{-n2 k1} B[r(k1)][n2]|^2 for P2 n1 + n2 < n.
//
// CT columns at once: thread (t, column) with the column in the low bits of the thread index, so
// that a row's CT values are read straight into registers as one contiguous run, all 16 loads of
// a thread in flight, and the exchanges (values of the CT columns side by side, one buffer used
// twice) are free of bank conflicts.  The twiddle of slot (g, k3) is a base per g times a step
// per k3: two sincospif per thread and 8 per column.  B is marked streaming where two templates'
// B do not fit L2 (2^23: 4471 us, 4598 if not; 2^22: 2256 against 2287).
template <int P2>
__device__ __forceinline__ void col_inv(const float2 *__restrict__ B, const float2 *__restrict__ tw1,
                                        float *__restrict__ out, int64_t n, int n2_0, float2 *fd_smem)
{
    using namespace fd;
    constexpr int R = Geo<P1>::R, Q = Geo<P1>::Q, NT = NT1, LD = NT + 1;
    static_assert(R == 8, "slots (g, k3) of the 1024-point transform");
    constexpr float two_over_p = 2.0f / ((float)P1 * (float)P2);
    float2 *ex = fd_smem, *step = fd_smem + (size_t)16 * LD * CT;
    const int col = threadIdx.x % CT, t = threadIdx.x / CT, k1 = t & 15, hi = t >> 4;
    const int n2 = n2_0 + col;
    if (t < 8) step[t * CT + col] = twiddle_p(n2 * 16 * Q * t, two_over_p, 1.f);   // n2 k1 < 2^23
    const float2 base0 = twiddle_p(n2 * (k1 + 16 * hi), two_over_p, 1.f);
    const float2 base1 = twiddle_p(n2 * (k1 + 16 * (hi + NT / 16)), two_over_p, 1.f);
    wait_prerequisites();   // the rows have written B
    float2 v[16];
    const float2 *src = B + (size_t)t * P2 + n2;
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = P2 > 2048 ? __ldcs(src + (size_t)j * NT * P2) : __ldcg(src + (size_t)j * NT * P2);
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

// One launch: the rows of one template (H given) and the columns of the one before (out given),
// each on half of the blocks; two B buffers alternate.  The row pass waits on memory (X and H
// from DRAM) while the column pass keeps the load/store pipe busy: together they take less than
// one after the other (10 / 2 / 1 % of a call at P = 2^21 / 2^22 / 2^23 when it was made).  Blocks of the
// two kinds in turn, so that an SM holds one of each; P = 2^21 with the rows first, since its 512 blocks
// are two waves and the rows, which start before the launch ahead has ended, fill the first (in turn
// 1154 us against 1048; no gain above).
template <int P2>
__global__ void __launch_bounds__(fd::NT_INV, 2) fdfir_inv_step(const float2 *__restrict__ X, const float2 *__restrict__ H,
                                                               float2 *__restrict__ Bw, const float2 *__restrict__ Br,
                                                               const float2 *__restrict__ tw1, const float2 *__restrict__ tw2,
                                                               const float2 *__restrict__ twr, float *__restrict__ out,
                                                               int64_t n, bool up)
{
    using namespace fd;
    extern __shared__ float2 fd_smem[];
    constexpr int NB = P2 / CT;
    static_assert(NB * NT_INV * 16 == P1 * P2, "as many blocks of rows as of columns");
    launch_dependents();
    const bool both = H && out;
    const int b = !both ? blockIdx.x : P2 > 2048 ? blockIdx.x >> 1 : blockIdx.x % NB;
    if (both ? (P2 > 2048 ? (blockIdx.x & 1) == 0 : blockIdx.x < NB) : H != nullptr)
        row_inv<P2>(X, H, Bw, tw2, twr, up ? b : NB - 1 - b, fd_smem);
    else
        col_inv<P2>(Br, tw1, out, n, b * CT, fd_smem);
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
        e = cudaFuncSetAttribute(fdfir_row_fwd<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fd::row_smem_bytes<P2>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(fdfir_inv_step<P2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fd::inv_smem_bytes<P2>());
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

// Forward P-point transform of in[0, len) (zero-padded) into A, times scale.
template <int P2>
static cudaError_t fdfir_forward_l(const float2 *in, int64_t len, const FdfirTables &tw, float2 *A, float scale, cudaStream_t s)
{
    cudaError_t e = fdfir_attrs<P2>();
    if (e != cudaSuccess) return e;
    fdfir_col_fwd<P2><<<P2 / fd::CT, fd::NT_INV, fd::col_smem_bytes(), s>>>(in, len, tw.w1, A, scale);
    fdfir_row_fwd<P2><<<fd::P1, dim3(fd::row_threads(P2), fd::row_halves(P2)), fd::row_smem_bytes<P2>(), s>>>(A, tw.wr);
    return cudaGetLastError();
}

// Inverse transforms of X . H_z into the power rows out[z][0, n).
template <int P2>
static cudaError_t fdfir_inverse_l(const float2 *X, const float2 *H, int M, float2 *B, const FdfirTables &tw, float *out,
                                   int64_t n, cudaStream_t s)
{
    cudaError_t e = fdfir_attrs<P2>();
    if (e != cudaSuccess) return e;
    constexpr int64_t P = (int64_t)fd::P1 * P2;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(fd::NT_INV);
    cfg.dynamicSmemBytes = fd::inv_smem_bytes<P2>();
    cfg.stream = s;
    cfg.attrs = &attr;
    auto step = [&](int zr, int zc) {   // rows of template zr and columns of template zc, -1: none
        cfg.gridDim = dim3((zr >= 0 && zc >= 0 ? 2 : 1) * (P2 / fd::CT));
        cfg.numAttrs = zr == 0 ? 0 : 1;   // the first rows follow the transform that writes X
        return cudaLaunchKernelEx(&cfg, fdfir_inv_step<P2>, X, zr >= 0 ? H + zr * P : nullptr, B + (zr & 1) * P,
                                  (const float2 *)(B + (zc & 1) * P), tw.w1, tw.w2, tw.wr,
                                  zc >= 0 ? out + (size_t)zc * n : nullptr, n, zr % 2 == 0);
    };
    for (int z = 0; z <= M && e == cudaSuccess; ++z) e = step(z < M ? z : -1, z - 1);
    return e;
}

cudaError_t fdfir_forward(int P2, const float2 *in, int64_t len, const FdfirTables &tw, float2 *A, float scale, cudaStream_t s)
{
    switch (P2) {
    case 2048: return fdfir_forward_l<2048>(in, len, tw, A, scale, s);
    case 4096: return fdfir_forward_l<4096>(in, len, tw, A, scale, s);
    case 8192: return fdfir_forward_l<8192>(in, len, tw, A, scale, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t fdfir_inverse(int P2, const float2 *X, const float2 *H, int M, float2 *B, const FdfirTables &tw, float *out,
                          int64_t n, cudaStream_t s)
{
    switch (P2) {
    case 2048: return fdfir_inverse_l<2048>(X, H, M, B, tw, out, n, s);
    case 4096: return fdfir_inverse_l<4096>(X, H, M, B, tw, out, n, s);
    case 8192: return fdfir_inverse_l<8192>(X, H, M, B, tw, out, n, s);
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
    float2 *d_B = nullptr;      // [2][P] row-pass outputs of the inverse, used in turn
    float2 *d_tw1 = nullptr;    // [P1] W_P1, FP32 from FP64
    float2 *d_tw2 = nullptr;    // W of the in-block row transform, then the factors of its last pass
    float2 *d_twr = nullptr;    // [P2] W_P2
    fdas::FdfirTables tables() const { return {d_tw1, d_tw2, d_twr}; }
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
    cudaFree(f->d_twr);
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
    const int PR = fdas::fd::row_points(f->P2);
    cudaError_t e;
    float2 *d_h = nullptr;
    const size_t h_bytes = sizeof(float2) * (size_t)M * K;
    int rc = FDAS_OK;
    if ((e = cudaMalloc(&f->d_H, sizeof(float2) * (size_t)M * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc spectra");
    else if ((e = cudaMalloc(&f->d_X, sizeof(float2) * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc input spectrum");
    else if ((e = cudaMalloc(&f->d_B, 2 * sizeof(float2) * P)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc scratch");
    else if ((e = cudaMalloc(&f->d_tw1, sizeof(float2) * fdas::fd::P1)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&f->d_tw2, sizeof(float2) * (PR + PR / 2))) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&f->d_twr, sizeof(float2) * f->P2)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&f->d_tw64, sizeof(double2) * f->P2)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc twiddles");
    else if ((e = cudaMalloc(&d_h, h_bytes)) != cudaSuccess) rc = fdfir_cuda(e, "cudaMalloc template staging");
    else if ((e = cudaMemcpy(d_h, templates, h_bytes, cudaMemcpyHostToDevice)) != cudaSuccess) rc = fdfir_cuda(e, "copy templates");
    else if ((e = fdas::launch_twiddles(fdas::fd::P1, f->d_tw64, f->d_tw1, nullptr)) != cudaSuccess) rc = fdfir_cuda(e, "twiddles");
    else if ((e = fdas::launch_twiddles(PR, f->d_tw64, f->d_tw2, nullptr)) != cudaSuccess) rc = fdfir_cuda(e, "twiddles");
    else if ((e = fdas::launch_twiddles(f->P2, f->d_tw64, f->d_twr, nullptr)) != cudaSuccess) rc = fdfir_cuda(e, "twiddles");
    if (rc == FDAS_OK) fdas::fdfir_factors<<<1, 256>>>(PR, f->d_tw2);
    for (int z = 0; rc == FDAS_OK && z < M; ++z) {
        e = fdas::fdfir_forward(f->P2, d_h + (size_t)z * K, K, f->tables(), f->d_H + (size_t)z * P, 1.0f / (float)P, nullptr);
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
    cudaError_t e = fdas::fdfir_forward(f->P2, static_cast<const float2 *>(in), n, f->tables(), f->d_X, 1.0f, s);
    if (e == cudaSuccess) e = fdas::fdfir_inverse(f->P2, f->d_X, f->d_H, f->M, f->d_B, f->tables(), out, n, s);
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
