// sigma = H c of small spaces in one kernel (all three terms of Eq. 8, string
// driven, plain FP64 or FP32 multiply-adds).
//
// Below about 1e7 multiply-adds (FP64; CAS(9; 5,4) has 1.06e7) the arithmetic is
// a few microseconds, and the tensor-core pipeline of larger spaces - operand
// planes of C, one product per term, their launches and pipeline fills - is all
// latency (FP64 CAS(6,6) 62 us, here 8.6; CAS(8,8) 74, here 16; FP32 CAS(9; 5,4)
// 44, here 18.5; FP64 errors 3e-16 instead of 1e-13 to 1e-12).  Here a CTA owns one alpha row, or a share of its beta
// strings: it stages the rows C(J_a, :) of the row's off-diagonal alpha
// replacements and C(I_a, :) itself (a = last, standing for all E_kk, with their
// summed integral row), transposed so that the replacements of one beta string
// are contiguous, and the signed integral rows s_a (p_a | q) likewise.  Then
//   sigma_3(I_a, I_b) = sum over b of s_b sum over a of W[p_b][a] R[J_b][a]
// is a short dot product per beta replacement; sigma_1 gathers from the staged
// row itself, sigma_2 reads C along rows.  The replacements and matrix elements
// of one determinant are dealt to several threads, whose sums are added in a
// fixed order (bit-reproducible).  FP32 adds the dot products into a
// double-float sum, which keeps the rounding of a determinant's few hundred
// terms below that of one FP32 sum.
#include <algorithm>

#include "internal.cuh"

namespace fci {
namespace sml {

constexpr int kThreads = 256;

template <typename T>
struct Vec;
template <>
struct Vec<float> {
    typedef float4 type;
    static constexpr int n = 4;
};
template <>
struct Vec<double> {
    typedef double2 type;
    static constexpr int n = 2;
};

// staged replacements per row (one more than the off-diagonal ones), padded to an
// odd number of 16-byte words: the records of different strings then start in
// different banks
template <typename T>
__host__ __device__ inline int row_len(int noff) {
    constexpr int n = Vec<T>::n;
    const int words = (noff + 1 + n - 1) / n;
    return (words | 1) * n;
}

__device__ __forceinline__ float dot(float4 x, float4 y, float4 &acc) {
    acc.x = fmaf(x.x, y.x, acc.x);
    acc.y = fmaf(x.y, y.y, acc.y);
    acc.z = fmaf(x.z, y.z, acc.z);
    acc.w = fmaf(x.w, y.w, acc.w);
    return 0.f;
}
__device__ __forceinline__ float total(float4 a) { return (a.x + a.y) + (a.z + a.w); }
__device__ __forceinline__ double dot(double2 x, double2 y, double2 &acc) {
    acc.x = fma(x.x, y.x, acc.x);
    acc.y = fma(x.y, y.y, acc.y);
    return 0.0;
}
__device__ __forceinline__ double total(double2 a) { return a.x + a.y; }

// Running sum: FP64 as it is, FP32 as a double-float pair (TwoSum).
template <typename T>
struct Sum;
template <>
struct Sum<double> {
    double v = 0.0;
    __device__ void add(double x) { v += x; }
    __device__ void fma_(double a, double b) { v = fma(a, b, v); }
    __device__ double get() const { return v; }
};
template <>
struct Sum<float> {
    float h = 0.f, l = 0.f;
    __device__ void add(float x) {
        const float t = h + x, b = t - h;
        l += (h - (t - b)) + (x - b);
        h = t;
    }
    __device__ void fma_(float a, float b) {
        const float p = a * b;
        l += fmaf(a, b, -p);
        add(p);
    }
    __device__ float get() const { return h + l; }
};

template <typename T>
__global__ void __launch_bounds__(kThreads) k_sigma_small(const T *__restrict__ C, T *__restrict__ sig, SpinTables A,
                                                          SpinTables B, const T *__restrict__ W,
                                                          const T *__restrict__ ga, const T *__restrict__ gb, int npair,
                                                          int len, const int *__restrict__ active) {
    if (active != nullptr && *active == 0) return;  // gated launch (batched engine)
    typedef typename Vec<T>::type V;
    constexpr int VN = Vec<T>::n;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nsa = (int)A.ns, nsb = (int)B.ns, row = blockIdx.x, tid = threadIdx.x;
    const int noff = A.nsingle - A.ne, na = row_len<T>(noff);
    T *sR = reinterpret_cast<T *>(smem_raw);  // [nsb][na]
    T *sW = sR + (size_t)nsb * na;            // [npair][na]
    T *sRed = sW + (size_t)npair * na;        // [kThreads]
    // staged rows and signed integral rows (padding: zeros)
    for (int t = tid; t < na * nsb; t += kThreads) {
        const int a = t / nsb, j = t - a * nsb;
        T v = T(0);
        if (a <= noff) v = C[(size_t)(a < noff ? (int)ent_target(A.tabo[(size_t)a * nsa + row]) : row) * nsb + j];
        sR[j * na + a] = v;
    }
    const uint32_t occ = A.str[row];
    for (int t = tid; t < na * npair; t += kThreads) {
        const int a = t / npair, q = t - a * npair;
        T w = T(0);
        if (a < noff) {
            const uint32_t e = A.tabo[(size_t)a * nsa + row];
            w = W[(size_t)ent_pair(e) * npair + q];
            if (ent_negative(e)) w = -w;
        } else if (a == noff) {
            for (uint32_t m = occ; m; m &= m - 1u) {
                const int k = __ffs(m) - 1;
                w += W[(size_t)(k * (k + 1) / 2 + k) * npair + q];
            }
        }
        sW[q * na + a] = w;
    }
    __syncthreads();
    // determinants c0 .. c1 of the row; `parts` threads share one determinant
    const int c0 = blockIdx.y * len, c1 = min(nsb, c0 + len), cnt = c1 - c0;
    const int parts = cnt >= kThreads ? 1 : kThreads / cnt;
    for (int base = 0; base < cnt; base += kThreads) {  // one round unless cnt > kThreads
        const int width = min(cnt - base, kThreads);
        const int p = tid / width, i = base + tid - p * width, ib = c0 + i;
        const bool on = p < parts;
        if (on) {
            Sum<T> s;
#pragma unroll 2
            for (int b = p; b < B.nsingle; b += parts) {
                const uint32_t e = B.tab[(size_t)b * nsb + ib];
                const V *w = reinterpret_cast<const V *>(sW + (size_t)ent_pair(e) * na);
                const V *r = reinterpret_cast<const V *>(sR + (size_t)ent_target(e) * na);
                V acc{};
                for (int k = 0; k < na / VN; ++k) dot(w[k], r[k], acc);
                const T d = total(acc);
                s.add(ent_negative(e) ? -d : d);
            }
#pragma unroll 4
            for (int e = p; e < B.nsame; e += parts)
                s.fma_(gb[(size_t)e * nsb + ib], sR[(size_t)B.gcol[(size_t)e * nsb + ib] * na + noff]);
#pragma unroll 4
            for (int e = p; e < A.nsame; e += parts)
                s.fma_(ga[(size_t)e * nsa + row], C[(size_t)A.gcol[(size_t)e * nsa + row] * nsb + ib]);
            sRed[tid] = s.get();
        }
        __syncthreads();
        if (on && p == 0) {
            // as above: up to 256 parts, one of which holds the diagonal (a plain FP32 sum of
            // them left 4e-7 of the result at CAS(12; 6,12), this one 7e-8)
            Sum<T> v;
            for (int k = 0; k < parts; ++k) v.add(sRed[tid + k * width]);
            sig[(size_t)row * nsb + ib] = v.get();
        }
        __syncthreads();
    }
}

template <typename T>
static size_t smem_bytes(const fci_ctx *ctx) {
    const int na = row_len<T>(ctx->A.nsingle - ctx->A.ne);
    return sizeof(T) * ((size_t)(ctx->B.ns + ctx->npair) * na + kThreads);
}

template <typename T>
static double macs(const fci_ctx *ctx) {  // multiply-adds of the call
    const SpinTables &A = ctx->A, &B = ctx->B;
    return (double)ctx->ndet * ((double)row_len<T>(A.nsingle - A.ne) * B.nsingle + A.nsame + B.nsame);
}

}  // namespace sml

// FP64 up to kSmall64 multiply-adds (CAS(9; 5,4), 1.1e7: 37 us against 81 us with
// the sliced products; CAS(10; 5,3), 2.4e7: 89 with them).  FP32 up to kSmall32 for
// unequal spins (CAS(10; 5,4): 51 us against 68 with the dense products; CAS(11;
// 6,5), 3.5e8: 270 against 115) and kSmall32Same for one string space, whose same-spin
// terms the fused table walk of sigma.cu takes next (15876 determinants of CAS(9; 4,4):
// 19 us against 28; CAS(11; 3,3), 2e7: 44 both; CAS(10; 4,4), 4e7: 50 against 44).
// Both spins with replacements (the single-spin terms alone stay with the staged
// kernels), default kernel choices.
constexpr double kSmall64 = 1.5e7, kSmall32 = 8e7, kSmall32Same = 2.5e7;

bool sigma_small_ok(const fci_ctx *ctx, int dtype) {
    const fci_options &o = ctx->opt;
    if (ctx->A.nsingle == 0 || ctx->B.nsingle == 0) return false;
    if (dtype == FCI_F64)
        return o.f64_kernels == FCI_F64_AUTO && o.f64_same_spin == FCI_SS_AUTO && sml::macs<double>(ctx) <= kSmall64 &&
               sml::smem_bytes<double>(ctx) <= 100 * 1024;
    return o.same_spin_tc == 0 && o.f32_row_global == 0 &&
           sml::macs<float>(ctx) <= (ctx->A.ne == ctx->B.ne ? kSmall32Same : kSmall32) &&
           sml::smem_bytes<float>(ctx) <= 100 * 1024;
}

int prepare_sigma_small(const fci_ctx *ctx) {
    FCI_CUDA(opt_in_max_smem((const void *)sml::k_sigma_small<double>, ctx->device));
    FCI_CUDA(opt_in_max_smem((const void *)sml::k_sigma_small<float>, ctx->device));
    return FCI_OK;
}

template <typename T>
static int launch_small(fci_ctx *ctx, const T *C, T *sig, cudaStream_t s, const int *active) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const T *W, *ga, *gb;
    if constexpr (sizeof(T) == 8) {
        W = ctx->W;
        ga = A.gval;
        gb = B.gval;
    } else {
        W = ctx->Wf;
        ga = A.gvalf;
        gb = B.gvalf;
    }
    // shares of a row: about two CTAs per SM, at least 32 determinants each
    const int nsa = (int)A.ns, nsb = (int)B.ns;
    const int shares = std::max(1, std::min((nsb + 31) / 32, 304 / nsa));
    const int len = (nsb + shares - 1) / shares;
    sml::k_sigma_small<T><<<dim3((unsigned)nsa, (unsigned)((nsb + len - 1) / len)), sml::kThreads, sml::smem_bytes<T>(ctx), s>>>(
        C, sig, A, B, W, ga, gb, ctx->npair, len, active);
    FCI_CUDA(cudaGetLastError());
    return FCI_OK;
}

int launch_sigma_small(fci_ctx *ctx, const void *C, void *sig, int dtype, cudaStream_t s, const int *active) {
    if (dtype == FCI_F64) return launch_small<double>(ctx, (const double *)C, (double *)sig, s, active);
    return launch_small<float>(ctx, (const float *)C, (float *)sig, s, active);
}

}  // namespace fci
