// Device code shared by the single-instance and the batched Davidson drivers:
// cross-lane sums of several FP64 accumulators, and the eigensolver of the
// projected matrix.
//
// Both are written around GB300's FP64 rate: an SM retires about two FP64
// operations per clock, so one FP64 instruction of a warp holds its scheduler
// for 64 cycles, whether it is part of a product or of a reduction.
#pragma once
#include <stdint.h>

namespace fci {
namespace sd {

// Sums over the warp of the eight acc[j], in 9 additions per lane instead of
// the 40 of eight separate shuffle trees: at every halving a lane gives away
// half of the accumulators it still holds.  Lane l returns the sum of
// acc[j(l)], j(l) = 4 (l >> 4 & 1) + 2 (l >> 3 & 1) + (l >> 2 & 1).
__device__ __forceinline__ int reduce8_index(int lane) { return (lane >> 4 & 1) * 4 + (lane >> 3 & 1) * 2 + (lane >> 2 & 1); }
__device__ __forceinline__ double warp_reduce8(const double (&acc)[8], int lane) {
    double a[4], b[2], v;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const bool up = lane & 16;
        const double got = __shfl_xor_sync(0xFFFFFFFFu, up ? acc[j] : acc[j + 4], 16);
        a[j] = (up ? acc[j + 4] : acc[j]) + got;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const bool up = lane & 8;
        const double got = __shfl_xor_sync(0xFFFFFFFFu, up ? a[j] : a[j + 2], 8);
        b[j] = (up ? a[j + 2] : a[j]) + got;
    }
    {
        const bool up = lane & 4;
        const double got = __shfl_xor_sync(0xFFFFFFFFu, up ? b[0] : b[1], 4);
        v = (up ? b[1] : b[0]) + got;
    }
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
    return v;
}

// Sum of v over a block of 256 threads (fixed order), valid in thread 0; red: 8 doubles of shared memory.
__device__ __forceinline__ double block_sum256(double v, double *red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < 8; ++w) t += red[w];
    return t;
}

// Whether this block is the last of `total` to get here (all threads get the
// answer); what the others wrote before is then visible.  The counter is left
// at zero for the next launch.
__device__ __forceinline__ bool last_block(int *counter, int total) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(counter, 1) == total - 1;
        if (s_last) *counter = 0;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

constexpr int kEigMax = 32;

// Eigenvalues (ascending, stable) and eigenvectors (columns of V[m][m]) of the
// symmetric part of the m x m matrix A (row-major, leading dimension lda), by
// one block of 256 threads.
//
// Parallel cyclic Jacobi (textbook; round-robin pairs: each step rotates m / 2
// disjoint pairs) in two stages, because FP64 rotations are what it costs (270
// to 300 us at m = 24 with every sweep in FP64, 130 to 215 us this way):
//  1. in FP32 until the off-diagonal elements are at FP32 rounding;
//  2. its vectors are made orthogonal in FP64 (two Newton-Schulz steps, V <- V
//     (3/2 - V^T V / 2): an orthogonality error e becomes 3/8 e^2), A is transformed with
//     them in FP64, and FP64 sweeps finish on the nearly diagonal matrix until a
//     sweep rotates nothing (|a_pq| <= 2^-46 max(|a_pp|, |a_qq|) is skipped).
// A rotation's tangent is formed in FP32 (an inexact angle leaves 1e-7 of the
// element for the next sweep).  Where the matrix may be out of FP32's range (RESCALE,
// told by the integrals, fci_ctx::eig_rescale) one whose largest element is not between 2^-40
// and 2^100 is scaled by a power of two and its eigenvalues scaled back; elements below
// 2^-100 are not rotated.  (With the look at the elements in every launch the kernel took
// 2 us more of 103.)  The rotation's cosine is 1 / sqrt(1 + t^2) to FP64 rounding by
// one third-order correction of the FP32 reciprocal root, so that every rotation is
// orthogonal to FP64 rounding.  A non-finite matrix ends both stages at once and comes
// back as non-finite eigenvalues.
struct EigShared {
    double a[kEigMax][kEigMax + 1], v[kEigMax][kEigMax + 1], t[kEigMax][kEigMax + 1];
    float af[kEigMax][kEigMax + 1], vf[kEigMax][kEigMax + 1];
    double c[kEigMax / 2], s[kEigMax / 2];
    float cf[kEigMax / 2], sf[kEigMax / 2];
    int order[kEigMax];
    int rotated;
};

// The pair at position k of step `step` (round robin over n players, 0 fixed; p < q).
__device__ __forceinline__ void rr_pair(int k, int step, int n, int &p, int &q) {
    auto player = [&](int at) {
        int x = at - 1 - step;  // > -n: one wrap
        if (x < 0) x += n - 1;
        return at == 0 ? 0 : 1 + x;
    };
    const int x = player(k), y = player(n - 1 - k);
    p = min(x, y);
    q = max(x, y);
}

// Sweeps of rotations on a (m x m, symmetric) with the vectors in v; c and s:
// the rotations of a step.  Blocks of 256 threads.
template <typename T>
__device__ __forceinline__ void jacobi_sweeps(T (*a)[kEigMax + 1], T (*v)[kEigMax + 1], T *cs, T *sn, int m, int *rotated,
                                              int max_sweeps) {
    const int tid = threadIdx.x;
    const int me = m + (m & 1), half = me / 2;  // index m is a dummy when m is odd
    // this thread's 2 x 2 block (pairs k1 <= k2): the tid-th of the half (half + 1) / 2
    int k1 = 0, k2 = tid;
    while (k1 < half && k2 >= half) {
        ++k1;
        k2 += k1 - half;
    }
    const bool block = k1 < half;
    // eigenvector rows: threads from the last down, so that they are not the
    // block threads where there are enough
    const int vt = 255 - tid, r = vt & 31;
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        if (tid == 0) *rotated = 0;
        __syncthreads();
        for (int step = 0; step < me - 1; ++step) {
            if (tid < half) {
                int p, q;
                rr_pair(tid, step, me, p, q);
                T c = T(1), s = T(0);
                if (q < m) {
                    const T apq = a[p][q], app = a[p][p], aqq = a[q][q];
                    bool rot;
                    if constexpr (sizeof(T) == 8) {  // |a_pq| > 2^-46 max(|a_pp|, |a_qq|), on the exponents
                        const int h = __double2hiint(apq) & 0x7FFFFFFF;
                        const int g = max(__double2hiint(app) & 0x7FFFFFFF, __double2hiint(aqq) & 0x7FFFFFFF);
                        rot = h > g - (46 << 20) && h < 0x7FF00000 && h >= 923 << 20;
                    } else {
                        rot = fabsf(apq) > fmaf(2e-7f, fmaxf(fabsf(app), fabsf(aqq)), 0x1p-100f);
                    }
                    if (rot) {
                        const float th = __fdividef((float)(aqq - app), 2.0f * (float)apq);
                        const float tf = copysignf(1.0f, th) * __fdividef(1.0f, fabsf(th) + sqrtf(fmaf(th, th, 1.0f)));
                        const float yf = rsqrtf(fmaf(tf, tf, 1.0f));
                        if constexpr (sizeof(T) == 8) {
                            const double td = tf, y = yf;
                            const double e = fma(-fma(td, td, 1.0), y * y, 1.0);  // 1 - x y^2, about 2^-22
                            c = fma(y, e * fma(e, 0.375, 0.5), y);
                            s = td * c;
                        } else {
                            c = yf;
                            s = tf * yf;
                        }
                        if (tf != 0.0f) *rotated = 1;
                    }
                }
                cs[tid] = c;
                sn[tid] = s;
            }
            __syncthreads();
            // a <- J^T a J by 2 x 2 blocks, v <- v J
            if (block) {
                const T s1 = sn[k1], s2 = sn[k2];
                if (s1 != T(0) || s2 != T(0)) {
                    const T c1 = cs[k1], c2 = cs[k2];
                    int p1, q1, p2, q2;
                    rr_pair(k1, step, me, p1, q1);
                    rr_pair(k2, step, me, p2, q2);
                    const T x = a[p1][p2], y = a[p1][q2], z = a[q1][p2], w = a[q1][q2];  // row and column m: zeros
                    const T xc = c2 * x - s2 * y, yc = s2 * x + c2 * y, zc = c2 * z - s2 * w, wc = s2 * z + c2 * w;
                    const T xn = c1 * xc - s1 * zc, yn = c1 * yc - s1 * wc, zn = s1 * xc + c1 * zc, wn = s1 * yc + c1 * wc;
                    a[p1][p2] = a[p2][p1] = xn;
                    a[p1][q2] = a[q2][p1] = yn;
                    a[q1][p2] = a[p2][q1] = zn;
                    a[q1][q2] = a[q2][q1] = wn;
                }
            }
            if (r < m)
                for (int k = vt >> 5; k < half; k += 8) {
                    const T s = sn[k];
                    if (s == T(0)) continue;
                    const T c = cs[k];
                    int p, q;
                    rr_pair(k, step, me, p, q);
                    const T vp = v[r][p], vq = v[r][q];
                    v[r][p] = c * vp - s * vq;
                    v[r][q] = s * vp + c * vq;
                }
            __syncthreads();
        }
        if (!*rotated) break;
        __syncthreads();
    }
}

// S.t and S.af scaled to a largest element in [1, 2) where it is not between 2^-40 and
// 2^100 (above the batch's padding of 1e30); the factor back.  Zero and non-finite matrices
// stay as they are.
__device__ __forceinline__ double eig_rescale(int m, EigShared &S) {
    int ex = 0;
    for (int t = threadIdx.x; t < m * m; t += blockDim.x) ex = max(ex, (__double2hiint(S.t[t / m][t % m]) >> 20) & 0x7FF);
    if (threadIdx.x == 0) S.rotated = 0;
    __syncthreads();
    atomicMax(&S.rotated, ex);
    __syncthreads();
    ex = S.rotated;
    double back = 1.0;
    if (ex > 0 && ex < 0x7FF && (ex < 983 || ex > 1123)) {
        const int e = max(2046 - ex, 1);
        const double f = __hiloint2double(e << 20, 0);
        back = __hiloint2double((2046 - e) << 20, 0);
        for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
            S.t[t / m][t % m] *= f;
            S.af[t / m][t % m] = (float)S.t[t / m][t % m];
        }
    }
    __syncthreads();
    return back;
}

template <bool RESCALE>
__device__ __forceinline__ void eig_symmetric(const double *A, int lda, int m, double *w, double *V, EigShared &S) {
    const int tid = threadIdx.x;
    for (int t = tid; t < kEigMax * (kEigMax + 1); t += 256) {
        (&S.af[0][0])[t] = 0.0f;
        (&S.a[0][0])[t] = 0.0;
    }
    __syncthreads();
    for (int t = tid; t < m * m; t += blockDim.x) {
        const int i = t / m, j = t % m;
        const double x = 0.5 * (A[i * lda + j] + A[j * lda + i]);
        S.t[i][j] = x;
        S.af[i][j] = (float)x;
        S.vf[i][j] = i == j ? 1.0f : 0.0f;
    }
    __syncthreads();
    double back = 1.0;
    if constexpr (RESCALE) back = eig_rescale(m, S);
    jacobi_sweeps<float>(S.af, S.vf, S.cf, S.sf, m, &S.rotated, 12);
    __syncthreads();
    for (int t = tid; t < m * m; t += blockDim.x) S.v[t / m][t % m] = (double)S.vf[t / m][t % m];
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
        for (int t = tid; t < m * m; t += blockDim.x) {  // a = 3/2 - V^T V / 2
            const int i = t / m, j = t % m;
            if (i > j) continue;
            double x = 0.0;
            for (int k = 0; k < m; ++k) x = fma(S.v[k][i], S.v[k][j], x);
            S.a[i][j] = S.a[j][i] = (i == j ? 1.5 : 0.0) - 0.5 * x;
        }
        __syncthreads();
        double y[4];
        int n = 0;
        for (int t = tid; t < m * m; t += blockDim.x, ++n) {
            const int i = t / m, j = t % m;
            double x = 0.0;
            for (int k = 0; k < m; ++k) x = fma(S.v[i][k], S.a[k][j], x);
            y[n & 3] = x;
        }
        __syncthreads();
        n = 0;
        for (int t = tid; t < m * m; t += blockDim.x, ++n) S.v[t / m][t % m] = y[n & 3];
        __syncthreads();
    }
    {  // a = V^T A V
        double y[4];
        int n = 0;
        for (int t = tid; t < m * m; t += blockDim.x, ++n) {
            const int i = t / m, j = t % m;
            double x = 0.0;
            for (int k = 0; k < m; ++k) x = fma(S.t[i][k], S.v[k][j], x);
            y[n & 3] = x;
        }
        __syncthreads();
        n = 0;
        for (int t = tid; t < m * m; t += blockDim.x, ++n) S.t[t / m][t % m] = y[n & 3];
        __syncthreads();
        for (int t = tid; t < m * m; t += blockDim.x) {
            const int i = t / m, j = t % m;
            if (i > j) continue;
            double x = 0.0;
            for (int k = 0; k < m; ++k) x = fma(S.v[k][i], S.t[k][j], x);
            S.a[i][j] = S.a[j][i] = x;
        }
        __syncthreads();
    }
    jacobi_sweeps<double>(S.a, S.v, S.c, S.s, m, &S.rotated, 60);
    __syncthreads();
    if (tid == 0) {
        for (int i = 0; i < m; ++i) S.order[i] = i;
        for (int i = 1; i < m; ++i) {  // insertion sort, stable
            const int o = S.order[i];
            int j = i - 1;
            while (j >= 0 && S.a[S.order[j]][S.order[j]] > S.a[o][o]) {
                S.order[j + 1] = S.order[j];
                --j;
            }
            S.order[j + 1] = o;
        }
    }
    __syncthreads();
    for (int t = tid; t < m; t += blockDim.x) w[t] = RESCALE ? S.a[S.order[t]][S.order[t]] * back : S.a[S.order[t]][S.order[t]];
    for (int t = tid; t < m * m; t += blockDim.x) V[t] = S.v[t / m][S.order[t % m]];
}

}  // namespace sd
}  // namespace fci
