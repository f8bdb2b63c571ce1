// Spin-summed one-particle density gamma_pq = <c| E_pq |c> (Eq. 7), the
// density the paper builds in an extra CI pass after the Davidson iterations
// (Section 4, Table 2 "1e/2e Density Matrices").
//
// gamma = gamma_alpha + gamma_beta.  A replacement a+_k a_l |J> = s |T> gives
//   alpha: s <C(T, :), C(J, :)>      (dot of two rows)
//   beta:  s <C(:, T), C(:, J)>      (dot of two columns)
// to gamma_kl, and T's entry back to J the same to gamma_lk.  The dots are FP64
// multiply-adds on a pipe that retires two per clock and SM, so each is computed
// once: a pair list per spin holds, string by string, the string with itself
// (its norm, which every E_kk of it shares) and its replacements to higher
// addresses, 25.5 entries per string at CAS(14,14) instead of 56.  Then
//  * alpha: a CTA per string J, a warp per pair;
//  * beta: eight pairs per thread, whose sums stay in registers while the rows of
//    a chunk of C pass through shared memory (two rows staged, the next one
//    arriving); one partial per pair and row chunk;
//  * one CTA per pair of orbitals sums its partials in a fixed order: the result
//    is bitwise reproducible.
// CAS(14,14), the whole blocking call: 3.5 ms with one dot per replacement (a
// thread's column dots gathered from global memory), 1.45 ms this way (6e8
// multiply-adds: 1.0 ms of the FP64 pipe).
#include <algorithm>
#include <cstdio>
#include <cstring>

#include "internal.cuh"

namespace fci {
namespace {

constexpr int kPairsPerThread = 8;
constexpr int kBetaThreads = 512;
constexpr int kPairsPerBlock = kPairsPerThread * kBetaThreads;
constexpr int kMinRows = 8;       // of a beta row chunk
constexpr int kListStrings = 512;

struct RdmSpin {
    int32_t *off = nullptr;
    uint32_t *ent = nullptr;
    double *part = nullptr;
    int64_t np = 0;
    int nr = 0;  // 0: the spin has no electrons
};

// The pair lists, a CTA per 512 strings: for string x first x itself (pair index
// kPairMask), then its replacements to higher addresses (packed entries), from
// off[x] on; off[ns] is the length.  Strings are in ascending order, so a+_k a_l goes
// to a higher address where k > l, and the entries of the strings before a CTA's own
// are counted from the bitmasks alone (one CTA per spin that carried the count along
// took 33 us for 1716 strings, 350 for 12870).
__global__ void __launch_bounds__(kListStrings) k_rdm_lists(SpinTables A, SpinTables B, int norb, RdmSpin a, RdmSpin b) {
    const SpinTables &S = blockIdx.y ? B : A;
    const RdmSpin &R = blockIdx.y ? b : a;
    const int64_t x0 = (int64_t)blockIdx.x * kListStrings, x = x0 + threadIdx.x;
    if (R.nr == 0 || x0 >= S.ns) return;
    const uint32_t all = (1u << norb) - 1u;
    auto count = [&](int64_t y) {
        const uint32_t occ = S.str[y], empty = all & ~occ;
        int n = 1;
        for (uint32_t m = occ; m; m &= m - 1u) n += __popc(empty & ~(m ^ (m - 1u)));
        return n;
    };
    int before = 0;
    for (int64_t y = threadIdx.x; y < x0; y += kListStrings) before += count(y);
    const int n = x < S.ns ? count(x) : 0;
    __shared__ int warp_sum[kListStrings / 32], warp_before[kListStrings / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    before = __reduce_add_sync(0xFFFFFFFFu, before);
    int v = n;  // inclusive sum over the warp
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) {
        warp_sum[warp] = v;
        warp_before[warp] = before;
    }
    __syncthreads();
    for (int w = 0; w < kListStrings / 32; ++w) v += warp_before[w] + (w < warp ? warp_sum[w] : 0);
    if (x >= S.ns) return;
    if (x == 0) R.off[0] = 0;
    R.off[x + 1] = v;
    uint32_t *out = R.ent + (v - n);
    *out++ = (uint32_t)x | (kPairMask << kPairShift);
    const int noff = S.nsingle - S.ne;
#pragma unroll 8
    for (int e = 0; e < noff; ++e) {
        const uint32_t t = S.tabo[(int64_t)e * S.ns + x];
        if ((int64_t)ent_target(t) > x) *out++ = t;
    }
}

// alpha partials: block J, a warp per pair (J, T): s <C(T, :), C(J, :)>
template <typename T>
__global__ void __launch_bounds__(256) k_rdm_alpha(const T *__restrict__ C, int64_t nsb, const int32_t *__restrict__ off,
                                                   const uint32_t *__restrict__ ent, double *__restrict__ part) {
    const int64_t j = blockIdx.x;
    const int lane = threadIdx.x & 31;
    const T *x = C + j * nsb;
    for (int i = off[j] + (threadIdx.x >> 5); i < off[j + 1]; i += 8) {
        const uint32_t e = ent[i];
        const T *y = C + (int64_t)ent_target(e) * nsb;
        double a0 = 0.0, a1 = 0.0;
        int64_t b = lane;
        for (; b + 96 < nsb; b += 128) {  // four loads of either row in flight
            const T x0 = x[b], x1 = x[b + 32], x2 = x[b + 64], x3 = x[b + 96];
            const T y0 = y[b], y1 = y[b + 32], y2 = y[b + 64], y3 = y[b + 96];
            a0 = fma((double)x0, (double)y0, a0);
            a1 = fma((double)x1, (double)y1, a1);
            a0 = fma((double)x2, (double)y2, a0);
            a1 = fma((double)x3, (double)y3, a1);
        }
        for (; b < nsb; b += 32) a0 = fma((double)x[b], (double)y[b], a0);
        a0 += a1;
        for (int o = 16; o > 0; o >>= 1) a0 += __shfl_down_sync(0xFFFFFFFFu, a0, o);
        if (lane == 0) part[i] = ent_negative(e) ? -a0 : a0;
    }
}

// beta partials: pairs blockIdx.x kPairsPerBlock .. (eight consecutive ones per
// thread) over the rows of chunk blockIdx.y; staged: rows pass through shared
// memory as doubles (two buffers of nsb), else the pairs are read from C itself.
template <typename T>
__global__ void __launch_bounds__(kBetaThreads) k_rdm_beta(const T *__restrict__ C, int64_t nsa, int64_t nsb,
                                                           const int32_t *__restrict__ off,
                                                           const uint32_t *__restrict__ ent, int64_t np, int64_t rows,
                                                           int staged, double *__restrict__ part) {
    extern __shared__ double sRow[];
    const int64_t i0 = (int64_t)blockIdx.x * kPairsPerBlock + (int64_t)threadIdx.x * kPairsPerThread;
    const int64_t r0 = blockIdx.y * rows, r1 = min(nsa, r0 + rows);
    int js[kPairsPerThread], ts[kPairsPerThread];
    double acc[kPairsPerThread];
    {   // strings of the pairs: the last x with off[x] <= i
        int64_t lo = 0, hi = nsb;
        const int64_t i = min(i0, np - 1);
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) / 2;
            if (off[mid] <= i)
                lo = mid;
            else
                hi = mid;
        }
#pragma unroll
        for (int u = 0; u < kPairsPerThread; ++u) {
            const int64_t at = min(i0 + u, np - 1);
            while (off[lo + 1] <= at) ++lo;
            js[u] = (int)lo;
            ts[u] = (int)ent_target(ent[at]);
            acc[u] = 0.0;
        }
    }
    if (staged) {
        // the next row is loaded into registers while the current one is used
        constexpr int kPre = 16;  // nsb <= kPre * kBetaThreads (host rule)
        T pre[kPre];
        auto load = [&](int64_t r) {
#pragma unroll
            for (int k = 0; k < kPre; ++k) {
                const int64_t b = threadIdx.x + k * kBetaThreads;
                if (b < nsb) pre[k] = C[r * nsb + b];
            }
        };
        load(r0);
        for (int64_t r = r0; r < r1; ++r) {
            double *row = sRow + ((r - r0) & 1) * nsb;
#pragma unroll
            for (int k = 0; k < kPre; ++k) {
                const int64_t b = threadIdx.x + k * kBetaThreads;
                if (b < nsb) row[b] = (double)pre[k];
            }
            if (r + 1 < r1) load(r + 1);
            __syncthreads();  // one barrier per row: the buffer used before is free by then
#pragma unroll
            for (int u = 0; u < kPairsPerThread; ++u) acc[u] = fma(row[js[u]], row[ts[u]], acc[u]);
        }
    } else {
        for (int64_t r = r0; r < r1; ++r)
#pragma unroll
            for (int u = 0; u < kPairsPerThread; ++u)
                acc[u] = fma((double)C[r * nsb + js[u]], (double)C[r * nsb + ts[u]], acc[u]);
    }
#pragma unroll
    for (int u = 0; u < kPairsPerThread; ++u)
        if (i0 + u < np) part[blockIdx.y * np + i0 + u] = ent_negative(ent[i0 + u]) ? -acc[u] : acc[u];
}

// part[i] = sum over the nr row chunks of part[r np + i], in order
__global__ void k_rdm_chunks(double *__restrict__ part, int64_t np, int nr) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    double v = 0.0;
#pragma unroll 4
    for (int r = 0; r < nr; ++r) v += part[r * np + i];
    part[i] = v;
}

// Sum of one spin's dots of orbital pair P = {k, l}: gamma_kl (the pairs hold one
// of gamma_kl, gamma_lk each)
__device__ double rdm_bin(const SpinTables &S, const int32_t *off, const uint32_t *ent, const double *part, int64_t np,
                          int P, int k, int l) {
    double acc = 0.0;
    if (k == l) {
        for (int64_t x = threadIdx.x; x < S.ns; x += blockDim.x)
            if (S.str[x] >> k & 1u) acc += part[off[x]];
    } else {
#pragma unroll 8
        for (int64_t i = threadIdx.x; i < np; i += blockDim.x)
            if ((int)ent_pair(ent[i]) == P) acc += part[i];
    }
    return acc;
}

__global__ void __launch_bounds__(1024) k_rdm_bins(SpinTables A, SpinTables B, RdmSpin a, RdmSpin b, int norb,
                                                  double *__restrict__ gamma) {
    const int P = blockIdx.x;
    int k = 0;
    while ((k + 1) * (k + 2) / 2 <= P) ++k;
    const int l = P - k * (k + 1) / 2;
    double acc = 0.0;
    if (a.nr) acc += rdm_bin(A, a.off, a.ent, a.part, a.np, P, k, l);
    if (b.nr) acc += rdm_bin(B, b.off, b.ent, b.part, b.np, P, k, l);
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 32; ++w) v += red[w];
        gamma[k * norb + l] = v;
        gamma[l * norb + k] = v;
    }
}

// Small spaces, one launch: a CTA per pair of orbitals {k, l} finds the strings'
// entries of that pair in the tables (to higher addresses, or E_kk), and its
// warps add their dots lane by lane; one reduction at the end.
constexpr int kScan = 4;  // table entries per thread in flight
template <typename T>
__global__ void __launch_bounds__(256) k_rdm_small(const T *__restrict__ C, SpinTables A, SpinTables B, int norb,
                                                   double *__restrict__ gamma) {
    const int P = blockIdx.x, lane = threadIdx.x & 31;
    int k = 0;
    while ((k + 1) * (k + 2) / 2 <= P) ++k;
    const int l = P - k * (k + 1) / 2;
    const int nsa = (int)A.ns, nsb = (int)B.ns;
    double acc = 0.0;
    for (int spin = 0; spin < 2; ++spin) {
        const SpinTables &S = spin ? B : A;
        const int ns = spin ? nsb : nsa, len = spin ? nsa : nsb;         // strings, length of a dot
        const int ld = spin ? 1 : nsb, step = spin ? nsb : 1;            // between strings, along a dot
        const int total = ns * S.nsingle;
        for (int t0 = threadIdx.x - lane; t0 < total; t0 += 256 * kScan) {
            uint32_t es[kScan];
#pragma unroll
            for (int u = 0; u < kScan; ++u) {
                const int t = t0 + u * 256 + lane;
                es[u] = t < total ? S.tab[t] : kPairMask << kPairShift;  // no pair has that index
            }
#pragma unroll
            for (int u = 0; u < kScan; ++u) {
                const uint32_t e = es[u];
                int x = 0;
                bool match = false;
                if ((int)ent_pair(e) == P) {
                    x = (t0 + u * 256 + lane) % ns;
                    match = k == l || (int)ent_target(e) > x;
                }
                for (uint32_t m = __ballot_sync(0xFFFFFFFFu, match); m; m &= m - 1u) {
                    const int from = __ffs(m) - 1;
                    const uint32_t ee = __shfl_sync(0xFFFFFFFFu, e, from);
                    const int xx = __shfl_sync(0xFFFFFFFFu, x, from);
                    const T *a = C + (size_t)xx * ld, *b = C + (size_t)ent_target(ee) * ld;
                    double d = 0.0;
                    for (int i = lane; i < len; i += 32) d = fma((double)a[(size_t)i * step], (double)b[(size_t)i * step], d);
                    acc += ent_negative(ee) ? -d : d;
                }
            }
        }
    }
    __shared__ double red[8];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
    if (lane == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[w];
        gamma[k * norb + l] = v;
        gamma[l * norb + k] = v;
    }
}

// Where the one launch is the faster way: few elements in the dots of a pair of orbitals
// (CAS(9; 5,4), 8800: 53 us against 72; (11; 3,3), 11000: 79 against 70; CAS(10,10), 32000:
// 143 against 74), some more where one spin has few strings, which leave the other kernels
// few CTAs ((11; 2,5), 10600; (18; 1,4), 12600).  With one alpha string the other kernels'
// only work is the beta spin's, whose columns lie together, and the search through the
// tables costs more from about 30000 entries on ((11; 11,5), 16000: 40 against 50; (12;
// 12,6), 39000: 72 against 60; (16; 16,8), 927000: 636 against 485).
bool one_launch(const fci_ctx *ctx) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const int64_t limit = std::min(A.ns, B.ns) < 64 ? 13000 : 10000;
    return ctx->ndet * (A.nsingle + B.nsingle) <= 2 * limit * ctx->npair && (A.ns > 1 || B.ns * B.nsingle <= 30000);
}

// Entries of a spin's pair list: a string each and half of the off-diagonal replacements.
int64_t pair_count(const SpinTables &S) { return S.ns + S.ns * (int64_t)(S.nsingle - S.ne) / 2; }

// Scratch, carved from one buffer of doubles: gamma, then per spin the offsets,
// the list and the partials (the beta spin's per row chunk).
struct RdmPlan {
    RdmSpin a, b;
    int64_t rows = 0;     // rows of C per beta chunk
    size_t doubles = 0;
    double *gamma = nullptr;
    int64_t ga = 0, gb = 0;  // places in the buffer

    RdmPlan(const fci_ctx *ctx, int max_chunks) {
        const SpinTables &A = ctx->A, &B = ctx->B;
        if (one_launch(ctx)) {  // gamma alone
            doubles = (size_t)ctx->norb * ctx->norb;
            return;
        }
        size_t at = (size_t)ctx->norb * ctx->norb;
        auto spin = [&](const SpinTables &S, RdmSpin &R, int nr, int64_t &where) {
            if (!S.nsingle) return;
            R.np = pair_count(S);
            R.nr = nr;
            where = (int64_t)at;
            at += (size_t)((S.ns + 2) / 2 + (R.np + 1) / 2 + R.np * nr);
        };
        spin(A, a, 1, ga);
        // enough row chunks to give every SM two blocks, at least kMinRows rows each
        int chunks = 1;
        if (B.nsingle) {
            const int64_t blocks = (pair_count(B) + kPairsPerBlock - 1) / kPairsPerBlock;
            chunks = (int)std::min<int64_t>(std::max<int64_t>(1, 304 / blocks), std::max<int64_t>(1, A.ns / kMinRows));
            chunks = std::min(chunks, max_chunks);
            rows = (A.ns + chunks - 1) / chunks;
            chunks = (int)((A.ns + rows - 1) / rows);
        }
        spin(B, b, chunks, gb);
        doubles = at;
    }
    void place(const fci_ctx *ctx, double *base) {
        gamma = base;
        auto spin = [&](const SpinTables &S, RdmSpin &R, int64_t where) {
            if (!R.nr) return;
            R.off = reinterpret_cast<int32_t *>(base + where);
            R.ent = reinterpret_cast<uint32_t *>(base + where + (S.ns + 2) / 2);
            R.part = base + where + (S.ns + 2) / 2 + (R.np + 1) / 2;
        };
        spin(ctx->A, a, ga);
        spin(ctx->B, b, gb);
    }
};

// The kernels of one density, into P.gamma (device), on stream s.
template <typename T>
int launch_rdm1(fci_ctx *ctx, const T *C, const RdmPlan &P, cudaStream_t s) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    if (one_launch(ctx)) {
        k_rdm_small<T><<<ctx->npair, 256, 0, s>>>(C, A, B, ctx->norb, P.gamma);
        FCI_CUDA(cudaGetLastError());
        return FCI_OK;
    }
    RdmSpin a = P.a, b = P.b;
    const bool shared = a.nr && b.nr && A.tabo == B.tabo;  // one string space: one list
    if (shared) {
        b.off = a.off;
        b.ent = a.ent;
    }
    if (a.nr || b.nr) {
        k_rdm_lists<<<dim3(ceil_div(std::max(A.ns, B.ns), kListStrings), shared ? 1 : 2), kListStrings, 0, s>>>(
            A, B, ctx->norb, a, b);
        FCI_CUDA(cudaGetLastError());
    }
    if (a.nr) {
        k_rdm_alpha<T><<<(unsigned)A.ns, 256, 0, s>>>(C, B.ns, a.off, a.ent, a.part);
        FCI_CUDA(cudaGetLastError());
    }
    if (b.nr) {
        // staged while two rows fit in 96 KB (two CTAs per SM) and in the registers of the prefetch
        const size_t smem = 2 * sizeof(double) * (size_t)B.ns;
        const int staged = smem <= 96 * 1024;
        if (staged && smem > 48 * 1024) FCI_CUDA(opt_in_max_smem((const void *)k_rdm_beta<T>, ctx->device));
        k_rdm_beta<T><<<dim3(ceil_div(b.np, kPairsPerBlock), (unsigned)b.nr), kBetaThreads, staged ? smem : 0, s>>>(
            C, A.ns, B.ns, b.off, b.ent, b.np, P.rows, staged, b.part);
        if (b.nr > 1) k_rdm_chunks<<<ceil_div(b.np, 256), 256, 0, s>>>(b.part, b.np, b.nr);
        FCI_CUDA(cudaGetLastError());
    }
    k_rdm_bins<<<ctx->npair, 1024, 0, s>>>(A, B, a, b, ctx->norb, P.gamma);
    FCI_CUDA(cudaGetLastError());
    return FCI_OK;
}

template <typename T>
int rdm_impl(fci_ctx *ctx, const T *C, double *gamma_host) {
    RdmPlan P(ctx, 1 << 20);
    DensityScratch mem(ctx);
    int rc = mem.take(sizeof(double) * P.doubles);
    if (rc == FCI_ERR_OOM && P.b.nr > 1) {  // one row chunk needs a partial per pair only
        P = RdmPlan(ctx, 1);
        rc = mem.take(sizeof(double) * P.doubles);
    }
    if (rc) return rc;
    P.place(ctx, reinterpret_cast<double *>(mem.dev));
    const size_t bytes = sizeof(double) * ctx->norb * ctx->norb;
    if (mem.host) P.gamma = mem.host;  // the last kernel writes the density into pinned host memory
    cudaStream_t s = ctx->stream;
    rc = launch_rdm1<T>(ctx, C, P, s);
    cudaError_t e = cudaSuccess;
    if (rc == FCI_OK && !mem.host) e = cudaMemcpyAsync(gamma_host, P.gamma, bytes, cudaMemcpyDeviceToHost, s);
    const cudaError_t done = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = done;
    if (rc == FCI_OK && e != cudaSuccess) rc = cuda_fail(e, "rdm1");
    if (rc == FCI_OK && mem.host) memcpy(gamma_host, mem.host, bytes);
    return rc;
}

}  // namespace

int run_rdm1(fci_ctx *ctx, const void *c, int dtype, double *gamma) {
    if (dtype == FCI_F64) return rdm_impl<double>(ctx, (const double *)c, gamma);
    return rdm_impl<float>(ctx, (const float *)c, gamma);
}

}  // namespace fci

// ---------------------------------------------------------------------------
// fci_rdm1_noalloc: the same density as fci_rdm1, with its scratch in a
// file-scope device array instead of per-call cudaMalloc/cudaFree.
//
// The array below is a host-side stand-in in host code: its device address
// is looked up with cudaGetSymbolAddress once per device (with that device
// current) and cached; kernels receive that address.  Every call shares the
// one array, so calls whose GPU work overlaps race on it.
// ---------------------------------------------------------------------------
#include <mutex>

static __device__ __align__(256) double g_rdm1_scratch[FCI_RDM1_NOALLOC_MAX_DOUBLES];

namespace fci {
namespace {
std::mutex g_scratch_mu;
constexpr int kMaxDevices = 64;
double *g_scratch_addr[kMaxDevices] = {};

// Device address of g_rdm1_scratch on the current device `dev`.
int scratch_address(int dev, double **out) {
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (dev < 0 || dev >= kMaxDevices) return fail(FCI_ERR_ARG, "device ordinal out of range for the scratch cache");
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_rdm1_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(rdm1 scratch)");
        g_scratch_addr[dev] = (double *)p;
    }
    *out = g_scratch_addr[dev];
    return FCI_OK;
}

template <typename T>
int rdm_noalloc_impl(fci_ctx *ctx, const T *C, double *gamma_host, cudaStream_t s) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const int n = ctx->norb;
    const size_t na = (size_t)A.ns * A.nsingle, nb = (size_t)B.ns * B.nsingle, ng = (size_t)n * n;
    if (na + nb + ng > (size_t)FCI_RDM1_NOALLOC_MAX_DOUBLES) {
        char buf[200];
        snprintf(buf, sizeof(buf),
                 "fci_rdm1_noalloc needs %zu scratch doubles, above its fixed limit of %d "
                 "(FCI_RDM1_NOALLOC_MAX_DOUBLES); use fci_rdm1",
                 na + nb + ng, FCI_RDM1_NOALLOC_MAX_DOUBLES);
        return fail(FCI_ERR_ARG, buf);
    }
    // fewer row chunks where the array does not hold them all (one chunk needs at most 0.83 (na +
    // nb) doubles and a few per string)
    RdmPlan P(ctx, 1 << 20);
    if (P.doubles > (size_t)FCI_RDM1_NOALLOC_MAX_DOUBLES) {
        const size_t over = P.doubles - (size_t)FCI_RDM1_NOALLOC_MAX_DOUBLES;
        const int64_t drop = (int64_t)((over + P.b.np - 1) / P.b.np);
        P = RdmPlan(ctx, (int)std::max<int64_t>(1, P.b.nr - drop));
    }
    if (P.doubles > (size_t)FCI_RDM1_NOALLOC_MAX_DOUBLES)
        return fail(FCI_ERR_ARG, "fci_rdm1_noalloc: the space exceeds its fixed scratch; use fci_rdm1");
    double *base = nullptr;
    if (int rc = scratch_address(ctx->device, &base)) return rc;
    P.place(ctx, base);
    if (int rc = launch_rdm1<T>(ctx, C, P, s)) return rc;
    FCI_CUDA(cudaMemcpyAsync(gamma_host, P.gamma, sizeof(double) * ng, cudaMemcpyDeviceToHost, s));
    FCI_CUDA(cudaStreamSynchronize(s));
    return FCI_OK;
}
}  // namespace
}  // namespace fci

extern "C" int fci_rdm1_noalloc(fci_ctx *ctx, const void *c, int dtype, double *gamma, void *stream) {
    using namespace fci;
    if (!ctx || !c || !gamma) return fail(FCI_ERR_ARG, "NULL argument");
    if (dtype != FCI_F64 && dtype != FCI_F32) return fail(FCI_ERR_ARG, "dtype must be FCI_F64 or FCI_F32");
    // the caller's current device is restored on every return path
    int prev = -1;
    FCI_CUDA(cudaGetDevice(&prev));
    FCI_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    const int rc = dtype == FCI_F64 ? rdm_noalloc_impl<double>(ctx, (const double *)c, gamma, s)
                                    : rdm_noalloc_impl<float>(ctx, (const float *)c, gamma, s);
    const cudaError_t e = cudaSetDevice(prev);
    if (rc == FCI_OK && e != cudaSuccess) return cuda_fail(e, "cudaSetDevice (restoring the caller's device)");
    return rc;
}
