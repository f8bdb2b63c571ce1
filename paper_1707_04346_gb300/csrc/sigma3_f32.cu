// sigma_3 (the alpha-beta term of Eq. 8) for FP32 CI vectors, in the shape of the
// FP64 per-row kernel (sigma3_sliced_kernel.cuh): per output alpha string I_a
//   G[J_b][q] = sum_a C(J_a, J_b) s_a (q | p_a)     (tensor cores, K = a)
//   sigma(I_a, I_b) += s_b G[J_b][q]                (integer adds, shared memory)
//
// C is scaled row by row to below one (an exact power of two) and cut into NS
// bf16 slices, rounded to nearest with the remainder carried on (NS = 3: 24 bits
// relative to the value itself; NS = 2: split-BF16x3), once per call, in planes
// [slice][row][pitch]; the integral operand carries the rows' scales, as in the
// FP64 kernel.  The NS (NS + 1) / 2 slice products i + j < NS accumulate in FP32
// in tensor memory, the small ones first in every K-step.  G is below K <= 96 in
// these scales: the epilogue writes it as round(2^37 G) = 2^22 h + l with two
// magic-number additions and adds h and l to two 32-bit words of the target's
// slot of the sigma row in shared memory (|h| < 2^22 and |l| <= 2^21, at most 96
// adds: neither overflows; exact, in any order: the result is bit-reproducible).
//
// The kernel before this one (sigma_tc_kernel.cuh, which still takes smaller spaces
// and rows that do not fit) split C into slices once per replacement, 56 times a
// value at CAS(14,14), in the producers' registers, and gathered each target's
// contributions on four warps.  sigma_3 of one call, slices included, before and
// now: 2.97 and 2.24 ms at CAS(14,14), 55.7 and 36.4 ms at CAS(16,16).
//
// What bounds it at CAS(14,14): the copies of C's rows (0.75 GB of cp.async through
// L2 for 56 replacements x 3 slices, with their hand-over to the MMAs) and the shared
// adds take about equal parts; with the epilogue's adds left out it takes 1.5 ms,
// with neither adds, copies nor MMAs (row set-up and hand-overs alone) 1.2 ms.  Four
// producer warps that hand over every K-step together, each waiting for its own
// copies, took 2.79 ms, three warps with pairs of K-steps 2.32, a warp per K-step
// 2.21 (but 45.9 ms at CAS(16,16), whose ring holds four K-steps).  Two 32-bit
// adds of split words against a 64-bit sum with carry: the carry waits for the old
// value of the low word, 0.9 ms of the 2.79.
//
// CTA (544 threads), one per SM, persistent over rows: warps 0-3 copy the planes'
// row segments into a ring of MN-major K-steps with 16-byte asynchronous copies
// (rows past the replacement list are filled with zeros), warps 4-15 epilogue,
// warp 16 MMAs into two accumulators in turn.  All waits are bounded.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sigma3_sliced_kernel.cuh"

namespace fci {
namespace s3f {

using sl::kEpiGroups;
using sl::kEpiThreads;
using sl::kMmaWarp;
using sl::kThreads;
using tc::kM;

constexpr int kMaxStages = 8;
constexpr int kBars = 2 * kMaxStages + 5;     // a_full[], a_free[], acc_full[2], acc_empty[2], drain

struct Layout {
    uint32_t bytesB, offA, offAcc, offEa, offBar, total;
};

// Shared memory: B slices [NS][npad x kpad], A stages [nst][NS][4 KB], the sigma
// row (low words, high words), the alpha list, barriers and words.
__host__ __device__ inline Layout make_layout(int ns, int kpad, int npad, int nst, int64_t nsb, int nsingle_a) {
    Layout L;
    L.bytesB = (uint32_t)(npad * kpad * 2);
    L.offA = ((uint32_t)ns * L.bytesB + 1023u) & ~1023u;
    L.offAcc = L.offA + (uint32_t)(nst * ns) * 4096u;
    L.offEa = L.offAcc + (uint32_t)((nsb * 8 + 15) / 16 * 16);
    L.offBar = L.offEa + (uint32_t)((nsingle_a + 3) / 4 * 16);
    L.total = L.offBar + kBars * 8 + 16;
    return L;
}

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16u : 0u) : "memory");
}

// out[r] = largest biased exponent of row r of C (at least 1); a warp per row
__global__ void k_row_exponents_f32(const float *__restrict__ C, int64_t nrows, int64_t ncols, int *__restrict__ out,
                                    const int *__restrict__ active) {
    if (active != nullptr && *active == 0) return;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= nrows) return;
    unsigned mx = 1;
    for (int64_t j = lane; j < ncols; j += 32) mx = max(mx, (__float_as_uint(__ldg(C + r * ncols + j)) >> 23) & 0xFFu);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if (lane == 0) out[r] = (int)mx;
}

// 2^e for any e of interest (|e| < 280): the product of two powers, exact where
// the scaled value is a normal number
__device__ __forceinline__ float scale2(float x, int e) {
    const int h = e / 2;
    return x * __int_as_float((127 + h) << 23) * __int_as_float((127 + e - h) << 23);
}

// Slices of C 2^-(exponent of the row) (below one in magnitude; zero in a
// non-finite row, whose results are NaN anyway), 8 columns per thread, zeros up
// to the pitch.
template <int NS>
__global__ void k_slice_f32(const float *__restrict__ C, const int *__restrict__ rowexp, int64_t nrows, int64_t ncols,
                            int64_t pitch, uint16_t *__restrict__ planes, const int *__restrict__ active) {
    if (active != nullptr && *active == 0) return;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t groups = pitch / 8;
    if (t >= nrows * groups) return;
    const int64_t r = t / groups, j0 = (t - r * groups) * 8;
    const int e = __ldg(rowexp + r);
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        v[i] = (j0 + i < ncols && e < 0xFF) ? scale2(__ldg(C + r * ncols + j0 + i), 126 - e) : 0.f;
    uint32_t w[NS][4];
    tc::split8p<NS>(v, w);
#pragma unroll
    for (int s = 0; s < NS; ++s)
        *reinterpret_cast<uint4 *>(planes + (s * nrows + r) * pitch + j0) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

template <int KPAD, int NS>
__global__ void __launch_bounds__(kThreads, 1)
    k_sigma3_f32(const uint16_t *__restrict__ planes, int64_t pitch, float *__restrict__ sig, SpinTables A, SpinTables B,
                 const float *__restrict__ Wf, const int *__restrict__ rowexp, int npair, int npad, int nst, int eW,
                 uint32_t tmem_cols, int *err, const int *__restrict__ active) {
    if (active != nullptr && *active == 0) return;
    constexpr int NKS = KPAD / 16;
    constexpr int kgroups = KPAD / 8;
    constexpr uint32_t sbo = (uint32_t)(KPAD / 8) * 128u;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int64_t nsb = B.ns;
    const int sa_n = A.nsingle;
    const Layout L = make_layout(NS, KPAD, npad, nst, nsb, sa_n);
    unsigned char *sB = smem;
    uint32_t *sLo = reinterpret_cast<uint32_t *>(smem + L.offAcc);  // sum of l
    uint32_t *sHi = sLo + nsb;                                      // sum of h
    uint32_t *sEa = reinterpret_cast<uint32_t *>(smem + L.offEa);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.offBar);
    volatile int *s_fail = reinterpret_cast<volatile int *>(smem + L.offBar + kBars * 8);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + L.offBar + kBars * 8 + 4);
    volatile int *s_emax = reinterpret_cast<volatile int *>(smem + L.offBar + kBars * 8 + 8);
    const uint32_t bar0 = tc::smem_u32(bars);
    const uint32_t a0 = tc::smem_u32(smem + L.offA);
    auto a_full = [&](int st) { return bar0 + 8u * (uint32_t)st; };
    auto a_free = [&](int st) { return bar0 + 8u * (uint32_t)(kMaxStages + st); };
    auto acc_full = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + 2 + b); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kMaxStages + 4);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const bool elected = tc::elect_one();

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tslot)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < nst; ++i) {
            tc::mbar_init(a_full(i), 64);
            tc::mbar_init(a_free(i), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(acc_full(b), 1);
            tc::mbar_init(acc_empty(b), kEpiThreads);
        }
        tc::mbar_init(drain, 1);
        *s_fail = 0;
    }
    for (int64_t j = tid; j < nsb; j += kThreads) sLo[j] = sHi[j] = 0u;
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tslot;
    const int64_t ntiles = (nsb + kM - 1) / kM;
    int64_t T = 0;  // tiles done by this CTA (barrier phases)

    for (int64_t row = blockIdx.x; row < A.ns; row += gridDim.x) {
        // ---- row set-up: alpha list, common exponent, B slices ----
        for (int e = tid; e < sa_n; e += kThreads) sEa[e] = A.tab[(int64_t)e * A.ns + row];
        __syncthreads();
        if (warp == 0) {
            int mx = 0;
            for (int e = lane; e < sa_n; e += 32) mx = max(mx, __ldg(rowexp + ent_target(sEa[e])));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            if (lane == 0) *s_emax = mx;
        }
        __syncthreads();
        const int emax = *s_emax;
        // B[q][a] = s_a (q | p_a) 2^(e_row(J_a) - emax - eW), K-major per slice
        for (int item = tid; item < npad * kgroups; item += kThreads) {
            const int q = item / kgroups, kg = item % kgroups;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int a = kg * 8 + i;
                float x = 0.f;
                if (q < npair && a < sa_n) {
                    const uint32_t ea = sEa[a];
                    const int d = __ldg(rowexp + ent_target(ea)) - emax;
                    x = d < -126 ? 0.f : scale2(__ldg(Wf + (int64_t)q * npair + ent_pair(ea)), d - eW);
                    if (ent_negative(ea)) x = -x;
                }
                v[i] = x;
            }
            tc::store_split8p<NS>(v, sB, L.bytesB, tc::kmajor_offset(q, kg, KPAD));
        }
        tc::fence_async_smem();
        tc::fence_before();
        __syncthreads();
        tc::fence_after();

        if (warp < 4) {
            // ---- producers: two pairs of warps take alternate K-steps, so that the
            // waits and proxy fences (several hundred cycles each) of one overlap the
            // other's; a K-step is handed over when the pair has issued its next one,
            // or before it blocks on a buffer that is not free yet ----
            const int64_t plane = A.ns * pitch, end = (T + ntiles) * NKS;
            int64_t held = -1;  // K-step issued and not yet handed over
            const int c = lane & 15, sub = (warp >> 1) * 2 + (lane >> 4);  // replacement rows sub, sub + 4, ...
            bool ok = true;
            auto hand_over = [&]() {
                tc::fence_async_smem();
                tc::mbar_arrive(a_full((int)(held % nst)));
                held = -1;
            };
            for (int64_t g = T * NKS + (warp & 1); g < end; g += 2) {
                const int st = (int)(g % nst);
                const uint32_t ph = (uint32_t)((g / nst - 1) & 1);
                if (g >= nst && !tc::mbar_try_wait(a_free(st), ph)) {
                    if (held >= 0) {
                        sl::cp_async_wait<0>();
                        hand_over();
                    }
                    if (!tc::mbar_wait_bounded(a_free(st), ph)) {
                        ok = false;
                        break;
                    }
                }
                const int64_t t = g / NKS - T;
                const int ks = (int)(g - (t + T) * NKS);
                const uint16_t *col = planes + t * kM + c * 8;
                const uint32_t base = a0 + (uint32_t)(st * NS) * 4096u + (uint32_t)((c >> 3) * 2048);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int al = r * 4 + sub, a = ks * 16 + al;
                    const bool live = a < sa_n;
                    const uint16_t *q = col + (live ? (int64_t)ent_target(sEa[a]) * pitch : 0);
                    const uint32_t dst = base + (uint32_t)((al >> 3) * 1024 + (al & 7) * 128 + (((c & 7) ^ (al & 7)) << 4));
#pragma unroll
                    for (int s = 0; s < NS; ++s) cp_async16_zfill(dst + (uint32_t)s * 4096u, q + s * plane, live);
                }
                sl::cp_async_commit();
                if (held >= 0) {
                    sl::cp_async_wait<1>();
                    hand_over();
                }
                held = g;
            }
            sl::cp_async_wait<0>();
            if (!ok)
                *s_fail = 1;
            else if (held >= 0)
                hand_over();
        } else if (warp < kMmaWarp) {
            // ---- epilogue: lane m of the tile, 8-column chunks grp, grp + 3, ... ----
            const int quarter = warp & 3, grp = (warp - 4) >> 2;
            const int m = quarter * 32 + lane;
            const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
            const uint32_t lo0 = tc::smem_u32(sLo), hi0 = tc::smem_u32(sHi);
            const int nchunks = npad / 8;
            for (int64_t t = 0; t < ntiles; ++t) {
                const int64_t Tt = T + t;
                const int b = (int)(Tt & 1);
                const int64_t jb = t * kM + m;
                const bool live = jb < nsb;
                const uint4 *trow = reinterpret_cast<const uint4 *>(B.tabp + (live ? jb : 0) * npad);
                auto fetch = [&](int c) { return live ? sl::ld_early_v4(trow + c) : make_uint4(~0u, ~0u, ~0u, ~0u); };
                uint4 ent = make_uint4(~0u, ~0u, ~0u, ~0u);
                if (grp < nchunks) ent = fetch(grp);
                if (!tc::mbar_wait_bounded(acc_full(b), (uint32_t)((Tt >> 1) & 1))) {
                    *s_fail = 1;
                    break;
                }
                tc::fence_after();
                if (grp >= nchunks) {
                    tc::fence_before();
                    tc::mbar_arrive(acc_empty(b));
                }
                for (int c = grp; c < nchunks; c += kEpiGroups) {
                    uint32_t r[8];
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                                   "=r"(r[7])
                                 : "r"(lane_base + (uint32_t)(b * npad + c * 8)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (c + kEpiGroups >= nchunks) {  // last chunk of this thread: release the accumulator
                        tc::fence_before();
                        tc::mbar_arrive(acc_empty(b));
                    }
                    const uint32_t ew[4] = {ent.x, ent.y, ent.z, ent.w};
                    if (c + kEpiGroups < nchunks) ent = fetch(c + kEpiGroups);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        constexpr float M = 12582912.0f;  // 1.5 2^23
                        constexpr int MB = 0x4B400000;
                        const uint32_t v16 = (j & 1) ? (ew[j >> 1] >> 16) : (ew[j >> 1] & 0xFFFFu);
                        const float x = __uint_as_float(r[j] ^ ((v16 & 0x8000u) << 16));  // sign of the replacement
                        const float t1 = fmaf(x, 0x1p15f, M);              // round(2^15 x), |x| <= 2^7
                        const float rem = fmaf(-(t1 - M), 0x1p-15f, x);    // exact
                        const uint32_t at = 4u * (v16 & 0x7FFFu);
                        sl::red_add_if(hi0 + at, (uint32_t)(__float_as_int(t1) - MB), v16 != 0xFFFFu);
                        sl::red_add_if(lo0 + at, (uint32_t)(__float_as_int(fmaf(rem, 0x1p37f, M)) - MB), v16 != 0xFFFFu);
                    }
                }
                if (*s_fail) break;
            }
        } else if (warp == kMmaWarp) {
            // ---- MMAs (all lanes run the loop, the elected one issues) ----
            const uint64_t ad = sl::smem_desc_mn(a0, 2048, 1024);
            const uint64_t bd = tc::smem_desc(tc::smem_u32(sB), 128, sbo);
            const uint32_t idesc = tc::instr_desc(kM, npad) | sl::kTransposeA;
            int64_t g = T * NKS;
            bool ok = true;
            for (int64_t t = 0; t < ntiles && ok; ++t) {
                const int64_t Tt = T + t;
                const int b = (int)(Tt & 1);
                if (Tt >= 2 && !tc::mbar_wait_bounded(acc_empty(b), (uint32_t)(((Tt - 2) >> 1) & 1))) ok = false;
#pragma unroll
                for (int ks = 0; ks < NKS; ++ks, ++g) {
                    const int st = (int)(g % nst);
                    if (ok && !tc::mbar_wait_bounded(a_full(st), (uint32_t)((g / nst) & 1))) ok = false;
                    if (!ok) break;
                    tc::fence_after();
                    if (!elected) continue;
#pragma unroll
                    for (int lv = NS - 1; lv >= 0; --lv)  // slice products i + j = lv
#pragma unroll
                        for (int i = 0; i <= lv; ++i)
                            tc::mma_bf16(tmem + (uint32_t)(b * npad), ad + (uint64_t)((st * NS + i) * 256),
                                         bd + (uint64_t)(((lv - i) * L.bytesB >> 4) + ks * 16), idesc,
                                         (ks == 0 && lv == NS - 1 && i == 0) ? 0u : 1u);
                    tc::mma_commit(a_free(st));
                }
                if (!ok) {
                    *s_fail = 1;
                    break;
                }
                if (elected) tc::mma_commit(acc_full(b));
            }
        }
        // ---- row end: every entry of the row has been added ----
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        T += ntiles;
        if (*s_fail) break;
        const int e2 = emax - 126 + eW - 37;
        float *out = sig + row * nsb;
        for (int64_t j = tid; j < nsb; j += kThreads) {
            const long long v = (long long)(int)sHi[j] * 4194304ll + (int)sLo[j];
            out[j] += emax == 0xFF ? __int_as_float(0x7FC00000) : (float)sl::scaled_i64(v, e2);
            sLo[j] = sHi[j] = 0u;
        }
        __syncthreads();
    }
    // ---- exit: wait for every MMA this CTA issued, then free tensor memory ----
    if (warp == kMmaWarp) {
        if (elected) tc::mma_commit(drain);
        if (!tc::mbar_wait_bounded(drain, 0u)) *s_fail = 1;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (*s_fail && tid == 0) atomicOr(err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

// (no space of norb <= 30 with kMinRows strings has 32 replacements or fewer)
template <int NS>
static void *kernel(int kpad) {
    switch (kpad) {
        case 48: return (void *)k_sigma3_f32<48, NS>;
        case 64: return (void *)k_sigma3_f32<64, NS>;
        case 80: return (void *)k_sigma3_f32<80, NS>;
        case 96: return (void *)k_sigma3_f32<96, NS>;
        default: return nullptr;
    }
}

struct Plan {
    int kpad = 0, npad = 0, nst = 0;
    uint32_t cols = 0, smem = 0;
    void *kern = nullptr;
};

// A row's set-up (exponents, integral slices) and the slicing pass pay off over
// seven tiles of beta strings and four rows per SM: 792 x 792 strings 156 us against
// 159 with the kernel of sigma_tc_kernel.cuh, 924 x 924 201 against 209, 1287 x 1287
// 359 against 385; below, 715 x 715 strings 137 against 121, 364 x 1001 114 against
// 105, 252 x 252 32 against 22.
constexpr int64_t kMinRows = 600, kMinStrings = 769;

// Sizes for this context (the ring as deep as fits, at least four K-steps);
// false when the kernel does not cover it.
static bool plan(const fci_ctx *ctx, Plan *P) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const int ns = ctx->opt.f32_splits;
    P->kpad = (A.nsingle + 15) / 16 * 16;
    P->npad = (ctx->npair + 15) / 16 * 16;
    if (A.nsingle == 0 || B.nsingle == 0 || P->kpad < 48 || P->kpad > 96 || P->npad > 256 || B.ns > 0x7FFF || B.nsingle > 96 ||
        A.ns < kMinRows || B.ns < kMinStrings)
        return false;
    int lim = 0;
    if (cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device) != cudaSuccess) return false;
    for (P->nst = kMaxStages; P->nst >= 4; --P->nst) {
        P->smem = make_layout(ns, P->kpad, P->npad, P->nst, B.ns, A.nsingle).total;
        if ((int)P->smem <= lim) break;
    }
    if (P->nst < 4) return false;
    P->cols = 32;
    while ((int)P->cols < 2 * P->npad) P->cols <<= 1;
    P->kern = ns == 2 ? kernel<2>(P->kpad) : kernel<3>(P->kpad);
    return true;
}

}  // namespace s3f

bool sigma3_f32_ok(const fci_ctx *ctx) { return ctx->rowexp32 != nullptr; }

// Row exponents, the slice planes (those of the FP64 kernels when the context has
// them: one call at a time uses either) and the pair-major beta table.
int build_sigma3_f32(fci_ctx *ctx, const double *eri_host) {
    s3f::Plan P;
    if (ctx->opt.f32_row_global != 0 || sigma_small_ok(ctx, FCI_F32) || !s3f::plan(ctx, &P)) return FCI_OK;
    const int n = ctx->norb;
    double wmax = 0.0;
    for (int64_t i = 0; i < (int64_t)n * n * n * n; ++i) wmax = std::fmax(wmax, std::fabs(eri_host[i]));
    if (wmax > 0) std::frexp(wmax, &ctx->eW32);  // |W| < 2^eW32
    const size_t bytes = sizeof(uint16_t) * ctx->opt.f32_splits * (size_t)ctx->A.ns * plane_pitch(ctx->B.ns);
    int rc = grow_buffer(ctx, (void **)&ctx->planes, &ctx->planes_bytes, bytes);
    if (!rc && !ctx->B.tabp) rc = build_pair_table16(ctx);
    ctx->rowexp32 = rc ? nullptr : (int *)dalloc(ctx, sizeof(int) * (size_t)ctx->A.ns, &rc);
    if (rc) return rc;
    FCI_CUDA(opt_in_max_smem(P.kern, ctx->device));
    return FCI_OK;
}

void free_sigma3_f32(fci_ctx *ctx) {
    dfree(ctx, ctx->rowexp32, sizeof(int) * (size_t)ctx->A.ns);
    ctx->rowexp32 = nullptr;
}

// sig += sigma_3 (stream-ordered; the opt-in was done at fci_init)
int launch_sigma3_f32(fci_ctx *ctx, const float *C, float *sig, cudaStream_t s, const int *active) {
    s3f::Plan P;
    if (!sigma3_f32_ok(ctx) || !s3f::plan(ctx, &P)) return fail(FCI_ERR_STATE, "FP32 sigma_3 tables were not built for this context");
    const SpinTables &A = ctx->A, &B = ctx->B;
    int64_t pitch = plane_pitch(B.ns);
    s3f::k_row_exponents_f32<<<ceil_div(A.ns * 32, 256), 256, 0, s>>>(C, A.ns, B.ns, ctx->rowexp32, active);
    const unsigned grid8 = ceil_div(A.ns * (pitch / 8), 256);
    if (ctx->opt.f32_splits == 2)
        s3f::k_slice_f32<2><<<grid8, 256, 0, s>>>(C, ctx->rowexp32, A.ns, B.ns, pitch, ctx->planes, active);
    else
        s3f::k_slice_f32<3><<<grid8, 256, 0, s>>>(C, ctx->rowexp32, A.ns, B.ns, pitch, ctx->planes, active);
    FCI_CUDA(cudaGetLastError());
    int nsm = 0;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    const unsigned grid = (unsigned)std::min<int64_t>(nsm, A.ns);
    SpinTables At = A, Bt = B;
    const uint16_t *planes = ctx->planes;
    void *args[] = {(void *)&planes,        (void *)&pitch,       (void *)&sig,    (void *)&At,    (void *)&Bt,
                    (void *)&ctx->Wf,       (void *)&ctx->rowexp32, (void *)&ctx->npair, (void *)&P.npad, (void *)&P.nst,
                    (void *)&ctx->eW32,     (void *)&P.cols,      (void *)&ctx->d_err, (void *)&active};
    FCI_CUDA(cudaLaunchKernel(P.kern, dim3(grid), dim3(s3f::kThreads), args, P.smem, s));
    return FCI_OK;
}

}  // namespace fci
