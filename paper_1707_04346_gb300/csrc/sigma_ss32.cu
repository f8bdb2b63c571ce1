// FP32 same-spin sigma terms (sigma_1 and sigma_2 of Eq. 8) as dense products on
// the bf16 tensor cores:
//   sigma_1(I_a, I_b) = sum_{J_b} G_b(I_b, J_b) C(I_a, J_b)
//   sigma_2(I_a, I_b) = sum_{J_a} G_a(I_a, J_a) C(J_a, I_b)
// with the off-diagonal part of the dense same-spin Hamiltonians G_s (see
// sigma_ss.cu) and the diagonal, which dwarfs the couplings, applied in FP32 in
// sigma_2's epilogue.
//
// FP32 accuracy: every value is split into three bf16 slices (rounded to
// nearest, the remainder carried on: 24 bits relative to the value itself), and
// the six slice products i + j < 3 accumulate in FP32 in tensor memory.  The
// tensor cores' FP32 accumulation does not round to nearest, so few terms go
// through it: every 64 terms the epilogue adds the accumulator to FP32 sums in
// registers, and within such a group the small products come first (i + j = 2,
// then 1, then the leading ones of the four K-steps last).
//
// One launch computes both terms.  The narrow operand A (the MMA's M) is G in
// blocks of 128 rows, whose all-zero K-steps are left out (7 % at CAS(14,14), 28
// % at CAS(16,16)); B is C in blocks of NB rows:
//   sigma_1: m = I_b, n = I_a, k = J_b;   sigma_2: m = I_a, n = I_b, k = J_a.
// Operand tiles are contiguous ([block][K-step][3][rows x 16], one bulk copy
// each).  NB = 256 keeps the six MMAs of a K-step at full width (768 cycles; an
// M = 128 MMA re-reads 4 KB of A) with two accumulators in tensor memory; NB =
// 64 for small spaces, so that their tiles spread over the SMs.  Both terms meet
// on each element: sigma starts at zero and takes two atomic adds, whose order
// does not change the sum of two addends onto zero.
//
// Both terms with their passes over C, against the fused table-driven FP32 kernel
// before (unequal spins: one kernel per term): CAS(14,14) 2.24 -> 0.75 ms,
// CAS(16,16) 80.3 -> 25.7 ms.
#include <algorithm>

#include "sliced_mma.cuh"

namespace fci {
namespace s32 {

using sm::bulk_g2s;
using sm::mbar_expect_tx;
using tc::kM;

constexpr int kSl = 3;      // bf16 slices
constexpr int kGroup = 4;   // K-steps (64 terms) per accumulator
constexpr uint32_t kBytesA = kSl * 4096;

template <int NB>
struct Shape {
    static constexpr uint32_t kBytesB = kSl * NB * 32;
    static constexpr uint32_t kStageBytes = kBytesA + kBytesB;
    static constexpr int kStages = NB == 256 ? 6 : 8;
    static constexpr int kSub = NB == 256 ? 2 : 1;  // epilogue warps per lane quarter
    static constexpr int kCols = NB / kSub;         // columns per epilogue thread
    static constexpr int kEpiThreads = 128 * kSub;
    static constexpr int kThreads = 64 + kEpiThreads;
    static constexpr uint32_t kTmem = 2 * NB;
    static constexpr int kBars = 2 * kStages + 5;  // full, free, acc_full[2], acc_empty[2], drain
    static constexpr uint32_t kSmem = kStages * kStageBytes + kBars * 8 + 16;
};

inline int64_t nblocks(int64_t rows, int nb) { return (rows + nb - 1) / nb; }
inline int64_t ksteps(int64_t k) { return (k + 15) / 16; }
inline size_t c_bytes(int64_t rows, int64_t k, int nb) { return (size_t)ksteps(k) * nblocks(rows, nb) * kSl * nb * 32; }

__device__ __forceinline__ uint32_t core_offset(int r, int kk) {
    return (uint32_t)((r >> 3) * 256 + (kk >> 3) * 128 + (r & 7) * 16 + (kk & 7) * 2);
}

// off-diagonal ELL entries of G into their slices (each row's columns are
// distinct; the planes start at zero)
__global__ void k_s32_gplanes(const int32_t *__restrict__ gcol, const double *__restrict__ gval, int64_t ns, int nsame,
                              int64_t nks, const int *__restrict__ slot, unsigned char *__restrict__ planes) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ns || t >= ns * (int64_t)nsame) return;  // slot 0: the diagonal
    const int64_t x = t % ns;
    double v = gval[t];
    if (v == 0.0) return;
    const int col = gcol[t];
    unsigned char *tile = planes + (size_t)slot[x / kM * nks + (col >> 4)] * kBytesA;
    const uint32_t off = core_offset((int)(x % kM), col & 15);
#pragma unroll
    for (int s = 0; s < kSl; ++s) {
        const __nv_bfloat16 b = __float2bfloat16_rn((float)v);
        *reinterpret_cast<__nv_bfloat16 *>(tile + s * 4096 + off) = b;
        v -= (double)__bfloat162float(b);
    }
}

// C's slices by rows (plane row = row of C, k = column; nullptr: not wanted) and
// by columns from one read of a 64 x 64 tile; plane rows past the matrix are
// written as zeros up to whole NB-row blocks (the grid covers them).
template <int NB>
__global__ void __launch_bounds__(256) k_s32_cplanes(const float *__restrict__ C, int64_t nrows, int64_t ncols,
                                                     unsigned char *__restrict__ prow, unsigned char *__restrict__ pcol,
                                                     const int *__restrict__ active) {
    if (active != nullptr && *active == 0) return;
    __shared__ float t[64][65];
    const int64_t c0 = (int64_t)blockIdx.x * 64, r0 = (int64_t)blockIdx.y * 64;
    for (int i = threadIdx.x; i < 64 * 64; i += 256) {
        const int64_t r = r0 + (i >> 6), c = c0 + (i & 63);
        t[i >> 6][i & 63] = (r < nrows && c < ncols) ? C[r * ncols + c] : 0.f;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < 1024; it += 256) {
        const bool cols = it >= 512;
        unsigned char *planes = cols ? pcol : prow;
        if (planes == nullptr) continue;
        const int x = it & 63, g = (it >> 6) & 7;
        const int64_t r = (cols ? c0 : r0) + x, k0 = (cols ? r0 : c0) + g * 8;
        const int64_t rows = cols ? ncols : nrows, klen = cols ? nrows : ncols, nnb = (rows + NB - 1) / NB;
        if (k0 >= (klen + 15) / 16 * 16 || r >= nnb * NB) continue;
        float v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = cols ? t[g * 8 + i][x] : t[x][g * 8 + i];
        unsigned char *tile = planes + ((size_t)(k0 >> 4) * nnb + r / NB) * (kSl * NB * 32);
        tc::store_split8p<kSl>(v, tile, NB * 32, core_offset((int)(r % NB), (int)(k0 & 15)));
    }
}

struct Product {
    const unsigned char *A, *B;
    const int *koff, *kidx;     // K-steps of row block mb of A
    int M, N;
    int64_t sm, sn;             // out[m sm + n sn] += (one of sm, sn is 1)
    const float *dm, *dn;       // diagonal: += (dm[m] + dn[n]) C at the same place (dm null: none; dn may be null)
};

struct Args {
    Product P[2];
    int t0, ntiles;             // tiles of P[0], of both
    float *out;
    const float *C;
    int *err;
    const int *active;
};

template <int NB>
__global__ void __launch_bounds__(Shape<NB>::kThreads, 1) k_s32_tc(const __grid_constant__ Args Q) {
    if (Q.active != nullptr && *Q.active == 0) return;
    using S = Shape<NB>;
    constexpr int kStages = S::kStages;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kStages * S::kStageBytes);
    volatile int *s_fail = reinterpret_cast<volatile int *>(smem + kStages * S::kStageBytes + S::kBars * 8);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + kStages * S::kStageBytes + S::kBars * 8 + 4);
    const uint32_t sbase = tc::smem_u32(smem);
    const uint32_t bar0 = tc::smem_u32(bars);
    auto full = [&](int st) { return bar0 + 8u * (uint32_t)st; };
    auto freeb = [&](int st) { return bar0 + 8u * (uint32_t)(kStages + st); };
    auto acc_full = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kStages + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kStages + 2 + b); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kStages + 4);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const bool elected = tc::elect_one();

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tslot)),
                     "r"(S::kTmem)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kStages; ++i) {
            tc::mbar_init(full(i), 1);
            tc::mbar_init(freeb(i), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(acc_full(b), 1);
            tc::mbar_init(acc_empty(b), S::kEpiThreads);
        }
        tc::mbar_init(drain, 1);
        *s_fail = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tslot;
    // product, row blocks and K-step list of tile t
    auto tile = [&](int t, int &w, int &mb, int &nb, int &k0, int &k1) {
        w = t >= Q.t0;
        const Product &P = Q.P[w];
        const int r = w ? t - Q.t0 : t, nmb = (P.M + kM - 1) / kM;
        mb = r % nmb;
        nb = r / nmb;
        k0 = __ldg(P.koff + mb);
        k1 = __ldg(P.koff + mb + 1);
    };

    int64_t G_copied = 0;
    if (warp == 0 && lane == 0) {
        // ---- copies ----
        int64_t &G = G_copied;
        for (int t = blockIdx.x; t < Q.ntiles && !*s_fail; t += gridDim.x) {
            int w, mb, nb, k0, k1;
            tile(t, w, mb, nb, k0, k1);
            const Product &P = Q.P[w];
            const int nnb = (P.N + NB - 1) / NB;
            for (int k = k0; k < k1; ++k, ++G) {
                const int st = (int)(G % kStages);
                const size_t ks = (size_t)__ldg(P.kidx + k);
                if (G >= kStages && !tc::mbar_wait_bounded(freeb(st), (uint32_t)((G / kStages - 1) & 1))) {
                    *s_fail = 1;
                    break;
                }
                mbar_expect_tx(full(st), S::kStageBytes);
                const uint32_t dst = sbase + (uint32_t)st * S::kStageBytes;
                bulk_g2s(dst, P.A + (size_t)k * kBytesA, kBytesA, full(st));
                bulk_g2s(dst + kBytesA, P.B + (ks * nnb + nb) * S::kBytesB, S::kBytesB, full(st));
            }
        }
    } else if (warp == 1) {
        // ---- MMAs (all lanes run the loop, the elected one issues) ----
        const uint64_t a0 = tc::smem_desc(sbase, 128, 256), b0 = tc::smem_desc(sbase + kBytesA, 128, 256);
        constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
        int64_t G = 0, Tt = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < Q.ntiles && ok; t += gridDim.x) {
            int w, mb, nb, k0, k1;
            tile(t, w, mb, nb, k0, k1);
            for (int k = k0; k < k1 && ok; k += kGroup, ++Tt) {
                const int b = (int)(Tt & 1), n = min(kGroup, k1 - k);
                if (Tt >= 2 && !tc::mbar_wait_bounded(acc_empty(b), (uint32_t)(((Tt - 2) >> 1) & 1))) {
                    ok = false;
                    break;
                }
#pragma unroll
                for (int lv = kSl - 1; lv >= 0; --lv)  // products i + j = lv
                    for (int j = 0; j < n && ok; ++j) {
                        const int st = (int)((G + j) % kStages);
                        if (lv == kSl - 1 && !tc::mbar_wait_bounded(full(st), (uint32_t)(((G + j) / kStages) & 1))) {
                            ok = false;
                            break;
                        }
                        tc::fence_after();
                        if (!elected) continue;
                        const uint64_t so = (uint64_t)((st * S::kStageBytes) >> 4);
#pragma unroll
                        for (int i = 0; i <= lv; ++i)
                            tc::mma_bf16(tmem + b * NB, a0 + so + (uint64_t)(i * 256), b0 + so + (uint64_t)((lv - i) * NB * 2),
                                         idesc, (lv == kSl - 1 && i == 0 && j == 0) ? 0u : 1u);
                        if (lv == 0) tc::mma_commit(freeb(st));
                    }
                G += n;
                if (ok && elected) tc::mma_commit(acc_full(b));
            }
        }
        if (!ok) *s_fail = 1;
    } else if (warp >= 2) {
        // ---- epilogue: lane m of the tile, columns kCols sub .. ----
        constexpr int kCols = S::kCols;
        const int quarter = warp & 3, sub = (warp - 2) >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(sub * kCols);
        int64_t Tt = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < Q.ntiles && ok; t += gridDim.x) {
            int w, mb, nb, k0, k1;
            tile(t, w, mb, nb, k0, k1);
            const Product &P = Q.P[w];
            float sum[kCols];
#pragma unroll
            for (int j = 0; j < kCols; ++j) sum[j] = 0.f;
            for (int k = k0; k < k1; k += kGroup, ++Tt) {
                const int b = (int)(Tt & 1);
                if (!tc::mbar_wait_bounded(acc_full(b), (uint32_t)((Tt >> 1) & 1))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
#pragma unroll
                for (int h = 0; h < kCols; h += 16) {
                    uint32_t r[16];
                    asm volatile(
                        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                          "=r"(r[15])
                        : "r"(lane_base + (uint32_t)(b * NB + h)));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[h + j] += __uint_as_float(r[j]);
                }
                tc::fence_before();
                tc::mbar_arrive(acc_empty(b));
            }
            if (!ok) break;
            const int mrow = mb * kM + quarter * 32, ncol = nb * NB + sub * kCols;
            auto put = [&](int m, int n, float v) {
                if (m >= P.M || n >= P.N) return;
                const int64_t o = m * P.sm + n * P.sn;
                if (P.dm) v = fmaf(P.dm[m] + (P.dn ? P.dn[n] : 0.f), Q.C[o], v);
                atomicAdd(Q.out + o, v);
            };
            if (P.sn == 1) {
                // transpose 32 x 32 blocks over the warp: the adds run along a row of sigma
#pragma unroll
                for (int h = 0; h < kCols; h += 32) {
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1)
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (!(j & d)) {
                                const bool up = (lane & d) != 0;
                                const float got = __shfl_xor_sync(0xFFFFFFFFu, up ? sum[h + j] : sum[h + j + d], d);
                                sum[h + j] = up ? got : sum[h + j];
                                sum[h + j + d] = up ? sum[h + j + d] : got;
                            }
#pragma unroll
                    for (int j = 0; j < 32; ++j) put(mrow + j, ncol + h + lane, sum[h + j]);
                }
            } else {
#pragma unroll
                for (int j = 0; j < kCols; ++j) put(mrow + lane, ncol + j, sum[j]);
            }
        }
        if (!ok) *s_fail = 1;
    }
    // ---- exit: wait for every MMA this CTA issued and every copy it started,
    // then free tensor memory ----
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 1) {
        if (elected) tc::mma_commit(drain);
        if (!tc::mbar_wait_bounded(drain, 0u)) *s_fail = 1;
    }
    if (warp == 0 && lane == 0) {
        for (int st = 0; st < kStages; ++st) {
            const int64_t fills = G_copied / kStages + (st < G_copied % kStages ? 1 : 0);
            if (fills > 0 && !tc::mbar_wait_bounded(full(st), (uint32_t)((fills - 1) & 1))) *s_fail = 1;
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (*s_fail && tid == 0) atomicOr(Q.err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kTmem) : "memory");
}

// Rows of C per tile: 256 where the tiles of both terms fill half of the chip, else 64.
static int tile_rows(const fci_ctx *ctx, int nsm) {
    const int64_t a = ctx->A.ns, b = ctx->B.ns;
    return 2 * (nblocks(a, kM) * nblocks(b, 256) + nblocks(b, kM) * nblocks(a, 256)) >= nsm ? 256 : 64;
}

}  // namespace s32

bool sigma_ss32_ok(const fci_ctx *ctx) { return ctx->ss32Ga.planes != nullptr; }

// Built where FCI_F32 covers the space at all (replacements of both spins on the
// tensor cores, see sigma_tc.cu), neither string space exceeds 16384 strings (as
// for the FP64 products) and neither the one-kernel sigma nor the caller's choice of
// the intermediate-string kernels takes the space anyway.
int build_ss32_tables(fci_ctx *ctx) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    if (A.nsingle == 0 || B.nsingle == 0 || A.nsingle > 96 || ctx->npair > 256 || A.ns > 16384 || B.ns > 16384) return FCI_OK;
    if (sigma_small_ok(ctx, FCI_F32) || ctx->opt.same_spin_tc == 1) return FCI_OK;
    int rc = FCI_OK, nsm = 0;
    cudaStream_t s = ctx->stream;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    auto build = [&](const SpinTables &T, SsOperand &O) -> int {
        int *slot = nullptr;
        size_t slot_bytes = 0;
        auto fill = [&]() -> int {
            if (int r = ss_kstep_lists(ctx, T, s32::kM, O, &slot, &slot_bytes)) return r;
            O.plane_bytes = O.nsteps * (size_t)s32::kBytesA;
            O.planes = (unsigned char *)dalloc(ctx, O.plane_bytes, &rc);
            if (rc) return rc;
            FCI_CUDA(cudaMemsetAsync(O.planes, 0, O.plane_bytes, s));
            s32::k_s32_gplanes<<<ceil_div(T.ns * (int64_t)T.nsame, 256), 256, 0, s>>>(
                T.gcol, T.gval, T.ns, T.nsame, s32::ksteps(T.ns), slot, O.planes);
            FCI_CUDA(cudaGetLastError());
            FCI_CUDA(cudaStreamSynchronize(s));
            return FCI_OK;
        };
        const int r = fill();
        dfree(ctx, slot, slot_bytes);
        return r;
    };
    if ((rc = build(A, ctx->ss32Ga))) return rc;
    if (A.gval == B.gval)
        ctx->ss32Gb = ctx->ss32Ga;
    else if ((rc = build(B, ctx->ss32Gb)))
        return rc;
    ctx->ss32_rows = s32::tile_rows(ctx, nsm);
    if ((rc = alloc_c_planes(ctx, s32::c_bytes(A.ns, B.ns, ctx->ss32_rows), s32::c_bytes(B.ns, A.ns, ctx->ss32_rows))))
        return rc;
    FCI_CUDA(opt_in_max_smem((const void *)s32::k_s32_tc<256>, ctx->device));
    FCI_CUDA(opt_in_max_smem((const void *)s32::k_s32_tc<64>, ctx->device));
    return FCI_OK;
}

void free_ss32_tables(fci_ctx *ctx) {
    if (ctx->ss32Gb.lists != ctx->ss32Ga.lists) free_ss_operand(ctx, ctx->ss32Gb, 0);
    ctx->ss32Gb = SsOperand{};
    free_ss_operand(ctx, ctx->ss32Ga, 0);
}

template <int NB>
static int launch_ss32(fci_ctx *ctx, const float *C, float *sig, int which, cudaStream_t s, const int *active) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const int64_t nsa = A.ns, nsb = B.ns;
    int nsm = 0;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    FCI_CUDA(cudaMemsetAsync(sig, 0, sizeof(float) * (size_t)ctx->ndet, s));
    s32::k_s32_cplanes<NB><<<dim3((unsigned)(s32::nblocks(nsb, NB) * (NB / 64)), (unsigned)(s32::nblocks(nsa, NB) * (NB / 64))),
                             256, 0, s>>>(C, nsa, nsb, which & 1 ? ctx->ssCr : nullptr, which & 2 ? ctx->ssCc : nullptr,
                                          active);
    FCI_CUDA(cudaGetLastError());
    s32::Args Q{};
    Q.out = sig;
    Q.C = C;
    Q.err = ctx->d_err;
    Q.active = active;
    int n = 0;
    auto add = [&](const SsOperand &G, int64_t M, const unsigned char *Bp, int64_t N, int64_t sm, int64_t sn, const float *dm,
                   const float *dn) {
        s32::Product &P = Q.P[n++];
        P.A = G.planes;
        P.koff = G.lists;
        P.kidx = G.lists + G.nnb + 1;
        P.B = Bp;
        P.M = (int)M;
        P.N = (int)N;
        P.sm = sm;
        P.sn = sn;
        P.dm = dm;
        P.dn = dn;
        Q.ntiles += (int)(s32::nblocks(M, s32::kM) * s32::nblocks(N, NB));
        if (n == 1) Q.t0 = Q.ntiles;
    };
    // sigma_2 with the diagonal of the spins asked for, sigma_1
    if (which & 2) add(ctx->ss32Ga, nsa, ctx->ssCc, nsb, nsb, 1, A.gvalf, which & 1 ? B.gvalf : nullptr);
    if (which & 1) add(ctx->ss32Gb, nsb, ctx->ssCr, nsa, 1, nsb, nullptr, nullptr);
    const unsigned grid = (unsigned)std::min<int64_t>(Q.ntiles, nsm);
    s32::k_s32_tc<NB><<<grid, s32::Shape<NB>::kThreads, s32::Shape<NB>::kSmem, s>>>(Q);
    FCI_CUDA(cudaGetLastError());
    return FCI_OK;
}

int launch_sigma_ss32(fci_ctx *ctx, const float *C, float *sig, int which, cudaStream_t s, const int *active) {
    if (!sigma_ss32_ok(ctx)) return fail(FCI_ERR_STATE, "FP32 same-spin planes were not built for this context");
    return ctx->ss32_rows == 256 ? launch_ss32<256>(ctx, C, sig, which, s, active)
                                 : launch_ss32<64>(ctx, C, sig, which, s, active);
}

}  // namespace fci
