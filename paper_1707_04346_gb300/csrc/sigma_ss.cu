// FP64 same-spin sigma terms (sigma_1 and sigma_2 of Eq. 8) as dense sliced
// contractions on the bf16 tensor cores.
//
// With G_s the Hamiltonian of spin s alone between the strings of that spin
// (the one-spin part of Eq. 6: diagonal, single and double replacements;
// symmetric),
//   sigma_1(I_a, I_b) = sum_{J_b} G_b(I_b, J_b) C(I_a, J_b)
//   sigma_2(I_a, I_b) = sum_{J_a} G_a(I_a, J_a) C(J_a, I_b).
// G_s has 1 + n(N-n) + C(n,2) C(N-n,2) nonzeros per row (491 of 3432 at
// CAS(14,14)).  Its diagonal (one-spin energies, tens of Eh against couplings
// well below one) is applied in FP64 separately; the off-diagonal part as a
// dense matrix makes both terms square matrix products, and
// the bf16 tensor pipe (1937 TFLOP/s measured) outruns the FP32 pipe (70) by
// far more than the zeros cost.  FP64 accuracy comes from the digit scheme of
// sliced_mma.cuh: every row of G_s and every row or column of C in 46-bit
// fixed point relative to its own largest power of two, six 8-bit digits, 21
// digit products with exact per-weight accumulation flushed into 64-bit
// integers every 256 terms, and at the end one FP64 conversion per element
// with the two scales of its row and column.
//
// One kernel computes out(m, n) += sum_k A(m, k) B(n, k) for a plane set A of C
// (rows m, the MMA's M: 128 per tile) and one B of G (rows n: NB per tile), each
// row with its own exponent:
//   sigma_1: A = C by rows (m = I_a, k = J_b), B = G_b (n = I_b);
//   sigma_2: A = C by columns (m = I_b, k = J_a), B = G_a (n = I_a); its epilogue
//            also applies the FP64 diagonal of both spins.
// Layout: an operand tile (six digit planes of its rows x 16 columns in the
// K-major no-swizzle core-matrix layout) is contiguous, so that one bulk copy
// stages it: A [K-step][128-row block][6][4 KB], B [row block][K-step][6][32 NB].
// (An SM issues a bulk copy about every 100 cycles whatever its size, and the
// twelve copies of 1.5 to 4 KB per K-step of a plane-by-plane layout were the
// 1190 cycles that a K-step of 48 columns took.)
// G_s between strings that differ by more than two replacements is zero, and
// strings in address order share their high orbitals: of the K-steps of a
// 96-row block of G, 9 % (CAS(14,14)) and 33 % (CAS(16,16)) hold only zeros.
// B keeps the others, with their list per block; rows of G as the narrow side
// of the tile skip more than as the 128-row side.
// NB = 96 where the tiles fill the chip: the digit products run as MMAs of N =
// 192 (two digits stacked along N, writing two neighbouring weights) or 96;
// 575 cycles per K-step and 48 columns against 730 to 800 for NB = 48 (an M =
// 128 MMA reads its 4 KB of A each time, so narrow ones wait for shared
// memory).  The five accumulators of 96 columns fill tensor memory once, so
// the next flush group cannot simply alternate buffers: the epilogue releases
// weight by weight, last first, and the first three K-steps of a group are
// issued weight by weight in that order (the eleven products of weights 4 and
// 5 first), which hides the read-out.  NB = 16 for small spaces, where 96-row
// tiles would leave most SMs idle.
// G_s's planes are built once at fci_init; C's two plane sets per call.
//
// sigma_1 + sigma_2 with their passes over C: CAS(14,14) 3.74 -> 2.59 ms,
// CAS(16,16) 179 -> 82 ms.  At CAS(16,16) the product runs at 1500 TFLOP/s of
// executed MMA work (cuBLAS sustains 1705 there, at the power cap); at CAS(14,14)
// its 972 tiles are 6.4 waves of 152.
#include <algorithm>
#include <vector>

#include "sliced_mma.cuh"

namespace fci {
namespace ss {

using sl::kSlices;
using tc::kM;
using sm::bulk_g2s;
using sm::mbar_expect_tx;

constexpr int kKTile = 16;           // K-steps (256 terms) per accumulator flush
constexpr int kLead = 3;             // K-steps of a flush group issued weight by weight
constexpr int kLevels = 5;
constexpr int kF = 34;               // integer unit 2^-34 of the accumulator scale
constexpr uint32_t kBytesA = 6 * 4096;

// Tile shape of NB rows of G: stages of operands in flight, epilogue warps per
// lane quarter, weights per MMA (N = kWide NB <= 256), tensor-memory columns.
template <int NB>
struct Shape {
    static constexpr uint32_t kBytesB = 6 * NB * 32;
    static constexpr uint32_t kStageBytes = kBytesA + kBytesB;
    static constexpr int kStages = NB == 96 ? 5 : 8;
    static constexpr int kSub = NB == 96 ? 3 : 1;
    static constexpr int kCols = NB / kSub;  // columns per epilogue thread
    static constexpr int kWide = NB == 96 ? 2 : 5;
    static constexpr int kEpiThreads = 128 * kSub;
    static constexpr int kThreads = 64 + kEpiThreads;  // warp 0 copies, warp 1 issues the MMAs
    static constexpr uint32_t kTmem = NB == 96 ? 512 : 128;
    static constexpr int kBars = 2 * kStages + 1 + kLevels + 1;  // full, free, acc_full, acc_empty[level], drain
    static constexpr uint32_t kSmem = kStages * kStageBytes + kBars * 8 + 16;
};

inline int64_t nblocks(int64_t rows, int nb) { return (rows + nb - 1) / nb; }
inline int64_t ksteps(int64_t k) { return (k + 15) / 16; }
inline size_t c_bytes(int64_t rows, int64_t k) { return (size_t)ksteps(k) * nblocks(rows, kM) * kBytesA; }

// byte offset of (row r, column kk) of a K-step inside one plane of a tile
__device__ __forceinline__ uint32_t core_offset(int r, int kk) {
    return (uint32_t)((r >> 3) * 256 + (kk >> 3) * 128 + (r & 7) * 16 + (kk & 7) * 2);
}

__device__ __forceinline__ long long fixed46(double x, int emax) {
    const unsigned long long b = __double_as_longlong(x);
    return sl::fixed47((uint32_t)b, (uint32_t)(b >> 32), emax + 1);
}

// largest biased exponent of the off-diagonal part of each row of the ELL
// same-spin Hamiltonian (slot 0 is the diagonal, applied separately)
__global__ void k_ss_rowexp(const double *__restrict__ gval, int64_t ns, int nsame, int *__restrict__ e) {
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= ns) return;
    unsigned m = 0;
    for (int k = 1; k < nsame; ++k)
        m = max(m, (unsigned)((__double_as_longlong(gval[(int64_t)k * ns + x]) >> 52) & 0x7FF));
    e[x] = (int)m;
}

// used[nb * nks + ks] = 1 for every K-step of every block of NB rows that holds
// an off-diagonal nonzero
__global__ void k_ss_used(const int32_t *__restrict__ gcol, const double *__restrict__ gval, int64_t ns, int nsame,
                          int NB, int64_t nks, unsigned char *__restrict__ used) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ns || t >= ns * (int64_t)nsame) return;  // slot 0 (t < ns): the diagonal
    if (gval[t] != 0.0) used[(t % ns) / NB * nks + (gcol[t] >> 4)] = 1;
}

// G planes: every off-diagonal ELL entry (row x, column gcol, value gval)
// scattered into the kept K-step slot[nb * nks + ks] (each row's columns are
// distinct; the planes start at zero)
__global__ void k_ss_gplanes(const int32_t *__restrict__ gcol, const double *__restrict__ gval, int64_t ns, int nsame,
                             const int *__restrict__ e, int NB, int64_t nks, const int *__restrict__ slot,
                             unsigned char *__restrict__ planes) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < ns || t >= ns * (int64_t)nsame) return;
    const int64_t x = t % ns;
    const double v = gval[t];
    if (v == 0.0) return;
    const int col = gcol[t];
    float f[kSlices];
    sl::digits6(fixed46(v, e[x]), f);
    unsigned char *tile = planes + (size_t)slot[x / NB * nks + (col >> 4)] * 6 * NB * 32;
    const uint32_t off = core_offset((int)(x % NB), col & 15);
#pragma unroll
    for (int s = 0; s < kSlices; ++s)  // exact: an 8-bit integer times a power of two
        *reinterpret_cast<__nv_bfloat16 *>(tile + s * NB * 32 + off) = __float2bfloat16_rn(f[s]);
}

// largest biased exponent of each row (erow) and each column (ecol) of the
// nrows x ncols matrix C, both from one coalesced pass: block (32, 8) over a
// 32 x 32 tile, integer atomicMax into erow / ecol (zeroed beforehand)
__global__ void k_ss_cexp(const double *__restrict__ C, int64_t nrows, int64_t ncols, int *__restrict__ erow,
                          int *__restrict__ ecol) {
    __shared__ unsigned colmax[8][32];
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    unsigned cm = 0;
    for (int i = 0; i < 4; ++i) {
        const int64_t r = (int64_t)blockIdx.y * 32 + threadIdx.y * 4 + i;
        unsigned e = 0;
        if (r < nrows && c < ncols) e = (unsigned)((__double_as_longlong(C[r * ncols + c]) >> 52) & 0x7FF);
        cm = max(cm, e);
        unsigned rm = e;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) rm = max(rm, __shfl_xor_sync(0xFFFFFFFFu, rm, o));
        if (threadIdx.x == 0 && r < nrows) atomicMax(erow + r, (int)rm);
    }
    colmax[threadIdx.y][threadIdx.x] = cm;
    __syncthreads();
    if (threadIdx.y == 0 && c < ncols) {
        unsigned m = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) m = max(m, colmax[k][threadIdx.x]);
        atomicMax(ecol + c, (int)m);
    }
}

// C's planes by rows (plane row = row of C, k = column; nullptr: not wanted) and
// by columns (plane row = column of C, k = row), both from one read of a 64 x 64
// tile of C through shared memory; 8 threads write the 128 bytes of 8 rows' core
// matrix.  Plane rows and columns past the matrix are written as zeros up to the
// ends of the 128-row tiles and K-steps (the grid covers them).
__global__ void __launch_bounds__(256) k_ss_cplanes(const double *__restrict__ C, int64_t nrows, int64_t ncols,
                                                    const int *__restrict__ erow, const int *__restrict__ ecol,
                                                    unsigned char *__restrict__ prow, unsigned char *__restrict__ pcol) {
    __shared__ double t[64][65];
    const int64_t c0 = (int64_t)blockIdx.x * 64, r0 = (int64_t)blockIdx.y * 64;
    for (int i = threadIdx.x; i < 64 * 64; i += 256) {
        const int64_t r = r0 + (i >> 6), c = c0 + (i & 63);
        t[i >> 6][i & 63] = (r < nrows && c < ncols) ? C[r * ncols + c] : 0.0;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < 1024; it += 256) {
        const bool cols = it >= 512;
        unsigned char *planes = cols ? pcol : prow;
        if (planes == nullptr) continue;
        const int x = it & 63, g = (it >> 6) & 7;  // plane row of the tile, group of 8 k
        const int64_t r = (cols ? c0 : r0) + x, k0 = (cols ? r0 : c0) + g * 8;
        const int64_t rows = cols ? ncols : nrows, klen = cols ? nrows : ncols;
        if (k0 >= (klen + 15) / 16 * 16 || r >= (rows + kM - 1) / kM * kM) continue;
        const int e = r < rows ? (cols ? ecol[r] : erow[r]) : 0;
        uint32_t w[kSlices][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float f0[kSlices], f1[kSlices];
            const int k = g * 8 + 2 * i;
            sl::digits6(fixed46(cols ? t[k][x] : t[x][k], e), f0);
            sl::digits6(fixed46(cols ? t[k + 1][x] : t[x][k + 1], e), f1);
#pragma unroll
            for (int s = 0; s < kSlices; ++s) w[s][i] = sl::pack_bf16(f0[s], f1[s]);
        }
        unsigned char *tile = planes + ((size_t)(k0 >> 4) * ((rows + kM - 1) / kM) + (r >> 7)) * kBytesA;
        const uint32_t off = core_offset((int)(r & 127), (int)(k0 & 15));
#pragma unroll
        for (int s = 0; s < kSlices; ++s)
            *reinterpret_cast<uint4 *>(tile + s * 4096 + off) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

struct SsArgs {
    const unsigned char *A, *B;  // plane sets
    const int *koff, *kidx;      // K-steps of row block nb of B: kidx[koff[nb] .. koff[nb + 1])
    int M, N;                    // rows of A (output lanes) and of B (output columns) in use
    const int *eA, *eB;          // biased exponent of each row
    double *out;
    int64_t sm, sn;              // out[m sm + n sn] +=
    const double *C;             // with it, out += (dn[n] + dm[m]) C at the same place first (dm may be null)
    const double *dn, *dm;
    int *err;
};

// value = V 2^(eA + eB - 12 - f), eA/eB the unbiased exponents of the row maxima
// (given biased); a non-finite operand row (exponent 0x7FF) gives NaN
__device__ __forceinline__ double element(long long V, int ea, int eb) {
    if (ea == 0x7FF || eb == 0x7FF) return __longlong_as_double(0x7FF8000000000000ll);
    return sl::scaled_i64(V, (ea - 1022) + (eb - 1022) - 12 - kF);
}

// The integer i of an FP32 value holding i 2^-k exactly, |i| <= 2^24, as
// 4 h + r with h = round(i / 4): both from magic-number additions, which are
// exact up to 2^22; no conversion instructions.
__device__ __forceinline__ int exact_int(float v, float quarter_scale, float unit) {
    constexpr float M = 12582912.0f;  // 1.5 2^23
    constexpr int MB = 0x4B400000;
    const float t = fmaf(v, quarter_scale, M);          // round(i / 4)
    const float r = fmaf(-(t - M), 4.0f * unit, v);     // (i - 4 h) 2^-k, exact
    const float u = fmaf(r, 4.0f * quarter_scale, M);   // i - 4 h
    return 4 * (__float_as_int(t) - MB) + (__float_as_int(u) - MB);
}

// Tiles: 128 rows of A x NB rows of B, t = nb * nmb + mb; CTA b takes tiles
// b, b + grid, ...  (the CTAs of one wave share A and B K-steps through L2,
// advancing through K at one rate).
template <int NB>
__global__ void __launch_bounds__(Shape<NB>::kThreads, 1) k_ss_tc(SsArgs P) {
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
    const uint32_t acc_full = bar0 + 8u * (uint32_t)(2 * kStages);
    auto acc_empty = [&](int lv) { return bar0 + 8u * (uint32_t)(2 * kStages + 1 + lv); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kStages + 1 + kLevels);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const bool elected = tc::elect_one();
    const int nmb = (P.M + 127) / 128, nnb = (P.N + NB - 1) / NB;
    const int ntiles = nmb * nnb;

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
        tc::mbar_init(acc_full, 1);
        for (int lv = 0; lv < kLevels; ++lv) tc::mbar_init(acc_empty(lv), S::kEpiThreads);
        tc::mbar_init(drain, 1);
        *s_fail = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tslot;

    int64_t G_copied = 0;
    if (warp == 0 && lane == 0) {
        // ---- copies: the A and B tiles of one K-step per stage ----
        int64_t &G = G_copied;
        for (int t = blockIdx.x; t < ntiles && !*s_fail; t += gridDim.x) {
            const int mb = t % nmb, nb = t / nmb;
            const int k1 = __ldg(P.koff + nb + 1);
            for (int k = __ldg(P.koff + nb); k < k1; ++k, ++G) {
                const int st = (int)(G % kStages);
                const size_t ks = (size_t)__ldg(P.kidx + k);
                if (G >= kStages && !tc::mbar_wait_bounded(freeb(st), (uint32_t)((G / kStages - 1) & 1))) {
                    *s_fail = 1;
                    break;
                }
                mbar_expect_tx(full(st), S::kStageBytes);
                const uint32_t dst = sbase + (uint32_t)st * S::kStageBytes;
                bulk_g2s(dst, P.A + (ks * nmb + mb) * kBytesA, kBytesA, full(st));
                bulk_g2s(dst + kBytesA, P.B + (size_t)k * S::kBytesB, S::kBytesB, full(st));
            }
        }
    } else if (warp == 1) {
        // ---- MMAs (all lanes run the loop, the elected one issues) ----
        const uint64_t a0 = tc::smem_desc(sbase, 128, 256), b0 = tc::smem_desc(sbase + kBytesA, 128, 256);
        auto A = [&](int st, int s) { return a0 + (uint64_t)((st * S::kStageBytes + s * 4096) >> 4); };
        auto B = [&](int st, int d) { return b0 + (uint64_t)((st * S::kStageBytes + d * NB * 32) >> 4); };
        int64_t G = 0, Tt = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const int nb = t / nmb;
            const int nk = __ldg(P.koff + nb + 1) - __ldg(P.koff + nb);
            for (int kt = 0; kt < nk && ok; kt += kKTile, ++Tt) {
                const int ke = min(nk - kt, kKTile), lead = min(ke, kLead);
                // the first K-steps of the group weight by weight, as the epilogue
                // releases the accumulators of the group before (weights 4 and 5
                // share one); each accumulator's first MMA overwrites it
#pragma unroll
                for (int lv = kLevels - 1; lv >= 0; --lv) {
                    if (ok && Tt >= 1 && !tc::mbar_wait_bounded(acc_empty(lv), (uint32_t)((Tt - 1) & 1))) ok = false;
                    for (int j = 0; j < lead && ok; ++j) {
                        const int st = (int)((G + j) % kStages);
                        if (lv == kLevels - 1 &&
                            !tc::mbar_wait_bounded(full(st), (uint32_t)(((G + j) / kStages) & 1))) {
                            ok = false;
                            break;
                        }
                        tc::fence_after();
                        if (!elected) continue;
#pragma unroll
                        for (int s = 0; s < kSlices; ++s) {
                            if (s <= lv)
                                tc::mma_bf16(tmem + lv * NB, A(st, s), B(st, lv - s), tc::instr_desc(kM, NB),
                                             (j == 0 && s == 0) ? 0u : 1u);
                            if (lv == kLevels - 1)
                                tc::mma_bf16(tmem + lv * NB, A(st, s), B(st, 5 - s), tc::instr_desc(kM, NB), 1u);
                        }
                        if (lv == 0) tc::mma_commit(freeb(st));
                    }
                }
                G += lead;
                // the others digit by digit of A, kWide weights per MMA
                for (int j = lead; j < ke && ok; ++j, ++G) {
                    const int st = (int)(G % kStages);
                    if (!tc::mbar_wait_bounded(full(st), (uint32_t)((G / kStages) & 1))) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    if (!elected) continue;
#pragma unroll
                    for (int s = 0; s < kSlices; ++s) {
#pragma unroll
                        for (int d = 0; d < kSlices; d += S::kWide)
                            if (s + d < kLevels) {
                                const int w = kLevels - s - d < S::kWide ? kLevels - s - d : S::kWide;
                                tc::mma_bf16(tmem + (s + d) * NB, A(st, s), B(st, d), tc::instr_desc(kM, w * NB), 1u);
                            }
                        tc::mma_bf16(tmem + (kLevels - 1) * NB, A(st, s), B(st, 5 - s), tc::instr_desc(kM, NB), 1u);
                    }
                    tc::mma_commit(freeb(st));
                }
                if (ok && elected) tc::mma_commit(acc_full);
            }
        }
        if (!ok) *s_fail = 1;
    } else if (warp >= 2) {
        // ---- epilogue: kSub warps per lane quarter (warp % 4); lane m of the
        // tile, columns kCols sub .. ----
        constexpr int kCols = S::kCols;
        const int quarter = warp & 3, sub = (warp - 2) >> 2;
        const int ml = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(sub * kCols);
        float top2 = 0.f, top3 = 0.f;
        int64_t Tt = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const int mb = t % nmb, nb = t / nmb;
            const int nk = __ldg(P.koff + nb + 1) - __ldg(P.koff + nb);
            const int m = mb * 128 + ml;
            long long acc[kCols];
#pragma unroll
            for (int j = 0; j < kCols; ++j) acc[j] = 0;
            for (int kt = 0; kt < nk; kt += kKTile, ++Tt) {
                if (!tc::mbar_wait_bounded(acc_full, (uint32_t)(Tt & 1))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                // weights 0-3 hold integers in units 2^-8L (|.| <= 2^20, 2^22, 2^23
                // and 3 2^22: top digits within +-64, others within +-128, 256
                // terms), weights 4 and 5 FP32 below 2^-6; units of the sum 2^-34
#pragma unroll
                for (int lv = kLevels - 1; lv >= 0; --lv)
#pragma unroll
                    for (int h = 0; h < kCols; h += 16) {
                        uint32_t r[16];
                        asm volatile(
                            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                              "=r"(r[14]), "=r"(r[15])
                            : "r"(lane_base + (uint32_t)(lv * NB + h)));
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        if (h + 16 >= kCols) {  // this weight is read: the next group may overwrite it
                            tc::fence_before();
                            tc::mbar_arrive(acc_empty(lv));
                        }
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            constexpr float M = 12582912.0f;
                            constexpr int MB = 0x4B400000;
                            const float v = __uint_as_float(r[j]);
                            if (lv == 4) {
                                const float t1 = fmaf(v, 262144.f, M);              // round(2^18 v)
                                const float q1 = fmaf(-(t1 - M), 0x1p-18f, v);      // exact rest
                                const float t2 = fmaf(q1, 0x1p34f, M);
                                acc[h + j] += (long long)((__float_as_int(t1) - MB) * 65536 + (__float_as_int(t2) - MB));
                            } else if (lv == 3) {
                                top3 = fmaxf(top3, fabsf(v));
                                acc[h + j] += (long long)exact_int(v, 0x1p22f, 0x1p-24f) << 10;
                            } else if (lv == 2) {
                                top2 = fmaxf(top2, fabsf(v));
                                acc[h + j] += (long long)exact_int(v, 0x1p14f, 0x1p-16f) << 18;
                            } else if (lv == 1) {
                                acc[h + j] += (long long)(__float_as_int(fmaf(v, 256.f, M)) - MB) << 26;
                            } else {
                                acc[h + j] += (long long)(__float_as_int(v + M) - MB) << 34;
                            }
                        }
                    }
            }
            if (!ok) break;
            // sigma_1's strides only (it carries no diagonal): with one beta string sigma_2
            // has sm = sn = 1 (asking for P.C == nullptr here costs 6 us a product at CAS(14,14))
            if (kCols == 32 && P.sn < P.sm) {
                // a thread holds consecutive columns of one row: transpose the warp's
                // 32 x 32 block so that its stores run along the row
#pragma unroll
                for (int d = kCols / 2; d > 0; d >>= 1)
#pragma unroll
                    for (int j = 0; j < kCols; ++j)
                        if (!(j & d)) {
                            const bool up = (lane & d) != 0;
                            const long long got = __shfl_xor_sync(0xFFFFFFFFu, up ? acc[j] : acc[j + d], d);
                            acc[j] = up ? got : acc[j];
                            acc[j + d] = up ? acc[j + d] : got;
                        }
                const int n = nb * NB + sub * kCols + lane, m0 = mb * 128 + quarter * 32;
                if (n < P.N) {
                    const int ebn = P.eB[n];
#pragma unroll
                    for (int j = 0; j < kCols; ++j)
                        if (m0 + j < P.M) {
                            const int eam = P.eA[m0 + j];
                            P.out[(m0 + j) * P.sm + n] += element(acc[j], eam, ebn);
                        }
                }
            } else if (m < P.M) {
                const int eam = P.eA[m];
                const double dm = P.dm ? P.dm[m] : 0.0;
#pragma unroll
                for (int j = 0; j < kCols; ++j) {
                    const int n = nb * NB + sub * kCols + j;
                    if (n < P.N) {
                        const double v = element(acc[j], eam, P.eB[n]);
                        double *o = P.out + m * P.sm + n * P.sn;
                        if (P.C)
                            *o = fma(P.dn[n] + dm, P.C[m * P.sm + n * P.sn], *o) + v;
                        else
                            *o += v;
                    }
                }
            }
        }
        if (!ok) *s_fail = 1;
        if (top2 > 256.f || top3 > 1.f) atomicOr(P.err, 2);  // beyond 2^24 units: not reached with these digits
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
    if (*s_fail && tid == 0) atomicOr(P.err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::kTmem) : "memory");
}

}  // namespace ss

// The dense path applies when both spins have replacements, no string space
// exceeds 16384 strings (the planes of G stay below 2 GB) and the context asks
// for it (fci_options.f64_same_spin).
bool sigma_ss_ok(const fci_ctx *ctx) { return ctx->ssGa.planes != nullptr; }

// Rows of G per tile: 96 where its tiles fill half of the chip, else 16.
static int tile_rows(int64_t M, int64_t N, int nsm) { return ss::nblocks(M, ss::kM) * ss::nblocks(N, 96) * 2 >= nsm ? 96 : 16; }

// The K-steps of every block of nb rows of G_s that hold a nonzero (every block
// keeps at least one), into O.lists, and on the device for each (block, K-step)
// its place in the planes, *slot (to be freed by the caller).
int ss_kstep_lists(fci_ctx *ctx, const SpinTables &T, int nb, SsOperand &O, int **slot, size_t *slot_bytes) {
    int rc = FCI_OK;
    cudaStream_t s = ctx->stream;
    const int64_t nks = ss::ksteps(T.ns), nnb = ss::nblocks(T.ns, nb);
    std::vector<unsigned char> used((size_t)(nnb * nks));
    std::vector<int> place(used.size(), 0), tab;
    O.nb = nb;
    O.nnb = (int)nnb;
    O.list_bytes = sizeof(int) * (size_t)(nnb + 1 + nnb * nks);
    O.lists = (int *)dalloc(ctx, O.list_bytes, &rc);  // koff [nnb + 1], kidx
    *slot_bytes = sizeof(int) * place.size();
    *slot = (int *)dalloc(ctx, *slot_bytes, &rc);
    if (rc) return rc;
    unsigned char *dused = reinterpret_cast<unsigned char *>(*slot);  // read back before the places go there
    FCI_CUDA(cudaMemsetAsync(dused, 0, used.size(), s));
    ss::k_ss_used<<<ceil_div(T.ns * (int64_t)T.nsame, 256), 256, 0, s>>>(T.gcol, T.gval, T.ns, T.nsame, nb, nks, dused);
    FCI_CUDA(cudaGetLastError());
    FCI_CUDA(cudaMemcpyAsync(used.data(), dused, used.size(), cudaMemcpyDeviceToHost, s));
    FCI_CUDA(cudaStreamSynchronize(s));
    std::vector<int> kidx;
    tab.push_back(0);
    for (int64_t b = 0; b < nnb; ++b) {
        for (int64_t k = 0; k < nks; ++k)
            if (used[b * nks + k] || (k == nks - 1 && (int)kidx.size() == tab.back())) {
                place[b * nks + k] = (int)kidx.size();
                kidx.push_back((int)k);
            }
        tab.push_back((int)kidx.size());
    }
    O.nsteps = kidx.size();
    tab.insert(tab.end(), kidx.begin(), kidx.end());
    FCI_CUDA(cudaMemcpyAsync(O.lists, tab.data(), sizeof(int) * tab.size(), cudaMemcpyHostToDevice, s));
    FCI_CUDA(cudaMemcpyAsync(*slot, place.data(), *slot_bytes, cudaMemcpyHostToDevice, s));
    FCI_CUDA(cudaStreamSynchronize(s));
    return FCI_OK;
}

int build_ss_tables(fci_ctx *ctx) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    if (ctx->opt.f64_same_spin == FCI_SS_FAMILY) return FCI_OK;
    if (A.nsingle == 0 || B.nsingle == 0 || A.ns > 16384 || B.ns > 16384) return FCI_OK;
    int rc = FCI_OK, nsm = 0;
    cudaStream_t s = ctx->stream;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    const bool shared = (&A == &B) || (A.gval == B.gval);
    auto build = [&](const SpinTables &T, int64_t M, SsOperand &O) -> int {
        const int nb = tile_rows(M, T.ns, nsm);
        int *slot = nullptr;
        size_t slot_bytes = 0;
        auto fill = [&]() -> int {
            if (int r = ss_kstep_lists(ctx, T, nb, O, &slot, &slot_bytes)) return r;
            O.plane_bytes = O.nsteps * (size_t)(6 * nb * 32);
            O.planes = (unsigned char *)dalloc(ctx, O.plane_bytes, &rc);
            O.e = (int *)dalloc(ctx, sizeof(int) * (size_t)T.ns, &rc);
            if (rc) return rc;
            FCI_CUDA(cudaMemsetAsync(O.planes, 0, O.plane_bytes, s));
            ss::k_ss_rowexp<<<ceil_div(T.ns, 256), 256, 0, s>>>(T.gval, T.ns, T.nsame, O.e);
            ss::k_ss_gplanes<<<ceil_div(T.ns * (int64_t)T.nsame, 256), 256, 0, s>>>(
                T.gcol, T.gval, T.ns, T.nsame, O.e, nb, ss::ksteps(T.ns), slot, O.planes);
            FCI_CUDA(cudaGetLastError());
            FCI_CUDA(cudaStreamSynchronize(s));
            return FCI_OK;
        };
        const int r = fill();
        dfree(ctx, slot, slot_bytes);
        return r;
    };
    if ((rc = build(A, B.ns, ctx->ssGa))) return rc;
    if (shared)
        ctx->ssGb = ctx->ssGa;
    else if ((rc = build(B, A.ns, ctx->ssGb)))
        return rc;
    // per-call workspace: C by rows (K = J_b) and by columns (K = J_a), and their exponents
    if ((rc = alloc_c_planes(ctx, ss::c_bytes(A.ns, B.ns), ss::c_bytes(B.ns, A.ns)))) return rc;
    ctx->ssEr = (int *)dalloc(ctx, sizeof(int) * (size_t)(A.ns + B.ns + 1), &rc);
    if (rc) return rc;
    ctx->ssEc = ctx->ssEr + A.ns;
    FCI_CUDA(opt_in_max_smem((const void *)ss::k_ss_tc<96>, ctx->device));
    FCI_CUDA(opt_in_max_smem((const void *)ss::k_ss_tc<16>, ctx->device));
    return FCI_OK;
}

// The operand planes of C by rows and by columns, shared by the FP64 and the FP32
// products (each call writes all of what it reads): made, or made larger.
int alloc_c_planes(fci_ctx *ctx, size_t row_bytes, size_t col_bytes) {
    if (int rc = grow_buffer(ctx, (void **)&ctx->ssCr, &ctx->ssCr_bytes, row_bytes)) return rc;
    return grow_buffer(ctx, (void **)&ctx->ssCc, &ctx->ssCc_bytes, col_bytes);
}

void free_c_planes(fci_ctx *ctx) {
    dfree(ctx, ctx->ssCr, ctx->ssCr_bytes);
    dfree(ctx, ctx->ssCc, ctx->ssCc_bytes);
    ctx->ssCr = ctx->ssCc = nullptr;
    ctx->ssCr_bytes = ctx->ssCc_bytes = 0;
}

void free_ss_operand(fci_ctx *ctx, SsOperand &O, int64_t ns) {
    dfree(ctx, O.planes, O.plane_bytes);
    dfree(ctx, O.lists, O.list_bytes);
    dfree(ctx, O.e, sizeof(int) * (size_t)ns);
    O = SsOperand{};
}

void free_ss_tables(fci_ctx *ctx) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    if (ctx->ssGb.lists != ctx->ssGa.lists) free_ss_operand(ctx, ctx->ssGb, B.ns);
    ctx->ssGb = SsOperand{};
    free_ss_operand(ctx, ctx->ssGa, A.ns);
    free_c_planes(ctx);
    dfree(ctx, ctx->ssEr, sizeof(int) * (size_t)(A.ns + B.ns + 1));
    ctx->ssEr = ctx->ssEc = nullptr;
}

// sigma += sigma_1 (which = 1), sigma_2 (which = 2) or both (which = 3), in that
// order, from the dense planes; sigma_2's pass also applies the diagonal of the
// alpha strings' Hamiltonian and, with sigma_1, of the beta strings'.
int launch_sigma_ss(fci_ctx *ctx, const double *C, double *sig, int which, cudaStream_t s, int rec, int slot) {
    const SpinTables &A = ctx->A, &B = ctx->B;
    const int64_t nsa = A.ns, nsb = B.ns;
    int nsm = 0;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    auto gemm = [&](const unsigned char *Ap, int64_t M, const int *eA, const SsOperand &O, int64_t N, int64_t sm, int64_t sn,
                    const double *dn, const double *dm) -> int {
        ss::SsArgs P;
        P.A = Ap;
        P.B = O.planes;
        P.koff = O.lists;
        P.kidx = O.lists + O.nnb + 1;
        P.M = (int)M;
        P.N = (int)N;
        P.eA = eA;
        P.eB = O.e;
        P.out = sig;
        P.sm = sm;
        P.sn = sn;
        P.C = dn ? C : nullptr;
        P.dn = dn;
        P.dm = dm;
        P.err = ctx->d_err;
        const unsigned grid = (unsigned)std::min<int64_t>(ss::nblocks(M, ss::kM) * O.nnb, nsm);
        if (O.nb == 96)
            ss::k_ss_tc<96><<<grid, ss::Shape<96>::kThreads, ss::Shape<96>::kSmem, s>>>(P);
        else
            ss::k_ss_tc<16><<<grid, ss::Shape<16>::kThreads, ss::Shape<16>::kSmem, s>>>(P);
        FCI_CUDA(cudaGetLastError());
        return FCI_OK;
    };
    // exponents of C's rows (I_a) and columns (I_b), then its planes
    FCI_CUDA(cudaMemsetAsync(ctx->ssEr, 0, sizeof(int) * (size_t)(nsa + nsb), s));
    ss::k_ss_cexp<<<dim3(ceil_div(nsb, 32), ceil_div(nsa, 32)), dim3(32, 8), 0, s>>>(C, nsa, nsb, ctx->ssEr, ctx->ssEc);
    FCI_CUDA(cudaGetLastError());
    ss::k_ss_cplanes<<<dim3(2 * ceil_div(nsb, ss::kM), 2 * ceil_div(nsa, ss::kM)), 256, 0, s>>>(
        C, nsa, nsb, ctx->ssEr, ctx->ssEc, which & 1 ? ctx->ssCr : nullptr, which & 2 ? ctx->ssCc : nullptr);
    FCI_CUDA(cudaGetLastError());
    if (which & 1) {  // sigma_1: A = C by rows (m = I_a), B = G_b (n = I_b), K = J_b
        if (int rc = gemm(ctx->ssCr, nsa, ctx->ssEr, ctx->ssGb, nsb, nsb, 1, nullptr, nullptr)) return rc;
        prof_mark(ctx, rec, slot, s);
        ++slot;
    }
    if (which & 2) {  // sigma_2: A = C by columns (m = I_b), B = G_a (n = I_a), K = J_a, and the diagonal
        if (int rc = gemm(ctx->ssCc, nsb, ctx->ssEc, ctx->ssGa, nsa, 1, nsb, A.gval, which & 1 ? B.gval : nullptr))
            return rc;
        prof_mark(ctx, rec, slot, s);
    }
    return FCI_OK;
}

}  // namespace fci
