// Spin-summed two-particle density Gamma_pqrs = <c| E_pq E_rs |c>, the
// density of the two-electron term of Eq. 6 (with gamma = <c|E_pq|c>,
// <c|H|c> = sum h_pq gamma_pq + 1/2 sum (pq|rs) (Gamma_pqrs - delta_qr gamma_ps)),
// the second half of the density step the paper runs after the Davidson
// iterations (Section 4, Table 2 "1e/2e Density Matrices").
//
// With the identity resolved over the determinants K of the space,
//   Gamma_pqrs = sum_K D_qp(K) D_rs(K),   D_rs(K) = <K| E_rs |c>.
// For K = (K_a, K_b), one entry a+_k a_l |K_a> = sign |T> of K_a's single-replacement list (Eq. 7)
// gives <K_a| a+_l a_k |T> = sign, that is D_lk(K) += sign c(T, K_b), and the
// entries of K_b's beta list D_lk(K) += sign c(K_a, T) (k == l entries: the
// occupation numbers).  One spin's entries of one determinant have distinct
// (l, k), so D needs no atomics: the alpha entries are stored, then the beta
// entries added.
//
// E_rs = (S_rs + A_rs) / 2 with S_rs = E_rs + E_sr symmetric and
// A_rs = E_rs - E_sr antisymmetric operators.  The mixed terms of the product,
// <S c|A c> = 1/2 <c|[S, A] c>, are commutators, so with the unitary group's
// [E_pq, E_rs] = d_qr E_ps - d_ps E_rq
//   4 Gamma_pqrs = <S_qp c|S_rs c> + <A_qp c|A_rs c> + 2 (d_qr gamma_ps - d_ps gamma_rq):
// two Gram matrices, of the n (n + 1) / 2 rows S c with one more row c (which gives
// gamma = <c|S c> / 2) and of the n (n - 1) / 2 rows A c, in place of one of all
// n^2 + 1 rows of D: about half the products.
//
// Both are dense contractions over all N determinants, run on the bf16 tensor
// cores with FP64 accuracy in the way of the sliced sigma kernels:
//  * c in fixed point relative to its largest power of two (|c| < 2^eD),
//    X = round(c 2^(45 - eD)); the rows' values are exact integer sums of these
//    (below 2^47, top digit in [-128, 128]), cut into six balanced 8-bit digits
//    that bf16 holds exactly;
//  * k_rdm2_fixed writes c's fixed-point integers once and k_rdm2_rows the pair
//    {l, k} of every replacement-list entry;
//  * k_rdm2_digits writes, per K-step of 16 determinants, the digit planes
//    D_0 .. D_5 and D_2 / 2 of both blocks' rows in the tensor cores' K-major
//    no-swizzle layout (8 x 8 core matrices of 128 bytes, 8-row groups 256 bytes
//    apart), a block's seven planes one after the other;
//  * k_rdm2_tc.  A Gram matrix is symmetric: D_i D_j^T is the transpose of
//    D_j D_i^T, so only the twelve products i <= j of the 21 with i + j <= 5 are
//    formed, over the whole square, and element (a, b) takes K_ab + K_ba (the
//    half plane gives the product 2, 2 the same weight).  A tile is 128 rows (the
//    MMA's M) x at most 80 columns; six accumulators: weights 0, 1, 2, 3 and 4 + 5
//    together, and the product 1, 1 of weight 2 by itself, since its element is
//    not doubled.  All but the last weights hold exact integers (at most 2^24 units
//    for the 512 determinants after which the epilogue reads them); the first MMAs of a
//    group overwrite, so nothing is reset.  The groups are fixed (K-steps 32j .. 32j +
//    31), each is accumulated in one order and their sum is taken in integers in units
//    2^-40 (the lowest product digit's), in registers and shared memory and at the end
//    of a work item by global integer adds in any order, so the result is the same bits
//    on every run and for every chunking;
//  * k_rdm2_finish combines the integers (the factor 4 included, so Gamma is rounded
//    once) and scales them to FP64.
// Left out are the digit products of weight >= 6 (below 2^-46 of the leading
// product) and c's fixed-point rounding (2^-46 of max |c|).  Products of a digit with
// itself do not cancel over the determinants, so the error grows with N max |c|^2: 1e-14
// to 3e-14 of it (measured, 63504 to 853776 determinants), 1e-10 of ||c||^2 for a CI vector
// at CAS(12,12), 4e-13 for a random one.
//
// CAS(12,12) (853,776 determinants): the whole call 3.04 ms before (one Gram matrix of
// D's rows in 128 x 48 tiles with all 21 products, twelve copies per K-step, 1 GiB of
// scratch), 1.34 ms now: digits 0.40, Gram 0.39 (MMAs 0.2, the rest the epilogue, which
// tensor memory lets overlap only in blocks of up to 42 columns), 0.23 for allocating
// and freeing the scratch (0.8 for 1 GiB), the rest launches, the small kernels and the
// copies to the host.  Converting each group of 512 to one integer in a unit set by
// ||c||^2 took the Gram kernel 0.61 ms and the call a round trip to the host.
#include "sliced_mma.cuh"

#include <algorithm>
#include <type_traits>

namespace fci {
namespace r2 {

using sl::kSlices;
using tc::kM;
using sm::bulk_g2s;
using sm::mbar_expect_tx;

constexpr int kThreads = 448;        // warp 0 copies, warp 1 issues the MMAs, warps 2-13 epilogue
constexpr int kEpiThreads = 384;
constexpr int kPlanes = 7;           // D_0 .. D_5, D_2 / 2
constexpr int kLv = 6;               // accumulators per tile: weights 0, 1, 2, 3, 4 + 5 and the product 1, 1
constexpr int kMaxBN = 80;           // columns per tile: kLv x 80 of the 512 tensor memory columns
constexpr int kKTile = 32;           // K-steps (512 determinants) per accumulator flush and work item
constexpr int kMaxStages = 10;       // K-steps of operands in flight
constexpr uint32_t kRing = 152u * 1024u;
constexpr int kEls = 32;             // elements per epilogue thread: 80 columns in chunks of 8 over 3 warps
constexpr uint32_t kRemBytes = kEls * kEpiThreads * 4;
constexpr uint32_t kSlack = 4096u;   // descriptors of the last rows reach past a plane (columns not read back)
constexpr int kBars = 2 * kMaxStages + 5;    // full[], free[], acc_full[2], acc_empty[2], drain
constexpr uint32_t kSmem = kRing + kSlack + kRemBytes + kBars * 8 + 16;
constexpr int kStatBlocks = 1024;
constexpr uint32_t kRowSwap = 0x4000u, kRowDiag = 0x8000u;

// Fixed point of c relative to the largest biased exponent emax of the vector:
// round(|x| 2^(45 - eD)) with the sign of x, |x| < 2^eD.
__device__ __forceinline__ long long fixed45(double x, int emax) {
    const unsigned long long b = __double_as_longlong(x);
    return sl::fixed47((uint32_t)b, (uint32_t)(b >> 32), emax + 2);
}
__device__ __forceinline__ long long fixed45(float x, int emax) {
    const uint32_t b = __float_as_uint(x);
    const int ex = (int)((b >> 23) & 0xFFu);
    const long long m = (long long)((b & 0x7FFFFFu) | (ex ? 0x800000u : 0u));
    // x = m 2^(max(ex,1) - 150), eD = emax - 126: X = m 2^(max(ex,1) - emax + 21)
    const int sh = (ex ? ex : 1) - emax + 21;
    long long X;
    if (sh >= 0)
        X = m << sh;  // sh <= 21 since ex <= emax
    else
        X = -sh > 30 ? 0ll : (m + (1ll << (-sh - 1))) >> -sh;
    return (b >> 31) ? -X : X;
}

template <typename T>
__device__ __forceinline__ unsigned biased_exponent(T x);
template <>
__device__ __forceinline__ unsigned biased_exponent<double>(double x) {
    return (unsigned)((__double_as_longlong(x) >> 52) & 0x7FF);
}
template <>
__device__ __forceinline__ unsigned biased_exponent<float>(float x) {
    return (__float_as_uint(x) >> 23) & 0xFFu;
}

// Largest biased exponent of c (atomicMax).
template <typename T>
__global__ void __launch_bounds__(256) k_rdm2_stats(const T *__restrict__ c, int64_t n, int *__restrict__ emax) {
    unsigned mx = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        mx = max(mx, biased_exponent<T>(__ldg(c + i)));
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(emax, (int)mx);
}

// (l, k) of the entry a+_k a_l |x> = sign |t> (x, t bitmasks; pair index p of {k, l})
__device__ __forceinline__ void entry_orbitals(uint32_t x, uint32_t t, uint32_t p, int &l, int &k) {
    if (x != t) {
        l = __ffs(x & ~t) - 1;
        k = __ffs(t & ~x) - 1;
    } else {  // k == l: pair index l (l + 1) / 2 + l
        int o = 0;
        while ((uint32_t)(o * (o + 3) / 2) < p) ++o;
        l = k = o;
    }
}

// c in fixed point, once per call: Xc[i] = round(c_i 2^(45 - eD)); zero where no
// value is a normal number.
template <typename T>
__global__ void k_rdm2_fixed(const T *__restrict__ c, int64_t n, const int *__restrict__ d_emax,
                             long long *__restrict__ Xc) {
    const int emax = *d_emax;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) Xc[i] = emax > 0 ? fixed45(c[i], emax) : 0;
}

// rows[e * ns + x] = the pair {l, k} (max (max + 1) / 2 + min) that the entry a+_k a_l |x> =
// sign |target> of string x feeds, with kRowSwap where l < k and kRowDiag where l = k;
// entry-major like SpinTables::tab.
__global__ void k_rdm2_rows(SpinTables S, uint16_t *__restrict__ rows) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= S.ns * (int64_t)S.nsingle) return;
    const uint32_t ent = S.tab[t];
    int l, k;
    entry_orbitals(S.str[t % S.ns], S.str[ent_target(ent)], ent_pair(ent), l, k);
    const int i = max(l, k), j = min(l, k);
    rows[t] = (uint16_t)((uint32_t)(i * (i + 1) / 2 + j) | (l < k ? kRowSwap : 0u) | (l == k ? kRowDiag : 0u));
}

// One Gram matrix: R rows (Rd with padding, a multiple of 16), tiles of 128 rows x
// NB columns.  Up to 128 rows the seven planes of a K-step are staged whole by one
// bulk copy (an SM issues such a copy every hundred cycles whatever its size; the
// kernel before, with twelve copies per K-step, was bound by them), and a tile takes
// its operand rows from there; above that a tile copies its rows of each plane.
struct Block {
    int R, Rd, NB, nct, nrb;
    int whole;       // planes staged whole
    uint32_t bytes;  // staged per K-step
    // rows of a staged plane of the A / B operand
    __host__ __device__ uint32_t planeA() const { return (whole ? Rd : 128) * 32u; }
    __host__ __device__ uint32_t planeB() const { return (whole ? Rd : NB) * 32u; }
    __host__ __device__ uint32_t offB() const { return whole ? 0u : 3u * 128u * 32u; }
};

static Block make_block(int R) {
    Block b{};
    b.R = R;
    if (R <= 0) return b;
    b.Rd = (R + 15) / 16 * 16;
    b.nct = (b.Rd + kMaxBN - 1) / kMaxBN;
    b.NB = ((b.Rd + b.nct - 1) / b.nct + 15) / 16 * 16;
    b.nrb = (b.Rd + 127) / 128;
    b.whole = b.Rd <= 128;
    b.bytes = b.whole ? kPlanes * b.planeA() : 3u * b.planeA() + kPlanes * b.planeB();
    return b;
}

// 64-bit words of one determinant's rows S, c and A in k_rdm2_digits
__host__ __device__ inline int row_stride(int n) { return (n * (n + 1) + 1) | 1; }

// One block per K-step of 16 determinants: the integers of the rows S_ij (i >= j), c
// and A_ij (stored under the same pair index) in shared memory, then the seven
// planes of both blocks into dg (K-step ks - ks0 of the chunk): row r, determinant kk
// of the K-step of a plane at (r/8) 256 + (kk/8) 128 + (r%8) 16 + (kk%8) 2.  A
// replacement (l, k) needs l occupied and k empty, so one spin's entries of one
// determinant have distinct pairs {l, k} and S and A are stored and added to as D
// was; the determinant-major layout with an odd stride spreads the 16 determinants
// of one entry, and the consecutive rows of the digit pass, over the banks.  The
// loads of a thread's list entries are issued together (a block's time is their
// latency, twice: entry, then c).
__global__ void __launch_bounds__(256) k_rdm2_digits(const long long *__restrict__ Xc, SpinTables A, SpinTables B,
                                                     const uint16_t *__restrict__ rows_a,
                                                     const uint16_t *__restrict__ rows_b, int n, Block bs, Block ba,
                                                     int64_t ks0, int64_t N, uint4 *__restrict__ dg) {
    extern __shared__ __align__(16) long long X[];  // [16][row_stride(n)]
    const int npair = n * (n + 1) / 2, offA = npair + 1, Rs = row_stride(n);
    const int64_t ks = ks0 + blockIdx.x;
    const int64_t nsb = B.ns;
    const int tid = threadIdx.x, kk = tid & 15;
    const int64_t K = ks * 16 + kk;
    const bool in = K < N;
    const int64_t ka = !in ? 0 : N <= 0xFFFFFFFFll ? (int64_t)((uint32_t)K / (uint32_t)nsb) : K / nsb, kb = in ? K - ka * nsb : 0;
    long long *Xk = X + kk * Rs;
    for (int i = tid; i < Rs * 16; i += blockDim.x) X[i] = 0;
    __syncthreads();
    constexpr int kBatch = 3;  // 16 entries per block pass
    // alpha entries stored, then beta entries added
    auto entries = [&](auto first, const SpinTables &S, const uint16_t *rows, int64_t x, const long long *src,
                       int64_t stride) {
        for (int e0 = tid >> 4; e0 < S.nsingle; e0 += 16 * kBatch) {
            uint32_t ent[kBatch];
            uint32_t row[kBatch];
            long long v[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const bool ok = in && e0 + 16 * u < S.nsingle;
                const int64_t at = (int64_t)(e0 + 16 * u) * S.ns + x;
                ent[u] = ok ? __ldg(S.tab + at) : 0u;
                row[u] = ok ? (uint32_t)__ldg(rows + at) : ~0u;
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) v[u] = row[u] != ~0u ? __ldg(src + (int64_t)ent_target(ent[u]) * stride) : 0;
#pragma unroll
            for (int u = 0; u < kBatch; ++u)
                if (row[u] != ~0u) {
                    const long long d = ent_negative(ent[u]) ? -v[u] : v[u];
                    long long *q = Xk + (row[u] & 0x3FFFu);
                    const long long sv = (row[u] & kRowDiag) ? 2 * d : d, av = (row[u] & kRowSwap) ? -d : d;
                    if (first) {
                        q[0] = sv;
                        q[offA] = av;
                    } else {
                        q[0] += sv;
                        q[offA] += av;
                    }
                }
        }
    };
    entries(std::true_type{}, A, rows_a, ka, Xc + kb, nsb);
    if (tid < 16 && in) Xk[npair] = Xc[K];
    __syncthreads();
    entries(std::false_type{}, B, rows_b, kb, Xc + ka * nsb, 1);
    __syncthreads();
    // digits: item (r/8) 16 + g 8 + r%8 of a block owns 16 bytes at 16 x item of each plane
    uint4 *out = dg + (ks - ks0) * kPlanes * (int64_t)(bs.Rd + ba.Rd) * 2;
    for (int it = tid; it < (bs.Rd + ba.Rd) * 2; it += blockDim.x) {
        const bool anti = it >= bs.Rd * 2;
        const int item = anti ? it - bs.Rd * 2 : it;
        const int Rd = anti ? ba.Rd : bs.Rd, R = anti ? ba.R : bs.R;
        const int r = (item >> 4) * 8 + (item & 7), g = (item >> 3) & 1;
        int at = r;
        if (anti) {  // r = i (i - 1) / 2 + j, i > j: the pair index is r + i
            int i = (int)((sqrtf(8.f * (float)r + 1.f) + 1.f) * 0.5f);
            while (i * (i - 1) / 2 > r) --i;
            while (i * (i + 1) / 2 <= r) ++i;
            at = offA + r + i;
        }
        const long long *x = X + g * 8 * Rs + at;
        uint32_t w[kPlanes][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            float f0[kSlices], f1[kSlices];
            sl::digits6(r < R ? x[2 * u * Rs] : 0, f0);
            sl::digits6(r < R ? x[(2 * u + 1) * Rs] : 0, f1);
#pragma unroll
            for (int s = 0; s < kSlices; ++s) w[s][u] = sl::pack_bf16(f0[s], f1[s]);
            w[6][u] = sl::pack_bf16(0.5f * f0[2], 0.5f * f1[2]);
        }
        uint4 *o = out + (anti ? kPlanes * (int64_t)bs.Rd * 2 : 0) + item;
#pragma unroll
        for (int s = 0; s < kPlanes; ++s) o[(int64_t)s * Rd * 2] = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

struct TcArgs {
    const unsigned char *dg;  // digit planes of the chunk
    int64_t nks, step;        // K-steps in the chunk, bytes of one
    Block blk[2];             // S and A
    int ntile;
    unsigned long long *G;    // per block [Rd][Rd][2] words, element a <= b at b Rd + a; S first
    int *err;
};

// Tile t: block, row block rb (128 rows), column block cb (NB columns).
struct Tile {
    const Block *b;
    int anti, rb, cb;
    __device__ Tile(const TcArgs &P, int t) {
        const int ns = P.blk[0].nrb * P.blk[0].nct;
        anti = t >= ns;
        if (anti) t -= ns;
        b = &P.blk[anti];
        rb = t / b->nct;
        cb = t - rb * b->nct;
    }
};

// Work of CTA b: with at least ntile CTAs (a multiple of ntile), CTA b keeps
// tile b % ntile for the whole launch and takes the K-ranges g, g + ng, ...
// (g = b / ntile, ng = grid / ntile), so that its sums stay in registers and
// the ntile CTAs of a group read each K-range at about the same time; with
// fewer CTAs than tiles, CTA b takes tiles b, b + grid, ... over every K-range.
struct Work {
    int t0, tstep, g, ng;
    __device__ Work(int ntile) {
        if ((int)gridDim.x >= ntile) {
            t0 = blockIdx.x % ntile;
            tstep = ntile;
            g = blockIdx.x / ntile;
            ng = gridDim.x / ntile;
        } else {
            t0 = blockIdx.x;
            tstep = gridDim.x;
            g = 0;
            ng = 1;
        }
    }
};

__global__ void __launch_bounds__(kThreads, 1) k_rdm2_tc(const __grid_constant__ TcArgs P) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kRing + kSlack + kRemBytes);
    volatile int *s_fail = reinterpret_cast<volatile int *>(smem + kRing + kSlack + kRemBytes + kBars * 8);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + kRing + kSlack + kRemBytes + kBars * 8 + 4);
    const uint32_t sbase = tc::smem_u32(smem);
    const uint32_t bar0 = tc::smem_u32(bars);
    auto full = [&](int st) { return bar0 + 8u * (uint32_t)st; };
    auto freeb = [&](int st) { return bar0 + 8u * (uint32_t)(kMaxStages + st); };
    auto acc_full = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + b); };
    auto acc_empty = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kMaxStages + 2 + b); };
    const uint32_t drain = bar0 + 8u * (uint32_t)(2 * kMaxStages + 4);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const bool elected = tc::elect_one();
    const int64_t nkr = (P.nks + kKTile - 1) / kKTile;
    const Work W(P.ntile);
    // one ring and one accumulator count for both blocks: a CTA with several tiles
    // keeps its stages and barrier phases
    const uint32_t stage = max(P.blk[0].bytes, P.blk[1].bytes);
    const int nst = min(kMaxStages, (int)(kRing / stage));
    const int nbuf = kLv * P.blk[0].NB <= 256 && kLv * P.blk[1].NB <= 256 ? 2 : 1;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < nst; ++i) {
            tc::mbar_init(full(i), 1);
            tc::mbar_init(freeb(i), 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(acc_full(b), 1);
            tc::mbar_init(acc_empty(b), kEpiThreads);
        }
        tc::mbar_init(drain, 1);
        *s_fail = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tslot;

    int64_t G_copied = 0;  // K-steps whose copies warp 0 issued
    if (warp == 0) {
        // ---- copies: one K-step per stage ----
        int64_t &G = G_copied;
        bool ok = true;
        for (int t = W.t0; t < P.ntile && ok; t += W.tstep) {
            const Tile T(P, t);
            const Block &b = *T.b;
            const size_t blk_off = T.anti ? (size_t)kPlanes * P.blk[0].Rd * 32 : 0;
            const uint32_t ra = (uint32_t)min(128, b.Rd - T.rb * 128) * 32u;
            const uint32_t rc = (uint32_t)min(b.NB, b.Rd - T.cb * b.NB) * 32u;
            for (int64_t kr = W.g; kr < nkr && ok; kr += W.ng) {
                const int64_t k1 = min(P.nks, (kr + 1) * kKTile);
                for (int64_t ks = kr * kKTile; ks < k1; ++ks, ++G) {
                    const int st = (int)(G % nst);
                    if (G >= nst && !tc::mbar_wait_bounded(freeb(st), (uint32_t)((G / nst - 1) & 1))) {
                        ok = false;
                        break;
                    }
                    if (!elected) continue;
                    const unsigned char *src = P.dg + (size_t)ks * P.step + blk_off;
                    const uint32_t dst = sbase + (uint32_t)st * stage;
                    if (b.whole) {
                        mbar_expect_tx(full(st), b.bytes);
                        bulk_g2s(dst, src, b.bytes, full(st));
                    } else {
                        mbar_expect_tx(full(st), 3u * ra + kPlanes * rc);
                        for (int p = 0; p < 3; ++p)
                            bulk_g2s(dst + (uint32_t)p * b.planeA(), src + ((size_t)p * b.Rd + T.rb * 128) * 32, ra, full(st));
                        for (int p = 0; p < kPlanes; ++p)
                            bulk_g2s(dst + b.offB() + (uint32_t)p * b.planeB(),
                                     src + ((size_t)p * b.Rd + T.cb * b.NB) * 32, rc, full(st));
                    }
                }
            }
        }
        if (!ok) *s_fail = 1;
    } else if (warp == 1) {
        // ---- MMAs (all lanes run the loop, the elected one issues) ----
        int64_t G = 0, Tt = 0;
        bool ok = true;
        for (int t = W.t0; t < P.ntile && ok; t += W.tstep) {
            const Tile T(P, t);
            const Block &b = *T.b;
            const bool stacked = b.planeB() == (uint32_t)b.NB * 32u;  // the planes' columns adjoin
            const uint32_t pa = b.planeA() >> 4, pb = b.planeB() >> 4, nb = (uint32_t)b.NB;
            const uint64_t ad = tc::smem_desc(sbase, 128, 256);  // one row block when whole
            const uint64_t bd = tc::smem_desc(sbase + b.offB() + (b.whole ? (uint32_t)T.cb * nb * 32u : 0u), 128, 256);
            const uint32_t id1 = tc::instr_desc(kM, b.NB), id2 = tc::instr_desc(kM, 2 * b.NB),
                           id3 = tc::instr_desc(kM, 3 * b.NB);
            for (int64_t kr = W.g; kr < nkr && ok; kr += W.ng, ++Tt) {
                const int buf = nbuf == 2 ? (int)(Tt & 1) : 0;
                const int64_t k0 = kr * kKTile, k1 = min(P.nks, k0 + kKTile);
                if (Tt >= nbuf && !tc::mbar_wait_bounded(acc_empty(buf), (uint32_t)(((Tt - nbuf) / nbuf) & 1))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                const uint32_t acc = tmem + (uint32_t)buf * 256u;
                for (int64_t ks = k0; ks < k1; ++ks, ++G) {
                    const int st = (int)(G % nst);
                    if (!tc::mbar_wait_bounded(full(st), (uint32_t)((G / nst) & 1))) {
                        ok = false;
                        break;
                    }
                    tc::fence_after();
                    if (!elected) continue;
                    const uint64_t so = (uint64_t)(((uint32_t)st * stage) >> 4);
                    const uint64_t a = ad + so, d = bd + so;
                    const uint32_t on = ks == k0 ? 0u : 1u;  // the first products overwrite
                    // accumulators 0-3: weights 0-3, 4: weights 4 and 5, 5: the product 1, 1
                    if (stacked) {
                        tc::mma_bf16(acc, a, d, id3, on);
                        tc::mma_bf16(acc + 3 * nb, a, d + 3 * pb, id2, on);
                        tc::mma_bf16(acc + 5 * nb, a + pa, d + pb, id1, on);
                        tc::mma_bf16(acc + 3 * nb, a + pa, d + 2 * pb, id2, 1u);
                    } else {
#pragma unroll
                        for (uint32_t j = 0; j < 5; ++j) tc::mma_bf16(acc + j * nb, a, d + j * pb, id1, on);
                        tc::mma_bf16(acc + 5 * nb, a + pa, d + pb, id1, on);
                        tc::mma_bf16(acc + 3 * nb, a + pa, d + 2 * pb, id1, 1u);
                        tc::mma_bf16(acc + 4 * nb, a + pa, d + 3 * pb, id1, 1u);
                    }
                    tc::mma_bf16(acc + 4 * nb, a, d + 5 * pb, id1, 1u);
                    tc::mma_bf16(acc + 4 * nb, a + pa, d + 4 * pb, id1, 1u);
                    tc::mma_bf16(acc + 4 * nb, a + 2 * pa, d + 6 * pb, id1, 1u);
                    tc::mma_bf16(acc + 4 * nb, a + 2 * pa, d + 3 * pb, id1, 1u);
                    tc::mma_commit(freeb(st));
                }
                if (!ok) break;
                if (elected) tc::mma_commit(acc_full(buf));
            }
        }
        if (!ok) *s_fail = 1;
    } else {
        // ---- epilogue: three warps per lane quarter (warp % 4); lane m of the
        // tile, column chunks of 8 sub, sub + 3, ... ----
        const int quarter = warp & 3, sub = (warp - 2) >> 2;
        const int m = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        constexpr int kChunks = kEls / 8;
        // Sums of this thread's elements, exact: units 2^-24 in registers, the rest of
        // the FP32 weights in units 2^-40 (below 2^15 a group) in shared memory.
        int *rem = reinterpret_cast<int *>(smem + kRing + kSlack) + (tid - 64);
        bool range_bad = false;
        int64_t Tt = 0;
        bool ok = true;
        for (int t = W.t0; t < P.ntile && ok; t += W.tstep) {
            const Tile T(P, t);
            const Block &b = *T.b;
            const int row = T.rb * 128 + m, col0 = T.cb * b.NB;
            const int nc = min(b.NB, b.R - col0);  // columns read back (may be <= 0)
            long long acc[kChunks][8];
            auto clear = [&]() {
#pragma unroll
                for (int h = 0; h < kChunks; ++h)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        acc[h][j] = 0;
                        rem[(h * 8 + j) * kEpiThreads] = 0;
                    }
            };
            // adds acc 2^16 + rem (units 2^-40) to the element's words hi 2^32 + lo: lo below
            // 2^33 a flush, hi below 2^56 in all for up to 2^33 determinants
            auto flush = [&]() {
                unsigned long long *Gb = P.G + (T.anti ? (size_t)2 * P.blk[0].Rd * P.blk[0].Rd : 0);
                int c0 = sub * 8, rd = b.Rd;
                asm volatile("" : "+r"(c0), "+r"(rd));
#pragma unroll
                for (int h = 0; h < kChunks; ++h)
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int c = c0 + 24 * h + j, col = col0 + c;
                        if (row >= b.R || c >= nc) continue;
                        unsigned long long *g = Gb + 2 * (max(row, col) * rd + min(row, col));
                        const long long lo = ((acc[h][j] & 0xFFFFll) << 16) + rem[(h * 8 + j) * kEpiThreads];
                        atomicAdd(g, (unsigned long long)(acc[h][j] >> 16));
                        atomicAdd(g + 1, (unsigned long long)lo);
                    }
            };
            clear();
            const bool rows_live = T.rb * 128 + quarter * 32 < b.R;  // uniform in the warp
            int groups = 0;
            for (int64_t kr = W.g; kr < nkr; kr += W.ng, ++Tt) {
                const int buf = nbuf == 2 ? (int)(Tt & 1) : 0;
                if (!tc::mbar_wait_bounded(acc_full(buf), (uint32_t)((Tt / nbuf) & 1))) {
                    ok = false;
                    break;
                }
                tc::fence_after();
                if (rows_live) {
                    // opaque, or the comparisons of all 32 elements are kept in registers
                    int above = row - col0, ncols = row < b.R ? nc : 0;
                    asm volatile("" : "+r"(above), "+r"(ncols));
#pragma unroll
                    for (int h = 0; h < 2 * kChunks; ++h) {  // halves of chunks: 24 registers in flight
                        const int c = (sub + 3 * (h >> 1)) * 8 + 4 * (h & 1);
                        if (c >= nc) continue;
                        uint32_t r[kLv][4];
#pragma unroll
                        for (int lv = 0; lv < kLv; ++lv)
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                         : "=r"(r[lv][0]), "=r"(r[lv][1]), "=r"(r[lv][2]), "=r"(r[lv][3])
                                         : "r"(lane_base + (uint32_t)(buf * 256 + lv * b.NB + c)));
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            // symmetric products count once per pair (a, b), the others in both
                            // orders: K_ab here, K_ba by the thread of (b, a), twice on the diagonal
                            const bool live = c + j < ncols, once = above <= c + j;
                            const int tw = above == c + j ? 2 : 1;
                            const float v2 = __uint_as_float(r[2][j]), v3 = __uint_as_float(r[3][j]),
                                        d2 = __uint_as_float(r[5][j]), v4 = __uint_as_float(r[4][j]);
                            range_bad |= live && !(fmaxf(fmaxf(fabsf(v2), fabsf(d2)), 256.f * fabsf(v3)) <= 256.f);
                            constexpr float M = 12582912.0f;  // 1.5 2^23
                            constexpr int MB = 0x4B400000;
                            const float t1 = fmaf(v4, 0x1p24f, M);            // round(2^24 v4), |v4| < 2^-7
                            const float q = fmaf(-(t1 - M), 0x1p-24f, v4);    // exact
                            const int h2 = __float_as_int(fmaf(q, 0x1p40f, M)) - MB;
                            const int i1 = __float2int_rn(__uint_as_float(r[1][j]) * 256.f);
                            const int i2 = __float2int_rn(v2 * 65536.f);
                            const int i3 = __float2int_rn(v3 * 16777216.f) + (__float_as_int(t1) - MB);
                            const int i0 = once ? __float2int_rn(__uint_as_float(r[0][j])) : 0;
                            const int id = once ? __float2int_rn(d2 * 65536.f) : 0;
                            acc[h >> 1][4 * (h & 1) + j] += (long long)i0 * 16777216 + (long long)(tw * i1) * 65536 +
                                         (long long)(tw * i2 + id) * 256 + tw * i3;
                            rem[(h * 4 + j) * kEpiThreads] += tw * h2;
                        }
                    }
                }
                tc::fence_before();
                tc::mbar_arrive(acc_empty(buf));
                if (++groups == 4096 || kr + W.ng >= nkr) {  // |acc| < 2^49 a group, |rem| <= 2^16
                    flush();
                    clear();
                    groups = 0;
                }
            }
        }
        if (!ok) *s_fail = 1;
        if (range_bad) atomicOr(P.err, 2);
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
    if (warp == 0) {  // at once unless a wait gave up
        for (int st = 0; st < nst; ++st) {
            const int64_t fills = G_copied / nst + (st < G_copied % nst ? 1 : 0);
            if (fills > 0 && !tc::mbar_wait_bounded(full(st), (uint32_t)((fills - 1) & 1))) *s_fail = 1;
        }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (*s_fail && tid == 0) atomicOr(P.err, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// T 2^e2 as FP64, rounded to nearest even (results below the normal range flush to
// zero): the leading 63 bits, the rest as a sticky bit.
__device__ __forceinline__ double scaled_i128(__int128 T, int e2) {
    const bool neg = T < 0;
    unsigned __int128 m = neg ? -(unsigned __int128)T : (unsigned __int128)T;
    const unsigned long long hi = (unsigned long long)(m >> 62);
    if (hi) {
        const int sh = 64 - __clzll((long long)hi);
        const bool sticky = (m & (((unsigned __int128)1 << sh) - 1)) != 0;
        m >>= sh;
        m |= sticky ? 1u : 0u;
        e2 += sh;
    }
    const long long v = (long long)m;
    return sl::scaled_i64(neg ? -v : v, e2);
}

// 4 Gamma[p][q][r][s] = <S_qp|S_rs> + <A_qp|A_rs> + d_qr <c|S_ps> - d_ps <c|S_rq> and
// 2 gamma[p][q] = <c|S_pq> from the integers (element (a, b) read at a <= b), in units
// 2^(2 eD - 50), eD = emax - bias; NaN everywhere when c held a non-finite value
// (emax >= inf).
__global__ void k_rdm2_finish(const unsigned long long *__restrict__ G, int RdS, int RdA, int n,
                              const int *__restrict__ d_emax, int bias, int inf, double *__restrict__ g2,
                              double *__restrict__ g1) {
    const int64_t n2 = (int64_t)n * n, n4 = n2 * n2;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n4 + n2) return;
    const int emax = *d_emax, e2 = 2 * (emax - bias) - 50;
    const unsigned long long *GA = G + (size_t)2 * RdS * RdS;
    const int crow = n * (n + 1) / 2;
    auto sidx = [](int a, int b) { return a > b ? a * (a + 1) / 2 + b : b * (b + 1) / 2 + a; };
    auto aidx = [](int a, int b) { return a > b ? a * (a - 1) / 2 + b : b * (b - 1) / 2 + a; };
    auto at = [](const unsigned long long *M, int Rd, int a, int b) {
        const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(M + 2 * ((size_t)max(a, b) * Rd + min(a, b)));
        return (__int128)(long long)w.x * ((__int128)1 << 32) + (long long)w.y;
    };
    auto cS = [&](int a, int b) { return at(G, RdS, crow, sidx(a, b)); };
    double v;
    if (i < n4) {
        const int p = (int)(i / (n2 * n)), q = (int)((i / n2) % n), r = (int)(i / n % n), s = (int)(i % n);
        __int128 x = at(G, RdS, sidx(q, p), sidx(r, s));
        if (q != p && r != s) {
            const __int128 y = at(GA, RdA, aidx(q, p), aidx(r, s));
            x += (q > p) == (r > s) ? y : -y;
        }
        if (q == r) x += cS(p, s);
        if (p == s) x -= cS(r, q);
        v = scaled_i128(x, e2 - 2);
    } else {
        const int p = (int)((i - n4) / n), q = (int)((i - n4) % n);
        v = scaled_i128(cS(p, q), e2 - 1);
    }
    if (emax >= inf) v = __longlong_as_double(0x7FF8000000000000ll);
    if (i < n4)
        g2[i] = v;
    else
        g1[i - n4] = v;
}

// Digit planes of one chunk when the caller names no size.
constexpr size_t kDefaultChunk = (size_t)256 << 20;

inline unsigned grid_blocks(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16); }

template <typename T>
int rdm2_impl(fci_ctx *ctx, const T *C, double *g1_host, double *g2_host) {
    const int n = ctx->norb;
    const Block bs = make_block(n * (n + 1) / 2 + 1), ba = make_block(n * (n - 1) / 2);
    const int64_t N = ctx->ndet, nks = (N + 15) / 16;
    const int64_t n2 = (int64_t)n * n, n4 = n2 * n2;
    const int ntile = bs.nrb * bs.nct + ba.nrb * ba.nct;
    cudaStream_t s = ctx->stream;
    const size_t step_bytes = (size_t)kPlanes * (bs.Rd + ba.Rd) * 32;
    size_t budget = ctx->opt.rdm2_chunk_bytes > 0 ? (size_t)ctx->opt.rdm2_chunk_bytes : kDefaultChunk;
    // whole flush groups per chunk: every 512-determinant group K-steps [32j, 32j + 32)
    // is accumulated in the same order whatever the chunking, so the result is
    // the same bits for every chunk size
    int64_t chunk = (int64_t)(budget / step_bytes);
    if (chunk < nks) chunk = std::max<int64_t>(kKTile, chunk / kKTile * kKTile);
    int nsm = 0;
    FCI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    // whole rounds of the tensor kernel's CTAs (the default size rounded up to them)
    const int64_t round = (int64_t)std::max(1, nsm / ntile) * kKTile;
    if (ctx->opt.rdm2_chunk_bytes > 0)
        chunk = chunk < nks && chunk >= round ? chunk / round * round : chunk;
    else
        chunk = (chunk + round - 1) / round * round;
    if (chunk > nks) chunk = nks;
    // one allocation: planes, Gram integers, results, statistics, c's integers, rows; with
    // smaller chunks (down to one flush group) where it does not fit
    size_t total = 0, o_dg = 0, o_stat = 0, o_G = 0, o_out = 0, o_x = 0, o_rows = 0;
    const size_t gbytes = sizeof(long long) * 2 * ((size_t)bs.Rd * bs.Rd + (size_t)ba.Rd * ba.Rd);
    DensityScratch scratch(ctx);
    for (;;) {
        total = 0;
        auto part = [&](size_t bytes) {
            const size_t at = total;
            total += (bytes + 255) / 256 * 256;
            return at;
        };
        o_dg = part(step_bytes * (size_t)chunk), o_stat = part(sizeof(int) * 2), o_G = part(gbytes);
        o_out = part(sizeof(double) * (size_t)(n4 + n2)), o_x = part(sizeof(long long) * (size_t)N);
        o_rows = part(sizeof(uint16_t) * ((size_t)ctx->A.ns * ctx->A.nsingle + (size_t)ctx->B.ns * ctx->B.nsingle));
        const int rc = scratch.take(total);
        if (rc == FCI_OK) break;
        if (rc != FCI_ERR_OOM || chunk <= kKTile) return rc;
        chunk = std::max<int64_t>(kKTile, chunk / 2 / kKTile * kKTile);
    }
    unsigned char *mem = scratch.dev;
    unsigned char *dg = mem + o_dg;
    unsigned long long *G = reinterpret_cast<unsigned long long *>(mem + o_G);
    double *out = reinterpret_cast<double *>(mem + o_out);
    long long *Xc = reinterpret_cast<long long *>(mem + o_x);
    uint16_t *rows = reinterpret_cast<uint16_t *>(mem + o_rows);
    int *d_emax = reinterpret_cast<int *>(mem + o_stat), *d_err = d_emax + 1;
    int herr = 0;
    // per-kernel timing (fci_profile_*) when the call runs as one chunk
    static const char *const names[5] = {"rdm2_stats", "rdm2_prep", "rdm2_digits", "rdm2_tc", "rdm2_finish"};
    const int rec = chunk >= nks ? prof_begin(ctx, s, 5, names) : -1;
    cudaError_t e = cudaMemsetAsync(mem + o_stat, 0, o_out - o_stat, s);  // statistics and G
    if (e == cudaSuccess) {
        k_rdm2_stats<T><<<(unsigned)std::min<int64_t>(ceil_div(N, 256), kStatBlocks), 256, 0, s>>>(C, N, d_emax);
        e = cudaGetLastError();
    }
    prof_mark(ctx, rec, 0, s);
    if (e == cudaSuccess) e = opt_in_max_smem((const void *)k_rdm2_digits, ctx->device);
    if (e == cudaSuccess) e = cudaFuncSetAttribute((const void *)k_rdm2_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e == cudaSuccess) {
        const SpinTables &SA = ctx->A, &SB = ctx->B;
        uint16_t *rows_a = rows, *rows_b = rows + (size_t)SA.ns * SA.nsingle;
        k_rdm2_fixed<T><<<grid_blocks(N), 256, 0, s>>>(C, N, d_emax, Xc);
        if (SA.nsingle) k_rdm2_rows<<<ceil_div(SA.ns * (int64_t)SA.nsingle, 256), 256, 0, s>>>(SA, rows_a);
        if (SB.nsingle) k_rdm2_rows<<<ceil_div(SB.ns * (int64_t)SB.nsingle, 256), 256, 0, s>>>(SB, rows_b);
        e = cudaGetLastError();
        prof_mark(ctx, rec, 1, s);
        for (int64_t k0 = 0; k0 < nks && e == cudaSuccess; k0 += chunk) {
            const int64_t kn = std::min<int64_t>(chunk, nks - k0);
            k_rdm2_digits<<<(unsigned)kn, 256, (size_t)row_stride(n) * 16 * sizeof(long long), s>>>(
                Xc, SA, SB, rows_a, rows_b, n, bs, ba, k0, N, reinterpret_cast<uint4 *>(dg));
            e = cudaGetLastError();
            if (e != cudaSuccess) break;
            prof_mark(ctx, rec, 2, s);
            TcArgs P;
            P.dg = dg;
            P.nks = kn;
            P.step = (int64_t)step_bytes;
            P.blk[0] = bs;
            P.blk[1] = ba;
            P.ntile = ntile;
            P.G = G;
            P.err = d_err;
            // a multiple of ntile CTAs (one tile each) when the tiles fit the
            // SMs, no more groups than K-ranges
            const int64_t nkr = (kn + kKTile - 1) / kKTile;
            const unsigned grid = ntile <= nsm ? (unsigned)(ntile * std::min<int64_t>(nsm / ntile, nkr)) : (unsigned)nsm;
            k_rdm2_tc<<<grid, kThreads, kSmem, s>>>(P);
            e = cudaGetLastError();
            prof_mark(ctx, rec, 3, s);
        }
    }
    if (e == cudaSuccess) {
        k_rdm2_finish<<<ceil_div(n4 + n2, 256), 256, 0, s>>>(
            G, bs.Rd, ba.Rd, n, d_emax, sizeof(T) == 8 ? 1022 : 126, sizeof(T) == 8 ? 0x7FF : 0xFF, out, out + n4);
        e = cudaGetLastError();
        prof_mark(ctx, rec, 4, s);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(g2_host, out, sizeof(double) * n4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && g1_host) e = cudaMemcpyAsync(g1_host, out + n4, sizeof(double) * n2, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, d_err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "rdm2");
    if (herr & 1) return fail(FCI_ERR_TIMEOUT, "rdm2: a bounded wait in the tensor-core kernel gave up");
    if (herr) return fail(FCI_ERR_RANGE, "rdm2: an exact accumulator left its range");
    return FCI_OK;
}

}  // namespace r2

int run_rdm2(fci_ctx *ctx, const void *c, int dtype, double *gamma1, double *gamma2) {
    if (dtype == FCI_F64) return r2::rdm2_impl<double>(ctx, (const double *)c, gamma1, gamma2);
    return r2::rdm2_impl<float>(ctx, (const float *)c, gamma1, gamma2);
}

}  // namespace fci
