// pd_hxf.cu -- y = H x by pair removal on the tensor cores (variant 2, FP32).
//
// The off-diagonal part of Eq. 2 is a product of two sparse maps with a dense
// matrix in between,
//     V(t)_j = x(t + j),   Z(t) = G V(t),   y(s) = sum_{i in s} Z(s - i)_i,
// t running over the states with one pair less (t + j: a pair added on orbit j,
// j empty in t).  One gather of the M = Omega - N + 1 elements around t serves
// all M (M - 1) hops that pass through t, where a row-by-row kernel loads,
// addresses and multiplies every hop on its own.  The middle step is one small
// dense product per t with the same matrix, so 128 words t make one tile
//     Z [128 x Omega] = V [128 x Omega] G
// on the 5th-generation tensor cores.
//
// Precision.  tcgen05.mma kind::tf32 keeps 11 significant bits of an operand, so
// V and G are split in two, v = v_hi + v_lo with v_hi = v rounded to TF32 (the
// difference is exact), and Z = V_hi G_lo + V_lo G_hi + V_hi G_hi accumulates in
// FP32, the small products first (the accumulator truncates: mean row error 0.189
// -> 0.170 x 2^-23 at C(24,12) against V_hi G_hi first).  Of a term at most 4 x
// 2^-23 is dropped: V_lo G_lo (2^-22: a low part is at most 2^-11), the last bit of
// V_lo, which the unit cuts off, and the rounding of G_lo (2^-23 each).  A row sum
// is a tree of depth two instead of a chain of N (Omega - N) additions, so rows are
// more exact than row by row (norm of the error at C(24,12) 1.34e-7 / 3.23e-7,
// C(14,7) 0.73e-7 / 1.95e-7), but not a row with one dominant hop (1.0e-7 / 0.34e-7).
// Measured and not kept: V_lo G_lo as a fourth product, 0.56 to 0.82e-7 for such a
// row, the same 1.34e-7 for the others, and C(30,15) 6.55 -> 6.80 ms.  Elements that are
// not finite (or that overflow when rounded to TF32) cannot be split; a tile
// that meets one sets a flag, and the second kernel then forms the rows that it
// reaches term by term.
//
// Layout.  Low orbits: the L <= 12 lowest; high word h, block as in
// pd_internal.h.  remove_kernel takes one high word at a time (a block of t):
// one thread gathers one t, writes the split row into tensor memory (operand A
// of the product), and reads its row of Z back from there.  Results for low
// orbits belong to rows of the block h itself and meet in shared memory (slot
// [orbit][row], one writer each); the block's partial y is written once.
// Results for a high orbit q belong to block h + q at the same low word: they go
// to a scratch vector, ordered by (block of y, ordinal of q, row), where
// add_kernel streams them: y(h, l) += sum_a scratch(h, a, l).  The scratch is
// written and read as data used once, so that L2 keeps x and the caller's
// vectors (plain stores / streaming stores: C(24,12) 96.2 / 94.7 us and 10.09 /
// 9.96 ms for a solve around it, C(28,14) 1.71 / 1.61 ms, C(30,15) 6.89 / 6.53 ms).  No two threads
// add to the same element, so the sums have a fixed order.
#include "pd_internal.h"

#include <math_constants.h>

#include <climits>
#include <cstring>
#include <type_traits>
#include <utility>

namespace pd {
namespace {

constexpr int kLT = 12;                  // low orbits
constexpr int kRows = 924;               // most rows of a block: C(12,6)
constexpr int kSpare = kRows;            // slot of hops that do not exist (reads 0, writes ignored)
constexpr int kStride = 928;             // floats per orbit of the partial results
// Scratch (floats): all rows at once up to 2 GiB, else class by class (the rows
// with k low pairs, k ascending), which bounds it at the largest class: 1.62 GB
// instead of 5.58 GB at Omega=30, 6.83 GB instead of 24.0 GB at Omega=32.  Measured,
// when the line was drawn, at once / by class: Omega=24 0.096 / 0.28 ms (26 short launches), Omega=28
// 1.79 / 1.97 ms, Omega=30 7.45 / 7.36 ms.
constexpr int64_t kScratchAll = (int64_t)2048 << 18;
constexpr int kTile = 128;               // words t per tile: the lanes of tensor memory
constexpr int kMaxHigh = 28;             // high orbits (12 + 28 = 40 columns)
constexpr size_t kSmemMax = 112 * 1024;   // two CTAs per SM
constexpr int kTmemCols = 256;           // tensor-memory columns of a CTA: two CTAs fill an SM
constexpr int kDrainPolls = 1 << 12;     // polls of the wait for a product in flight after its wait gave up

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~size_t(15); }
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

template <class F, int... I>
__device__ __forceinline__ void for_each_impl(F &&f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
// f(0), ..., f(N - 1) with the index as a compile-time constant
template <int N, class F>
__device__ __forceinline__ void for_each(F &&f)
{
    for_each_impl(f, std::make_integer_sequence<int, N>{});
}

// Columns of a tile: low orbit p at p, high orbit q at 12 + q, zero-padded to KP
// (K of the product) and NP (its N).  Tensor memory per group of four warps:
// V_hi [KP], V_lo [KP], Z [NP].  Groups per CTA: as many as 256 columns hold.
template <int KP>
struct Cfg {
    static constexpr int kN = (KP + 15) / 16 * 16;
    static constexpr int kCols = 2 * KP + kN;
    static constexpr int kGroups = KP <= 24 ? 3 : 2;
    static constexpr int kSets = KP <= 32 ? 2 : 1;       // sets of partial results in shared memory
    static constexpr int kWarps = 4 * kGroups;           // and one warp that prepares the next block
    static constexpr int kThreads = 32 * (kWarps + 1);
    static_assert(kGroups * kCols <= kTmemCols, "tensor memory of a CTA");
};

// ---- tables ---------------------------------------------------------------------
__device__ int colex_rank(uint32_t w, const uint64_t *__restrict__ binom)
{
    int r = 0, c = 0;
    for (; w; w &= w - 1) r += (int)__ldg(binom + (__ffs(w) - 1) * kBinomStride + ++c);
    return r;
}
// Low words and their hops.  Word w = the r-th of c pairs is row lo_off[c] + r.
// For orbit j: byte offset 4 * rank(w with orbit j added), 4 * kSpare if j is in
// w or not an orbit.  Two orbits per 32-bit entry, the entries of one pair of
// orbits contiguous over the rows (table[pair << L | row]), so that a warp's 32
// rows are one coalesced load.
__global__ void hop_table_kernel(int L, const uint64_t *__restrict__ binom, uint16_t *__restrict__ low,
                                 uint32_t *__restrict__ up)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ((kLT / 2) << L)) return;
    const uint32_t w = (uint32_t)i & ((1u << L) - 1u);
    const int pair = i >> L;
    int row = colex_rank(w, binom);
    for (int c = 0; c < __popc(w); ++c) row += (int)__ldg(binom + L * kBinomStride + c);
    uint32_t u = 0;
    for (int t = 1; t >= 0; --t) {
        const int j = 2 * pair + t;
        u = u << 16 | (uint32_t)((j < L && !(w >> j & 1u)) ? 4 * colex_rank(w | (1u << j), binom) : 4 * kSpare);
    }
    up[(pair << L) + row] = u;
    if (pair == 0) low[row] = (uint16_t)w;
}

// High words by class (pairs in the high orbits), ascending within a class
// (colex unranking)
struct WordClasses {
    int n;
    int ph[kLT + 1];
    int64_t first[kLT + 2];              // number of the class's first word
};
__global__ void high_words_kernel(const WordClasses C, int H, const uint64_t *__restrict__ binom,
                                  uint32_t *__restrict__ words)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C.first[C.n]) return;
    int c = 0;
    while (i >= C.first[c + 1]) ++c;
    uint64_t idx = (uint64_t)(i - C.first[c]);
    uint32_t w = 0;
    int p = H - 1;
    for (int j = C.ph[c]; j > 0; --j) {
        while (__ldg(binom + p * kBinomStride + j) > idx) --p;
        idx -= __ldg(binom + p * kBinomStride + j);
        w |= 1u << p;
        --p;
    }
    words[i] = w;
}

// ---- pair removal ---------------------------------------------------------------
constexpr int kPartBytes = 4 * kLT * kStride;

struct __align__(16) BlockSmem {         // one block of t
    const float *xe[32];                 // block h + q of x, by high orbit q; zeros if q is occupied
    float *ze[32];                       // where the results for orbit q go
    float x[kStride];                    // block h of x; x[kSpare] = 0
    uint32_t h, base;
    float dh;                            // diagonal sum of its high orbits
    long long b;                         // its number; >= end: none left
};

struct LayoutR {
    size_t b, buf, dlow, bin, crk, dh, total;
};
__host__ __device__ inline LayoutR layout_r(int KP, int H, int N)
{
    LayoutR s;
    const int h1 = H > 0 ? H : 1;
    const int np = (KP + 15) / 16 * 16;
    size_t off = (KP <= 32 ? 2 : 1) * kPartBytes;   // the partial results lie at 0
    s.b = off;    off = align16(off + sizeof(float) * 2 * np * KP);
    s.buf = off;  off = align16(off + 3 * sizeof(BlockSmem));
    s.dlow = off; off = align16(off + sizeof(float) * 128);
    s.bin = off;  off = align16(off + sizeof(uint32_t) * h1 * (N + 2));
    s.crk = off;  off = align16(off + sizeof(uint32_t) * h1 * (h1 + 2));
    s.dh = off;   off = align16(off + sizeof(float) * h1);
    s.total = off;
    return s;
}

struct RemoveArgs {
    int omega, N, L, H;
    int lo_off[kLT + 2];
    int polls;                           // of a wait before it gives up
    int64_t first, end;                  // blocks of t of this launch, in words
    int64_t zbase[kLT + 1];              // scratch of the rows with k low pairs
    const uint32_t *words;
    const uint16_t *low;
    const uint32_t *up;
    const uint64_t *binom;
    const float *zeros;                  // kRows zeros
    float *scratch;
};

__device__ __forceinline__ void copy_async4(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Block of t with high word h, by one warp; lane j: high orbit j.  k = N -
// popcount(h) low pairs in block h of x, k - 1 in the words t.  With A, B(j) the
// binomials of the pair on j at its own ordinal and one lower, EA, EB their sums
// over the occupied high orbits below j, block h + q of x starts at
//     EB(q) + C(L + q, k + #below) + base(h) - EA(q)     (modulo 2^32)
// and its place among the words of its class is, with R(j) = C(j, ordinal from 1)
// and S(j) = C(j, ordinal + 1),   ER(q) + C(q, #below + 1) + sum S - ES(q).
struct HighWord {
    uint32_t base;                       // start of block h of x
    float dh;                            // diagonal sum of its high orbits
    bool hop;                            // this lane's orbit exists and is empty; if so:
    uint32_t x;                          // start of block h + q of x
    int64_t z;                           // where the results for orbit q go in the scratch
};
__device__ __forceinline__ HighWord high_word(const RemoveArgs &A, const uint32_t h, const uint32_t *bin,
                                              const uint32_t *crk, const float *dh)
{
    const int lane = threadIdx.x & 31;
    const int N = A.N, H = A.H;
    const int ph = __popc(h), k = N - ph;
    const bool occ = (h >> lane) & 1u;
    const int io = __popc(h & ((1u << lane) - 1u));
    uint32_t a = 0, bq = 0, c1 = 0, c2 = 0;
    if (lane < H) {
        bq = bin[lane * (N + 2) + k + io];
        c1 = crk[lane * (H + 2) + io + 1];
    }
    if (occ) {
        a = bin[lane * (N + 2) + k + io + 1];
        c2 = crk[lane * (H + 2) + io + 2];
    }
    uint32_t ia = a, ib = occ ? bq : 0u, ir = occ ? c1 : 0u, is = c2;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t ta = __shfl_up_sync(0xffffffffu, ia, o);
        const uint32_t tb = __shfl_up_sync(0xffffffffu, ib, o);
        const uint32_t tr = __shfl_up_sync(0xffffffffu, ir, o);
        const uint32_t ts = __shfl_up_sync(0xffffffffu, is, o);
        if (lane >= o) { ia += ta; ib += tb; ir += tr; is += ts; }
    }
    const uint32_t stot = __shfl_sync(0xffffffffu, is, 31);
    HighWord w;
    w.base = __shfl_sync(0xffffffffu, ia, 31);
    w.hop = lane < H && !occ;
    // (lanes of empty orbits: the inclusive sums are the exclusive ones)
    w.x = ib + bq + w.base - ia;
    const uint64_t place = (uint32_t)(ir + c1 + stot - is);
    const int nt = A.lo_off[k] - A.lo_off[k - 1];
    w.z = A.zbase[k - 1] + (int64_t)(place * (uint64_t)(ph + 1) + (uint64_t)io) * nt;
    w.dh = occ ? dh[lane] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w.dh += __shfl_xor_sync(0xffffffffu, w.dh, o);
    return w;
}

// the last warp: block of t with high word h into buffer bs
__device__ __forceinline__ void prepare_block(BlockSmem &bs, const RemoveArgs &A, const uint32_t h,
                                              const uint32_t *bin, const uint32_t *crk, const float *dh,
                                              const float *__restrict__ x)
{
    const int lane = threadIdx.x & 31;
    const int k = A.N - __popc(h);
    const HighWord w = high_word(A, h, bin, crk, dh);
    if (k <= A.L) {                               // block h exists (t is not the full low word)
        const int nk = A.lo_off[k + 1] - A.lo_off[k];
        for (int r = lane; r < nk; r += 32) copy_async4(bs.x + r, x + w.base + r);
    }
    bs.xe[lane] = w.hop ? x + w.x : A.zeros;
    if (w.hop) bs.ze[lane] = A.scratch + w.z;
    if (lane == 0) {
        bs.h = h;
        bs.base = w.base;
        bs.dh = w.dh;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// shared memory matrix descriptor of G: K-major, no swizzle, core matrices of 8
// rows x 16 bytes, 128 bytes apart in K and KP * 32 bytes apart in N
template <int KP>
__device__ __forceinline__ uint64_t g_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(128u >> 4) << 16;
    d |= (uint64_t)((KP * 32u) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t phase, int polls)
{
    for (int it = 0; it < polls; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(done)
                     : "r"(bar), "r"(phase), "r"(1000000u)
                     : "memory");
        if (done) return true;
    }
    return false;
}

// A bounded wait for a product.  When it expires, what the launch writes is void
// (the add kernels write NaN) and the CTA takes no more blocks, at most one that
// is prepared already; the product's operands and tensor memory are still in use,
// so it is waited for once more.
__device__ __noinline__ void expired(uint32_t bar, uint32_t phase, int *s_void)
{
    *reinterpret_cast<volatile int *>(s_void) = 1;
    mbar_poll(bar, phase, kDrainPolls);
}
__device__ __forceinline__ void wait_product(uint32_t bar, uint32_t phase, int polls, int *s_void)
{
    if (!mbar_poll(bar, phase, polls)) expired(bar, phase, s_void);
}

__device__ __forceinline__ float to_tf32(float v)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
    return __uint_as_float(r);
}

// eight columns of this thread's row of tensor memory
__device__ __forceinline__ void tmem_st8(uint32_t addr, const float (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(addr),
                 "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                 "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
                 "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr)
                 : "memory");
}

// G and the tables of a CTA into shared memory
template <int KP>
__device__ __forceinline__ void stage_tables(const RemoveArgs &A, const float *__restrict__ G, const float *__restrict__ d,
                                             unsigned char *g_smem, uint32_t *bin, uint32_t *crk, float *dh, float *dlow,
                                             const int threads)
{
    using C = Cfg<KP>;
    const int omega = A.omega, L = A.L, H = A.H, N = A.N, tid = threadIdx.x;
    // G in the operand layout, high and low parts (row n: the orbit that
    // receives the pair, column k: the orbit it leaves)
    for (int i = tid; i < C::kN * KP; i += threads) {
        const int n = i / KP, k = i % KP;
        auto orbit = [&](int c) { return c < kLT ? (c < L ? c : -1) : (c - kLT < H ? L + c - kLT : -1); };
        const int on = orbit(n), ok = orbit(k);
        const float g = (on >= 0 && ok >= 0 && on != ok) ? G[on * omega + ok] : 0.0f;
        const float hi = to_tf32(g);
        unsigned char *p = g_smem + (n >> 3) * (KP * 32) + (k >> 2) * 128 + (n & 7) * 16 + (k & 3) * 4;
        *reinterpret_cast<float *>(p) = hi;
        *reinterpret_cast<float *>(p + 4 * C::kN * KP) = to_tf32(g - hi);
    }
    for (int i = tid; i < H * (N + 2); i += threads)
        bin[i] = (uint32_t)__ldg(A.binom + (L + i / (N + 2)) * kBinomStride + i % (N + 2));
    for (int i = tid; i < H * (H + 2); i += threads)
        crk[i] = (uint32_t)__ldg(A.binom + (i / (H + 2)) * kBinomStride + i % (H + 2));
    for (int i = tid; i < H; i += threads) dh[i] = d[L + i];
    for (int i = tid; i < 128; i += threads) {   // diagonal sums of the two halves of a low word
        const int w = i & 63, p0 = i < 64 ? 0 : 6;
        float v = 0.0f;
        for (int p = 0; p < 6; ++p)
            if ((w >> p & 1) && p0 + p < L) v += d[p0 + p];
        dlow[i] = v;
    }
}

// Z = V G of one tile (one thread): TF32 operands, FP32 accumulator, both K-major, M = 128
template <int KP>
__device__ __forceinline__ void issue_product(const uint32_t tmem, const uint32_t g_smem, const uint32_t bar)
{
    using C = Cfg<KP>;
    constexpr uint32_t idesc =
        (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(C::kN >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
    const uint64_t b0 = g_desc<KP>(g_smem);
#pragma unroll
    for (int s = 0; s < 3; ++s)                   // V_hi G_lo, V_lo G_hi, V_hi G_hi
#pragma unroll
        for (int kk = 0; kk < KP / 8; ++kk) {
            const uint32_t a = tmem + (s == 1 ? KP : 0) + 8 * kk;
            const uint64_t db = b0 + (uint64_t)(((s == 0 ? 4 * C::kN * KP : 0) + kk * 256) >> 4);
            const uint32_t accum = (s || kk) ? 1u : 0u;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                         "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem + 2 * KP),
                         "r"(a), "l"(db), "r"(idesc), "r"(accum)
                         : "memory");
        }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// What bounds it: instruction issue and the latency of a tile's chain (gather,
// split, tensor-memory store, product, load, scatter).  Two CTAs of three groups
// share an SM's tensor memory, so that one group's gathers overlap another's
// product; the high orbits of the next tile are loaded while the product runs;
// the ninth (thirteenth) warp prepares the next block's pointers.  Omega=24:
// 78 us alone with a cold cache for 3.9e8 hops (47e6 warp instructions, 0.54 of
// the issue slots), where the row-by-row kernel (pd_hx.cu, variant 3) took
// 215 us; both kernels together 0.0964 ms.  Measured and not kept: FP32
// multiply-adds instead of the tensor cores (packed pairs, coefficients from
// shared memory or the constant bank, 8, 10 or 12 low orbits, hops between high
// orbits in registers): 0.127 to 0.18 ms.
__device__ __forceinline__ void report_void(Tickets *tk)
{
    atomicOr(&tk->mark, kMarkVoid);
    atomicExch(&tk->expired, 1);
}

template <int KP>
__device__ __forceinline__ void remove_blocks(const RemoveArgs &A, const float *__restrict__ G, const float *__restrict__ d,
                                              const float *__restrict__ x, float *__restrict__ y, Tickets *tk,
                                              const unsigned ctas)
{
    using C = Cfg<KP>;
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_bar[C::kGroups];
    __shared__ uint32_t s_tmem;
    __shared__ int s_void;                        // a wait gave up
    const int L = A.L, H = A.H, N = A.N;
    const LayoutR lay = layout_r(KP, H, N);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, group = warp >> 2;
    uint32_t *bin = reinterpret_cast<uint32_t *>(smem + lay.bin), *crk = reinterpret_cast<uint32_t *>(smem + lay.crk);
    float *dlow = reinterpret_cast<float *>(smem + lay.dlow), *dh = reinterpret_cast<float *>(smem + lay.dh);
    BlockSmem *bufs = reinterpret_cast<BlockSmem *>(smem + lay.buf);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int g = 0; g < C::kGroups; ++g)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s_bar[g])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    stage_tables<KP>(A, G, d, smem + lay.b, bin, crk, dh, dlow, C::kThreads);
    if (tid < 3) bufs[tid].x[kSpare] = 0.0f;
    if (tid == 0) s_void = 0;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // G: generic stores -> tensor core reads
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem + (uint32_t)(group < C::kGroups ? group : 0) * C::kCols;
    const uint32_t trow = tmem + ((uint32_t)(warp & 3) << 21);       // this warp's 32 lanes
    const uint32_t bar = smem_u32(&s_bar[group < C::kGroups ? group : 0]);
    uint32_t phase = 0;
    bool odd = false;                             // a row of Z is NaN

    auto take = [&](BlockSmem &bs) {              // the last warp
        long long b = A.end;                      // (none after a wait gave up)
        if (lane == 0 && !*reinterpret_cast<volatile int *>(&s_void)) b = A.first + (long long)atomicAdd(&tk->hx_next, 1ull);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b < A.end) prepare_block(bs, A, __ldg(A.words + b), bin, crk, dh, x);
        if (lane == 0) bs.b = b;
    };
    // rows of a finished block: its slots summed per row, the diagonal, y
    auto rows = [&](const BlockSmem &bs, const float *part) {
        const int k = N - __popc(bs.h);
        if (k > L) return;                        // no such block
        const int lo_k = A.lo_off[k], nk = A.lo_off[k + 1] - lo_k;
        for (int r = tid; r < nk; r += 32 * C::kWarps) {
            const uint32_t l = __ldg(A.low + lo_k + r);
            const float D = (dlow[l & 63u] + dlow[64 + (l >> 6)]) + bs.dh;
            float s = 0.0f;
#pragma unroll
            for (int o = 0; o < kLT; ++o)
                if (l >> o & 1u) s += part[o * kStride + r];
            y[bs.base + r] = fmaf(D, bs.x[r], s);
        }
    };
    // One barrier per block: after it the slots of block i are complete and
    // buffer i + 1 is filled; the warps then sum the rows of block i and go on
    // to the words of block i + 1 (slots alternate between two sets, buffers
    // rotate over three: rows, words, preparation).
    if (warp == C::kWarps) take(bufs[0]);
    __syncthreads();
    int cur = 0;                                  // buffer of block i
    for (int i = 0;; ++i) {
        const BlockSmem &bs = bufs[cur];
        const int nxt = cur == 2 ? 0 : cur + 1;
        const bool more = bs.b < A.end;
        if (warp == C::kWarps) {
            if (more) take(bufs[nxt]);
        } else {
            if (i > 0) rows(bufs[cur == 0 ? 2 : cur - 1], reinterpret_cast<const float *>(smem + (C::kSets == 2 ? ((i - 1) & 1) * kPartBytes : 0)));
            if constexpr (C::kSets == 1) asm volatile("bar.sync 4, %0;\n" ::"n"(32 * C::kWarps) : "memory");
            if (more) {
                const uint32_t h = bs.h;
                const int k = N - __popc(h);      // k >= 1
                const int lo_t = A.lo_off[k - 1], nt = A.lo_off[k] - lo_t;
                const uint32_t empty = ~h & ((1u << H) - 1u);   // high orbits that receive results
                const uint32_t poff = C::kSets == 2 ? (uint32_t)(i & 1) * (kPartBytes * 0x10001u) : 0u;
                constexpr int kPre = KP <= 24 ? KP - kLT : 8;   // high orbits loaded one tile ahead
                uint32_t hop[kLT / 2];
                float vh[kPre];
                auto load = [&](int c) {
                    const int rc = min(c * kTile + (tid & (kTile - 1)), nt - 1);
#pragma unroll
                    for (int p = 0; p < kLT / 2; ++p) hop[p] = __ldg(A.up + (p << L) + lo_t + rc);
#pragma unroll
                    for (int q = 0; q < kPre; ++q) vh[q] = __ldg(bs.xe[q] + rc);
                };
                if (group * kTile < nt) load(group);
                for (int c = group; c * kTile < nt; c += C::kGroups) {
                    const int r = c * kTile + (tid & (kTile - 1));
                    const bool in = r < nt;
                    // gather and split, eight columns at a time
                    for_each<KP / 8>([&](auto gc) {
                        constexpr int g = decltype(gc)::value;
                        float v[8], hi[8];
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            const int p = 8 * g + t;
                            if (p < kLT) {
                                const uint32_t off = (p & 1) ? hop[p / 2] >> 16 : hop[p / 2] & 0xffffu;
                                v[t] = *reinterpret_cast<const float *>(reinterpret_cast<const char *>(bs.x) + off);
                            } else if (p - kLT < kPre) {
                                v[t] = vh[p - kLT];
                            } else {
                                v[t] = __ldg(bs.xe[p - kLT] + (in ? r : nt - 1));
                            }
                        }
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            hi[t] = to_tf32(v[t]);
                            v[t] -= hi[t];        // NaN where v is not finite, and with it the whole row of Z
                        }
                        tmem_st8(trow + 8 * g, hi);
                        tmem_st8(trow + KP + 8 * g, v);
                    });
                    // one test per store instead of three (in the block, an orbit, empty): the
                    // product at Omega=30 7.15 -> 6.89 ms, Omega=24 98.2 -> 96.2 us
                    const uint32_t to = in ? empty : 0u;
                    uint32_t slot[kLT / 2];
#pragma unroll
                    for (int p = 0; p < kLT / 2; ++p) slot[p] = hop[p] + poff;
                    asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                    asm volatile("bar.sync %0, 128;\n" ::"r"(group + 1) : "memory");
                    if ((tid & (kTile - 1)) == 0) {
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        issue_product<KP>(tmem, smem_u32(smem + lay.b), bar);
                    }
                    __syncwarp();
                    if ((c + C::kGroups) * kTile < nt) load(c + C::kGroups);   // overlaps the product
                    wait_product(bar, phase, A.polls, &s_void);
                    phase ^= 1u;
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    for_each<KP / 8>([&](auto gc) {
                        constexpr int g = decltype(gc)::value;
                        uint32_t z[8];
                        tmem_ld8(trow + 2 * KP + 8 * g, z);
                        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                        if (g == 0) odd |= __uint_as_float(z[0]) != __uint_as_float(z[0]);
#pragma unroll
                        for (int t = 0; t < 8; ++t) {
                            const int p = 8 * g + t;
                            if (p < kLT) {
                                const uint32_t off = (p & 1) ? slot[p / 2] >> 16 : slot[p / 2] & 0xffffu;
                                *reinterpret_cast<float *>(smem + p * kStride * 4 + off) = __uint_as_float(z[t]);
                            } else if (to >> (p - kLT) & 1u) {
                                __stcs(bs.ze[p - kLT] + r, __uint_as_float(z[t]));
                            }
                        }
                    });
                    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
                }
            }
        }
        if (!more) break;
        __syncthreads();
        cur = nxt;
    }
    if (odd) atomicOr(&tk->mark, kMarkSplit);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(s_tmem), "r"(kTmemCols) : "memory");
    if (tid == 0 && s_void) report_void(tk);
    if (arrive_last(&tk->hx_done, ctas) && tid == 0) tk->hx_next = 0ull;
}

template <int KP>
__global__ void __launch_bounds__(Cfg<KP>::kThreads, 2)
remove_kernel(const __grid_constant__ RemoveArgs A, const float *__restrict__ G, const float *__restrict__ d,
              const float *__restrict__ x, float *__restrict__ y, Tickets *tk, const int *__restrict__ skip)
{
    if (skip && *skip) return;                    // CTA-uniform
    remove_blocks<KP>(A, G, d, x, y, tk, gridDim.x);
}

// ---- pair removal, small blocks -------------------------------------------------
// Classes whose blocks have few words t (1, 12 or 66 of the 128 of a tile): a
// group of four warps takes several high words of one class together.  Far from
// half filling these are nearly all blocks: 565,000 of the 600,000 of Omega=34,
// N=9, whose lone tiles held 12 words and less and left one of the two groups of
// remove_kernel's CTA without work.
constexpr int kSmallWords = 66;          // most words t per block of such a class
constexpr int kSmallRows = 660;          // most rows, and words t, of the blocks taken together
constexpr int kSmallStride = 664;        // floats per orbit of their partial results
constexpr int kSmallBlocks = 32;         // most blocks taken together
constexpr int kSmallClasses = 6;
constexpr int kSmallGroups = 2;          // groups per CTA; two CTAs per SM
// Fewest such blocks that get a launch of their own (in remove_kernel / on their
// own): 990 blocks, C(30,4), 31.0 / 38.7 us, 1456, C(26,5), 33.8 / 40.4 us, 3682,
// C(40,4), 71.8 / 43.1 us.
constexpr int kSmallMin = 2000;

struct SmallArgs {
    RemoveArgs r;
    int n;                               // classes
    int k[kSmallClasses], m[kSmallClasses];   // low pairs of the rows; blocks per item
    int64_t first[kSmallClasses], end[kSmallClasses];   // words of the class
    int64_t item[kSmallClasses + 1];     // number of the class's first item
};
struct LayoutS {
    size_t b, dlow, bin, crk, dh, group, part, x, h, base, bdh, xe, ze, per_group, total;
};
__host__ __device__ inline LayoutS layout_s(int KP, int H, int N)
{
    LayoutS s;
    const int np = (KP + 15) / 16 * 16;
    size_t off = 0;
    s.b = off;    off = align16(off + sizeof(float) * 2 * np * KP);
    s.dlow = off; off = align16(off + sizeof(float) * 128);
    s.bin = off;  off = align16(off + sizeof(uint32_t) * H * (N + 2));
    s.crk = off;  off = align16(off + sizeof(uint32_t) * H * (H + 2));
    s.dh = off;   off = align16(off + sizeof(float) * H);
    s.group = off;
    off = 0;      // per group
    s.part = off; off += sizeof(float) * kLT * kSmallStride;
    s.x = off;    off += sizeof(float) * kSmallStride;
    s.h = off;    off += sizeof(uint32_t) * kSmallBlocks;
    s.base = off; off += sizeof(uint32_t) * kSmallBlocks;
    s.bdh = off;  off += sizeof(float) * kSmallBlocks;
    s.xe = off;   off += sizeof(uint32_t) * kSmallBlocks * H;
    s.ze = off;   off += sizeof(uint32_t) * kSmallBlocks * H;
    s.per_group = align16(off);
    s.total = s.group + kSmallGroups * s.per_group;
    return s;
}

// What bounds it: the latency of an item's chain (starts of the blocks, gather,
// product, scatter, rows: about 8 us), of which only four overlap per SM, because
// the operands of four tiles fill its tensor memory.  Omega=34, N=9: 0.72 ms for
// these blocks and 0.51 ms for the others, against 5.1 ms for both in
// remove_kernel.  Measured and not kept: the rows' sums over the set bits of a
// low word instead of twelve predicated loads, 0.76 ms.
template <int KP>
__global__ void __launch_bounds__(128 * kSmallGroups, 2)
remove_small_kernel(const __grid_constant__ SmallArgs S, const float *__restrict__ G, const float *__restrict__ d,
                    const float *__restrict__ x, float *__restrict__ y, Tickets *tk, const int *__restrict__ skip)
{
    using C = Cfg<KP>;
    static_assert(kSmallGroups * C::kCols <= kTmemCols, "tensor memory of a CTA");
    if (skip && *skip) return;                    // CTA-uniform
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t s_bar[kSmallGroups];
    __shared__ uint32_t s_tmem;
    __shared__ int s_void[kSmallGroups][2];       // a wait gave up in an item of this parity
    const RemoveArgs &A = S.r;
    const int L = A.L, H = A.H, N = A.N;
    const LayoutS lay = layout_s(KP, H, N);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, group = warp >> 2, gt = tid & 127;
    uint32_t *bin = reinterpret_cast<uint32_t *>(smem + lay.bin), *crk = reinterpret_cast<uint32_t *>(smem + lay.crk);
    float *dlow = reinterpret_cast<float *>(smem + lay.dlow), *dh = reinterpret_cast<float *>(smem + lay.dh);
    unsigned char *mine = smem + lay.group + group * lay.per_group;
    float *part = reinterpret_cast<float *>(mine + lay.part), *bx = reinterpret_cast<float *>(mine + lay.x);
    uint32_t *bh = reinterpret_cast<uint32_t *>(mine + lay.h), *bbase = reinterpret_cast<uint32_t *>(mine + lay.base);
    float *bdh = reinterpret_cast<float *>(mine + lay.bdh);
    uint32_t *xe = reinterpret_cast<uint32_t *>(mine + lay.xe), *ze = reinterpret_cast<uint32_t *>(mine + lay.ze);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int g = 0; g < kSmallGroups; ++g)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&s_bar[g])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    stage_tables<KP>(A, G, d, smem + lay.b, bin, crk, dh, dlow, 128 * kSmallGroups);
    if (gt == 0) bx[kSmallRows] = 0.0f;
    if (gt < 2) s_void[group][gt] = 0;
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // G: generic stores -> tensor core reads
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = s_tmem + (uint32_t)group * C::kCols;
    const uint32_t trow = tmem + ((uint32_t)(warp & 3) << 21);       // this warp's 32 lanes
    const uint32_t bar = smem_u32(&s_bar[group]);
    uint32_t phase = 0;
    bool odd = false;
    auto sync = [&] { asm volatile("bar.sync %0, 128;\n" ::"r"(group + 1) : "memory"); };

    // Items in turn (sorted by class, so every group gets its share of each).
    // Block i of an item belongs to warp i % 4; lane j holds the word of the
    // warp's j-th block, loaded one item ahead.
    struct Item {
        int k, m;                        // low pairs of the rows, blocks
        uint32_t word;
    };
    int c = 0;
    auto fetch = [&](int64_t it) {
        Item t{0, 0, 0u};
        if (it >= S.item[S.n]) return t;
        while (it >= S.item[c + 1]) ++c;
        const int64_t b = S.first[c] + (it - S.item[c]) * S.m[c];
        t.k = S.k[c];
        t.m = (int)min((int64_t)S.m[c], S.end[c] - b);
        const int i = (warp & 3) + 4 * lane;
        if (i < t.m) t.word = __ldg(A.words + b + i);
        return t;
    };
    const int64_t step = (int64_t)gridDim.x * kSmallGroups;
    int64_t it = (int64_t)blockIdx.x * kSmallGroups + group;
    Item cur = fetch(it);
    for (int parity = 0; cur.m > 0; parity ^= 1) {
        it += step;
        const Item nxt = fetch(it);
        const int k = cur.k, m = cur.m;
        const int lo_t = A.lo_off[k - 1], nt = A.lo_off[k] - lo_t;
        const int lo_k = A.lo_off[k], nk = k <= L ? A.lo_off[k + 1] - lo_k : 0;
        for (int j = 0, i = warp & 3; i < m; ++j, i += 4) {
            const uint32_t h = __shfl_sync(0xffffffffu, cur.word, j);
            const HighWord w = high_word(A, h, bin, crk, dh);
            for (int r = lane; r < nk; r += 32) copy_async4(bx + i * nk + r, x + w.base + r);
            if (w.hop) {
                xe[i * H + lane] = w.x;
                ze[i * H + lane] = (uint32_t)w.z;
            }
            if (lane == 0) {
                bh[i] = h;
                bbase[i] = w.base;
                bdh[i] = w.dh;
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        sync();
        const int words = m * nt;
        for (int r0 = 0; r0 < words; r0 += kTile) {
            const bool in = r0 + gt < words;
            const int r = in ? r0 + gt : words - 1;
            const int i = r / nt, t = r - i * nt;
            const uint32_t empty = ~bh[i] & ((1u << H) - 1u), to = in ? empty : 0u;
            uint32_t hop[kLT / 2];
            // offsets into the item's rows; beyond its last row: the spare element
            const uint32_t shift = (uint32_t)(4 * i * nk) * 0x10001u;
#pragma unroll
            for (int p = 0; p < kLT / 2; ++p)
                hop[p] = __vminu2(__ldg(A.up + (p << L) + lo_t + t) + shift, 4 * kSmallRows * 0x10001u);
            float vh[KP - kLT];
#pragma unroll
            for (int q = 0; q < KP - kLT; ++q)
                vh[q] = empty >> q & 1u ? __ldg(x + (uint32_t)(xe[i * H + q] + t)) : 0.0f;
            for_each<KP / 8>([&](auto gc) {
                constexpr int g = decltype(gc)::value;
                float v[8], hi[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int p = 8 * g + u;
                    if (p < kLT) {
                        const uint32_t off = (p & 1) ? hop[p / 2] >> 16 : hop[p / 2] & 0xffffu;
                        v[u] = *reinterpret_cast<const float *>(reinterpret_cast<const char *>(bx) + off);
                    } else {
                        v[u] = vh[p - kLT];
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    hi[u] = to_tf32(v[u]);
                    v[u] -= hi[u];
                }
                tmem_st8(trow + 8 * g, hi);
                tmem_st8(trow + KP + 8 * g, v);
            });
            asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            sync();
            if (gt == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                issue_product<KP>(tmem, smem_u32(smem + lay.b), bar);
            }
            __syncwarp();
            wait_product(bar, phase, A.polls, &s_void[group][parity]);
            phase ^= 1u;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            for_each<KP / 8>([&](auto gc) {
                constexpr int g = decltype(gc)::value;
                uint32_t z[8];
                tmem_ld8(trow + 2 * KP + 8 * g, z);
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                if (g == 0) odd |= __uint_as_float(z[0]) != __uint_as_float(z[0]);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int p = 8 * g + u;
                    if (p < kLT) {
                        const uint32_t off = (p & 1) ? hop[p / 2] >> 16 : hop[p / 2] & 0xffffu;
                        *reinterpret_cast<float *>(reinterpret_cast<char *>(part) + p * kSmallStride * 4 + off) =
                            __uint_as_float(z[u]);
                    } else if (to >> (p - kLT) & 1u) {
                        __stcs(A.scratch + (uint32_t)(ze[i * H + p - kLT] + t), __uint_as_float(z[u]));
                    }
                }
            });
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        }
        sync();
#pragma unroll 2
        for (int r = gt; r < m * nk; r += 128) {
            const int i = r / nk, t = r - i * nk;
            const uint32_t l = __ldg(A.low + lo_k + t);
            const float D = (dlow[l & 63u] + dlow[64 + (l >> 6)]) + bdh[i];
            float s = 0.0f;
#pragma unroll
            for (int o = 0; o < kLT; ++o)
                if (l >> o & 1u) s += part[o * kSmallStride + r];
            y[bbase[i] + t] = fmaf(D, bx[r], s);
        }
        sync();
        // (group-uniform: the flag is next written two items on)
        if (s_void[group][parity]) break;         // once a wait has given up, no more items
        cur = nxt;
    }
    if (odd) atomicOr(&tk->mark, kMarkSplit);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(s_tmem), "r"(kTmemCols) : "memory");
    if (gt == 0 && (s_void[group][0] || s_void[group][1])) report_void(tk);
}

// ---- pair addition --------------------------------------------------------------
constexpr int kAThreads = 128;
constexpr int kARows = 4;                // rows per thread and pass
constexpr int kACtas = 10;               // CTAs per SM

struct AddArgs {
    int omega, N, L, H;
    int lo_off[kLT + 2];
    int ph[kLT + 1];
    int64_t first[kLT + 2];              // number of the class's first word in words
    int c0, c1;                          // classes of this launch
    int64_t zbase[kLT + 1];
    const uint32_t *words;
    const uint16_t *low;
    const uint64_t *binom;
    const float *scratch;
    int first_launch, last_launch;       // of the product
};

// One row term by term, by a warp (its hops over the lanes)
__device__ float row_slow(const AddArgs &A, const float *__restrict__ G, const float *__restrict__ d,
                          const float *__restrict__ x, uint64_t s, float xs)
{
    if (xs != xs) return xs;                      // NaN stays
    const int lane = threadIdx.x & 31, M = A.omega - A.N;
    float D = 0.0f;
    for (int p = lane; p < A.omega; p += 32)
        if (s >> p & 1ull) D += d[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
    float acc = lane == 0 ? D * xs : 0.0f;
    for (int i = lane; i < A.N * M; i += 32) {
        uint64_t wo = s, we = ~s;
        for (int j = i / M; j > 0; --j) wo &= wo - 1;
        for (int j = i % M; j > 0; --j) we &= we - 1;
        const int o = __ffsll((long long)wo) - 1, e = __ffsll((long long)we) - 1;
        uint64_t idx = 0;
        int c = 0;
        for (uint64_t w = s ^ (1ull << o) ^ (1ull << e); w; w &= w - 1)
            idx += __ldg(A.binom + (__ffsll((long long)w) - 1) * kBinomStride + ++c);
        acc = fmaf(G[e * A.omega + o], x[idx], acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// the last CTA sums the partial dot products
__device__ __forceinline__ void finish_add(const AddArgs &A, const DotAcc<float> &dot, Tickets *tk, double *part,
                                           double *dot_out, double *sred, const unsigned ctas)
{
    if (part) {
        const double v = block_reduce(dot, sred);
        if (threadIdx.x == 0) part[blockIdx.x] = v;
    }
    if (!arrive_last(&tk->hx_done, ctas)) return;
    if (A.last_launch && threadIdx.x == 0) tk->mark = 0u;
    if (!part) return;
    double s = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kAThreads) s += __ldcg(part + i);
    s = block_sum(s, sred);
    if (threadIdx.x == 0) *dot_out = A.first_launch ? s : *dot_out + s;
}

// The addition after a marked product (a function and a loop of its own, so that
// the usual ones keep their registers).  An element that cannot be split makes its
// tiles' rows of Z NaN, so exactly the rows that it reaches are not finite (and
// those that overflow anyway): they are formed term by term, the others are as
// usual.  C(24,12) with one such element: 12.3 ms when every row was formed that way.
__device__ __noinline__ void add_marked(const AddArgs &A, const float *__restrict__ G, const float *__restrict__ d,
                                        const float *__restrict__ x, float *__restrict__ y, Tickets *tk, double *part,
                                        double *dot_out, const int cta, const int ctas, const uint32_t *bin, double *sred,
                                        const unsigned mark, const bool tree)
{
    const int lane = threadIdx.x & 31, NB = A.N + 2;
    DotAcc<float> dot;
    int c = A.c0;
    for (int64_t b = A.first[A.c0] + cta; b < A.first[A.c1]; b += ctas) {
        while (b >= A.first[c + 1]) ++c;
        const int ph = A.ph[c], k = A.N - ph;
        const int lo_k = A.lo_off[k], nk = A.lo_off[k + 1] - lo_k;
        const uint32_t h = __ldg(A.words + b);
        uint32_t base = 0;
        float Dh = 0.0f;
        int o = k;
        for (uint32_t w = h; w; w &= w - 1) {
            const int j = __ffs(w) - 1;
            base += bin[j * NB + ++o];
            Dh += d[A.L + j];
        }
        if (tree) {                               // (in the order of the kernel that this one stands in for)
            Dh = h >> lane & 1u ? d[A.L + lane] : 0.0f;
#pragma unroll
            for (int p = 16; p > 0; p >>= 1) Dh += __shfl_xor_sync(0xffffffffu, Dh, p);
        }
        const float *z = A.scratch + A.zbase[k] + (b - A.first[c]) * (int64_t)ph * nk;
#pragma unroll 1
        for (int r0 = threadIdx.x & ~31; r0 < nk; r0 += kAThreads) {      // whole warps
            const bool in = r0 + lane < nk;
            const int r = in ? r0 + lane : nk - 1;
            const float xr = __ldg(x + base + r);
            float acc = k == 0 ? Dh * xr : y[base + r];                   // (no pair removal writes rows with k = 0)
            const float *zr = z + r;
#pragma unroll 4
            for (int a = 0; a < ph; ++a, zr += nk) acc += __ldcs(zr);
            if (mark & kMarkVoid) acc = CUDART_NAN_F;
            const uint64_t s = (uint64_t)h << A.L | __ldg(A.low + lo_k + r);
            const bool again = in && !(mark & kMarkVoid) && !isfinite(acc);
            for (unsigned m = __ballot_sync(0xffffffffu, again); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const float v = row_slow(A, G, d, x, __shfl_sync(0xffffffffu, s, src), __shfl_sync(0xffffffffu, xr, src));
                if (lane == src) acc = v;
            }
            __syncwarp();
            if (!in) continue;
            y[base + r] = acc;
            dot.add(xr, acc);
        }
    }
    finish_add(A, dot, tk, part, dot_out, sred, ctas);
}

// y(h, l) += sum over the pairs a of h of scratch(h, a, l); fused x^T y.  Bound
// by the latency of streaming reads: 16 loads per thread in flight, small CTAs
// so that blocks of very different sizes balance.  Omega=24 (65 MB of scratch,
// mostly in L2): 23 us alone with a cold cache; 25 us before the rows of marked
// products left its loop, 32 us then with 256 threads, 40 us with two rows per thread.
__device__ __forceinline__ void add_blocks(const AddArgs &A, const float *__restrict__ G, const float *__restrict__ d,
                                           const float *__restrict__ x, float *__restrict__ y, Tickets *tk, double *part,
                                           double *dot_out, const int cta, const int ctas)
{
    __shared__ double sred[kAThreads / 32];
    __shared__ uint32_t bin[kMaxHigh * (kMaxHigh + kLT + 1)];   // C(L + p, m), m < N + 2, N < omega
    const int lane = threadIdx.x & 31;
    const int NB = A.N + 2;
    for (int i = threadIdx.x; i < A.H * NB; i += kAThreads)
        bin[i] = (uint32_t)__ldg(A.binom + (A.L + i / NB) * kBinomStride + i % NB);
    const unsigned mark = __ldcg(&tk->mark);
    __syncthreads();
    if (mark) {
        add_marked(A, G, d, x, y, tk, part, dot_out, cta, ctas, bin, sred, mark, true);
        return;
    }
    DotAcc<float> dot;
    int c = A.c0;
    int64_t b = A.first[A.c0] + cta;
    const int64_t end = A.first[A.c1];
    uint32_t hn = b < end ? __ldg(A.words + b) : 0u;
    for (; b < end; b += ctas) {
        while (b >= A.first[c + 1]) ++c;
        const int ph = A.ph[c], k = A.N - ph;
        const int lo_k = A.lo_off[k], nk = A.lo_off[k + 1] - lo_k;
        const uint32_t h = hn;
        if (b + ctas < end) hn = __ldg(A.words + b + ctas);
        const bool occ = h >> lane & 1u;
        uint32_t base = occ ? bin[lane * NB + k + 1 + __popc(h & ((1u << lane) - 1u))] : 0u;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
        const float *z = A.scratch + A.zbase[k] + (b - A.first[c]) * (int64_t)ph * nk;
        float Dh = 0.0f;
        if (k == 0) {                             // no pair removal writes these rows
            Dh = occ ? d[A.L + lane] : 0.0f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) Dh += __shfl_xor_sync(0xffffffffu, Dh, o);
        }
        for (int r0 = threadIdx.x; r0 < nk; r0 += kARows * kAThreads) {
            float acc[kARows], xr[kARows];
            bool in[kARows];
#pragma unroll
            for (int i = 0; i < kARows; ++i) {
                const int r = r0 + i * kAThreads;
                in[i] = r < nk;
                xr[i] = in[i] && (part || k == 0) ? __ldg(x + base + r) : 0.0f;
                acc[i] = k == 0 ? Dh * xr[i] : in[i] ? y[base + r] : 0.0f;
            }
            const float *zr = z + r0;
            int a = 0;
            for (; a + 4 <= ph; a += 4) {
                float v[4][kARows];
#pragma unroll
                for (int u = 0; u < 4; ++u, zr += nk)
#pragma unroll
                    for (int i = 0; i < kARows; ++i) v[u][i] = in[i] ? __ldcs(zr + i * kAThreads) : 0.0f;
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int i = 0; i < kARows; ++i) acc[i] += v[u][i];
            }
            for (; a < ph; ++a, zr += nk)
#pragma unroll
                for (int i = 0; i < kARows; ++i)
                    if (in[i]) acc[i] += __ldcs(zr + i * kAThreads);
#pragma unroll
            for (int i = 0; i < kARows; ++i) {
                const int r = r0 + i * kAThreads;
                if (!in[i]) continue;
                y[base + r] = acc[i];
                if (part) dot.add(xr[i], acc[i]);
            }
        }
    }
    finish_add(A, dot, tk, part, dot_out, sred, ctas);
}

__global__ void __launch_bounds__(kAThreads, kACtas)
add_kernel(const __grid_constant__ AddArgs A, const float *__restrict__ G, const float *__restrict__ d,
           const float *__restrict__ x, float *__restrict__ y, Tickets *tk, const int *__restrict__ skip, double *part,
           double *dot_out)
{
    if (skip && *skip) return;                    // CTA-uniform
    add_blocks(A, G, d, x, y, tk, part, dot_out, blockIdx.x, gridDim.x);
}

// The rows of classes with small blocks (at most kAddSmall rows): one thread per
// row, numbered through the class, where add_kernel has one block per CTA and
// pass.  Omega=34, N=9 (990,000 blocks of 1, 12 and 66 rows): 0.18 ms for these
// rows and 0.22 ms for the others, against 1.68 ms for both in add_kernel; 396 us
// for 1.6 GB is 0.61 of the measured copy rate, the scattered y rows included.
constexpr int kAddSmall = 66;
__global__ void __launch_bounds__(kAThreads, kACtas)
add_small_kernel(const __grid_constant__ AddArgs A, const float *__restrict__ G, const float *__restrict__ d,
                 const float *__restrict__ x, float *__restrict__ y, Tickets *tk, const int *__restrict__ skip,
                 double *part, double *dot_out)
{
    if (skip && *skip) return;                    // CTA-uniform
    __shared__ double sred[kAThreads / 32];
    __shared__ uint32_t bin[kMaxHigh * (kMaxHigh + kLT + 1)];
    __shared__ float dh[kMaxHigh];
    const int NB = A.N + 2;
    for (int i = threadIdx.x; i < A.H * NB; i += kAThreads)
        bin[i] = (uint32_t)__ldg(A.binom + (A.L + i / NB) * kBinomStride + i % NB);
    for (int i = threadIdx.x; i < A.H; i += kAThreads) dh[i] = d[A.L + i];
    const unsigned mark = __ldcg(&tk->mark);
    __syncthreads();
    if (mark) {
        add_marked(A, G, d, x, y, tk, part, dot_out, blockIdx.x, gridDim.x, bin, sred, mark, false);
        return;
    }
    DotAcc<float> dot;
    for (int c = A.c0; c < A.c1; ++c) {
        const int ph = A.ph[c], k = A.N - ph;
        const uint32_t lo_k = A.lo_off[k], nk = A.lo_off[k + 1] - lo_k;
        const int64_t rows = (A.first[c + 1] - A.first[c]) * nk;    // < 2^32
        for (int64_t i = (int64_t)blockIdx.x * kAThreads + threadIdx.x; i < rows; i += (int64_t)gridDim.x * kAThreads) {
            const uint32_t b = (uint32_t)i / nk, r = (uint32_t)i - b * nk;
            const uint32_t h = __ldg(A.words + A.first[c] + b);
            uint32_t base = r;
            float Dh = 0.0f;
            int o = k;
            for (uint32_t w = h; w; w &= w - 1) {
                const int j = __ffs(w) - 1;
                base += bin[j * NB + ++o];
                Dh += dh[j];
            }
            const float xr = part || k == 0 ? __ldg(x + base) : 0.0f;
            float acc = k == 0 ? Dh * xr : y[base];
            const float *z = A.scratch + A.zbase[k] + (int64_t)b * ph * nk + r;
#pragma unroll 4
            for (int a = 0; a < ph; ++a, z += nk) acc += __ldg(z);
            y[base] = acc;
            if (part) dot.add(xr, acc);
        }
    }
    finish_add(A, dot, tk, part, dot_out, sred, gridDim.x);
}

// ---- many problems in one launch ------------------------------------------------
// Each CTA belongs to one problem; it takes blocks from that problem's ticket.
// Bound as the kernels of one problem are, and at the same rate: five problems of
// 650,000 states 107 us for the removal and 29 us for the addition.  (One pair of
// launches per problem, in one to eight parallel branches of the solver's graph,
// was no faster than the row-by-row kernel over all of them: a launch of 250
// blocks is mostly the start of its CTAs.)
struct FacItem {
    RemoveArgs r;
    AddArgs a;
    const float *G, *d;
    Tickets *tk;
    int64_t off;                         // of its vectors
    int p;                               // number of its skip flag
    int ctas_t, ctas_y;
};
static_assert(sizeof(FacItem) % 4 == 0, "copied in words");

__device__ __forceinline__ void copy_item(FacItem &to, const FacItem *from)
{
    for (int i = threadIdx.x; i < (int)(sizeof(FacItem) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(&to)[i] = __ldg(reinterpret_cast<const uint32_t *>(from) + i);
    __syncthreads();
}

template <int KP>
__global__ void __launch_bounds__(Cfg<KP>::kThreads, 2)
remove_batch_kernel(const FacItem *__restrict__ items, const int2 *__restrict__ ctas, const float *x, float *y,
                    const int *__restrict__ skip, int skip_stride)
{
    __shared__ FacItem it;
    const int2 c = ctas[blockIdx.x];
    if (skip[items[c.x].p * skip_stride]) return;   // CTA-uniform
    copy_item(it, items + c.x);
    remove_blocks<KP>(it.r, it.G, it.d, x + it.off, y + it.off, it.tk, it.ctas_t);
}

__global__ void __launch_bounds__(kAThreads, kACtas)
add_batch_kernel(const FacItem *__restrict__ items, const int2 *__restrict__ ctas, const float *x, float *y,
                 const int *__restrict__ skip, int skip_stride)
{
    __shared__ FacItem it;
    const int2 c = ctas[blockIdx.x];
    if (skip[items[c.x].p * skip_stride]) return;   // CTA-uniform
    copy_item(it, items + c.x);
    add_blocks(it.a, it.G, it.d, x + it.off, y + it.off, it.tk, nullptr, nullptr, c.y, it.ctas_y);
}

const void *remove_batch_fn_of(int KP)
{
    return KP == 16   ? (const void *)remove_batch_kernel<16>
           : KP == 24 ? (const void *)remove_batch_kernel<24>
           : KP == 32 ? (const void *)remove_batch_kernel<32>
                      : (const void *)remove_batch_kernel<40>;
}

template <int KP>
const void *remove_fn() { return (const void *)remove_kernel<KP>; }
int padded(int omega)
{
    const int c = omega > kLT ? omega : kLT;
    return c <= 16 ? 16 : (c + 7) / 8 * 8;
}
const void *remove_fn_of(int KP)
{
    return KP == 16 ? remove_fn<16>() : KP == 24 ? remove_fn<24>() : KP == 32 ? remove_fn<32>() : remove_fn<40>();
}
// (up to 12 high orbits there are too few small blocks for a launch of their own)
const void *remove_small_fn_of(int KP)
{
    return KP == 32 ? (const void *)remove_small_kernel<32> : KP == 40 ? (const void *)remove_small_kernel<40> : nullptr;
}
int remove_threads(int KP)
{
    return KP == 16 ? Cfg<16>::kThreads : KP == 24 ? Cfg<24>::kThreads : KP == 32 ? Cfg<32>::kThreads : Cfg<40>::kThreads;
}

}  // namespace

int fac_low(int omega) { return omega < kLT ? omega : kLT; }

bool fac_fits(int omega, int n, int64_t dim)
{
    const int H = omega - fac_low(omega);
    return n >= 1 && n < omega && dim < ((int64_t)1 << 32) && H <= kMaxHigh &&
           layout_r(padded(omega), H, n).total <= kSmemMax;
}

// Where the rows of variant 2 have been at least as exact as row by row in every
// draw (norm of the error against 64-bit rows, removal / rows).  Up to two thirds of
// the orbits occupied (rounded up) everywhere: C(14,7) 0.7 / 2.0e-7, C(24,12) 1.3 /
// 3.2e-7.  Above that from 30000 states on: means of six draws C(24,19) 2.0 / 3.1e-7,
// C(34,30) 2.4 / 3.8e-7; in smaller spaces the mean is lower too (C(22,19) 2.0 /
// 2.6e-7, C(24,20) 2.2 / 2.9e-7, C(30,26) 2.5 / 2.7e-7), but one or two of the six
// draws were higher.
bool fac_exact(int omega, int n, int64_t dim)
{
    return dim >= 30000 || 3 * n <= 2 * omega + 2;
}

// Where variant 2 is taken unasked (FP32, rows / removal, a cold L2 before each):
// C(17,6) 15.7 / 18.5 us, C(18,9) = 48620 18.7 / 20.6 us, C(20,10) = 184756 31 /
// 22.6 us, C(24,12) 215 / 96 us, C(30,15) 16.5 / 6.5 ms, C(34,9) 12.8 / 1.7 ms.  Up
// to two thirds filling (rounded up); above, it is taken on request and by the
// autotuner, which finds it the faster one in large spaces there too: C(22,16) 46 /
// 31 us, C(24,17) 134 / 64 us, C(24,18) 54 / 54 us, C(28,22) 146 / 97 us.
bool fac_pays(int omega, int n, int64_t dim)
{
    return dim >= 60000 && 3 * n <= 2 * omega + 2 && fac_fits(omega, n, dim);
}

// The same line for many problems in one launch, which has its launches and the
// start of its CTAs once for all.  Five problems of 650,000 states, row by row /
// by removal: 224 / 136 us; fourteen of 200,000 to 490,000: 286 / 199 us.  A solve
// of 96 problems of 10 to 22 orbits with the line at 60000 / 15000 / 3000 states:
// 95.5 / 94.5 / 94.7 ms; of twelve of 18 to 22 orbits 86.7 / 84.9 / 84.9 ms; of 96
// of 10 to 14 orbits 11.3 / 11.3 / 12.1 ms.
bool fac_pays_batch(int omega, int n, int64_t dim)
{
    return dim >= 15000 && omega > kLT && 3 * n <= 2 * omega + 2 && fac_fits(omega, n, dim);
}

// classes of words with `pairs` pairs in all, the largest blocks first
static void word_classes(int L, int H, int pairs, WordClasses &C)
{
    int ks[kLT + 1], n = 0;
    for (int k = 0; k <= L; ++k)
        if (pairs - k >= 0 && pairs - k <= H) ks[n++] = k;
    for (int i = 1; i < n; ++i)
        for (int j = i; j > 0 && host_binom(L, ks[j]) > host_binom(L, ks[j - 1]); --j) {
            const int t = ks[j];
            ks[j] = ks[j - 1];
            ks[j - 1] = t;
        }
    C = WordClasses{};
    C.n = n;
    for (int i = 0; i < n; ++i) {
        C.ph[i] = pairs - ks[i];
        C.first[i + 1] = C.first[i] + (int64_t)host_binom(H, pairs - ks[i]);
    }
}

size_t fac_zeros() { return kStride; }

void fac_sizes(int omega, int n, FacPlan &p)
{
    p = FacPlan{};
    p.omega = omega;
    p.n = n;
    p.L = fac_low(omega);
    const int H = omega - p.L;
    WordClasses ct, cy;
    word_classes(p.L, H, n - 1, ct);
    word_classes(p.L, H, n, cy);
    p.nt = ct.first[ct.n];
    p.ny = cy.first[cy.n];
    p.table = (int64_t)(kLT / 2) << p.L;
    int64_t all = 0, most = 0;
    for (int i = 0; i < cy.n; ++i) {
        const int64_t z = (int64_t)host_binom(H, cy.ph[i]) * cy.ph[i] * (int64_t)host_binom(p.L, n - cy.ph[i]);
        all += z;
        if (z > most) most = z;
    }
    p.by_class = all > kScratchAll;
    p.scratch_len = p.by_class ? most : all;
}

cudaError_t fac_build(FacPlan &p, const uint64_t *binom, cudaStream_t st)
{
    p.on = false;
    const int H = p.omega - p.L;
    WordClasses ct, cy;
    word_classes(p.L, H, p.n - 1, ct);
    word_classes(p.L, H, p.n, cy);
    cudaError_t ez = cudaMemsetAsync(p.zeros, 0, sizeof(float) * fac_zeros(), st);
    if (ez != cudaSuccess) return ez;
    hop_table_kernel<<<(unsigned)((p.table + 255) / 256), 256, 0, st>>>(p.L, binom, p.low, p.up);
    high_words_kernel<<<(unsigned)((p.nt + 255) / 256), 256, 0, st>>>(ct, H, binom, p.twords);
    high_words_kernel<<<(unsigned)((p.ny + 255) / 256), 256, 0, st>>>(cy, H, binom, p.ywords);
    count_launches(3);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int KP = padded(p.omega);
    p.smem = layout_r(KP, H, p.n).total;
    e = cudaFuncSetAttribute(remove_fn_of(KP), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e == cudaSuccess && remove_small_fn_of(KP))
        e = cudaFuncSetAttribute(remove_small_fn_of(KP), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
    p.grid_t = 2 * sm_count();                    // two CTAs per SM share its tensor memory
    p.grid_y = kACtas * sm_count();
    p.on = true;
    return cudaSuccess;
}

int64_t fac_partials() { return (int64_t)kACtas * sm_count(); }


static void fill_args(const FacPlan &p, const uint64_t *binom, WordClasses &ct, WordClasses &cy, RemoveArgs &R, AddArgs &A)
{
    const int L = p.L, H = p.omega - L, N = p.n;
    word_classes(L, H, N - 1, ct);
    word_classes(L, H, N, cy);
    R = RemoveArgs{};
    A = AddArgs{};
    R.omega = A.omega = p.omega;
    R.N = A.N = N;
    R.polls = p.polls;
    R.L = A.L = L;
    R.H = A.H = H;
    for (int k = 0; k <= kLT; ++k) {
        R.lo_off[k + 1] = R.lo_off[k] + (int)host_binom(L, k);
        A.lo_off[k + 1] = R.lo_off[k + 1];
    }
    R.words = p.twords;
    R.up = p.up;
    R.low = A.low = p.low;
    R.binom = A.binom = binom;
    R.scratch = p.scratch;
    R.zeros = p.zeros;
    A.scratch = p.scratch;
    A.words = p.ywords;
    for (int i = 0; i < cy.n; ++i) A.ph[i] = cy.ph[i];
    for (int i = 0; i <= cy.n; ++i) A.first[i] = cy.first[i];
    int64_t z = 0;
    for (int i = 0; i < cy.n && !p.by_class; ++i) {
        const int k = N - cy.ph[i];
        R.zbase[k] = A.zbase[k] = z;
        z += (int64_t)host_binom(H, cy.ph[i]) * cy.ph[i] * (int64_t)host_binom(L, k);
    }
}

cudaError_t fac_launch(const FacPlan &p, const uint64_t *binom, const float *G, const float *d, const float *x, float *y,
                       Tickets *tk, cudaStream_t st, const int *skip, const HxDot *dot)
{
    const int L = p.L, H = p.omega - L, N = p.n, KP = padded(p.omega);
    WordClasses ct, cy;
    RemoveArgs R;
    AddArgs A;
    fill_args(p, binom, ct, cy, R, A);
    const void *small_fn = remove_small_fn_of(KP);
    // classes [c0, c1) of t: those of small blocks, at the end, on their own if
    // they are many
    auto remove = [&](int c0, int c1) -> cudaError_t {
        int cs = c1;
        while (cs > c0 && small_fn) {
            const int ph = ct.ph[cs - 1], nt = (int)host_binom(L, N - 1 - ph);
            const int64_t z = R.zbase[N - 1 - ph] + (int64_t)host_binom(H, ph + 1) * (ph + 1) * nt;
            if (nt > kSmallWords || z > (int64_t)UINT32_MAX) break;   // (32-bit offsets into the scratch)
            --cs;
        }
        if (ct.first[c1] - ct.first[cs] < kSmallMin) cs = c1;
        if (cs > c0) {
            R.first = ct.first[c0];
            R.end = ct.first[cs];
            const int64_t grid = p.grid_t < R.end - R.first ? p.grid_t : R.end - R.first;
            const void *args[] = {&R, &G, &d, &x, &y, &tk, &skip};
            const cudaError_t e = cudaLaunchKernel(remove_fn_of(KP), dim3((unsigned)grid), dim3((unsigned)remove_threads(KP)),
                                                   const_cast<void **>(args), p.smem, st);
            if (e != cudaSuccess) return e;
            count_launches(1);
        }
        if (cs == c1) return cudaSuccess;
        SmallArgs S{};
        S.r = R;
        S.n = c1 - cs;
        for (int i = 0; i < S.n; ++i) {
            const int k = N - ct.ph[cs + i];
            const int nt = (int)host_binom(L, k - 1), nk = k <= L ? (int)host_binom(L, k) : 0;
            const int m = kSmallRows / (nt > nk ? nt : nk);
            S.k[i] = k;
            S.m[i] = m < kSmallBlocks ? m : kSmallBlocks;
            S.first[i] = ct.first[cs + i];
            S.end[i] = ct.first[cs + i + 1];
            S.item[i + 1] = S.item[i] + (S.end[i] - S.first[i] + S.m[i] - 1) / S.m[i];
        }
        const int64_t need = (S.item[S.n] + kSmallGroups - 1) / kSmallGroups;
        const int64_t grid = p.grid_t < need ? p.grid_t : need;
        const void *args[] = {&S, &G, &d, &x, &y, &tk, &skip};
        count_launches(1);
        return cudaLaunchKernel(small_fn, dim3((unsigned)grid), dim3(128 * kSmallGroups), const_cast<void **>(args),
                                layout_s(KP, H, N).total, st);
    };
    int left = cy.n;                              // classes of y to go
    A.first_launch = 1;
    auto add_range = [&](int c0, int c1, bool small) -> cudaError_t {
        if (c1 <= c0) return cudaSuccess;
        A.c0 = c0;
        A.c1 = c1;
        A.last_launch = (left -= c1 - c0) == 0;
        const int64_t nb = cy.first[c1] - cy.first[c0];
        const int64_t grid = p.grid_y < nb ? p.grid_y : nb;
        (small ? add_small_kernel : add_kernel)<<<(unsigned)grid, kAThreads, 0, st>>>(
            A, G, d, x, y, tk, skip, dot ? dot->blk_part : nullptr, dot ? dot->out : nullptr);
        A.first_launch = 0;
        count_launches(1);
        return cudaGetLastError();
    };
    auto add = [&](int c0, int c1) -> cudaError_t {
        int cs = c1;
        while (cs > c0 && (int)host_binom(L, N - cy.ph[cs - 1]) <= kAddSmall) --cs;
        if (cy.first[c1] - cy.first[cs] < kSmallMin) cs = c1;
        const cudaError_t e = add_range(c0, cs, false);
        return e != cudaSuccess ? e : add_range(cs, c1, true);
    };
    if (!p.by_class) {
        const cudaError_t e = remove(0, ct.n);
        return e != cudaSuccess ? e : add(0, cy.n);
    }
    // class by class, the low pairs k ascending: the words t with k low pairs give
    // the scratch of the rows with k and the partial y of the rows with k + 1
    for (int k = 0; k <= L; ++k) {
        for (int i = 0; i < ct.n; ++i)
            if (N - 1 - ct.ph[i] == k) {
                const cudaError_t e = remove(i, i + 1);
                if (e != cudaSuccess) return e;
            }
        for (int i = 0; i < cy.n; ++i)
            if (N - cy.ph[i] == k) {
                const cudaError_t e = add(i, i + 1);
                if (e != cudaSuccess) return e;
            }
    }
    return cudaSuccess;
}

size_t fac_item_size() { return sizeof(FacItem); }
int fac_columns(int omega) { return padded(omega); }

void fac_item(const FacPlan &p, const uint64_t *binom, const float *G, const float *d, int64_t off, int number, Tickets *tk,
              int ctas_t, int ctas_y, void *out)
{
    FacItem it{};
    WordClasses ct, cy;
    fill_args(p, binom, ct, cy, it.r, it.a);
    it.r.first = 0;
    it.r.end = p.nt;
    it.a.c0 = 0;
    it.a.c1 = cy.n;
    it.a.first_launch = it.a.last_launch = 1;
    it.G = G;
    it.d = d;
    it.tk = tk;
    it.off = off;
    it.p = number;
    it.ctas_t = ctas_t;
    it.ctas_y = ctas_y;
    std::memcpy(out, &it, sizeof it);
}

cudaError_t fac_batch_launch(const FacBatch &b, const float *x, float *y, cudaStream_t st, const int *skip, int skip_stride)
{
    const FacItem *items = static_cast<const FacItem *>(b.items);
    const void *fn = remove_batch_fn_of(b.columns);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
    const void *args[] = {&items, &b.ctas_t, &x, &y, &skip, &skip_stride};
    e = cudaLaunchKernel(fn, dim3((unsigned)b.grid_t), dim3((unsigned)remove_threads(b.columns)), const_cast<void **>(args),
                         b.smem, st);
    if (e != cudaSuccess) return e;
    add_batch_kernel<<<(unsigned)b.grid_y, kAThreads, 0, st>>>(items, b.ctas_y, x, y, skip, skip_stride);
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace pd
