// ff_gemv.cu -- float-float GEMV Y = A X, its adjoint dX = A^T dY and the
// weight gradient dA = dY X^T, each term a Mul22 and each accumulation an
// Add22 (the paper's operators), plus a binary64 GEMV baseline with the same
// layouts.
//
// Layouts: A is m x n row-major (row stride lda); X, dX are n x k and Y, dY
// are m x k, all column-major (column strides ldx, lddx, ldy, lddy).
//
// ff_gemv: one warp per row, four rows per block (eight where rows are short), a
// tile of up to four right-hand sides per warp, all tiles in one launch.  Lane l walks the row in two-
// column steps (j = 2l + 64t, 16-byte loads of A and of each column of X; single
// columns j = l + 32t on 8-byte access) and keeps one float-float accumulator
// per right-hand side.  The 32 lane accumulators are combined by a shuffle-down
// Add22 tree.
//
// ff_gemv_t: a thread sums one column or two columns of A over one row block in
// order, for a tile of up to four right-hand sides; a block holds several row
// blocks of its columns and adds their sums in row-block order, or the sums go
// to the workspace and a second kernel adds them.
//
// ff_gemv_dA: one thread per column or pair of adjacent columns of dA, its X
// values in registers, the block's rows walked four elements at a time with dY
// staged in shared memory; every element adds its k terms in order from (0, 0).
// Larger k runs on the GEMM kernel.
//
// All three are bound by FP32 issue from two right-hand sides on (28
// instructions per term as Mul22 + Add22) and use the Fast2Sum forms of
// ff_core.cuh (22): the weight gradient checks its operands once, the other
// two, which use each operand pair once, check every product (23) and repeat a
// sum with the full forms when one falls outside their condition.
#include <cmath>
#include <type_traits>

#include "ff_core.cuh"
#include "ff_first_term.cuh"
#include "ff_host.cuh"

namespace {

constexpr int kGBlock = 256;
constexpr int kGWarps = kGBlock / 32;
constexpr int kMaxK = 64;
constexpr int kFWarps = 4;   // rows (one per warp) of a forward block, unless its launch says otherwise

__device__ __forceinline__ float2 shfl_down2(float2 v, int off)
{
    return make_float2(__shfl_down_sync(0xffffffffu, v.x, off), __shfl_down_sync(0xffffffffu, v.y, off));
}

// ---------------------------------------------------------------------------
// Y = A X
// ---------------------------------------------------------------------------
// One lane's sums over its chunks of a row (two values each with VEC, one
// without): chunks lane, lane + 32, ... in order, U of them loaded before they
// are used (with PIPE, the next U of A before these are added).
// FAST uses the Fast2Sum forms and returns true when a product fell outside
// their condition; the caller then repeats the lane's sums with FAST false.
// Chunk numbers are 32-bit within segments of kSegment chunks.
constexpr int64_t kSegment = 1 << 24;

template <int KT, bool VEC, int U, bool PIPE, bool FAST, int LOOP = 1>
__device__ __forceinline__ bool gemv_lane(const float2* __restrict__ Ar, const float2* __restrict__ X, int64_t n,
                                          int64_t ldx, unsigned lane, float2 (&acc)[KT])
{
    using V = std::conditional_t<VEC, float4, float2>;
    const int64_t chunks = VEC ? n >> 1 : n;
    bool bad = false;
    auto term = [&](float2& s, float2 a, float2 x) {
        if (FAST)
            s = ffk::add22_fast(s, ffk::mul22_fast_checked(a, x, bad));
        else
            s = ffk::add22(s, ffk::mul22(a, x));
    };
    auto chunk = [&](float2& s, const V& a, const V& x) {
        term(s, make_float2(a.x, a.y), make_float2(x.x, x.y));
        if constexpr (VEC) term(s, make_float2(a.z, a.w), make_float2(x.z, x.w));
    };
#pragma unroll
    for (int c = 0; c < KT; ++c) acc[c] = make_float2(0.0f, 0.0f);
    for (int64_t s0 = 0; s0 < chunks; s0 += kSegment) {
        const unsigned nch = static_cast<unsigned>(chunks - s0 < kSegment ? chunks - s0 : kSegment);
        const V* Av = reinterpret_cast<const V*>(Ar) + s0;
        const V* Xv = reinterpret_cast<const V*>(X) + s0;
        const int64_t ldv = VEC ? ldx >> 1 : ldx;
        unsigned t = lane;
        if constexpr (U > 1) {
            auto add = [&](const V (&a)[U], unsigned t) {
#pragma unroll
                for (int c = 0; c < KT; ++c) {
                    V x[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) x[u] = __ldg(Xv + c * ldv + (t + 32 * u));
#pragma unroll
                    for (int u = 0; u < U; ++u) chunk(acc[c], a[u], x[u]);
                }
            };
            if constexpr (PIPE) {
                V a[U], b[U];
                bool full = t + 32 * (U - 1) < nch;
                if (full) {
#pragma unroll
                    for (int u = 0; u < U; ++u) a[u] = __ldcs(Av + (t + 32 * u));
                }
#pragma unroll 1
                while (full) {
                    full = t + 32 * (2 * U - 1) < nch;
                    if (full) {
#pragma unroll
                        for (int u = 0; u < U; ++u) b[u] = __ldcs(Av + (t + 32 * (U + u)));
                    }
                    add(a, t);
#pragma unroll
                    for (int u = 0; u < U; ++u) a[u] = b[u];
                    t += 32 * U;
                }
            } else {
#pragma unroll 1
                for (; t + 32 * (U - 1) < nch; t += 32 * U) {
                    V a[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) a[u] = __ldcs(Av + (t + 32 * u));
                    add(a, t);
                }
            }
        }
        if constexpr (U > 2) {   // the rest in pairs, then singly
#pragma unroll 1
            for (; t + 32 < nch; t += 64) {
                const V a0 = __ldcs(Av + t), a1 = __ldcs(Av + (t + 32));
#pragma unroll
                for (int c = 0; c < KT; ++c) {
                    const V x0 = __ldg(Xv + c * ldv + t), x1 = __ldg(Xv + c * ldv + (t + 32));
                    chunk(acc[c], a0, x0);
                    chunk(acc[c], a1, x1);
                }
            }
        }
#pragma unroll LOOP
        for (; t < nch; t += 32) {
            const V a = __ldcs(Av + t);
#pragma unroll
            for (int c = 0; c < KT; ++c) chunk(acc[c], a, __ldg(Xv + c * ldv + t));
        }
    }
    return bad;
}

// One level of the shuffle-down tree for two sums at once: lanes with bit `off`
// clear combine p with that of lane + off, the others q with that of lane -
// off, lower lane first in both.
__device__ __forceinline__ float2 tree_pair(float2 p, float2 q, int lane, int off)
{
    const bool up = (lane & off) != 0;
    const float2 mine = up ? q : p, give = up ? p : q;
    const float2 got = make_float2(__shfl_xor_sync(0xffffffffu, give.x, off), __shfl_xor_sync(0xffffffffu, give.y, off));
    return ffk::add22_fast(up ? got : mine, up ? mine : got);
}

// The lanes' KT sums combined by the shuffle-down Add22 tree (offsets 16 .. 1)
// and stored.  Two or more sums share the levels: each halves the lanes that
// hold one sum, so four sums take 6 additions per lane instead of 20 (16000 x
// 64, k = 64: 181 -> 134 us).
template <int KT>
__device__ __forceinline__ void gemv_tree_store(const float2 (&acc)[KT], int lane, float2* __restrict__ Yr, int64_t ldy)
{
    static_assert(KT <= 4, "two shared levels");
    float2 v;
    int c = 0, low = 32;   // lanes with lane % low == 0 end with sum c
    if constexpr (KT == 1) {
        v = acc[0];
    } else {
        const float2 p = tree_pair(acc[0], acc[1], lane, 16);
        c = lane >> 4;
        low = 16;
        v = p;
        if constexpr (KT > 2) {
            const float2 q = tree_pair(acc[2], acc[KT - 1], lane, 16);
            v = tree_pair(p, q, lane, 8);
            c += (lane >> 2) & 2;
            low = 8;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        if (off < low) v = ffk::add22_fast(v, shfl_down2(v, off));
    if (lane % low == 0 && c < KT) Yr[c * ldy] = ffk::ff_overflow_lo(v);
}

template <int KT, bool VEC, int U, bool PIPE, int LOOP>
__device__ __forceinline__ void gemv_row(const float2* __restrict__ Ar, const float2* __restrict__ X, int64_t n,
                                         int64_t ldx, float2* __restrict__ Yr, int64_t ldy)
{
    const unsigned lane = threadIdx.x & 31;
    float2 acc[KT];
    if (gemv_lane<KT, VEC, U, PIPE, true, LOOP>(Ar, X, n, ldx, lane, acc))
        gemv_lane<KT, VEC, 1, false, false>(Ar, X, n, ldx, lane, acc);
    gemv_tree_store(acc, static_cast<int>(lane), Yr, ldy);
}

// blockIdx.x: rows, one per warp; blockIdx.y: tile of right-hand sides, the
// first `na` of them KA wide, the others KB wide.
template <int KA, int KB, bool VEC, int U, bool PIPE, int MINB, int WARPS, int LOOP>
__global__ void __launch_bounds__(32 * WARPS, MINB)
gemv_kernel(const float2* __restrict__ A, int64_t m, int64_t n, int64_t lda, const float2* __restrict__ X,
            int64_t ldx, float2* __restrict__ Y, int64_t ldy, int na)
{
    const unsigned zero = ffk::prior_kernel_done();
    const int64_t r = static_cast<int64_t>(blockIdx.x + zero) * WARPS + (threadIdx.x >> 5);
    if (r >= m) return;
    const int y = blockIdx.y;
    X += zero;
    if (KA == KB || y < na) {
        const int64_t c0 = static_cast<int64_t>(y) * KA;
        gemv_row<KA, VEC, U, PIPE, LOOP>(A + r * lda, X + c0 * ldx, n, ldx, Y + c0 * ldy + r, ldy);
    } else {
        const int64_t c0 = static_cast<int64_t>(na) * KA + static_cast<int64_t>(y - na) * KB;
        gemv_row<KB, VEC, U, PIPE, LOOP>(A + r * lda, X + c0 * ldx, n, ldx, Y + c0 * ldy + r, ldy);
    }
}

// Tiles of right-hand sides: `na` of width ka, then `nb` of width kb, all in
// one launch.  Four wide is the best trade of operand reuse against registers
// (16384^2, k = 8: 1.48e12 terms/s forward in tiles of four, 1.42e12 in one of
// eight; adjoint 1.43e12 against 1.24e12); 5 and 6 split into threes and a two.
struct TileSplit {
    int ka, kb;
    int64_t na, nb;
};

inline TileSplit split_tiles(int64_t k)
{
    if (k == 1) return {1, 1, 1, 0};
    if (k == 2) return {2, 1, 1, 0};
    if (k == 3) return {3, 2, 1, 0};
    if (k == 5) return {3, 2, 1, 1};
    if (k == 6) return {3, 2, 2, 0};
    const int64_t threes = (4 - k % 4) % 4;
    return {4, 3, (k - 3 * threes) / 4, threes};
}

inline int f64_tile_for(int64_t k) { return k >= 16 ? 16 : k >= 8 ? 8 : k >= 4 ? 4 : k >= 2 ? 2 : 1; }

template <int KA, int KB, bool VEC, int U, bool PIPE, int MINB, int WARPS = kFWarps, int LOOP = 1>
ff_status launch_gemv(const TileSplit& t, const float2* A, int64_t m, int64_t n, int64_t lda, const float2* X,
                      int64_t ldx, float2* Y, int64_t ldy, cudaStream_t s)
{
    const dim3 grid(static_cast<unsigned>((m + WARPS - 1) / WARPS), static_cast<unsigned>(t.na + t.nb));
    return ffh::launch_kernel(&gemv_kernel<KA, KB, VEC, U, PIPE, MINB, WARPS, LOOP>, grid, 32 * WARPS, s, A, m, n, lda, X,
                              ldx, Y, ldy, static_cast<int>(t.na));
}

// Chunks in flight (U) and the register budget that lets the compiler issue
// their loads together (MINB) were chosen by sweeps over 300 x 1000 to 32768^2;
// left to itself the compiler took fewer registers and spread the loads out
// (16383^2, k = 1: 344 us; 302 with the budget below).  On 16-byte access a
// single right-hand side over many rows, bound by HBM, runs best with four
// chunks and the next four of A ahead (32768^2: 1.16 ms = 7.4 TB/s, 1.21 with
// eight and none ahead; 2000 rows and fewer prefer the latter: 300 x 20000 31.5
// -> 21.4 us).
// Short rows never fill four or eight chunks in flight, and serve better with one or
// two, few registers and so twice the warps, in blocks of eight: 65536 rows, k = 1, n =
// 64 15.2 -> 14.4 us, 100 22.2 -> 18.4, 200 41.7 -> 28.9, 1000 90 -> 82; odd rows n = 33, k = 5
// 54.7 -> 41.9, n = 101, k = 2 32.4 -> 26.3, n = 201, k = 5 110 -> 87.  The lines lie where the
// sweep crosses: fewer rows than 16 a quarter gain nothing, 2500 x 512 3.4 -> 3.7.  The
// same kernel takes 8 to 12 rows a quarter at any length, where the pipelined one
// starts a second wave that it does not fill (5000 x 16384: 128 -> 110 us; 8000 156, 152).
// Few rows leave SMs idle under a wide tile, since a row is one warp's: below
// one warp per SM quarter the right-hand sides get a warp each (400 x 2000, k =
// 4: 6.9 us in pairs, 5.7 singly), below two they go in pairs (800 x 2000, k = 4:
// 10.5 us in fours, 8.1).  Tiles of four take four chunks on rows below 8192
// values (6000^2, k = 8: 208 us, 213 with eight) and eight above (16384^2: 1.42
// ms, 1.44 with four).
template <bool VEC>
ff_status gemv_forward(const float2* A, int64_t m, int64_t n, int64_t lda, const float2* X, int64_t ldx, int64_t k,
                       float2* Y, int64_t ldy, int sm_count, cudaStream_t s)
{
    const TileSplit t = split_tiles(k);
    const int64_t warps = m * ((k + 3) / 4);
    const int64_t quarters = 4 * static_cast<int64_t>(sm_count);
    if constexpr (VEC) {
        if (k == 1 && n <= 128 && m >= 16 * quarters)
            return launch_gemv<1, 1, true, 1, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        if (k == 1 && n > 128 && m > 8 * quarters && (m <= 12 * quarters || n <= 400 || (n <= 2048 && m >= 24 * quarters)))
            return launch_gemv<1, 1, true, 1, false, 0, 8, 2>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        if (k == 1 && m >= 4 * quarters)
            return launch_gemv<1, 1, true, 4, true, 0>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    } else if (n <= 128 && m >= 16 * quarters) {
        if (k == 1) return launch_gemv<1, 1, false, 1, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        if (k == 2) return launch_gemv<2, 1, false, 1, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        if (t.ka == 3) return launch_gemv<3, 2, false, 1, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        return launch_gemv<4, 3, false, 1, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    } else if (n <= 256 && k == 1 && m >= 16 * quarters) {
        return launch_gemv<1, 1, false, 4, false, 5, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    } else if (n <= 256 && m >= 64 * quarters) {
        if (k == 2) return launch_gemv<2, 1, false, 2, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        if (t.ka == 3) return launch_gemv<3, 2, false, 2, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
        return launch_gemv<4, 3, false, 2, false, 0, 8>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    }
    if (k == 1 || warps < quarters)
        return launch_gemv<1, 1, VEC, 8, false, 4>({1, 1, k, 0}, A, m, n, lda, X, ldx, Y, ldy, s);
    if (k == 2 || warps < 2 * quarters)
        return launch_gemv<2, 1, VEC, VEC ? 4 : 8, false, VEC ? 6 : 4>({2, 1, k / 2, k % 2}, A, m, n, lda, X, ldx, Y,
                                                                       ldy, s);
    if (t.ka == 3) return launch_gemv<3, 2, VEC, VEC ? 4 : 8, false, 6>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    if (VEC && n < 8192) return launch_gemv<4, 3, VEC, 4, false, 6>(t, A, m, n, lda, X, ldx, Y, ldy, s);
    return launch_gemv<4, 3, VEC, 8, false, VEC ? 4 : 6>(t, A, m, n, lda, X, ldx, Y, ldy, s);
}

// ---------------------------------------------------------------------------
// dX = A^T dY
// ---------------------------------------------------------------------------
// A thread's columns: two adjacent ones (16-byte access), one, or two `apart`
// columns from one another (8-byte access; they share the loads of dY).
enum Columns { kAdjacent, kSingle, kApart };

// One thread's sums of its columns over the rows [r0, r1) in order, R rows
// loaded before they are added.  FAST uses the Fast2Sum forms and returns
// true when a product fell outside their condition; the caller then repeats
// the sums with FAST false.
template <int KT, Columns C, int R, bool FAST>
__device__ __forceinline__ bool gemv_t_sums(const float2* __restrict__ Aj, int apart, int64_t lda,
                                            const float2* __restrict__ dY, int64_t lddy, int64_t r0, int64_t r1,
                                            float2 (&acc)[KT][C == kSingle ? 1 : 2])
{
    constexpr int E = C == kSingle ? 1 : 2;
    using V = std::conditional_t<E == 2, float4, float2>;
    bool bad = false;
    auto term = [&](float2& s, float2 a, float2 d) {
        if (FAST)
            s = ffk::add22_fast(s, ffk::mul22_fast_checked(a, d, bad));
        else
            s = ffk::add22(s, ffk::mul22(a, d));
    };
    auto row = [&](float2 (&s)[E], const V& a, float2 d) {
        term(s[0], make_float2(a.x, a.y), d);
        if constexpr (E == 2) term(s[1], make_float2(a.z, a.w), d);
    };
    auto load = [&](int64_t r) {
        const float2* p = Aj + r * lda;
        if constexpr (C == kApart) {
            const float2 a = __ldcs(p), b = __ldcs(p + apart);
            return make_float4(a.x, a.y, b.x, b.y);
        } else {
            return __ldcs(reinterpret_cast<const V*>(p));
        }
    };
#pragma unroll
    for (int c = 0; c < KT; ++c)
#pragma unroll
        for (int e = 0; e < E; ++e) acc[c][e] = make_float2(0.0f, 0.0f);
    int64_t r = r0;
#pragma unroll 1
    for (; r + R <= r1; r += R) {
        V a[R];
#pragma unroll
        for (int q = 0; q < R; ++q) a[q] = load(r + q);
#pragma unroll
        for (int c = 0; c < KT; ++c)
#pragma unroll
            for (int q = 0; q < R; ++q) row(acc[c], a[q], __ldg(dY + c * lddy + r + q));
    }
    if (R > 1 && r < r1) {   // the last R - 1 rows at most, loaded together
        V a[R];
#pragma unroll
        for (int q = 0; q < R - 1; ++q)
            if (r + q < r1) a[q] = load(r + q);
#pragma unroll
        for (int c = 0; c < KT; ++c)
#pragma unroll
            for (int q = 0; q < R - 1; ++q)
                if (r + q < r1) row(acc[c], a[q], __ldg(dY + c * lddy + r + q));
    }
    return bad;
}

// The full forms, out of line: inlined, they took registers from the fast ones as
// soon as they loaded more than one row ahead (8192^2, k = 1, pairs that are not
// normalised: 246 us with one row, 171 with four; float-float operands 0.3% faster).
// A check for them within the fast loops cost those 4 to 7%.
template <int KT, Columns C, int R>
__device__ __noinline__ void gemv_t_sums_full(const float2* Aj, int apart, int64_t lda, const float2* dY, int64_t lddy,
                                              int64_t r0, int64_t r1, float2 (*sums)[C == kSingle ? 1 : 2])
{
    constexpr int E = C == kSingle ? 1 : 2;
    float2 acc[KT][E];
    gemv_t_sums<KT, C, R, false>(Aj, apart, lda, dY, lddy, r0, r1, acc);
#pragma unroll
    for (int c = 0; c < KT; ++c)
#pragma unroll
        for (int e = 0; e < E; ++e) sums[c][e] = acc[c][e];
}

// The block's tile of KT right-hand sides; see gemv_t_kernel.
template <int KT, Columns C, int R>
__device__ __forceinline__ void gemv_t_tile(const float2* __restrict__ A, int64_t m, int64_t n, int64_t lda,
                                            const float2* __restrict__ dY, int64_t lddy, int64_t rpb, int64_t nrb,
                                            int cx, float2* __restrict__ out, int64_t out_ld, int64_t rb_stride,
                                            float2 (*part)[kGBlock], unsigned zero)
{
    const int shift = 31 - __clz(cx);   // cx is a power of two
    const int tx = threadIdx.x & (cx - 1);
    const int ty = threadIdx.x >> shift;
    const int rg = kGBlock >> shift;
    constexpr int E = C == kSingle ? 1 : 2;
    const int64_t j = static_cast<int64_t>(blockIdx.x + zero) * cx * E + (C == kAdjacent ? 2 * tx : tx);   // first column
    const int apart = C == kAdjacent ? 1 : cx;   // to the second one
    const bool second = C == kAdjacent || j + apart < n;
    const int64_t rb = static_cast<int64_t>(blockIdx.y + zero) * rg + ty;
    const int64_t r0 = rb * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;
    float2 acc[KT][E];
    const bool active = j < n && rb < nrb;
    const int step = second ? apart : 0;
    if (active && gemv_t_sums<KT, C, R, true>(A + j, step, lda, dY, lddy, r0, r1, acc)) {
        if constexpr (R > 2) {
            float2 sums[KT][E];
            gemv_t_sums_full<KT, C, 4>(A + j, step, lda, dY, lddy, r0, r1, sums);
#pragma unroll
            for (int c = 0; c < KT; ++c)
#pragma unroll
                for (int e = 0; e < E; ++e) acc[c][e] = sums[c][e];
        } else {
            gemv_t_sums<KT, C, 1, false>(A + j, step, lda, dY, lddy, r0, r1, acc);
        }
    }
    if (rg == 1 || gridDim.y > 1) {
        if (!active) return;
        float2* o = out + rb * rb_stride + j;
#pragma unroll
        for (int c = 0; c < KT; ++c) {
            o[c * out_ld] = ffk::ff_overflow_lo(acc[c][0]);
            if constexpr (E == 2)
                if (second) o[c * out_ld + apart] = ffk::ff_overflow_lo(acc[c][1]);
        }
        return;
    }
    if (active) {
#pragma unroll
        for (int c = 0; c < KT; ++c)
#pragma unroll
            for (int e = 0; e < E; ++e) part[c * E + e][threadIdx.x] = acc[c][e];
    }
    __syncthreads();
    if (j >= n) return;
    for (int w = ty; w < KT * E; w += rg) {   // the thread's column w % E of right-hand side w / E
        if (w % E && !second) continue;
        float2 v = part[w][tx];
#pragma unroll 4
        for (int b = 1; b < nrb; ++b) v = ffk::add22_fast(v, part[w][b * cx + tx]);
        out[(w / E) * out_ld + j + (w % E) * apart] = ffk::ff_overflow_lo(v);
    }
}

// Grid: x groups of cx columns or column pairs, y groups of row
// blocks, z tiles of right-hand sides, the first `na` KA wide and the others
// KB.  A block is cx columns wide and 256 / cx row blocks high: thread (tx, ty)
// sums row block blockIdx.y * (256 / cx) + ty.  With one group of several row
// blocks the block adds its row blocks' sums in order through shared memory
// and writes dX; otherwise thread sums go to out[rb * rb_stride + c * out_ld +
// j] (dX itself when there is a single row block, else the workspace that
// gemv_t_combine reads).
template <int KA, int KB, Columns C, int R, int MINB>
__global__ void __launch_bounds__(kGBlock, MINB)
gemv_t_kernel(const float2* __restrict__ A, int64_t m, int64_t n, int64_t lda, const float2* __restrict__ dY,
              int64_t lddy, int64_t rpb, int64_t nrb, int cx, float2* __restrict__ out, int64_t out_ld,
              int64_t rb_stride, int na)
{
    __shared__ float2 part[KA * (C == kSingle ? 1 : 2)][kGBlock];
    const unsigned zero = ffk::prior_kernel_done();
    const int z = blockIdx.z;
    if (KA == KB || z < na) {
        const int64_t c0 = static_cast<int64_t>(z) * KA;
        gemv_t_tile<KA, C, R>(A, m, n, lda, dY + c0 * lddy, lddy, rpb, nrb, cx, out + c0 * out_ld, out_ld, rb_stride,
                              part, zero);
    } else {
        const int64_t c0 = static_cast<int64_t>(na) * KA + static_cast<int64_t>(z - na) * KB;
        gemv_t_tile<KB, C, R>(A, m, n, lda, dY + c0 * lddy, lddy, rpb, nrb, cx, out + c0 * out_ld, out_ld, rb_stride,
                              part, zero);
    }
}

// dX[c, j] = ws[0][c][j] (+) ws[1][c][j] (+) ... in row-block order.
__global__ void __launch_bounds__(kGBlock)
gemv_t_combine(const float2* __restrict__ ws, int64_t n, int64_t k, int64_t nrb, float2* __restrict__ dX,
               int64_t lddx)
{
    const int64_t idx = static_cast<int64_t>(blockIdx.x + ffk::prior_kernel_done()) * kGBlock + threadIdx.x;
    if (idx >= n * k) return;
    const int64_t c = idx / n, j = idx - c * n;
    float2 acc = ws[c * n + j];
#pragma unroll 8
    for (int64_t rb = 1; rb < nrb; ++rb) acc = ffk::add22_fast(acc, __ldg(ws + (rb * k + c) * n + j));
    dX[c * lddx + j] = ffk::ff_overflow_lo(acc);
}

// How the adjoint is cut: blocks cx columns (or column pairs: adjacent ones on
// 16-byte access, `pairs` apart on 8-byte access) wide and 256 / cx row blocks
// high, gy of them down the rows, right-hand sides in tiles of 1 (wide false)
// or as split_tiles says.
struct AdjointPlan {
    bool wide, pairs;
    int cx;
    int64_t gy, nrb, rpb;
};

// Row blocks for at most `want` of them: nrb blocks of rpb = ceil(m / nrb)
// rows, none empty.
inline void cut_rows(int64_t m, int64_t want, int64_t* nrb, int64_t* rpb)
{
    const int64_t w = want < m ? want : (m > 0 ? m : 1);
    *rpb = (m + w - 1) / w;
    *nrb = *rpb > 0 ? (m + *rpb - 1) / *rpb : 1;
}

// Rows of A a thread loads before it adds them: the fewer terms a row gives,
// the more rows must be in flight to cover the load latency.
inline int adjoint_rows(const AdjointPlan& p, int ka, int64_t k, bool vec)
{
    if (k == 1 && p.gy > 1) return 16;
    return ka <= 2 || !(vec || p.pairs) ? 8 : 4;
}

// Modelled cycles of a cut, fitted to sweeps of all cuts of 619 shapes (64^2 to
// 16384^2, tall and wide, down to 2 rows and up to 10^6 columns, k = 1-64, even and
// odd rows; of the cuts with a short enough chain it picks one within 1.2% of the
// best measured on average, at worst 25%): FP32 issue of the SM with the most
// blocks; memory traffic (bytes per cycle of the L2, or of HBM beyond it; short row
// segments touch more sectors than they use, and more L1 lines per load); a part-
// filled last wave; the latency of the rows loaded together (single columns in
// wide tiles wait for more of them); and the ordered combination, through shared
// memory, which every wave of blocks pays, so that a matrix wide enough to fill the
// device is cut into few row blocks (16 x 1000000, k = 16: 290 -> 196 us, 48 x 1000000, k =
// 5 290 -> 186, 100 x 100001, k = 5 67 -> 46, where it counted for three waves at most),
// or by a second launch over the workspace.
double adjoint_cycles(const AdjointPlan& p, int64_t m, int64_t n, int64_t k, bool vec, int sm_count)
{
    const TileSplit t = p.wide ? split_tiles(k) : TileSplit{1, 1, k, 0};
    const int e = vec || p.pairs ? 2 : 1;
    const int64_t cols = (n + e - 1) / e;
    const int64_t z = t.na + t.nb;
    const int rows = adjoint_rows(p, t.ka, k, vec);
    const double blocks = static_cast<double>((cols + p.cx - 1) / p.cx) * static_cast<double>(p.gy * z);
    const double resident = static_cast<double>(sm_count) * (t.ka >= 2 || rows == 16 ? 3 : 4);
    const double waves = blocks / resident;
    double per = std::ceil(blocks / sm_count);   // blocks of the fullest SM
    double over = 1.0;                           // and how far that is above the mean
    if (waves > 1.0) {
        const double part = waves - std::floor(waves);
        over = (std::floor(waves) + (part > 0.0 ? 0.29 + 0.71 * part : 0.0)) / waves;
        per = over * blocks / sm_count;
    }
    const double issue = per * 2.0 * p.rpb * t.ka * e * (24.5 + (vec ? 0.0 : p.pairs ? 1.0 : 3.2));
    const double bytes = 8.0 * m * n * z * (1.0 + (vec ? 23.0 : p.pairs ? 32.0 : 16.0) / (8.0 * p.cx * e));
    // 128-byte lines per warp and row: of A, and one of dY per row block and
    // right-hand side
    const double rbw = p.cx < 32 ? 32.0 / p.cx : 1.0;
    const double l1 = 0.46 * per * 8.0 * p.rpb * (std::fmax(rbw * (vec ? 1.0 : 1.4), 2.0 * e) + t.ka * rbw);
    const double mem = std::fmax(l1, over * bytes / (8.0 * m * n > 100e6 ? 3800.0 : 6000.0) + 8.0 * n * k / 6000.0);
    const double rounds = 1.0 + 0.36 * (std::fmin(std::ceil(waves), 3.0) - 1.0);
    double c = std::fmax(issue, mem) + 0.24 * std::fmin(issue, mem) +
               rounds * (464.0 * ((p.rpb + rows - 1) / rows) + 1590.0) + (e == 1 ? 50.0 * (t.ka - 1) * rows : 0.0);
    if (p.gy > 1)
        c += 14000.0 + 350.0 * p.nrb + 16.0 * p.nrb * n * k / 3800.0;
    else if (p.nrb > 1)
        c += 700.0 + 59.0 * p.nrb + std::fmax(waves - 0.5, 0.0) * (2000.0 + 40.0 * p.nrb);
    return c;
}

// The longest chain of additions behind one result that a cut may have: rows of a
// row block plus row blocks.  The error of a sum grows with it, so time alone does
// not choose.  The limit is a tenth above what row blocks of at least 32 rows, at
// most 64 of them, give (about the least any cut reaches, 2 sqrt(m), up to 4096
// rows): a tenth is 5% of the error, and without it the powers of two that cuts
// come in miss the limit by a hair.  By time alone 1035 x 4196, k = 13 was cut into 4
// blocks of 259 rows, 1.4 times the RMS error of 32 blocks of 33.
double longest_chain(int64_t m)
{
    int64_t blocks = m / 32;
    blocks = blocks < 1 ? 1 : blocks > 64 ? 64 : blocks;
    return 1.1 * static_cast<double>(blocks + (m + blocks - 1) / blocks);
}

// The cut with the least modelled time and no longer chain than that.  Against column groups of 256 and at
// most 64 row blocks in two launches of eight right-hand sides each, before:
// 32768^2, k = 16: 13.8 -> 11.7 ms (with the Fast2Sum forms); 1024^2: 12.6 ->
// 5.1 us; 10000 x 100, k = 3: 41 -> 14 us; 2001 x 3001, k = 5: 51 -> 32 us.
AdjointPlan search_adjoint_plan(int64_t m, int64_t n, int64_t k, bool vec, int sm_count)
{
    AdjointPlan best{true, false, kGBlock, 1, 1, m > 0 ? m : 0};
    if (m < 1 || n < 1) return best;
    // On 8-byte access a thread takes two columns apart, which share the loads of
    // dY, where the matrix gives every thread enough to do: 8191^2, k = 2 141 -> 126
    // us, 4000 x 6001, k = 5 123 -> 110, 12001^2, k = 1 190 -> 176.  Smaller or
    // narrower ones lose more to the halved number of threads (2001 x 3001, k = 5 29
    // -> 34, 3333 x 401 11.8 -> 12.7, 1024 x 1025, k = 64 57 -> 60), unless dX alone
    // has enough columns for all of them (4 x 50001, k = 16 7.0 -> 5.3).
    const double values = static_cast<double>(m) * n;
    const bool pairs = !vec && n >= 1024 && ((values >= 2e6 && values * k >= 64e6) || static_cast<double>(n) * k >= 2e5);
    const double chain = longest_chain(m);
    double least = -1.0;
    auto consider = [&](int cx, int64_t gy, bool wide) {
        AdjointPlan p{};
        p.cx = cx;
        const int64_t rg = kGBlock / cx;
        cut_rows(m, rg * gy, &p.nrb, &p.rpb);
        if (static_cast<double>(p.rpb + p.nrb) > chain) return;
        p.gy = (p.nrb + rg - 1) / rg;
        p.pairs = pairs;
        p.wide = wide;
        const double c = adjoint_cycles(p, m, n, k, vec, sm_count);
        if (least < 0.0 || c < least) {
            least = c;
            best = p;
        }
    };
    const int widths = k > 1 ? 2 : 1;
    for (int cx = 2; cx <= kGBlock; cx *= 2)
        for (int w = 0; w < widths; ++w) consider(cx, 1, w == 1);
    // Two launches cost more than a short sum takes in one.  Of their cuts only those
    // that just fill a number of waves are tried: of 4000 shapes 9 would take another
    // one, for at most 7%, and the search is 5 times as fast.
    const int64_t most = m / 2 < 64 ? m / 2 : 64;
    if (most < 2 || (least >= 0.0 && least <= 14000.0)) return best;
    const int64_t width = vec || pairs ? 256 : 128;
    for (int w = 0; w < widths; ++w) {
        const TileSplit t = w == 1 ? split_tiles(k) : TileSplit{1, 1, k, 0};
        const int64_t blocks = (n + width - 1) / width * (t.na + t.nb);
        const int64_t resident = static_cast<int64_t>(sm_count) * (t.ka >= 2 || k == 1 ? 3 : 4);
        for (int64_t gy = 1; gy < most;) {
            const int64_t waves = ((gy + 1) * blocks + resident - 1) / resident;
            gy = waves * resident / blocks;
            if (gy > most) gy = most;
            consider(128, gy, w == 1);
        }
    }
    return best;
}

struct AdjointPlans {
    AdjointPlan access8, access16;
};

// The plans of a call's sizes.  A search takes 0.2 to 1 us and a call asks for its
// plan several times (workspace size, for both access widths, then the launch):
// each host thread keeps those of the last sizes, four to a set.
const AdjointPlans& adjoint_plans(int64_t m, int64_t n, int64_t k, int sm_count)
{
    struct Entry {
        int64_t m, n, k;
        int sm_count;   // 0: empty
        AdjointPlans plans;
    };
    constexpr unsigned kSets = 16, kWays = 4;
    static thread_local Entry kept[kSets][kWays];
    static thread_local unsigned char oldest[kSets];
    const uint64_t h = (static_cast<uint64_t>(m) * 0x9e3779b97f4a7c15ull + static_cast<uint64_t>(n)) * 0xc2b2ae3d27d4eb4full +
                       static_cast<uint64_t>(k) * 0x165667b19e3779f9ull;
    const unsigned set = static_cast<unsigned>((h >> 48) % kSets);
    for (const Entry& e : kept[set])
        if (e.m == m && e.n == n && e.k == k && e.sm_count == sm_count) return e.plans;
    Entry& e = kept[set][oldest[set]++ % kWays];
    e = Entry{m, n, k, sm_count, {search_adjoint_plan(m, n, k, false, sm_count), search_adjoint_plan(m, n, k, true, sm_count)}};
    return e.plans;
}

inline const AdjointPlan& adjoint_plan(int64_t m, int64_t n, int64_t k, bool vec, int sm_count)
{
    const AdjointPlans& p = adjoint_plans(m, n, k, sm_count);
    return vec ? p.access16 : p.access8;
}

template <int KA, int KB, Columns C, int R, int MINB>
ff_status launch_adjoint(const AdjointPlan& p, const TileSplit& t, const float2* A, int64_t m, int64_t n, int64_t lda,
                         const float2* dY, int64_t lddy, float2* out, int64_t out_ld, int64_t rb_stride,
                         cudaStream_t s)
{
    const int64_t width = static_cast<int64_t>(p.cx) * (C == kSingle ? 1 : 2);
    const dim3 grid(static_cast<unsigned>((n + width - 1) / width), static_cast<unsigned>(p.gy),
                    static_cast<unsigned>(t.na + t.nb));
    return ffh::launch_kernel(&gemv_t_kernel<KA, KB, C, R, MINB>, grid, kGBlock, s, A, m, n, lda, dY, lddy, p.rpb, p.nrb,
                              p.cx, out, out_ld, rb_stride, static_cast<int>(t.na));
}

// ---------------------------------------------------------------------------
// dA = dY X^T.  Every element accumulates its k terms Mul22(dY[r, c], X[j, c])
// in order c = 0 .. k-1 from (0, 0), so the result is the oracle's
// left-to-right sum bit for bit.  Up to max_dA right-hand sides run here; larger k
// runs as the matrix product op(dY) X on the GEMM kernel (the same terms in the same
// order).
// ---------------------------------------------------------------------------

// Rows per shared-memory chunk of dY (a multiple of four).
constexpr int kTChunk = 128;

// One thread holds E adjacent columns (two with 16-byte access along the rows
// of dA, else one) and their KT values of X; block row y takes the rows [y rpb,
// (y + 1) rpb), 4 / E at a time, so a thread forms four elements per step.  The
// block stages the dY values of kTChunk rows at a time in shared memory, where
// one 16-byte read gives two rows of one right-hand side.  Every element is
// Add22((0, 0), term_0), then Add22 of terms 1 .. KT-1, in order.
// The chunk's dY and the threads' X are checked once, in the staging barrier:
// a chunk whose values are all normalised takes the Fast2Sum forms, any other the
// full ones; the first of several steps from (0, 0) takes two additions either way,
// since a finite product is normalised whatever its operands are.
// Threads past the last column work on the last one and do not store, so that
// every thread reaches the barriers.
template <int KT, int E>
__global__ void __launch_bounds__(kGBlock)
gemv_dA_small_kernel(const float2* __restrict__ dY, int64_t m, int64_t lddy, const float2* __restrict__ X, int64_t n,
                     int64_t ldx, float2* __restrict__ dA, int64_t ldda, int64_t rpb)
{
    using V = std::conditional_t<E == 2, float4, float2>;
    constexpr int RS = 4 / E;   // rows per step
    __shared__ __align__(16) float2 sdy[KT][kTChunk];
    const unsigned zero = ffk::prior_kernel_done();
    const int64_t j_raw = (static_cast<int64_t>(blockIdx.x + zero) * kGBlock + threadIdx.x) * E;
    const bool store = j_raw < n;
    const int64_t j = store ? j_raw : n - E + zero;
    float2 x[KT][E];
    bool okx = true;
#pragma unroll
    for (int c = 0; c < KT; ++c) {
        const V v = __ldg(reinterpret_cast<const V*>(X + c * ldx + j));
        x[c][0] = make_float2(v.x, v.y);
        if constexpr (E == 2) x[c][1] = make_float2(v.z, v.w);
#pragma unroll
        for (int e = 0; e < E; ++e) okx &= ffk::normalised(x[c][e]);
    }
    const int64_t r0 = static_cast<int64_t>(blockIdx.y + zero) * rpb;
    const int64_t r1 = r0 + rpb < m ? r0 + rpb : m;

    // R rows of the chunk from row q on
    auto rows = [&](auto fast_c, auto r_c, int q, V (&v)[decltype(r_c)::value]) {
        constexpr bool FAST = decltype(fast_c)::value;
        constexpr int R = decltype(r_c)::value;
        float2 a[R][E];
#pragma unroll
        for (int c = 0; c < KT; ++c) {
            float2 d[R];
            if constexpr (R % 2 == 0) {
#pragma unroll
                for (int r = 0; r < R; r += 2) {
                    const float4 p = *reinterpret_cast<const float4*>(&sdy[c][q + r]);
                    d[r] = make_float2(p.x, p.y);
                    d[r + 1] = make_float2(p.z, p.w);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) d[r] = sdy[c][q + r];
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const float2 t = FAST ? ffk::mul22_fast(d[r], x[c][e]) : ffk::mul22(d[r], x[c][e]);
                    if (c == 0)
                        a[r][e] = FAST || KT > 1 ? ffk::add22_from_zero_fast(t) : ffk::add22(make_float2(0.0f, 0.0f), t);
                    else
                        a[r][e] = FAST ? ffk::add22_fast(a[r][e], t) : ffk::add22(a[r][e], t);
                }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                a[r][e] = KT == 1 ? ffk::from_zero_infinite(a[r][e]) : ffk::ff_overflow_lo(a[r][e]);
            if constexpr (E == 2)
                v[r] = make_float4(a[r][0].x, a[r][0].y, a[r][1].x, a[r][1].y);
            else
                v[r] = a[r][0];
        }
    };
    auto chunk = [&](auto fast_c, int64_t cb, int n_rows) {
        float2* out = dA + cb * ldda + j;
        int q = 0;
#pragma unroll 1
        for (; q + RS <= n_rows; q += RS, out += RS * ldda) {
            V v[RS];
            rows(fast_c, std::integral_constant<int, RS>(), q, v);
            if (store) {
#pragma unroll
                for (int r = 0; r < RS; ++r) __stcs(reinterpret_cast<V*>(out + r * ldda), v[r]);
            }
        }
#pragma unroll 1
        for (; q < n_rows; ++q, out += ldda) {
            V v[1];
            rows(fast_c, std::integral_constant<int, 1>(), q, v);
            if (store) __stcs(reinterpret_cast<V*>(out), v[0]);
        }
    };
    for (int64_t cb = r0; cb < r1; cb += kTChunk) {
        const int n_rows = static_cast<int>(r1 - cb < kTChunk ? r1 - cb : kTChunk);
        if (cb > r0) __syncthreads();   // the previous chunk's reads are done
        bool ok = okx;
        auto stage = [&](unsigned c, unsigned q) {
            const float2 d = __ldg(dY + c * lddy + cb + q);
            ok &= ffk::normalised(d);
            sdy[c][q] = d;
        };
        if constexpr (KT <= 5) {   // at most three rounds
            for (int i = threadIdx.x; i < KT * kTChunk; i += kGBlock)
                if (i % kTChunk < n_rows) stage(i / kTChunk, i % kTChunk);
        } else {   // rounds by the rows there are: the division costs less than rounds with few of them
            const unsigned per = n_rows, staged = KT * per;
            for (unsigned i = threadIdx.x; i < staged; i += kGBlock) stage(i / per, i % per);
        }
        if (__syncthreads_and(ok))
            chunk(std::true_type(), cb, n_rows);
        else
            chunk(std::false_type(), cb, n_rows);
    }
}

// Widest k of a column pair per thread, and of the kernel at all.  A pair's X
// takes 4 k registers: at k = 12 (95 registers) 1.63e12 terms/s on 8192^2, single
// columns 1.54e12; beyond, single columns (k = 13-20: 1.61 -> 1.54e12) against
// the GEMM kernel's 1.38-1.43e12 and the 1.35-1.53e12 of two passes over dA,
// which they replace.  Odd row lengths take single columns throughout (4001^2,
// k = 5: 1.46e12 terms/s; with X re-read for every element 0.59e12).  Above 20
// columns it depends on the size, over 28 shapes of 10^6 to 4 10^8 values, square, tall
// and wide: k = 21-24 take 0.88-0.96 of the GEMM kernel's time from 4 10^6 values on (1.04-
// 1.07 at 10^6), k = 26 0.94-1.00 from 6.5 10^7 on (0.99-1.02 from 2.5 to 4.2 10^7), k = 28
// 0.98-1.06; narrow ones leave threads of their last block idle (100 columns, k = 24 1.11).
constexpr int kDAPair = 12;
constexpr int kDAMax = 26;

inline int max_dA(int64_t m, int64_t n)
{
    const double values = static_cast<double>(m) * n;
    return n < 1024 || values < 4e6 ? 20 : values < 6.5e7 ? 24 : kDAMax;
}

// Grid: as many block rows as fill 1 to 8 waves of resident blocks, whichever
// takes the fewest rows in turn, a wave's start counted as four rows.  One wave
// alone leaves up to a block row of slots empty: at 32768 columns and three
// blocks per SM 384 of 456 slots, k = 20 15.9 ms, 13.4 in two waves.
template <int KT, int E>
ff_status launch_dA(const float2* dY, int64_t m, int64_t lddy, const float2* X, int64_t n, int64_t ldx, float2* dA,
                    int64_t ldda, int sm_count, cudaStream_t s)
{
    const int64_t col_blocks = (n / E + kGBlock - 1) / kGBlock;
    const int occ = ffh::occupancy(reinterpret_cast<const void*>(&gemv_dA_small_kernel<KT, E>), kGBlock);
    const int64_t slots = static_cast<int64_t>(sm_count) * (occ > 0 ? occ : 1);
    constexpr int64_t RS = 4 / E;
    int64_t rpb = 0, least = 0;
    for (int w = 1; w <= 8; ++w) {
        int64_t gy = w * slots / col_blocks;
        if (gy > (m + RS - 1) / RS) gy = (m + RS - 1) / RS;
        if (gy > 65535) gy = 65535;
        if (gy < 1) gy = 1;
        const int64_t rows = ((m + gy - 1) / gy + RS - 1) / RS * RS;
        const int64_t waves = (col_blocks * ((m + rows - 1) / rows) + slots - 1) / slots;
        if (w == 1 || waves * (rows + 4) < least) {
            rpb = rows;
            least = waves * (rows + 4);
        }
    }
    const dim3 grid(static_cast<unsigned>(col_blocks), static_cast<unsigned>((m + rpb - 1) / rpb));
    return ffh::launch_kernel(&gemv_dA_small_kernel<KT, E>, grid, kGBlock, s, dY, m, lddy, X, n, ldx, dA, ldda, rpb);
}

// k <= KT right-hand sides.
template <int KT, int E>
ff_status dA_small(int64_t k, const float2* dY, int64_t m, int64_t lddy, const float2* X, int64_t n, int64_t ldx,
                   float2* dA, int64_t ldda, int sm_count, cudaStream_t s)
{
    if constexpr (KT > 1)
        if (k < KT) return dA_small<KT - 1, E>(k, dY, m, lddy, X, n, ldx, dA, ldda, sm_count, s);
    return launch_dA<KT, E>(dY, m, lddy, X, n, ldx, dA, ldda, sm_count, s);
}

// ---------------------------------------------------------------------------
// binary64 GEMV (one warp per row, fma accumulation, shuffle tree)
// ---------------------------------------------------------------------------
template <int KT>
__global__ void __launch_bounds__(kGBlock)
gemv_f64_kernel(const double* __restrict__ A, int64_t m, int64_t n, int64_t lda, const double* __restrict__ X,
                int64_t ldx, double* __restrict__ Y, int64_t ldy)
{
    const unsigned zero = ffk::prior_kernel_done();
    const int lane = threadIdx.x & 31;
    const int64_t r = static_cast<int64_t>(blockIdx.x + zero) * kGWarps + (threadIdx.x >> 5);
    X += zero;
    if (r >= m) return;
    double acc[KT];
#pragma unroll
    for (int c = 0; c < KT; ++c) acc[c] = 0.0;
    const double* Ar = A + r * lda;
    for (int64_t j = lane; j < n; j += 32) {
        const double a = __ldcs(Ar + j);
#pragma unroll
        for (int c = 0; c < KT; ++c) acc[c] = __fma_rn(a, __ldg(X + c * ldx + j), acc[c]);
    }
#pragma unroll
    for (int c = 0; c < KT; ++c) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[c] = __dadd_rn(acc[c], __shfl_down_sync(0xffffffffu, acc[c], off));
    }
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < KT; ++c) Y[c * ldy + r] = acc[c];
    }
}

template <int KT>
ff_status launch_f64(unsigned grid, const double* A, int64_t m, int64_t n, int64_t lda, const double* X, int64_t ldx,
                     double* Y, int64_t ldy, cudaStream_t s)
{
    return ffh::launch_kernel(&gemv_f64_kernel<KT>, grid, kGBlock, s, A, m, n, lda, X, ldx, Y, ldy);
}

bool bad_dims(int64_t m, int64_t n, int64_t k) { return m < 0 || n < 0 || k < 1 || k > kMaxK; }

size_t adjoint_ws(const AdjointPlan& p, int64_t n, int64_t k)
{
    return p.gy <= 1 ? 16 : static_cast<size_t>(p.nrb) * static_cast<size_t>(n) * static_cast<size_t>(k) * sizeof(float2);
}

}  // namespace

extern "C" {

ff_status ff_gemv(const ff2* A_, int64_t m, int64_t n, int64_t lda, const ff2* X_, int64_t ldx, int64_t k,
                  ff2* Y_, int64_t ldy, cudaStream_t s)
{
    if (bad_dims(m, n, k) || lda < n || ldx < n || ldy < m) return FF_ERR_INVALID_ARG;
    const size_t an = static_cast<size_t>(m) * static_cast<size_t>(n);
    if (!ffh::ok_ptr(A_, an) || !ffh::ok_ptr(X_, static_cast<size_t>(n)) || !ffh::ok_ptr(Y_, static_cast<size_t>(m)))
        return FF_ERR_INVALID_ARG;
    if (m == 0) return FF_OK;
    ffh::DeviceInfo di;
    const ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    auto* A = reinterpret_cast<const float2*>(A_);
    auto* X = reinterpret_cast<const float2*>(X_);
    auto* Y = reinterpret_cast<float2*>(Y_);
    const bool vec = (n % 2 == 0) && (lda % 2 == 0) && (ldx % 2 == 0) && ffh::aligned(A, 16) && ffh::aligned(X, 16);
    return vec ? gemv_forward<true>(A, m, n, lda, X, ldx, k, Y, ldy, di.sm_count, s)
               : gemv_forward<false>(A, m, n, lda, X, ldx, k, Y, ldy, di.sm_count, s);
}

size_t ff_gemv_t_workspace_bytes(int64_t m, int64_t n, int64_t k)
{
    if (bad_dims(m, n, k)) return 0;
    ffh::DeviceInfo di;
    if (ffh::device_info(&di) != FF_OK) return 0;
    // the workspace must cover either access path: take the larger
    const AdjointPlans& p = adjoint_plans(m, n, k, di.sm_count);
    const size_t a = adjoint_ws(p.access16, n, k), b = adjoint_ws(p.access8, n, k);
    return a > b ? a : b;
}

ff_status ff_gemv_t_launch_shape(const ff2* A, int64_t m, int64_t n, int64_t lda, int64_t k, int64_t* nrb,
                                 int* vector)
{
    if (bad_dims(m, n, k) || lda < n || nrb == nullptr || vector == nullptr) return FF_ERR_INVALID_ARG;
    ffh::DeviceInfo di;
    const ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    const bool vec = (n % 2 == 0) && (lda % 2 == 0) && ffh::aligned(A, 16);
    *nrb = adjoint_plan(m, n, k, vec, di.sm_count).nrb;
    *vector = vec ? 1 : 0;
    return FF_OK;
}

ff_status ff_gemv_t(const ff2* A_, int64_t m, int64_t n, int64_t lda, const ff2* dY_, int64_t lddy, int64_t k,
                    ff2* dX_, int64_t lddx, void* ws, size_t ws_bytes, cudaStream_t s)
{
    if (bad_dims(m, n, k) || lda < n || lddy < m || lddx < n) return FF_ERR_INVALID_ARG;
    const size_t an = static_cast<size_t>(m) * static_cast<size_t>(n);
    if (!ffh::ok_ptr(A_, an) || !ffh::ok_ptr(dY_, static_cast<size_t>(m)) || !ffh::ok_ptr(dX_, static_cast<size_t>(n)))
        return FF_ERR_INVALID_ARG;
    if (n == 0) return FF_OK;
    ffh::DeviceInfo di;
    ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    auto* A = reinterpret_cast<const float2*>(A_);
    auto* dY = reinterpret_cast<const float2*>(dY_);
    auto* dX = reinterpret_cast<float2*>(dX_);
    const bool vec = (n % 2 == 0) && (lda % 2 == 0) && ffh::aligned(A, 16);
    const AdjointPlan p = adjoint_plan(m, n, k, vec, di.sm_count);
    float2* out = dX;
    int64_t out_ld = lddx, rb_stride = 0;
    if (p.gy > 1) {
        if (ws == nullptr || ws_bytes < adjoint_ws(p, n, k) || !ffh::aligned(ws, 16))
            return FF_ERR_WORKSPACE;
        out = static_cast<float2*>(ws);
        out_ld = n;
        rb_stride = k * n;
    }
    const TileSplit t = p.wide ? split_tiles(k) : TileSplit{1, 1, k, 0};
    // rows loaded together as adjoint_rows says; the residency leaves the
    // registers that keep those loads in flight
    const Columns c = vec ? kAdjacent : p.pairs ? kApart : kSingle;
#define FF_ADJOINT_RS(KA, KB, R, RS, MINB)                                                                           \
    (c == kAdjacent ? launch_adjoint<KA, KB, kAdjacent, R, MINB>(p, t, A, m, n, lda, dY, lddy, out, out_ld, rb_stride, s) \
     : c == kApart  ? launch_adjoint<KA, KB, kApart, R, MINB>(p, t, A, m, n, lda, dY, lddy, out, out_ld, rb_stride, s)    \
                    : launch_adjoint<KA, KB, kSingle, RS, MINB>(p, t, A, m, n, lda, dY, lddy, out, out_ld, rb_stride, s))
#define FF_ADJOINT_R(KA, KB, R, MINB) FF_ADJOINT_RS(KA, KB, R, R, MINB)
#define FF_ADJOINT(KA, KB, R, MINB) FF_ADJOINT_RS(KA, KB, R, (R > 8 ? R : 8), MINB)
    // Row blocks of at most three rows have no batch of rows to load together; a
    // thread does little more than store, and more resident warps pay instead (1 x
    // 1000000, k = 1 6.2 -> 3.9 us, k = 16 38.9 -> 30.9; 3 x 1000001, k = 2 11.4 -> 9.0).
    if (p.rpb <= 3)
        st = t.ka == 1   ? FF_ADJOINT_R(1, 1, 2, 6)
             : t.ka == 2 ? FF_ADJOINT_R(2, 1, 2, 5)
             : t.ka == 3 ? FF_ADJOINT_R(3, 2, 2, 4)
                         : FF_ADJOINT_R(4, 3, 2, 4);
    else if (k == 1 && p.gy > 1)
        st = FF_ADJOINT(1, 1, 16, 3);
    else if (t.ka == 1)
        st = FF_ADJOINT(1, 1, 8, 4);
    else if (t.ka == 2)
        st = FF_ADJOINT(2, 1, 8, 3);
    else if (t.ka == 3)
        st = FF_ADJOINT(3, 2, 4, 3);
    else
        st = FF_ADJOINT(4, 3, 4, 3);
#undef FF_ADJOINT
#undef FF_ADJOINT_R
#undef FF_ADJOINT_RS
    if (st != FF_OK) return st;
    if (p.gy > 1) {
        const int64_t total = n * k;
        st = ffh::launch_kernel(&gemv_t_combine, static_cast<unsigned>((total + kGBlock - 1) / kGBlock), kGBlock, s,
                                static_cast<float2*>(ws), n, k, p.nrb, dX, lddx);
    }
    return st;
}

ff_status ff_gemv_dA(const ff2* dY_, int64_t m, int64_t lddy, const ff2* X_, int64_t n, int64_t ldx, int64_t k,
                     ff2* dA_, int64_t ldda, cudaStream_t s)
{
    if (bad_dims(m, n, k) || lddy < m || ldx < n || ldda < n) return FF_ERR_INVALID_ARG;
    const size_t an = static_cast<size_t>(m) * static_cast<size_t>(n);
    if (!ffh::ok_ptr(dY_, static_cast<size_t>(m)) || !ffh::ok_ptr(X_, static_cast<size_t>(n)) || !ffh::ok_ptr(dA_, an))
        return FF_ERR_INVALID_ARG;
    if (m == 0 || n == 0) return FF_OK;
    // beyond max_dA right-hand sides, dA is a matrix product op(dY) X with dY read
    // transposed in place: the GEMM kernel computes every element with the same
    // Mul22(dY[r, c], X[j, c]) terms in the same order (bit-identical)
    if (k > max_dA(m, n))
        return ff_gemm(1, 0, m, n, k, dY_, lddy, X_, ldx, dA_, ldda, s);
    auto* dY = reinterpret_cast<const float2*>(dY_);
    auto* X = reinterpret_cast<const float2*>(X_);
    auto* dA = reinterpret_cast<float2*>(dA_);
    const bool vec = (n % 2 == 0) && (ldx % 2 == 0) && (ldda % 2 == 0) && ffh::aligned(X, 16) && ffh::aligned(dA, 16);
    ffh::DeviceInfo di;
    const ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    return vec && k <= kDAPair ? dA_small<kDAPair, 2>(k, dY, m, lddy, X, n, ldx, dA, ldda, di.sm_count, s)
                               : dA_small<kDAMax, 1>(k, dY, m, lddy, X, n, ldx, dA, ldda, di.sm_count, s);
}

ff_status ff_f64_gemv(const double* A, int64_t m, int64_t n, int64_t lda, const double* X, int64_t ldx, int64_t k,
                      double* Y, int64_t ldy, cudaStream_t s)
{
    if (bad_dims(m, n, k) || lda < n || ldx < n || ldy < m) return FF_ERR_INVALID_ARG;
    const size_t an = static_cast<size_t>(m) * static_cast<size_t>(n);
    if (!ffh::ok_ptr(A, an) || !ffh::ok_ptr(X, static_cast<size_t>(n)) || !ffh::ok_ptr(Y, static_cast<size_t>(m)))
        return FF_ERR_INVALID_ARG;
    if (m == 0) return FF_OK;
    const unsigned grid = static_cast<unsigned>((m + kGWarps - 1) / kGWarps);
    for (int64_t c0 = 0; c0 < k;) {
        const int kt = f64_tile_for(k - c0);
        const double* Xc = X + c0 * ldx;
        double* Yc = Y + c0 * ldy;
        ff_status st = FF_OK;
        switch (kt) {
        case 16: st = launch_f64<16>(grid, A, m, n, lda, Xc, ldx, Yc, ldy, s); break;
        case 8: st = launch_f64<8>(grid, A, m, n, lda, Xc, ldx, Yc, ldy, s); break;
        case 4: st = launch_f64<4>(grid, A, m, n, lda, Xc, ldx, Yc, ldy, s); break;
        case 2: st = launch_f64<2>(grid, A, m, n, lda, Xc, ldx, Yc, ldy, s); break;
        default: st = launch_f64<1>(grid, A, m, n, lda, Xc, ldx, Yc, ldy, s); break;
        }
        if (st != FF_OK) return st;
        c0 += kt;
    }
    return FF_OK;
}

}  // extern "C"
