// ff_gemm.cu -- float-float matrix product C = op(A) op(B), each term a Mul22
// and each accumulation an Add22 (the paper's operators, Section 4.1).
//
// Every output accumulates its terms in increasing order of the inner index,
// starting from (0, 0), one thread per output: the result does not depend on
// the launch shape and equals the plain triple loop bit for bit.
//
// The work is FP32-instruction bound: 22 instructions per term with the
// Fast2Sum forms of ff_core.cuh, against 8 bytes of A and B read from L2 per 64
// terms.  Every value is checked once, when its slice goes to shared memory,
// for RN(hi + lo) == hi; the check is combined over the block in the slice's
// barrier, and a slice with any other value (or a NaN) runs on the full Mul22 +
// Add22 (28 instructions), with the same bits either way.  4096^3: 54.4 ms with
// the full forms alone, 44.2 ms with the fast ones, 43.1 ms with addresses kept
// from slice to slice instead of formed for each value (1.59e12 terms/s).
//
// A block computes one tile of C from slices of A and B in shared memory,
// double buffered; the next slice is loaded into registers while the current
// one is computed.  Four tile shapes (see tile choice at ff_gemm): the large
// ones reuse operands more, the small ones spread a small C over all SMs.
// Packed binary32 pairs (add / mul / fma f32x2) were measured for the 22-
// instruction term and not kept: 15.1 instructions per term, but bound by
// register operands at the same time (2048^3: 5.59-5.73 against 5.50 ms).
// Global loads are coalesced for each operand layout (row-major or
// transposed); the shared-memory tiles are k-major with padded rows so that
// the transposing stores do not serialise on one bank.
#include <cmath>

#include "ff_core.cuh"
#include "ff_host.cuh"

namespace {

// One tile shape: a block of T threads computes BM x BN outputs, each thread
// a TM x TN sub-tile (rows ty + r BM / TM, columns tx + c BN / TN, or adjacent
// columns when TN = 2), from slices BK deep of A and B in shared memory.
template <int BM_, int BN_, int TM_, int TN_, int BK_, int MINB_>
struct Tile {
    static constexpr int BM = BM_, BN = BN_, TM = TM_, TN = TN_, BK = BK_, MINB = MINB_;
    static constexpr int TX = BN / TN, TY = BM / TM, T = TX * TY;
    static constexpr int LA = BM * BK / T, LB = BN * BK / T;      // values of one slice per thread
    static constexpr int LDA = BM + 1;                            // shared row lengths: a transposing
    static constexpr int LDB = TN == 2 ? BN + 2 : BN + 1;         // store spreads over the banks
    static_assert(T % 32 == 0 && BM * BK % T == 0 && BN * BK % T == 0, "whole values per thread");
};

struct Dims {
    int64_t m, n, k, lda, ldb, ldc;
    int64_t tiles_n, tiles;
};

// One operand's slices as a thread reads them: N rows (of op(A)) or columns (of
// op(B)) from the tile's first on, BK inner indices per slice.  KMAJOR: the
// operand is stored contiguous along the rows / columns (transposed A, row-major
// B), so neighbouring threads take neighbouring rows; otherwise contiguous along
// the inner index.  The thread's first address is kept and moved on slice by
// slice; its L values lie a fixed stride apart.
template <int N, int BK, int T, int L, bool KMAJOR>
struct Slices {
    static constexpr int kStep = KMAJOR ? T / N : T / BK;   // inner indices / rows between a thread's values
    static_assert(T % (KMAJOR ? N : BK) == 0, "a thread's values share their row / inner index");
    const float2* p;
    int64_t stride, advance;
    int row, inner;   // the thread's first value: row of the tile, inner index of the slice
    int rows;         // rows of the tile that exist

    __device__ __forceinline__ Slices(const float2* M, int64_t ld, int64_t extent, int64_t i0)
    {
        row = KMAJOR ? threadIdx.x % N : threadIdx.x / BK;
        inner = KMAJOR ? threadIdx.x / N : threadIdx.x % BK;
        rows = static_cast<int>(extent - i0 < N ? extent - i0 : N);
        p = M + (KMAJOR ? inner * ld + i0 + row : (i0 + row) * ld + inner);
        stride = kStep * ld;
        advance = KMAJOR ? BK * ld : BK;
    }

    // The next slice, of which `left` inner indices exist.  Others, and rows past
    // the last, read as (0, 0); they are never used for a stored output nor for a
    // term beyond k.
    __device__ __forceinline__ void load(int left, float2 (&v)[L])
    {
#pragma unroll
        for (int s = 0; s < L; ++s) {
            const bool in = KMAJOR ? row < rows && inner + s * kStep < left : row + s * kStep < rows && inner < left;
            v[s] = in ? __ldg(p + s * stride) : make_float2(0.0f, 0.0f);
        }
        p += advance;
    }
};

template <int N, int BK, int T, int L, int LD, bool KMAJOR>
__device__ __forceinline__ void store_slice(float2 (*S)[LD], const float2 (&v)[L])
{
#pragma unroll
    for (int s = 0; s < L; ++s) {
        const int e = threadIdx.x + s * T;
        S[KMAJOR ? e / N : e % BK][KMAJOR ? e % N : e / BK] = v[s];
    }
}

// One inner index of the slice: TM x TN terms, one per accumulator.
template <class S, bool FAST>
__device__ __forceinline__ void step(const float2* Ar, const float2* Br, int ty, int tx, float2 (&acc)[S::TM][S::TN])
{
    float2 a[S::TM], b[S::TN];
#pragma unroll
    for (int r = 0; r < S::TM; ++r) a[r] = Ar[ty + S::TY * r];
    if constexpr (S::TN == 2) {
        const float4 q = *reinterpret_cast<const float4*>(Br + 2 * tx);
        b[0] = make_float2(q.x, q.y);
        b[1] = make_float2(q.z, q.w);
    } else {
#pragma unroll
        for (int c = 0; c < S::TN; ++c) b[c] = Br[tx + S::TX * c];
    }
#pragma unroll
    for (int r = 0; r < S::TM; ++r)
#pragma unroll
        for (int c = 0; c < S::TN; ++c)
            acc[r][c] = FAST ? ffk::add22_fast(acc[r][c], ffk::mul22_fast(a[r], b[c]))
                             : ffk::add22(acc[r][c], ffk::mul22(a[r], b[c]));
}

template <class S, bool TA, bool TB>
__global__ void __launch_bounds__(S::T, S::MINB)
gemm_kernel(const float2* __restrict__ A, const float2* __restrict__ B, float2* __restrict__ C, Dims d)
{
    __shared__ __align__(16) float2 As[2][S::BK][S::LDA];
    __shared__ __align__(16) float2 Bs[2][S::BK][S::LDB];
    const int tx = threadIdx.x % S::TX;
    const int ty = threadIdx.x / S::TX;
    const int64_t nslices = (d.k + S::BK - 1) / S::BK;
    // A slice is unrolled to about 1,400 instructions at most: the fully unrolled
    // slice of the 4 x 4 sub-tile overflows the instruction cache.
    constexpr int U = 32 / (S::TM * S::TN) < 8 ? 32 / (S::TM * S::TN) : 8;

    for (int64_t tile = blockIdx.x + ffk::prior_kernel_done(); tile < d.tiles; tile += gridDim.x) {
        const int64_t i0 = (tile / d.tiles_n) * S::BM;
        const int64_t j0 = (tile % d.tiles_n) * S::BN;
        float2 acc[S::TM][S::TN];
#pragma unroll
        for (int r = 0; r < S::TM; ++r)
#pragma unroll
            for (int c = 0; c < S::TN; ++c) acc[r][c] = make_float2(0.0f, 0.0f);

        float2 va[S::LA], vb[S::LB];
        Slices<S::BM, S::BK, S::T, S::LA, TA> slices_a(A, d.lda, d.m, i0);
        Slices<S::BN, S::BK, S::T, S::LB, !TB> slices_b(B, d.ldb, d.n, j0);
        auto load = [&](int64_t sl) {
            const int64_t rest = d.k - sl * S::BK;
            const int left = static_cast<int>(rest < S::BK ? rest : S::BK);
            slices_a.load(left, va);
            slices_b.load(left, vb);
        };
        // to shared memory; true when every value this thread loaded is normalised
        auto store = [&](int buf) {
            store_slice<S::BM, S::BK, S::T, S::LA, S::LDA, TA>(As[buf], va);
            store_slice<S::BN, S::BK, S::T, S::LB, S::LDB, !TB>(Bs[buf], vb);
            bool ok = true;
#pragma unroll
            for (int s = 0; s < S::LA; ++s) ok &= ffk::normalised(va[s]);
#pragma unroll
            for (int s = 0; s < S::LB; ++s) ok &= ffk::normalised(vb[s]);
            return ok;
        };
        bool ok = true;
        if (nslices > 0) {
            load(0);
            ok = store(0);
        }
        // the whole slice is normalised (block-uniform): its terms take the fast forms
        bool fast = __syncthreads_and(ok);
        for (int64_t sl = 0; sl < nslices; ++sl) {
            const int cur = static_cast<int>(sl & 1);
            const bool more = sl + 1 < nslices;
            if (more) load(sl + 1);
            const int64_t rem = d.k - sl * S::BK;
            const int kn = static_cast<int>(rem < S::BK ? rem : S::BK);
            if (!fast) {
#pragma unroll 1
                for (int kk = 0; kk < kn; ++kk) step<S, false>(As[cur][kk], Bs[cur][kk], ty, tx, acc);
            } else if (kn == S::BK) {
#pragma unroll U
                for (int kk = 0; kk < S::BK; ++kk) step<S, true>(As[cur][kk], Bs[cur][kk], ty, tx, acc);
            } else {
                // a last slice of fewer inner indices; one loop for both lengths
                // costs 1% on the whole slices
                int kk = 0;
#pragma unroll 1
                for (; kk + U <= kn; kk += U) {
#pragma unroll
                    for (int u = 0; u < U; ++u) step<S, true>(As[cur][kk + u], Bs[cur][kk + u], ty, tx, acc);
                }
#pragma unroll 1
                for (; kk < kn; ++kk) step<S, true>(As[cur][kk], Bs[cur][kk], ty, tx, acc);
            }
            ok = more ? store(cur ^ 1) : true;
            fast = __syncthreads_and(ok);
        }

#pragma unroll
        for (int r = 0; r < S::TM; ++r) {
            const int64_t i = i0 + ty + S::TY * r;
            if (i >= d.m) continue;
#pragma unroll
            for (int c = 0; c < S::TN; ++c) {
                const int64_t j = j0 + (S::TN == 2 ? 2 * tx + c : tx + S::TX * c);
                if (j < d.n) C[i * d.ldc + j] = ffk::ff_overflow_lo(acc[r][c]);
            }
        }
    }
}

template <class S>
ff_status launch(bool ta, bool tb, const float2* A, const float2* B, float2* C, Dims d, cudaStream_t s)
{
    d.tiles_n = (d.n + S::BN - 1) / S::BN;
    d.tiles = ((d.m + S::BM - 1) / S::BM) * d.tiles_n;
    // one block per tile up to the 1-D grid limit; blocks loop over the rest
    const int64_t cap = 0x7fffffffLL;
    const unsigned grid = static_cast<unsigned>(d.tiles < cap ? d.tiles : cap);
    const auto kernel = ta ? (tb ? &gemm_kernel<S, true, true> : &gemm_kernel<S, true, false>)
                           : (tb ? &gemm_kernel<S, false, true> : &gemm_kernel<S, false, false>);
    return ffh::launch_kernel(kernel, grid, S::T, s, A, B, C, d);
}

// Tile choice.  Every output is one serial chain of k terms, so C is cut by
// outputs only, and the time is that of the SM with the most tiles: measured
// cycles with q tiles on an SM are close to  (a q + b) k + f q + g  (a: the tile's
// outputs per lane times the cycles per term, which grow as the tile's operand
// reuse shrinks: 25.1, 26.4, 27.6 and 30.2; b: the part of a chain's latency that
// the few resident warps leave uncovered; f, g: a tile's first loads and its stores,
// per tile and once).  The shape with the least of it runs; over 167 shapes with k =
// 1 to 400 that is within 0.4% of the best one on average, at worst 10%.  500 x 300 x
// 700: 392 us with 64 x 64 tiles alone (40 of 152 SMs busy), 82 us; 100 x 100 x 1000: 508
// -> 29 us; 1024^3: 1042 -> 737 us; from about 2048 rows and columns the largest tile is
// always taken.  Without f and g small k took small tiles: 1000 x 2000 x 1 19.3 -> 6.3 us
// (the largest tile alone: 6.6), 900 x 900 x 4 10.7 -> 6.2 (7.0).
//
// The small tiles do few terms per inner index, so the work of one slice (its
// loads, stores and barrier) is spread over 64 of them: 90 us at 500 x 300 x 700
// with slices of 16, 82 with 64.  64 x 64 tiles gain nothing from deeper slices.
using Tile64 = Tile<64, 64, 4, 4, 16, 2>;
using Tile32 = Tile<32, 32, 2, 2, 32, 2>;
using Tile16 = Tile<16, 16, 1, 2, 64, 4>;
using Tile8 = Tile<8, 16, 1, 1, 64, 4>;

template <class S>
double cycles(const Dims& d, int sm_count, double a, double b, double f, double g)
{
    const double tiles = static_cast<double>((d.m + S::BM - 1) / S::BM) * static_cast<double>((d.n + S::BN - 1) / S::BN);
    const double q = std::ceil(tiles / sm_count), k = static_cast<double>(d.k);
    return (a * q + b) * k + f * q + g;
}

ff_status launch_best(bool ta, bool tb, const float2* A, const float2* B, float2* C, const Dims& d, int sm_count,
                      cudaStream_t s)
{
    const double c64 = cycles<Tile64>(d, sm_count, 803.0, 45.0, 1600.0, 700.0);
    const double c32 = cycles<Tile32>(d, sm_count, 211.0, 20.0, 1190.0, 0.0);
    const double c16 = cycles<Tile16>(d, sm_count, 55.2, 28.0, 600.0, 100.0);
    const double c8 = cycles<Tile8>(d, sm_count, 30.2, 28.0, 530.0, 200.0);
    const double best = std::fmin(std::fmin(c64, c32), std::fmin(c16, c8));
    if (best == c64) return launch<Tile64>(ta, tb, A, B, C, d, s);
    if (best == c32) return launch<Tile32>(ta, tb, A, B, C, d, s);
    if (best == c16) return launch<Tile16>(ta, tb, A, B, C, d, s);
    return launch<Tile8>(ta, tb, A, B, C, d, s);
}

}  // namespace

extern "C" {

ff_status ff_gemm(int transa, int transb, int64_t m, int64_t n, int64_t k, const ff2* A_, int64_t lda,
                  const ff2* B_, int64_t ldb, ff2* C_, int64_t ldc, cudaStream_t s)
{
    if (m < 0 || n < 0 || k < 0) return FF_ERR_INVALID_ARG;
    if ((transa != 0 && transa != 1) || (transb != 0 && transb != 1)) return FF_ERR_INVALID_ARG;
    const int64_t a_cols = transa ? m : k;  // row length of A as stored
    const int64_t b_cols = transb ? k : n;
    if (lda < (a_cols > 1 ? a_cols : 1) || ldb < (b_cols > 1 ? b_cols : 1) || ldc < (n > 1 ? n : 1))
        return FF_ERR_INVALID_ARG;
    if (m == 0 || n == 0) return FF_OK;  // nothing to write, no pointer read
    const size_t an = static_cast<size_t>(m) * static_cast<size_t>(k);
    const size_t bn = static_cast<size_t>(k) * static_cast<size_t>(n);
    const size_t cn = static_cast<size_t>(m) * static_cast<size_t>(n);
    if (!ffh::ok_ptr(A_, an) || !ffh::ok_ptr(B_, bn) || !ffh::ok_ptr(C_, cn)) return FF_ERR_INVALID_ARG;
    ffh::DeviceInfo di;
    const ff_status st = ffh::device_info(&di);
    if (st != FF_OK) return st;
    Dims d;
    d.m = m; d.n = n; d.k = k; d.lda = lda; d.ldb = ldb; d.ldc = ldc;
    d.tiles_n = d.tiles = 0;
    auto* A = reinterpret_cast<const float2*>(A_);
    auto* B = reinterpret_cast<const float2*>(B_);
    auto* C = reinterpret_cast<float2*>(C_);
    return launch_best(transa != 0, transb != 0, A, B, C, d, di.sm_count, s);
}

}  // extern "C"
