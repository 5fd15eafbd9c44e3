// ntt.cu -- negacyclic transforms at N = 2^10 .. 2^15 (N = 2^16: kernels.cu).
//
// Cooley-Tukey forward with twiddles psi^brv(m + i) (natural order in,
// bit-reversed order out), Gentleman-Sande inverse.  Every thread holds 16
// elements in registers and runs three or four stages between shared-memory
// exchanges (radix-16 rounds, or two radix-8 groups).
//   * Up to N = 2^13 one block transforms a whole limb: one launch and one
//     read and write of global memory per transform.
//   * N = 2^14, 2^15, small batches at 2^12 and 2^13 and batches at 2^13 whose
//     last wave of whole limbs would be far from full take two passes: the first
//     seven stages on 128-row columns (16 columns a block), the rest inside rows
//     of 32 to 256 (2048 elements a block).
// The last round's twiddles, one set per thread, come from a table of their own
// (d_fwd_last, d_inv_last: [prime][group of the round][thread of the limb]) so
// that a warp reads consecutive entries.
//
// What bounds it: the integer multiplier (FMA-heavy pipe), as at N = 2^16, for
// large batches; latency for small ones.  The radix-4 passes through shared
// memory that this replaces took two launches, a shared-memory round trip every
// two stages and twiddle reads with strides.  Measured, forward, us with 6 us of
// event overhead (before / now): 608 limbs of N = 2^15 305 / 209, of 2^14 138 /
// 103, of 2^13 72 / 58, of 2^12 41 / 31; 8 limbs 17 / 15, 19 / 15, 16 / 15, 16 /
// 13.
#include <type_traits>

#include "ntt.cuh"

namespace {

// stages per round of a transform of 2^LS elements
template <int LS> struct Rounds;
template <> struct Rounds<5>  { static constexpr int n = 2, r[4] = {1, 4, 0, 0}; };
template <> struct Rounds<6>  { static constexpr int n = 2, r[4] = {3, 3, 0, 0}; };
template <> struct Rounds<7>  { static constexpr int n = 2, r[4] = {4, 3, 0, 0}; };
template <> struct Rounds<8>  { static constexpr int n = 2, r[4] = {4, 4, 0, 0}; };
template <> struct Rounds<10> { static constexpr int n = 3, r[4] = {4, 3, 3, 0}; };
template <> struct Rounds<11> { static constexpr int n = 3, r[4] = {4, 4, 3, 0}; };
template <> struct Rounds<12> { static constexpr int n = 3, r[4] = {4, 4, 4, 0}; };
template <> struct Rounds<13> { static constexpr int n = 4, r[4] = {4, 3, 3, 3}; };

// stages before round K
template <int LS>
constexpr int before(int k)
{
    int s = 0;
    for (int i = 0; i < k; i++) s += Rounds<LS>::r[i];
    return s;
}

// Round K of thread t: 16 >> r groups of 2^r elements; group u of the
// transform is (blk, low) with low the bits below the round's, and element j of
// it is blk | j | low.
template <int LS, int K>
struct Round {
    static constexpr int r = Rounds<LS>::r[K], s = before<LS>(K), R = 1 << r, G = 16 >> r;
    static constexpr int lw = LS - s - r, T = (1 << LS) / 16;
    static __device__ __forceinline__ int blk(int t, int g) { return (t + T * g) >> lw; }
    static __device__ __forceinline__ int elem(int t, int g, int j)
    {
        const int u = t + T * g;
        return (u >> lw) << (LS - s) | j << lw | (u & ((1 << lw) - 1));
    }
};

// Twiddles of the stages S0 .. S0 + LS - 1 of limb-wide stage numbering inside
// sub-transform `row`: tab for all rounds but the last, `last` (entry of this
// thread's first group; NB entries per group of the round) for the last.
template <int LS, int S0>
struct Tw {
    const ulonglong2 *tab;
    int row;
    __device__ __forceinline__ ulonglong2 operator()(int s, int st, int blk, int g) const
    {
        return __ldg(tab + (1 << (S0 + s + st)) + (((row << s) + blk) << st) + g);
    }
};

template <int LS, int K, int S0, bool LAZY>
__device__ __forceinline__ void fwd_round(u64 (&v)[16], int t, const Tw<LS, S0> &tw, const ulonglong2 *last, int nb,
                                          u64 q)
{
    typedef Round<LS, K> A;
#pragma unroll
    for (int g = 0; g < A::G; g++) {
        const int blk = A::blk(t, g);
        if (last && K == Rounds<LS>::n - 1) {
            const ulonglong2 *p = last + A::T * g;
            ct_round<A::R, LAZY>(v + g * A::R, [&](int st, int x) { return __ldg(p + (size_t)((1 << st) - 1 + x) * nb); },
                                 q, 4 * q);
        } else {
            ct_round<A::R, LAZY>(v + g * A::R, [&](int st, int x) { return tw(A::s, st, blk, x); }, q, 4 * q);
        }
    }
}

template <int LS, int K, int S0, bool LAZY>
__device__ __forceinline__ void inv_round(u64 (&v)[16], int t, const Tw<LS, S0> &tw, const ulonglong2 *last, int nb,
                                          u64 q, int k0)
{
    typedef Round<LS, K> A;
#pragma unroll
    for (int g = 0; g < A::G; g++) {
        const int blk = A::blk(t, g);
        if (last && K == Rounds<LS>::n - 1) {
            const ulonglong2 *p = last + A::T * g;
            gs_round<A::R, LAZY>(v + g * A::R, [&](int st, int x) { return __ldg(p + (size_t)((1 << st) - 1 + x) * nb); },
                                 q, 4 * q, k0);
        } else {
            gs_round<A::R, LAZY>(v + g * A::R, [&](int st, int x) { return tw(A::s, st, blk, x); }, q, 4 * q, k0);
        }
    }
}

// the elements of round FROM through shared memory to those of round TO
template <int LS, int FROM, int TO, class At>
__device__ __forceinline__ void exchange(u64 (&v)[16], int t, u64 *sm, At at, bool again)
{
    typedef Round<LS, FROM> A;
    typedef Round<LS, TO> B;
    if (again) __syncthreads();   // the previous exchange has been read
#pragma unroll
    for (int m = 0; m < 16; m++) sm[at(A::elem(t, m / A::R, m % A::R))] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[at(B::elem(t, m / B::R, m % B::R))];
}

// all rounds; v holds the elements of the first round (forward) or of the last
// (inverse) and ends with those of the other
template <int LS, int S0, bool LAZY, class At>
__device__ __forceinline__ void fwd_all(u64 (&v)[16], int t, u64 *sm, At at, const Tw<LS, S0> &tw,
                                        const ulonglong2 *last, int nb, u64 q)
{
    constexpr int n = Rounds<LS>::n;
    fwd_round<LS, 0, S0, LAZY>(v, t, tw, last, nb, q);
    exchange<LS, 0, 1>(v, t, sm, at, false);
    fwd_round<LS, 1, S0, LAZY>(v, t, tw, last, nb, q);
    if constexpr (n > 2) {
        exchange<LS, 1, 2>(v, t, sm, at, true);
        fwd_round<LS, 2, S0, LAZY>(v, t, tw, last, nb, q);
    }
    if constexpr (n > 3) {
        exchange<LS, 2, 3>(v, t, sm, at, true);
        fwd_round<LS, 3, S0, LAZY>(v, t, tw, last, nb, q);
    }
}

template <int LS, int S0, bool LAZY, class At>
__device__ __forceinline__ void inv_all(u64 (&v)[16], int t, u64 *sm, At at, const Tw<LS, S0> &tw,
                                        const ulonglong2 *last, int nb, u64 q, int k0)
{
    constexpr int n = Rounds<LS>::n;
    if constexpr (n > 3) {
        inv_round<LS, 3, S0, LAZY>(v, t, tw, last, nb, q, k0);
        exchange<LS, 3, 2>(v, t, sm, at, false);
    }
    if constexpr (n > 2) {
        inv_round<LS, 2, S0, LAZY>(v, t, tw, last, nb, q, k0 + LS - before<LS>(3));
        exchange<LS, 2, 1>(v, t, sm, at, n > 3);
    }
    inv_round<LS, 1, S0, LAZY>(v, t, tw, last, nb, q, k0 + LS - before<LS>(2));
    exchange<LS, 1, 0>(v, t, sm, at, n > 2);
    inv_round<LS, 0, S0, LAZY>(v, t, tw, last, nb, q, k0 + LS - before<LS>(1));
}

// Rows of 2^LS contiguous elements, 2^LS / 16 threads each; the last stages of
// the limb (S0 .. LOGN - 1).  Whole limbs are the case LS = LOGN.
template <int LOGN, int LS>
struct RowPass {
    static constexpr int S0 = LOGN - LS, T = (1 << LS) / 16;
    static constexpr int ROWS = LS == LOGN || T >= 128 ? 1 : 128 / T, THREADS = T * ROWS;
    static constexpr int NB = (1 << LOGN) >> Rounds<LS>::r[Rounds<LS>::n - 1];   // groups of the last round in a limb
    static constexpr int PADDED = (1 << LS) + (1 << LS) / 16;
    typedef Round<LS, Rounds<LS>::n - 1> Last;
    static __device__ __forceinline__ auto pad()
    {
        return [](int e) { return e + (e >> 4); };
    }
    // the last round's groups are contiguous: 16-byte accesses
    static __device__ __forceinline__ void load(u64 (&v)[16], const u64 *p, int t)
    {
#pragma unroll
        for (int m = 0; m < 16; m += 2) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(p + Last::elem(t, m / Last::R, m % Last::R));
            v[m] = a.x;
            v[m + 1] = a.y;
        }
    }
};

// blocks per SM to budget the registers for: 64 to 80 a thread
template <int LOGN, int LS>
constexpr int row_blocks() { return RowPass<LOGN, LS>::THREADS >= 512 ? 2 : RowPass<LOGN, LS>::THREADS >= 256 ? 3 : 6; }

// first / only pass over rows.  FIRST (whole limbs): reads src, else in place.
template <int LOGN, int LS, bool FIN>
__global__ void __launch_bounds__(RowPass<LOGN, LS>::THREADS, row_blocks<LOGN, LS>())
ntt_rows_fwd(const __grid_constant__ Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ tw,
             const ulonglong2 *__restrict__ tw_last, const Finish fin)
{
    typedef RowPass<LOGN, LS> W;
    typedef Round<LS, 0> A;
    constexpr int N = 1 << LOGN;
    const int limb = blockIdx.y, col = limb % bt.per_row, lrow = limb / bt.per_row, pi = bt.pidx[col];
    if (pi < 0) return;
    extern __shared__ u64 sm[];
    const int t = threadIdx.x % W::T, row = blockIdx.x * W::ROWS + threadIdx.x / W::T;
    u64 *s = sm + threadIdx.x / W::T * W::PADDED;
    const PrimeC P = primes[pi];
    const u64 *src = (LS == LOGN ? bt.src + ((size_t)lrow * bt.src_stride + col) * N
                                 : bt.dst + ((size_t)lrow * bt.dst_stride + col) * N) + ((size_t)row << LS);
    u64 *dst = bt.dst + ((size_t)lrow * bt.dst_stride + col) * N;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = src[A::elem(t, m / A::R, m % A::R)];
    const Tw<LS, W::S0> w{tw + (size_t)pi * N, row};
    const ulonglong2 *last = tw_last + (size_t)pi * N + ((size_t)row << LS >> Rounds<LS>::r[Rounds<LS>::n - 1]) + t;
    const auto put = [&](auto lazy) {   // the last round's groups are contiguous
#pragma unroll
        for (int m = 0; m < 16; m += 2)
            put_pair<decltype(lazy)::value, FIN>(
                v[m], v[m + 1], dst, ((size_t)row << LS) + W::Last::elem(t, m / W::Last::R, m % W::Last::R), fin, lrow, col,
                N, P);
    };
    if (P.q < (1ull << 47)) {
        fwd_all<LS, W::S0, true>(v, t, s, W::pad(), w, last, W::NB, P.q);
        put(std::true_type());
    } else {
        fwd_all<LS, W::S0, false>(v, t, s, W::pad(), w, last, W::NB, P.q);
        put(std::false_type());
    }
}

template <int LOGN, int LS>
__global__ void __launch_bounds__(RowPass<LOGN, LS>::THREADS, row_blocks<LOGN, LS>())
ntt_rows_inv(const __grid_constant__ Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ itw,
             const ulonglong2 *__restrict__ itw_last, const u64 *__restrict__ ninv)
{
    typedef RowPass<LOGN, LS> W;
    typedef Round<LS, 0> A;
    constexpr int N = 1 << LOGN;
    const int limb = blockIdx.y, col = limb % bt.per_row, lrow = limb / bt.per_row, pi = bt.pidx[col];
    if (pi < 0) return;
    extern __shared__ u64 sm[];
    const int t = threadIdx.x % W::T, row = blockIdx.x * W::ROWS + threadIdx.x / W::T;
    u64 *s = sm + threadIdx.x / W::T * W::PADDED;
    const u64 q = primes[pi].q;
    u64 v[16];
    W::load(v, bt.src + ((size_t)lrow * bt.src_stride + col) * N + ((size_t)row << LS), t);
    const Tw<LS, W::S0> w{itw + (size_t)pi * N, row};
    const ulonglong2 *last = itw_last + (size_t)pi * N + ((size_t)row << LS >> Rounds<LS>::r[Rounds<LS>::n - 1]) + t;
    if (q < (1ull << 47)) inv_all<LS, W::S0, true>(v, t, s, W::pad(), w, last, W::NB, q, 0);
    else inv_all<LS, W::S0, false>(v, t, s, W::pad(), w, last, W::NB, q, 0);
    u64 *dst = bt.dst + ((size_t)lrow * bt.dst_stride + col) * N + ((size_t)row << LS);
    const u64 ni = ninv[2 * pi], nis = ninv[2 * pi + 1];
#pragma unroll
    for (int m = 0; m < 16; m++)   // whole limbs: scaled; else lazy (< 2^(LS + 1) q or < 4q)
        dst[A::elem(t, m / A::R, m % A::R)] = LS == LOGN ? shoup_mul(v[m], ni, nis, q) : v[m];
}

// the first seven stages on columns of 128 rows, 16 columns a block
constexpr int kColS = 7, kCols = 16;

template <int LOGN>
__global__ void __launch_bounds__(128, 6)
ntt_cols_fwd(const __grid_constant__ Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ tw)
{
    typedef Round<kColS, 0> A;
    typedef Round<kColS, 1> B;
    constexpr int N = 1 << LOGN, N2 = N >> kColS;
    const int limb = blockIdx.y, col = limb % bt.per_row, lrow = limb / bt.per_row, pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[kCols << kColS];
    const int c = threadIdx.x % kCols, t = threadIdx.x / kCols, c0 = blockIdx.x * kCols + c;
    const u64 q = primes[pi].q;
    const u64 *src = bt.src + ((size_t)lrow * bt.src_stride + col) * N + c0;
    u64 *dst = bt.dst + ((size_t)lrow * bt.dst_stride + col) * N + c0;
    auto at = [c](int e) { return e * kCols + c; };
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = src[(size_t)A::elem(t, m / A::R, m % A::R) * N2];
    const Tw<kColS, 0> w{tw + (size_t)pi * N, 0};
    if (q < (1ull << 47)) fwd_all<kColS, 0, true>(v, t, sm, at, w, nullptr, 0, q);
    else fwd_all<kColS, 0, false>(v, t, sm, at, w, nullptr, 0, q);
#pragma unroll
    for (int m = 0; m < 16; m++) dst[(size_t)B::elem(t, m / B::R, m % B::R) * N2] = v[m];   // lazy
}

template <int LOGN>
__global__ void __launch_bounds__(128, 6)
ntt_cols_inv(const __grid_constant__ Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ itw,
             const u64 *__restrict__ ninv)
{
    typedef Round<kColS, 0> A;
    typedef Round<kColS, 1> B;
    constexpr int N = 1 << LOGN, N2 = N >> kColS;
    const int limb = blockIdx.y, col = limb % bt.per_row, lrow = limb / bt.per_row, pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[kCols << kColS];
    const int c = threadIdx.x % kCols, t = threadIdx.x / kCols;
    const u64 q = primes[pi].q;
    u64 *d = bt.dst + ((size_t)lrow * bt.dst_stride + col) * N + blockIdx.x * kCols + c;
    auto at = [c](int e) { return e * kCols + c; };
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = d[(size_t)B::elem(t, m / B::R, m % B::R) * N2];
    const Tw<kColS, 0> w{itw + (size_t)pi * N, 0};
    if (q < (1ull << 47)) inv_all<kColS, 0, true>(v, t, sm, at, w, nullptr, 0, q, LOGN - kColS);
    else inv_all<kColS, 0, false>(v, t, sm, at, w, nullptr, 0, q, LOGN - kColS);
    const u64 ni = ninv[2 * pi], nis = ninv[2 * pi + 1];
#pragma unroll
    for (int m = 0; m < 16; m++) d[(size_t)A::elem(t, m / A::R, m % A::R) * N2] = shoup_mul(v[m], ni, nis, q);
}

// last[(2^st - 1 + x) nb + b] = tab[2^(log_n - r + st) + (b << st) + x]: group x of
// the round's stage st, group b of elements, nb = N >> r; blockIdx.y: the prime
__global__ void k_last_table(const ulonglong2 *__restrict__ tab, ulonglong2 *last, int log_n, int r)
{
    const int N = 1 << log_n, nb = N >> r, k = blockIdx.x * blockDim.x + threadIdx.x;
    const int grp = k / nb, b = k - grp * nb;
    if (grp >= (1 << r) - 1) return;
    const int st = 31 - __clz(grp + 1), x = grp + 1 - (1 << st);
    last[(size_t)blockIdx.y * N + k] = tab[(size_t)blockIdx.y * N + (1 << (log_n - r + st)) + ((size_t)b << st) + x];
}

template <int LOGN, int LS, bool FIN>
void launch_rows_fwd(fg_ctx *ctx, const Batch &bt, int count, const Finish &fin)
{
    typedef RowPass<LOGN, LS> W;
    const size_t sm = (size_t)W::ROWS * W::PADDED * 8;
    const dim3 g((1 << (LOGN - LS)) / W::ROWS, count);
    if (sm > 48 * 1024)
        CUDA_TRY(cudaFuncSetAttribute(ntt_rows_fwd<LOGN, LS, FIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    ntt_rows_fwd<LOGN, LS, FIN><<<g, W::THREADS, sm, ctx->stream>>>(
        bt, ctx->d_primes, (const ulonglong2 *)ctx->d_fwd, (const ulonglong2 *)ctx->d_fwd_last, fin);
}

template <int LOGN, int LS>
void launch_rows(fg_ctx *ctx, const Batch &bt, int count, bool inverse, const Finish *fin)
{
    if (!inverse) {
        if (fin) launch_rows_fwd<LOGN, LS, true>(ctx, bt, count, *fin);
        else launch_rows_fwd<LOGN, LS, false>(ctx, bt, count, Finish());
        return;
    }
    typedef RowPass<LOGN, LS> W;
    const size_t sm = (size_t)W::ROWS * W::PADDED * 8;
    const dim3 g((1 << (LOGN - LS)) / W::ROWS, count);
    if (sm > 48 * 1024)
        CUDA_TRY(cudaFuncSetAttribute(ntt_rows_inv<LOGN, LS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    ntt_rows_inv<LOGN, LS><<<g, W::THREADS, sm, ctx->stream>>>(bt, ctx->d_primes, (const ulonglong2 *)ctx->d_inv,
                                                              (const ulonglong2 *)ctx->d_inv_last, ctx->d_ninv);
}

template <int LOGN>
void two_passes(fg_ctx *ctx, const Batch &bt, int count, bool inverse, const Finish *fin)
{
    const dim3 g((1 << (LOGN - kColS)) / kCols, count);
    Batch b2 = bt;
    b2.src = b2.dst;
    b2.src_stride = b2.dst_stride;
    if (!inverse) {
        ntt_cols_fwd<LOGN><<<g, 128, 0, ctx->stream>>>(bt, ctx->d_primes, (const ulonglong2 *)ctx->d_fwd);
        launch_rows<LOGN, LOGN - kColS>(ctx, b2, count, false, fin);
    } else {
        launch_rows<LOGN, LOGN - kColS>(ctx, bt, count, true, nullptr);
        ntt_cols_inv<LOGN><<<g, 128, 0, ctx->stream>>>(b2, ctx->d_primes, (const ulonglong2 *)ctx->d_inv, ctx->d_ninv);
    }
}

}  // namespace

void ntt_last_tables(fg_ctx *ctx)
{
    int r = 0;
    switch (ctx->log_n) {
    case 10: r = Rounds<10>::r[2]; break;
    case 11: r = Rounds<11>::r[2]; break;
    case 12: r = Rounds<12>::r[2]; break;   // = Rounds<5>::r[1]
    case 13: r = Rounds<13>::r[3]; break;   // = Rounds<6>::r[1]
    case 14: r = Rounds<7>::r[1]; break;
    case 15: r = Rounds<8>::r[1]; break;
    default: throw fg_error(FG_EINVAL, "ntt: unsupported ring degree");
    }
    const dim3 g(ctx->n / 256, ctx->nq + ctx->np);
    k_last_table<<<g, 256, 0, ctx->stream>>>((const ulonglong2 *)ctx->d_fwd, (ulonglong2 *)ctx->d_fwd_last, ctx->log_n, r);
    k_last_table<<<g, 256, 0, ctx->stream>>>((const ulonglong2 *)ctx->d_inv, (ulonglong2 *)ctx->d_inv_last, ctx->log_n, r);
    CUDA_TRY(cudaGetLastError());
    CUDA_TRY(cudaStreamSynchronize(ctx->stream));
}

void ntt_small(fg_ctx *ctx, const Batch &bt, int count, int working, bool inverse, const Finish *fin)
{
    bool one = ctx->log_n <= 11;
    switch (ctx->log_n) {
    case 10: launch_rows<10, 10>(ctx, bt, count, inverse, fin); break;
    case 11: launch_rows<11, 11>(ctx, bt, count, inverse, fin); break;
    case 12:
        // Two passes below 80 limbs: a rotation (3 to 12 limbs a transform, six
        // transforms) 118 / 111 us; 96 limbs 12.2 / 13.8 us.  Limbs left alone
        // count here: in two passes they cost four blocks instead of one, and
        // with the line at 80 or 64 working limbs a product of eight pairs (64
        // of 304 limbs at work in its ModDown) took 255 instead of 248 us, or a
        // batch of three small queries (72 limbs, all at work) 4.07 instead of
        // 4.03 ms.
        one = count >= 80;
        if (one) launch_rows<12, 12>(ctx, bt, count, inverse, fin);
        else two_passes<12>(ctx, bt, count, inverse, fin);
        break;
    case 13: {
        // One pass runs one limb an SM at a time, two passes fill the chip at
        // any count, so one pass pays where its last wave is nearly full (us,
        // one pass / two, with 6 of event overhead, 45-bit primes forward: 8
        // limbs 18.8 / 13.8, 104 19.3 / 20.0, 152 19.7 / 22.2, 160 31.0 / 24.0,
        // 256 30.9 / 31.7, 304 31.0 / 34.5, 312 41.2 / 34.9, 456 43.1 / 44.6,
        // 480 53.4 / 47.5; inverse and 60-bit primes within 2 us of these).
        // In whole calls: a product of sixteen pairs, 10 primes, 395 -> 376 us.
        constexpr int kSms = 152;
        one = working >= 150 * ((working + kSms - 1) / kSms) - 50;
        if (one) launch_rows<13, 13>(ctx, bt, count, inverse, fin);
        else two_passes<13>(ctx, bt, count, inverse, fin);
        break;
    }
    case 14: two_passes<14>(ctx, bt, count, inverse, fin); break;
    case 15: two_passes<15>(ctx, bt, count, inverse, fin); break;
    default: throw fg_error(FG_EINVAL, "ntt: unsupported ring degree");
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw fg_error(FG_ECUDA, std::string("ntt: ") + cudaGetErrorString(e));
    ctx->launches += one ? 1 : 2;
}
