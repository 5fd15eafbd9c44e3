// kernels.cu -- sm_103a kernels of the encrypted GCN layer.
//
// Every kernel works on 64-bit RNS words with the reductions of
// modarith.cuh on CUDA cores.  Layouts are limb-major: a polynomial limb is
// N consecutive words; a batch of limbs is addressed as rows of `per_row`
// limbs (row r, column c at base + (r * row_stride + c) * N), and limb
// column c is reduced modulo prime pidx[c] (pidx < 0: leave that limb).
#include <cstdio>

#include "ntt.cuh"

namespace {

Batch make_batch(u64 *src, int src_stride, u64 *dst, int dst_stride, int per_row, int rows,
                 const std::vector<int> &pidx)
{
    FG_CHECK(per_row <= kPidxMax && (int)pidx.size() == per_row, FG_EINVAL,
             "limb batch wider than the prime-index table");
    Batch b;
    b.src = src;
    b.dst = dst;
    b.src_stride = src_stride;
    b.dst_stride = dst_stride;
    b.per_row = per_row;
    b.rows = rows;
    for (int i = 0; i < per_row; i++) b.pidx[i] = (int8_t)pidx[i];
    return b;
}

inline void check_launch(fg_ctx *ctx, const char *what, int kernels = 1)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw fg_error(FG_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
    ctx->launches += kernels;
}

// ------------------------------------------------------------------------
// NTT at N = 2^16 (smaller rings: ntt.cu): negacyclic, Cooley-Tukey forward
// with twiddles psi^brv(m+i) (natural order in, bit-reversed order out: out[j]
// = a(psi^(2 brv(j) + 1))), Gentleman-Sande inverse, Harvey's lazy butterflies.
// N = 256 x 256: pass A runs stages 0..7 on the columns, pass B stages 8..15
// inside the rows, each as two radix-16 register rounds (ct_round, gs_round)
// with one shared-memory exchange.
// ------------------------------------------------------------------------
// A round's 15 twiddles either held in registers for the whole round
// (OD = false: loaded up front) or loaded where each stage uses them (OD =
// true: fewer live registers, so more CTAs per SM).
template <bool OD, class F>
struct Twiddles {
    ulonglong2 w[OD ? 1 : 15];
    F f;
    __device__ __forceinline__ explicit Twiddles(F g) : f(g)
    {
        if (!OD) {
#pragma unroll
            for (int st = 0; st < 4; st++)
#pragma unroll
                for (int gg = 0; gg < (1 << st); gg++) w[OD ? 0 : (1 << st) - 1 + gg] = f(st, gg);
        }
    }
    __device__ __forceinline__ ulonglong2 operator()(int st, int g) const
    {
        return OD ? f(st, g) : w[OD ? 0 : (1 << st) - 1 + g];
    }
};
template <bool OD, class F>
__device__ __forceinline__ Twiddles<OD, F> twiddles(F f) { return Twiddles<OD, F>(f); }

constexpr int kR16Row = 272;   // 256 elements + 16 pad words per row (pass B shared memory)
__device__ __forceinline__ int pad16(int pos) { return pos + (pos >> 4); }

// Tiles: pass A takes COLS (16 or 8) of the 256 columns per CTA, one
// thread per (column, group of 16 rows), 16 x COLS threads; pass B takes
// ROWS (16 or 8) of the 256 rows per CTA, 16 threads per row.  Both tile
// sizes compute the same transform word for word; the batched form picks
// one per shape by timing.
// pass A's two rounds on values already in registers (element (r + 16 m) of
// this thread's column), written to d (the tile's first column)
template <bool LAZY, int COLS, bool OD>
__device__ __forceinline__ void fwd_a16_rounds(u64 (&v)[16], u64 *d, const ulonglong2 *stw, u64 q, u64 *sm)
{
    const int t = threadIdx.x, c = t % COLS, r = t / COLS;   // r: r0 in round 1, r1 in round 2
    constexpr int N2 = 256;
    const u64 q4 = 4 * q;
    // stage st, group g at (1 << st) + g
    ct_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return stw[(1 << st) + g]; }), q, q4);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[(r + 16 * m) * COLS + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[(16 * r + m) * COLS + c];
    ct_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return stw[(1 << (st + 4)) + (r << st) + g]; }), q, q4);
#pragma unroll
    for (int m = 0; m < 16; m++) d[(size_t)(16 * r + m) * N2 + c] = v[m];   // lazy
}

template <bool LAZY, int COLS, bool OD>
__device__ __forceinline__ void fwd_a16_body(const u64 *s, u64 *d, const ulonglong2 *stw, u64 q, u64 *sm)
{
    const int t = threadIdx.x, c = t % COLS, r = t / COLS;
    constexpr int N2 = 256;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = s[(size_t)(r + 16 * m) * N2 + c];
    fwd_a16_rounds<LAZY, COLS, OD>(v, d, stw, q, sm);
}

template <int COLS, bool OD>
__global__ void __launch_bounds__(16 * COLS, (OD ? 64 : 48) / COLS)
ntt16_fwd_a(const Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ tw)
{
    const int limb = blockIdx.y;
    const int col = limb % bt.per_row, row = limb / bt.per_row;
    const int pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[256 * COLS];
    __shared__ ulonglong2 stw[256];
    const u64 q = primes[pi].q;
    const ulonglong2 *twp = tw + (size_t)pi * 65536;
    for (int k = threadIdx.x; k < 256; k += blockDim.x) stw[k] = twp[k];
    __syncthreads();
    const int c0 = blockIdx.x * COLS;
    const u64 *src = bt.src + ((size_t)row * bt.src_stride + col) * 65536 + c0;
    u64 *dst = bt.dst + ((size_t)row * bt.dst_stride + col) * 65536 + c0;
    if (q < (1ull << 47)) fwd_a16_body<true, COLS, OD>(src, dst, stw, q, sm);
    else fwd_a16_body<false, COLS, OD>(src, dst, stw, q, sm);
}

template <bool LAZY, bool OD, bool FIN>
__device__ __forceinline__ void fwd_b16_body(u64 *d, const ulonglong2 *twp, const ulonglong2 *rows, int row0,
                                             const PrimeC &P, u64 *sm, const Finish &fin, int lrow, int lcol)
{
    const int t = threadIdx.x, j = t & 15, r = t >> 4;
    constexpr int S1 = 8;
    const u64 q = P.q, q4 = 4 * q;
    u64 v[16];
    const int grow = row0 + r;
    u64 *drow = d + (size_t)r * 256;
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = drow[j + 16 * m];
    ct_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return twp[(1 << (S1 + st)) + (grow << st) + g]; }), q, q4);
    u64 *srow = sm + r * kR16Row;
#pragma unroll
    for (int m = 0; m < 16; m++) srow[pad16(j + 16 * m)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = srow[pad16(16 * j + m)];
    // row stages 12..15 from the row-blocked table (consecutive per row)
    ct_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return rows[((size_t)grow * 15 + (1 << st) - 1 + g) * 16 + j]; }),
               q, q4);
    // d: the tile's first word, row0 rows into the limb
#pragma unroll
    for (int m = 0; m < 16; m += 2)
        put_pair<LAZY, FIN>(v[m], v[m + 1], d - (size_t)row0 * 256, (size_t)grow * 256 + 16 * j + m, fin, lrow, lcol, 65536, P);
}

template <int ROWS, bool OD, bool FIN>
__global__ void __launch_bounds__(16 * ROWS, (OD ? 64 : 48) / ROWS)
ntt16_fwd_b(const Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ tw,
            const ulonglong2 *__restrict__ tw_rows, const Finish fin)
{
    const int limb = blockIdx.y;
    const int col = limb % bt.per_row, row = limb / bt.per_row;
    const int pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[ROWS * kR16Row];
    const PrimeC P = primes[pi];
    const ulonglong2 *twp = tw + (size_t)pi * 65536;
    const int row0 = blockIdx.x * ROWS;
    u64 *d = bt.dst + ((size_t)row * bt.dst_stride + col) * 65536 + (size_t)row0 * 256;
    const ulonglong2 *rows = tw_rows + (size_t)pi * 256 * 15 * 16;
    if (P.q < (1ull << 47)) fwd_b16_body<true, OD, FIN>(d, twp, rows, row0, P, sm, fin, row, col);
    else fwd_b16_body<false, OD, FIN>(d, twp, rows, row0, P, sm, fin, row, col);
}

template <bool LAZY, bool OD>
__device__ __forceinline__ void inv_b16_body(const u64 *s, u64 *d, const ulonglong2 *twp,
                                             const ulonglong2 *rows, int row0, u64 q, u64 *sm)
{
    const int t = threadIdx.x, j = t & 15, r = t >> 4;
    constexpr int S1 = 8;
    const u64 q4 = 4 * q;
    u64 v[16];
    const int grow = row0 + r;
    const ulonglong2 *in = reinterpret_cast<const ulonglong2 *>(s + (size_t)r * 256 + 16 * j);
#pragma unroll
    for (int m = 0; m < 16; m += 2) {
        const ulonglong2 a = in[m / 2];
        v[m] = a.x;
        v[m + 1] = a.y;
    }
    gs_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return rows[((size_t)grow * 15 + (1 << st) - 1 + g) * 16 + j]; }),
               q, q4, 0);
    u64 *srow = sm + r * kR16Row;
#pragma unroll
    for (int m = 0; m < 16; m++) srow[pad16(16 * j + m)] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = srow[pad16(j + 16 * m)];
    gs_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return twp[(1 << (S1 + st)) + (grow << st) + g]; }), q, q4, 4);
    u64 *drow = d + (size_t)r * 256;
#pragma unroll
    for (int m = 0; m < 16; m++) drow[j + 16 * m] = v[m];   // lazy (< 2^9 q or < 4q)
}

template <int ROWS, bool OD>
__global__ void __launch_bounds__(16 * ROWS, (OD ? 64 : 48) / ROWS)
ntt16_inv_b(const Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ itw,
            const ulonglong2 *__restrict__ itw_rows)
{
    const int limb = blockIdx.y;
    const int col = limb % bt.per_row, row = limb / bt.per_row;
    const int pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[ROWS * kR16Row];
    const u64 q = primes[pi].q;
    const ulonglong2 *twp = itw + (size_t)pi * 65536;
    const int row0 = blockIdx.x * ROWS;
    const u64 *s = bt.src + ((size_t)row * bt.src_stride + col) * 65536 + (size_t)row0 * 256;
    u64 *d = bt.dst + ((size_t)row * bt.dst_stride + col) * 65536 + (size_t)row0 * 256;
    const ulonglong2 *rows = itw_rows + (size_t)pi * 256 * 15 * 16;
    if (q < (1ull << 47)) inv_b16_body<true, OD>(s, d, twp, rows, row0, q, sm);
    else inv_b16_body<false, OD>(s, d, twp, rows, row0, q, sm);
}

template <bool LAZY, int COLS, bool OD>
__device__ __forceinline__ void inv_a16_body(u64 *d, const ulonglong2 *stw, u64 q, u64 ni, u64 nis,
                                             u64 *sm)
{
    const int t = threadIdx.x, c = t % COLS, r = t / COLS;
    constexpr int N2 = 256;
    const u64 q4 = 4 * q;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = d[(size_t)(16 * r + m) * N2 + c];
    gs_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return stw[(1 << (st + 4)) + (r << st) + g]; }), q, q4, 8);
#pragma unroll
    for (int m = 0; m < 16; m++) sm[(16 * r + m) * COLS + c] = v[m];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 16; m++) v[m] = sm[(r + 16 * m) * COLS + c];
    gs_round<16, LAZY>(v, twiddles<OD>([&](int st, int g) { return stw[(1 << st) + g]; }), q, q4, 12);
#pragma unroll
    for (int m = 0; m < 16; m++) d[(size_t)(r + 16 * m) * N2 + c] = shoup_mul(v[m], ni, nis, q);
}

// col_scale (may be null): per limb column of the batch, a constant (and
// its Shoup companion) that replaces N^-1 in the final scaling
template <int COLS, bool OD>
__global__ void __launch_bounds__(16 * COLS, (OD ? 64 : 48) / COLS)
ntt16_inv_a(const Batch bt, const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ itw,
            const u64 *__restrict__ ninv, const u64 *__restrict__ col_scale)
{
    const int limb = blockIdx.y;
    const int col = limb % bt.per_row, row = limb / bt.per_row;
    const int pi = bt.pidx[col];
    if (pi < 0) return;
    __shared__ u64 sm[256 * COLS];
    __shared__ ulonglong2 stw[256];
    const u64 q = primes[pi].q;
    const ulonglong2 *twp = itw + (size_t)pi * 65536;
    for (int k = threadIdx.x; k < 256; k += blockDim.x) stw[k] = twp[k];
    __syncthreads();
    const int c0 = blockIdx.x * COLS;
    u64 *d = bt.dst + ((size_t)row * bt.dst_stride + col) * 65536 + c0;
    const u64 ni = col_scale ? col_scale[2 * col] : ninv[2 * pi];
    const u64 nis = col_scale ? col_scale[2 * col + 1] : ninv[2 * pi + 1];
    if (q < (1ull << 47)) inv_a16_body<true, COLS, OD>(d, stw, q, ni, nis, sm);
    else inv_a16_body<false, COLS, OD>(d, stw, q, ni, nis, sm);
}

// ModUp, N = 2^16: the base conversion of one digit to one output prime,
// fused into the first pass (column stages 0..7) of that output limb's
// forward NTT.  y: [ncol][nl][N], the conversion's inputs y_i = [x_i (D_j /
// q_i)^-1]_{q_i} in the coefficient domain (the inverse NTT of c1, scaled
// by modup_scale_tab); digits: [ncol][beta][E][N], pass-A output of every
// limb outside the digit (pass B follows as for any forward NTT).  Grid:
// (256 / COLS column tiles, output index t, column f x beta + digit).
template <int NMAX, int COLS, bool OD>
__global__ void __launch_bounds__(16 * COLS, (OD ? 64 : 48) / COLS)
k_modup_ntt16_a(const u64 *__restrict__ y, int nl, u64 *digits, int beta, int E,
                const ConvTab *__restrict__ tabs, const PrimeC *__restrict__ primes,
                const ulonglong2 *__restrict__ tw)
{
    const int f = blockIdx.z / beta, dg = blockIdx.z % beta, t = blockIdx.y;
    const ConvTab &T = tabs[dg];
    if (t >= T.n_out) return;
    __shared__ u64 sm[256 * COLS];
    __shared__ ulonglong2 stw[256];
    const int pi = T.out_p[t];
    const PrimeC P = primes[pi];
    const ulonglong2 *twp = tw + (size_t)pi * 65536;
    for (int k = threadIdx.x; k < 256; k += blockDim.x) stw[k] = twp[k];
    u64 hm_[NMAX];
    const u64 *src[NMAX];
#pragma unroll
    for (int k = 0; k < NMAX; k++) {
        hm_[k] = k < T.n_in ? T.hmod[k][t] : 0;
        src[k] = y + ((size_t)f * nl + (k < T.n_in ? T.in_l[k] : 0)) * 65536;
    }
    const int c = threadIdx.x % COLS, r = threadIdx.x / COLS, c0 = blockIdx.x * COLS;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) {
        const size_t idx = (size_t)(r + 16 * m) * 256 + c0 + c;
        u64 a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
        for (int k = 0; k < NMAX; k++)
            if (k < T.n_in) mac_split(a0, a1, a2, split30(src[k][idx]), hm_[k]);
        v[m] = reduce30<NMAX>(a0, a1, a2, P);
    }
    __syncthreads();   // stw
    u64 *d = digits + (((size_t)f * beta + dg) * E + T.out_l[t]) * 65536 + c0;
    if (P.q < (1ull << 47)) fwd_a16_rounds<true, COLS, OD>(v, d, stw, P.q, sm);
    else fwd_a16_rounds<false, COLS, OD>(v, d, stw, P.q, sm);
}

// ------------------------------------------------------------------------
// element-wise kernels over a Batch (grid: x blocks, limbs)
// ------------------------------------------------------------------------
__device__ __forceinline__ const u64 *limb_ptr(const u64 *base, int stride, int per_row, int limb,
                                               int N)
{
    return base + ((size_t)(limb / per_row) * stride + (limb % per_row)) * N;
}

// split: the words are left as split halves (split_word), the form in which
// the group MAC and the masked products take plan masks; pmodq: a mask of
// kept values, its limbs of Q (prime index below nq) times P, the others 0
__global__ void k_to_mont(const Batch bt, const PrimeC *__restrict__ primes, int N, int split,
                          const u64 *__restrict__ pmodq, int nq)
{
    const int limb = blockIdx.y;
    const int pi = bt.pidx[limb % bt.per_row];
    if (pi < 0) return;
    const PrimeC P = primes[pi];
    u64 *d = const_cast<u64 *>(limb_ptr(bt.dst, bt.dst_stride, bt.per_row, limb, N));
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        u64 m = mont_mul(d[x], P.r2, P);
        if (pmodq) m = pi < nq ? shoup_mul(m, pmodq[2 * pi], pmodq[2 * pi + 1], P.q) : 0;
        d[x] = split ? split_word(m, P.q) : m;
    }
}

__global__ void k_from_mont(const Batch bt, const PrimeC *__restrict__ primes, int N)
{
    const int limb = blockIdx.y;
    const int pi = bt.pidx[limb % bt.per_row];
    if (pi < 0) return;
    const PrimeC P = primes[pi];
    u64 *d = const_cast<u64 *>(limb_ptr(bt.dst, bt.dst_stride, bt.per_row, limb, N));
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        d[x] = redc(0, d[x], P);
}

// c = a * b (both plain NTT-domain values)
__global__ void k_pointwise(const u64 *a, const u64 *b, u64 *c, const Batch bt,
                            const PrimeC *__restrict__ primes, int N)
{
    const int limb = blockIdx.y;
    const int pi = bt.pidx[limb % bt.per_row];
    if (pi < 0) return;
    const PrimeC P = primes[pi];
    const size_t off = (size_t)limb * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        c[off + x] = mont_mul(mont_mul(a[off + x], b[off + x], P), P.r2, P);
}

// Tensor product of n pairs (a0, a1) x (b0, b1) (NTT domain, [n][2][nl][N]):
// lane = (a0 b0, a1 b1), d1 = P (a0 b1 + a1 b0), one pass over the operands
// instead of four products, a sum and a scaling each through memory.
__global__ void __launch_bounds__(256)
k_tensor(const u64 *a, const u64 *b, u64 *lane, u64 *d1, int nl, const PrimeC *__restrict__ primes,
         const u64 *__restrict__ pmodq, int N)
{
    const int i = blockIdx.y, c = blockIdx.z, x = blockIdx.x * blockDim.x + threadIdx.x;
    const PrimeC P = primes[i];
    const u64 pr2 = mont_mul(mont_mul(pmodq[2 * i], P.r2, P), P.r2, P);   // P R^2
    const size_t o0 = ((size_t)c * 2 * nl + i) * N + x, o1 = o0 + (size_t)nl * N;
    const u64 a0 = a[o0], a1 = a[o1], b0 = b[o0], b1 = b[o1];
    lane[o0] = mont_mul(mont_mul(a0, b0, P), P.r2, P);
    lane[o1] = mont_mul(mont_mul(a1, b1, P), P.r2, P);
    u64 hi = mulhi64(a0, b1), lo = a0 * b1;   // the sum of two products is below q 2^64
    mac128(hi, lo, a1, b0);
    d1[((size_t)c * nl + i) * N + x] = mont_mul(redc(hi, lo, P), pr2, P);
}

// part 1 of n extended ciphertexts u [n][2][E][N] += d [n][nl][N] on the limbs of Q
__global__ void __launch_bounds__(256)
k_add_part1(u64 *u, int E, const u64 *__restrict__ d, int nl, const PrimeC *__restrict__ primes, int N)
{
    const int i = blockIdx.y, c = blockIdx.z, x = blockIdx.x * blockDim.x + threadIdx.x;
    u64 *p = u + (((size_t)c * 2 + 1) * E + i) * N + x;
    *p = add_mod(*p, d[((size_t)c * nl + i) * N + x], primes[i].q);
}

__global__ void k_add(const u64 *a, const u64 *b, u64 *c, const Batch bt,
                      const PrimeC *__restrict__ primes, int N)
{
    const int limb = blockIdx.y;
    const int pi = bt.pidx[limb % bt.per_row];
    if (pi < 0) return;
    const u64 q = primes[pi].q;
    const size_t off = (size_t)limb * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        c[off + x] = add_mod(a[off + x], b[off + x], q);
}

__global__ void k_neg(const u64 *a, u64 *c, const Batch bt, const PrimeC *__restrict__ primes,
                      int N)
{
    const int limb = blockIdx.y;
    const int pi = bt.pidx[limb % bt.per_row];
    if (pi < 0) return;
    const u64 q = primes[pi].q;
    const size_t off = (size_t)limb * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        u64 v = a[off + x];
        c[off + x] = v ? q - v : 0;
    }
}

// c = a * s_limb (scalar per limb column, Shoup), s given as (w, w') pairs
__global__ void k_scalar(const u64 *a, u64 *c, const Batch bt, const PrimeC *__restrict__ primes,
                         const u64 *__restrict__ scal, int N)
{
    const int limb = blockIdx.y;
    const int col = limb % bt.per_row;
    const int pi = bt.pidx[col];
    if (pi < 0) return;
    const u64 q = primes[pi].q, w = scal[2 * col], ws = scal[2 * col + 1];
    const size_t off = (size_t)limb * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        c[off + x] = shoup_mul(a[off + x], w, ws, q);
}

__global__ void k_automorphism(const u64 *a, u64 *c, int nlimbs, uint32_t g, int log_n)
{
    const int N = 1 << log_n;
    const size_t off = (size_t)blockIdx.y * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        c[off + x] = a[off + auto_src(x, g, log_n)];
}

// small signed coefficients -> residues of each listed prime
__global__ void k_small_to_res(const int8_t *e, u64 *out, const int *pidx, const PrimeC *primes,
                               int N)
{
    const int limb = blockIdx.y;
    const u64 q = primes[pidx[limb]].q;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        int v = e[x];
        out[(size_t)limb * N + x] = v < 0 ? q - (u64)(-v) : (u64)v;
    }
}

// SplitMix64's output function (Steele, Lea and Flood, OOPSLA 2014)
__device__ __forceinline__ u64 sm_mix_dev(u64 z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// The uniform part of seeded ciphertexts: column c is ciphertext index0 + c,
// whose stream (seed, purpose, index) starts from s0 = mix(seed ^ (purpose
// << 48) ^ index) and has word j = mix(s0 + (j + 1) gamma); coefficient x of
// limb i is (w_hi 2^64 + w_lo) mod q_i with w_lo, w_hi the words 2(i N + x)
// and 2(i N + x) + 1.  [w_hi]_q 2^64 mod q is the Montgomery product of
// [w_hi]_q with R^2 mod q (R = 2^64).  Ciphertext c is written at ct + c *
// ct_pitch: its uniform part at offset nl N, and, when c0 is given, its c0
// copied from c0 + c * nl N.
__global__ void k_expand_uniform(u64 *ct, size_t ct_pitch, const u64 *__restrict__ c0, int nl, u64 seed,
                                 u64 purpose, u64 index0, const PrimeC *__restrict__ primes, int N)
{
    const int i = blockIdx.y, c = blockIdx.z;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const PrimeC P = primes[i];
    const u64 gamma = 0x9E3779B97F4A7C15ull;
    const u64 s0 = sm_mix_dev(seed ^ (purpose << 48) ^ (index0 + (u64)c));
    const u64 j = 2 * ((u64)i * (u64)N + (u64)x);
    const u64 lo = sm_mix_dev(s0 + (j + 1) * gamma), hi = sm_mix_dev(s0 + (j + 2) * gamma);
    const u64 h = mont_mul(reduce_word(hi, P), P.r2, P);
    u64 *o = ct + (size_t)c * ct_pitch + (size_t)i * N + x;
    o[(size_t)nl * N] = add_mod(h, reduce_word(lo, P), P.q);
    if (c0) *o = c0[((size_t)c * nl + i) * N + x];
}

__global__ void k_copy_limbs(const u64 *src, int src_ls, u64 *dst, int dst_ls, int nl, int N)
{
    const int poly = blockIdx.z, i = blockIdx.y;
    const u64 *s = src + ((size_t)poly * src_ls + i) * N;
    u64 *d = dst + ((size_t)poly * dst_ls + i) * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        d[x] = s[x];
}

// ------------------------------------------------------------------------
// combination: Z[j][p][i] = sum_f c[i][f][j] * X[f][p][i]   (coefficient domain)
// constants in Montgomery form, one Montgomery reduction at the end.  For
// primes below 2^46 the products are 23-bit split sums (mac_split); for the
// others 128-bit sums with the high word folded mod q every chunk.
// ------------------------------------------------------------------------
constexpr int kCombJ = 8;
constexpr int kCombChunk = 128;

// Columns fb..fe-1 of X; with accumulate set, the result is added to Z.
// The nj = ceil(Fp / kCombJ) output blocks of one slot range are
// neighbouring CTAs (blockIdx.x = slot block * nj + output block), so they
// run together and the later ones find the input words in L2: X is read from
// HBM once for all F' outputs.
__global__ void __launch_bounds__(256)
k_comb(const u64 *__restrict__ X, int F, int fb, int fe, int accumulate, int Fp, int nj, int level,
       const u64 *__restrict__ consts, u64 *Z, int z_ls, const PrimeC *__restrict__ primes,
       int N)
{
    __shared__ u64 cs[kCombChunk][kCombJ];
    const int i = blockIdx.y, p = blockIdx.z;
    const int j0 = (blockIdx.x % nj) * kCombJ;
    const int x = (blockIdx.x / nj) * blockDim.x + threadIdx.x;
    const PrimeC P = primes[i];
    const bool split = P.q < (1ull << 46);
    const int nl = level + 1;
    u64 a0[kCombJ], a1[kCombJ], a2[kCombJ];   // split: A0, A1, A2; else lo, hi, unused
#pragma unroll
    for (int j = 0; j < kCombJ; j++) a0[j] = a1[j] = a2[j] = 0;
    for (int f0 = fb; f0 < fe; f0 += kCombChunk) {
        const int fc = min(kCombChunk, fe - f0);
        __syncthreads();
        for (int idx = threadIdx.x; idx < kCombChunk * kCombJ; idx += blockDim.x) {
            int ff = idx / kCombJ, jj = idx % kCombJ;
            const u64 c = (ff < fc && j0 + jj < Fp) ? consts[((size_t)i * F + f0 + ff) * Fp + j0 + jj] : 0;
            cs[ff][jj] = split ? split23(c) : c;
        }
        __syncthreads();
        if (x < N) {
            if (split) {
                for (int ff = 0; ff < fc; ff++) {
                    const u64 xv = split23(X[(((size_t)(f0 + ff) * 2 + p) * nl + i) * N + x]);
#pragma unroll
                    for (int j = 0; j < kCombJ; j++) mac_split(a0[j], a1[j], a2[j], xv, cs[ff][j]);
                }
            } else {
                for (int ff = 0; ff < fc; ff++) {
                    const u64 xv = X[(((size_t)(f0 + ff) * 2 + p) * nl + i) * N + x];
#pragma unroll
                    for (int j = 0; j < kCombJ; j++) mac128(a1[j], a0[j], xv, cs[ff][j]);
                }
#pragma unroll
                for (int j = 0; j < kCombJ; j++) a1[j] = reduce_word(a1[j], P);
            }
        }
    }
    if (x < N) {
#pragma unroll
        for (int j = 0; j < kCombJ; j++)
            if (j0 + j < Fp) {
                u64 *z = Z + (((size_t)(j0 + j) * 2 + p) * z_ls + i) * N + x;
                const u64 r = split ? fold_split(a0[j], a1[j], a2[j], P) : redc(a1[j], a0[j], P);
                *z = accumulate ? add_mod(*z, r, P.q) : r;
            }
    }
}

// ------------------------------------------------------------------------
// rescale
// ------------------------------------------------------------------------
// Rescale rounds: c <- floor((c + h) / q_l), h = (q_l - 1) / 2, so the
// error of every coefficient is centred (a floor biases all of them by -1/2,
// and decryption amplifies that bias at the slots near 1).  Per limb:
//   out_i = (in_i + [h]_{q_i} - [r]_{q_i}) * q_l^-1,  r = [in_l + h]_{q_l}.
// coefficient domain
__global__ void k_rescale_coef(const u64 *in, int in_ls, u64 *out, int out_ls, int level,
                               const PrimeC *__restrict__ primes, const u64 *__restrict__ tab,
                               int N)
{
    const int i = blockIdx.y, poly = blockIdx.z;
    const PrimeC P = primes[i], Pl = primes[level];
    const u64 inv = tab[2 * i], invs = tab[2 * i + 1];
    const u64 h = Pl.q >> 1, hi = reduce_word(h, P);
    const u64 *top = in + ((size_t)poly * in_ls + level) * N;
    const u64 *src = in + ((size_t)poly * in_ls + i) * N;
    u64 *dst = out + ((size_t)poly * out_ls + i) * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const u64 r = reduce_word(reduce_word(top[x], Pl) + h, Pl);
        dst[x] = shoup_mul(sub_mod(add_mod(src[x], hi, P.q), reduce_word(r, P), P.q), inv, invs, P.q);
    }
}

// the top limb l (coefficient domain, one per poly) -> [r]_{q_i} - [h]_{q_i}
// for i < level, r = [c_l + h]_{q_l}: what the rounded rescale subtracts
// (after its NTT) from limb i
__global__ void k_bcast_reduce(const u64 *r, int r_ls, int r_limb, u64 *out, int level,
                               const PrimeC *__restrict__ primes, int N)
{
    const int i = blockIdx.y, poly = blockIdx.z;
    const PrimeC P = primes[i], Pl = primes[r_limb];
    const u64 h = Pl.q >> 1, hi = reduce_word(h, P);
    const u64 *src = r + ((size_t)poly * r_ls + r_limb) * N;
    u64 *dst = out + ((size_t)poly * level + i) * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const u64 t = reduce_word(reduce_word(src[x], Pl) + h, Pl);
        dst[x] = sub_mod(reduce_word(t, P), hi, P.q);
    }
}

// NTT domain finish: ct_i = (ct_i - r_i) * q_l^-1
__global__ void k_rescale_finish(u64 *ct, int ls, const u64 *rr, int level,
                                 const PrimeC *__restrict__ primes, const u64 *__restrict__ tab,
                                 int N)
{
    const int i = blockIdx.y, poly = blockIdx.z;
    const u64 q = primes[i].q, inv = tab[2 * i], invs = tab[2 * i + 1];
    u64 *c = ct + ((size_t)poly * ls + i) * N;
    const u64 *r = rr + ((size_t)poly * level + i) * N;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x)
        c[x] = shoup_mul(sub_mod(c[x], r[x], q), inv, invs, q);
}


// ------------------------------------------------------------------------
// base conversion (approximate, no overflow correction):
//   out_p = sum_k [x_k * (B/b_k)^-1]_{b_k} * (B/b_k) mod p
// y_k in [0, b_k), (B/b_k) mod p in Montgomery form, n_in <= 8 products of
// two words below 2^61 accumulate below p * 2^64, so one Montgomery
// reduction gives the exact residue.
// ------------------------------------------------------------------------
// NMAX bounds T.n_in at compile time, so that y stays in registers.  y and
// the table hold 30-bit halves: at most 8 products per partial sum, and the
// total below 8 2^60 p keeps its high word below p for the Montgomery step.
template <int NMAX>
__device__ __forceinline__ u64 conv_point(const ConvTab &T, const u64 *y, int t, const PrimeC &P,
                                          int c = 0)
{
    static_assert(NMAX <= 8, "at most 8 inputs per conversion");
    u64 a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
    for (int k = 0; k < NMAX; k++)
        if (k < T.n_in) mac_split(a0, a1, a2, y[k], T.hmod[k][t]);
    // centred conversion: c B subtracted (c <= 7: the product adds below
    // 2^34 to the partial sums, within the 8-term bound for K <= 7)
    if (c) mac_split(a0, a1, a2, (u64)c, T.negb[t]);
    return reduce30<NMAX>(a0, a1, a2, P);
}

// returns the number of inputs y_k above b_k / 2: taking those as y_k - b_k
// centres the conversion (see k_moddown_conv)
template <int NMAX>
__device__ __forceinline__ int conv_inputs(const ConvTab &T, const u64 *src, size_t limb_stride,
                                           u64 *y, const PrimeC *__restrict__ primes)
{
    int c = 0;
#pragma unroll
    for (int k = 0; k < NMAX; k++)
        if (k < T.n_in) {
            const u64 v = src[(size_t)T.in_l[k] * limb_stride];
            const u64 b = primes[T.in_p[k]].q;
            const u64 yk = shoup_mul(v, T.hinv[k], T.hinv_s[k], b);
            c += yk > (b >> 1);
            y[k] = split30(yk);
        }
    return c;
}

// ModUp conversion.  c1c: [ncol][nl][N] coefficient domain (nl = level+1);
// digits: [ncol][beta][E][N]; writes every limb outside digit dg.
template <int NMAX>
__global__ void __launch_bounds__(256)
k_modup_conv(const u64 *__restrict__ c1c, int nl, u64 *digits, int beta, int E,
             const ConvTab *__restrict__ tabs, const PrimeC *__restrict__ primes, int N)
{
    const int f = blockIdx.z / beta, dg = blockIdx.z % beta;
    const ConvTab &T = tabs[dg];
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 y[NMAX];
    conv_inputs<NMAX>(T, c1c + (size_t)f * nl * N + x, N, y, primes);
    u64 *out = digits + ((size_t)f * beta + dg) * E * N;
    for (int t = 0; t < T.n_out; t++) {
        const PrimeC P = primes[T.out_p[t]];
        out[(size_t)T.out_l[t] * N + x] = conv_point<NMAX>(T, y, t, P);
    }
}

// ModDown conversion P -> q_0..q_level.  u: [npoly][E][N] (P limbs in the
// coefficient domain at positions level+1..), conv: [npoly][level+1][N].
// The ModDown's conversion is centred: y_k = [u_k (P/p_k)^-1]_{p_k} taken
// in (-p_k/2, p_k/2], i.e. the plain conversion minus c P with c the number
// of y_k above p_k/2.  Then (u - Conv)/P differs from u/P by minus
// sum_k y_k / p_k, which has mean zero; the plain conversion (y_k in
// [0, p_k)) biases every coefficient by -K/2, and in c1 decryption
// multiplies that bias by s and amplifies it at the slots near 1.
template <int NMAX>
__global__ void __launch_bounds__(256)
k_moddown_conv(const u64 *__restrict__ u, int E, u64 *conv, int nl,
               const ConvTab *__restrict__ tab, const PrimeC *__restrict__ primes, int N)
{
    const int poly = blockIdx.y;
    const ConvTab &T = *tab;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 y[NMAX];
    const int c = conv_inputs<NMAX>(T, u + (size_t)poly * E * N + x, N, y, primes);
    for (int t = 0; t < T.n_out; t++) {
        const PrimeC P = primes[T.out_p[t]];
        conv[((size_t)poly * nl + T.out_l[t]) * N + x] = conv_point<NMAX>(T, y, t, P, c);
    }
}

// A thread that owns two adjacent slots x, x+1 makes 16-byte accesses.  In the
// bit-reversed NTT order the automorphism maps every aligned pair {x, x+1}
// onto an aligned pair {2m, 2m+1}, so the gather is one 16-byte load plus a
// swap when sigma(x) is odd.
__device__ __forceinline__ ulonglong2 gather_pair(const u64 *limb, int m2, bool swap)
{
    const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(limb)[m2 >> 1];
    return swap ? make_ulonglong2(v.y, v.x) : v;
}

// ------------------------------------------------------------------------
// ModDown finish of one rotation:
//   out_p = (u_p - conv_p) * P^-1  (+ phi_g(c0) for p = 0)
// ------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
k_moddown_finish(const u64 *__restrict__ u, int E, const u64 *__restrict__ conv, const u64 *__restrict__ lane, int ls,
                 int ncol, int level, uint32_t g, int log_n, const u64 *__restrict__ pinv, u64 *out, int out_ls,
                 const PrimeC *__restrict__ primes)
{
    const int N = 1 << log_n;
    const int i = blockIdx.y;
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const u64 q = primes[i].q, pv = pinv[2 * i], pvs = pinv[2 * i + 1];
    const int sx = auto_src(x, g, log_n);
    const bool swap = sx & 1;
    const int nl = level + 1;
    for (int f = 0; f < ncol; f++) {
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const int poly = f * 2 + p;
            const ulonglong2 uu = *reinterpret_cast<const ulonglong2 *>(u + ((size_t)poly * E + i) * N + x);
            const ulonglong2 cc = *reinterpret_cast<const ulonglong2 *>(conv + ((size_t)poly * nl + i) * N + x);
            u64 r0 = shoup_mul(sub_mod(uu.x, cc.x, q), pv, pvs, q);
            u64 r1 = shoup_mul(sub_mod(uu.y, cc.y, q), pv, pvs, q);
            if (p == 0) {
                const ulonglong2 c0 = gather_pair(lane + ((size_t)(f * 2) * ls + i) * N, sx, swap);
                r0 = add_mod(r0, c0.x, q);
                r1 = add_mod(r1, c0.y, q);
            }
            *reinterpret_cast<ulonglong2 *>(out + ((size_t)poly * out_ls + i) * N + x) = make_ulonglong2(r0, r1);
        }
    }
}

constexpr int kMaxDest = 8;
struct DestList {
    int n;
    int out_ls;
    u64 *out[kMaxDest];
    const u64 *mask[kMaxDest];
};

// out_d += mask_d (x) lane (the kept values of a lane, rotation 0)
__global__ void __launch_bounds__(256)
k_stay_mac(const u64 *__restrict__ lane, int ls, int ncol, int level, const DestList dl,
           const PrimeC *__restrict__ primes, int N)
{
    const int i = blockIdx.y;
    const int x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x >= N) return;
    const PrimeC P = primes[i];
    ulonglong2 m[kMaxDest];
#pragma unroll
    for (int d = 0; d < kMaxDest; d++)
        if (d < dl.n) {
            m[d] = *reinterpret_cast<const ulonglong2 *>(dl.mask[d] + (size_t)i * N + x);
            m[d] = make_ulonglong2(join_word(m[d].x, P.q), join_word(m[d].y, P.q));
        }
    for (int f = 0; f < ncol; f++) {
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const int poly = f * 2 + p;
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(lane + ((size_t)poly * ls + i) * N + x);
#pragma unroll
            for (int d = 0; d < kMaxDest; d++) {
                if (d < dl.n) {
                    ulonglong2 *o = reinterpret_cast<ulonglong2 *>(dl.out[d] + ((size_t)poly * dl.out_ls + i) * N + x);
                    ulonglong2 ov = *o;
                    ov.x = add_mod(ov.x, mont_mul(v.x, m[d].x, P), P.q);
                    ov.y = add_mod(ov.y, mont_mul(v.y, m[d].y, P), P.q);
                    *o = ov;
                }
            }
        }
    }
}

// ModDown followed by the rescale by q_l, equal word for word to the two
// done in turn.  With conv_i the base conversion of the special limbs and
// o_l = (ext_l - conv_l) P^-1 mod q_l (coefficient domain: the limb the
// rescale drops), the rescaled limbs are
//   ((ext_i - conv_i) P^-1 - [o_l]_{q_i}) q_l^-1 = (ext_i - (conv_i + P o_l)) (P q_l)^-1,
// so one forward NTT of w_i = conv_i + P o_l mod q_i per kept limb replaces
// the NTT of conv_i and the rescale's NTT of [o_l]_{q_i}.  The conversion
// is centred (see k_moddown_conv) and the rescale rounds: its offset
// (q_l - 1) / 2, seen before the division by P, is H = P (q_l - 1) / 2,
// which vanishes on the special limbs, enters limb l through o_l and the
// kept limbs as w_i - [H]_{q_i}.
// ext: [npoly][E][N], limbs l and l+1.. in the coefficient domain;
// w: [npoly][l][N] coefficient domain.
template <int NMAX>
__global__ void __launch_bounds__(256)
k_moddown_rescale_conv(const u64 *__restrict__ ext, int E, u64 *w, int l,
                       const ConvTab *__restrict__ tab, const u64 *__restrict__ pinv,
                       const u64 *__restrict__ hq,
                       const PrimeC *__restrict__ primes, int N)
{
    const int poly = blockIdx.y;
    const ConvTab &T = *tab;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 y[NMAX];
    const int c = conv_inputs<NMAX>(T, ext + (size_t)poly * E * N + x, N, y, primes);
    const PrimeC Pl = primes[l];
    // hq[i] = [H]_{q_i}, H = P (q_l - 1) / 2
    const u64 el = add_mod(ext[((size_t)poly * E + l) * N + x], hq[l], Pl.q);
    const u64 ol = shoup_mul(sub_mod(el, conv_point<NMAX>(T, y, l, Pl, c), Pl.q), pinv[2 * l],
                             pinv[2 * l + 1], Pl.q);
    // conv_t + P o_l - H = sum_k y_k h_k + P (o_l - c + 8) - (H + 8 P): one more
    // term and a constant of the same sums, reduced once (c <= 7: at most seven
    // special primes; the constant, a reduced word, goes whole into the lowest
    // sum).  With a Shoup product for P o_l, a term for c and an addition for H
    // this kernel took a quarter longer: 4.24 against 3.38 ms in a layer of 29
    // launches of 32 polynomials, N = 2^16, four special primes.
    const u64 o = split30(ol + (u64)(8 - c));
    for (int t = 0; t < l; t++) {
        const PrimeC P = primes[t];
        u64 a0 = hq[l + 1 + t], a1 = 0, a2 = 0;
#pragma unroll
        for (int k = 0; k < NMAX; k++)
            if (k < T.n_in) mac_split(a0, a1, a2, y[k], T.hmod[k][t]);
        mac_split(a0, a1, a2, o, T.posb[t]);
        w[((size_t)poly * l + t) * N + x] = reduce30<(NMAX < 8 ? NMAX + 1 : 8)>(a0, a1, a2, P);
    }
}

// ModDown + rescale at N = 2^16, the conversion fused into the first NTT
// pass of w (see k_moddown_rescale_conv for what w is).  First
// k_moddown_prep, per coefficient of each polynomial: y_k (the inverse NTT
// of the special limbs scaled to [u_k (P/p_k)^-1]_{p_k}), c = #{y_k > p_k/2},
// o_l = ((ext_l + [H]_{q_l}) - Conv_l(y) + c [P]_{q_l}) P^-1 mod q_l, and
// o_l | c << 60 written over limb l (q_l < 2^60; limb l is not read again).
// Then k_moddown_ntt16_a per (column tile, kept limb t, polynomial): w_t =
// Conv_t(y, c) + P o_l - [H]_{q_t} mod q_t, straight into pass A of w_t.
template <int NMAX>
__global__ void __launch_bounds__(256)
k_moddown_prep(u64 *ext, int E, int l, const ConvTab *__restrict__ tab, const u64 *__restrict__ pinv,
               const u64 *__restrict__ hq, const PrimeC *__restrict__ primes, int N)
{
    const int poly = blockIdx.y;
    const ConvTab &T = *tab;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    u64 y[NMAX];
    int c = 0;
    const u64 *src = ext + (size_t)poly * E * N + x;
#pragma unroll
    for (int k = 0; k < NMAX; k++)
        if (k < T.n_in) {
            const u64 yk = src[(size_t)T.in_l[k] * N];
            c += yk > (primes[T.in_p[k]].q >> 1);
            y[k] = split30(yk);
        }
    const PrimeC Pl = primes[l];
    u64 *el = ext + ((size_t)poly * E + l) * N + x;
    const u64 e = add_mod(*el, hq[l], Pl.q);
    const u64 ol = shoup_mul(sub_mod(e, conv_point<NMAX>(T, y, l, Pl, c), Pl.q), pinv[2 * l], pinv[2 * l + 1], Pl.q);
    *el = ol | ((u64)c << 60);
}

template <int NMAX, bool OD>
__global__ void __launch_bounds__(256, OD ? 4 : 3)
k_moddown_ntt16_a(const u64 *__restrict__ ext, int E, u64 *w, int l, const ConvTab *__restrict__ tab,
                  const u64 *__restrict__ pmodq, const u64 *__restrict__ hq,
                  const PrimeC *__restrict__ primes, const ulonglong2 *__restrict__ tw)
{
    const int t = blockIdx.y, poly = blockIdx.z;
    const ConvTab &T = *tab;
    __shared__ u64 sm[256 * 16];
    __shared__ ulonglong2 stw[256];
    const PrimeC P = primes[t];
    const ulonglong2 *twp = tw + (size_t)t * 65536;
    stw[threadIdx.x] = twp[threadIdx.x];
    const u64 pw = pmodq[2 * t], pws = pmodq[2 * t + 1], ht = hq[t];
    u64 hm_[NMAX], nb = T.negb[t];
#pragma unroll
    for (int k = 0; k < NMAX; k++) hm_[k] = k < T.n_in ? T.hmod[k][t] : 0;
    const u64 *base = ext + (size_t)poly * E * 65536;
    const int c = threadIdx.x & 15, r = threadIdx.x >> 4, c0 = blockIdx.x * 16;
    u64 v[16];
#pragma unroll
    for (int m = 0; m < 16; m++) {
        const size_t idx = (size_t)(r + 16 * m) * 256 + c0 + c;
        const u64 pk = base[(size_t)l * 65536 + idx];
        const u64 ol = pk & ((1ull << 60) - 1);
        const int cc = (int)(pk >> 60);
        u64 a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
        for (int k = 0; k < NMAX; k++)
            if (k < T.n_in) mac_split(a0, a1, a2, split30(base[(size_t)T.in_l[k] * 65536 + idx]), hm_[k]);
        if (cc) mac_split(a0, a1, a2, (u64)cc, nb);
        const u64 conv = reduce30<NMAX>(a0, a1, a2, P);
        v[m] = sub_mod(add_mod(conv, shoup_mul(ol, pw, pws, P.q), P.q), ht, P.q);
    }
    __syncthreads();   // stw
    u64 *d = w + ((size_t)poly * l + t) * 65536 + c0;
    if (P.q < (1ull << 47)) fwd_a16_rounds<true, 16, OD>(v, d, stw, P.q, sm);
    else fwd_a16_rounds<false, 16, OD>(v, d, stw, P.q, sm);
}

// residues mod the special primes of a polynomial given by its limb 0,
// read as a centred integer (valid when |coefficient| < q_0 / 2)
__global__ void k_lift_special(const u64 *limb0, u64 q0, u64 *out, int np, int nq,
                               const PrimeC *__restrict__ primes, int N)
{
    const int k = blockIdx.y;
    const PrimeC P = primes[nq + k];
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < N; x += gridDim.x * blockDim.x) {
        const u64 v = limb0[x];
        u64 r;
        if (v <= q0 / 2) {
            r = reduce_word(v, P);
        } else {
            const u64 m = reduce_word(q0 - v, P);
            r = m ? P.q - m : 0;
        }
        out[(size_t)k * N + x] = r;
    }
}

}  // namespace

// ========================================================================
// host wrappers
// ========================================================================
// launch a kernel templated on the number of base-conversion inputs
#define FG_NIN_DISPATCH(n, LAUNCH)                                               \
    switch (n) {                                                                 \
    case 1: LAUNCH(1); break;                                                    \
    case 2: LAUNCH(2); break;                                                    \
    case 3: LAUNCH(3); break;                                                    \
    case 4: LAUNCH(4); break;                                                    \
    case 5: LAUNCH(5); break;                                                    \
    case 6: LAUNCH(6); break;                                                    \
    case 7: LAUNCH(7); break;                                                    \
    case 8: LAUNCH(8); break;                                                    \
    default: throw fg_error(FG_EINVAL, "base conversion with more than 8 inputs"); \
    }

namespace kern {

KTimer::KTimer(fg_ctx *c, const char *cls, double alg_bytes) : ctx(c), bytes(alg_bytes)
{
    on = !c->time_class.empty() && c->time_class == cls;
    if (on) {
        a = c->event();
        cudaEventRecord(a, c->stream);
    }
}

KTimer::~KTimer()
{
    if (on) {
        cudaEvent_t b = ctx->event();
        cudaEventRecord(b, ctx->stream);
        ctx->timed.push_back({a, b, bytes});
    }
}


// N = 2^16 forward pass B alone (the whole second half of a transform), in
// place on bt.dst or finished
template <bool OD>
static void ntt16_pass_b_od(fg_ctx *ctx, const Batch &bt, int count, const Finish *fin = nullptr)
{
    const auto *fwd = (const ulonglong2 *)ctx->d_fwd;
    const auto *rows = (const ulonglong2 *)ctx->d_fwd_rows;
    const int R = ctx->tune.ntt_rows == 8 ? 8 : 16;
    auto kern = R == 8 ? (fin ? ntt16_fwd_b<8, OD, true> : ntt16_fwd_b<8, OD, false>)
                       : (fin ? ntt16_fwd_b<16, OD, true> : ntt16_fwd_b<16, OD, false>);
    kern<<<dim3(256 / R, count), 16 * R, 0, ctx->stream>>>(bt, ctx->d_primes, fwd, rows, fin ? *fin : Finish());
}

template <int COLS, int ROWS, bool OD>
static void ntt16_launch_t(fg_ctx *ctx, const Batch &bt, int count, bool inverse, const u64 *col_scale,
                           const Finish *fin)
{
    const auto *fwd = (const ulonglong2 *)ctx->d_fwd;
    const auto *inv = (const ulonglong2 *)ctx->d_inv;
    dim3 gA(256 / COLS, count), gB(256 / ROWS, count);
    Batch b2 = bt;
    b2.src = b2.dst;
    b2.src_stride = b2.dst_stride;
    if (!inverse) {
        ntt16_fwd_a<COLS, OD><<<gA, 16 * COLS, 0, ctx->stream>>>(bt, ctx->d_primes, fwd);
        ntt16_pass_b_od<OD>(ctx, b2, count, fin);
    } else {
        ntt16_inv_b<ROWS, OD><<<gB, 16 * ROWS, 0, ctx->stream>>>(bt, ctx->d_primes, inv,
                                                                (const ulonglong2 *)ctx->d_inv_rows);
        ntt16_inv_a<COLS, OD><<<gA, 16 * COLS, 0, ctx->stream>>>(b2, ctx->d_primes, inv, ctx->d_ninv,
                                                                col_scale);
    }
}

// the tile and twiddle form of the N = 2^16 transform from the context's tuning
template <bool OD>
static void ntt16_launch_od(fg_ctx *ctx, const Batch &bt, int count, bool inverse, const u64 *col_scale,
                            const Finish *fin)
{
    const bool ca = ctx->tune.ntt_cols == 8, rb = ctx->tune.ntt_rows == 8;
    if (!ca && !rb) ntt16_launch_t<16, 16, OD>(ctx, bt, count, inverse, col_scale, fin);
    else if (ca && !rb) ntt16_launch_t<8, 16, OD>(ctx, bt, count, inverse, col_scale, fin);
    else if (!ca && rb) ntt16_launch_t<16, 8, OD>(ctx, bt, count, inverse, col_scale, fin);
    else ntt16_launch_t<8, 8, OD>(ctx, bt, count, inverse, col_scale, fin);
}

static void ntt16_launch(fg_ctx *ctx, const Batch &bt, int count, bool inverse,
                         const u64 *col_scale = nullptr, const Finish *fin = nullptr)
{
    if (ctx->tune.ntt_tw) ntt16_launch_od<true>(ctx, bt, count, inverse, col_scale, fin);
    else ntt16_launch_od<false>(ctx, bt, count, inverse, col_scale, fin);
}

static void launch_ntt(fg_ctx *ctx, const LimbSet &src, const LimbSet &dst, bool inverse, const Finish *fin = nullptr)
{
    FG_CHECK(src.per_row == dst.per_row && src.rows == dst.rows, FG_EINVAL, "ntt: shape mismatch");
    if (src.rows == 0 || src.per_row == 0) return;
    Batch bt = make_batch(src.base, src.stride, dst.base, dst.stride, src.per_row, src.rows,
                          src.pidx);
    const int count = src.rows * src.per_row;
    FG_CHECK(count <= 65535, FG_EINVAL, "ntt: more than 65535 limbs in one batch");
    int active = 0;
    for (int v : src.pidx) active += v >= 0;
    // finishing: ext read as well, and out when it accumulates
    KTimer kt(ctx, "ntt", (double)active * src.rows * ctx->n * 8 * (fin ? 3 + fin->accumulate : 2));
    if (ctx->log_n < 16) {
        ntt_small(ctx, bt, count, active * src.rows, inverse, fin);
        return;
    }
    ntt16_launch(ctx, bt, count, inverse, nullptr, fin);
    check_launch(ctx, "ntt", 2);
}

void ntt_fwd(fg_ctx *ctx, const LimbSet &src, const LimbSet &dst) { launch_ntt(ctx, src, dst, false); }
void ntt_inv(fg_ctx *ctx, const LimbSet &src, const LimbSet &dst) { launch_ntt(ctx, src, dst, true); }

static inline dim3 ew_grid(int N, int count) { return dim3((N + 255) / 256, count); }

static Batch contiguous(u64 *p, int count, const std::vector<int> &pidx)
{
    const int per = (int)pidx.size();
    return make_batch(p, per, p, per, per, count / per, pidx);
}

void to_mont(fg_ctx *ctx, u64 *data, int count, const std::vector<int> &pidx, bool split, bool times_p)
{
    if (!count) return;
    KTimer kt(ctx, "to_mont", 0);
    k_to_mont<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(contiguous(data, count, pidx),
                                                               ctx->d_primes, ctx->n, split ? 1 : 0,
                                                               times_p ? ctx->d_pmodq : nullptr, ctx->nq);
    check_launch(ctx, "to_mont");
}

void from_mont(fg_ctx *ctx, u64 *data, int count, const std::vector<int> &pidx)
{
    if (!count) return;
    KTimer kt(ctx, "from_mont", 0);
    k_from_mont<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(contiguous(data, count, pidx),
                                                                 ctx->d_primes, ctx->n);
    check_launch(ctx, "from_mont");
}

void pointwise(fg_ctx *ctx, const u64 *a, const u64 *b, u64 *c, int count,
               const std::vector<int> &pidx)
{
    if (!count) return;
    KTimer kt(ctx, "pointwise", 0);
    k_pointwise<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(
        a, b, c, contiguous(c, count, pidx), ctx->d_primes, ctx->n);
    check_launch(ctx, "pointwise");
}

void add(fg_ctx *ctx, const u64 *a, const u64 *b, u64 *c, int count, const std::vector<int> &pidx)
{
    if (!count) return;
    KTimer kt(ctx, "add", 0);
    k_add<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(a, b, c, contiguous(c, count, pidx),
                                                           ctx->d_primes, ctx->n);
    check_launch(ctx, "add");
}

void tensor(fg_ctx *ctx, const u64 *a, const u64 *b, u64 *lane, u64 *d1, int n, int nl)
{
    KTimer kt(ctx, "tensor", (double)n * nl * ctx->n * 8 * (a == b ? 5 : 7));
    k_tensor<<<dim3(ctx->n / 256, nl, n), 256, 0, ctx->stream>>>(a, b, lane, d1, nl, ctx->d_primes, ctx->d_pmodq, ctx->n);
    check_launch(ctx, "tensor");
}

void add_part1(fg_ctx *ctx, u64 *u, int E, const u64 *d, int n, int nl)
{
    KTimer kt(ctx, "add", (double)n * nl * ctx->n * 8 * 3);
    k_add_part1<<<dim3(ctx->n / 256, nl, n), 256, 0, ctx->stream>>>(u, E, d, nl, ctx->d_primes, ctx->n);
    check_launch(ctx, "add_part1");
}

void neg(fg_ctx *ctx, const u64 *a, u64 *c, int count, const std::vector<int> &pidx)
{
    if (!count) return;
    KTimer kt(ctx, "neg", 0);
    k_neg<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(a, c, contiguous(c, count, pidx),
                                                           ctx->d_primes, ctx->n);
    check_launch(ctx, "neg");
}

void scalar(fg_ctx *ctx, const u64 *a, u64 *c, int count, const std::vector<int> &pidx,
            const u64 *d_scal)
{
    if (!count) return;
    KTimer kt(ctx, "scalar", 0);
    k_scalar<<<ew_grid(ctx->n, count), 256, 0, ctx->stream>>>(
        a, c, contiguous(c, count, pidx), ctx->d_primes, d_scal, ctx->n);
    check_launch(ctx, "scalar");
}

void automorphism(fg_ctx *ctx, const u64 *a, u64 *c, int nlimbs, uint32_t g)
{
    if (!nlimbs) return;
    KTimer kt(ctx, "automorphism", 0);
    k_automorphism<<<ew_grid(ctx->n, nlimbs), 256, 0, ctx->stream>>>(a, c, nlimbs, g, ctx->log_n);
    check_launch(ctx, "automorphism");
}

void small_to_res(fg_ctx *ctx, const int8_t *e, u64 *out, int n_limbs, const int *d_pidx)
{
    KTimer kt(ctx, "small_to_res", 0);
    k_small_to_res<<<ew_grid(ctx->n, n_limbs), 256, 0, ctx->stream>>>(e, out, d_pidx,
                                                                      ctx->d_primes, ctx->n);
    check_launch(ctx, "small_to_res");
}

void expand_uniform(fg_ctx *ctx, cudaStream_t st, u64 *ct, size_t ct_pitch, const u64 *c0, int ncols,
                    int nl, u64 seed, u64 index0)
{
    if (!ncols || !nl) return;
    FG_CHECK(ncols <= 65535 && nl <= ctx->nq, FG_EINVAL, "expand_uniform: bad shape");
    dim3 g((ctx->n + 255) / 256, nl, ncols);
    k_expand_uniform<<<g, 256, 0, st>>>(ct, ct_pitch, c0, nl, seed, hm::kSeededPurpose, index0,
                                        ctx->d_primes, ctx->n);
    check_launch(ctx, "expand_uniform");
}

void copy_limbs(fg_ctx *ctx, const u64 *src, int src_ls, u64 *dst, int dst_ls, int npoly, int nl)
{
    if (!npoly || !nl) return;
    KTimer kt(ctx, "copy", (double)npoly * nl * ctx->n * 16);
    dim3 g((ctx->n + 255) / 256, nl, npoly);
    k_copy_limbs<<<g, 256, 0, ctx->stream>>>(src, src_ls, dst, dst_ls, nl, ctx->n);
    check_launch(ctx, "copy_limbs");
}

void comb_const_mac(fg_ctx *ctx, const u64 *X, int F, int Fp, int level, const u64 *consts, u64 *Z,
                    int z_ls, int fb, int fe, bool accumulate)
{
    // split partial sums stay below 2^64 for up to 2^16 terms
    FG_CHECK(F < (1 << 16), FG_EINVAL, "combination over more than 2^16 input columns");
    if (fe < 0) fe = F;
    FG_CHECK(0 <= fb && fb < fe && fe <= F, FG_EINVAL, "combination column range");
    const int nj = (Fp + kCombJ - 1) / kCombJ;
    // inputs read once, outputs written once (read too when accumulating)
    KTimer kt(ctx, "comb", ((double)(fe - fb) + Fp * (accumulate ? 2 : 1)) * 2 * (level + 1) * ctx->n * 8);
    dim3 g(((ctx->n + 255) / 256) * nj, level + 1, 2);
    k_comb<<<g, 256, 0, ctx->stream>>>(X, F, fb, fe, accumulate ? 1 : 0, Fp, nj, level, consts, Z, z_ls,
                                       ctx->d_primes, ctx->n);
    check_launch(ctx, "comb");
}

void rescale_coef(fg_ctx *ctx, const u64 *in, int in_ls, u64 *out, int out_ls, int npoly, int level)
{
    FG_CHECK(level >= 1, FG_ELEVEL, "rescale needs level >= 1");
    KTimer kt(ctx, "rescale", (double)npoly * (2 * level + 1) * ctx->n * 8);
    dim3 g((ctx->n + 255) / 256, level, npoly);
    k_rescale_coef<<<g, 256, 0, ctx->stream>>>(in, in_ls, out, out_ls, level, ctx->d_primes,
                                               ctx->rescale_tab(level), ctx->n);
    check_launch(ctx, "rescale_coef");
}

void rescale_ntt(fg_ctx *ctx, u64 *ct, int ls, int npoly, int level)
{
    FG_CHECK(level >= 1, FG_ELEVEL, "rescale needs level >= 1");
    const int N = ctx->n;
    // top limb back to the coefficient domain (in place; it is dropped anyway)
    std::vector<int> top(ls, -1);
    top[level] = level;
    LimbSet s{ct, ls, ls, npoly, top};
    ntt_inv(ctx, s, s);
    u64 *rr = (u64 *)ctx->buf("rescale_r", (size_t)npoly * level * N * 8);
    dim3 g((N + 255) / 256, level, npoly);
    {
        KTimer kt(ctx, "rescale", (double)npoly * (level + 1) * N * 8);
        k_bcast_reduce<<<g, 256, 0, ctx->stream>>>(ct, ls, level, rr, level, ctx->d_primes, N);
        check_launch(ctx, "bcast_reduce");
    }
    std::vector<int> pid(level);
    for (int i = 0; i < level; i++) pid[i] = i;
    LimbSet r{rr, level, level, npoly, pid};
    ntt_fwd(ctx, r, r);
    KTimer kt(ctx, "rescale", (double)npoly * level * N * 8 * 3);
    k_rescale_finish<<<g, 256, 0, ctx->stream>>>(ct, ls, rr, level, ctx->d_primes,
                                                 ctx->rescale_tab(level), N);
    check_launch(ctx, "rescale_finish");
}

// ModUp at N = 2^16 with the conversion fused into the digits' first NTT
// pass: the inverse NTT of c1 scaled to give the conversion's inputs y_i,
// one kernel per (column, digit, output limb, column tile) converting and
// running stages 0..7, then pass B over every digit limb
template <bool OD>
static void modup16_fused(fg_ctx *ctx, const u64 *lane, int ls, int ncol, int level, u64 *digits)
{
    const int N = ctx->n, nl = level + 1, E = ctx->ext(level), beta = ctx->n_digits(level);
    u64 *y = (u64 *)ctx->buf("modup_c1", (size_t)ncol * nl * N * 8);
    std::vector<int> pid(nl);
    for (int i = 0; i < nl; i++) pid[i] = i;
    {
        Batch bt = make_batch(const_cast<u64 *>(lane) + (size_t)ls * N, 2 * ls, y, nl, nl, ncol, pid);
        KTimer kt(ctx, "ntt", (double)nl * ncol * N * 8 * 2);
        ntt16_launch(ctx, bt, ncol * nl, true, ctx->modup_scale_tab(level));
        check_launch(ctx, "ntt", 2);
    }
    const int nmax = std::min(ctx->alpha, nl);
    int n_out = 0;
    for (int d = 0; d < beta; d++) n_out = std::max(n_out, E - std::min(ctx->alpha, nl - d * ctx->alpha));
    const ConvTab *tabs = ctx->modup_tabs(level);
    const auto *fwd = (const ulonglong2 *)ctx->d_fwd;
    {
        KTimer kt(ctx, "modup_conv", (double)ncol * (nl + (double)beta * (E - ctx->alpha)) * N * 8);
        const bool c8 = ctx->tune.ntt_cols == 8;
        dim3 g(c8 ? 32 : 16, n_out, ncol * beta);
#define FG_LAUNCH(M)                                                                                  \
        if (c8)                                                                                       \
            k_modup_ntt16_a<M, 8, OD><<<g, 128, 0, ctx->stream>>>(y, nl, digits, beta, E, tabs,       \
                                                                  ctx->d_primes, fwd);                \
        else                                                                                          \
            k_modup_ntt16_a<M, 16, OD><<<g, 256, 0, ctx->stream>>>(y, nl, digits, beta, E, tabs,      \
                                                                   ctx->d_primes, fwd)
        FG_NIN_DISPATCH(nmax, FG_LAUNCH)
#undef FG_LAUNCH
        check_launch(ctx, "modup_ntt16_a");
    }
    std::vector<int> dp(beta * E);
    for (int d = 0; d < beta; d++)
        for (int i = 0; i < E; i++)
            dp[d * E + i] = (i <= level && i / ctx->alpha == d) ? -1 : ctx->ext_prime(level, i);
    Batch bd = make_batch(digits, beta * E, digits, beta * E, beta * E, ncol, dp);
    int active = 0;
    for (int v : dp) active += v >= 0;
    KTimer kt(ctx, "ntt", (double)active * ncol * N * 8 * 2 / 2);
    ntt16_pass_b_od<OD>(ctx, bd, ncol * beta * E);
    check_launch(ctx, "ntt16_fwd_b");
}

void modup(fg_ctx *ctx, const u64 *lane, int ls, int ncol, int level, u64 *digits)
{
    if (ctx->log_n == 16 && ctx->tune.modup_fused) {
        if (ctx->tune.ntt_tw) modup16_fused<true>(ctx, lane, ls, ncol, level, digits);
        else modup16_fused<false>(ctx, lane, ls, ncol, level, digits);
        return;
    }
    const int N = ctx->n, nl = level + 1, E = ctx->ext(level), beta = ctx->n_digits(level);
    u64 *c1c = (u64 *)ctx->buf("modup_c1", (size_t)ncol * nl * N * 8);
    std::vector<int> pid(nl);
    for (int i = 0; i < nl; i++) pid[i] = i;
    LimbSet src{const_cast<u64 *>(lane) + (size_t)ls * N, 2 * ls, nl, ncol, pid};
    LimbSet dst{c1c, nl, nl, ncol, pid};
    ntt_inv(ctx, src, dst);
    dim3 g((N + 255) / 256, 1, ncol * beta);
    {
    KTimer kt(ctx, "modup_conv", (double)ncol * (nl + (double)beta * E - nl) * N * 8);
#define FG_LAUNCH(M)                                                                       \
    k_modup_conv<M><<<g, 256, 0, ctx->stream>>>(c1c, nl, digits, beta, E, ctx->modup_tabs(level), \
                                                ctx->d_primes, N)
    FG_NIN_DISPATCH(std::min(ctx->alpha, nl), FG_LAUNCH)
#undef FG_LAUNCH
    check_launch(ctx, "modup_conv");
    }
    std::vector<int> dp(beta * E);
    for (int d = 0; d < beta; d++)
        for (int i = 0; i < E; i++)
            dp[d * E + i] = (i <= level && i / ctx->alpha == d) ? -1 : ctx->ext_prime(level, i);
    LimbSet ds{digits, beta * E, beta * E, ncol, dp};
    ntt_fwd(ctx, ds, ds);
}

void rotate(fg_ctx *ctx, const KeyDev &key, const u64 *lane, int ls, int ncol, int level, const u64 *digits, u64 *out,
            int out_ls)
{
    const int N = ctx->n, nl = level + 1, E = ctx->ext(level), beta = ctx->n_digits(level);
    u64 *u = (u64 *)ctx->buf("ks_u", (size_t)ncol * 2 * E * N * 8);
    ks_launch(ctx, {&key}, {u}, lane, ls, ncol, level, digits, false);
    std::vector<int> pp(E);
    for (int i = 0; i < E; i++) pp[i] = i <= level ? -1 : ctx->ext_prime(level, i);
    LimbSet us{u, E, E, 2 * ncol, pp};
    ntt_inv(ctx, us, us);
    u64 *conv = (u64 *)ctx->buf("ks_conv", (size_t)ncol * 2 * nl * N * 8);
    dim3 g2((N + 255) / 256, 2 * ncol);
    {
    KTimer kt(ctx, "moddown_conv", (double)2 * ncol * (ctx->np + nl) * N * 8);
#define FG_LAUNCH(M)                                                                       \
    k_moddown_conv<M><<<g2, 256, 0, ctx->stream>>>(u, E, conv, nl, ctx->moddown_tab(level),   \
                                                   ctx->d_primes, N)
    FG_NIN_DISPATCH(ctx->np, FG_LAUNCH)
#undef FG_LAUNCH
    check_launch(ctx, "moddown_conv");
    }
    std::vector<int> pq(nl);
    for (int i = 0; i < nl; i++) pq[i] = i;
    LimbSet cs{conv, nl, nl, 2 * ncol, pq};
    ntt_fwd(ctx, cs, cs);
    dim3 g3((N / 2 + 255) / 256, nl);
    KTimer kt(ctx, "moddown_mac", (double)7 * ncol * nl * N * 8);
    k_moddown_finish<<<g3, 256, 0, ctx->stream>>>(u, E, conv, lane, ls, ncol, level, key.galois, ctx->log_n,
                                                  ctx->pinv_tab(level), out, out_ls, ctx->d_primes);
    check_launch(ctx, "moddown_finish");
}

void stay_mac(fg_ctx *ctx, const u64 *lane, int ls, int ncol, int level,
              const std::vector<Dest> &dests, int out_ls)
{
    const int N = ctx->n;
    for (size_t d0 = 0; d0 < dests.size(); d0 += kMaxDest) {
        DestList dl;
        dl.n = (int)std::min<size_t>(kMaxDest, dests.size() - d0);
        dl.out_ls = out_ls;
        for (int d = 0; d < dl.n; d++) {
            dl.out[d] = dests[d0 + d].out;
            dl.mask[d] = dests[d0 + d].mask;
        }
        dim3 g((N / 2 + 255) / 256, level + 1);
        const int nl = level + 1;
        KTimer kt(ctx, "stay_mac", ((double)2 * ncol * nl + (double)dl.n * nl +
                                     (double)dl.n * ncol * 2 * nl * 2) * N * 8);
        k_stay_mac<<<g, 256, 0, ctx->stream>>>(lane, ls, ncol, level, dl, ctx->d_primes, N);
        check_launch(ctx, "stay_mac");
    }
}


void lift_special(fg_ctx *ctx, const u64 *limb0, u64 *out)
{
    KTimer kt(ctx, "lift", 0);
    k_lift_special<<<ew_grid(ctx->n, ctx->np), 256, 0, ctx->stream>>>(limb0, ctx->primes[0], out,
                                                                      ctx->np, ctx->nq,
                                                                      ctx->d_primes, ctx->n);
    check_launch(ctx, "lift_special");
}

// ModDown + rescale at N = 2^16 with the conversion fused into w's first
// NTT pass (see k_moddown_ntt16_a)
template <bool OD>
static void moddown16_fused(fg_ctx *ctx, u64 *ext, int ncol, int level, u64 *out, int ls, bool accumulate)
{
    const int N = ctx->n, l = level, E = ctx->ext(level), npoly = 2 * ncol;
    std::vector<int> pp(E, -1);
    pp[l] = l;
    for (int i = l + 1; i < E; i++) pp[i] = ctx->ext_prime(level, i);
    {
        Batch bt = make_batch(ext, E, ext, E, E, npoly, pp);
        KTimer kt(ctx, "ntt", (double)npoly * (ctx->np + 1) * N * 8 * 2);
        ntt16_launch(ctx, bt, npoly * E, true, ctx->moddown_scale_tab(level));
        check_launch(ctx, "ntt", 2);
    }
    u64 *w = (u64 *)ctx->buf("ks_conv", (size_t)npoly * l * N * 8);
    const ConvTab *tab = ctx->moddown_tab(level);
    const u64 *hq = ctx->moddown_rescale_half_tab(level);
    {
        KTimer kt(ctx, "moddown_conv", (double)npoly * (ctx->np + 2 + l) * N * 8);
        dim3 g1((N + 255) / 256, npoly);
#define FG_LAUNCH(M) \
        k_moddown_prep<M><<<g1, 256, 0, ctx->stream>>>(ext, E, l, tab, ctx->pinv_tab(level), hq, ctx->d_primes, N)
        FG_NIN_DISPATCH(ctx->np, FG_LAUNCH)
#undef FG_LAUNCH
        check_launch(ctx, "moddown_prep");
        dim3 g2(16, l, npoly);
#define FG_LAUNCH(M)                                                                                \
        k_moddown_ntt16_a<M, OD><<<g2, 256, 0, ctx->stream>>>(ext, E, w, l, tab, ctx->d_pmodq, hq,    \
                                                              ctx->d_primes,                          \
                                                              (const ulonglong2 *)ctx->d_fwd)
        FG_NIN_DISPATCH(ctx->np, FG_LAUNCH)
#undef FG_LAUNCH
        check_launch(ctx, "moddown_ntt16_a");
    }
    {
        std::vector<int> pq(l);
        for (int i = 0; i < l; i++) pq[i] = i;
        Batch bw = make_batch(w, l, w, l, l, npoly, pq);
        const Finish fin{ext, out, ctx->moddown_rescale_tab(level), E, ls, accumulate ? 1 : 0};
        KTimer kt(ctx, "ntt", (double)npoly * l * N * 8 * (2 + fin.accumulate));
        ntt16_pass_b_od<OD>(ctx, bw, npoly * l, &fin);
        check_launch(ctx, "ntt16_fwd_b");
    }
}

void moddown_rescale_to_lane(fg_ctx *ctx, u64 *ext, int ncol, int level, u64 *out, int ls, bool accumulate)
{
    if (ctx->log_n == 16 && ctx->tune.moddown_fused && level >= 1) {
        if (ctx->tune.ntt_tw) moddown16_fused<true>(ctx, ext, ncol, level, out, ls, accumulate);
        else moddown16_fused<false>(ctx, ext, ncol, level, out, ls, accumulate);
        return;
    }
    FG_CHECK(level >= 1, FG_ELEVEL, "rescale needs level >= 1");
    const int N = ctx->n, l = level, E = ctx->ext(level), npoly = 2 * ncol;
    std::vector<int> pp(E, -1);
    pp[l] = l;
    for (int i = l + 1; i < E; i++) pp[i] = ctx->ext_prime(level, i);
    LimbSet us{ext, E, E, npoly, pp};
    ntt_inv(ctx, us, us);
    u64 *w = (u64 *)ctx->buf("ks_conv", (size_t)npoly * l * N * 8);
    {
        KTimer kt(ctx, "moddown_conv", (double)npoly * (ctx->np + 1 + l) * N * 8);
        dim3 g2((N + 255) / 256, npoly);
#define FG_LAUNCH(M)                                                                        \
        k_moddown_rescale_conv<M><<<g2, 256, 0, ctx->stream>>>(ext, E, w, l, ctx->moddown_tab(level), \
                                                               ctx->pinv_tab(level),                 \
                                                               ctx->moddown_rescale_half_tab(level), \
                                                               ctx->d_primes, N)
        FG_NIN_DISPATCH(ctx->np, FG_LAUNCH)
#undef FG_LAUNCH
        check_launch(ctx, "moddown_rescale_conv");
    }
    std::vector<int> pq(l);
    for (int i = 0; i < l; i++) pq[i] = i;
    // the rescaled limbs (ext_i - NTT(w)_i) (P q_l)^-1 straight from the
    // transform's last pass
    LimbSet ws{w, l, l, npoly, pq};
    const Finish fin{ext, out, ctx->moddown_rescale_tab(level), E, ls, accumulate ? 1 : 0};
    launch_ntt(ctx, ws, ws, false, &fin);
}

}  // namespace kern
