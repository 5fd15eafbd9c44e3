// ntt.cuh -- a batch of limbs for the transforms and element-wise kernels, and
// the register rounds the transforms are built from.
#pragma once
#include "fg_internal.h"
#include "modarith.cuh"

constexpr int kPidxMax = 1024;

struct Batch {
    u64 *src;          // read from
    u64 *dst;          // written to (may equal src)
    int src_stride;    // limbs between rows
    int dst_stride;
    int per_row;
    int rows;
    int8_t pidx[kPidxMax];
};

// A radix-R round of R elements in registers, log2 R stages; tw(st, g):
// twiddle of group g at the round's stage st.  Products take the three-product
// quotient shoup_lazy4 and lie in [0, 4q).  LAZY (primes below 2^47): no
// conditional reduction, forward values grow by at most 4q per stage (< 65q
// after 16 stages), inverse values are below 2^(k+1) q after k stages (< 2^64
// for q < 2^47).  Larger primes (below 2^61) subtract 4q once per butterfly:
// forward values stay below 8q, inverse ones below 4q.
template <int R, bool LAZY, class TW>
__device__ __forceinline__ void ct_round(u64 *v, TW tw, u64 q, u64 q4)
{
    constexpr int LR = R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1;
#pragma unroll
    for (int st = 0; st < LR; st++) {
        const int h = R >> (st + 1);
#pragma unroll
        for (int m = 0; m < R; m++) {
            if ((m & h) == 0) {
                const ulonglong2 w = tw(st, m >> (LR - st));
                u64 X = v[m], Y = v[m + h];
                if (LAZY) {
                    const u64 T = shoup_lazy4(Y, w.x, w.y, q);
                    v[m + h] = X - T + q4;
                    v[m] = X + T;
                } else {
                    X = X >= q4 ? X - q4 : X;
                    const u64 T = shoup_lazy4(Y, w.x, w.y, q);
                    v[m + h] = X - T + q4;
                    v[m] = X + T;
                }
            }
        }
    }
}

// k0: number of inverse stages already applied to these values (lazy bound 2^k0 q)
template <int R, bool LAZY, class TW>
__device__ __forceinline__ void gs_round(u64 *v, TW tw, u64 q, u64 q4, int k0)
{
    constexpr int LR = R == 16 ? 4 : R == 8 ? 3 : R == 4 ? 2 : 1;
#pragma unroll
    for (int st = LR - 1; st >= 0; st--) {
        const int h = R >> (st + 1);
        const u64 qb = LAZY ? (q << (k0 + LR - st)) : q4;   // above the bound of V
#pragma unroll
        for (int m = 0; m < R; m++) {
            if ((m & h) == 0) {
                const ulonglong2 w = tw(st, m >> (LR - st));
                const u64 U = v[m], V = v[m + h];
                const u64 S = U + V;
                v[m] = LAZY ? S : (S >= q4 ? S - q4 : S);
                v[m + h] = shoup_lazy4(U - V + qb, w.x, w.y, q);
            }
        }
    }
}

// What a forward transform may do with its results w instead of storing them:
// out_i (+)= (ext_i - w_i) c_i mod q_i for limb i of every row, c with its Shoup
// companion at c[2 i].  ext and out have E and ls limbs a row.
struct Finish {
    const u64 *ext;
    u64 *out;
    const u64 *c;
    int E, ls, accumulate;
};

// Two neighbouring results of one limb (row, col), at word offset pos: reduced
// and stored at d + pos, or finished.  w is lazy: below 65 q (LAZY) or 8 q.
template <bool LAZY, bool FIN>
__device__ __forceinline__ void put_pair(u64 w0, u64 w1, u64 *d, size_t pos, const Finish &f, int row, int col, int N,
                                         const PrimeC &P)
{
    ulonglong2 *o;
    ulonglong2 r;
    if (FIN) {
        const u64 q = P.q, c = f.c[2 * col], cs = f.c[2 * col + 1], up = (LAZY ? 65 : 8) * q;
        const ulonglong2 e = *reinterpret_cast<const ulonglong2 *>(f.ext + ((size_t)row * f.E + col) * N + pos);
        r = make_ulonglong2(shoup_mul(e.x + up - w0, c, cs, q), shoup_mul(e.y + up - w1, c, cs, q));
        o = reinterpret_cast<ulonglong2 *>(f.out + ((size_t)row * f.ls + col) * N + pos);
        if (f.accumulate) {
            const ulonglong2 b = *o;
            r = make_ulonglong2(add_mod(r.x, b.x, q), add_mod(r.y, b.y, q));
        }
    } else {
        r = LAZY ? make_ulonglong2(reduce_word(w0, P), reduce_word(w1, P))
                 : make_ulonglong2(reduce8(w0, P.q), reduce8(w1, P.q));
        o = reinterpret_cast<ulonglong2 *>(d + pos);
    }
    *o = r;
}

// N = 2^10 .. 2^15 (ntt.cu); count limbs, of which `working` are transformed
// and the others left alone (pidx < 0); fin: forward only
void ntt_small(fg_ctx *ctx, const Batch &bt, int count, int working, bool inverse, const Finish *fin = nullptr);
