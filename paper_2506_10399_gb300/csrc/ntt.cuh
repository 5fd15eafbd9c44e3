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

// N = 2^10 .. 2^15 (ntt.cu)
void ntt_small(fg_ctx *ctx, const Batch &bt, int count, bool inverse);
