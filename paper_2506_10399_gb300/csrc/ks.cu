// ks.cu -- key switching inner product with the automorphism folded into the
// gather (k_ks_ip):
//   u_p[f][i][x] = sum_d D_d[f][i][sigma_g(x)] evk_g[d][p][i][x]  (+ P phi_g(c0) for p = 0)
// D_d limb i is the lane's own c1 limb when i belongs to digit d, else the
// ModUp output.  The keys (Montgomery form, [beta_L][2][nq+np][N]) of a thread's
// slot are held in registers, split into halves, for every column.
//
// Several rotations of one lane share a launch: blockIdx.y picks the rotation
// and blockIdx.z the limb, so the blocks of one limb run together and the
// lane's digits of that limb (ncol x beta limbs) are read from HBM once and
// gathered again from L2 by the other rotations.  In the bit-reversed NTT order
// the automorphism maps every aligned block of 2^k slots onto an aligned block,
// so a warp's gather of 32 words still reads 256 consecutive bytes.
//
// What bounds it: the FMA-heavy pipe (a 32 x 32 -> 64-bit product holds it for
// four cycles a warp).  Primes below 2^46 take Karatsuba's form on 23-bit halves
// (three products), P phi(c0) is one more term of the same sums instead of a
// modular product of its own, and the reductions are fold_split's and redc30's.
// One slot a thread: half the registers of two, twice the warps.  Measured at
// N = 2^16, 16 columns, 6 rotations: five digits (21 limbs) 1.17 ms, four (17
// limbs) 0.85 ms, 3.3 TB/s of what must move, half of the issue slots used; the
// form with two slots a thread, 30-bit halves for every prime and P phi(c0) as a
// modular product took 8 to 12% longer.  Loading the next columns' words
// early, advancing pointers instead of indexing and other register budgets were
// slower or equal: the loads are not what it waits for.
#include <cstring>

#include "fg_internal.h"
#include "modarith.cuh"

namespace {

constexpr int kMaxBeta = 16;   // digits
constexpr int kKsMulti = 24;   // rotations per launch

struct KsSet {
    int n;
    const u64 *key[kKsMulti];
    uint32_t g[kKsMulti];
    u64 *u[kKsMulti];
};

// blocks of 256 threads per SM the registers are budgeted for (the words a
// thread keeps grow with the digits); d: tune.ks_split's one fewer or one more
constexpr int ks_blocks(int beta, int d) { return (beta <= 3 ? 5 : beta <= 4 ? 4 : beta <= 8 ? 3 : 2) + d; }

// With pmodq given (P mod q_i at pmodq[2 i]), part 0 also receives P phi_g(c0)
// on the limbs of Q, so that ModDown of u is Rot(c) itself: ModDown(A + P B) =
// ModDown(A) + B exactly.
template <int BETA, int D>
__global__ void __launch_bounds__(256, ks_blocks(BETA, D))
k_ks_ip(const __grid_constant__ KsSet ks, int KL, const u64 *__restrict__ lane, int ls,
        const u64 *__restrict__ digits, int ncol, int level, int E, int alpha, int nq, int log_n,
        const PrimeC *__restrict__ primes, const u64 *__restrict__ pmodq)
{
    const int N = 1 << log_n;
    const int rot = blockIdx.y, i = blockIdx.z;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int pi = i <= level ? i : nq + (i - level - 1);
    const PrimeC P = primes[pi];
    const int sx = auto_src(x, ks.g[rot], log_n);
    const int own = i <= level ? i / alpha : -1;
    const bool small = P.q < (1ull << 46), c0 = pmodq && i <= level;
    const u64 *key = ks.key[rot] + (size_t)pi * N + x;
    u64 kb[BETA], ka[BETA];
#pragma unroll
    for (int d = 0; d < BETA; d++) {
        kb[d] = key[(size_t)(2 * d) * KL * N];
        ka[d] = key[(size_t)(2 * d + 1) * KL * N];
    }
    const u64 *dig = digits + (size_t)i * N + sx;
    const u64 *c0p = lane + (size_t)i * N + sx, *c1p = c0p + (size_t)ls * N;
    u64 *u = ks.u[rot] + (size_t)i * N + x;
    auto word = [&](int f, int d) {
        return d == own ? c1p[(size_t)f * 2 * ls * N] : dig[((size_t)f * BETA + d) * E * N];
    };
    if (small) {
        // P in Montgomery form, so that P c0 joins the sums; 0 without it
        const u64 pw = c0 ? split23(mont_mul(pmodq[2 * i], P.r2, P)) : 0;
#pragma unroll
        for (int d = 0; d < BETA; d++) {
            kb[d] = split23(kb[d]);
            ka[d] = split23(ka[d]);
        }
        for (int f = 0; f < ncol; f++) {
            u64 v[BETA];
#pragma unroll
            for (int d = 0; d < BETA; d++) v[d] = word(f, d);
            u64 a[6] = {0, 0, 0, 0, 0, 0};
            if (c0) mac_kara(a[0], a[1], a[2], split23(c0p[(size_t)f * 2 * ls * N]), pw);
#pragma unroll
            for (int d = 0; d < BETA; d++) {
                const u64 h = split23(v[d]);
                mac_kara(a[0], a[1], a[2], h, kb[d]);
                mac_kara(a[3], a[4], a[5], h, ka[d]);
            }
            u[(size_t)f * 2 * E * N] = fold_kara(a[0], a[1], a[2], P);
            u[((size_t)f * 2 + 1) * E * N] = fold_kara(a[3], a[4], a[5], P);
        }
    } else {
        // Words below 2^60 in 30-bit halves: three 64-bit partial sums hold up
        // to 8 products per sum, more digits take 128-bit sums.  The total,
        // below (BETA + 1) 2^60 q, keeps its high word below q for the
        // Montgomery step.
        constexpr bool SPLIT = BETA <= 8, SUM_C0 = BETA + 1 <= 8;
        const u64 pw = !c0 ? 0 : SUM_C0 ? split30(mont_mul(pmodq[2 * i], P.r2, P)) : pmodq[2 * i];
        const u64 pws = c0 ? pmodq[2 * i + 1] : 0;
        if (SPLIT) {
#pragma unroll
            for (int d = 0; d < BETA; d++) {
                kb[d] = split30(kb[d]);
                ka[d] = split30(ka[d]);
            }
        }
        for (int f = 0; f < ncol; f++) {
            u64 h0 = 0, l0 = 0, h1 = 0, l1 = 0;
            u64 a[6] = {0, 0, 0, 0, 0, 0};
            const u64 w = c0 ? c0p[(size_t)f * 2 * ls * N] : 0;
            if (SUM_C0 && c0) mac_split(a[0], a[1], a[2], split30(w), pw);
#pragma unroll
            for (int d = 0; d < BETA; d++) {
                const u64 v = word(f, d);
                if (SPLIT) {
                    const u64 h = split30(v);
                    mac_split(a[0], a[1], a[2], h, kb[d]);
                    mac_split(a[3], a[4], a[5], h, ka[d]);
                } else {
                    mac128(h0, l0, v, kb[d]);
                    mac128(h1, l1, v, ka[d]);
                }
            }
            u64 r = SPLIT ? reduce30<SUM_C0 ? BETA + 1 : 8>(a[0], a[1], a[2], P) : redc(h0, l0, P);
            if (!SUM_C0 && c0) r = add_mod(r, shoup_mul(w, pw, pws, P.q), P.q);
            u[(size_t)f * 2 * E * N] = r;
            u[((size_t)f * 2 + 1) * E * N] =
                SPLIT ? reduce30<SPLIT ? BETA : 8>(a[3], a[4], a[5], P) : redc(h1, l1, P);
        }
    }
}

}  // namespace

namespace kern {

// key-switch inner products of up to kKsMulti rotations of one lane (with
// P phi(c0) folded in when add_c0 is set)
void ks_launch(fg_ctx *ctx, const std::vector<const KeyDev *> &keys, const std::vector<u64 *> &us, const u64 *lane,
               int ls, int ncol, int level, const u64 *digits, bool add_c0)
{
    const int N = ctx->n, E = ctx->ext(level), beta = ctx->n_digits(level);
    FG_CHECK(beta <= kMaxBeta, FG_EINVAL, "too many key-switching digits");
    FG_CHECK(!keys.empty() && keys.size() <= (size_t)kKsMulti && keys.size() == us.size(), FG_EINVAL,
             "ks_launch: 1 to 24 rotations");
    const int KL = ctx->nq + ctx->np;
    KsSet ks;
    memset(&ks, 0, sizeof(ks));
    ks.n = (int)keys.size();
    for (int r = 0; r < ks.n; r++) {
        ks.key[r] = keys[r]->d;
        ks.g[r] = keys[r]->galois;
        ks.u[r] = us[r];
    }
    const u64 *pmodq = add_c0 ? ctx->d_pmodq : nullptr;
    const dim3 g(N / 256, ks.n, E);
    // digits and c0 once per launch, keys and outputs once per rotation
    KTimer kt(ctx, "ks_ip", ((double)ncol * beta * E + (add_c0 ? (double)ncol * (level + 1) : 0) +
                             (double)ks.n * (2.0 * beta * E + 2.0 * ncol * E)) * N * 8);
    const int v = ctx->tune.ks_split;
#define FG_KS_CASE(B)                                                                                                 \
    case B: {                                                                                                         \
        auto kern = v == 1 ? k_ks_ip<B, -1> : v == 2 ? k_ks_ip<B, 1> : k_ks_ip<B, 0>;                                 \
        kern<<<g, 256, 0, ctx->stream>>>(ks, KL, lane, ls, digits, ncol, level, E, ctx->alpha, ctx->nq, ctx->log_n,   \
                                         ctx->d_primes, pmodq);                                                       \
        break;                                                                                                        \
    }
    switch (beta) {
        FG_KS_CASE(1) FG_KS_CASE(2) FG_KS_CASE(3) FG_KS_CASE(4) FG_KS_CASE(5) FG_KS_CASE(6)
        FG_KS_CASE(7) FG_KS_CASE(8) FG_KS_CASE(9) FG_KS_CASE(10) FG_KS_CASE(11) FG_KS_CASE(12)
        FG_KS_CASE(13) FG_KS_CASE(14) FG_KS_CASE(15) FG_KS_CASE(16)
    default: throw fg_error(FG_EINVAL, "too many key-switching digits");
    }
#undef FG_KS_CASE
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw fg_error(FG_ECUDA, std::string("ks_ip: ") + cudaGetErrorString(e));
    ctx->launches += 1;
}

// With ctx->tune.ks_cols = 2 the columns are split over two launches, so
// that the digits a limb's blocks gather from L2 are half as many (the keys
// are then read once per half).
void ks_multi(fg_ctx *ctx, const std::vector<const KeyDev *> &keys, const std::vector<u64 *> &us, const u64 *lane,
              int ls, int ncol, int level, const u64 *digits)
{
    const int E = ctx->ext(level), beta = ctx->n_digits(level), N = ctx->n;
    const int parts = std::max(1, std::min(ctx->tune.ks_cols, ncol));
    for (int h = 0; h < parts; h++) {
        const int f0 = ncol * h / parts, f1 = ncol * (h + 1) / parts;
        if (f1 == f0) continue;
        for (size_t r0 = 0; r0 < keys.size(); r0 += kKsMulti) {
            const size_t r1 = std::min(keys.size(), r0 + kKsMulti);
            std::vector<u64 *> uh;
            for (size_t r = r0; r < r1; r++) uh.push_back(us[r] + (size_t)f0 * 2 * E * N);
            ks_launch(ctx, std::vector<const KeyDev *>(keys.begin() + r0, keys.begin() + r1), uh,
                      lane + (size_t)f0 * 2 * ls * N, ls, f1 - f0, level, digits + (size_t)f0 * beta * E * N, true);
        }
    }
}

}  // namespace kern
