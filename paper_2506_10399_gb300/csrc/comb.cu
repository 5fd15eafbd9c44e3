// comb.cu -- the combination Z = X W on the tensor cores.
//
// Z[j][p][i] = sum_f c[f][j] X[f][p][i] mod q_i over coefficients x: for every
// (part p, limb i) a product of the integers X [F] x [N] by the integer
// constants c = round(W q_l) [F'] x [F], the only contraction of the layer
// whose second factor does not change with x.  k_comb spends four 32 x 32-bit
// products of the integer pipe on each term; here both factors are cut into
// signed 8-bit digits, and tcgen05.mma multiplies them exactly:
//   X = sum_a (d_a + 128) 256^a, d_a in [-128, 127], Da = 5..8 digits by limb,
//   c = sum_b c_b 256^b, c_b in [-128, 127], Dc digits (the largest |c| of the
//   plan decides; the same integers serve every limb),
//   D_e[x][j] = sum_{a + b = e} sum_f d_a[x][f] c_b[f][j].
// Digits are f16, products below 2^14, and D_e is read after at most kSeg =
// 128 columns, so |D_e| <= min(Da, Dc) 128 2^14 <= 2^24: every partial sum is
// an integer that f32 accumulation holds exactly.  Then
//   Z = sum_e D_e 256^e + 128 (256^Da - 1) / 255 sum_f c  mod q,
// the last term a constant per limb and output (CombPlan::corr).
//
// One block an SM, persistent over tiles of 128 coefficients of one (part,
// limb) and 16 outputs.  One warp brings in the words of X by TMA, a box of 16
// columns x 128 coefficients (16 KB) a stage; two groups of four warps cut
// alternate stages and write the digits to shared memory as core matrices of
// 8 x 16 bytes (K-major, no swizzle: consecutive lanes write consecutive
// 16-byte rows, no bank conflict); one warp issues the products (digit a: M =
// 128, N = 16 Dc, into the 16 (a + b) columns of its D_e); eight warps read
// the accumulators, zero them for the next segment and collect 64-bit sums.
// The constants' digits are laid out once per plan as the shared-memory image
// of each block of columns and arrive by a bulk copy.  Two accumulator sets
// of 256 TMEM columns let a segment's products run while the previous one is
// read.
//
// Measured on 500 columns, 16 outputs, 6 limbs, N = 2^16: 0.90 ms, 3.5 TB/s of
// X (k_comb: 4.2 ms).  Neither HBM nor the tensor cores (19% busy) are full: a
// stage of 16 KB takes 1450 cycles, its copies alone 820 (6.2 TB/s), copies and
// cutting 1110, copies and products 1310.  Copies of 1 KB rows instead of
// boxes, words through registers or cp.async instead of TMA, other splits of
// the ring: all slower by 3 to 30%.
#include <algorithm>
#include <cstring>

#include <cuda.h>

#include "fg_internal.h"
#include "modarith.cuh"

namespace {

constexpr int kSeg = 128;          // columns f per accumulator
constexpr int kKB = 16;            // columns per stage: one step of the products
constexpr int kRaw = 6;            // stages of words
constexpr int kStages = 3;         // stages of digits
constexpr int kTileX = 128;
constexpr int kEpi = 256, kProd = 256, kThreads = kEpi + kProd + 64;
constexpr int kGroup = kProd / 2;  // two groups of warps cut alternate stages
// A group's consecutive slots are at most three apart (its own second half,
// then up to two of the other group): with three slots or more its wait for an
// empty slot is never more than one phase ahead of the barrier.
static_assert(kStages >= 3, "slots");
constexpr u32 kWaitTries = fg_ctx::kWaitTries;
constexpr int kMaxCols = 8192;     // columns per launch: the 64-bit sums hold 64 segments
constexpr int kDigBytes = kTileX * kKB * 2;                        // one digit of X in a stage
constexpr int kStageBytes = 8 * kDigBytes + 8 * 16 * kKB * 2;      // 8 digits of X, 8 of c
constexpr int kRawBytes = kKB * kTileX * 8;
constexpr int kSmem = kRaw * kRawBytes + kStages * kStageBytes;
// a group's consecutive stages are two apart, so with two stages or more its
// waits are never more than one phase ahead of a barrier
static_assert(kStages >= 2 && kRaw >= 2, "stages");

struct Limb {
    u64 c40, c40s, c80, c80s;   // 2^40, 2^80 mod q and their Shoup companions
    u64 bias;                   // the least multiple of q that is at least 2^62 + 2^58
    u64 da;                     // digits of X
};

__device__ __forceinline__ u32 smem_u32(const void *p) { return (u32)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(u32 bar, u32 count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(u32 bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(u32 bar, u32 bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_poll(u32 bar, u32 parity)
{
    u32 ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Waits for the phase of the given parity.  Every wait is bounded: after
// `tries` polls, or once another role of the block has given up, it sets
// the block's stop flag and returns false, and the role leaves its loop.
__device__ __forceinline__ bool mbar_wait(u32 bar, u32 parity, volatile int *stop, u32 tries)
{
    for (u32 n = 0; n < tries; n++) {
        if (mbar_poll(bar, parity)) return true;
        if (*stop) return false;
    }
    *stop = 1;
    return false;
}
// The same once a role has given up, for what is still under way: always with
// the default limit, and nothing to report.
__device__ __forceinline__ void mbar_drain(u32 bar, u32 parity)
{
    for (u32 n = 0; n < kWaitTries; n++)
        if (mbar_poll(bar, parity)) return;
}

// shared-memory matrix descriptor: K-major, no swizzle; lbo: bytes between
// core matrices along K, sbo: between groups of eight rows
__device__ __forceinline__ u64 mma_desc(u32 addr, u32 lbo, u32 sbo)
{
    return (u64)((addr & 0x3FFFF) >> 4) | (u64)(lbo >> 4) << 16 | (u64)(sbo >> 4) << 32 | 1ull << 46;
}

__device__ __forceinline__ void mma_f16(u32 d, u64 a, u64 b, u32 idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, 1, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(idesc)
                 : "memory");
}

// the barrier is arrived at once the products issued so far are done
__device__ __forceinline__ void mma_commit(u32 bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld8(u32 addr, u32 (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
}

__device__ __forceinline__ void tmem_zero8(u32 addr)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(addr), "r"(0)
                 : "memory");
}

// eight words' digit a as f16 integers in [-128, 127]: byte a of each word
// under the f16 pattern of 1024 (0x64 in the high byte) is 1024 + byte
__device__ __forceinline__ uint4 digit8(const u32 (&lo)[8], const u32 (&hi)[8], int a)
{
    u32 o[4];
    const u32 sel = (a & 3) | (a & 3) << 4 | (4 + (a & 3)) << 8 | (4 + (a & 3)) << 12;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const u32 p = a < 4 ? lo[2 * k] : hi[2 * k], q = a < 4 ? lo[2 * k + 1] : hi[2 * k + 1];
        const u32 t = (__byte_perm(p, q, sel) & 0x00FF00FF) | 0x64006400;
        asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o[k]) : "r"(t), "r"(0xE480E480));   // - 1152
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// DA digits of a thread's sixteen words into a stage
template <int DA>
__device__ __forceinline__ void cut(unsigned char *dst, const u32 (&lo)[2][8], const u32 (&hi)[2][8])
{
#pragma unroll
    for (int c = 0; c < 2; c++)
#pragma unroll
        for (int a = 0; a < DA; a++)
            *reinterpret_cast<uint4 *>(dst + c * (kTileX * 16) + a * kDigBytes) = digit8(lo[c], hi[c], a);
}

__device__ __forceinline__ void bulk_copy(u32 dst, const void *src, u32 bytes, u32 bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// a box of kKB columns x kTileX coefficients at (x, row, f)
__device__ __forceinline__ void tma_load(u32 dst, const CUtensorMap *map, int x, int row, int f, u32 bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                 "%4}], [%5];" ::"r"(dst), "l"(map), "r"(x), "r"(row), "r"(f), "r"(bar) : "memory");
}

struct CombArgs {
    u64 *Z;
    const unsigned char *dig;   // [output block][16-column block][2][16 Dc][16 bytes]
    const Limb *limb;           // [nl]
    const u64 *corr;            // [nl][64-column blocks + 1][16 nj]
    const PrimeC *primes;
    int *err;
    int Fp, nl, N, z_ls, nj, dc, tiles;
    int f0, f1, kb_all, corr0, corr1, corr_blocks, accumulate;
    u32 tries;                  // polls after which a wait gives up
    uint8_t da[64];             // digits of X by limb
    CUtensorMap map;            // X as [columns][part x limb][coefficients]
};

// the block's tiles in turn: output block fastest, then coefficients, limb, part
struct Tile {
    int t, jb, xb, i, p, da;
    __device__ __forceinline__ void set(const CombArgs &A, int t_)
    {
        t = t_;
        jb = t % A.nj;
        const int u = t / A.nj, nx = A.N / kTileX, v = u / nx;
        xb = u - v * nx;
        p = v >= A.nl;
        i = p ? v - A.nl : v;
        da = t < A.tiles ? A.da[i] : 1;
    }
};

__global__ void __launch_bounds__(kThreads, 1) k_comb_mma(const __grid_constant__ CombArgs A)
{
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) u64 bars[2 * kStages + 4 + 2 * kRaw];
    __shared__ u32 tmem_base_s;
    __shared__ volatile int stop;
    __shared__ u32 cut_end[2];   // stages up to which each group of cutting warps has issued digit copies
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 full = smem_u32(bars), empty = full + 8 * kStages, acc_full = empty + 8 * kStages,
              acc_empty = acc_full + 16, raw_full = acc_empty + 16, raw_empty = raw_full + 8 * kRaw;
    if (tid == 0) {
        stop = 0;
        for (int s = 0; s < kStages; s++) {
            mbar_init(full + 8 * s, kGroup / 32 + 1);
            mbar_init(empty + 8 * s, 1);
        }
        for (int s = 0; s < kRaw; s++) {
            mbar_init(raw_full + 8 * s, 1);
            mbar_init(raw_empty + 8 * s, kGroup / 32);
        }
        for (int s = 0; s < 2; s++) {
            mbar_init(acc_full + 8 * s, 1);
            mbar_init(acc_empty + 8 * s, kEpi);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                     "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const u32 tmem = tmem_base_s;
    unsigned char *dig0 = sm + kRaw * kRawBytes;   // words, then digits
    const u32 raw0 = smem_u32(sm), smem0 = smem_u32(dig0);
    const int nkb = (A.f1 - A.f0 + kKB - 1) / kKB;   // stages per tile
    constexpr int kbs = kSeg / kKB;                  // stages per segment
    const u32 bbytes = (u32)A.dc * 16 * kKB * 2;
    u32 it = 0, seg = 0;   // stages and segments of the block so far

    if (warp < 8) {
        // ---- accumulators -> 64-bit sums -> Z
        const int quad = warp & 3, half = warp >> 2;
        const u32 tq = tmem + ((u32)(quad * 32) << 16) + half * 8;
        for (int c = 0; c < 512; c += 16) tmem_zero8(tq + c);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(acc_empty);
        mbar_arrive(acc_empty + 8);
        bool ok = true;
        Tile T;
        for (T.set(A, blockIdx.x); T.t < A.tiles && ok; T.set(A, T.t + gridDim.x)) {
            const int ne = T.da + A.dc - 1;   // columns D_0 .. D_{ne - 1}, at most 15
            i64 g[3][8];
#pragma unroll
            for (int r = 0; r < 3; r++)
#pragma unroll
                for (int j = 0; j < 8; j++) g[r][j] = 0;
            for (int kb = 0; kb < nkb && ok; kb += kbs, seg++) {
                const u32 b = seg & 1, ta = tq + b * 256;
                ok = mbar_wait(acc_full + 8 * b, seg >> 1 & 1, &stop, A.tries);
                ok = __all_sync(0xFFFFFFFFu, ok);   // the tcgen05 loads are warp-wide
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int e0 = 0; e0 < 15; e0 += 3) {   // three columns at a time; D_e into g[e / 5], weight 2^(40 e / 5)
                    if (e0 < ne) {
                        u32 d[3][8];
#pragma unroll
                        for (int k = 0; k < 3; k++)
                            if (e0 + k < ne) tmem_ld8(ta + (e0 + k) * 16, d[k]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int k = 0; k < 3; k++)
                            if (e0 + k < ne) {
                                const int e = e0 + k;
#pragma unroll
                                for (int j = 0; j < 8; j++) {
                                    // the load's results must not be used before the wait above
                                    asm volatile("" : "+r"(d[k][j]));
                                    const int v = __float2int_rn(__uint_as_float(d[k][j]));
                                    g[e / 5][j] += e % 5 < 4 ? (i64)v * (1 << (8 * (e % 5))) : (i64)((u64)(u32)v << 32);
                                }
                                tmem_zero8(ta + e * 16);
                            }
                    }
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive(acc_empty + 8 * b);
            }
            if (!ok) break;
            // Z = g0 + g1 2^40 + g2 2^80 + corr; |g| < 2^62 + 2^57, so g + bias
            // is a positive word; four terms below 2q, then one reduction
            const int i = T.i, jb = T.jb;
            const Limb L = A.limb[i];
            const PrimeC P = A.primes[i];
            const size_t co = ((size_t)i * (A.corr_blocks + 1)) * (16 * A.nj) + 16 * jb + 8 * half;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const int jj = 16 * jb + 8 * half + j;
                if (jj < A.Fp) {
                    const u64 c0 = A.corr[co + (size_t)A.corr0 * (16 * A.nj) + j];
                    const u64 c1 = A.corr[co + (size_t)A.corr1 * (16 * A.nj) + j];
                    u64 s = sub_mod(c1, c0, P.q) + shoup_lazy((u64)g[0][j] + L.bias, 1, P.one_s, P.q) +
                            shoup_lazy((u64)g[1][j] + L.bias, L.c40, L.c40s, P.q) +
                            shoup_lazy((u64)g[2][j] + L.bias, L.c80, L.c80s, P.q);
                    u64 *z = A.Z + (((size_t)jj * 2 + T.p) * A.z_ls + i) * A.N + (size_t)T.xb * kTileX + quad * 32 + lane;
                    if (A.accumulate) s += *z;
                    *z = reduce_word(s, P);
                }
            }
        }
    } else if (warp < 16) {
        // ---- words of X -> digits
        const int x = (tid - kEpi) % kGroup;               // kGroup == kTileX
        const u32 grp = (u32)(tid - kEpi) / kGroup;
        u32 mine = 0;      // the group cuts the stages with it % 2 == grp; one past the last of them
        bool ok = true;
        Tile T;
        for (T.set(A, blockIdx.x); T.t < A.tiles && ok; T.set(A, T.t + gridDim.x)) {
            const unsigned char *dig = A.dig + ((size_t)T.jb * A.kb_all + A.f0 / kKB) * bbytes;
            for (int kb = 0; kb < nkb; kb++, it++) {
                if ((it & 1) != grp) continue;
                const u32 s = it % kStages, rs = it % kRaw;
                ok = mbar_wait(raw_full + 8 * rs, it / kRaw & 1, &stop, A.tries);
                if (ok && it >= kStages) ok = mbar_wait(empty + 8 * s, (it / kStages - 1) & 1, &stop, A.tries);
                ok = __all_sync(0xFFFFFFFFu, ok);   // lanes may differ; they meet again below
                if (!ok) break;
                if (x == 0) {
                    mbar_arrive_tx(full + 8 * s, bbytes);
                    bulk_copy(smem0 + s * kStageBytes + 8 * kDigBytes, dig + (size_t)kb * bbytes, bbytes, full + 8 * s);
                }
                mine = it + 1;
                const unsigned char *src = sm + rs * kRawBytes + x * 8;
                unsigned char *dst = dig0 + s * kStageBytes + x * 16;
                u32 lo[2][8], hi[2][8];
#pragma unroll
                for (int u = 0; u < 16; u++) {
                    const u64 w = *reinterpret_cast<const u64 *>(src + u * (kTileX * 8));
                    lo[u / 8][u % 8] = (u32)w;
                    hi[u / 8][u % 8] = (u32)(w >> 32);
                }
                if (T.da == 6) cut<6>(dst, lo, hi);
                else if (T.da <= 5) cut<5>(dst, lo, hi);
                else cut<8>(dst, lo, hi);   // digits above da are not multiplied
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(raw_empty + 8 * rs);
                    mbar_arrive(full + 8 * s);
                }
            }
        }
        if (x == 0) cut_end[grp] = mine;
    } else if (warp == 17) {
        // ---- words of X: columns past the last arrive as zeros
        if (lane == 0) {
            bool ok = true;
            Tile T;
            for (T.set(A, blockIdx.x); T.t < A.tiles && ok; T.set(A, T.t + gridDim.x)) {
                for (int kb = 0; kb < nkb; kb++, it++) {
                    const u32 rs = it % kRaw;
                    if (it >= kRaw) ok = mbar_wait(raw_empty + 8 * rs, (it / kRaw - 1) & 1, &stop, A.tries);
                    if (!ok) break;
                    mbar_arrive_tx(raw_full + 8 * rs, kRawBytes);
                    tma_load(raw0 + rs * kRawBytes, &A.map, T.xb * kTileX, T.p * A.nl + T.i, A.f0 + kb * kKB,
                             raw_full + 8 * rs);
                }
            }
        }
        __syncwarp();
    } else {
        // ---- the products
        const u32 idesc = 1u << 4 | (u32)(2 * A.dc) << 17 | (u32)(kTileX >> 4) << 24;   // f32 += f16 f16, N = 16 Dc
        bool ok = true;
        Tile T;
        for (T.set(A, blockIdx.x); T.t < A.tiles && ok; T.set(A, T.t + gridDim.x)) {
            for (int kb = 0; kb < nkb && ok; kb++, it++) {
                const u32 b = seg & 1, s = it % kStages;
                if (kb % kbs == 0) ok = mbar_wait(acc_empty + 8 * b, seg >> 1 & 1, &stop, A.tries);
                ok = ok && mbar_wait(full + 8 * s, it / kStages & 1, &stop, A.tries);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const bool last = kb % kbs == kbs - 1 || kb == nkb - 1;
                if (lane == 0) {
                    const u32 st = smem0 + s * kStageBytes;
                    const u64 bd = mma_desc(st + 8 * kDigBytes, (u32)A.dc * 256, 128);
                    for (int a = 0; a < T.da; a++)
                        mma_f16(tmem + b * 256 + a * 16, mma_desc(st + a * kDigBytes, kTileX * 16, 128), bd, idesc);
                    mma_commit(empty + 8 * s);
                    if (last) mma_commit(acc_full + 8 * b);
                }
                __syncwarp();
                if (last) seg++;
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // When no wait has run out, the last sums have been read, so every product
    // is done and every copy has been used.  When one has, a role that had
    // already finished, or left later, may have copies into this block's shared
    // memory or products under way: nothing is issued any more, and whoever
    // issued them waits for them (bounded) before the block can end.
    if (stop) {
        if (tid == 17 * 32)   // words: the last use of every slot
            for (u32 k = it > kRaw ? it - kRaw : 0; k < it; k++) mbar_drain(raw_full + 8 * (k % kRaw), k / kRaw & 1);
        if (tid == kEpi || tid == kEpi + kGroup) {   // digits: the group's last two slots, unless used again since
            const u32 grp = tid != kEpi, end = cut_end[grp];
            for (u32 k = end >= 3 ? end - 3 : end ? end - 1 : 0; k < end; k += 2)
                if (cut_end[grp ^ 1] < k + kStages + 1) mbar_drain(full + 8 * (k % kStages), k / kStages & 1);
        }
        if (tid == 16 * 32 && it > 0) {
            mbar_drain(empty + 8 * ((it - 1) % kStages), (it - 1) / kStages & 1);
            if (seg > 0) mbar_drain(acc_full + 8 * ((seg - 1) & 1), (seg - 1) >> 1 & 1);
        }
        if (tid == 0) *A.err = 1;
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 16)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// The words of X [F][rows][N] for TMA.  Boxes start at multiples of kTileX
// words, so every copy starts on a 16-byte boundary when X does.
CUtensorMap word_map(const u64 *X, int F, int rows, int N)
{
    typedef CUresult (*Encode)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                               const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &r) != cudaSuccess ||
            r != cudaDriverEntryPointSuccess)
            fn = nullptr;
        return (Encode)fn;
    }();
    FG_CHECK(encode != nullptr, FG_ECUDA, "cuTensorMapEncodeTiled is not available");
    CUtensorMap m;
    const cuuint64_t dim[3] = {(cuuint64_t)N, (cuuint64_t)rows, (cuuint64_t)F};
    const cuuint64_t stride[2] = {(cuuint64_t)N * 8, (cuuint64_t)N * 8 * rows};
    const cuuint32_t box[3] = {kTileX, 1, kKB}, step[3] = {1, 1, 1};
    const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<u64 *>(X), dim, stride, box, step,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    FG_CHECK(r == CUDA_SUCCESS, FG_ECUDA, "tensor map of the combination's inputs");
    return m;
}

// the f16 of an integer in [-128, 127]
uint16_t half_of(int v)
{
    if (v == 0) return 0;
    const int s = v < 0, m = s ? -v : v;
    int e = 0;
    while ((m >> (e + 1)) != 0) e++;
    return (uint16_t)(s << 15 | (e + 15) << 10 | ((m << (10 - e)) & 0x3FF));
}

}  // namespace

void CombPlan::release()
{
    if (dig) cudaFree(dig);
    if (limb) cudaFree(limb);
    if (corr) cudaFree(corr);
}

// Digits of the constants, laid out as the shared-memory image of every
// 16-column block, and the per-limb tables.  Nothing is built (dc stays 0)
// when a constant needs more than eight digits.
void CombPlan::build(const fg_ctx &ctx, const std::vector<i64> &c, int F, int Fp, int level)
{
    int most = 1;
    for (i64 v : c) {
        int n = 0;
        for (i64 r = v; r != 0; n++) r = (r - (i64)(int8_t)r) >> 8;   // exact: the low byte is cleared first
        most = std::max(most, n);
    }
    // r - (int8_t)r can leave i64 only for |v| near 2^63, where nine digits are needed
    for (i64 v : c)
        if (v > 0x7F7F7F7F7F7F7F7Fll || v < -0x7F7F7F7F7F7F7F7Fll) most = 9;
    if (most > 8) return;
    const int nl = level + 1, J = (Fp + 15) / 16, kb = (F + kKB - 1) / kKB;
    std::vector<uint16_t> h((size_t)J * kb * most * 16 * kKB, 0);
    for (int f = 0; f < F; f++)
        for (int j = 0; j < Fp; j++) {
            i64 r = c[(size_t)f * Fp + j];
            const size_t blk = ((size_t)(j / 16) * kb + f / kKB) * (most * 16 * kKB);
            for (int b = 0; b < most; b++) {
                const int d = (int8_t)r;
                r = (r - d) >> 8;
                h[blk + ((size_t)(f % kKB / 8) * most * 16 + b * 16 + j % 16) * 8 + f % 8] = half_of(d);
            }
        }
    corr_blocks = (F + 63) / 64;
    std::vector<Limb> lim(nl);
    std::vector<u64> co((size_t)nl * (corr_blocks + 1) * 16 * J, 0);
    for (int i = 0; i < nl; i++) {
        const u64 q = ctx.primes[i];
        Limb &L = lim[i];
        L.c40 = (1ull << 40) % q;
        L.c40s = hm::shoup(L.c40, q);
        L.c80 = hm::mulmod(L.c40, L.c40, q);
        L.c80s = hm::shoup(L.c80, q);
        L.bias = ((1ull << 62) + (1ull << 58) + q - 1) / q * q;
        L.da = 1;
        while (L.da < 8 && (q - 1) >> (8 * L.da)) L.da++;
        u64 off = 0;   // 128 (256^Da - 1) / 255
        for (u64 a = 0; a < L.da; a++) off = (hm::mulmod(off, 256 % q, q) + 128) % q;
        for (int j = 0; j < Fp; j++) {
            u64 s = 0;
            for (int f = 0; f < F; f++) {
                const i64 v = c[(size_t)f * Fp + j];
                const u64 r = v >= 0 ? (u64)v % q : (q - (u64)(-v) % q) % q;
                s = (s + r) % q;
                if (f % 64 == 63 || f == F - 1)
                    co[((size_t)i * (corr_blocks + 1) + f / 64 + 1) * 16 * J + j] = hm::mulmod(s, off, q);
            }
        }
    }
    CUDA_TRY(cudaMalloc(&dig, h.size() * 2));
    CUDA_TRY(cudaMemcpy(dig, h.data(), h.size() * 2, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMalloc(&limb, lim.size() * sizeof(Limb)));
    CUDA_TRY(cudaMemcpy(limb, lim.data(), lim.size() * sizeof(Limb), cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMalloc(&corr, co.size() * 8));
    CUDA_TRY(cudaMemcpy(corr, co.data(), co.size() * 8, cudaMemcpyHostToDevice));
    for (const Limb &L : lim) da.push_back((int)L.da);
    nj = J;
    kb_all = kb;
    dc = most;
}

namespace kern {

void combine(fg_ctx *ctx, const fg_plan *pl, const u64 *X, u64 *Z, int z_ls, int fb, int fe, bool accumulate)
{
    const CombPlan &C = pl->comb;
    const int F = pl->F, Fp = pl->Fp, level = pl->in_level;
    if (fe < 0) fe = F;
    FG_CHECK(F < (1 << 16), FG_EINVAL, "combination over more than 2^16 input columns");
    FG_CHECK(0 <= fb && fb < fe && fe <= F, FG_EINVAL, "combination column range");
    // The tensor cores take over where a block's fixed work (TMEM, one
    // reading of the accumulators and eight reductions a thread) is paid for:
    // with 16 outputs, N = 2^14, 10 limbs (ms, integer pipe / tensor cores) 8
    // columns 0.059 / 0.094, 16 0.088 / 0.095, 24 0.116 / 0.100, 64 0.254 /
    // 0.112; k_comb's time goes with the blocks of 8 outputs, the other with
    // those of 16.  TMA takes 16-byte aligned words.
    const bool pays = (fe - fb) * ((Fp + 7) / 8) >= kCombMmaMin * C.nj;
    if (!C.dc || !pays || (uintptr_t)X % 16 || fb % 64 || (fe != F && fe % 64)) {
        comb_const_mac(ctx, X, F, Fp, level, pl->d_comb, Z, z_ls, fb, fe, accumulate);
        return;
    }
    KTimer kt(ctx, "comb", ((double)(fe - fb) + Fp * (accumulate ? 2 : 1)) * 2 * (level + 1) * ctx->n * 8);
    int sms = 0;
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
    CUDA_TRY(cudaFuncSetAttribute(k_comb_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    for (int f0 = fb; f0 < fe; f0 += kMaxCols) {
        CombArgs A;
        memset(&A, 0, sizeof(A));
        A.map = word_map(X, F, 2 * (level + 1), ctx->n);
        A.Z = Z;
        A.dig = (const unsigned char *)C.dig;
        A.limb = (const Limb *)C.limb;
        A.corr = C.corr;
        A.primes = ctx->d_primes;
        A.err = ctx->wait_error();
        A.Fp = Fp;
        A.nl = level + 1;
        A.N = ctx->n;
        A.z_ls = z_ls;
        A.nj = C.nj;
        A.dc = C.dc;
        A.f0 = f0;
        A.f1 = std::min(fe, f0 + kMaxCols);
        A.kb_all = C.kb_all;
        A.corr0 = f0 / 64;
        A.corr1 = (A.f1 + 63) / 64;
        A.corr_blocks = C.corr_blocks;
        A.accumulate = accumulate || f0 > fb;
        A.tries = ctx->wait_tries;
        A.tiles = A.nj * (A.N / kTileX) * A.nl * 2;
        for (int i = 0; i < A.nl; i++) A.da[i] = (uint8_t)C.da[i];
        k_comb_mma<<<std::min(A.tiles, sms), kThreads, kSmem, ctx->stream>>>(A);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) throw fg_error(FG_ECUDA, std::string("comb: ") + cudaGetErrorString(e));
        ctx->launches += 1;
    }
}

}  // namespace kern
