// gmac.cu -- the SpIntra-CA group's masked sums (k_group_mac).
//
// One group, all outputs at once (double hoisting): for each output d,
//   ext_d = sum over its rotated sources r of mask (x) (u_r + P phi_r(c0))
//         + sum over its kept sources of P mask (x) lane
// in the extended basis q_0..q_l, p_0..p_{K-1} (the P terms vanish mod p_k;
// the plan stores the masks of kept values times P).
// ModDown(ext_d) is then exactly the sum of mask (x) Rot and mask (x) lane,
// since ModDown(A + P B) = ModDown(A) + B.
//
// What bounds it.  A 32 x 32 -> 64-bit multiply-add holds the FMA-heavy pipe
// of an SM quarter for four cycles (30 a clock and SM, measured with operands
// that change; the low word alone takes two), so a product of two words of a
// prime below 2^46 costs 12 cycles a warp in Karatsuba's form (three
// products of 23-bit halves) and one of a 60-bit word 16.  k_group_mac, the
// form for up to six outputs, is laid out so that little else is issued per
// product:
//   * a warp holds 32 neighbouring slots of one column, both parts of the
//     ciphertext, and the running sums of every output in registers;
//   * the loop runs over the sources, so that a source word is read from
//     shared memory and split once for all outputs, and a mask word, stored
//     in split halves by the plan, is read once for both parts;
//   * which outputs a source feeds is the same for the whole grid, so it is
//     read and branched on in the uniform datapath;
//   * sources and masks arrive through a ring of kGmStages shared-memory
//     stages filled by cp.async two stages ahead, so that no word is staged
//     long before it is needed.
// Measured on 22 sources, 75 terms, 5 outputs, 16 columns, 9 limbs of 45 and
// 5 of 60 bits at N = 2^16: 2.05 ms (3.4 TB/s) against 2.26 ms for the tiled
// form below, which took 2.5 ms before its masks were stored split.  Half of
// the issue slots are used: 128 registers leave 16 warps an SM, and the
// fixed latencies of 60 instructions a source and 9 a term are not all
// hidden.
#include <algorithm>
#include <cstring>

#include "fg_internal.h"
#include "modarith.cuh"

namespace {

constexpr int kGmXs = 6;       // most outputs whose sums one warp holds
constexpr int kGmStages = 3;
constexpr int kGmChunk = 4;    // sources per stage
constexpr uint32_t kGmKept = 1u << 31;

// The launch's program, passed by value (kernel parameters sit in the
// constant bank).  Stage: kGmChunk consecutive sources and their masks, a row of 32 slots per (slot
// block, source, output) whether there is such a term or not, so that the
// shared-memory reads of the inner loop have constant offsets.
struct GProg {
    int nsrc, nstage, accumulate;
    int npairs, pw, lts;                    // columns; columns per block; log2 of the tile's slots
    int stage_words;                        // a stage in shared memory
    u64 *outs[kGmXs];
    const u64 *src[kern::kGmacSrc];         // rotation: key-switch output (limb stride E); kept lane (stride ls)
    uint32_t bits[kern::kGmacSrc + kGmChunk];   // the outputs a source feeds; kGmKept
    int tstage[kern::kGmacSrc + 1];         // a stage's first term
    uint8_t trow[kern::kGmacTerms];         // the term's mask row in its stage: source in stage x XS + output
    const u64 *tmask[kern::kGmacTerms];
};

__device__ __forceinline__ void cp_async16(u64 *smem, const u64 *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

// The warp's sums over one stage's sources for outputs bit 0..XS-1.  SMALL:
// primes below 2^46, a[d][p] = (A0, K, A2) of mac_kara, at most 2^16 terms.
// Otherwise 30-bit halves, a[d][p] = (A0, A1, A2) of mac_split with x3[d][p]
// the overflow of A2 past 2^60: norm() carries the sums up every eight terms
// (A0 and A1 back below 2^30, A2 below 2^60), so that A1, two products below
// 2^60 a term, stays below 16 (2^30 - 1)^2 + 2^30 + 2^34 < 2^64.
template <int XS>
__device__ __forceinline__ void norm30(u64 (&a)[XS][2][3], u32 (&x3)[XS][2])
{
#pragma unroll
    for (int d = 0; d < XS; d++)
#pragma unroll
        for (int p = 0; p < 2; p++) {
            a[d][p][1] += a[d][p][0] >> 30;
            a[d][p][0] &= 0x3FFFFFFF;
            a[d][p][2] += a[d][p][1] >> 30;
            a[d][p][1] &= 0x3FFFFFFF;
            x3[d][p] += (u32)(a[d][p][2] >> 60);
            a[d][p][2] &= (1ull << 60) - 1;
        }
}

template <int XS, bool SMALL>
__device__ __forceinline__ void gmac_tile(const GProg &pg, u64 *sm, int i, bool isq, const PrimeC &P, int E, int ls,
                                          int N)
{
    // block: (column group, slot tile, limb), the first fastest, so that the
    // blocks that share masks run together
    const int col0 = blockIdx.x * pg.pw, tile = blockIdx.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pw = pg.pw, lts = pg.lts;
    const int sub = warp / pw, pl = warp - sub * pw;
    // the last column group may have fewer columns: its spare warps repeat
    // the last column and store nothing
    const int pair = min(col0 + pl, pg.npairs - 1);
    const int x0 = (tile << lts) + (sub << 5), x = x0 + lane;   // this warp's 32 slots
    // word offset of the 16 bytes this lane copies of a source (part lane /
    // 16); a kept lane has no special limbs (its masks are zero there): limb
    // 0 stands in for them
    const int cpoly = 2 * pair + (lane >> 4), cx = x0 + 2 * (lane & 15);
    const size_t uoff = ((size_t)cpoly * E + i) * N + cx, loff = ((size_t)cpoly * ls + (isq ? i : 0)) * N + cx;
    // a stage: [source][warp][part][32], then [slot block][source][output][32]
    const int srcw = blockDim.x * 2;   // words of one source in a stage
    const int vofs = warp * 64, mofs = kGmChunk * srcw + sub * (kGmChunk * XS * 32) + lane;
    u64 *cdst = sm + vofs + 2 * lane;
    const size_t moff = (size_t)i * N + (tile << lts);

    auto issue = [&](int k) {
        if (k < pg.nstage) {
            const int st = k % kGmStages * pg.stage_words, s0 = k * kGmChunk;
#pragma unroll
            for (int c = 0; c < kGmChunk; c++)
                if (s0 + c < pg.nsrc)
                    cp_async16(cdst + st + c * srcw,
                               pg.src[s0 + c] + (pg.bits[s0 + c] & kGmKept ? loff : uoff));
            const int t0 = pg.tstage[k], n = (pg.tstage[k + 1] - t0) << (lts - 1);
            for (int c = threadIdx.x; c < n; c += blockDim.x) {
                const int t = t0 + (c >> (lts - 1)), o = 2 * (c & ((1 << (lts - 1)) - 1));
                cp_async16(sm + st + kGmChunk * srcw + (((o >> 5) * (kGmChunk * XS) + pg.trow[t]) << 5) + (o & 31),
                           pg.tmask[t] + moff + o);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    u64 a[XS][2][3];
    u32 x3[XS][2];
#pragma unroll
    for (int d = 0; d < XS; d++)
#pragma unroll
        for (int p = 0; p < 2; p++) {
            a[d][p][0] = a[d][p][1] = a[d][p][2] = 0;
            x3[d][p] = 0;
        }
#pragma unroll
    for (int k = 0; k < kGmStages - 1; k++) issue(k);
    for (int k = 0; k < pg.nstage; k++) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kGmStages - 2) : "memory");
        __syncthreads();   // stage k has arrived; stage k - 1 is free
        issue(k + kGmStages - 1);
        const u64 *vp = sm + k % kGmStages * pg.stage_words + vofs + lane;
        const u64 *mp = sm + k % kGmStages * pg.stage_words + mofs;
#pragma unroll
        for (int c = 0; c < kGmChunk; c++) {
            const u32 bits = pg.bits[k * kGmChunk + c];   // 0 past the last source
            u64 m[XS];
#pragma unroll
            for (int d = 0; d < XS; d++) m[d] = mp[(c * XS + d) * 32];   // rows without a term are not used
            u32 v0[2], v1[2], vs[2];
#pragma unroll
            for (int p = 0; p < 2; p++) {
                const u64 v = vp[c * srcw + p * 32];
                const u64 h = SMALL ? split23(v) : split30(v);
                v0[p] = (u32)h;
                v1[p] = (u32)(h >> 32);
                vs[p] = v0[p] + v1[p];
            }
#pragma unroll
            for (int d = 0; d < XS; d++)
                if (bits >> d & 1) {
                    const u32 m0 = (u32)m[d], m1 = (u32)(m[d] >> 32);
#pragma unroll
                    for (int p = 0; p < 2; p++) {
                        u64 *t = a[d][p];
                        t[0] = mad_wide(v0[p], m0, t[0]);
                        t[2] = mad_wide(v1[p], m1, t[2]);
                        if (SMALL) {
                            t[1] = mad_wide(vs[p], m0 + m1, t[1]);
                        } else {
                            t[1] = mad_wide(v0[p], m1, t[1]);
                            t[1] = mad_wide(v1[p], m0, t[1]);
                        }
                    }
                }
        }
        if (!SMALL && (k & 1)) norm30<XS>(a, x3);   // two stages: at most eight sources
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (col0 + pl >= pg.npairs) return;
    if (!SMALL) norm30<XS>(a, x3);
#pragma unroll
    for (int d = 0; d < XS; d++)
#pragma unroll
        for (int p = 0; p < 2; p++) {
            u64 r;
            if (SMALL) {
                r = fold_kara(a[d][p][0], a[d][p][1], a[d][p][2], P);
            } else {   // A0 + A1 2^30 + A2 2^60 + x3 2^120, A0, A1 < 2^30
                const u64 w = a[d][p][0] | a[d][p][1] << 30;   // < 2^60
                const u64 lo = w | a[d][p][2] << 60;
                const u64 hi = (a[d][p][2] >> 4) + ((u64)x3[d][p] << 56);
                r = redc(reduce_word(hi, P), lo, P);
            }
            u64 *o = pg.outs[d] + ((size_t)(2 * pair + p) * E + i) * N + x;
            *o = pg.accumulate ? add_mod(*o, r, P.q) : r;
        }
}

template <int XS>
__global__ void __launch_bounds__(256, XS <= 3 ? 3 : 2)
k_group_mac(const __grid_constant__ GProg pg, int level, int E, int ls, int log_n, const PrimeC *__restrict__ primes,
            int nq)
{
    extern __shared__ __align__(16) u64 gsm[];
    const int i = blockIdx.z;
    const bool isq = i <= level;
    const PrimeC P = primes[isq ? i : nq + (i - level - 1)];
    if (P.q < (1ull << 46)) gmac_tile<XS, true>(pg, gsm, i, isq, P, E, ls, 1 << log_n);
    else gmac_tile<XS, false>(pg, gsm, i, isq, P, E, ls, 1 << log_n);
}

typedef void (*GmacKernel)(const GProg, int, int, int, int, const PrimeC *, int);
const GmacKernel kGmacKernels[kGmXs] = {k_group_mac<1>, k_group_mac<2>, k_group_mac<3>,
                                        k_group_mac<4>, k_group_mac<5>, k_group_mac<6>};

// ------------------------------------------------------------------------
// More than kGmXs outputs: whole tiles.  A tile is PPC polynomials (column,
// part) times PPN neighbouring slot pairs of one limb, thread = one
// polynomial at one slot pair (PPC = min(npoly, 16), PPN = min(128 / PPC,
// 16): for 32 polynomials two tiles of 16 x 8, 128-byte runs per
// polynomial).  A block holds one tile and G thread groups that share its
// staged words: every group copies a share of the sources (split in place)
// and masks, then computes its own contiguous slice of the outputs (balanced
// by term count on the host), each a register sum over its terms.  With
// seven or more outputs G = 3: the block gets three times the warps for the
// same shared memory (measured on a 66-source, 12-output group: 9% faster
// than one group).
constexpr int kGmacTile = 128;    // threads per group: PPC x PPN (idle ones when npoly < 8)
constexpr int kGmacGroups = 3;    // most output groups per block
constexpr int kGmacThreads = kGmacTile * kGmacGroups;

struct TProg {
    int nsrc, nterm, accumulate;
    int ppc, ppn;                       // tile: polynomials x slot pairs
    int groups;                         // thread groups (blockDim = groups x kGmacTile)
    int gfirst[kGmacGroups + 1];        // first output of each thread group
    const u64 *src[kern::kGmacSrc];     // rotation: key-switch output (limb stride E); kept lane (stride ls)
    uint8_t kept[kern::kGmacSrc];
    u32 tvoff[kern::kGmacTerms];        // terms sorted by output: byte offset of the source's row in vsm
    const u64 *tmask[kern::kGmacTerms];
    int dfirst[kern::kGmacOut + 1];
    u64 *outs[kern::kGmacOut];
};

// 16-byte shared-memory load by 32-bit shared address (volatile: it must
// stay after the barrier that publishes the staged words)
__device__ __forceinline__ ulonglong2 lds128(u32 addr)
{
    ulonglong2 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(addr));
    return v;
}

// MINB: blocks of kGmacThreads threads per SM the registers are budgeted for
// (2: up to 85 registers a thread; 3: up to 56, more warps resident).
// KARA: the 23-bit split products in Karatsuba's form (mac_kara: three
// products instead of four; the same sums).
template <int MINB, bool KARA>
__global__ void __launch_bounds__(kGmacThreads, MINB)
k_group_mac_tile(const __grid_constant__ TProg pg, int ncol, int level, int E, int ls, int log_n,
            const PrimeC *__restrict__ primes, int nq)
{
    extern __shared__ __align__(16) u64 gsm[];
    const int npoly = 2 * ncol, PPC = pg.ppc, PPN = pg.ppn;
    const int npg = (npoly + PPC - 1) / PPC;
    const int nsrc = pg.nsrc, nterm = pg.nterm;
    ulonglong2 *vsm = reinterpret_cast<ulonglong2 *>(gsm);                  // [nsrc][kGmacTile]
    ulonglong2 *msm = vsm + (size_t)nsrc * kGmacTile;                       // [nterm][PPN]
    const int N = 1 << log_n;
    const int grp = threadIdx.x / kGmacTile, lt = threadIdx.x % kGmacTile;
    const int pl = lt / PPN, pp = lt - pl * PPN;
    const int pgi = blockIdx.x % npg, blk = blockIdx.x / npg;
    const int poly = pgi * PPC + pl;
    const int x = 2 * (blk * PPN + pp);
    const bool xin = pl < PPC && x < N;          // a slot pair of the tile
    const bool act = xin && poly < npoly;        // ... of an existing polynomial
    const int i = blockIdx.y;
    const bool isq = i <= level;
    const PrimeC P = primes[isq ? i : nq + (i - level - 1)];
    const u64 q = P.q;
    const bool split = q < (1ull << 46);
    const size_t ext_off = ((size_t)poly * E + i) * N + x;
    const int G = pg.groups;
    // 1. asynchronous copies: the masks of terms grp PPC + pl (step G PPC)
    // at this slot pair, the sources grp, grp + G, ... of this thread's slot
    // (a kept lane has no special limbs, and its masks are zero there: limb 0
    // stands in for them)
    if (xin)
        for (int t = grp * PPC + pl; t < nterm; t += G * PPC)
            cp_async16(reinterpret_cast<u64 *>(msm + t * PPN + pp), pg.tmask[t] + (size_t)i * N + x);
    if (act)
        for (int s = grp; s < nsrc; s += G)
            cp_async16(reinterpret_cast<u64 *>(vsm + (size_t)s * kGmacTile + lt),
                       pg.src[s] + (pg.kept[s] ? ((size_t)poly * ls + (isq ? i : 0)) * N + x : ext_off));
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    // 2. in place, each thread on the words it copied: source words split
    // into halves (the masks are stored split)
    if (act)
        for (int s = grp; s < nsrc; s += G) {
            ulonglong2 *dst = vsm + (size_t)s * kGmacTile + lt;
            const ulonglong2 v = *dst;
            *dst = split ? make_ulonglong2(split23(v.x), split23(v.y)) : make_ulonglong2(split30(v.x), split30(v.y));
        }
    __syncthreads();
    if (!act) return;
    // 3. this group's outputs.  Shared-memory reads by 32-bit address: the
    // source row of a term is a constant offset from this thread's slot, the
    // mask row steps by PPN words per term.
    const int d0 = pg.gfirst[grp], d1 = pg.gfirst[grp + 1];
    const u32 vbase = (u32)__cvta_generic_to_shared(vsm + lt);
    const u32 mstep = (u32)PPN * 16;
    u32 maddr = (u32)__cvta_generic_to_shared(msm + pp) + (u32)pg.dfirst[d0] * mstep;
    for (int d = d0; d < d1; d++) {
        ulonglong2 *o = reinterpret_cast<ulonglong2 *>(pg.outs[d] + ext_off);
        const ulonglong2 b = pg.accumulate ? *o : make_ulonglong2(0, 0);
        const int t0 = pg.dfirst[d], t1 = pg.dfirst[d + 1];
        ulonglong2 r;
        if (split) {
            u64 a0 = 0, a1 = 0, a2 = 0, c0 = 0, c1 = 0, c2 = 0;
            if (KARA) {
                for (int t = t0; t < t1; t++, maddr += mstep) {
                    const ulonglong2 v = lds128(vbase + pg.tvoff[t]);
                    const ulonglong2 m = lds128(maddr);
                    mac_kara(a0, a1, a2, v.x, m.x);
                    mac_kara(c0, c1, c2, v.y, m.y);
                }
                r = make_ulonglong2(fold_kara(a0, a1, a2, P), fold_kara(c0, c1, c2, P));
            } else {
                for (int t = t0; t < t1; t++, maddr += mstep) {
                    const ulonglong2 v = lds128(vbase + pg.tvoff[t]);
                    const ulonglong2 m = lds128(maddr);
                    mac_split(a0, a1, a2, v.x, m.x);
                    mac_split(c0, c1, c2, v.y, m.y);
                }
                r = make_ulonglong2(fold_split(a0, a1, a2, P), fold_split(c0, c1, c2, P));
            }
        } else {
            // 30-bit halves: partial sums folded into 128 bits every 8 terms
            u64 lo0 = 0, hi0 = 0, lo1 = 0, hi1 = 0;
            for (int t = t0; t < t1;) {
                const int te = min(t + 8, t1);
                u64 a0 = 0, a1 = 0, a2 = 0, c0 = 0, c1 = 0, c2 = 0;
                for (; t < te; t++, maddr += mstep) {
                    const ulonglong2 v = lds128(vbase + pg.tvoff[t]);
                    const ulonglong2 m = lds128(maddr);
                    mac_split(a0, a1, a2, v.x, m.x);
                    mac_split(c0, c1, c2, v.y, m.y);
                }
                fold30(hi0, lo0, a0, a1, a2);
                fold30(hi1, lo1, c0, c1, c2);
            }
            r = make_ulonglong2(redc(reduce_word(hi0, P), lo0, P), redc(reduce_word(hi1, P), lo1, P));
        }
        if (pg.accumulate) {
            r.x = add_mod(r.x, b.x, q);
            r.y = add_mod(r.y, b.y, q);
        }
        *o = r;
    }
}

}  // namespace

namespace kern {

// Lets a kernel take more than 48 KB of dynamic shared memory: always up to all
// a block can have, since the limit belongs to the kernel, and a limit of this
// launch's own size would undercut a launch that another thread is about to
// make.  (Not a stream operation: allowed while capturing.)
template <class K>
static void allow_shared(K kern, size_t bytes)
{
    if (bytes > 48 * 1024)
        CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
}

// more than kGmXs outputs: k_group_mac_tile
static void group_mac_tile(fg_ctx *ctx, const std::vector<GroupSource> &srcs, const std::vector<Dest> &terms_in,
                           const std::vector<int> &term_dest, const std::vector<u64 *> &outs, bool accumulate, int ncol,
                           int level, int ls)
{
    const int N = ctx->n, E = ctx->ext(level), X = (int)outs.size();
    TProg pg;
    memset(&pg, 0, sizeof(pg));
    pg.nsrc = (int)srcs.size();
    pg.nterm = (int)terms_in.size();
    pg.accumulate = accumulate ? 1 : 0;
    std::vector<int> src_of(terms_in.size());
    for (size_t s = 0; s < srcs.size(); s++) {
        pg.src[s] = srcs[s].u ? srcs[s].u : srcs[s].lane;
        pg.kept[s] = srcs[s].u ? 0 : 1;
        for (int t = srcs[s].t0; t < srcs[s].t1; t++) src_of[t] = (int)s;
    }
    int n = 0;
    for (int d = 0; d < X; d++) {   // terms sorted by output
        pg.dfirst[d] = n;
        pg.outs[d] = outs[d];
        for (size_t t = 0; t < terms_in.size(); t++)
            if (term_dest[t] == d) {
                pg.tvoff[n] = (u32)src_of[t] * kGmacTile * 16;
                pg.tmask[n] = terms_in[t].mask;
                n++;
            }
    }
    pg.dfirst[X] = n;
    // thread groups and their output slices, cut where the running term
    // count passes k / G of the total
    const int G = X >= ctx->tune.gmac_groups ? kGmacGroups : 1;
    pg.groups = G;
    pg.gfirst[0] = 0;
    int k = 1;
    for (int d = 0; d < X && k < G; d++)
        while (k < G && (int64_t)pg.dfirst[d + 1] * G >= (int64_t)k * n) pg.gfirst[k++] = d + 1;
    for (; k <= kGmacGroups; k++) pg.gfirst[k] = X;
    const int npoly = 2 * ncol;
    pg.ppc = std::min(npoly, 16);
    pg.ppn = std::min(kGmacTile / pg.ppc, 16);
    const int npg = (npoly + pg.ppc - 1) / pg.ppc;
    dim3 g(((N / 2 + pg.ppn - 1) / pg.ppn) * npg, E);
    FG_CHECK(g.x < (1u << 31), FG_EINVAL, "group_mac: grid too large");
    const size_t sm = (size_t)pg.nsrc * kGmacTile * 16 + (size_t)pg.nterm * pg.ppn * 16;
    const int v = (ctx->tune.gmac_regs ? 1 : 0) + (ctx->tune.kara ? 2 : 0);
    auto kern = v == 0 ? k_group_mac_tile<2, false> : v == 1 ? k_group_mac_tile<3, false>
              : v == 2 ? k_group_mac_tile<2, true> : k_group_mac_tile<3, true>;
    allow_shared(kern, sm);
    kern<<<g, G * kGmacTile, sm, ctx->stream>>>(pg, ncol, level, E, ls, ctx->log_n, ctx->d_primes, ctx->nq);
}

// up to kGmXs outputs: k_group_mac
static void group_mac_stream(fg_ctx *ctx, const std::vector<GroupSource> &srcs, const std::vector<Dest> &terms,
                             const std::vector<int> &term_dest, const std::vector<u64 *> &outs, bool accumulate,
                             int ncol, int level, int ls)
{
    const int N = ctx->n, E = ctx->ext(level), X = (int)outs.size();
    GProg pg;
    memset(&pg, 0, sizeof(pg));
    pg.nsrc = (int)srcs.size();
    pg.accumulate = accumulate ? 1 : 0;
    std::vector<const u64 *> mask((size_t)pg.nsrc * X, nullptr);
    for (int d = 0; d < X; d++) pg.outs[d] = outs[d];
    for (int s = 0; s < pg.nsrc; s++) {
        pg.src[s] = srcs[s].u ? srcs[s].u : srcs[s].lane;
        pg.bits[s] = srcs[s].u ? 0 : kGmKept;
        for (int t = srcs[s].t0; t < srcs[s].t1; t++) {
            const int d = term_dest[t];
            FG_CHECK(!(pg.bits[s] >> d & 1), FG_EINVAL, "group_mac: a source feeds an output twice");
            pg.bits[s] |= 1u << d;
            mask[(size_t)s * X + d] = terms[t].mask;
        }
    }
    // the tile: up to eight columns x 32 slots, more slots with fewer columns
    pg.npairs = ncol;
    const int npg = (ncol + 7) / 8;
    pg.pw = (ncol + npg - 1) / npg;
    pg.lts = 5;
    while ((pg.pw << (pg.lts - 4)) <= 8) pg.lts++;
    pg.nstage = (pg.nsrc + kGmChunk - 1) / kGmChunk;
    int n = 0;
    for (int s = 0; s < pg.nsrc; s++) {
        if (s % kGmChunk == 0) pg.tstage[s / kGmChunk] = n;
        for (int d = 0; d < X; d++)
            if (pg.bits[s] >> d & 1) {
                pg.trow[n] = (uint8_t)(s % kGmChunk * X + d);
                pg.tmask[n++] = mask[(size_t)s * X + d];
            }
    }
    pg.tstage[pg.nstage] = n;
    // 22 KB a stage with eight columns and six outputs; 64 KB with one column
    pg.stage_words = kGmChunk * ((2 * pg.pw << pg.lts) + (X << pg.lts));
    const size_t sm = (size_t)kGmStages * pg.stage_words * 8;
    const dim3 g(npg, N >> pg.lts, E);
    const GmacKernel kern = kGmacKernels[X - 1];
    allow_shared(kern, sm);
    kern<<<g, pg.pw << pg.lts, sm, ctx->stream>>>(pg, level, E, ls, ctx->log_n, ctx->d_primes, ctx->nq);
}

void group_mac(fg_ctx *ctx, const std::vector<GroupSource> &srcs, const std::vector<Dest> &terms,
               const std::vector<int> &term_dest, const std::vector<u64 *> &outs, bool accumulate, int ncol,
               int level, int ls)
{
    const int N = ctx->n, E = ctx->ext(level), X = (int)outs.size();
    if (srcs.empty() || X == 0) return;
    FG_CHECK((int)srcs.size() <= kGmacSrc && (int)terms.size() <= kGmacTerms && X <= kGmacOut, FG_EINVAL,
             "group_mac: launch larger than its program limits");
    double src_limbs = 0;
    for (const auto &gs : srcs) src_limbs += gs.u ? E : level + 1;
    KTimer kt(ctx, "group_mac",
              (src_limbs * 2 * ncol + (double)terms.size() * E +
               (double)X * 2 * ncol * E * (accumulate ? 2 : 1)) * N * 8);
    // Both forms timed over 22 to 36 sources at 65% of the terms, N = 2^16, 9
    // limbs of 45 bits and 5 of 60 (ms, streamed against tiles): 3 outputs
    // 1.41 / 1.62, 5 2.05 / 2.26, 6 3.08 / 4.73; with two blocks of up to six
    // outputs each the streamed form took 7 outputs 4.15 / 3.89, 12 outputs
    // 7.02 / 6.41.
    if (X > kGmXs)
        group_mac_tile(ctx, srcs, terms, term_dest, outs, accumulate, ncol, level, ls);
    else
        group_mac_stream(ctx, srcs, terms, term_dest, outs, accumulate, ncol, level, ls);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw fg_error(FG_ECUDA, std::string("group_mac: ") + cudaGetErrorString(e));
    ctx->launches += 1;
}

}  // namespace kern
