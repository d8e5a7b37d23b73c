// Persistent two-sided block Jacobi eigensolver for the Gram matrix G = B B^T of the projected input
// (Rayleigh-Ritz step of the basis extraction, Sec. 4.2: the rotation that diagonalises G turns the
// orthonormal range basis into singular vectors, X' = [sigma_i v_i]).
//
// One cooperative launch diagonalises every sequence of a batch. Each sequence owns a fixed group of
// CTAs (pivot CTAs, one a pair as a rule, and workers; see launch and seat_of) that loops over sweeps and steps on its own and leaves when its matrix has converged; the
// CTAs of a group meet at a counter in global memory (bounded spin) instead of at kernel boundaries.
// Blocks of 32 rows; a step handles n/64 disjoint block pairs (round-robin order) in two phases:
//   pivot : per pair, the 64 x 64 pivot block is rotated on chip by cyclic Jacobi (first step of a sweep: all
//           2016 pairs of its 64 rows once, in 63 rounds; other steps: the 1024 pairs across its two blocks, in
//           32 rounds). The block lives in registers (see "pivot phase" below); a round is a rotation per row
//           pair, one block barrier and a shift of the pairing. The accumulated row transform Vt (64 x 64)
//           is published, and of a step of 32 rounds the two diagonal blocks of the rotated pivot block. The pivot
//           block of the NEXT step is formed on chip from those and one block of the matrix before this step's update
//           (pivot_form_cross; after a sweep's first step from three blocks, pivot_form), so the chain of pivot solves
//           runs beside the update and never waits for it.
//   apply : every 64 x 64 block (p, q) of G becomes Vt_p G_pq Vt_q^T (upper triangle computed, mirror
//           stored), rows of Wt become Vt_p Wt, both in place. The pivot CTAs of the step read blocks of G as they
//           were before the update; a counter of fetched pivot blocks holds the first store of every updating
//           CTA back until they have them on chip. The 64^3 products run on the tensor cores from two fp16 parts per operand
//           (split_mma.cuh; see "published transforms" for the scaling); fp32 inputs use the fp32 units.
// G and Wt are stored with a leading dimension padded to a multiple of 64; the padding of G is zero
// (zero diagonal entries are never rotated), the padding of Wt is the identity.
#pragma once
#include "common.cuh"
#include "group_barrier.cuh"
#include "split_mma.cuh"
#include <mutex>
#include <algorithm>

namespace j3 {

constexpr int JB = 32;            // block height
constexpr int BLK = 64;           // pivot block = one pair of blocks
constexpr int NT = 256;           // threads per CTA
constexpr int LDA = 68;           // shared-memory row stride (floats) of A-operand style tiles
constexpr int LDB = 72;           // shared-memory row stride of B-operand style tiles
constexpr int MAXSEQ = 32;        // sequences per launch
constexpr int SYNC_WORDS = 64;
// Rows of G whose diagonal entry is at most NEGLIGIBLE times the largest one (rows of B below 2^-37 of the longest) are what a
// rank-deficient input leaves: rounding, with a Gram matrix that is not even positive, so that rotations among such rows do not
// end. No pass waits for their entries, they are not rotated against each other, and one whose diagonal entry is not positive is
// not rotated at all. (A token that is that small stays in use: rotations against longer rows go on as long as a pass does.)
constexpr float NEGLIGIBLE = 0x1p-74f;
constexpr int VSTRIDE = 2 * BLK * BLK + 2 * BLK + 2 * JB * JB;   // floats of a published transform (see below)

struct Seq {
    float *G, *Wt, *Vbuf;         // G, Wt: np x np (ld = np); Vbuf: 2 x npairs x VSTRIDE (by step parity)
    int *vflag;                   // 2 x npairs: the pair rotated in this step
    unsigned *sync;               // SYNC_WORDS words (in the first sequence of a launch the list of SMs, 2 words an SM, lies behind
                                  // them). [0]: arrivals at the group barrier (monotonic); largest scaled off-diagonal
                                  // entry, slot sweep % 4: [1..4] met in a sweep, [8..11] in the whole matrix after it;
                                  // [5]: sweeps used; [6]: largest diagonal entry at the start; by step parity: [16..17] work
                                  // tickets of the update, [20..21] pivot blocks fetched; [32]: arrivals of the whole launch
    int n, np, nb;                // size, padded size (multiple of 64), number of 32-row blocks (even)
    int ncta, npu;                // CTAs that own this sequence; those of them that solve pivot blocks
    int pivot0, worker0;          // numbers of the first of its pivot CTAs and of the first of the others (see seat_of)
};
struct Batch {
    Seq s[MAXSEQ]; int count;
    int pivots;                   // pivot CTAs of all sequences
    bool seated;                  // two CTAs to an SM: roles by seat_of, else by block number
    unsigned *grid_sync, *smids;  // arrivals of all CTAs of the launch (zero at the start); the SM of each of them
};

// Bytes of dynamic shared memory: four tile slots of 64 x LDB floats (pivot phase: the old blocks and the
// transforms the pivot block is formed from, then A and Vt; apply phase: Vt_p, Vt_q, T and the G block).
constexpr int SLOT = BLK * LDB;
constexpr size_t SMEM_BYTES = (size_t)4 * SLOT * sizeof(float);

__device__ __forceinline__ void rr_pair(int nb, int step, int t, int &I, int &J)
{
    const int m = nb - 1;                    // 0 <= step < m, 0 <= t < nb / 2
    if (t == 0) { I = m; J = step; }
    else { I = step + t; J = step - t; I -= I >= m ? m : 0; J += J < 0 ? m : 0; }
    if (I > J) { const int x = I; I = J; J = x; }
}
// The pair t that block b is in at a step, and whether b is the second of its two blocks.
__device__ __forceinline__ void rr_locate(int nb, int step, int b, int &t, int &h)
{
    const int m = nb - 1;
    int x = b - step, other;
    x += x < 0 ? m : 0;
    if (b == m) { t = 0; other = step; }
    else if (x == 0) { t = 0; other = m; }
    else if (x < nb / 2) { t = x; other = step - t; other += other < 0 ? m : 0; }
    else { t = m - x; other = step + t; other -= other >= m ? m : 0; }
    h = b > other;
}

using ::group_barrier;

// ---- pivot phase -------------------------------------------------------------------------------
// The 64 rows of a pivot block sit in 32 "even" and 32 "odd" slots. A phase of width M rotates, in M rounds, every
// even slot k with the odd slots of its own group of M: in round rd with slot base(k) + ((k - rd) mod M). Width 32
// pairs every row of the first block with every row of the second; widths 16, 8, 4, 2, 1 pair the rows inside the
// blocks; together the 63 rounds rotate each of the 2016 pairs exactly once. Slot -> logical row (0..31 first block,
// 32..63 second block): the logical rows are cut in groups of 2M; the first M of a group are even slots, the last M odd.
//
// What bounds a round is the chain rotation -> entry of the next pair -> next rotation, so the layout makes that
// chain live in one warp. Lane k of a warp holds, for offsets d = 0 .. M/2, the 2 x 2 blocks between the pairs k and
// k + d (mod M; the matrix is symmetric, so half of the offsets suffice):
//     ee[d] = A[E(k)][E(k+d)]   eo[d] = A[E(k)][O(k+d)]   oe[d] = A[O(k)][E(k+d)]   oo[d] = A[O(k)][O(k+d)]
// with O(k) the odd row now paired with E(k). Moving to the next pairing, O(k) <- O(k-1), is then
//     oo[d] <- oo[d] of lane k-1,   oe[d] <- oe[d+1] of lane k-1,   eo[d] <- eo[d-1] of the same lane,
//     eo[0] <- oe[1] of lane k-1,   oe[M/2] <- eo[M/2-1] of lane k+M/2,
// and the 2 x 2 problem of the next round needs the offsets 0 and 1 only: warp 0 owns them, derives the next 32
// rotations from two shuffles and publishes them. Width 32: offsets 0-2, 3-7, 8-12, 13-16 live in warps 0-3, and the
// entries that cross a warp boundary go through shared memory; one block barrier a round. Widths <= 16 only need the
// diagonal sub-blocks (the block itself is discarded afterwards, only the transform is kept): warp 0 holds them all.
// Warps 4-7 apply the published rotations to the transform: lane = two columns, warp = a quarter of the row pairs.
// Second bound: issue slots, FMA and shared-memory cycles of those updates. The rotations are therefore applied without
// their common factor c (Gentleman's fast Givens form): row = d * stored row, and with t = s / c
//     x~ <- x~ - beta y~,  y~ <- y~ + gamma x~,   beta = t d_y / d_x,  gamma = t d_x / d_y,   d_x, d_y <- c d_x, c d_y,
// two multiply-adds instead of four operations; |t| <= 1, so d loses at most a factor 2^-16 in 32 rounds. The factors
// live in warp 0 and are multiplied back at the end of a phase.
// Cross phase of 32 rounds, one CTA alone on an SM: 31500 -> 9600 cycles; all 63 rounds: 68000 -> 23600 (the layout
// before put a quarter of the rows in each thread: every round moved a row between warps behind a second barrier, and
// the next rotation waited for all of it). Packed fp32x2 arithmetic was slower: 13900 cycles, it adds register moves.
constexpr int LDP = 65;           // row stride of the logical pivot block and transform in shared memory

struct PivotShared {
    float2 bg[2][32];             // (beta, gamma) of the current round, by round parity
    float2 vx[2][4][32];          // last odd row of each quarter of the transform
    float up[2][3][32];           // eo of the last offset of warp w, for warp w + 1
    float dn[2][3][32];           // oe of the first offset of warp w + 1, for warp w
    float sd[2][64];              // row factors d at the end of a phase (even slots, odd slots), by phase parity
    float red[4];
    float d[64];                  // powers of two above the square roots of the diagonal
};

__device__ __forceinline__ float rsqrt_ftz(float x) { float y; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

// 2^-e for x in [2^e, 2^(e+1)), from the exponent field (kept to normal numbers)
__device__ __forceinline__ float inv_exponent(float x)
{
    return __uint_as_float(0x7f000000u - min(max(__float_as_uint(x) & 0x7f800000u, 0x01000000u), 0x7e800000u));
}

// The rotations of the pairs of warp 0, one per lane, with the row factors of the pair (and their reciprocals) and the
// two diagonal entries.
struct Rotor {
    float de, ie, dod, io, gpp, gqq;
    __device__ __forceinline__ void reset(float ee, float oo) { de = ie = dod = io = 1.f; gpp = ee; gqq = oo; }
    // Rotation that annihilates the entry between the rows p (even) and q (odd) of a symmetric matrix, stored as eo;
    // identity when the entry is already small against its diagonal. With a = g_qq - g_pp, b = 2 g_pq,
    // r = sqrt(a^2 + b^2):
    //   cos 2t = |a| / r,  c = sqrt((1 + cos 2t) / 2),  tan t = sign(a) b / (2 r c^2)      (|t| <= pi/4).
    // What does not depend on eo (it arrives last) comes first. The squares are taken of entries scaled by the power of two
    // that brings the larger diagonal entry into [1, 2): an entry worth rotating is then far above the flush to zero of the
    // approximate reciprocal root (1 / 0 times 0 otherwise), whatever the scale of the matrix. Returns (beta, gamma) and
    // advances the factors and the diagonal.
    __device__ __forceinline__ float2 next(float eo, float tol2)
    {
        const float w = de * dod, dp = fmaxf(gpp, 0.f), dq = fmaxf(gqq, 0.f);
        const float sc = inv_exponent(fmaxf(fabsf(gpp), fabsf(gqq)));
        const float a = (gqq - gpp) * sc, a2 = a * a, ah = 0.5f * fabsf(a), sgw = copysignf(sc, a) * w;
        const float thr = fmaxf(4.f * tol2 * (dp * sc) * (dq * sc), 0x1p-120f), scw = 2.f * sc * w, kb = dod * ie, kg = de * io;
        const float b = eo * scw, b2 = b * b;
        const float r2 = b2 + a2;
        const float rh = rsqrt_ftz(r2);
        const float c2 = fmaf(ah, rh, 0.5f);
        const float rc = rsqrt_ftz(c2);
        const float gpq = eo * w;
        const bool on = b2 > thr;
        const float t = on ? (eo * sgw) * rh * (rc * rc) : 0.f;
        const float2 out = make_float2(t * kb, t * kg);
        gpp = fmaf(-t, gpq, gpp); gqq = fmaf(t, gpq, gqq);
        // c = 1 / sqrt(1 + t^2) for the t that is applied: one Newton step from c0 = cos t above. The bias of the approximate
        // roots in c^2 (1 + t^2) would add up over the rotations of a row.
        const float c0 = on ? c2 * rc : 1.f, cc = c0 * c0, ch = 0.5f * c0;
        const float q2 = fmaf(t, t, 1.f), c = fmaf(ch, fmaf(-cc, q2, 1.f), c0), ic = q2 * c;
        de *= c; dod *= c; ie *= ic; io *= ic;
        ie = ie * fmaf(-de, ie, 2.f); io = io * fmaf(-dod, io, 2.f);      // keeps d * (1 / d) = 1 to the last bit or so
        return out;
    }
    __device__ __forceinline__ void shift(int km)
    {
        dod = __shfl_sync(0xffffffffu, dod, km); io = __shfl_sync(0xffffffffu, io, km); gqq = __shfl_sync(0xffffffffu, gqq, km);
    }
};

// [ee eo; oe oo] <- R(ra) [ee eo; oe oo] R(rb)^T with R(r) = [1 -beta; gamma 1]
__device__ __forceinline__ void rotate_block(float2 ra, float2 rb, float &ee, float &eo, float &oe, float &oo)
{
    const float r0 = fmaf(-ra.x, oe, ee), r1 = fmaf(-ra.x, oo, eo);
    const float r2 = fmaf(ra.y, ee, oe), r3 = fmaf(ra.y, eo, oo);
    ee = fmaf(-rb.x, r1, r0); eo = fmaf(rb.y, r0, r1);
    oe = fmaf(-rb.x, r3, r2); oo = fmaf(rb.y, r2, r3);
}

// Offsets of a width-32 phase in warp W of 0..3: 0-2, 3-7, 8-12, 13-16 (warp 0 has the rotations to do as well).
template <int W> struct Band {
    static constexpr int D0 = W == 0 ? 0 : 5 * W - 2, ND = W == 0 ? 3 : (W == 3 ? 4 : 5);
    float ee[ND], eo[ND], oe[ND], oo[ND];
    // loads the offsets from As, without the entries that are not rotated (see NEGLIGIBLE; rows with a diagonal entry of at most
    // `least`), and returns the largest scaled off-diagonal entry among those that a pass waits for
    __device__ __forceinline__ float load(const float *As, float least)
    {
        const int k = threadIdx.x & 31;
        const float de = As[k * (LDP + 1)], dd = As[(32 + k) * (LDP + 1)];
        const float re = de > least ? rsqrtf(de) : 0.f, ro = dd > least ? rsqrtf(dd) : 0.f;
        float me = 0.f, mo = 0.f;                                // in the even rows and in the odd ones, without re and ro
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const int l = (k + D0 + i) & 31;
            ee[i] = As[k * LDP + l]; eo[i] = As[k * LDP + 32 + l];
            oe[i] = As[(32 + k) * LDP + l]; oo[i] = As[(32 + k) * LDP + 32 + l];
            const float le = __shfl_sync(0xffffffffu, re, l), lo = __shfl_sync(0xffffffffu, ro, l);
            if (D0 + i > 0) { me = fmaxf(me, fabsf(ee[i]) * le); mo = fmaxf(mo, fabsf(oo[i]) * lo); }
            me = fmaxf(me, fabsf(eo[i]) * lo); mo = fmaxf(mo, fabsf(oe[i]) * le);
        }
        mo = fmaxf(me * re, mo * ro);
        // (zero: padding, or a row of zeros)
        if (__any_sync(0xffffffffu, (de <= least && de != 0.f) || (dd <= least && dd != 0.f))) {
            auto keep = [&](float &g, float a, float b) { if (fminf(a, b) <= 0.f || fmaxf(a, b) <= least) g = 0.f; };
#pragma unroll
            for (int i = 0; i < ND; ++i) {
                const int l = (k + D0 + i) & 31;
                const float fe = __shfl_sync(0xffffffffu, de, l), fo = __shfl_sync(0xffffffffu, dd, l);
                keep(eo[i], de, fo); keep(oe[i], dd, fe);
                if (D0 + i > 0) { keep(ee[i], de, fe); keep(oo[i], dd, fo); }
            }
        }
        return mo;
    }
    // the 32 rounds; the diagonal quadrants (both blocks after the cross rotations) go back to As
    __device__ __forceinline__ void rounds(float *As, PivotShared &sh, float tol2)
    {
        const int k = threadIdx.x & 31, km = (k - 1) & 31;
        float2 own = make_float2(0.f, 0.f), nxt = own;           // warp 0: rotations of the pairs k and k + 1
        Rotor rot;
        auto publish = [&](int par, bool last) {
            own = rot.next(eo[0], tol2);
            sh.bg[par][k] = own;
            if (last) { sh.sd[0][k] = rot.de; sh.sd[0][32 + ((k + 1) & 31)] = rot.dod; }
            rot.shift(km);
            nxt.x = __shfl_sync(0xffffffffu, own.x, (k + 1) & 31);
            nxt.y = __shfl_sync(0xffffffffu, own.y, (k + 1) & 31);
        };
        if (W == 0) { rot.reset(ee[0], oo[0]); publish(0, false); }
        __syncthreads();
#pragma unroll 2
        for (int rd = 0; rd < 32; ++rd) {
            const int par = rd & 1;
            const float2 ra = W == 0 ? own : sh.bg[par][k];
            float2 rb[ND];
#pragma unroll
            for (int i = 0; i < ND; ++i) rb[i] = W == 0 && i == 0 ? own : W == 0 && i == 1 ? nxt : sh.bg[par][(k + D0 + i) & 31];
            if (rd > 0) {                                        // entries that crossed a warp boundary in the last shift
                if (W > 0) eo[0] = sh.up[par ^ 1][W > 0 ? W - 1 : 0][k];
                if (W < 3) oe[ND - 1] = sh.dn[par ^ 1][W < 3 ? W : 0][km];
            }
#pragma unroll
            for (int i = 0; i < ND; ++i) rotate_block(ra, rb[i], ee[i], eo[i], oe[i], oo[i]);
            // next pairing
            if (W < 3) sh.up[par][W < 3 ? W : 0][k] = eo[ND - 1];
            if (W > 0) sh.dn[par][W > 0 ? W - 1 : 0][k] = oe[0];
            float wrap = 0.f, in0 = 0.f;
            if (W == 0) in0 = __shfl_sync(0xffffffffu, oe[1], km);
            if (W == 3) wrap = __shfl_sync(0xffffffffu, eo[ND - 2], k ^ 16);
#pragma unroll
            for (int i = 0; i < ND; ++i) oo[i] = __shfl_sync(0xffffffffu, oo[i], km);
#pragma unroll
            for (int i = ND - 1; i > 0; --i) eo[i] = eo[i - 1];
            if (W == 0) eo[0] = in0;
            if (W == 0 && rd < 31) publish(par ^ 1, rd == 30);
#pragma unroll
            for (int i = 0; i + 1 < ND; ++i) oe[i] = __shfl_sync(0xffffffffu, oe[i + 1], km);
            if (W == 3) oe[ND - 1] = wrap;
            __syncthreads();
        }
        const float de = sh.sd[0][k], dd = sh.sd[0][32 + k];
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const int l = (k + D0 + i) & 31;
            if (D0 + i == 16 && k >= 16) continue;               // (two lanes have these entries, equal but for rounding)
            const float e = ee[i] * de * sh.sd[0][l], o = oo[i] * dd * sh.sd[0][32 + l];
            As[k * LDP + l] = e; As[l * LDP + k] = e;
            As[(32 + k) * LDP + 32 + l] = o; As[(32 + l) * LDP + 32 + k] = o;
        }
    }
};

// A phase of width M <= 16 on the diagonal sub-blocks of 2M rows, in warp 0; one block barrier per round. ph: phase parity.
template <int M> __device__ __forceinline__ void inner_phase(float *As, PivotShared &sh, float tol2, int ph)
{
    constexpr int ND = M / 2 + 1;
    const int k = threadIdx.x & 31, g = k & ~(M - 1), q = k & (M - 1);
    const int E = 2 * g + q, km = g | ((q - 1) & (M - 1)), kp = g | ((q + 1) & (M - 1)), kh = g | ((q + M / 2) & (M - 1));
    float ee[ND], eo[ND], oe[ND], oo[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) {
        const int F = 2 * g + ((q + i) & (M - 1));
        ee[i] = As[E * LDP + F]; eo[i] = As[E * LDP + F + M];
        oe[i] = As[(E + M) * LDP + F]; oo[i] = As[(E + M) * LDP + F + M];
    }
    Rotor rot;
    rot.reset(ee[0], oo[0]);
    float2 own = rot.next(eo[0], tol2);
    sh.bg[0][k] = own;
    if (M == 1) { sh.sd[ph][k] = rot.de; sh.sd[ph][32 + k] = rot.dod; }
    rot.shift(km);
#pragma unroll 1
    for (int rd = 0; rd < M; ++rd) {
        const int par = rd & 1;
        __syncthreads();
        float2 rb[ND];
#pragma unroll
        for (int i = 0; i < ND; ++i) rb[i] = i == 0 ? own : sh.bg[par][g | ((q + i) & (M - 1))];
#pragma unroll
        for (int i = 0; i < ND; ++i) rotate_block(own, rb[i], ee[i], eo[i], oe[i], oo[i]);
        if (M > 1) {
            const float in0 = __shfl_sync(0xffffffffu, oe[ND > 1 ? 1 : 0], km);
            const float wrap = __shfl_sync(0xffffffffu, eo[ND > 1 ? ND - 2 : 0], kh);
#pragma unroll
            for (int i = 0; i < ND; ++i) oo[i] = __shfl_sync(0xffffffffu, oo[i], km);
#pragma unroll
            for (int i = ND - 1; i > 0; --i) eo[i] = eo[i - 1];
            eo[0] = in0;
            if (rd + 1 < M) {
                own = rot.next(eo[0], tol2);
                sh.bg[par ^ 1][k] = own;
                if (rd + 2 == M) { sh.sd[ph][k] = rot.de; sh.sd[ph][32 + kp] = rot.dod; }
                rot.shift(km);
            }
#pragma unroll
            for (int i = 0; i + 1 < ND; ++i) oe[i] = __shfl_sync(0xffffffffu, oe[i + 1], km);
            oe[ND - 1] = wrap;
        }
    }
    if (M > 1) {
        const float de = sh.sd[ph][k], dd = sh.sd[ph][32 + k];
#pragma unroll
        for (int i = 0; i < ND; ++i) {
            const int l = (q + i) & (M - 1), F = 2 * g + l;
            const float e = ee[i] * de * sh.sd[ph][g + l], o = oo[i] * dd * sh.sd[ph][32 + g + l];
            As[E * LDP + F] = e; As[F * LDP + E] = e;
            As[(E + M) * LDP + F + M] = o; As[(F + M) * LDP + E + M] = o;
        }
        __syncwarp();
    }
}

// The transform's share of a phase (warps 4..7): lane = columns 2 l and 2 l + 1, warp 4 + h = the rows of the pairs
// 8 h .. 8 h + 7. Widths 32 and 16: ve / vo = even and odd rows in slot order; the odd row that leaves the quarter goes to
// the next quarter of its group through shared memory. Widths <= 8: the 16 rows 16 h .. 16 h + 15 in v.
__device__ __forceinline__ void rotate_rows(float b, float g, float2 &x, float2 &y)
{
    const float2 t = x;
    x = make_float2(fmaf(-b, y.x, t.x), fmaf(-b, y.y, t.y));
    y = make_float2(fmaf(g, t.x, y.x), fmaf(g, t.y, y.y));
}
__device__ __forceinline__ void scale_row(float2 &x, float d) { x.x *= d; x.y *= d; }
__device__ __forceinline__ void transform_wide(float2 (&ve)[8], float2 (&vo)[8], PivotShared &sh, int rounds, int h, int from)
{
    const int l = threadIdx.x & 31;
#pragma unroll 2
    for (int rd = 0; rd < rounds; ++rd) {
        const int par = rd & 1;
        __syncthreads();
        if (rd > 0) vo[0] = sh.vx[par ^ 1][from][l];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const float4 r = *(const float4 *)&sh.bg[par][8 * h + i];
            rotate_rows(r.x, r.y, ve[i], vo[i]);
            rotate_rows(r.z, r.w, ve[i + 1], vo[i + 1]);
        }
        sh.vx[par][h][l] = vo[7];
#pragma unroll
        for (int i = 7; i > 0; --i) vo[i] = vo[i - 1];
    }
}
template <int M> __device__ __forceinline__ void transform_inner(float2 (&v)[16], PivotShared &sh, int h, int ph)
{
#pragma unroll 1
    for (int rd = 0; rd < M; ++rd) {
        const int par = rd & 1;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const float4 r = *(const float4 *)&sh.bg[par][8 * h + i];
            const int e0 = 2 * M * (i / M) + i % M, e1 = 2 * M * ((i + 1) / M) + (i + 1) % M;
            rotate_rows(r.x, r.y, v[e0], v[e0 + M]);
            rotate_rows(r.z, r.w, v[e1], v[e1 + M]);
        }
#pragma unroll
        for (int g = 0; g < 8 / M; ++g) {                        // odd rows of a group move on by one slot
            const int o = 2 * M * g + M;
            const float2 last = v[o + M - 1];
#pragma unroll
            for (int i = M - 1; i > 0; --i) v[o + i] = v[o + i - 1];
            v[o] = last;
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = 2 * M * (i / M) + i % M;
        scale_row(v[e], sh.sd[ph][8 * h + i]); scale_row(v[e + M], sh.sd[ph][32 + 8 * h + i]);
    }
}

// global row / column of local index l of the pair (I, J)
__device__ __forceinline__ int glob_of_loc(int I, int J, int l) { return (l < JB ? I : J) * JB + (l & (JB - 1)); }

// Copies the 64 x 64 pivot block of the pair (I, J) from G to the logical copy As (stride LDP).
__device__ void pivot_load(float *sm, const float *G, int np, int I, int J)
{
    float *As = sm;
    for (int f = threadIdx.x; f < BLK * (BLK / 4); f += NT) {
        const int li = f >> 4, lj = (f & 15) * 4;
        const float4 v = __ldcg((const float4 *)(G + (size_t)glob_of_loc(I, J, li) * np + glob_of_loc(I, J, lj)));
        float *dst = As + li * LDP + lj;
        dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
    }
}

// Rotates the 64 x 64 pivot block held in As = sm (stride LDP, complete before the call: the routine starts with
// a block barrier) and publishes the accumulated row transform Vt (new rows = Vt * old rows, logical order) to
// vout. cross_only: the 32 rounds that pair the two blocks' rows; otherwise all 63 rounds. Returns the largest
// scaled off-diagonal entry found in the block before rotating (block-uniform); when it is <= tol_rot nothing is
// rotated or published.
template <int W> __device__ __forceinline__ float pivot_warp(float *As, PivotShared &sh, bool cross_only, float tol_rot, float least, float *quad)
{
    const float tol2 = tol_rot * tol_rot;
    Band<W> band;
    float mo = band.load(As, least);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mo = fmaxf(mo, __shfl_xor_sync(0xffffffffu, mo, o));
    if ((threadIdx.x & 31) == 0) sh.red[W] = mo;
    __syncthreads();
    mo = fmaxf(fmaxf(sh.red[0], sh.red[1]), fmaxf(sh.red[2], sh.red[3]));
    if (!(mo > tol_rot)) return mo;
    band.rounds(As, sh, tol2);
    if (cross_only) {
        asm volatile("bar.sync 3, 128;" ::: "memory");           // these four warps
        const int f = threadIdx.x & 127;
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int q = it >> 1, e = (f + (it & 1) * 128) * 4;
            const float *src = As + (q * JB + (e >> 5)) * LDP + q * JB + (e & 31);
            *(float4 *)(quad + q * JB * JB + e) = make_float4(src[0], src[1], src[2], src[3]);
        }
    } else {
        __syncthreads();
        if (W == 0) {
            inner_phase<16>(As, sh, tol2, 1); inner_phase<8>(As, sh, tol2, 0); inner_phase<4>(As, sh, tol2, 1);
            inner_phase<2>(As, sh, tol2, 0); inner_phase<1>(As, sh, tol2, 1);
        } else {
#pragma unroll 1
            for (int rd = 0; rd < 31; ++rd) __syncthreads();
        }
    }
    return mo;
}
// Published transforms. fp32 inputs: Vt as 64 x 64 floats. Otherwise, for products from fp16 parts, with powers of two
//     d_i >= sqrt(g_ii)  per row of the pivot block before the rotation,     s_i > max_k |vt_ik| d_k  per row of Vt:
//   VS  = diag(1/s) Vt diag(d)  (entries below 1), 64 x 64 fp16 high parts, then the low parts, times V_SCALE: rotates G,
//         whose blocks diag(1/d_p) G_pq diag(1/d_q) have entries of at most 1 however the rows are graded; the result is scaled
//         back by s_p, s_q. What is left out is below 2^-35 s_i s_j, on top of 2^-22 of the entries themselves.
//   VU  = Vt times V_SCALE in the same form: rotates the rows of Wt, whose entries are at most 1.
//   d, s as 64 floats each (s = d where the pair was not rotated).
// Behind them, for every input and where the 32 rounds alone were done: the two 32 x 32 diagonal blocks of the rotated pivot block.
constexpr float V_SCALE = 8192.f, G_SCALE = 1024.f, T_SCALE = 256.f;
constexpr int V_VU = BLK * BLK, V_D = 2 * BLK * BLK, V_S = V_D + BLK, V_Q = V_S + BLK;     // offsets in floats
constexpr int LDV = 66;           // row stride of the transform in shared memory
__device__ __forceinline__ float inv_pow2(float x) { return __uint_as_float(0x7f000000u - __float_as_uint(x)); }

template <bool TENSOR>
__device__ float pivot_rotate(float *sm, bool cross_only, float tol_rot, float least, float *vout, bool &rotated)
{
    __shared__ __align__(16) PivotShared sh;
    const int tid = threadIdx.x, warp = tid >> 5, l = tid & 31;
    float *As = sm, *Vs = sm + BLK * LDP;
    float mo;
    __syncthreads();
    if (TENSOR && tid < BLK) {
        // g < 2^(E - 126): d = 2^ceil((E - 126) / 2)
        const float g = As[tid * (LDP + 1)];
        const int e = g > 0.f ? min(max(((int)(__float_as_uint(g) >> 23) - 125) >> 1, -60), 63) : -60;
        const float d = __int_as_float((127 + e) << 23);
        sh.d[tid] = d;
        vout[V_D + tid] = d;
        vout[V_S + tid] = d;                                     // (overwritten below where rows are rotated)
    }
    if (warp == 0) mo = pivot_warp<0>(As, sh, cross_only, tol_rot, least, vout + V_Q);
    else if (warp == 1) mo = pivot_warp<1>(As, sh, cross_only, tol_rot, least, vout + V_Q);
    else if (warp == 2) mo = pivot_warp<2>(As, sh, cross_only, tol_rot, least, vout + V_Q);
    else if (warp == 3) mo = pivot_warp<3>(As, sh, cross_only, tol_rot, least, vout + V_Q);
    else {
        const int h = warp - 4;
        __syncthreads();
        mo = fmaxf(fmaxf(sh.red[0], sh.red[1]), fmaxf(sh.red[2], sh.red[3]));
        if (mo > tol_rot) {
            float2 ve[8], vo[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int e = 8 * h + i, o = 32 + e;
                ve[i] = make_float2(e == 2 * l ? 1.f : 0.f, e == 2 * l + 1 ? 1.f : 0.f);
                vo[i] = make_float2(o == 2 * l ? 1.f : 0.f, o == 2 * l + 1 ? 1.f : 0.f);
            }
            transform_wide(ve, vo, sh, 32, h, (h - 1) & 3);
            __syncthreads();
            vo[0] = sh.vx[1][(h - 1) & 3][l];
#pragma unroll
            for (int i = 0; i < 8; ++i) { scale_row(ve[i], sh.sd[0][8 * h + i]); scale_row(vo[i], sh.sd[0][32 + 8 * h + i]); }
            auto put = [&](int row, float2 v) { *(float2 *)(Vs + row * LDV + 2 * l) = v; };
            auto get = [&](int row) { return *(const float2 *)(Vs + row * LDV + 2 * l); };
            auto publish = [&](int row, float2 v) {
                if (!TENSOR) { *(float2 *)(vout + row * BLK + 2 * l) = v; return; }
                auto parts = [&](float *dst, float x, float y) {
                    const __half2 hi = __floats2half2_rn(x, y);
                    const float2 f = __half22float2(hi);
                    ((__half2 *)dst)[row * 32 + l] = hi;
                    ((__half2 *)dst)[2048 + row * 32 + l] = __floats2half2_rn(x - f.x, y - f.y);
                };
                parts(vout + V_VU, v.x * V_SCALE, v.y * V_SCALE);
                const float x = v.x * sh.d[2 * l], y = v.y * sh.d[2 * l + 1];
                const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(fabsf(x), fabsf(y))));
                const int e = min(max((int)(m >> 23), 20), 250);                  // largest entry < 2^(e - 126)
                const float is = __int_as_float((266 - e) << 23);                 // V_SCALE * 2^(126 - e)
                parts(vout, x * is, y * is);
                if (l == 0) vout[V_S + row] = __int_as_float((e + 1) << 23);
            };
            auto vbar = [] { asm volatile("bar.sync 1, 128;" ::: "memory"); };          // the warps of the transform
            if (cross_only) {
#pragma unroll
                for (int i = 0; i < 8; ++i) { publish(8 * h + i, ve[i]); publish(32 + 8 * h + i, vo[i]); }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) { put(8 * h + i, ve[i]); put(32 + 8 * h + i, vo[i]); }
                vbar();
                const int e16 = 32 * (h >> 1) + 8 * (h & 1);     // width 16: even rows e16 + i, odd rows 16 further on
#pragma unroll
                for (int i = 0; i < 8; ++i) { ve[i] = get(e16 + i); vo[i] = get(e16 + 16 + i); }
                __syncthreads();
                transform_wide(ve, vo, sh, 16, h, h ^ 1);
                vbar();
                vo[0] = sh.vx[1][h ^ 1][l];
#pragma unroll
                for (int i = 0; i < 8; ++i) { scale_row(ve[i], sh.sd[1][8 * h + i]); scale_row(vo[i], sh.sd[1][32 + 8 * h + i]); }
#pragma unroll
                for (int i = 0; i < 8; ++i) { put(e16 + i, ve[i]); put(e16 + 16 + i, vo[i]); }
                vbar();
                float2 v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = get(16 * h + i);
                transform_inner<8>(v, sh, h, 0); transform_inner<4>(v, sh, h, 1); transform_inner<2>(v, sh, h, 0);
                transform_inner<1>(v, sh, h, 1);
#pragma unroll
                for (int i = 0; i < 16; ++i) publish(16 * h + i, v[i]);
            }
        }
    }
    rotated = mo > tol_rot;
    return mo;
}

// ---- apply phase -------------------------------------------------------------------------------
// A 64^3 product on the fp32 FMA units: B[k][n] = Bs[k * ldb + n], or Bs[n * ldb + k] when B_TRANS; rows of A at stride LDA (this
// thread: rows m0 + g and m0 + g + 8, columns n0 + 8 nt + 2 t, + 1). Used for fp32 inputs, whose
// convergence threshold (1e-6) sits below the rounding of the split-precision product (~2^-21).
template <bool B_TRANS>
__device__ __forceinline__ void product64_fma(const float *As, const float *Bs, int ldb, int m0, int n0, float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[nt][i] = 0.f;
#pragma unroll 2
    for (int k0 = 0; k0 < BLK; k0 += 4) {
        const float4 a0 = *(const float4 *)(As + (m0 + g) * LDA + k0);
        const float4 a1 = *(const float4 *)(As + (m0 + g + 8) * LDA + k0);
        const float av0[4] = {a0.x, a0.y, a0.z, a0.w}, av1[4] = {a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
                const int n = n0 + nt * 8 + 2 * t;
                float b0, b1;
                if (B_TRANS) { b0 = Bs[n * ldb + k0 + kk]; b1 = Bs[(n + 1) * ldb + k0 + kk]; }
                else { const float2 b = *(const float2 *)(Bs + (k0 + kk) * ldb + n); b0 = b.x; b1 = b.y; }
                acc[nt][0] = fmaf(av0[kk], b0, acc[nt][0]); acc[nt][1] = fmaf(av0[kk], b1, acc[nt][1]);
                acc[nt][2] = fmaf(av1[kk], b0, acc[nt][2]); acc[nt][3] = fmaf(av1[kk], b1, acc[nt][3]);
            }
        }
    }
}

// Forms, on chip, the pivot block that a pair of the NEXT step will have once the current step's update is done,
// from the state before that update. The pair's first block sits in half h1 of the current pair p1, its second in
// half h2 of the current pair p2. With W1 / W2 the 32 rows of Vt_p1 / Vt_p2 that produce those blocks (rows of
// the identity where the pair was not rotated: f1 / f2 = 0) and X_ab the old blocks between the pairs a and b,
//   N = [ W1 X11 W1^T   W1 X12 W2^T ]
//       [   (mirror)    W2 X22 W2^T ]
// in three 64^3 products: [W1 X11; W2 X22] and W1 X12 first, then the multiplication by [W1; W2]^T from the
// right. The result lands in As = sm (stride LDP). So the chain of pivot solves never waits for the update.
__device__ void pivot_form(float *sm, const Seq &sq, const float *Gsrc, const float *Vcur, int step, int p1, int h1, int f1, int p2, int h2, int f2, unsigned *fetched)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    float *Wc = sm, *S1 = sm + SLOT, *S2 = sm + 2 * SLOT, *S3 = sm + 3 * SLOT;
    int I1, J1, I2, J2;
    rr_pair(sq.nb, step, p1, I1, J1);
    rr_pair(sq.nb, step, p2, I2, J2);
    const int np = sq.np;
    for (int f = tid; f < BLK * (BLK / 4); f += NT) {
        const int i = f >> 4, c = (f & 15) * 4;
        const bool up = i < JB;
        const int row = (up ? h1 : h2) * JB + (i & (JB - 1));
        float4 w;
        if (up ? f1 : f2) w = __ldcg((const float4 *)(Vcur + (size_t)(up ? p1 : p2) * VSTRIDE + row * BLK + c));
        else w = make_float4(row == c ? 1.f : 0.f, row == c + 1 ? 1.f : 0.f, row == c + 2 ? 1.f : 0.f, row == c + 3 ? 1.f : 0.f);
        *(float4 *)(Wc + i * LDA + c) = w;
        const size_t r1 = (size_t)glob_of_loc(I1, J1, i) * np, r2 = (size_t)glob_of_loc(I2, J2, i) * np;
        *(float4 *)(S1 + i * LDB + c) = __ldcg((const float4 *)(Gsrc + r1 + glob_of_loc(I1, J1, c)));
        *(float4 *)(S2 + i * LDB + c) = __ldcg((const float4 *)(Gsrc + r2 + glob_of_loc(I2, J2, c)));
        *(float4 *)(S3 + i * LDB + c) = __ldcg((const float4 *)(Gsrc + r1 + glob_of_loc(I2, J2, c)));
    }
    __syncthreads();
    if (tid == 0) atomicAdd(fetched, 1u);                       // the old blocks are on chip: the update may overwrite them
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    const bool up = m0 < JB;
    float accd[4][4], acco[4][4];
    product64_fma<false>(Wc, up ? S1 : S2, LDB, m0, n0, accd);
    if (up) {
        product64_fma<false>(Wc, S3, LDB, m0, n0, acco);
    }
    __syncthreads();
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int c = n0 + nt * 8 + 2 * t;
        *(float2 *)(S1 + (m0 + g) * LDA + c) = make_float2(accd[nt][0], accd[nt][1]);
        *(float2 *)(S1 + (m0 + g + 8) * LDA + c) = make_float2(accd[nt][2], accd[nt][3]);
        if (up) {
            *(float2 *)(S2 + (m0 + g) * LDA + c) = make_float2(acco[nt][0], acco[nt][1]);
            *(float2 *)(S2 + (m0 + g + 8) * LDA + c) = make_float2(acco[nt][2], acco[nt][3]);
        }
    }
    __syncthreads();
    const bool lower_left = !up && n0 == 0;                     // mirror of the upper right part
    if (!lower_left) {
        const float *Ta = (up && n0 != 0) ? S2 : S1;
        product64_fma<true>(Ta, Wc, LDA, m0, n0, accd);
    }
    __syncthreads();
    float *As = sm;
    if (!lower_left) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = m0 + g + (e >> 1) * 8, j = n0 + nt * 8 + 2 * t + (e & 1);
                As[i * LDP + j] = accd[nt][e];
                if (up && n0 != 0) As[j * LDP + i] = accd[nt][e];
            }
    }
}


// four values as two fp16 parts, kept inside fp16's range (a scaled entry of G beyond 1 is rounding noise of a row whose
// diagonal entry is noise itself)
__device__ __forceinline__ void put4_clamped(__half *tile, int row, int c, float4 v, float4 cs, float rs)
{
    auto k = [&](float x, float s) { return fminf(fmaxf(x * s * rs, -60000.f), 60000.f); };
    hs::put4(tile, row, c, make_float4(k(v.x, cs.x), k(v.y, cs.y), k(v.z, cs.z), k(v.w, cs.w)));
}
__device__ __forceinline__ float4 inv_pow2_4(float4 v) { return make_float4(inv_pow2(v.x), inv_pow2(v.y), inv_pow2(v.z), inv_pow2(v.w)); }
// accumulator of a product, times k, as fp16 parts of the same 64 x 64 tile position
template <int NTILE>
__device__ __forceinline__ void put_acc(__half *tile, int m0, int n0, const float (&acc)[NTILE][4], float k)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NTILE; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float x = fminf(fmaxf(acc[nt][2 * e] * k, -60000.f), 60000.f), y = fminf(fmaxf(acc[nt][2 * e + 1] * k, -60000.f), 60000.f);
            const __half2 hi = __floats2half2_rn(x, y);
            const float2 f = __half22float2(hi);
            __half *dst = tile + (m0 + g + 8 * e) * hs::LDH + n0 + nt * 8 + 2 * t;
            *(__half2 *)dst = hi;
            *(__half2 *)(dst + hs::PLANE) = __floats2half2_rn(x - f.x, y - f.y);
        }
}
// rows of a published transform (64 x 64, high parts then low parts) to a tile; 256 threads
__device__ __forceinline__ void load_parts(__half *tile, const float *src)
{
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int f = threadIdx.x + it * NT, plane = f >> 9, r = (f >> 3) & 63, c = (f & 7) * 8;
        *(uint4 *)(tile + plane * hs::PLANE + r * hs::LDH + c) = __ldcg((const uint4 *)src + f);
    }
}

// The same with the products from fp16 parts. With the scaled transforms and blocks of "published transforms", N is formed
// as diag(s) [V'1 X'11 V'1^T ...] diag(s), s the scales of the 64 rows taken.
__device__ void pivot_form_half(float *sm, const Seq &sq, const float *Gsrc, const float *Vcur, int step, int p1, int h1, int f1, int p2, int h2, int f2, unsigned *fetched)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    __half *Wc = (__half *)sm, *S1 = Wc + 2 * hs::PLANE, *S2 = S1 + 2 * hs::PLANE, *S3 = S2 + 2 * hs::PLANE;
    __shared__ float srow[BLK];
    int I1, J1, I2, J2;
    rr_pair(sq.nb, step, p1, I1, J1);
    rr_pair(sq.nb, step, p2, I2, J2);
    const int np = sq.np;
    const float *P1 = Vcur + (size_t)p1 * VSTRIDE, *P2 = Vcur + (size_t)p2 * VSTRIDE;
    if (tid < BLK) srow[tid] = tid < JB ? __ldcg(P1 + V_S + h1 * JB + tid) : __ldcg(P2 + V_S + h2 * JB + tid - JB);
    const int c = (tid & 15) * 4;
    const float4 c1 = inv_pow2_4(__ldcg((const float4 *)(P1 + V_D + c))), c2 = inv_pow2_4(__ldcg((const float4 *)(P2 + V_D + c)));
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int i = (tid >> 4) + 16 * it;
        const size_t r1 = (size_t)glob_of_loc(I1, J1, i) * np, r2 = (size_t)glob_of_loc(I2, J2, i) * np;
        const float4 x1 = __ldcg((const float4 *)(Gsrc + r1 + glob_of_loc(I1, J1, c)));
        const float4 x2 = __ldcg((const float4 *)(Gsrc + r2 + glob_of_loc(I2, J2, c)));
        const float4 x3 = __ldcg((const float4 *)(Gsrc + r1 + glob_of_loc(I2, J2, c)));
        const float d1 = inv_pow2(__ldcg(P1 + V_D + i)) * G_SCALE, d2 = inv_pow2(__ldcg(P2 + V_D + i)) * G_SCALE;
        const bool up = i < JB;
        const int row = (up ? h1 : h2) * JB + (i & (JB - 1));
        if (up ? f1 : f2) {
            const uint2 *src = (const uint2 *)(up ? P1 : P2) + (row * BLK + c) / 4;
            *(uint2 *)(Wc + i * hs::LDH + c) = __ldcg(src);
            *(uint2 *)(Wc + hs::PLANE + i * hs::LDH + c) = __ldcg(src + BLK * BLK / 4);
        } else
            hs::put4(Wc, i, c, make_float4(row == c ? V_SCALE : 0.f, row == c + 1 ? V_SCALE : 0.f, row == c + 2 ? V_SCALE : 0.f, row == c + 3 ? V_SCALE : 0.f));
        put4_clamped(S1, i, c, x1, c1, d1);
        put4_clamped(S2, i, c, x2, c2, d2);
        put4_clamped(S3, i, c, x3, c2, d1);
    }
    __syncthreads();
    if (tid == 0) atomicAdd(fetched, 1u);                       // the old blocks are on chip: the update may overwrite them
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    const bool up = m0 < JB;
    float accd[4][4] = {}, acco[4][4] = {};
    hs::product64<false, false>(Wc, up ? S1 : S2, m0, n0, accd);
    if (up) hs::product64<false, false>(Wc, S3, m0, n0, acco);
    __syncthreads();
    constexpr float k1 = T_SCALE / (V_SCALE * G_SCALE), k2 = 1.f / (T_SCALE * V_SCALE);
    put_acc(S1, m0, n0, accd, k1);
    if (up) put_acc(S2, m0, n0, acco, k1);
    __syncthreads();
    const bool lower_left = !up && n0 == 0;                     // mirror of the upper right part
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) accd[nt][e] = 0.f;
    if (!lower_left) hs::product64<false, true>((up && n0 != 0) ? S2 : S1, Wc, m0, n0, accd);
    __syncthreads();
    float *As = sm;
    if (!lower_left) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = m0 + g + (e >> 1) * 8, j = n0 + nt * 8 + 2 * t + (e & 1);
                const float v = accd[nt][e] * k2 * srow[i] * srow[j];
                As[i * LDP + j] = v;
                if (up && n0 != 0) As[j * LDP + i] = v;
            }
    }
}

// The same where the current step did the 32 cross rounds only: the diagonal blocks of N are then those of the rotated pivot
// blocks, published with the transforms (or still in G, where the pair was not rotated; store_diagonal writes them to G, so that
// there is one version of them), and W1 X12 W2^T is all that is left
// to form: one block of G to fetch instead of three, a quarter of the arithmetic (10000 -> 6500 cycles of a step at r~ = 1088 in
// bf16, 15500 -> 9000 at r~ = 192 in fp32; jacobi_persistent of one 32768 x 1088 iterate 4730 -> 3740 us). Not for the step after
// a sweep's first one: the 31 rounds inside the blocks give a transform, no blocks, so those are formed from G.
template <bool TENSOR>
__device__ void pivot_form_cross(float *sm, const Seq &sq, const float *Vcur, int step, int b1, int p1, int h1, int f1, int b2, int p2, int h2, int f2, unsigned *fetched)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, np = sq.np;
    __shared__ float srow[BLK];
    int I1, J1, I2, J2;
    rr_pair(sq.nb, step, p1, I1, J1);
    rr_pair(sq.nb, step, p2, I2, J2);
    const float *P1 = Vcur + (size_t)p1 * VSTRIDE, *P2 = Vcur + (size_t)p2 * VSTRIDE;
    float *As = sm;                                              // slot 0; the operands live in the others
    const int c = (tid & 15) * 4;
    float4 x[4], q[2];
#pragma unroll
    for (int it = 0; it < 4; ++it)
        x[it] = __ldcg((const float4 *)(sq.G + (size_t)glob_of_loc(I1, J1, (tid >> 4) + 16 * it) * np + glob_of_loc(I2, J2, c)));
    const int qi = tid >> 3, qc = (tid & 7) * 4;
    q[0] = __ldcg((const float4 *)(f1 ? P1 + V_Q + h1 * JB * JB + qi * JB + qc : sq.G + (size_t)(b1 * JB + qi) * np + b1 * JB + qc));
    q[1] = __ldcg((const float4 *)(f2 ? P2 + V_Q + h2 * JB * JB + qi * JB + qc : sq.G + (size_t)(b2 * JB + qi) * np + b2 * JB + qc));
    if constexpr (TENSOR) {
        __half *Wc = (__half *)(sm + SLOT), *S = (__half *)(sm + 2 * SLOT);
        const float4 cs = inv_pow2_4(__ldcg((const float4 *)(P2 + V_D + c)));
        float d[4];
        uint4 w[4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            d[it] = __ldcg(P1 + V_D + (tid >> 4) + 16 * it);
            const int r = (tid >> 3) + 32 * (it & 1), e = (tid & 7) * 8, row = ((it & 1) ? h2 : h1) * JB + (r & (JB - 1));
            if ((it & 1) ? f2 : f1) w[it] = __ldcg((const uint4 *)(((it & 1) ? P2 : P1) + (it >> 1) * (BLK * BLK / 2) + (row * BLK + e) / 2));
            else {                                               // V_SCALE times the identity (0x7000: 8192 in fp16)
                uint32_t u[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) u[k] = it < 2 && (row - e) >> 1 == k ? ((row & 1) ? 0x70000000u : 0x7000u) : 0u;
                w[it] = make_uint4(u[0], u[1], u[2], u[3]);
            }
        }
        if (tid < BLK) srow[tid] = tid < JB ? __ldcg(P1 + V_S + h1 * JB + tid) : __ldcg(P2 + V_S + h2 * JB + tid - JB);
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            *(uint4 *)(Wc + (it >> 1) * hs::PLANE + ((tid >> 3) + 32 * (it & 1)) * hs::LDH + (tid & 7) * 8) = w[it];
            put4_clamped(S, (tid >> 4) + 16 * it, c, x[it], cs, inv_pow2(d[it]) * G_SCALE);
        }
    } else {
        float *Wc = sm + SLOT, *S = sm + 2 * SLOT;
        float4 w[4];
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int r = (tid >> 4) + 16 * it, row = (it < 2 ? h1 : h2) * JB + (r & (JB - 1));
            if (it < 2 ? f1 : f2) w[it] = __ldcg((const float4 *)((it < 2 ? P1 : P2) + row * BLK + c));
            else w[it] = make_float4(row == c ? 1.f : 0.f, row == c + 1 ? 1.f : 0.f, row == c + 2 ? 1.f : 0.f, row == c + 3 ? 1.f : 0.f);
        }
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            *(float4 *)(Wc + ((tid >> 4) + 16 * it) * LDA + c) = w[it];
            *(float4 *)(S + ((tid >> 4) + 16 * it) * LDB + c) = x[it];
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        float *dst = As + (k * JB + qi) * LDP + k * JB + qc;
        dst[0] = q[k].x; dst[1] = q[k].y; dst[2] = q[k].z; dst[3] = q[k].w;
    }
    __syncthreads();
    if (tid == 0) atomicAdd(fetched, 1u);                       // the old blocks are on chip: the update may overwrite them
    if constexpr (TENSOR) {
        __half *Wc = (__half *)(sm + SLOT), *S = (__half *)(sm + 2 * SLOT), *T = (__half *)(sm + 3 * SLOT);
        const int g = lane >> 2, t = lane & 3;
        {   // T = W1 X12: 32 x 64, a 16 x 16 part per warp
            const int m0 = (warp & 1) * 16, n0 = (warp >> 1) * 16;
            float acc[2][4] = {};
            hs::product16<false>(Wc, S, m0, n0, acc);
            constexpr float k1 = T_SCALE / (V_SCALE * G_SCALE);
            put_acc(T, m0, n0, acc, k1);
        }
        __syncthreads();
        if (warp < 4) {   // T W2^T: 32 x 32
            const int m0 = (warp & 1) * 16, n0 = (warp >> 1) * 16;
            float acc[2][4] = {};
            hs::product16<true>(T, Wc + JB * hs::LDH, m0, n0, acc);
            constexpr float k2 = 1.f / (T_SCALE * V_SCALE);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int i = m0 + g + (e >> 1) * 8, j = JB + n0 + nt * 8 + 2 * t + (e & 1);
                    const float v = acc[nt][e] * k2 * srow[i] * srow[j];
                    As[i * LDP + j] = v;
                    As[j * LDP + i] = v;
                }
        }
    } else {
        const float *Wc = sm + SLOT, *S = sm + 2 * SLOT;
        float *T = sm + 3 * SLOT;
        {   // two rows, four columns a thread
            const int r = (tid >> 4) * 2;
            float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = a0;
#pragma unroll 4
            for (int k = 0; k < BLK; ++k) {
                const float4 b = *(const float4 *)(S + k * LDB + c);
                const float u = Wc[r * LDA + k], v = Wc[(r + 1) * LDA + k];
                a0.x = fmaf(u, b.x, a0.x); a0.y = fmaf(u, b.y, a0.y); a0.z = fmaf(u, b.z, a0.z); a0.w = fmaf(u, b.w, a0.w);
                a1.x = fmaf(v, b.x, a1.x); a1.y = fmaf(v, b.y, a1.y); a1.z = fmaf(v, b.z, a1.z); a1.w = fmaf(v, b.w, a1.w);
            }
            *(float4 *)(T + r * LDA + c) = a0;
            *(float4 *)(T + (r + 1) * LDA + c) = a1;
        }
        __syncthreads();
        const int r = tid >> 3, j0 = tid & 7;                    // columns j0, j0 + 8, ...: rows of W2 without bank conflicts
        float acc[4] = {};
#pragma unroll 4
        for (int k = 0; k < BLK; k += 4) {
            const float4 a = *(const float4 *)(T + r * LDA + k);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 b = *(const float4 *)(Wc + (JB + j0 + 8 * e) * LDA + k);
                acc[e] = fmaf(a.x, b.x, acc[e]); acc[e] = fmaf(a.y, b.y, acc[e]);
                acc[e] = fmaf(a.z, b.z, acc[e]); acc[e] = fmaf(a.w, b.w, acc[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int j = JB + j0 + 8 * e;
            As[r * LDP + j] = acc[e];
            As[j * LDP + r] = acc[e];
        }
    }
}

// The update of a step is cut into items: a block (p, q), p <= q, of G, updated in place together with its mirror, or two
// 64-column chunks of the rows of pair p of Wt, in place. The pivot CTAs of the same step read blocks of G as they were before
// the update: before its first store of a step a CTA makes sure that all of them have fetched theirs (Fetched). Single blocks
// rather than rows of them: at r~ = 2112 a step has about four items for each of 296 CTAs, and the last ones to finish set its
// time (24 us; most of an item is the latency of its loads). The chunks of Wt share Vt_p, and the second one is fetched into
// registers during the product of the first.
constexpr int SEG_W = 2;

__device__ __forceinline__ void store_tile_acc(float *dst, int ld, int m0, int n0, const float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int c = n0 + nt * 8 + 2 * t;
        *(float2 *)(dst + (m0 + g) * ld + c) = make_float2(acc[nt][0], acc[nt][1]);
        *(float2 *)(dst + (m0 + g + 8) * ld + c) = make_float2(acc[nt][2], acc[nt][3]);
    }
}

struct Fetched {
    const unsigned *count; unsigned target; int *abort_flag;   // counter of pivot blocks fetched in this step, its final value
    bool ok;                                                    // already seen complete by this CTA
};
// Block-uniform, bounded: false when the wait ran out.
__device__ bool wait_fetched(Fetched &f)
{
    if (f.ok) return true;
    __shared__ int ok_s;
    if (threadIdx.x == 0) {
        int ok = 0;
        for (unsigned i = 0; i < SPIN_LIMIT; ++i) {
            if (*(volatile const unsigned *)f.count >= f.target) { ok = 1; break; }
            if ((i & 1023u) == 1023u && *(volatile int *)f.abort_flag) break;
        }
        if (!ok) wait_ran_out(f.abort_flag);
        ok_s = ok;
    }
    __syncthreads();
    f.ok = ok_s != 0;
    return f.ok;
}

// The two 32 x 32 diagonal blocks of a rotated pair go to G as its pivot solve left them (published behind the transform, in the
// steps of 32 rounds), not as the products of the item (p, p) give them. The next pivot block is formed from them, so G has to
// hold the same values: computed twice, the two versions of a diagonal block part with every step of a sweep, and where a row's
// diagonal entry is rounding noise (rank-deficient inputs) one may be negative and the other not, which clips good entries of G
// (put4_clamped).
__device__ __forceinline__ void store_diagonal(float *G, int np, int I, int J, const float *P)
{
    const int i = threadIdx.x >> 3, c = (threadIdx.x & 7) * 4;
    const float4 a = __ldcg((const float4 *)(P + V_Q + i * JB + c)), b = __ldcg((const float4 *)(P + V_Q + JB * JB + i * JB + c));
    *(float4 *)(G + (size_t)(I * JB + i) * np + I * JB + c) = a;
    *(float4 *)(G + (size_t)(J * JB + i) * np + J * JB + c) = b;
}

// A fragment of an updated block of G (rows gr0, gr1; columns gc, gc + 1) goes out with its mirror. Of a block (p, p) only what
// lies on and above the diagonal does: computed both ways, the two triangles differ by rounding, and a rotation, which reads one
// of them, never takes away the difference.
__device__ __forceinline__ void store_mirrored(float *G, int np, int gr0, int gr1, int gc, float v0, float v1, float v2, float v3)
{
    *(float2 *)(G + (size_t)gr0 * np + gc) = make_float2(v0, v1);
    *(float2 *)(G + (size_t)gr1 * np + gc) = make_float2(v2, v3);
    G[(size_t)gc * np + gr0] = v0; G[(size_t)(gc + 1) * np + gr0] = v1;
    G[(size_t)gc * np + gr1] = v2; G[(size_t)(gc + 1) * np + gr1] = v3;
}
__device__ __forceinline__ void store_upper(float *G, int np, int gr0, int gr1, int gc, float v0, float v1, float v2, float v3)
{
    auto put = [&](int r, int c, float v) { if (r <= c) { G[(size_t)r * np + c] = v; G[(size_t)c * np + r] = v; } };
    put(gr0, gc, v0); put(gr0, gc + 1, v1); put(gr1, gc, v2); put(gr1, gc + 1, v3);
}
// 0: this warp (rows m0 .., columns n0 .. of the block) stores nothing, 1: the triangle on and above the diagonal, 2: all, mirrored.
__device__ __forceinline__ int part_stored(bool diagonal, bool carried, int m0, int n0)
{
    const bool same_half = !((m0 ^ n0) & JB);
    if (!diagonal) return 2;
    return same_half ? (carried ? 0 : 1) : m0 < n0 ? 2 : 0;
}

// One block (p, q) of G on the fp32 units: Vt_p G_pq Vt_q^T.
__device__ bool g_block(float *sm, const Seq &sq, float *G, const float *Vbuf, const int *vflag, int step, int p, int q, Fetched &fetched)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32, np = sq.np;
    float *Vp = sm, *Vq = sm + BLK * LDA, *Tm = sm + 2 * BLK * LDA, *Bk = sm + 3 * BLK * LDA;
    const int fp = vflag[p], fq = vflag[q];
    if (!fp && !fq) return true;                                 // unchanged block
    int Ip, Jp, Iq, Jq;
    rr_pair(sq.nb, step, p, Ip, Jp);
    rr_pair(sq.nb, step, q, Iq, Jq);
    // the block goes to the B tile when a row transform comes first, else straight to the T tile
    float *blk_dst = fp ? Bk : Tm;
    const int blk_ld = fp ? LDB : LDA;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int f = tid + it * NT, i = f >> 4, c = (f & 15) * 4;
        *(float4 *)(blk_dst + i * blk_ld + c) = __ldcg((const float4 *)(G + (size_t)glob_of_loc(Ip, Jp, i) * np + glob_of_loc(Iq, Jq, c)));
        if (fp) *(float4 *)(Vp + i * LDA + c) = __ldcg((const float4 *)(Vbuf + (size_t)p * VSTRIDE + i * BLK + c));
        if (fq) *(float4 *)(Vq + i * LDA + c) = __ldcg((const float4 *)(Vbuf + (size_t)q * VSTRIDE + i * BLK + c));
    }
    __syncthreads();
    float acc[4][4];
    if (fp) {
        product64_fma<false>(Vp, Bk, LDB, m0, n0, acc);
        if (fq) {
            store_tile_acc(Tm, LDA, m0, n0, acc);
            __syncthreads();
        }
    }
    if (fq) product64_fma<true>(Tm, Vq, LDA, m0, n0, acc);       // out = T * Vt_q^T
    if (!wait_fetched(fetched)) return false;
    const bool carried = p == q && step > 0;                     // the diagonal blocks come from the pivot solve
    if (carried) store_diagonal(G, np, Ip, Jp, Vbuf + (size_t)p * VSTRIDE);
    const int gr0 = glob_of_loc(Ip, Jp, m0 + g), gr1 = glob_of_loc(Ip, Jp, m0 + g + 8);
    const int part = part_stored(p == q, carried, m0, n0);
    if (part)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int gc = glob_of_loc(Iq, Jq, n0 + nt * 8 + 2 * t);     // gc, gc + 1 are contiguous
            if (part == 2) store_mirrored(G, np, gr0, gr1, gc, acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
            else store_upper(G, np, gr0, gr1, gc, acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
        }
    __syncthreads();                                             // tiles are reused by the next block
    return true;
}

__device__ void wt_strip(float *sm, const Seq &sq, const float *Vbuf, const int *vflag, int step, int p, int c0, int cnt)
{
    if (!vflag[p]) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32, np = sq.np;
    float *Vp = sm, *Bk = sm + 3 * BLK * LDA;
    int Ip, Jp;
    rr_pair(sq.nb, step, p, Ip, Jp);
    float4 x[4];
    auto fetch = [&](int chunk) {
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int f = tid + it * NT, i = f >> 4, c = (f & 15) * 4;
            x[it] = __ldcg((const float4 *)(sq.Wt + (size_t)glob_of_loc(Ip, Jp, i) * np + chunk * BLK + c));
        }
    };
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int f = tid + it * NT, i = f >> 4, c = (f & 15) * 4;
        *(float4 *)(Vp + i * LDA + c) = __ldcg((const float4 *)(Vbuf + (size_t)p * VSTRIDE + i * BLK + c));
    }
    fetch(c0);
    const int gr0 = glob_of_loc(Ip, Jp, m0 + g), gr1 = glob_of_loc(Ip, Jp, m0 + g + 8);
    for (int j = 0; j < cnt; ++j) {
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int f = tid + it * NT, i = f >> 4, c = (f & 15) * 4;
            *(float4 *)(Bk + i * LDB + c) = x[it];
        }
        __syncthreads();
        if (j + 1 < cnt) fetch(c0 + j + 1);
        float acc[4][4];
        product64_fma<false>(Vp, Bk, LDB, m0, n0, acc);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int gc = (c0 + j) * BLK + n0 + nt * 8 + 2 * t;
            *(float2 *)(sq.Wt + (size_t)gr0 * np + gc) = make_float2(acc[nt][0], acc[nt][1]);
            *(float2 *)(sq.Wt + (size_t)gr1 * np + gc) = make_float2(acc[nt][2], acc[nt][3]);
        }
        __syncthreads();                                         // the B tile is reused by the next chunk
    }
}

// One block (p, q) of G, products from fp16 parts: with V' and the scaled block G' of "published transforms",
//   G_pq <- diag(s_p) V'_p G' V'_q^T diag(s_q)     (V' the identity and s = d for a pair that was not rotated).
__device__ bool g_block_half(float *sm, const Seq &sq, float *G, const float *Vbuf, const int *vflag, int step, int p, int q, Fetched &fetched)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32, np = sq.np;
    __half *Vp = (__half *)sm, *Vq = Vp + 2 * hs::PLANE, *Bk = Vq + 2 * hs::PLANE;
    __shared__ float sp[BLK], sqv[BLK];
    const int fp = vflag[p], fq = vflag[q];
    if (!fp && !fq) return true;                                 // unchanged block
    int Ip, Jp, Iq, Jq;
    rr_pair(sq.nb, step, p, Ip, Jp);
    rr_pair(sq.nb, step, q, Iq, Jq);
    const float *Pp = Vbuf + (size_t)p * VSTRIDE, *Pq = Vbuf + (size_t)q * VSTRIDE;
    const int c = (tid & 15) * 4;
    float4 x[4];
    float d[4];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int i = (tid >> 4) + 16 * it;
        x[it] = __ldcg((const float4 *)(G + (size_t)glob_of_loc(Ip, Jp, i) * np + glob_of_loc(Iq, Jq, c)));
        d[it] = __ldcg(Pp + V_D + i);
    }
    const float4 cs = inv_pow2_4(__ldcg((const float4 *)(Pq + V_D + c)));
    if (tid < BLK) sp[tid] = __ldcg(Pp + V_S + tid);
    else if (tid < 2 * BLK) sqv[tid - BLK] = __ldcg(Pq + V_S + tid - BLK);
    if (fp) load_parts(Vp, Pp);
    if (fq) load_parts(Vq, Pq);
#pragma unroll
    for (int it = 0; it < 4; ++it) put4_clamped(Bk, (tid >> 4) + 16 * it, c, x[it], cs, inv_pow2(d[it]) * G_SCALE);
    __syncthreads();
    float acc[4][4] = {};
    float k = 1.f / (V_SCALE * G_SCALE);
    if (fp) hs::product64<false, false>(Vp, Bk, m0, n0, acc);
    if (fq) {
        if (fp) {
            __syncthreads();
            put_acc(Bk, m0, n0, acc, T_SCALE * k);
            __syncthreads();
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[nt][e] = 0.f;
            k = 1.f / (V_SCALE * T_SCALE);
        }
        hs::product64<false, true>(Bk, Vq, m0, n0, acc);
    }
    if (!wait_fetched(fetched)) return false;
    const bool carried = p == q && step > 0;                     // the diagonal blocks come from the pivot solve
    if (carried) store_diagonal(G, np, Ip, Jp, Pp);
    const int gr0 = glob_of_loc(Ip, Jp, m0 + g), gr1 = glob_of_loc(Ip, Jp, m0 + g + 8);
    const float s0 = sp[m0 + g] * k, s1 = sp[m0 + g + 8] * k;
    const int part = part_stored(p == q, carried, m0, n0);
    if (part)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int lc = n0 + nt * 8 + 2 * t, gc = glob_of_loc(Iq, Jq, lc);    // gc, gc + 1 are contiguous
            const float q0 = sqv[lc], q1 = sqv[lc + 1];
            const float v0 = acc[nt][0] * s0 * q0, v1 = acc[nt][1] * s0 * q1, v2 = acc[nt][2] * s1 * q0, v3 = acc[nt][3] * s1 * q1;
            if (part == 2) store_mirrored(G, np, gr0, gr1, gc, v0, v1, v2, v3);
            else store_upper(G, np, gr0, gr1, gc, v0, v1, v2, v3);
        }
    __syncthreads();                                             // tiles are reused by the next block
    return true;
}

// Column chunks c0 .. c0 + cnt - 1 of the rows of pair p of Wt, products from fp16 parts.
__device__ void wt_strip_half(float *sm, const Seq &sq, const float *Vbuf, const int *vflag, int step, int p, int c0, int cnt)
{
    if (!vflag[p]) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32, np = sq.np;
    __half *Vp = (__half *)sm, *Bk = Vp + 2 * hs::PLANE;
    int Ip, Jp;
    rr_pair(sq.nb, step, p, Ip, Jp);
    float4 x[4];
    auto fetch = [&](int chunk) {
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int f = tid + it * NT, i = f >> 4, c = (f & 15) * 4;
            x[it] = __ldcg((const float4 *)(sq.Wt + (size_t)glob_of_loc(Ip, Jp, i) * np + chunk * BLK + c));
        }
    };
    fetch(c0);
    load_parts(Vp, Vbuf + (size_t)p * VSTRIDE + V_VU);
    const int gr0 = glob_of_loc(Ip, Jp, m0 + g), gr1 = glob_of_loc(Ip, Jp, m0 + g + 8);
    for (int j = 0; j < cnt; ++j) {
        __half *B = Bk + (j & 1) * 2 * hs::PLANE;                // two tiles: one barrier per chunk
#pragma unroll
        for (int it = 0; it < 4; ++it) {
            const int f = tid + it * NT;
            hs::put4(B, f >> 4, (f & 15) * 4, make_float4(x[it].x * V_SCALE, x[it].y * V_SCALE, x[it].z * V_SCALE, x[it].w * V_SCALE));
        }
        __syncthreads();
        if (j + 1 < cnt) fetch(c0 + j + 1);
        float acc[4][4] = {};
        hs::product64<false, false>(Vp, B, m0, n0, acc);
        constexpr float k = 1.f / (V_SCALE * V_SCALE);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int gc = (c0 + j) * BLK + n0 + nt * 8 + 2 * t;
            *(float2 *)(sq.Wt + (size_t)gr0 * np + gc) = make_float2(acc[nt][0] * k, acc[nt][1] * k);
            *(float2 *)(sq.Wt + (size_t)gr1 * np + gc) = make_float2(acc[nt][2] * k, acc[nt][3] * k);
        }
    }
    __syncthreads();
}

// Work items of the update: first the blocks of G (row by row of the upper triangle), then the chunks of Wt.
__host__ __device__ __forceinline__ int blocks_of_g(int npairs) { return npairs * (npairs + 1) / 2; }
template <bool TENSOR>
__device__ bool apply_item(float *sm, const Seq &sq, const float *Vbuf, const int *vflag, int step, int idx, int npairs, int items_g, int nw, Fetched &fetched)
{
    if (idx < items_g) {
        int p = 0;
        while (idx >= npairs - p) { idx -= npairs - p; ++p; }
        return TENSOR ? g_block_half(sm, sq, sq.G, Vbuf, vflag, step, p, p + idx, fetched) : g_block(sm, sq, sq.G, Vbuf, vflag, step, p, p + idx, fetched);
    }
    idx -= items_g;
    const int nseg = (nw + SEG_W - 1) / SEG_W, p = idx / nseg, c0 = (idx - p * nseg) * SEG_W;
    if (TENSOR) wt_strip_half(sm, sq, Vbuf, vflag, step, p, c0, min(SEG_W, nw - c0));
    else wt_strip(sm, sq, Vbuf, vflag, step, p, c0, min(SEG_W, nw - c0));
    return true;
}

// ---- the kernel --------------------------------------------------------------------------------
// Schedule of a group. The pivot block of a pair of step s+1 is a function of the matrix before the update of
// step s and of two pivot solves of step s (pivot_form, pivot_form_cross), all of which are complete at the barrier
// that ends step s-1. Every step therefore runs, side by side,
//   1. the pivot solves of the NEXT step (a few CTAs; this chain of rotation rounds is the critical path), and
//   2. the update of this step, its blocks handed out by a ticket counter so that the pivot CTAs join in when
//      they are through,
// followed by one group barrier. The update works in place; before its first store of a step a CTA waits
// (as a rule not at all: it has a block to load and multiply first) until every pivot CTA has fetched the
// blocks it forms its pivot block from. Vt and the rotated-flags are double buffered by step parity, because
// the pivots of step s+1 publish while the update of step s still reads.
// status[0]: sticky device status word of the context; status[1]: abort flag of bounded waits.
constexpr int MAXPAIRS = 72;                  // np <= 4608

// Number of this CTA in the order in which roles are given out: pivot solves go to CTAs on SMs of their own (two of them on one
// SM, or one beside a CTA of the update, take 13000 cycles for their 32 rounds instead of 9400, and blocks that follow one
// another do share an SM). First come the CTAs with the lowest block number of their SM, then the second CTAs of the SMs without
// a pivot, last those beside a pivot; numbers that no sequence uses leave the kernel. -1: the wait for the other CTAs ran out.
constexpr int MAXGRID = 1024;
__device__ int seat_of(const Batch &batch, int *abort_flag)
{
    __shared__ int first[MAXGRID];
    __shared__ unsigned prim[MAXGRID / 32], away[MAXGRID / 32], beside[MAXGRID / 32];
    const int tid = threadIdx.x, n = (int)gridDim.x, n32 = (n + 31) & ~31;
    unsigned sm;
    asm("mov.u32 %0, %%smid;" : "=r"(sm));
    if (tid == 0) batch.smids[blockIdx.x] = sm;
    for (int i = tid; i < MAXGRID; i += NT) first[i] = n;
    if (!group_barrier(batch.grid_sync, 1u, (unsigned)n, abort_flag)) return -1;
    auto sm_of = [&](int b) { return (int)(__ldcg(batch.smids + b) % MAXGRID); };
    auto below = [](const unsigned *mask, int b) {               // bits set below b
        int c = __popc(mask[b >> 5] & ((1u << (b & 31)) - 1u));
        for (int k = 0; k < b >> 5; ++k) c += __popc(mask[k]);
        return c;
    };
    for (int b = tid; b < n; b += NT) atomicMin(&first[sm_of(b)], b);
    __syncthreads();
    for (int b = tid; b < n32; b += NT) {
        const unsigned m = __ballot_sync(0xffffffffu, b < n && first[sm_of(b)] == b);
        if ((tid & 31) == 0) prim[b >> 5] = m;
    }
    __syncthreads();
    for (int b = tid; b < n32; b += NT) {
        const bool second = b < n && !(prim[b >> 5] >> (b & 31) & 1u), near = second && below(prim, first[sm_of(b)]) < batch.pivots;
        const unsigned m = __ballot_sync(0xffffffffu, second && !near), m2 = __ballot_sync(0xffffffffu, near);
        if ((tid & 31) == 0) { away[b >> 5] = m; beside[b >> 5] = m2; }
    }
    __syncthreads();
    const int b = (int)blockIdx.x;
    int seat = below(prim, b);
    if (!(prim[b >> 5] >> (b & 31) & 1u)) {
        const bool far = away[b >> 5] >> (b & 31) & 1u;
        int before = 0;                                          // all the CTAs of the classes before
        for (int k = 0; k < n32 / 32; ++k) before += __popc(prim[k]) + (far ? 0 : __popc(away[k]));
        seat = before + below(far ? away : beside, b);
    }
    __syncthreads();
    return seat;
}

// This CTA's share (rows rank, rank + ncta, ...) of the largest |g_ij| / sqrt(g_ii g_jj), i < j, negligible rows left out.
// rs: np floats of shared memory.
__device__ float matrix_max(float *rs, const Seq &sq, int rank, float least)
{
    __shared__ float part[NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = sq.n, np = sq.np;
#pragma unroll 4
    for (int i = tid; i < np; i += NT) {
        const float d = i < n ? __ldcg(sq.G + (size_t)i * np + i) : 0.f;
        rs[i] = d > least ? rsqrtf(d) : 0.f;
    }
    __syncthreads();
    float mo = 0.f;
    for (int i = rank * (NT / 32) + warp; i < n; i += sq.ncta * (NT / 32)) {
        const float *row = sq.G + (size_t)i * np;
        float m = 0.f;
#pragma unroll 4
        for (int j = (i & ~127) + lane * 4; j < n; j += 128) {
            const float4 g = __ldcg((const float4 *)(row + j)), r = *(const float4 *)(rs + j);
            m = fmaxf(m, fmaxf(j > i ? fabsf(g.x) * r.x : 0.f, j + 1 > i ? fabsf(g.y) * r.y : 0.f));
            m = fmaxf(m, fmaxf(j + 2 > i ? fabsf(g.z) * r.z : 0.f, j + 3 > i ? fabsf(g.w) * r.w : 0.f));
        }
        mo = fmaxf(mo, m * rs[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mo = fmaxf(mo, __shfl_xor_sync(0xffffffffu, mo, o));
    if (lane == 0) part[warp] = mo;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) mo = fmaxf(mo, part[w]);
    return mo;
}

template <bool TENSOR>
__global__ void __launch_bounds__(NT, 2)
jacobi_persistent_kernel(const __grid_constant__ Batch batch, float tol_conv, float tol_left, float tol_rot, int max_sweeps,
                         int raise_not_converged, int *status)
{
    extern __shared__ __align__(16) float j3sm[];
    __shared__ int flag_s[MAXPAIRS];              // the pairs rotated in the current step
    __shared__ int ticket_s;
    int si = -1, rank = 0;
    const int seat = batch.seated ? seat_of(batch, status + 1) : (int)blockIdx.x;
    if (seat < 0) return;
#pragma unroll 1
    for (int i = 0; i < batch.count; ++i) {                      // pivot CTAs are the first ones of their sequence
        const int p = seat - batch.s[i].pivot0, w = seat - batch.s[i].worker0, npu = batch.s[i].npu;
        if (p >= 0 && p < npu) { si = i; rank = p; }
        else if (w >= 0 && w < batch.s[i].ncta - npu) { si = i; rank = npu + w; }
    }
    if (si < 0) return;
    const Seq &sq = batch.s[si];
    const int tid = threadIdx.x;
    if (sq.np <= 0) return;
    const int npairs = sq.nb / 2, nw = sq.np / BLK;
    const int items_g = blocks_of_g(npairs), total = items_g + npairs * ((nw + SEG_W - 1) / SEG_W);
    const int nsteps = sq.nb - 1;
    int *abort_flag = status + 1;
    unsigned gen = 0, gstep = 0;
    bool converged = false, alive = true;
    const float least = __uint_as_float(__ldcg(sq.sync + 6)) * NEGLIGIBLE;

    // rotates the block held in shared memory for pair pr of (sweep, step); publishes to parity par
    auto pivot_finish = [&](int sweep, int step, int pr, int par) {
        bool rotated;
        const float mo = pivot_rotate<TENSOR>(j3sm, step > 0, tol_rot, least, sq.Vbuf + ((size_t)par * npairs + pr) * VSTRIDE, rotated);
        if (tid == 0) {
            sq.vflag[par * npairs + pr] = rotated ? 1 : 0;
            atomicMax(sq.sync + 1 + sweep % 4, __float_as_uint(mo));
        }
        __syncthreads();
    };

    // prologue: the pivots of the very first step, straight from G
    for (int pr = rank; pr < npairs; pr += sq.ncta) {
        int I, J;
        rr_pair(sq.nb, 0, pr, I, J);
        pivot_load(j3sm, sq.G, sq.np, I, J);
        pivot_finish(0, 0, pr, 0);
    }
    alive = group_barrier(sq.sync, ++gen, (unsigned)sq.ncta, abort_flag);

    int sweep = 0;
    for (; sweep < max_sweeps && alive; ++sweep) {
        if (rank == 0 && tid == 0) sq.sync[1 + (sweep + 2) % 4] = sq.sync[8 + (sweep + 2) % 4] = 0u;   // slots of sweep + 2, last read two sweeps ago
        for (int step = 0; step < nsteps && alive; ++step, ++gstep) {
            const int par = (int)(gstep & 1u);
            const bool has_next = !(sweep == max_sweeps - 1 && step == nsteps - 1);
            const int nstep = step + 1 == nsteps ? 0 : step + 1, nsweep = sweep + (step + 1 == nsteps ? 1 : 0);
            const float *Vcur = sq.Vbuf + (size_t)par * npairs * VSTRIDE;
            const int *fcur = sq.vflag + par * npairs;
            // a step in which no pair was rotated needs no update (the flags are read once: an L2 round trip per use otherwise)
            const int my_flag = tid < npairs ? __ldcg(fcur + tid) : 0;
            if (tid < npairs) flag_s[tid] = my_flag;
            const bool any_rot = __syncthreads_or(my_flag != 0) != 0;
            if (rank == 0 && tid == 0) {                                  // tickets and fetch count of the next step
                sq.sync[16 + (par ^ 1)] = 0u;
                sq.sync[20 + (par ^ 1)] = 0u;
            }
            Fetched fetched{sq.sync + 20 + par, has_next ? (unsigned)npairs : 0u, abort_flag, false};
            // 1. pivots of the next step
            if (has_next && rank < npairs) {
                for (int pr = rank; pr < npairs; pr += sq.ncta) {
                    int b1, b2, p1, h1, p2, h2;
                    rr_pair(sq.nb, nstep, pr, b1, b2);
                    rr_locate(sq.nb, step, b1, p1, h1);
                    rr_locate(sq.nb, step, b2, p2, h2);
                    const int f1 = flag_s[p1], f2 = flag_s[p2];
                    if (!f1 && !f2) {
                        pivot_load(j3sm, sq.G, sq.np, b1, b2);
                        __syncthreads();
                        if (tid == 0) atomicAdd(sq.sync + 20 + par, 1u);
                    } else if (step > 0) pivot_form_cross<TENSOR>(j3sm, sq, Vcur, step, b1, p1, h1, f1, b2, p2, h2, f2, sq.sync + 20 + par);
                    else if (TENSOR) pivot_form_half(j3sm, sq, sq.G, Vcur, step, p1, h1, f1, p2, h2, f2, sq.sync + 20 + par);
                    else pivot_form(j3sm, sq, sq.G, Vcur, step, p1, h1, f1, p2, h2, f2, sq.sync + 20 + par);
                    pivot_finish(nsweep, nstep, pr, par ^ 1);
                }
            }
            // 2. the update: the CTAs without a pivot take the first items by rank, everything else goes by tickets (the next
            // one is requested while a block is processed)
            const int fixed = has_next ? max(sq.ncta - npairs, 0) : sq.ncta, mine = has_next ? rank - npairs : rank;
            int t = total;
            if (any_rot && mine >= 0) t = mine;
            else if (any_rot) {
                if (tid == 0) ticket_s = fixed + (int)atomicAdd(sq.sync + 16 + par, 1u);
                __syncthreads();
                t = ticket_s;
            }
            while (t < total && alive) {
                int tn = 0;
                if (tid == 0) tn = fixed + (int)atomicAdd(sq.sync + 16 + par, 1u);
                alive = apply_item<TENSOR>(j3sm, sq, Vcur, flag_s, step, t, npairs, items_g, nw, fetched);
                __syncthreads();
                if (tid == 0) ticket_s = tn;
                __syncthreads();
                t = ticket_s;
            }
            alive = group_barrier(sq.sync, ++gen, (unsigned)sq.ncta, abort_flag) && alive;
        }
        if (!alive) break;
        const float mo = __uint_as_float(*(volatile unsigned *)(sq.sync + 1 + sweep % 4));
        if (mo <= tol_conv) { converged = true; ++sweep; break; }
        // The largest scaled off-diagonal entry of the matrix as the sweep has left it: a few microseconds, against a whole
        // sweep (65 steps at n = 2112) to find the same by visiting every pair again.
        const float left = matrix_max(j3sm, sq, rank, least);
        if (tid == 0) atomicMax(sq.sync + 8 + sweep % 4, __float_as_uint(left));
        alive = group_barrier(sq.sync, ++gen, (unsigned)sq.ncta, abort_flag);
        if (!alive) break;
        if (__uint_as_float(*(volatile unsigned *)(sq.sync + 8 + sweep % 4)) <= tol_left) { converged = true; ++sweep; break; }
    }
    if (rank == 0 && tid == 0) {
        if (alive && !converged && raise_not_converged) raise_status(status, ATP_ERR_NOT_CONVERGED);
        sq.sync[5] = (unsigned)sweep;
    }
}

// Wt = identity, padding of G = 0, synchronisation words = 0 but for the largest diagonal entry; a non-finite entry of G (an
// input with Inf / NaN, or one whose squares overflow fp32) raises ATP_ERR_RANGE. grid (x, count).
__global__ void init_kernel(const __grid_constant__ Batch batch, int *status)
{
    bool bad = false;
    const Seq &sq = batch.s[blockIdx.y];
    const size_t n2 = (size_t)sq.np * sq.np;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n2; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / sq.np), j = (int)(e - (size_t)i * sq.np);
        sq.Wt[e] = (i == j) ? 1.f : 0.f;
        if (i >= sq.n || j >= sq.n) sq.G[e] = 0.f;
        else if (!isfinite(sq.G[e])) bad = true;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) raise_status(status, ATP_ERR_RANGE);
    if (blockIdx.x == 0) {
        __shared__ unsigned top;
        if (threadIdx.x == 0) top = 0u;
        __syncthreads();
        float m = 0.f;
        for (int i = threadIdx.x; i < sq.n; i += blockDim.x) m = fmaxf(m, sq.G[(size_t)i * (sq.np + 1)]);
        atomicMax(&top, __float_as_uint(m));
        __syncthreads();
        if (threadIdx.x < SYNC_WORDS) sq.sync[threadIdx.x] = threadIdx.x == 6 ? top : 0u;
    }
}

// Host side: gives every sequence its group of CTAs and launches the kernel cooperatively, so that all groups are resident
// together and the group barriers cannot starve. Up to as many pairs of blocks as SMs a sequence gets a CTA for each of its pairs
// and shares the rest with the others in proportion to the items of their updates (at most one an item); beyond, all CTAs are
// shared by size, at least one to a sequence. An empty sequence gets none.
// The CTAs beside the pivots stay away (seat_of) as long as the others have at most MATE_ITEMS items each. The rotation of one
// iterate with r~ = 768: 1886 us, 2358 without seats; 1088: 3250, 3810; 1408, the largest below the line: 4694, 5311; 1472, the
// first above: 5585 without, 5678 with; 1792: 8692, 9368. Three iterates of 576: 1575, 1884; 8 of 320: 916, 1008; 16 of 320, above:
// 1130, 1260. (12 of 320, above as well, would be 3 % faster with seats.) Up to as many CTAs as SMs there is nothing to seat.
constexpr int MATE_ITEMS = 2;
template <bool TENSOR>
static inline atp_status launch(atp_ctx *ctx, Batch &jb, float tol_conv, float tol_left, float tol_rot, int max_sweeps, bool raise_not_converged)
{
    if (jb.count <= 0) return ATP_OK;
    static std::mutex mu;
    static int occ_dev[64] = {};
    int occ = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        const int dv = ctx->device;
        if (dv < 0 || dv >= 64 || occ_dev[dv] == 0) {
            ATP_CUDA_OK(ctx, cudaFuncSetAttribute(jacobi_persistent_kernel<TENSOR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
            ATP_CUDA_OK(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, jacobi_persistent_kernel<TENSOR>, NT, SMEM_BYTES));
            if (occ < 1) return ATP_ERR_CUDA;
            if (dv >= 0 && dv < 64) occ_dev[dv] = occ;
        } else occ = occ_dev[dv];
    }
    const int per_sm = std::min(occ, 2), total = ctx->sm_count * per_sm;
    double wsum = 0;
    int pairs = 0, all_items = 0, items[MAXSEQ];
    for (int i = 0; i < jb.count; ++i) {
        const Seq &q = jb.s[i];
        const int npairs = q.nb / 2;
        wsum += (double)q.np * q.np;
        pairs += npairs;
        items[i] = q.np > 0 ? blocks_of_g(npairs) + npairs * ((q.np / BLK + SEG_W - 1) / SEG_W) : 0;     // of the update
        all_items += items[i];
    }
    if (wsum <= 0) return ATP_OK;
    const bool own = pairs <= ctx->sm_count;
    auto share = [&](int workers, int i) { return (int)std::min<double>(items[i], (double)workers * items[i] / all_items); };
    bool apart = own && per_sm == 2;
    for (int i = 0; i < jb.count; ++i) apart = apart && items[i] <= MATE_ITEMS * share(total - 2 * pairs, i);
    int used = 0;
    jb.pivots = 0;
    for (int i = 0; i < jb.count; ++i) {
        Seq &q = jb.s[i];
        const int npairs = q.nb / 2;
        if (own) { q.npu = npairs; q.ncta = npairs + share(total - (apart ? 2 : 1) * pairs, i); }
        else {
            q.ncta = 1 + (int)std::min<double>(items[i], (total - jb.count) * ((double)q.np * q.np / wsum));      // (at most `total` together)
            q.npu = std::min(npairs, q.ncta);
        }
        if (q.np <= 0) q.npu = q.ncta = 0;
        q.pivot0 = jb.pivots;
        jb.pivots += q.npu;
        used += q.ncta;
    }
    for (int i = 0, next = jb.pivots; i < jb.count; ++i) {
        jb.s[i].worker0 = next;
        next += jb.s[i].ncta - jb.s[i].npu;
    }
    jb.seated = apart && used > ctx->sm_count && total <= MAXGRID;
    const int grid = jb.seated ? total : used;
    jb.grid_sync = jb.s[0].sync + 32;
    jb.smids = jb.s[0].sync + SYNC_WORDS;
    ATP_KERNEL(ctx, "jacobi_init", 0, wsum * 4.0);
    init_kernel<<<dim3(std::max(64, 4 * ctx->sm_count / jb.count), jb.count), 256, 0, ctx->stream>>>(jb, ctx->dev_status);
    ATP_LAUNCHED(ctx);
    int *status = ctx->dev_status;
    int ms = max_sweeps, rn = raise_not_converged ? 1 : 0;
    void *args[] = {(void *)&jb, (void *)&tol_conv, (void *)&tol_left, (void *)&tol_rot, (void *)&ms, (void *)&rn, (void *)&status};
    // bytes: one read and one write of G and Wt (what the kernel must move at least; it runs from L2)
    ATP_KERNEL(ctx, "jacobi_persistent", 0, wsum * 16.0);
    ATP_CUDA_OK(ctx, cudaLaunchCooperativeKernel((const void *)jacobi_persistent_kernel<TENSOR>, dim3(grid), dim3(NT), args, SMEM_BYTES, ctx->stream));
    ATP_LAUNCHED(ctx);
    return ATP_OK;
}

}  // namespace j3
