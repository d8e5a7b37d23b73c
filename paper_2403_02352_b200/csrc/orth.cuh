// Persistent block Gram-Schmidt: orthonormalises the columns of the range-finder iterates (Sec. 4.2:
// the basis U must satisfy U^T U = I) for every sequence of a batch in ONE cooperative launch.
//
// Panels of 64 columns, left to right; every panel runs `reps` times through
//   project   C = Q^T P against the finished columns Q (split over row ranges, partials summed in a fixed order)
//   update    P <- P - Q C
//   Gram      S = P^T P accumulated in fp64, scaled, Cholesky-factored and inverted in fp64 (panel_chol.cuh); from the
//             second repetition on, when S is within 5e-3 of the identity, the factor comes from a three-term series
//   apply     P <- P (D^-1 L^-T); columns found dependent are replaced by hash noise, which the next
//             repetition orthonormalises
// With two repetitions (what the extraction asks for) the passes are reordered so that the second projection runs
// beside the single-CTA factorisation of the first repetition and the first apply folds into the second Gram
// pass; see the panel program in the kernel.
// Two repetitions give orthonormality to working precision (the second also repairs the explicit inverse,
// which is only norm-wise stable). Each sequence owns a group of CTAs; the phases of a panel are separated by
// the group's barrier (bounded spin) instead of kernel boundaries, and every phase is a list
// of independent 64 x 64 tile jobs dealt out round-robin. The tile products of the projections (most of the arithmetic) run on
// the tensor cores from two fp16 parts per operand (split_mma.cuh), columns of the panel scaled by powers of two to a
// common range. The finished columns are kept as such parts: their tiles go to shared memory by cp.async, without a
// conversion, two of them for every tile of the panel (or of C), which is fetched and cut once for two products (from fp32
// tiles, one product per pair of fetched and cut tiles, 32768 x 1088 took 4920 us instead of 3710). The products
// with the factor run the same way: the panel's columns scaled as before, the factor's rows by the inverse and all of it to
// its largest entry. Plain TF32 is not enough even for the first repetition, because what a projection leaves of an
// ill-conditioned panel is far below 2^-11 of the panel.
// fp32 inputs keep every product on the fp32 units.
#pragma once
#include "jacobi3.cuh"
#include "panel_chol.cuh"
#include "split_mma.cuh"

namespace orth {

using j3::BLK; using j3::NT; using j3::LDA; using j3::LDB;
constexpr int MAXSEQ = 32;
constexpr int SYNC_WORDS = 256;   // words of Seq::sync before the SM list
constexpr int EXTRA = 6;          // repetitions of a panel beyond those asked for
// Length outside the finished columns and those before it in the panel at which a unit column that has been projected and factored
// `tries` times is given up: 1e-5, like a column whose pivot says so, then more, because what is new keeps its length once it has
// been projected. Where a panel has no other direction to offer (rows of zeros, rows repeated: all columns lie in the same few
// dimensions) every projection leaves the rounding of the one before, and normalising that gave U^T U - I of up to the number of
// panels.
constexpr float lost_length(int tries) { return tries <= 0 ? 0.f : tries == 1 ? 1e-5f : tries == 2 ? 1e-3f : 0.1f; }
constexpr int NRED = 8;           // second-level partial Gram sums (chunk ranges)

struct Seq {
    float *M; int n, rt, ld;                  // the iterate: n x rt, fp32, leading dimension ld
    __nv_bfloat16 *hi, *lo; int ldh;          // nullable: the finished columns also go out as a bf16 hi/lo pair
    __half *qh, *ql; int ldq;                 // bf16 inputs: the finished columns times QSCALE as two fp16 parts, n x ldq
    float *Cpart, *C, *Dpart, *W;             // tile scratch (see scratch_tiles)
    double *gpart, *gpart2;
    int *flags;
    unsigned *sync;                           // 64 words: group barrier; 3 x 64 words: largest entry of each column of the
                                              // panel (as bits), before the first projection (by panel parity) and before
                                              // the second; then one word per CTA of the group (its SM)
    int cta0, ncta, index;                    // CTA group (on entry to launch(): ncta = the cap the scratch was
                                              // sized for); index of the sequence in its batch (noise stream)
};
struct Batch { Seq s[MAXSEQ]; int count; };

// Number of 64 x 64 fp32 tiles of Cpart / C / Dpart, fp64 tiles of gpart, for a sequence of n rows and rt
// columns handled by at most `ncta` CTAs: the partial results of the panel that has most (see KS and G in the kernel).
struct Scratch { size_t cpart, c, dpart, gpart; };
static inline Scratch scratch_tiles(int n, int rt, int ncta, bool tensor)
{
    const int nt = (n + 63) / 64, np = (rt + 63) / 64, nr = tensor ? (nt + 1) / 2 : nt;
    Scratch s{1, (size_t)np + 1, 1, (size_t)std::max(nt, std::min(2 * nt, ncta)) + 1};
    for (int nj = 1; nj < np && nt > 0; ++nj) {
        const int nc = tensor ? (nj + 1) / 2 : nj;
        s.cpart = std::max(s.cpart, (size_t)nj * std::min(nt, (ncta + nc - 1) / nc));
        s.dpart = std::max(s.dpart, (size_t)nt * std::min(nj, (ncta + nr - 1) / nr));
    }
    return s;
}

// 64 x 64 tile of a row-major fp32 matrix, zero beyond rv rows / cv columns, in two halves so that the loads of
// the next tile can be in flight while the current one is multiplied: fetch_tile (global -> registers, four
// 16-byte pieces per thread) and stash_tile (registers -> shared memory at stride lds).
struct TileRegs { float4 v[4]; };
__device__ __forceinline__ void fetch_tile(TileRegs &tr, const float *src, int ld, int rv, int cv, bool vec)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int f = threadIdx.x + i * NT, r = f >> 4, c = (f & 15) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rv) {
            const float *p = src + (size_t)r * ld + c;
            if (vec && c + 3 < cv) v = __ldcg((const float4 *)p);
            else {
                if (c < cv) v.x = __ldcg(p);
                if (c + 1 < cv) v.y = __ldcg(p + 1);
                if (c + 2 < cv) v.z = __ldcg(p + 2);
                if (c + 3 < cv) v.w = __ldcg(p + 3);
            }
        }
        tr.v[i] = v;
    }
}
__device__ __forceinline__ void stash_tile(const TileRegs &tr, float *dst, int lds)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int f = threadIdx.x + i * NT, r = f >> 4, c = (f & 15) * 4;
        *(float4 *)(dst + r * lds + c) = tr.v[i];             // lds is a multiple of 4 floats: 16-byte aligned
    }
}

// sum of base[0], base[stride], ..., base[(count - 1) stride] in that order, eight loads in flight
template <typename T>
__device__ __forceinline__ T ordered_sum(const T *base, size_t stride, int count)
{
    T s = (T)0;
    int i = 0;
    for (; i + 8 <= count; i += 8) {
        T v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = __ldcg(base + (size_t)(i + k) * stride);
#pragma unroll
        for (int k = 0; k < 8; ++k) s += v[k];
    }
    for (; i < count; ++i) s += __ldcg(base + (size_t)i * stride);
    return s;
}

// acc += op(A) B on the fp32 units (fp32 inputs).
template <bool A_TRANS>
__device__ __forceinline__ void tile_mac(const float *As, int lda, const float *Bs, int ldb, int m0, int n0, float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll 4
    for (int k = 0; k < BLK; ++k) {
        const float a0 = A_TRANS ? As[k * lda + m0 + g] : As[(m0 + g) * lda + k];
        const float a1 = A_TRANS ? As[k * lda + m0 + g + 8] : As[(m0 + g + 8) * lda + k];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const float2 b = *(const float2 *)(Bs + k * ldb + n0 + nt * 8 + 2 * t);
            acc[nt][0] = fmaf(a0, b.x, acc[nt][0]); acc[nt][1] = fmaf(a0, b.y, acc[nt][1]);
            acc[nt][2] = fmaf(a1, b.x, acc[nt][2]); acc[nt][3] = fmaf(a1, b.y, acc[nt][3]);
        }
    }
}

// This thread's part of a 64 x 64 accumulator tile (rows m0 + g, + 8; columns n0 + 8 nt + 2 t, + 1).
__device__ __forceinline__ void store_acc(float *dst, int ld, int m0, int n0, const float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
        const int c = n0 + nt * 8 + 2 * t;
        *(float2 *)(dst + (size_t)(m0 + g) * ld + c) = make_float2(acc[nt][0], acc[nt][1]);
        *(float2 *)(dst + (size_t)(m0 + g + 8) * ld + c) = make_float2(acc[nt][2], acc[nt][3]);
    }
}

// TENSOR: bf16 inputs (tensor-core products); otherwise fp32 FMA everywhere.
template <bool TENSOR>
__global__ void __launch_bounds__(NT, 2)
orth_persistent_kernel(const __grid_constant__ Batch batch, int reps, uint64_t seed, int *status)
{
    extern __shared__ __align__(16) float osm[];
    float *sA = osm, *sB = osm + BLK * LDB;                   // two tiles at stride LDB (covers LDA too)
    double *Gs = (double *)(osm + 2 * BLK * LDB);             // 64 x LDC, behind them
    int si = 0;
#pragma unroll 1
    for (int i = 1; i < batch.count; ++i) if ((int)blockIdx.x >= batch.s[i].cta0) si = i;
    const Seq &sq = batch.s[si];
    const int rank = (int)blockIdx.x - sq.cta0, tid = threadIdx.x, warp = tid >> 5;
    if (rank >= sq.ncta || sq.n <= 0 || sq.rt <= 0) return;
    const int m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    const int n = sq.n, rt = sq.rt, ld = sq.ld, ncta = sq.ncta;
    const int ntile = (n + 63) / 64, npanel = (rt + 63) / 64;
    // The passes that form the Gram matrix go by half tiles where there are CTAs for them: the fp64 products of a tile alone take
    // 2300 cycles of its SM, 5000 to 9000 with what is around them (16 x 512 x 320: 1096 -> 1067 us for the three iterates, 512 x 192
    // in fp32: 655 -> 622).
    const int gh = 2 * ntile <= ncta ? 32 : 64, ngram = (n + gh - 1) / gh;
    const bool vec = (ld & 3) == 0 && ((size_t)sq.M & 15) == 0;
    int *abort_flag = status + 1;
    unsigned gen = 0;
    bool alive = true;
    auto barrier = [&]() { alive = j3::group_barrier(sq.sync, ++gen, (unsigned)ncta, abort_flag) && alive; };

    // The CTA that shares an SM with rank 0 (if it belongs to this group) stays out of the work that runs beside
    // rank 0's factorisation, which is a latency chain and slows down under a busy neighbour.
    unsigned smid;
    asm("mov.u32 %0, %%smid;" : "=r"(smid));
    if (tid == 0) sq.sync[SYNC_WORDS + rank] = smid;
    // Largest entry of each column of panel pj over the row tiles first, first + stride, ... (bits of non-negative floats
    // order like integers)
    auto column_max = [&](int pj, int first, int stride) {
        const int j0 = pj * 64, w = min(64, rt - j0), c = tid & 63;
        float m = 0.f;
        if (c < w)
            for (int t = first; t < ntile; t += stride) {
                const int r0 = t * 64 + (tid >> 6), r1 = min(n, (t + 1) * 64);
#pragma unroll 8
                for (int r = r0; r < r1; r += 4) m = fmaxf(m, fabsf(__ldcg(sq.M + (size_t)r * ld + j0 + c)));
            }
        if (m > 0.f) atomicMax(sq.sync + 64 + 64 * (pj & 1) + c, __float_as_uint(m));
    };
    if (TENSOR) column_max(0, rank, ncta);
    barrier();
    __shared__ int mate_s;
    if (tid == 0) mate_s = 1 << 30;
    __syncthreads();
    if (alive) {
        const unsigned sm0 = __ldcg(sq.sync + SYNC_WORDS);
        for (int r = 1 + tid; r < ncta; r += NT)
            if (__ldcg(sq.sync + SYNC_WORDS + r) == sm0) atomicMin(&mate_s, r);
    }
    __syncthreads();
    const int mate = mate_s < ncta ? mate_s : -1;
    const bool overlap = reps == 2 && ncta >= 4;
    const int nworkers = ncta - 1 - (mate > 0 ? 1 : 0);
    const int wid = (rank == 0 || rank == mate) ? -1 : rank - 1 - ((mate > 0 && rank > mate) ? 1 : 0);

    // Scales of the panel's columns for the fp16 parts: entries of P, and of C = Q^T P, are below the column norm, i.e. below
    // sqrt(n) times the largest entry of the column; after a first apply the columns have unit norm.
    __shared__ unsigned wmax[NT / 32];
    __shared__ __align__(16) float colscale[64], colinv[64];   // (read in 16-byte pieces)
    int half_log_n = 0;
    while ((1ll << (2 * half_log_n)) < n) ++half_log_n;
    constexpr float QSCALE = 16384.f;                         // entries of the finished columns: at most 1
    auto set_scales = [&](int slot) {                         // slot < 0: unit columns
        if (TENSOR && tid < 64) {
            const float2 sc = slot < 0 ? make_float2(8192.f, 1.f / 8192.f) : hs::scale_for(__ldcg(sq.sync + 64 + 64 * slot + tid), 15 - half_log_n);
            colscale[tid] = sc.x;
            colinv[tid] = sc.y * (1.f / QSCALE);
        }
        __syncthreads();
    };
    // Tiles of fp16 parts: two buffers of two tiles of finished columns, one tile of the panel or of C; the first four take
    // the place of sA, sB and Gs.
    auto htile = [&](int k) { return (__half *)osm + (size_t)k * 2 * hs::PLANE; };
    auto async_q = [&](__half *dst, int t, int jb) {           // rows of tile t, columns of panel jb
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int f = tid + i * NT, plane = f >> 9, r = (f >> 3) & 63, c = (f & 7) * 8, row = t * 64 + r;
            const __half *src = (plane ? sq.ql : sq.qh) + (size_t)(row < n ? row : 0) * sq.ldq + jb * 64 + c;
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + plane * hs::PLANE + r * hs::LDH + c);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(row < n ? 16 : 0) : "memory");
        }
    };
    auto async_commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    auto put_tile = [&](const TileRegs &tr, __half *dst, float4 sc) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int f = tid + i * NT;
            const float4 v = tr.v[i];
            hs::put4(dst, f >> 4, (f & 15) * 4, make_float4(v.x * sc.x, v.y * sc.y, v.z * sc.z, v.w * sc.w));
        }
    };
    // P <- P W on a tile: P (fp32, in registers) times W, result in acc. W's rows undo the column scales.
    auto times_factor = [&](const TileRegs &tr, float (&acc)[4][4]) {
        TileRegs rw;
        fetch_tile(rw, sq.W, 64, 64, 64, true);
        if constexpr (!TENSOR) {
            stash_tile(tr, sA, LDA);
            stash_tile(rw, sB, LDB);
            __syncthreads();
            tile_mac<false>(sA, LDA, sB, LDB, m0, n0, acc);
        } else {
            float rs[4], m = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                rs[i] = colinv[(tid >> 4) + 16 * i] * QSCALE;
                const float4 v = rw.v[i];
                m = fmaxf(m, rs[i] * fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
            }
            const unsigned mb = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if ((tid & 31) == 0) wmax[warp] = mb;
            put_tile(tr, htile(0), *(const float4 *)&colscale[(tid & 15) * 4]);
            __syncthreads();
            unsigned all = wmax[0];
#pragma unroll
            for (int k = 1; k < NT / 32; ++k) all = max(all, wmax[k]);
            const float2 sc = hs::scale_for(all, 15);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float k = rs[i] * sc.x;
                const float4 v = rw.v[i];
                hs::put4(htile(1), (tid >> 4) + 16 * i, (tid & 15) * 4, make_float4(v.x * k, v.y * k, v.z * k, v.w * k));
            }
            __syncthreads();
            hs::product64<false, false>(htile(0), htile(1), m0, n0, acc);
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[nt][e] *= sc.y;
        }
        __syncthreads();
    };
    auto unscale = [&](float (&acc)[4][4]) {
        const int t2 = (tid & 3) * 2;
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[nt][e] *= colinv[n0 + nt * 8 + t2 + (e & 1)];
    };

    // A panel is a short program of four kinds of passes, each written once below:
    //   PF      project (partial C over row ranges, jobs first, first + stride, ...) and / or, on rank 0, the factor
    //           of the panel's Gram matrix; SUMUPD  C = ordered sum of the partials, then partial D = Q C;
    //   GRAM    P -= sum D, optionally P <- P W, written back, Gram matrix in fp64 and its ordered sum;
    //   APPLY   P <- P W, dependent columns refilled, finished columns also as bf16 hi/lo.
    // Classic order per repetition: PF(project) SUMUPD GRAM PF(factor) APPLY. With two repetitions the second
    // projection is taken of the panel BEFORE the first factor is applied ((P - Q Q^T P) W = P W - Q Q^T (P W)), so
    // it runs beside rank 0's factorisation, and the first APPLY folds into the second GRAM pass:
    //   PF(project) SUMUPD GRAM | PF(project beside factor) SUMUPD GRAM(with W) | PF(series factor) APPLY.
    // A panel with dependent columns (their replacements must still be projected) returns to the classic order, and so does an
    // ill-conditioned one: W enlarges what rounding leaves of the finished columns in P - Q Q^T P by 1 / sqrt(least pivot),
    // and in this order nothing is projected after W. For the same reason a panel whose last factor was not benign (dependent
    // columns, a small pivot, little left of a column by the projection) gets another repetition, up to EXTRA of them.
    // (512 x 768, r 128, a spectrum that falls to 1e-6 of noise: X - U U^T X 1.5e-6 sigma_1 instead of 5e-4; 300 x 1000,
    // r 250, 1e-4 of noise: U^T U - I 4e-6 instead of 0.3.)
    enum { OP_PF, OP_SUMUPD, OP_GRAM, OP_APPLY };
    for (int pj = 0; pj < npanel && alive; ++pj) {
        const int j0 = pj * 64, w = min(64, rt - j0), nj = pj;            // nj finished panels
        // jobs of the projections: (columns, row range) and (rows, column range), by pairs of tiles with TENSOR
        const int nc = TENSOR ? (nj + 1) / 2 : nj, nr = TENSOR ? (ntile + 1) / 2 : ntile;
        const int KS = nj > 0 ? max(1, min(ntile, (ncta + nc - 1) / nc)) : 1;
        const int tper = (ntile + KS - 1) / KS;
        const int G = nj > 0 ? max(1, min(nj, (ncta + nr - 1) / nr)) : 1;
        const int jper = nj > 0 ? (nj + G - 1) / G : 1;
        const int nrange = max(1, min(8, ngram / 32)), cper = (ngram + nrange - 1) / nrange;
        int stage = overlap ? 0 : 30, rep = 0;
        while (stage >= 0 && alive) {
            int op = OP_PF, first = -1, stride = 1, arep = 0;
            bool do_factor = false, series_ok = false, with_w = false, last = false, skip = false;
            // which scales the panel's columns have: pj & 1 the panel as it came, 2 after the first projection, -1 unit columns
            const int scale_slot = stage <= 1 ? pj & 1 : stage <= 5 || stage == 20 ? 2 : stage < 30 ? -1 : rep == 0 ? pj & 1 : -1;
            switch (stage) {
                // overlapped order
                case 0: op = OP_PF; first = rank; stride = ncta; skip = nj == 0; break;
                case 1: op = OP_SUMUPD; skip = nj == 0; break;
                case 2: op = OP_GRAM; break;
                case 3: op = OP_PF; first = nj > 0 ? wid : -1; stride = nworkers; do_factor = true; break;
                case 4: op = OP_SUMUPD; skip = nj == 0; break;
                case 5: op = OP_GRAM; with_w = true; break;
                case 6: op = OP_PF; do_factor = true; series_ok = true; break;
                case 7: op = OP_APPLY; arep = 1; last = true; break;
                // dependent columns or a small pivot found by the first factor: classic remainder (rep counts its repetitions)
                case 20: op = OP_APPLY; arep = 0; break;
                case 21: op = OP_PF; first = rank; stride = ncta; skip = nj == 0; break;
                case 22: op = OP_SUMUPD; skip = nj == 0; break;
                case 23: op = OP_GRAM; break;
                case 24: op = OP_PF; do_factor = true; series_ok = true; break;
                case 25: op = OP_APPLY; arep = 1 + rep; last = true; break;
                // classic order, any number of repetitions
                case 30: op = OP_PF; first = rank; stride = ncta; skip = nj == 0; break;
                case 31: op = OP_SUMUPD; skip = nj == 0; break;
                case 32: op = OP_GRAM; break;
                case 33: op = OP_PF; do_factor = true; series_ok = rep > 0; break;
                default: op = OP_APPLY; arep = rep; last = rep >= reps - 1; break;      // 34
            }
            if (!skip) switch (op) {
            case OP_PF: {
                // beside the last factor of a panel the other CTAs note the column maxima of the next panel
                const bool scan = TENSOR && do_factor && stage != 3 && (stage != 33 || rep >= reps - 1) && pj + 1 < npanel;
                if (TENSOR && !do_factor && rank == 0 && tid < 64) sq.sync[192 + tid] = 0u;   // (used up by the panel before)
                if (scan && (rank > 0 || ncta == 1)) column_max(pj + 1, max(rank - 1, 0), max(ncta - 1, 1));
                if (do_factor && rank == 0) {
                    {   // all elements of a partial matrix in flight together
                        double2 g[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) g[i] = make_double2(0.0, 0.0);
                        for (int rg = 0; rg < nrange; ++rg) {
                            double2 x[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) x[i] = __ldcg((const double2 *)(sq.gpart2 + (size_t)rg * 4096) + tid + i * NT);
#pragma unroll
                            for (int i = 0; i < 8; ++i) { g[i].x += x[i].x; g[i].y += x[i].y; }
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            double *dst = Gs + ((tid + i * NT) >> 5) * LDC + ((tid + i * NT) & 31) * 2;
                            dst[0] = g[i].x; dst[1] = g[i].y;
                        }
                    }
                    __syncthreads();
                    // a nearly orthonormal panel gets its factor from a short series instead of the factorisation
                    if (!(series_ok && lowdin_64(Gs, w, sA, (__half *)sB, sq.W, sq.flags))) {
                        // given up (see lost_length): columns of which nothing is left, but not the replacements of the last factor.
                        // Where the factor is that of unit columns, one that has lost half of its length asks for another repetition:
                        // the factor enlarges what the finished columns' own errors have left in it, by up to 128 within the limits
                        // of a benign factor, and the next panel starts from that (581 x 952 tokens that fall by 60 octaves, six
                        // panels: U^T U - I of 0.2, 5e-3 with it).
                        const bool unit = stage == 24 || (stage == 33 && rep > 0);
                        const float lost = lost_length(stage == 24 ? rep : stage == 33 ? rep - 1 : 0);
                        const bool old = unit && tid < w && !(__ldcg(sq.flags + tid) & 1);
                        chol_invert_64(Gs, (double *)osm, w, sq.W, sq.flags);
                        if (unit) {
                            __syncthreads();
                            // the diagonal of the factor: 1 / length outside the columns before
                            if (old) {
                                const float inv = __ldcg(sq.W + tid * 65);
                                sq.flags[tid] |= (inv * lost >= 1.f ? 1 : 0) | (inv > 2.f ? 4 : 0);
                            }
                        }
                    }
                    __syncthreads();
                } else if (first >= 0) {
                    set_scales(scale_slot);
                    const float4 ps4 = *(const float4 *)&colscale[(tid & 15) * 4];
                    if constexpr (TENSOR) for (int it = first; it < nc * KS; it += stride) {
                        const int jb = it / KS * 2, ks = it - jb / 2 * KS;
                        const bool two = jb + 1 < nj;
                        float acc[2][4][4] = {};
                        const int t0 = ks * tper, t1 = min(ntile, (ks + 1) * tper);
                        TileRegs rb;
                        auto issue = [&](int t) {
                            __half *dst = htile(2 * ((t - t0) & 1));
                            async_q(dst, t, jb);
                            if (two) async_q(dst + 2 * hs::PLANE, t, jb + 1);
                        };
                        if (t0 < t1) {
                            issue(t0);
                            fetch_tile(rb, sq.M + (size_t)t0 * 64 * ld + j0, ld, min(64, n - t0 * 64), w, vec);
                        }
                        async_commit();
                        for (int t = t0; t < t1; ++t) {
                            put_tile(rb, htile(4), ps4);
                            if (t + 1 < t1) issue(t + 1);                   // next tiles in flight during the products
                            async_commit();
                            asm volatile("cp.async.wait_group 1;" ::: "memory");
                            __syncthreads();
                            if (t + 1 < t1) fetch_tile(rb, sq.M + (size_t)(t + 1) * 64 * ld + j0, ld, min(64, n - (t + 1) * 64), w, vec);
                            const __half *q = htile(2 * ((t - t0) & 1));
                            hs::product64<true, false>(q, htile(4), m0, n0, acc[0]);
                            if (two) hs::product64<true, false>(q + 2 * hs::PLANE, htile(4), m0, n0, acc[1]);
                            __syncthreads();
                        }
                        unscale(acc[0]);
                        store_acc(sq.Cpart + (size_t)(jb * KS + ks) * 4096, 64, m0, n0, acc[0]);
                        if (two) {
                            unscale(acc[1]);
                            store_acc(sq.Cpart + (size_t)((jb + 1) * KS + ks) * 4096, 64, m0, n0, acc[1]);
                        }
                    } else for (int it = first; it < nj * KS; it += stride) {
                        const int jb = it / KS, ks = it - jb * KS;
                        float acc[4][4] = {};
                        const int t0 = ks * tper, t1 = min(ntile, (ks + 1) * tper);
                        TileRegs ra, rb;
                        if (t0 < t1) {
                            fetch_tile(ra, sq.M + (size_t)t0 * 64 * ld + jb * 64, ld, min(64, n - t0 * 64), 64, vec);
                            fetch_tile(rb, sq.M + (size_t)t0 * 64 * ld + j0, ld, min(64, n - t0 * 64), w, vec);
                        }
                        for (int t = t0; t < t1; ++t) {
                            stash_tile(ra, sA, LDB);
                            stash_tile(rb, sB, LDB);
                            __syncthreads();
                            if (t + 1 < t1) {                               // next tiles in flight during the product
                                const int rv = min(64, n - (t + 1) * 64);
                                fetch_tile(ra, sq.M + (size_t)(t + 1) * 64 * ld + jb * 64, ld, rv, 64, vec);
                                fetch_tile(rb, sq.M + (size_t)(t + 1) * 64 * ld + j0, ld, rv, w, vec);
                            }
                            tile_mac<true>(sA, LDB, sB, LDB, m0, n0, acc);
                            __syncthreads();
                        }
                        store_acc(sq.Cpart + (size_t)it * 4096, 64, m0, n0, acc);
                    }
                }
                barrier();
            } break;
            case OP_SUMUPD: {
                for (int it = rank; it < nj * 4; it += ncta) {           // a quarter tile per job
                    const int jb = it >> 2;
                    const float4 *src = (const float4 *)(sq.Cpart + (size_t)jb * KS * 4096) + (it & 3) * NT + tid;
                    float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int ks = 0; ks < KS; ks += 8) {                 // in this order, eight loads in flight
                        float4 x[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) x[q] = ks + q < KS ? __ldcg(src + (size_t)(ks + q) * 1024) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < 8; ++q) { c4.x += x[q].x; c4.y += x[q].y; c4.z += x[q].z; c4.w += x[q].w; }
                    }
                    ((float4 *)(sq.C + (size_t)jb * 4096))[(it & 3) * NT + tid] = c4;
                }
                barrier();
                if (!alive) break;
                set_scales(scale_slot);
                const float4 ps4 = *(const float4 *)&colscale[(tid & 15) * 4];
                if constexpr (TENSOR) for (int it = rank; it < nr * G; it += ncta) {
                    const int t = it / G * 2, g = it - t / 2 * G;
                    const bool two = t + 1 < ntile;
                    float acc[2][4][4] = {};
                    const int jb0 = g * jper, jb1 = min(nj, (g + 1) * jper);
                    TileRegs rb;
                    auto issue = [&](int jb) {
                        __half *dst = htile(2 * ((jb - jb0) & 1));
                        async_q(dst, t, jb);
                        if (two) async_q(dst + 2 * hs::PLANE, t + 1, jb);
                    };
                    if (jb0 < jb1) {
                        issue(jb0);
                        fetch_tile(rb, sq.C + (size_t)jb0 * 4096, 64, 64, 64, true);
                    }
                    async_commit();
                    for (int jb = jb0; jb < jb1; ++jb) {
                        put_tile(rb, htile(4), ps4);
                        if (jb + 1 < jb1) issue(jb + 1);
                        async_commit();
                        asm volatile("cp.async.wait_group 1;" ::: "memory");
                        __syncthreads();
                        if (jb + 1 < jb1) fetch_tile(rb, sq.C + (size_t)(jb + 1) * 4096, 64, 64, 64, true);
                        const __half *q = htile(2 * ((jb - jb0) & 1));
                        hs::product64<false, false>(q, htile(4), m0, n0, acc[0]);
                        if (two) hs::product64<false, false>(q + 2 * hs::PLANE, htile(4), m0, n0, acc[1]);
                        __syncthreads();
                    }
                    unscale(acc[0]);
                    store_acc(sq.Dpart + (size_t)(t * G + g) * 4096, 64, m0, n0, acc[0]);
                    if (two) {
                        unscale(acc[1]);
                        store_acc(sq.Dpart + (size_t)((t + 1) * G + g) * 4096, 64, m0, n0, acc[1]);
                    }
                } else for (int it = rank; it < ntile * G; it += ncta) {
                    const int t = it / G, g = it - t * G;
                    const int rv = min(64, n - t * 64);
                    float acc[4][4] = {};
                    const int jb0 = g * jper, jb1 = min(nj, (g + 1) * jper);
                    TileRegs ra, rb;
                    if (jb0 < jb1) {
                        fetch_tile(ra, sq.M + (size_t)t * 64 * ld + jb0 * 64, ld, rv, 64, vec);
                        fetch_tile(rb, sq.C + (size_t)jb0 * 4096, 64, 64, 64, true);
                    }
                    for (int jb = jb0; jb < jb1; ++jb) {
                        stash_tile(ra, sA, LDA);
                        stash_tile(rb, sB, LDB);
                        __syncthreads();
                        if (jb + 1 < jb1) {
                            fetch_tile(ra, sq.M + (size_t)t * 64 * ld + (jb + 1) * 64, ld, rv, 64, vec);
                            fetch_tile(rb, sq.C + (size_t)(jb + 1) * 4096, 64, 64, 64, true);
                        }
                        tile_mac<false>(sA, LDA, sB, LDB, m0, n0, acc);
                        __syncthreads();
                    }
                    store_acc(sq.Dpart + (size_t)it * 4096, 64, m0, n0, acc);
                }
                barrier();
            } break;
            case OP_GRAM: {
                // the columns' largest entries are noted before a second projection of the same panel; the slot of the panel
                // before this one is cleared for the next panel (noted beside the factor that follows)
                const bool note_max = TENSOR && stage == 2;
                float4 cmax = make_float4(0.f, 0.f, 0.f, 0.f);
                if (TENSOR && rank == 0 && tid < 64) sq.sync[64 + 64 * ((pj + 1) & 1) + tid] = 0u;
                if (TENSOR && with_w) set_scales(scale_slot);
                for (int t = rank; t < ngram; t += ncta) {
                    const int row0 = t * gh, rv = min(gh, n - row0);
                    TileRegs ra;
                    fetch_tile(ra, sq.M + (size_t)row0 * ld + j0, ld, rv, w, vec);
                    if (nj > 0) {
                        const float4 *dp = (const float4 *)(sq.Dpart + (size_t)(row0 >> 6) * G * 4096 + (row0 & 63) * 64) + tid;
                        float4 d[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) d[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int g = 0; g < G; g += 2) {                 // in this order, eight loads in flight
                            float4 x[8];
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                x[q] = g + (q >> 2) < G && (q & 2) * 16 < gh ? __ldcg(dp + (size_t)(g + (q >> 2)) * 1024 + (q & 3) * NT) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                            for (int q = 0; q < 8; ++q) { float4 &a = d[q & 3]; a.x += x[q].x; a.y += x[q].y; a.z += x[q].z; a.w += x[q].w; }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {                    // (rows and columns beyond the tile are zero in both)
                            float4 &v = ra.v[i];
                            v.x -= d[i].x; v.y -= d[i].y; v.z -= d[i].z; v.w -= d[i].w;
                            const int f = tid + i * NT, r = f >> 4, c = (f & 15) * 4;
                            if (!with_w && r < rv) {
                                float *dm = sq.M + (size_t)(row0 + r) * ld + j0 + c;
                                if (vec && c + 3 < w) *(float4 *)dm = v;
                                else {
                                    if (c < w) dm[0] = v.x;
                                    if (c + 1 < w) dm[1] = v.y;
                                    if (c + 2 < w) dm[2] = v.z;
                                    if (c + 3 < w) dm[3] = v.w;
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 v = ra.v[i];
                        cmax.x = fmaxf(cmax.x, fabsf(v.x)); cmax.y = fmaxf(cmax.y, fabsf(v.y));
                        cmax.z = fmaxf(cmax.z, fabsf(v.z)); cmax.w = fmaxf(cmax.w, fabsf(v.w));
                    }
                    if (!with_w) {
                        stash_tile(ra, sA, LDA);
                        __syncthreads();
                    } else {
                        float acc[4][4] = {};
                        times_factor(ra, acc);
                        const int lane = tid & 31, g = lane >> 2, tq = lane & 3;
#pragma unroll
                        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int r = m0 + g + (i >= 2 ? 8 : 0), c = n0 + nt * 8 + 2 * tq + (i & 1);
                                const bool in = r < rv && c < w;
                                sA[r * LDA + c] = in ? acc[nt][i] : 0.f;
                                if (in) sq.M[(size_t)(row0 + r) * ld + j0 + c] = acc[nt][i];
                            }
                        __syncthreads();
                    }
                    gram_tile_64(sA, LDA, gh, Gs, sq.gpart + (size_t)t * 4096);
                    __syncthreads();
                }
                if (note_max) {
                    unsigned *cm = (unsigned *)colinv;                       // (free between the projections)
                    if (tid < 64) cm[tid] = 0u;
                    __syncthreads();
                    const float m[4] = {cmax.x, cmax.y, cmax.z, cmax.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) atomicMax(cm + (tid & 15) * 4 + k, __float_as_uint(m[k]));
                    __syncthreads();
                    if (tid < 64 && cm[tid] > 0u) atomicMax(sq.sync + 192 + tid, cm[tid]);
                }
                barrier();
                if (!alive) break;
                // ordered sum of the partial Gram matrices: 16 element slices x (up to 8) chunk ranges
                for (int it = rank; it < 16 * nrange; it += ncta) {
                    const int sl = it & 15, rg = it >> 4, e = sl * 256 + tid;
                    const int c0 = rg * cper, c1 = min(ngram, (rg + 1) * cper);
                    sq.gpart2[(size_t)rg * 4096 + e] = ordered_sum(sq.gpart + (size_t)c0 * 4096 + e, 4096, max(c1 - c0, 0));
                }
                barrier();
            } break;
            default: {                                                   // OP_APPLY
                const uint64_t nseed = seed + 7919ull * (uint64_t)(pj * 2 + (arep & 1)) + 0x51ED270Bull * (uint64_t)(arep >> 1);
                const float rscale = rsqrtf((float)n * (1.f / 3.f));     // replacement columns of about unit norm
                if (TENSOR) set_scales(scale_slot);
                int fl[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) fl[k] = __ldcg(sq.flags + (tid & 15) * 4 + k) & 1;
                for (int t = rank; t < ntile; t += ncta) {
                    const int rv = min(64, n - t * 64);
                    TileRegs ra;
                    fetch_tile(ra, sq.M + (size_t)t * 64 * ld + j0, ld, rv, w, vec);
                    float acc[4][4] = {};
                    times_factor(ra, acc);
                    store_acc(sA, LDA, m0, n0, acc);
                    __syncthreads();
                    // out row by row, four columns a thread (the flags are read once, before any store)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = (tid >> 4) + 16 * i, c = (tid & 15) * 4, grow = t * 64 + r;
                        if (r >= rv || c >= w) continue;
                        const float4 q = *(const float4 *)(sA + r * LDA + c);
                        float v[4] = {q.x, q.y, q.z, q.w};
                        __nv_bfloat162 h[2], l[2];
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (fl[k]) v[k] = rscale * hash_uniform(nseed, ((uint64_t)sq.index << 40) ^ ((uint64_t)grow << 8) ^ (uint64_t)(c + k));
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            h[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                            l[k] = __floats2bfloat162_rn(v[2 * k] - __low2float(h[k]), v[2 * k + 1] - __high2float(h[k]));
                        }
                        float *dm = sq.M + (size_t)grow * ld + j0 + c;
                        if (vec && c + 3 < w) *(float4 *)dm = make_float4(v[0], v[1], v[2], v[3]);
                        else for (int k = 0; k < 4 && c + k < w; ++k) dm[k] = v[k];
                        if (TENSOR && last && pj + 1 < npanel) {             // (the last panel is projected against by nobody)
                            const __half2 h0 = __floats2half2_rn(v[0] * QSCALE, v[1] * QSCALE), h1 = __floats2half2_rn(v[2] * QSCALE, v[3] * QSCALE);
                            const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
                            const __half2 l0 = __floats2half2_rn(v[0] * QSCALE - f0.x, v[1] * QSCALE - f0.y);
                            const __half2 l1 = __floats2half2_rn(v[2] * QSCALE - f1.x, v[3] * QSCALE - f1.y);
                            const size_t at = (size_t)grow * sq.ldq + j0 + c;
                            *(uint2 *)(sq.qh + at) = make_uint2(*(const uint32_t *)&h0, *(const uint32_t *)&h1);
                            *(uint2 *)(sq.ql + at) = make_uint2(*(const uint32_t *)&l0, *(const uint32_t *)&l1);
                        }
                        if (last && sq.hi) {
                            // the pair's rows are padded to multiples of 8 columns; what lies beyond rt is never read
                            *(uint2 *)(sq.hi + (size_t)grow * sq.ldh + j0 + c) = *(const uint2 *)h;
                            *(uint2 *)(sq.lo + (size_t)grow * sq.ldh + j0 + c) = *(const uint2 *)l;
                        }
                    }
                    __syncthreads();
                }
                barrier();
            } break;
            }
            // next stage
            if (stage == 3 || stage == 7 || stage == 25 || stage == 34) {
                // (lengths count from the second factor on: the panel had unit columns then)
                const bool again = __syncthreads_or(alive && tid < w && (__ldcg(sq.flags + tid) & (stage == 3 ? 5 : 7)) != 0) != 0;
                if (stage == 3) stage = again ? 20 : 4;
                else if (stage == 34) { ++rep; stage = rep < reps || (again && rep < reps + EXTRA) ? 30 : -1; }
                else stage = again && rep++ < EXTRA ? 21 : -1;
            }
            else ++stage;
        }
    }
}

__global__ void init_kernel(const __grid_constant__ Batch batch)
{
    const Seq &sq = batch.s[blockIdx.x];
    if ((int)threadIdx.x < SYNC_WORDS && sq.n > 0) sq.sync[threadIdx.x] = 0u;
}

// two fp32 tiles and the Gram matrix, or five tiles of fp16 parts
template <bool TENSOR> constexpr size_t SMEM_BYTES = TENSOR ? 5 * hs::TILE_BYTES : (size_t)(2 * BLK * LDB) * sizeof(float) + (size_t)PB * LDC * sizeof(double);
static_assert((size_t)(2 * BLK * LDB) * sizeof(float) + (size_t)PB * LDC * sizeof(double) <= 5 * hs::TILE_BYTES, "Gram matrix behind the tiles");

// Largest number of CTAs a launch hands to one sequence (workspace sizing and launch agree on it).
static inline int max_ctas_per_seq(int sm_count, int nseq) { return std::max(1, 2 * sm_count / std::max(nseq, 1)); }

template <bool TENSOR>
static inline atp_status launch(atp_ctx *ctx, Batch &ob, int reps, uint64_t seed)
{
    if (ob.count <= 0) return ATP_OK;
    static PerDeviceOnce attr_once;
    ATP_CUDA_OK(ctx, attr_once.run(ctx->device, [] {
        return cudaFuncSetAttribute(orth_persistent_kernel<TENSOR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES<TENSOR>);
    }));
    int occ = 0;
    ATP_CUDA_OK(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, orth_persistent_kernel<TENSOR>, NT, SMEM_BYTES<TENSOR>));
    if (occ < 1) return ATP_ERR_CUDA;
    const int total = ctx->sm_count * std::min(occ, 2);
    double wsum = 0;
    for (int i = 0; i < ob.count; ++i) wsum += (double)ob.s[i].n * ob.s[i].rt;
    if (wsum <= 0) return ATP_OK;
    int next = 0;
    for (int i = 0; i < ob.count; ++i) {
        Seq &q = ob.s[i];
        const int ntile = (q.n + 63) / 64;
        int c = (int)((double)total * ((double)q.n * q.rt / wsum));
        c = std::max(1, std::min(std::min(c, q.ncta), 4 * std::max(ntile, 1)));    // q.ncta: the cap the scratch was sized for
        q.cta0 = next; q.ncta = c; q.index = i;
        next += c;
    }
    if (next > total) return ATP_ERR_INVALID_ARG;      // cannot happen: shares sum to at most `total`
    ATP_KERNEL(ctx, "orth_init", 0, 0);
    init_kernel<<<ob.count, 256, 0, ctx->stream>>>(ob);
    ATP_LAUNCHED(ctx);
    int *status = ctx->dev_status;
    void *args[] = {(void *)&ob, (void *)&reps, (void *)&seed, (void *)&status};
    // bytes: one read and one write of every iterate
    ATP_KERNEL(ctx, "orth_persistent", 0, wsum * 8.0);
    ATP_CUDA_OK(ctx, cudaLaunchCooperativeKernel((const void *)orth_persistent_kernel<TENSOR>, dim3(next), dim3(NT), args, SMEM_BYTES<TENSOR>, ctx->stream));
    ATP_LAUNCHED(ctx);
    return ATP_OK;
}

}  // namespace orth
