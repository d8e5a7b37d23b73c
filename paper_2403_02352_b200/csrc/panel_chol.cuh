// Cholesky factorisation and inversion of a 64 x 64 Gram matrix in fp64, on 256 threads of a CTA.
// Gs (shared memory, 64 x 64 doubles, row-major) holds G = P^T P of a panel of n <= 64 columns. The
// matrix is scaled to unit diagonal, factored D^-1 G D^-1 = L L^T and the factor inverted; the result
// W = D^-1 L^-T (upper triangular, fp32, 64 x 64 row-major) goes to rinv, so that P W has orthonormal
// columns. A column whose scaled pivot falls below 1e-10 (its part outside the span of the earlier
// columns is below 1e-5 of its norm) is flagged as dependent in flags[0..63].
// Right-looking by blocks of four columns, in registers: thread (br, bc) owns the 4 x 4 blocks of G
// and of X (X starts as the identity and ends as L^-1) at rows 4 br, columns 4 bc. Block step jb:
//   1. the owner of the diagonal block factors it (four pivots) and publishes L_bb and 1 / L_jj;
//   2. the owners of the block column below it solve for their rows of L, the owners of block row jb of
//      X apply L_bb^-1 to it; both publish;
//   3. everybody below subtracts L_i L_k^T from G (columns right of jb) or L_i X_b from X (columns up
//      to jb): 64 independent multiply-adds per thread.
// Two barriers per four columns (named barrier 1, 256 threads: exactly the threads 0..255 must call).
// Bound by the chain of 64 pivots (reciprocal root, scaling, next pivot) and the two barriers of a block step. The
// published rows are stored column-wise (lc[c][row]), so that step 3 reads them in 16-byte pieces with at most two
// lanes on a bank; row-wise they collided 16-fold, and the reciprocal root went through two fp32 conversions:
// 40300 -> 34600 cycles.
#pragma once
#include "common.cuh"
#include "jacobi3.cuh"

constexpr int PB = 64;            // orthonormalisation panel width

__device__ __noinline__ void chol_invert_64(const double *Gs, int n, float *rinv, int *flags)
{
    __shared__ double rs[PB];          // 1 / sqrt(diagonal of the Gram matrix)
    __shared__ __align__(16) double lc[4][PB];    // block column jb of L (rows below the diagonal block), by column
    __shared__ __align__(16) double xrow4[4][PB]; // block row jb of L^-1
    __shared__ double Lbb[4][4];       // the factored diagonal block (strictly lower part)
    __shared__ double rinv4[4];        // 1 / L_jj, 0 for a dependent column
    __shared__ int dep[PB];
    auto bar256 = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    const int tid = threadIdx.x;
    const int br = tid >> 4, bc = tid & 15;
    // One 4 x 4 block per thread: it holds the thread's block of G until block step jb = bc has consumed it, and
    // the thread's block of X from then on (a block of G left of the current step is dead, a block of X right of
    // it is still its initial identity / zero block), which halves the register need.
    double blk[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) blk[a][b] = Gs[(4 * br + a) * PB + 4 * bc + b];
    auto to_x = [&]() {
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) blk[a][b] = (br == bc && a == b) ? 1.0 : 0.0;
    };
    if (br == bc) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = 4 * br + a;
            rs[i] = (i < n && blk[a][a] > 0.0) ? rsqrt(blk[a][a]) : 0.0;
            dep[i] = 0;
        }
    }
    bar256();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const double ra = rs[4 * br + a], rb = rs[4 * bc + b];
            blk[a][b] = (br == bc && a == b) ? (ra > 0.0 ? 1.0 : 0.0) : blk[a][b] * ra * rb;
        }
    const int nblk = (n + 3) >> 2;
    for (int jb = 0; jb < nblk; ++jb) {
        if (br == jb && bc == jb) {
            // 1. the diagonal block, column by column; a dependent column gets a unit pivot and zeros below
            double ri[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                double piv = blk[c][c];
#pragma unroll
                for (int k = 0; k < c; ++k) piv = fma(-blk[c][k], blk[c][k], piv);
                const bool bad = !(piv > 1e-10);
                // 1/sqrt from the hardware's 20-bit approximation and one Newton step: ~2^-40 relative, far below the
                // fp32 precision the result is stored in
                double y;
                asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(piv));
                y = fma(0.5 * y, fma(-piv * y, y, 1.0), y);
                ri[c] = bad ? 0.0 : y;
                if (bad && 4 * jb + c < n) dep[4 * jb + c] = 1;
#pragma unroll
                for (int r = c + 1; r < 4; ++r) {
                    double v = blk[r][c];
#pragma unroll
                    for (int k = 0; k < c; ++k) v = fma(-blk[r][k], blk[c][k], v);
                    blk[r][c] = v * ri[c];
                }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                rinv4[r] = ri[r];
#pragma unroll
                for (int c = 0; c < 4; ++c) Lbb[r][c] = (c < r) ? blk[r][c] : 0.0;
            }
            to_x();
        }
        bar256();
        if (bc == jb && br > jb) {
            // 2a. rows of L below the diagonal block: l_c = (g_c - sum_{k<c} l_k L_bb[c][k]) / L_cc
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                double l[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    double v = blk[a][c];
#pragma unroll
                    for (int k = 0; k < c; ++k) v = fma(-l[k], Lbb[c][k], v);
                    l[c] = v * rinv4[c];
                    lc[c][4 * br + a] = l[c];
                }
            }
            to_x();
        }
        if (br == jb && bc <= jb) {
            // 2b. block row jb of X: forward substitution with L_bb (a dependent column keeps its scale)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double sc = rinv4[c] > 0.0 ? rinv4[c] : 1.0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    double v = blk[c][b];
#pragma unroll
                    for (int k = 0; k < c; ++k) v = fma(-Lbb[c][k], blk[k][b], v);
                    blk[c][b] = v * sc;
                    xrow4[c][4 * bc + b] = blk[c][b];
                }
            }
        }
        bar256();
        if (br > jb && bc <= br) {
            // 3. trailing update, one column of L (and its row of X) at a time
            const double *rsrc = bc > jb ? &lc[0][4 * bc] : &xrow4[0][4 * bc];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double2 a0 = *(const double2 *)&lc[c][4 * br], a1 = *(const double2 *)&lc[c][4 * br + 2];
                const double2 b0 = *(const double2 *)(rsrc + c * PB), b1 = *(const double2 *)(rsrc + c * PB + 2);
                const double la[4] = {a0.x, a0.y, a1.x, a1.y}, rb[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) blk[a][b] = fma(-la[a], rb[b], blk[a][b]);
            }
        }
    }
    if (bc > br || bc >= nblk) to_x();      // blocks that never became part of X: above the diagonal, beyond n
    // W[k][c] = (L^-1)[c][k] / D_k ; this thread holds (L^-1)[4 br + a][4 bc + b]
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int k = 4 * bc + b;
        const double rk = rs[k];
        float4 w;
        w.x = (float)(rk * blk[0][b]); w.y = (float)(rk * blk[1][b]); w.z = (float)(rk * blk[2][b]); w.w = (float)(rk * blk[3][b]);
        *(float4 *)(rinv + k * PB + 4 * br) = w;
    }
    bar256();
    if (tid < PB) flags[tid] = (tid < n) ? (dep[tid] || !(rs[tid] > 0.0)) : 0;
}


// Orthonormalising factor of a panel that is already close to orthonormal (the second Gram-Schmidt repetition):
// with the Gram matrix scaled to unit diagonal, D^-1/2 G D^-1/2 = I + E, the symmetric factor
//   W = D^-1/2 (I - E/2 + 3/8 E^2)          (P W has orthonormal columns up to 5/16 |E|^3)
// needs one 64^3 product instead of a factorisation and its chain of 64 dependent pivots. Taken only when every
// diagonal entry is positive and the largest absolute row sum of E is at most LOWDIN_LIMIT (then the neglected
// term is below 4e-8); otherwise nothing is written and the caller factors the matrix. Returns the decision
// (block-uniform). Es: a 64 x LDE fp32 tile of shared memory; 256 threads.
// E^2 is at most 2.5e-5, so plain TF32 products (2^-10 relative) leave an error near 1e-8. Thread = 4 x 4 block: a row sum
// is complete within half a warp. 11600 -> 3300 cycles (per-element reductions, atomics and an fp32 product before).
constexpr float LOWDIN_LIMIT = 5e-3f;
constexpr int LDE = 72;
__device__ __noinline__ bool lowdin_64(const double *Gs, int n, float *Es, float *rinv, int *flags)
{
    __shared__ double rsq[PB];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    bool bad = false;
    if (tid < PB) {
        const double d = Gs[tid * PB + tid];
        const bool pos = tid < n && d > 0.0;
        rsq[tid] = pos ? rsqrt(d) : 0.0;
        bad = tid < n && !pos;
    }
    __syncthreads();
    float sum[4];
    const double sc[4] = {rsq[tx * 4], rsq[tx * 4 + 1], rsq[tx * 4 + 2], rsq[tx * 4 + 3]};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = ty * 4 + i;
        const double sr = rsq[r];
        const double2 g0 = *(const double2 *)&Gs[r * PB + tx * 4], g1 = *(const double2 *)&Gs[r * PB + tx * 4 + 2];
        const double g[4] = {g0.x, g0.y, g1.x, g1.y};
        float e[4];
        sum[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = tx * 4 + j;
            e[j] = r < n && c < n && r != c ? (float)(g[j] * sr * sc[j]) : 0.f;
            sum[i] += fabsf(e[j]);
        }
        *(float4 *)&Es[r * LDE + tx * 4] = make_float4(e[0], e[1], e[2], e[3]);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < 4; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
#pragma unroll
    for (int i = 0; i < 4; ++i) bad |= !(sum[i] <= LOWDIN_LIMIT);
    if (__syncthreads_or(bad)) return false;
    // E^2 (E is symmetric); this warp: rows m0 .. + 15, columns n0 .. + 31
    const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    float acc[4][4] = {};
    j3::product64_acc<true, false, 1>(Es, LDE, Es, LDE, m0, n0, acc);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = m0 + g + 8 * h;
        const float sr = (float)rsq[r];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
            const int c = n0 + nt * 8 + 2 * t;
            float w[2];
#pragma unroll
            for (int k = 0; k < 2; ++k)
                w[k] = r < n && c + k < n ? sr * ((r == c + k ? 1.f : 0.f) - 0.5f * Es[r * LDE + c + k] + 0.375f * acc[nt][2 * h + k]) : 0.f;
            *(float2 *)(rinv + r * PB + c) = make_float2(w[0], w[1]);
        }
    }
    if (tid < PB) flags[tid] = 0;
    return true;
}

// Partial Gram matrix of a 64 x 64 fp32 tile T (64 rows of a panel, row stride lds): dst[i][j] = sum_k T[k][i] T[k][j] in
// fp64, on the fp64 matrix units (mma.m8n8k4; 36 tiles of 8 x 8 by symmetry, four or five per warp). Td: 4096 doubles of
// shared memory for the converted tile, columns swizzled so that the fragment loads are conflict-free. Converting once
// instead of per product matters: 9500 -> 5100 cycles (fp64 FMA with conversions in the inner loop before: conversions
// run at 16 a cycle). 256 threads, T complete before the call; the caller synchronises before T or Td is reused.
__device__ __forceinline__ void gram_tile_64(const float *T, int lds, double *Td, double *dst)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = lane & 3, p = lane >> 2;
    for (int f = tid; f < PB * PB / 4; f += 256) {
        const int r = f >> 4, c = (f & 15) * 4, cs = c ^ ((r & 3) << 2);
        const float4 v = *(const float4 *)(T + r * lds + c);
        *(double2 *)&Td[r * PB + cs] = make_double2(v.x, v.y);
        *(double2 *)&Td[r * PB + cs + 2] = make_double2(v.z, v.w);
    }
    __syncthreads();
    // tiles (i, j), i <= j, numbered row by row: warp w takes w, w + 8, ...
    int ti[5], tj[5];
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        int t = warp + 8 * s, i = 0;
        while (i < 7 && t >= 8 - i) { t -= 8 - i; ++i; }
        ti[s] = i; tj[s] = min(i + t, 7);
    }
    double acc[5][2] = {};
#pragma unroll 2
    for (int k0 = 0; k0 < PB; k0 += 4) {
        const double *row = Td + (k0 + q) * PB;
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            if (s == 4 && warp >= 4) break;
            const double a = row[(8 * ti[s] + p) ^ (q << 2)], b = row[(8 * tj[s] + p) ^ (q << 2)];
            asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                : "+d"(acc[s][0]), "+d"(acc[s][1]) : "d"(a), "d"(b));
        }
    }
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        if (s == 4 && warp >= 4) break;
        const int r = 8 * ti[s] + p, c = 8 * tj[s] + 2 * q;
        *(double2 *)&dst[r * PB + c] = make_double2(acc[s][0], acc[s][1]);
        if (ti[s] != tj[s]) { dst[c * PB + r] = acc[s][0]; dst[(c + 1) * PB + r] = acc[s][1]; }
    }
}
