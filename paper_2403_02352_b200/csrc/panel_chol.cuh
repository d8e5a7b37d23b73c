// Cholesky factorisation and inversion of a 64 x 64 Gram matrix in fp64, on 256 threads of a CTA.
// Gs (shared memory, 64 rows of 64 doubles at stride LDC) holds G = P^T P of a panel of n <= 64 columns. The
// matrix is scaled to unit diagonal, factored D^-1 G D^-1 = L L^T and the factor inverted; the result
// W = D^-1 L^-T (upper triangular, fp32, 64 x 64 row-major) goes to rinv, so that P W has orthonormal
// columns. A column whose scaled pivot falls below 1e-10 (its part outside the span of the earlier
// columns is below 1e-5 of its norm) is flagged as dependent: bit 0 of its word in flags[0..63]. Bit 1: the column is shorter
// than SHRUNK; where it had unit length before the projection, what rounding left of the finished columns in it is no longer
// small against it. Bit 2: its scaled pivot is below ILL_PIVOT^2, so W enlarges a rounding error of the panel more than
// 1 / ILL_PIVOT times.
// Four panels of 16 columns. What bounds it is the chain of 64 pivots, so a panel's diagonal block is factored inside one
// warp, without a barrier: lane i < 16 holds row i of the block, lane 16 + j column j of its inverse (which starts as the
// identity); with m = (entry of column c) / L_cc in every lane, the right-looking step
//     entry[k] -= m * m_k        (m_k: m of lane k, the k-th entry of column c of L)
// is the update of the block in the lower lanes and the forward substitution for the inverse in the upper ones. The other
// warps finish the trailing update of the panel before meanwhile (the block that is factored next goes first), then all
// warps form the rows of L below the panel (A_21 X_11^T) and the blocks of the inverse left of it (-X_pp L_p,: X), in
// strips of 8 x 16 on the fp64 matrix units (with scalar multiply-adds these were bound by shared-memory reads).
// Cycles from block barrier to block barrier, in the kernel: 27000 -> 19600 (16 x 512 x 320 in bf16, 1024 x 764 the same), 38100 ->
// 23700 in fp32 (1024 x 764), since the diagonal blocks are straight code that updates what lies right of its column. The fp32
// kernel keeps more in registers around it and spills 72 bytes here, the bf16 kernel none. (The first form, 4 x 4 blocks per
// thread with 16-way bank conflicts, took 40300 in either.)
#pragma once
#include "common.cuh"
#include "jacobi3.cuh"
#include "split_mma.cuh"

constexpr int PB = 64;            // orthonormalisation panel width
constexpr double ILL_PIVOT = 0x1p-5, SHRUNK = 0.25;

constexpr int LDC = 68;           // row stride (doubles) in shared memory: the fragments below are free of bank conflicts

// acc (8 x 8 tiles n = 0, 1 of an 8 x 16 result) += sign * A B over K = 16 on the fp64 matrix units: A rows at a, stride LDC;
// B[k][n] = b[k * LDC + n], or b[n * LDC + k] when B_T. Lane: row lane / 4, columns 8 t + 2 (lane % 4), + 1.
template <bool B_T, bool NEG>
__device__ __forceinline__ void dmma_8x16x16(const double *a, const double *b, double (&acc)[2][2])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int k0 = 0; k0 < 16; k0 += 4) {
        const double x = a[g * LDC + k0 + q], av = NEG ? -x : x;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const double bv = B_T ? b[(8 * t + g) * LDC + k0 + q] : b[(k0 + q) * LDC + 8 * t + g];
            asm("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                : "+d"(acc[t][0]), "+d"(acc[t][1]) : "d"(av), "d"(bv));
        }
    }
}
__device__ __forceinline__ void dmma_load(const double *c, double (&acc)[2][2])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int t = 0; t < 2; ++t) { acc[t][0] = c[g * LDC + 8 * t + 2 * q]; acc[t][1] = c[g * LDC + 8 * t + 2 * q + 1]; }
}
__device__ __forceinline__ void dmma_store(double *c, const double (&acc)[2][2])
{
    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int t = 0; t < 2; ++t) { c[g * LDC + 8 * t + 2 * q] = acc[t][0]; c[g * LDC + 8 * t + 2 * q + 1] = acc[t][1]; }
}
// Gs is overwritten. work: 64 x LDC doubles of shared memory (ends as L^-1, lower triangle). 256 threads.
__device__ __noinline__ void chol_invert_64(double *Gs, double *work, int n, float *rinv, int *flags)
{
    __shared__ double rs[PB];          // 1 / sqrt(diagonal of the Gram matrix)
    __shared__ int dep[PB];
    __shared__ __align__(16) double xcol[2][16], xdiag[2][16];     // the column in work of a diagonal block and the diagonal entries, by step parity
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double *X = work;
    if (tid < PB) {
        const double g = Gs[tid * (LDC + 1)];
        rs[tid] = tid < n && g > 0.0 ? rsqrt(g) : 0.0;
        dep[tid] = 0;
    }
    __syncthreads();
    // D^-1 G D^-1 in place: unit diagonal (0 for a zero column); the ten 16 x 16 blocks of the lower triangle, which are all
    // that is read of the matrix
    {
        const int r = tid >> 4, c = tid & 15;
        double rr[4], rc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { rr[k] = rs[16 * k + r]; rc[k] = rs[16 * k + c]; }
#pragma unroll
        for (int bi = 0; bi < 4; ++bi)
#pragma unroll
            for (int bj = 0; bj <= bi; ++bj) {
                double *g = Gs + (16 * bi + r) * LDC + 16 * bj + c;
                *g = bi == bj && r == c ? (rr[bi] > 0.0 ? 1.0 : 0.0) : *g * rr[bi] * rc[bj];
            }
    }
    __syncthreads();
    for (int p = 0; p < 4; ++p) {
        const int b = 16 * p;
        if (warp == 0) {
            // the diagonal block: 16 dependent pivots. The unscaled column is exchanged through shared memory before its
            // pivot is known, and the next pivot comes from the current one and two entries that every lane already has
            // (d - e^2 / piv), so the chain per column is one reciprocal and two multiply-adds (11 cycles each). Instructions count
            // more than that chain: all 15 entries in every step of a loop over 16 columns (unrolled by 8) took 410 cycles a column
            // with what is around it, twice that chain. Straight code updates the entries right of the column only.
            // 16 x 512 x 320: 1067 -> 1008 us for the three iterates, 512 x 192 in fp32: 622 -> 566; same values.
            double e[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) e[k] = lane < 16 ? Gs[(b + lane) * LDC + b + k] : (lane - 16 == k ? 1.0 : 0.0);
            if (lane < 16) { xcol[0][lane] = e[0]; xdiag[0][lane] = e[1]; }
            __syncwarp();
            double piv = xcol[0][0];
            bool bad = false;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                double ck[16], dn = 0.0;
#pragma unroll
                for (int k = (c + 1) & ~1; k < 16; k += 2) {
                    const double2 v = *(const double2 *)&xcol[c & 1][k];
                    ck[k] = v.x; ck[k + 1] = v.y;
                }
                if (c < 15) dn = xdiag[c & 1][c + 1];
                const bool dep_c = !(piv > 1e-10);
                // 1/sqrt from the hardware's 20-bit approximation and one step of third order, ~2^-58 relative: an error of the
                // step goes into the entries that are left, which may be 1e-10 of those it comes from
                double y;
                asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(dep_c ? 1.0 : piv));
                const double h = fma(-piv * y, y, 1.0);
                y = fma(y * h, fma(0.375, h, 0.5), y);
                // a dependent column: unit pivot, zeros below; its row of the inverse keeps its scale
                const double ic = dep_c ? 0.0 : y * y, f = e[c] * ic;
                if (c < 15) piv = fma(-ck[c + 1] * ck[c + 1], ic, dn);
                bad |= dep_c && c == lane;
                if (lane >= 16) X[(b + c) * LDC + b + lane - 16] = c >= lane - 16 ? (dep_c ? e[c] : e[c] * y) : 0.0;
#pragma unroll
                for (int k = c + 1; k < 16; ++k) e[k] = fma(-f, ck[k], e[k]);
                if (lane < 16 && c < 15) {
                    xcol[(c + 1) & 1][lane] = e[c + 1];
                    if (c < 14) xdiag[(c + 1) & 1][lane] = e[c + 2];
                }
                __syncwarp();
            }
            if (lane < 16 && b + lane < n && bad) dep[b + lane] = 1;
        } else if (p > 0) {
            // the rest of the trailing update of panel p - 1: blocks (bi, bj), bj <= bi, below the diagonal block of panel p
            const int nb = 4 - p;
            for (int t = warp - 1; t < (nb * (nb + 1) / 2 - 1) * 2; t += 7) {
                int blk = (t >> 1) + 1, bi = 0;
                while (blk > bi) { blk -= bi + 1; ++bi; }
                const int r = b + 16 * bi + 8 * (t & 1), c = b + 16 * blk;
                double acc[2][2];
                dmma_load(Gs + r * LDC + c, acc);
                dmma_8x16x16<true, true>(Gs + r * LDC + b - 16, Gs + c * LDC + b - 16, acc);
                dmma_store(Gs + r * LDC + c, acc);
            }
        }
        __syncthreads();
        // strips of the rows of L below the panel, L = A X_pp^T (t < 2 (3 - p)), and of T = sum_k L_pk X_kq, q < p
        double acc[2][2] = {};
        const int nl = 2 * (3 - p), strip = warp;
        double *dst = nullptr;
        if (strip < nl) {
            double *a = Gs + (b + 16 + 8 * strip) * LDC + b;
            dmma_8x16x16<true, false>(a, X + b * LDC + b, acc);
            dst = a;
        } else if (strip < nl + 2 * p) {
            const int s = strip - nl, q16 = (s >> 1) * 16, r = b + 8 * (s & 1);
            for (int kb = q16; kb < b; kb += 16) dmma_8x16x16<false, false>(Gs + r * LDC + kb, X + kb * LDC + q16, acc);
            dst = X + r * LDC + q16;
        }
        __syncthreads();
        if (dst) dmma_store(dst, acc);
        __syncthreads();
        // X_pq = -X_pp T (in place: every warp reads before the barrier); the diagonal block of the next panel
#pragma unroll
        for (int t = 0; t < 2; ++t) acc[t][0] = acc[t][1] = 0.0;
        dst = nullptr;
        if (strip < 2 * p) {
            const int q16 = (strip >> 1) * 16, r = b + 8 * (strip & 1);
            dmma_8x16x16<false, true>(X + r * LDC + b, X + b * LDC + q16, acc);
            dst = X + r * LDC + q16;
        } else if (p < 3 && strip >= 6) {
            const int r = b + 16 + 8 * (strip - 6);
            dmma_load(Gs + r * LDC + b + 16, acc);
            dmma_8x16x16<true, true>(Gs + r * LDC + b, Gs + (b + 16) * LDC + b, acc);
            dst = Gs + r * LDC + b + 16;
        }
        __syncthreads();
        if (dst) dmma_store(dst, acc);
        if (strip >= 6) asm volatile("bar.arrive 2, 96;" ::: "memory");          // warp 0 goes on with the diagonal block
        else if (strip == 0) asm volatile("bar.sync 2, 96;" ::: "memory");
    }
    __syncthreads();
    // W[k][c] = (L^-1)[c][k] / D_k; the blocks of L^-1 above the diagonal have not been written
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int f = tid + 256 * i, k = f & 63, c = (f >> 6) * 4;
        const double rk = rs[k];
        float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k >> 4 <= c >> 4) {
            w.x = (float)(rk * X[c * LDC + k]); w.y = (float)(rk * X[(c + 1) * LDC + k]);
            w.z = (float)(rk * X[(c + 2) * LDC + k]); w.w = (float)(rk * X[(c + 3) * LDC + k]);
        }
        *(float4 *)(rinv + k * PB + c) = w;
    }
    // (the diagonal of L^-1 holds the reciprocal square roots of the pivots)
    if (tid < PB)
        flags[tid] = tid >= n ? 0 : (dep[tid] || !(rs[tid] > 0.0) ? 1 : 0) | (rs[tid] > 1.0 / SHRUNK ? 2 : 0) | (X[tid * (LDC + 1)] > 1.0 / ILL_PIVOT ? 4 : 0);
}


// Orthonormalising factor of a panel that is already close to orthonormal (the second Gram-Schmidt repetition):
// with the Gram matrix scaled to unit diagonal, D^-1/2 G D^-1/2 = I + E, the symmetric factor
//   W = D^-1/2 (I - E/2 + 3/8 E^2)          (P W has orthonormal columns up to 5/16 |E|^3)
// needs one 64^3 product instead of a factorisation and its chain of 64 dependent pivots. Taken only when every
// column has kept SHRUNK of its unit length and the largest absolute row sum of E is at most LOWDIN_LIMIT (then the neglected
// term is below 4e-8); otherwise nothing is written and the caller factors the matrix. Returns the decision
// (block-uniform). Es: a 64 x LDE fp32 tile of shared memory, Eh: a tile of fp16 parts; 256 threads.
// E^2 comes from two fp16 parts of E, E_SCALE E = hi + lo to 2^-25, so it is as good as an fp32 product (from one TF32 part, as
// before, it was off by 2^-10: 1e-8 in W). Thread = 4 x 4 block: a row sum is complete within half a warp.
constexpr float LOWDIN_LIMIT = 5e-3f;
constexpr int LDE = 72;
constexpr float E_SCALE = 0x1p20f;                               // an entry is at most LOWDIN_LIMIT: below 5300 then
__device__ __noinline__ bool lowdin_64(const double *Gs, int n, float *Es, __half *Eh, float *rinv, int *flags)
{
    __shared__ double rsq[PB];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    bool bad = false;
    if (tid < PB) {
        const double d = Gs[tid * (LDC + 1)];
        const bool kept = tid < n && d >= SHRUNK * SHRUNK;
        rsq[tid] = kept ? rsqrt(d) : 0.0;
        bad = tid < n && !kept;
    }
    __syncthreads();
    float sum[4];
    const double sc[4] = {rsq[tx * 4], rsq[tx * 4 + 1], rsq[tx * 4 + 2], rsq[tx * 4 + 3]};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = ty * 4 + i;
        const double sr = rsq[r];
        const double *gr = Gs + r * LDC + tx * 4, g[4] = {gr[0], gr[1], gr[2], gr[3]};
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
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 e = *(const float4 *)&Es[(ty * 4 + i) * LDE + tx * 4];
        hs::put4(Eh, ty * 4 + i, tx * 4, make_float4(e.x * E_SCALE, e.y * E_SCALE, e.z * E_SCALE, e.w * E_SCALE));
    }
    __syncthreads();
    // E^2 (E is symmetric); this warp: rows m0 .. + 15, columns n0 .. + 31
    const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, m0 = (warp & 3) * 16, n0 = (warp >> 2) * 32;
    float acc[4][4] = {};
    hs::product64<false, false>(Eh, Eh, m0, n0, acc);
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
                w[k] = r < n && c + k < n ? sr * ((r == c + k ? 1.f : 0.f) - 0.5f * Es[r * LDE + c + k] + 0.375f / (E_SCALE * E_SCALE) * acc[nt][2 * h + k]) : 0.f;
            *(float2 *)(rinv + r * PB + c) = make_float2(w[0], w[1]);
        }
    }
    if (tid < PB) flags[tid] = 0;
    return true;
}

// Partial Gram matrix of a rows x 64 fp32 tile T (32 or 64 rows of a panel, row stride lds): dst[i][j] = sum_k T[k][i] T[k][j] in
// fp64, on the fp64 matrix units (mma.m8n8k4; 36 tiles of 8 x 8 by symmetry, four or five per warp). Td: 4096 doubles of
// shared memory for the converted tile, columns swizzled so that the fragment loads are conflict-free. Converting once
// instead of per product matters: 9500 -> 5100 cycles (fp64 FMA with conversions in the inner loop before: conversions
// run at 16 a cycle). 256 threads, T complete before the call; the caller synchronises before T or Td is reused.
__device__ __forceinline__ void gram_tile_64(const float *T, int lds, int rows, double *Td, double *dst)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = lane & 3, p = lane >> 2;
    for (int f = tid; f < rows * PB / 4; f += 256) {
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
    for (int k0 = 0; k0 < rows; k0 += 4) {
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
