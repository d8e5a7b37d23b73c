// atp_alternating_basis: the paper's own approximate extraction (Algorithm 1, appendix B) - rank-1
// alternating fits with deflation - and atp_svd_entropy: Eq. 4 with the rank rule of Sec. 3.
//
// Algorithm 1 on the GPU. The method is a chain of matrix-vector products over the deflated matrix R (L x d, fp32): for
// every component, `inner` rounds of
//   u = R v / |v|^2,   v = R^T u / |u|^2,
// then R <- R - u v^T. One persistent cooperative launch runs the whole chain for all sequences of a batch: a group of CTAs
// per sequence, each with a share of the rows of R in shared memory (rows that do not fit stay in the workspace, L2). A
// round is one visit of the rows: phase A takes the dot products of the rows with v (four rows per warp; in the first
// round of a component it applies the deflation of the component before on the way), phase B multiplies the same rows by u
// column by column. The partial columns of the group's CTAs are summed in a fixed order around a group barrier. Dot
// products accumulate in fp64, so that the only rounding of a step is the fp32 storage of u, v and R.
// Bound by shared-memory reads and the widening of the elements to fp64 (half by the conversion instruction, 16 a clock and
// SM, half by three integer operations each), and by the barrier and the partial sums of a round.
// 16 sequences of 512 x 1024, r = 64, inner = 2: 5092 -> 1360 us (a chain of 320 launches that read R six times per
// component from L2 before).
#include "common.cuh"
#include "group_barrier.cuh"

constexpr int ALT_MAX = 32;        // sequences per launch
constexpr int ALT_NT = 512;        // threads per CTA
constexpr int ALT_DIRECT = 16;     // up to this many CTAs in a group every CTA sums the partial columns itself
struct AltSeq {
    const void *X;                 // first row of the sequence in the packed input
    float *R;                      // rows of the deflated matrix that do not fit in shared memory (of each CTA, dp floats a row)
    double *part;                  // partial columns: 2 (by round parity) x ncta x (dp + 4)
    float *vbuf;                   // v of a round, where it is summed in slices
    double *vecs;                  // u, v and the last v of every CTA, where they do not fit in shared memory
    unsigned *sync;                // words of the group barrier
    const float *v0;               // start vectors of this sequence (r x d, row stride ldv)
    void *U, *Xp;                  // outputs: U (L x r), X' (r x d)
    int L, r, ldx_in, ldu, ldx, ldv;
    int cta0, ncta, rows;          // CTA group, rows per CTA
};
struct AltBatch { AltSeq s[ALT_MAX]; int count; };

template <int W> __device__ __forceinline__ double block_sum(double x, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    const int w = threadIdx.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = x;
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < W; ++i) s += red[i];       // fixed order
    return s;
}

// x * 2^-896 in fp64, exactly, by shifting the bits of a finite x into place (the exponent field keeps its value, fp32
// denormals become fp64 denormals, zero stays zero). The other factor of a product is scaled by 2^896 (an fp32 value times
// 2^896 is an fp64 number), so the products and their sums are those of the converted values, whatever their size. Inf and NaN
// would come out as numbers: a warp with such rows takes their dot products again with conversions alone.
__device__ __forceinline__ double widen(float x)
{
    const int b = __float_as_int(x);
    return __hiloint2double((b >> 3) & (int)0x8fffffff, b << 29);
}
constexpr double WIDEN_SCALE = 0x1p896;

// dp: d rounded up to 4 (row stride of R; columns d .. dp - 1 are zero); srows: rows of a CTA kept in shared memory.
// FAR: the vectors do not fit in shared memory either (alternating_fixed), they lie in the workspace; srows = 0 then.
template <typename T, bool FAR>
__global__ void __launch_bounds__(ALT_NT, 1)
alternating_kernel(const __grid_constant__ AltBatch batch, int d, int dp, int srows, int maxrows, int inner, int *status)
{
    extern __shared__ __align__(16) unsigned char altsm[];
    constexpr int NW = ALT_NT / 32;
    __shared__ double red[NW], redu[NW], slice[ALT_NT];
    int si = 0;
#pragma unroll 1
    for (int i = 1; i < batch.count; ++i) if ((int)blockIdx.x >= batch.s[i].cta0) si = i;
    const AltSeq &q = batch.s[si];
    const int rank = (int)blockIdx.x - q.cta0, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (rank >= q.ncta || q.L <= 0) return;
    double *ud = FAR ? q.vecs + (size_t)rank * (maxrows + dp) : (double *)altsm;   // u of the current round
    float *vc = (float *)(ud + maxrows), *vo = vc + dp;        // v of the current round and of the last one
    float *sR = FAR ? nullptr : vo + dp;                       // rows of R
    const int row0 = rank * q.rows, nrow = max(0, min(q.rows, q.L - row0)), ns = min(srows, nrow);
    float *gR = q.R + (size_t)rank * max(q.rows - srows, 0) * dp;   // rows ns .. nrow - 1 of this CTA
    int *abort_flag = status + 1;
    unsigned gen = 0, round = 0;
    bool alive = true;

    float seen = 0.f;                                          // NaN once this lane has seen Inf or NaN in R
    for (int l = warp; l < nrow; l += NW) {
        const T *x = (const T *)q.X + (size_t)(row0 + l) * q.ldx_in;
        float *r = (l < ns ? sR + (size_t)l * dp : gR + (size_t)(l - ns) * dp);
        for (int k = lane; k < dp; k += 32) {
            const float v = k < d ? to_f32(x[k]) : 0.f;
            seen = fmaf(v, 0.f, seen);
            r[k] = v;
        }
    }
    for (int l = tid; l < maxrows; l += ALT_NT) ud[l] = 0.0;
    __syncthreads();

    for (int comp = 0; comp < q.r && alive; ++comp) {
        double un = 0.0, vpart = 0.0;                          // vpart: this thread's share of |v|^2
        { float *t = vc; vc = vo; vo = t; }                    // vo: v of the last component; vc: the start vector
        for (int k = tid; k < dp; k += ALT_NT) {
            const float v = k < d ? q.v0[(size_t)comp * q.ldv + k] : 0.f;
            vc[k] = v;
            vpart += (double)v * (double)v;
        }
        for (int j = 0; j < inner && alive; ++j, ++round) {
            const bool deflate = j == 0 && comp > 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) vpart += __shfl_xor_sync(0xffffffffu, vpart, o);
            if (lane == 0) red[warp] = vpart;
            // a row that lives in the workspace is fetched before anything else (first 1024 columns)
            float4 pre[8];
            const int pl = ns + warp;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                pre[i] = pl < nrow && lane * 4 + 128 * i < dp ? *(const float4 *)(gR + (size_t)(pl - ns) * dp + lane * 4 + 128 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();                                   // v and the parts of |v|^2
            double usq = 0.0, vv = -1.0;
            auto norm_v = [&]() {                              // fixed order
                if (vv < 0.0) {
                    vv = 0.0;
#pragma unroll
                    for (int i = 0; i < NW; ++i) vv += red[i];
                }
            };
            auto put_u = [&](int l, double acc) {              // u of row l, by one lane
                const float u = vv > 0.0 ? (float)(acc / vv) : 0.f;
                ud[l] = (double)u;
                usq += (double)u * (double)u;
            };
            auto lanes_sum = [&](double acc, int from) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) if (o <= from) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                return acc;
            };
            // one sum with converted and one with shifted elements
            auto factors = [&](double (&v)[4], int k) {
                const float4 f = *(const float4 *)(vc + k);
                v[0] = f.x; v[1] = (double)f.y * WIDEN_SCALE; v[2] = f.z; v[3] = (double)f.w * WIDEN_SCALE;
            };
            auto dot = [&](double &a, double &w, float4 x, const double (&v)[4]) {
                a = fma((double)x.x, v[0], a); w = fma(widen(x.y), v[1], w);
                a = fma((double)x.z, v[2], a); w = fma(widen(x.w), v[3], w);
            };
            auto see = [&](float4 x) { seen = fmaf(x.w, 0.f, fmaf(x.y, 0.f, seen)); };       // (the shifted elements)
            auto subtract = [&](float4 &x, float u, float4 p) {
                x.x = fmaf(-u, p.x, x.x); x.y = fmaf(-u, p.y, x.y); x.z = fmaf(-u, p.z, x.z); x.w = fmaf(-u, p.w, x.w);
            };

            // phase A: u = R v / |v|^2. Rows in shared memory, four of a warp together (v is read once for them)
            for (int l0 = warp; l0 < ns; l0 += NW * 4) {
                double acc[4] = {0.0, 0.0, 0.0, 0.0}, aw[4] = {0.0, 0.0, 0.0, 0.0};
                float *rp[4], up[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const int l = l0 + NW * a;
                    rp[a] = sR + (size_t)(l < ns ? l : l0) * dp;
                    up[a] = deflate && l < ns ? (float)ud[l] : 0.f;
                }
                for (int k = lane * 4; k < dp; k += 128) {
                    double v[4];
                    factors(v, k);
                    float4 x[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) x[a] = *(const float4 *)(rp[a] + k);
                    if (deflate) {
                        const float4 p = *(const float4 *)(vo + k);
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            subtract(x[a], up[a], p);
                            if (l0 + NW * a < ns) { *(float4 *)(rp[a] + k) = x[a]; see(x[a]); }
                        }
                    }
#pragma unroll
                    for (int a = 0; a < 4; ++a) dot(acc[a], aw[a], x[a], v);
                }
                __syncwarp();
                // the four sums over the lanes together: after two exchanges a quarter of the warp holds each row
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[a] += aw[a];
                const bool h1 = lane & 16, h0 = lane & 8;
                const double p0 = (h1 ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, h1 ? acc[0] : acc[2], 16);
                const double p1 = (h1 ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, h1 ? acc[1] : acc[3], 16);
                const double t = lanes_sum((h0 ? p1 : p0) + __shfl_xor_sync(0xffffffffu, h0 ? p0 : p1, 8), 4);
                norm_v();
                const int l = l0 + NW * (lane >> 3);
                if ((lane & 7) == 0 && l < ns) put_u(l, t);
            }
            // rows in the workspace, one of a warp at a time, eight loads in flight
            for (int l = pl; l < nrow; l += NW) {
                float *rp = gR + (size_t)(l - ns) * dp;
                const float up = deflate ? (float)ud[l] : 0.f;
                double acc = 0.0, aw = 0.0;
                for (int k0 = lane * 4; k0 < dp; k0 += 1024) {
                    if (l != pl || k0 >= 1024)
#pragma unroll
                        for (int i = 0; i < 8; ++i) pre[i] = k0 + 128 * i < dp ? *(const float4 *)(rp + k0 + 128 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int k = k0 + 128 * i;
                        if (k >= dp) continue;
                        if (deflate) { subtract(pre[i], up, *(const float4 *)(vo + k)); *(float4 *)(rp + k) = pre[i]; see(pre[i]); }
                        double v[4];
                        factors(v, k);
                        dot(acc, aw, pre[i], v);
                    }
                }
                __syncwarp();
                acc = lanes_sum(acc + aw, 16);
                norm_v();
                if (lane == 0) put_u(l, acc);
            }
            if (__any_sync(0xffffffffu, seen != 0.f)) {          // (the whole warp again)
                usq = 0.0;
                for (int l = warp; l < nrow; l += NW) {
                    const float *row = (l < ns ? sR + (size_t)l * dp : gR + (size_t)(l - ns) * dp);
                    double acc = 0.0;
                    for (int k = lane; k < dp; k += 32) acc = fma((double)row[k], (double)vc[k], acc);
                    acc = lanes_sum(acc, 16);
                    norm_v();
                    if (lane == 0) put_u(l, acc);
                }
            }
            usq = lanes_sum(usq, 16);
            if (lane == 0) redu[warp] = usq;
            __syncthreads();

            // phase B: this CTA's part of R^T u, two columns a thread; the first rows from the workspace are fetched early
            double *mine = q.part + ((size_t)(round & 1) * q.ncta + rank) * (dp + 4);
            for (int k = tid * 2; k < dp; k += ALT_NT * 2) {
                double a0 = 0.0, a1 = 0.0;
                float2 g[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) g[a] = ns + a < nrow ? *(const float2 *)(gR + (size_t)a * dp + k) : make_float2(0.f, 0.f);
                const float *col = sR + k;
                // (a row with Inf or NaN has an infinite or NaN u, so its shifted elements need no care here)
                auto add = [&](float2 x, double u) { a0 = fma((double)x.x, u, a0); a1 = fma(widen(x.y), u * WIDEN_SCALE, a1); };
                int l = 0;
                for (; l + 8 <= ns; l += 8, col += 8 * (size_t)dp) {
                    float2 x[8];
                    double2 u[4];
#pragma unroll
                    for (int a = 0; a < 8; ++a) x[a] = *(const float2 *)(col + a * (size_t)dp);
#pragma unroll
                    for (int a = 0; a < 4; ++a) u[a] = *(const double2 *)(ud + l + 2 * a);
#pragma unroll
                    for (int a = 0; a < 8; ++a) add(x[a], a & 1 ? u[a >> 1].y : u[a >> 1].x);
                }
                for (; l < ns; ++l, col += dp) add(*(const float2 *)col, ud[l]);
#pragma unroll
                for (int a = 0; a < 4; ++a) if (ns + a < nrow) add(g[a], ud[ns + a]);
#pragma unroll 4
                for (l = ns + 4; l < nrow; ++l) add(*(const float2 *)(gR + (size_t)(l - ns) * dp + k), ud[l]);
                *(double2 *)(mine + k) = make_double2(a0, a1);
            }
            if (tid == 0) {
                double s = 0.0;
#pragma unroll
                for (int i = 0; i < NW; ++i) s += redu[i];
                mine[dp] = s;
            }
            alive = group_barrier(q.sync, ++gen, (unsigned)q.ncta, abort_flag) && alive;
            if (!alive) break;
            // v = R^T u / |u|^2 from the partial columns, in rank order
            const size_t ps = (size_t)dp + 4;
            const double *all = q.part + (size_t)(round & 1) * q.ncta * ps;
            double uu = 0.0;
            for (int c = lane; c < q.ncta; c += 32) uu += __ldcg(all + (size_t)c * ps + dp);
            vpart = 0.0;
            auto keep = [&](int k, float v) { vc[k] = v; vpart += (double)v * (double)v; };
            auto all_lanes = [&](double x) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                return x;
            };
            if (q.ncta <= ALT_DIRECT) {                          // two columns a thread, all loads in flight
                bool first = true;
                for (int k0 = 0; k0 < dp; k0 += ALT_NT * 2) {
                    const int k = k0 + tid * 2;
                    double2 x[ALT_DIRECT];
#pragma unroll
                    for (int c = 0; c < ALT_DIRECT; ++c)
                        x[c] = c < q.ncta && k < dp ? __ldcg((const double2 *)(all + (size_t)c * ps + k)) : make_double2(0.0, 0.0);
                    if (first) { uu = all_lanes(uu); first = false; }
                    double s0 = 0.0, s1 = 0.0;
#pragma unroll
                    for (int c = 0; c < ALT_DIRECT; ++c) { s0 += x[c].x; s1 += x[c].y; }
                    if (k < dp) { keep(k, uu > 0.0 ? (float)(s0 / uu) : 0.f); keep(k + 1, uu > 0.0 ? (float)(s1 / uu) : 0.f); }
                }
            } else {                                             // a slice of columns per CTA, then everybody reads the whole
                uu = all_lanes(uu);
                const int per = (dp + q.ncta - 1) / q.ncta, c0 = rank * per, c1 = min(dp, c0 + per);
                for (int k0 = c0; k0 < c1; k0 += 32) {           // 32 columns at a time, the partials dealt to the warps
                    const int k = k0 + lane;
                    double s0 = 0.0;
                    if (k < c1)
#pragma unroll 4
                        for (int c = warp; c < q.ncta; c += NW) s0 += __ldcg(all + (size_t)c * ps + k);
                    slice[tid] = s0;
                    __syncthreads();
                    if (warp == 0 && k < c1) {
                        s0 = 0.0;
#pragma unroll
                        for (int i = 0; i < NW; ++i) s0 += slice[i * 32 + lane];
                        q.vbuf[k] = uu > 0.0 ? (float)(s0 / uu) : 0.f;
                    }
                    __syncthreads();
                }
                alive = group_barrier(q.sync, ++gen, (unsigned)q.ncta, abort_flag) && alive;
                if (!alive) break;
                for (int k = tid; k < dp; k += ALT_NT) keep(k, __ldcg(q.vbuf + k));
            }
            un = uu;
        }
        if (!alive) break;
        __syncthreads();
        un = sqrt(un);
        // the finished component: U[:, comp] = u / |u|, X'[comp, :] = v |u|
        for (int l = tid; l < nrow; l += ALT_NT)
            ((T *)q.U)[(size_t)(row0 + l) * q.ldu + comp] = from_f32<T>(un > 0.0 ? (float)(ud[l] / un) : 0.f);
        for (int k = rank * ALT_NT + tid; k < d; k += q.ncta * ALT_NT)
            ((T *)q.Xp)[(size_t)comp * q.ldx + k] = from_f32<T>((float)((double)vc[k] * un));
    }
}

__global__ void alternating_init_kernel(const __grid_constant__ AltBatch batch)
{
    if (threadIdx.x < 64) batch.s[blockIdx.x].sync[threadIdx.x] = 0u;
}

// CTAs of each sequence of a launch (at most `total` together): in proportion to the rows, at least one, and not more than
// leaves 16 rows (a row a warp) to a CTA.
static std::vector<int> alternating_ctas(const std::vector<SeqDims> &sd, size_t i0, size_t i1, int total)
{
    double rows = 0;
    for (size_t i = i0; i < i1; ++i) rows += sd[i].L;
    const int spare = std::max(0, total - (int)(i1 - i0));
    std::vector<int> c;
    for (size_t i = i0; i < i1; ++i)
        c.push_back(std::min(std::max(1, ceil_div(sd[i].L, 16)), 1 + (int)(rows > 0 ? spare * (sd[i].L / rows) : 0)));
    return c;
}

// Shared memory of a CTA, and what its vectors take of it: u of at most `rows` rows in fp64, two v of dp floats.
constexpr int ALT_SMEM = 226 * 1024 - 512 * 8;   // of 227 KB a CTA may have: the rest is the kernel's static share
static size_t alternating_fixed(int dp, int rows) { return (size_t)dp * 8 + align_up((size_t)std::max(rows, 1), 2) * 8 + 32; }

struct AltScratch { float *R; double *part; float *vbuf; double *vecs; unsigned *sync; int ncta, maxrows, srows; };
static void plan_alternating(Arena &ar, const std::vector<SeqDims> &sd, int d, int sm_count, std::vector<AltScratch> &out)
{
    const size_t dp = align_up((size_t)d, 4);
    for (size_t i0 = 0; i0 < sd.size(); i0 += ALT_MAX) {
        const size_t i1 = std::min(sd.size(), i0 + ALT_MAX);
        const std::vector<int> c = alternating_ctas(sd, i0, i1, sm_count);
        int rows = 1;
        for (size_t i = i0; i < i1; ++i) rows = std::max(rows, ceil_div(sd[i].L, c[i - i0]));
        rows = (int)align_up((size_t)rows, 2);
        // the vectors first, then as many rows of R as fit
        const size_t fixed = alternating_fixed((int)dp, rows);
        const bool far = fixed > (size_t)ALT_SMEM;
        const int srows = far ? 0 : (int)std::min<size_t>((ALT_SMEM - fixed) / (dp * 4), (size_t)rows);
        for (size_t i = i0; i < i1; ++i) {
            AltScratch a;
            a.ncta = c[i - i0];
            a.maxrows = rows; a.srows = srows;
            a.vecs = far ? ar.take<double>((size_t)a.ncta * (rows + dp)) : nullptr;
            a.R = ar.take<float>((size_t)a.ncta * std::max(ceil_div(sd[i].L, a.ncta) - srows, 0) * dp);
            a.part = ar.take<double>((size_t)2 * a.ncta * (dp + 4));
            a.vbuf = ar.take<float>(dp);
            a.sync = ar.take<unsigned>(64);
            out.push_back(a);
        }
    }
}

size_t alternating_workspace_bytes(const std::vector<SeqDims> &sd, int d, int sm_count)
{
    Arena ar(nullptr, (size_t)-1);
    std::vector<AltScratch> sc;
    plan_alternating(ar, sd, d, sm_count, sc);
    return ar.off;
}

template <typename T>
static atp_status alternating_impl(atp_ctx *ctx, const atp_mat *X, const std::vector<SeqDims> &sd, const atp_mat *V0, int inner,
                                   atp_mat *U_r, atp_mat *X_r)
{
    const int d = (int)X->cols, dp = (int)align_up((size_t)d, 4);
    Arena ar(ctx->workspace, ctx->workspace_bytes);
    std::vector<AltScratch> sc;
    plan_alternating(ar, sd, d, ctx->sm_count, sc);
    if (ar.overflow || !ctx->workspace) return ATP_ERR_WORKSPACE_TOO_SMALL;
    static PerDeviceOnce attr_once;
    ATP_CUDA_OK(ctx, attr_once.run(ctx->device, [] {
        return cudaFuncSetAttribute(alternating_kernel<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, ALT_SMEM);
    }));
    for (size_t i0 = 0; i0 < sd.size(); i0 += ALT_MAX) {
        AltBatch b; b.count = (int)std::min<size_t>(ALT_MAX, sd.size() - i0);
        int next = 0;
        double work = 0;
        for (int k = 0; k < b.count; ++k) {
            const SeqDims &s = sd[i0 + k];
            const AltScratch &a = sc[i0 + k];
            AltSeq &q = b.s[k];
            q.X = (const T *)X->data + (size_t)s.row0 * X->ld; q.ldx_in = (int)X->ld;
            q.R = a.R; q.part = a.part; q.vbuf = a.vbuf; q.vecs = a.vecs; q.sync = a.sync;
            q.v0 = (const float *)V0->data + (size_t)s.rank0 * V0->ld; q.ldv = (int)V0->ld;
            q.U = (T *)U_r->data + (size_t)s.row0 * U_r->ld; q.ldu = (int)U_r->ld;
            q.Xp = (T *)X_r->data + (size_t)s.rank0 * X_r->ld; q.ldx = (int)X_r->ld;
            q.L = s.L; q.r = s.r;
            q.cta0 = next; q.ncta = a.ncta; q.rows = ceil_div(s.L, a.ncta);
            next += a.ncta;
            work += (double)s.r * s.L * d * 4;
        }
        if (work == 0) continue;
        const int maxrows = sc[i0].maxrows;
        const bool far = alternating_fixed(dp, maxrows) > (size_t)ALT_SMEM;
        int srows = sc[i0].srows;
        const size_t smem = far ? 0 : alternating_fixed(dp, maxrows) + (size_t)srows * dp * 4;
        ATP_KERNEL(ctx, "alternating_init", 0, 0);
        alternating_init_kernel<<<b.count, 64, 0, ctx->stream>>>(b);
        ATP_LAUNCHED(ctx);
        int dd = d, ddp = dp, mr = maxrows, in = inner;
        int *status = ctx->dev_status;
        void *args[] = {(void *)&b, (void *)&dd, (void *)&ddp, (void *)&srows, (void *)&mr, (void *)&in, (void *)&status};
        // bytes: R once per round, written once per component (most of it in shared memory)
        ATP_KERNEL(ctx, "alternating", work / 4 * (4.0 * inner + 2), work * (inner + 1));
        const void *kern = far ? (const void *)alternating_kernel<T, true> : (const void *)alternating_kernel<T, false>;
        ATP_CUDA_OK(ctx, cudaLaunchCooperativeKernel(kern, dim3(next), dim3(ALT_NT), args, smem, ctx->stream));
        ATP_LAUNCHED(ctx);
    }
    return ATP_OK;
}

extern "C" atp_status atp_alternating_basis(atp_ctx *ctx, const atp_mat *X, const atp_seqs *seqs, const atp_mat *V0, int inner,
                                            atp_mat *U_r, atp_mat *X_r)
{
    if (!ctx) return ATP_ERR_INVALID_ARG;
    atp_status st;
    if ((st = check_mat(X)) != ATP_OK || (st = check_mat(U_r)) != ATP_OK || (st = check_mat(X_r)) != ATP_OK ||
        (st = check_mat(V0)) != ATP_OK) return st;
    if (V0->dtype != ATP_F32 || inner < 1 || inner > 64) return ATP_ERR_INVALID_ARG;
    if (U_r->dtype != X->dtype || X_r->dtype != X->dtype) return ATP_ERR_INVALID_ARG;
    std::vector<SeqDims> sd;
    if ((st = check_seqs(seqs, sd, X->rows)) != ATP_OK) return st;
    int maxr = 0, total_rank = 0;
    for (auto &s : sd) { maxr = std::max(maxr, s.r); total_rank += s.r; if (s.r > X->cols) return ATP_ERR_INVALID_RANK; }
    if (U_r->rows != X->rows || U_r->cols < maxr || X_r->rows != total_rank || X_r->cols != X->cols ||
        V0->rows != total_rank || V0->cols != X->cols) return ATP_ERR_INVALID_ARG;
    if (X->rows == 0 || X->cols == 0) return ATP_OK;
    ATP_CUDA_OK(ctx, cudaSetDevice(ctx->device));
    if (X->dtype == ATP_F32) return alternating_impl<float>(ctx, X, sd, V0, inner, U_r, X_r);
    return alternating_impl<__nv_bfloat16>(ctx, X, sd, V0, inner, U_r, X_r);
}

// ------------------------------------------------------------------------------------------------
// Eq. 4: mu = -log2(sum_i sbar_i^2), sbar_i = sigma_i / sum_j sigma_j; rank rule ceil(2^mu).
struct EntBatch { int off[ALT_MAX + 1]; int count; };
__global__ void __launch_bounds__(256) svd_entropy_kernel(const __grid_constant__ EntBatch batch, const float *sigma, float *mu, int *rank)
{
    __shared__ double red[8];
    const int b = blockIdx.x;
    const int lo = batch.off[b], hi = batch.off[b + 1];
    double p = 0.0;
    for (int i = lo + threadIdx.x; i < hi; i += 256) p += (double)sigma[i];
    const double tot = block_sum<8>(p, red);
    p = 0.0;
    for (int i = lo + threadIdx.x; i < hi; i += 256) { const double s = (double)sigma[i] / tot; p += s * s; }
    const double acc = block_sum<8>(p, red);
    if (threadIdx.x == 0) {
        const double m = (tot > 0.0 && acc > 0.0) ? -log2(acc) : 0.0;
        mu[b] = (float)m;
        if (rank) rank[b] = (tot > 0.0) ? (int)ceil(exp2(m) - 1e-9) : 0;
    }
}

extern "C" atp_status atp_svd_entropy(atp_ctx *ctx, const float *sigma, const int32_t *offsets, int32_t batch, float *mu,
                                      int32_t *rank)
{
    if (!ctx || batch < 0 || (batch > 0 && (!sigma || !offsets || !mu))) return ATP_ERR_INVALID_ARG;
    for (int b = 0; b < batch; ++b)
        if (offsets[b + 1] < offsets[b] || offsets[0] != 0) return ATP_ERR_INVALID_ARG;
    ATP_CUDA_OK(ctx, cudaSetDevice(ctx->device));
    for (int b0 = 0; b0 < batch; b0 += ALT_MAX) {
        EntBatch eb; eb.count = std::min(ALT_MAX, batch - b0);
        for (int k = 0; k <= eb.count; ++k) eb.off[k] = offsets[b0 + k];
        ATP_KERNEL(ctx, "svd_entropy", 0, (double)(eb.off[eb.count] - eb.off[0]) * 8);
        svd_entropy_kernel<<<eb.count, 256, 0, ctx->stream>>>(eb, sigma, mu + b0, rank ? rank + b0 : nullptr);
        ATP_LAUNCHED(ctx);
    }
    return ATP_OK;
}
