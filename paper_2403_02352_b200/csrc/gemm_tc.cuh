// Batched bf16 GEMM on the 5th-generation tensor cores (tcgen05.mma, accumulator in TMEM, operands
// staged in shared memory by TMA with the 128-byte swizzle): C = epilogue(op(A) * B).
//   A: M x K row-major (K-major operand) or K x M row-major (M-major operand), bf16
//   B: K x N row-major (N-major operand) or N x K row-major (K-major operand), bf16; optionally more
//      matrices of the same shape whose products are accumulated on top (split precision: B = B_hi + B_lo [+ B_lo2],
//      16 [24] mantissa bits), and a second matrix A_lo as well: A_hi B_hi + A_hi B_lo + A_lo B_hi carries
//      about 16 mantissa bits of both operands, for fp32 data cut into bf16 hi/lo pairs
//   C: M x N row-major, fp32 or bf16, or a bf16 hi/lo pair or hi/lo/lo2 triple; D (optional): M x N fp32
//   DUAL: two matrices B and B_gate side by side in one tile, C = silu(A B_gate) * (A B)
// Persistent: a CTA (or a pair of CTAs) walks over its tiles with two accumulators in TMEM, so that the epilogue of a tile
// runs beside the products of the next. Two forms (see choose_pairs for the rule):
//   CG = 2: a cluster of two CTAs makes 256 x 256 tiles (tcgen05.mma.cta_group::2): each CTA stages 128 rows of A and 128
//           columns of B. What bounds a bf16 GEMM here is the L2 -> shared-memory path, about 64 bytes a clock and SM: a
//           128 x 128 tile needs 128 bytes a clock at the full tensor rate, the pair's tile 64.
//   CG = 1: 128 x 128 tiles, for problems with too few 256 x 256 tiles to fill the GPU.
// Warp roles: EW epilogue warps (tcgen05.ld), one TMA warp, one warp that allocates TMEM and issues the MMAs. Extents come
// from per-problem tensor maps, so ragged M, N, K are zero-filled by TMA and masked at the store.
// Every mbarrier wait is bounded; on expiry the kernel records ATP_ERR_TIMEOUT and winds down.
#pragma once
#include "common.cuh"
#include "gemm_simt.cuh"
#include <cuda.h>

namespace tc {

constexpr int BM = 128, BN = 128, BK = 64;      // rows of A and columns of B staged by one CTA; K per stage
constexpr int MAX_PROB = 16;
constexpr uint32_t WAIT_LIMIT = 1u << 22;

struct Problem {
    CUtensorMap ta, ta2, tb, tb2, tb3; // ta2: low part of a split A; tb2, tb3: low parts of a split B, or (tb2) the gate matrix
    void *C; void *C2; void *C3; const float *D;
    int M, N, K, ldc, ldd;
    int tile0, tiles_n, tiles_m; // first linear tile index of this problem, tiles along N and along M
};
template <int P> struct Batch {         // (small launches carry a small parameter block)
    Problem p[P];
    int count, total_tiles;
};

enum OutKind { OUT_F32 = 0, OUT_BF16 = 1, OUT_BF16_SPLIT = 2, OUT_BF16_SPLIT3 = 3 };

// ---- PTX wrappers -----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: false when the limit ran out or another role already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 1023u) == 1023u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
// One lane of a converged warp. The compiler knows the branch to be taken by a single thread: with lane == 0 it guards every
// tcgen05 instruction against several active lanes, and issuing an MMA took 140 cycles (SwiGLU of 4096 rows at r 2048: 586 ->
// 555 us). Fetching the tensor maps ahead of the first copy (prefetch.tensormap) gave nothing measurable.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// The same MMA with the A operand in tensor memory (M = 128 lanes = rows, two 16-bit K elements per
// 32-bit column): only B is read from shared memory.
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// The same load without the wait: several loads can be in flight, then one tmem_ld_wait().
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle, Blackwell version field set.
//   K-major tile  (rows of 64 bf16 = 128 B, 8-row groups 1024 B apart):        lbo unused, sbo = 1024
//   MN-major tile (k-rows of 64 bf16 along M/N, 8-row groups 1024 B apart,
//                  64-element chunks `lbo` bytes apart):                        lbo = chunk stride, sbo = 1024
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;      // descriptor version
    d |= (uint64_t)2 << 61;      // SWIZZLE_128B
    return d;
}
// Instruction descriptor for kind::f16 with bf16 operands and fp32 accumulation.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N, bool a_mn_major, bool b_mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- cluster forms (CG = 2: a pair of CTAs, rank 0 leads) --------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
template <int CG> __device__ __forceinline__ void tma_load_cg(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar)
{
    if (CG == 1) tma_load_2d(dst, map, c0, c1, bar);
    else asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];"
                      ::"r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
template <int CG> __device__ __forceinline__ void tmem_alloc_cg(uint32_t dst_smem, uint32_t ncols)
{
    if (CG == 1) tmem_alloc(dst_smem, ncols);
    else {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
}
template <int CG> __device__ __forceinline__ void tmem_dealloc_cg(uint32_t taddr, uint32_t ncols)
{
    if (CG == 1) tmem_dealloc(taddr, ncols);
    else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
template <int CG> __device__ __forceinline__ void umma_cg(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    if (CG == 1) umma_bf16(d, ad, bd, idesc, acc);
    else asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                      ::"r"(d), "l"(ad), "l"(bd), "r"(idesc), "r"(acc) : "memory");
}
// completion of the MMAs issued so far arrives at the barrier of both CTAs of the pair
template <int CG> __device__ __forceinline__ void umma_commit_cg(uint32_t bar)
{
    if (CG == 1) umma_commit(bar);
    else asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                      ::"r"(bar), "h"((uint16_t)3) : "memory");
}
template <int CG> __device__ __forceinline__ void arrive_at(uint32_t bar)      // bar: an address of the leader (map_to_rank) for CG = 2
{
    if (CG == 1) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
    else asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

template <int CG, int NB, bool SPLIT_A> struct Cfg {
    static constexpr int A_BYTES = BM * BK * 2;                 // 16 KB
    static constexpr int B_BYTES = BK * BN * 2;                 // 16 KB
    static constexpr int B_OFF = A_BYTES * (SPLIT_A ? 2 : 1);
    static constexpr int STAGE_BYTES = B_OFF + B_BYTES * NB;
    // one CTA per SM and as many stages as fit; only the plain 128 x 128 form stays small enough for two
    static constexpr bool TWO_PER_SM = CG == 1 && NB == 1 && !SPLIT_A;
    static constexpr int STAGES = TWO_PER_SM ? 3 : 200 * 1024 / STAGE_BYTES;
    static constexpr int NACC = CG * BN;                        // accumulator columns of a tile
    static constexpr int EW = CG == 2 ? 8 : 4;                  // epilogue warps
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
};

__device__ __forceinline__ void store_32b(void *dst, const uint32_t (&v)[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
// 32 consecutive values of a row as bf16; part k = 0, 1, 2 of the hi / lo / lo2 cut leaves the remainder in v
__device__ __forceinline__ void store_row32_bf16(__nv_bfloat16 *dst, float (&v)[32], int valid, bool v32, bool v16, bool more)
{
    uint32_t h[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * t], v[2 * t + 1]);
        h[t] = *(const uint32_t *)&b;
        if (more) { v[2 * t] -= __low2float(b); v[2 * t + 1] -= __high2float(b); }
    }
    if (v32) {
#pragma unroll
        for (int t = 0; t < 16; t += 8) {
            const uint32_t q[8] = {h[t], h[t + 1], h[t + 2], h[t + 3], h[t + 4], h[t + 5], h[t + 6], h[t + 7]};
            store_32b(dst + 2 * t, q);
        }
    } else if (v16) {
#pragma unroll
        for (int t = 0; t < 16; t += 4) *(uint4 *)(dst + 2 * t) = make_uint4(h[t], h[t + 1], h[t + 2], h[t + 3]);
    } else {
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            const __nv_bfloat162 b = *(const __nv_bfloat162 *)&h[t];
            if (2 * t < valid) dst[2 * t] = __low2bfloat16(b);
            if (2 * t + 1 < valid) dst[2 * t + 1] = __high2bfloat16(b);
        }
    }
}

template <int CG, bool A_MN, int NB, int OUT, bool B_KMAJ, bool SPLIT_A, bool DUAL, int P>
__global__ void __launch_bounds__(Cfg<CG, NB, SPLIT_A>::EW * 32 + 64)
gemm_tc_kernel(const __grid_constant__ Batch<P> batch, GemmEpi epi, int *dev_status)
{
    using C_ = Cfg<CG, NB, SPLIT_A>;
    static_assert(!SPLIT_A || NB == 2, "a split A comes with a split B");
    static_assert(!DUAL || (NB == 1 && !SPLIT_A && !B_KMAJ), "the gated form takes plain row-major weights");
    constexpr int S = C_::STAGES, EW = C_::EW, TN = DUAL ? C_::NACC / 2 : C_::NACC;   // output columns of a tile
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;                // swizzled tiles need 1024-byte alignment
    uint8_t *gbase = smem_raw + (base - raw);
    const uint32_t bars = base + S * C_::STAGE_BYTES;            // full[S], empty[S], acc full[2], acc free[2], then tmem slot
    const uint32_t b_full = bars, b_empty = bars + 8 * S, b_afull = b_empty + 8 * S, b_afree = b_afull + 16;
    uint32_t *tmem_slot = (uint32_t *)(gbase + S * C_::STAGE_BYTES + 8 * (2 * S + 4));
    __shared__ int abort_flag;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const uint32_t rank = CG == 2 ? cluster_rank() : 0u;
    const int first = (int)blockIdx.x / CG, step = (int)gridDim.x / CG, total = batch.total_tiles;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < S; ++s) { mbar_init(b_full + 8 * s, 1); mbar_init(b_empty + 8 * s, 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(b_afull + 8 * a, 1); mbar_init(b_afree + 8 * a, CG * EW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == EW + 1) tmem_alloc_cg<CG>(smem_u32(tmem_slot), 2 * C_::NACC);
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();                                                  // set-up done; from here on memory of the launch before is touched
    pdl_trigger();

    // Tile t: problem, first row and column of the whole tile (both CTAs of a pair). Where N is much larger than M,
    // consecutive tiles walk along M: they share a tile of the large operand B, and the operand that is re-read from L2 is
    // the small one, A (a 4096 x 2048 x 11008 product read 1 GB from DRAM in row-major tile order).
    auto locate = [&](int t, int &m0, int &n0) -> const Problem & {
        int pi = 0;
#pragma unroll 1
        for (int i = 1; i < batch.count; ++i) if (t >= batch.p[i].tile0) pi = i;
        const Problem &pr = batch.p[pi];
        const int lt = t - pr.tile0;
        const bool along_m = pr.tiles_n > 2 * pr.tiles_m;
        m0 = (along_m ? lt % pr.tiles_m : lt / pr.tiles_n) * (CG * BM);
        n0 = (along_m ? lt / pr.tiles_m : lt % pr.tiles_n) * TN;
        return pr;
    };

    if (warp == EW) {
        if (elect_one()) {
            int ks = 0;                                          // stages filled so far
            bool ok = true;
            for (int t = first; t < total && ok; t += step) {
                int m0, n0;
                const Problem &pr = locate(t, m0, n0);
                m0 += rank * BM;
                const int num_kt = (pr.K + BK - 1) / BK;
                for (int kt = 0; kt < num_kt; ++kt, ++ks) {
                    const int s = ks % S;
                    if (ks >= S && !mbar_wait(b_empty + 8 * s, ((ks / S) - 1) & 1, &abort_flag)) { ok = false; break; }
                    const uint32_t full = CG == 2 ? map_to_rank(b_full + 8 * s, 0) : b_full + 8 * s;
                    const uint32_t sa = base + s * C_::STAGE_BYTES, sb = sa + C_::B_OFF;
                    if (rank == 0) mbar_expect_tx(b_full + 8 * s, CG * C_::STAGE_BYTES);
                    const int k0 = kt * BK;
                    auto load_a = [&](uint32_t dst, const CUtensorMap *m) {
                        if (!A_MN) tma_load_cg<CG>(dst, m, k0, m0, full);                    // box {64 k, 128 m}
                        else {
                            tma_load_cg<CG>(dst, m, m0, k0, full);                           // box {64 m, 64 k} x 2
                            tma_load_cg<CG>(dst + 8192, m, m0 + 64, k0, full);
                        }
                    };
                    load_a(sa, &pr.ta);
                    if (SPLIT_A) load_a(sa + C_::A_BYTES, &pr.ta2);
                    if (DUAL) {
                        // pair: CTA 0 stages 128 columns of B, CTA 1 the same columns of the gate; alone: 64 of each
                        const CUtensorMap *m0p = CG == 2 && rank == 1 ? &pr.tb2 : &pr.tb, *m1p = CG == 2 ? m0p : &pr.tb2;
                        tma_load_cg<CG>(sb, m0p, n0, k0, full);
                        tma_load_cg<CG>(sb + 8192, m1p, CG == 2 ? n0 + 64 : n0, k0, full);
                    } else {
                        const int nn = n0 + (int)rank * BN;
                        auto load_b = [&](uint32_t dst, const CUtensorMap *m) {
                            if (B_KMAJ) tma_load_cg<CG>(dst, m, k0, nn, full);               // box {64 k, 128 n}
                            else {
                                tma_load_cg<CG>(dst, m, nn, k0, full);                       // box {64 n, 64 k} x 2
                                tma_load_cg<CG>(dst + 8192, m, nn + 64, k0, full);
                            }
                        };
                        load_b(sb, &pr.tb);
                        if (NB > 1) load_b(sb + C_::B_BYTES, &pr.tb2);
                        if (NB > 2) load_b(sb + 2 * C_::B_BYTES, &pr.tb3);
                    }
                }
            }
        }
    } else if (warp == EW + 1) {
        if (rank == 0 && elect_one()) {
            constexpr uint32_t idesc = instr_desc(CG * BM, C_::NACC, A_MN, !B_KMAJ);
            bool ok = true;
            int ks = 0, it = 0;
            for (int t = first; t < total && ok; t += step, ++it) {
                int m0, n0;
                const Problem &pr = locate(t, m0, n0);
                const int num_kt = (pr.K + BK - 1) / BK, ab = it & 1;
                if (it >= 2) ok = mbar_wait(b_afree + 8 * ab, ((it >> 1) - 1) & 1, &abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem_base + ab * C_::NACC;
                for (int kt = 0; kt < num_kt; ++kt, ++ks) {
                    const int s = ks % S;
                    ok = mbar_wait(b_full + 8 * s, (ks / S) & 1, &abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + s * C_::STAGE_BYTES, sb = sa + C_::B_OFF;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk) {
                        auto adesc = [&](uint32_t a0) { return A_MN ? smem_desc(a0 + kk * 2048, 8192, 1024) : smem_desc(a0 + kk * 32, 16, 1024); };
                        auto bdesc = [&](uint32_t b0) { return B_KMAJ ? smem_desc(b0 + kk * 32, 16, 1024) : smem_desc(b0 + kk * 2048, 8192, 1024); };
                        const uint64_t ad = adesc(sa), bd = bdesc(sb);
                        uint32_t acc = (kt > 0 || kk > 0) ? 1u : 0u;
                        // small terms first, the hi * hi product last
                        if (NB > 2) { umma_cg<CG>(d, ad, bdesc(sb + 2 * C_::B_BYTES), idesc, acc); acc = 1u; }
                        if (SPLIT_A) { umma_cg<CG>(d, adesc(sa + C_::A_BYTES), bd, idesc, acc); acc = 1u; }
                        if (NB > 1) { umma_cg<CG>(d, ad, bdesc(sb + C_::B_BYTES), idesc, acc); acc = 1u; }
                        umma_cg<CG>(d, ad, bd, idesc, acc);
                    }
                    umma_commit_cg<CG>(b_empty + 8 * s);         // frees the stage once these MMAs have read it
                }
                if (ok) umma_commit_cg<CG>(b_afull + 8 * ab);    // accumulator complete
            }
        }
    } else {
        // epilogue: TMEM lane = row of the tile; EW = 8: warps 4..7 take the second half of the columns
        const int quad = warp & 3, half = warp >> 2;
        constexpr int CW = TN / (EW / 4);                        // output columns of this warp
        const uint32_t afree = CG == 2 ? map_to_rank(b_afree, 0) : b_afree;
        int it = 0;
        for (int t = first; t < total; t += step, ++it) {
            int m0, n0;
            const Problem &pr = locate(t, m0, n0);
            const int ab = it & 1;
            int ok_i = 0;
            if (lane == 0) ok_i = mbar_wait(b_afull + 8 * ab, (it >> 1) & 1, &abort_flag) ? 1 : 0;
            if (__shfl_sync(0xffffffffu, ok_i, 0) == 0) break;           // warp-uniform: tcgen05.ld is warp-collective
            tc_fence_after();
            const int row = m0 + (int)rank * BM + quad * 32 + lane;
            const uint32_t tacc = tmem_base + ab * C_::NACC + ((uint32_t)(quad * 32) << 16);
#pragma unroll 1
            for (int c = half * CW; c < half * CW + CW; c += 32) {
                uint32_t r[32], gte[32];
                tmem_ld32_nowait(tacc + c, r);
                if (DUAL) tmem_ld32_nowait(tacc + TN + c, gte);
                tmem_ld_wait();
                if (c + 32 == half * CW + CW) {                  // last read of this accumulator by this warp
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) arrive_at<CG>(afree + 8 * ab);
                }
                const int col0 = n0 + c, valid = pr.N - col0;
                if (row < pr.M && valid > 0) {
                    float v[32];
                    const bool full_chunk = valid >= 32;
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
                    if (DUAL) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] *= silu_f(__uint_as_float(gte[j]));
                    } else if (epi.kind == EPI_BIAS || epi.kind == EPI_BIAS_GELU) {
                        if (epi.bias)
#pragma unroll
                            for (int j = 0; j < 32; ++j) if (j < valid) v[j] += __ldg(epi.bias + col0 + j);
                        if (epi.kind == EPI_BIAS_GELU)
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = gelu_erf_f(v[j]);
                    } else if (epi.kind == EPI_ROPE) {
                        // pairs of columns turn by the angle of (row, pair of the head): D holds (cos, sin) per row and pair;
                        // the head width ldd is a multiple of 32, so the chunk lies inside one head
                        const float4 *cs = (const float4 *)(pr.D + (size_t)row * pr.ldd + col0 % pr.ldd);
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            const float4 t4 = __ldg(cs + j / 4);
                            const float x0 = v[j], y0 = v[j + 1], x1 = v[j + 2], y1 = v[j + 3];
                            v[j] = x0 * t4.x - y0 * t4.y; v[j + 1] = x0 * t4.y + y0 * t4.x;
                            v[j + 2] = x1 * t4.z - y1 * t4.w; v[j + 3] = x1 * t4.w + y1 * t4.z;
                        }
                    }
                    if (OUT == OUT_F32) {
                        float *dst = (float *)pr.C + (size_t)row * pr.ldc + col0;
                        if (full_chunk && ((uintptr_t)dst & 31) == 0) {
#pragma unroll
                            for (int j = 0; j < 32; j += 8) {
                                const uint32_t q[8] = {__float_as_uint(v[j]), __float_as_uint(v[j + 1]), __float_as_uint(v[j + 2]), __float_as_uint(v[j + 3]),
                                                       __float_as_uint(v[j + 4]), __float_as_uint(v[j + 5]), __float_as_uint(v[j + 6]), __float_as_uint(v[j + 7])};
                                store_32b(dst + j, q);
                            }
                        } else if (full_chunk && ((uintptr_t)dst & 15) == 0) {
#pragma unroll
                            for (int j = 0; j < 32; j += 4) *(float4 *)(dst + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j) if (j < valid) dst[j] = v[j];
                        }
                    } else {
                        const size_t at = (size_t)row * pr.ldc + col0;
                        __nv_bfloat16 *dst = (__nv_bfloat16 *)pr.C + at;
                        const bool v32 = full_chunk && (((uintptr_t)dst | (OUT >= OUT_BF16_SPLIT ? (uintptr_t)pr.C2 : 0) | (OUT == OUT_BF16_SPLIT3 ? (uintptr_t)pr.C3 : 0)) & 31) == 0 && ((pr.ldc & 15) == 0);
                        const bool v16 = full_chunk && ((pr.ldc & 7) == 0);
                        store_row32_bf16(dst, v, valid, v32, v16, OUT >= OUT_BF16_SPLIT);
                        if (OUT >= OUT_BF16_SPLIT) store_row32_bf16((__nv_bfloat16 *)pr.C2 + at, v, valid, v32, v16, OUT == OUT_BF16_SPLIT3);
                        if (OUT == OUT_BF16_SPLIT3) store_row32_bf16((__nv_bfloat16 *)pr.C3 + at, v, valid, v32, v16, false);
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag && dev_status) raise_status(dev_status, ATP_ERR_TIMEOUT);
    if (CG == 2) cluster_sync_all();                             // nobody leaves while the other CTA may still signal it
    if (warp == EW + 1) {
        tc_fence_after();
        tmem_dealloc_cg<CG>(tmem_base, 2 * C_::NACC);
    }
}

// ---- host side ---------------------------------------------------------------------------------
// Tensor map over a row-major bf16 matrix (rows x cols, ld elements): box {64 cols, box_rows rows}, 128-byte swizzle.
// The driver entry point is looked up at run time (the library does not link against libcuda, so it
// still loads on machines without a driver, where only the symbol table is inspected).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static inline EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}
static inline bool make_map(CUtensorMap *m, const void *ptr, uint64_t rows, uint64_t cols, uint64_t ld, uint32_t box_rows)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {ld * 2};
    cuuint32_t box[2] = {64, box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct HostProblem {
    const void *A; const void *B; const void *B2; void *C; void *C2; const float *D;
    int M, N, K, lda, ldb, ldc, ldd;
    const void *A2 = nullptr;     // low part of a split A
    const void *B3 = nullptr;     // third part of B
    void *C3 = nullptr;           // third part of C
};

template <int CG, bool A_MN, int NB, int OUT, bool B_KMAJ, bool SPLIT_A, bool DUAL, int P>
static atp_status launch_form(atp_ctx *ctx, const HostProblem *probs, int count, GemmEpi epi, const char *tag)
{
    using C_ = Cfg<CG, NB, SPLIT_A>;
    auto kern = gemm_tc_kernel<CG, A_MN, NB, OUT, B_KMAJ, SPLIT_A, DUAL, P>;
    static PerDeviceOnce attr_once;        // the shared-memory opt-in is a per-device attribute
    ATP_CUDA_OK(ctx, attr_once.run(ctx->device, [&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C_::SMEM); }));
    constexpr int TN = DUAL ? C_::NACC / 2 : C_::NACC;
    Batch<P> b; b.count = 0; b.total_tiles = 0;
    double flops = 0, bytes = 0;
    for (int i = 0; i < count; ++i) {
        const HostProblem &h = probs[i];
        Problem &p = b.p[b.count];
        auto amap = [&](CUtensorMap *m, const void *ptr) { return A_MN ? make_map(m, ptr, h.K, h.M, h.lda, 64) : make_map(m, ptr, h.M, h.K, h.lda, BM); };
        auto bmap = [&](CUtensorMap *m, const void *ptr) { return B_KMAJ ? make_map(m, ptr, h.N, h.K, h.ldb, BN) : make_map(m, ptr, h.K, h.N, h.ldb, 64); };
        bool ok = amap(&p.ta, h.A) && bmap(&p.tb, h.B);
        if (SPLIT_A) ok = ok && h.A2 && amap(&p.ta2, h.A2);
        if (NB > 1 || DUAL) ok = ok && h.B2 && bmap(&p.tb2, h.B2);
        if (NB > 2) ok = ok && h.B3 && bmap(&p.tb3, h.B3);
        if (!ok) return ATP_ERR_INVALID_ARG;
        p.C = h.C; p.C2 = h.C2; p.C3 = h.C3; p.D = h.D; p.M = h.M; p.N = h.N; p.K = h.K; p.ldc = h.ldc; p.ldd = h.ldd;
        p.tiles_n = ceil_div(h.N, TN);
        p.tiles_m = ceil_div(h.M, CG * BM);
        p.tile0 = b.total_tiles;
        b.total_tiles += p.tiles_m * p.tiles_n;
        b.count++;
        flops += 2.0 * h.M * h.N * h.K * (SPLIT_A || NB == 3 ? 3 : (NB == 2 || DUAL ? 2 : 1));
        bytes += 2.0 * ((double)h.M * h.K + (double)h.K * h.N * (DUAL ? 2 : NB)) + (double)h.M * h.N * (OUT == OUT_F32 ? 4 : 2 * (OUT == OUT_BF16 ? 1 : OUT));
    }
    const int slots = CG == 2 ? ctx->sm_count / 2 : ctx->sm_count * (C_::TWO_PER_SM ? 2 : 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(slots, b.total_tiles) * CG); cfg.blockDim = dim3(C_::EW * 32 + 64);
    cfg.dynamicSmemBytes = C_::SMEM; cfg.stream = ctx->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = CG; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = CG == 2 ? 2 : 1;
    ATP_KERNEL(ctx, tag ? tag : (SPLIT_A || NB == 3 ? "gemm_tc_split3" : (NB == 2 ? "gemm_tc_split" : "gemm_tc")), flops, bytes);
    ATP_CUDA_OK(ctx, cudaLaunchKernelEx(&cfg, kern, b, epi, ctx->dev_status));
    ATP_LAUNCHED(ctx);
    return ATP_OK;
}

// Pairs of CTAs (256 x 256 tiles) or single ones (128 x 128 tiles, 128 x 64 gated): the form with the smaller number of
// waves times the time of a stage of one tile. A stage takes a pair about 560 cycles whatever runs beside it; a single CTA
// about 330 when it has the L2 path to itself (all tiles in one wave), 500 when every SM loads at the full rate. The weights
// are those of one product; with two or three a stage takes both forms longer by about the same factor. All pairs / all
// single / as chosen, us a launch:
//   one product, linear layer (mean of its two launches) 512 rows, r 256, 1024 -> 1024  14.9 / 11.7 / 12.4
//                4096 rows, r 2048, 4096 -> 4096  54.6 / 61.4 / 58.1;  gated, -> 11008  244 / 292 / 238
//   two          Q = U_r Q', 1024 x 1024 x 256  16.9 / 11.0 / 10.8;  2048 x 4096 x 512  25.6 / 25.1 / 26.5
//                4096 x 4096 x 2048  95.4 / 106 / 95.8
//   three        rotary keys, 1024 x 1024 x 256  25.7 / 17.6 / 17.8;  4096 x 4096 x 2048  141 / 167 / 140
//                Gram matrix, 576 x 576 x 2048  40.1 / 27.0 / 26.0;  2112 x 2112 x 4096  127 / 86.5 / 85.7
// Over 24 such calls the choice is within 8 % of the better form, but for 1024 rows, r 256, 4096 columns (one product 35.3
// against 32.3, two 16.9 against 14.9).
template <bool DUAL>
static inline bool choose_pairs(const HostProblem *probs, int count, int sm_count)
{
    int t1 = 0, t2 = 0;
    for (int i = 0; i < count; ++i) {
        const int n2 = DUAL ? 128 : 256, n1 = n2 / 2;
        t2 += ceil_div(probs[i].M, 256) * ceil_div(probs[i].N, n2);
        t1 += ceil_div(probs[i].M, 128) * ceil_div(probs[i].N, n1);
    }
    return ceil_div(t2, sm_count / 2) * 560 <= ceil_div(t1, sm_count) * (t1 <= sm_count ? 330 : 500);
}

template <bool A_MN, int NB, int OUT, bool B_KMAJ = false, bool SPLIT_A = false, bool DUAL = false>
static atp_status launch(atp_ctx *ctx, const std::vector<HostProblem> &all, GemmEpi epi, const char *tag = nullptr)
{
    HostProblem probs[MAX_PROB];
    size_t i = 0;
    while (i < all.size()) {
        int n = 0;
        for (; i < all.size() && n < MAX_PROB; ++i)
            if (all[i].M > 0 && all[i].N > 0 && all[i].K > 0) probs[n++] = all[i];
        if (n == 0) continue;
        atp_status st;
        if (choose_pairs<DUAL>(probs, n, ctx->sm_count))
            st = n <= 2 ? launch_form<2, A_MN, NB, OUT, B_KMAJ, SPLIT_A, DUAL, 2>(ctx, probs, n, epi, tag)
                        : launch_form<2, A_MN, NB, OUT, B_KMAJ, SPLIT_A, DUAL, MAX_PROB>(ctx, probs, n, epi, tag);
        else
            st = n <= 2 ? launch_form<1, A_MN, NB, OUT, B_KMAJ, SPLIT_A, DUAL, 2>(ctx, probs, n, epi, tag)
                        : launch_form<1, A_MN, NB, OUT, B_KMAJ, SPLIT_A, DUAL, MAX_PROB>(ctx, probs, n, epi, tag);
        if (st != ATP_OK) return st;
    }
    return ATP_OK;
}

}  // namespace tc
