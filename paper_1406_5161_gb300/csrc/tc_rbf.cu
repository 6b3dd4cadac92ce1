// RBF contraction on the 5th-generation tensor cores (tcgen05, sm_103a):
//
//   out[q] = sum_k coef_k * exp(-gamma * (||z_q||^2 + ||x_k||^2 - 2 <z_q, x_k>))
//
// the inner loop of gradient reconstruction (Algorithm 6: f of the shrunk
// samples from all alpha > 0) and of the decision function (Eq. classi) in
// the mixed-precision mode. The inner products are a dense contraction: query
// rows and support vectors are densified once into BF16 row-major matrices
// (K = columns padded to 64), a CTA keeps a 128-row query tile in shared
// memory and streams 128-row support-vector tiles with TMA (128-byte
// swizzle); one thread issues tcgen05.mma (M = N = 128, K = 16, BF16 inputs,
// FP32 accumulators in tensor memory); the four warps then read the
// 128 x 128 FP32 tile from tensor memory (tcgen05.ld), apply the exp
// epilogue and accumulate coef * K per query row (FP32 within a tile, FP64
// across tiles). Support tiles and accumulators are double-buffered, so the
// load and MMA of the next tile overlap the epilogue. Padding rows carry
// coef = 0.
//
// All waits on mbarriers are bounded; on expiry the CTA records an error,
// waits (bounded) for its own asynchronous work, frees its tensor memory and
// returns, and the host reports SVM_ERR_TIMEOUT.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "svm_internal.cuh"

namespace svmgb {
namespace {

constexpr int kTile = 128;            // rows per query tile and per SV tile (M = N)
constexpr int kKB = 64;               // BF16 elements per 128-byte swizzle row
constexpr int kMaxKBlocks = 4;        // d_pad <= 256
constexpr uint32_t kTileBytes = kTile * kKB * 2;   // 16 KiB per k-block tile
constexpr long long kWaitLimit = 1ll << 26;        // mbarrier polls before giving up

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// true when the phase with the given parity completed; bounded
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    const uint32_t a = smem_u32(bar);
    for (long long i = 0; i < kWaitLimit; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// bulk copy global -> shared counted on an mbarrier (16-byte aligned, size a
// multiple of 16)
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows
// of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
    d |= (uint64_t)1 << 16;                          // leading byte offset (unused here)
    d |= (uint64_t)(1024 >> 4) << 32;                // stride byte offset: 8-row group
    d |= (uint64_t)1 << 46;                          // descriptor version
    d |= (uint64_t)2 << 61;                          // swizzle: 128-byte
    return d;
}

// Instruction descriptor of kind::f16: FP32 accumulate, BF16 A and B, both
// K-major, M = 128, N = 128.
constexpr uint32_t kIdesc = (1u << 4)                  // D format F32
                            | (1u << 7)                // A format BF16
                            | (1u << 10)               // B format BF16
                            | ((uint32_t)(kTile >> 3) << 17)   // N / 8
                            | ((uint32_t)(kTile >> 4) << 24);  // M / 16

struct TcArgs {
    int64_t nq, nsv;
    int kblocks;                 // d_pad / 64
    int stages;                  // support-tile slots in shared memory (2..4)
    const float *zc;             // per query: -gamma * log2(e) * ||z||^2
    const float *xc;             // per SV (padded): -gamma * log2(e) * ||x||^2
    const float *coef;           // per SV (padded): alpha * y (0 on padding)
    float g2;                    // 2 * gamma * log2(e)
    const int32_t *qrow;         // output index per query (row id or position)
    const int8_t *yq;            // subtract yq[qrow] when non-NULL
    double add_scalar;
    double *out;
    int *err;
    // few query tiles: the support tiles split over gridDim.y CTAs per query
    // tile, whose sums (part: [splits][nq]) the last CTA to finish adds in
    // split order (done: per query tile, zeroed)
    double *part;
    unsigned *done;
};

// 2^x on the special-function unit (flush to zero below 2^-126)
// packed pairs of FP32 values (f32x2 arithmetic, sm_100 and later)
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b,
                                                       unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ void tmem_ld_x32(uint32_t *r, uint32_t addr)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr)
        : "memory");
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One CTA: a 128-row query tile against all support-vector tiles, with the
// roles split by warp and handed over by mbarriers only (no CTA-wide barrier
// inside the tile loop):
//   warp 0 (one thread)  TMA loads of the support tiles and their constants
//                        into a ring of `stages` shared-memory slots;
//   warp 1 (one thread)  tcgen05.mma of each tile into one of two 128-column
//                        tensor-memory accumulators;
//   warps 2..9           the epilogue: each reads its 32-lane quadrant
//                        (warp % 4) and half of the columns of an accumulator
//                        with tcgen05.ld, evaluates coef * 2^(...) and sums.
// full[s]  : the tile in slot s has landed (TMA transaction bytes);
// empty[s] : slot s is free again (the MMA's commit + one arrival per
//            epilogue warp, which also read the slot's constants);
// accf[b]  : accumulator b holds a finished tile (MMA commit);
// acce[b]  : the epilogue has read accumulator b (one arrival per warp).
// Tile t uses slot t % stages (round t / stages) and accumulator t & 1 (use
// t >> 1); the k-th completion of a barrier has parity k & 1.
constexpr int kEpiWarps = 8;          // epilogue warps per accumulator
// Query tiles per CTA (RT). The epilogue's constants of a column, 8 bytes read
// from shared memory into every lane, bound it with one tile: a warp-wide
// 16-byte read takes 4 clocks of the SM's data path whatever its addresses, 8
// clocks per pair and scheduler against 6.5 of issue. With two tiles a thread
// holds a row of each and reads the constants once for both; one such CTA per
// SM (512 tensor-memory columns), whose 16 epilogue warps take the support
// tiles in turn, 8 each.
__host__ __device__ constexpr int tc_threads(int rt) { return 64 + 32 * kEpiWarps * rt; }
constexpr int kMaxStages = 4;

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait that also gives up once another role has failed. The thread
// sleeps in the barrier (suspend-time hint) until the phase completes or the
// hint runs out, so waiting warps take no issue slots from the epilogue; the
// whole wait is bounded by kWaitNs of the global timer.
constexpr uint64_t kWaitNs = 5ull * 1000 * 1000 * 1000;
__device__ __forceinline__ bool mbar_wait_or_fail(uint64_t *bar, uint32_t parity, const volatile int *fail)
{
    const uint32_t a = smem_u32(bar);
    uint64_t t0 = 0;
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity), "r"(20000u)
            : "memory");
        if (ok) return true;
        if (*fail) return false;
        const uint64_t now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > kWaitNs) return false;
    }
}

// 32 columns of one row: (columns j, j + 1) partial sums in two chains; the
// FP32 arithmetic runs on packed column pairs (f32x2), the same IEEE result in
// each lane as the scalar form. FACTORED: see the kernel.
template <bool FACTORED>
__device__ __forceinline__ void epi_quad(const uint32_t *rr, const ulonglong2 &x4, const ulonglong2 &c4,
                                         unsigned long long g2v, unsigned long long zc2, float nzc,
                                         unsigned long long &partA, unsigned long long &partB)
{
    const float cap = FACTORED ? nzc : 0.f;
    const unsigned long long xa = FACTORED ? x4.x : add_f32x2(x4.x, zc2), xb = FACTORED ? x4.y : add_f32x2(x4.y, zc2);
    float e0, e1, e2, e3;
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(rr[0]), __uint_as_float(rr[1])), g2v, xa), e0, e1);
    unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(rr[2]), __uint_as_float(rr[3])), g2v, xb), e2, e3);
    const unsigned long long k01 = pack_f32x2(ex2_approx(fminf(e0, cap)), ex2_approx(fminf(e1, cap)));
    const unsigned long long k23 = pack_f32x2(ex2_approx(fminf(e2, cap)), ex2_approx(fminf(e3, cap)));
    partA = fma_f32x2(c4.x, k01, partA);
    partB = fma_f32x2(c4.y, k23, partB);
}

template <int RT>
__global__ void __launch_bounds__(tc_threads(RT), RT == 1 ? 2 : 1)
    tc_rbf_kernel(const __grid_constant__ CUtensorMap mapZ, const __grid_constant__ CUtensorMap mapX, TcArgs a)
{
    extern __shared__ __align__(1024) unsigned char dsm_raw[];
    // 1024-byte alignment for the swizzled tiles
    unsigned char *dsm = reinterpret_cast<unsigned char *>(((uintptr_t)dsm_raw + 1023) & ~(uintptr_t)1023);
    const int S = a.stages;
    const size_t tile_all = (size_t)a.kblocks * kTileBytes;   // one tile, all k-blocks
    unsigned char *tileA = dsm;                               // the query tiles
    unsigned char *tileB = dsm + RT * tile_all;               // [S][kblocks][16 KiB]
    __shared__ __align__(8) uint64_t bar_q, bar_full[kMaxStages], bar_empty[kMaxStages], bar_accf[2],
        bar_acce[2], bar_drain;
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float s_xc[kMaxStages][kTile], s_coef[kMaxStages][kTile];
    __shared__ double s_acc[2 * RT][RT * kTile];   // the epilogue warps' row sums, by tile turn and column half
    __shared__ int s_fail, s_last;
    const volatile int *fail = &s_fail;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t q0 = (int64_t)blockIdx.x * (RT * kTile);
    if (tid == 0) {
        mbar_init(&bar_q, 1);
        for (int k = 0; k < kMaxStages; ++k) {
            mbar_init(&bar_full[k], 1);
            mbar_init(&bar_empty[k], 1 + kEpiWarps);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&bar_accf[k], 1);
            mbar_init(&bar_acce[k], kEpiWarps);
        }
        mbar_init(&bar_drain, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base)), "r"(2 * RT * kTile) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;
    const int64_t ntiles_all = (a.nsv + kTile - 1) / kTile;
    const int splits = gridDim.y;
    const int64_t tile0 = ntiles_all * (int64_t)blockIdx.y / splits;   // this CTA's first support tile
    const int64_t ntiles = ntiles_all * (int64_t)(blockIdx.y + 1) / splits - tile0;

    bool ok = true;
    int64_t issued = 0;         // producer: support tiles whose loads were issued
    bool q_issued = false;
    // epilogue warps: turn (support tiles t = turn, turn + RT, ..), column half
    // and 32-lane quadrant of tensor memory
    const int quad = warp & 3, half = ((warp - 2) >> 2) & 1, turn = (warp - 2) >> 3;
    const int my_row = quad * 32 + lane;                  // TMEM lane = query row in each tile
    double acc[RT];
#pragma unroll
    for (int i = 0; i < RT; ++i) acc[i] = 0.0;

    if (warp == 0) {
        // ---- producer
        if (lane == 0) {
            mbar_expect_tx(&bar_q, (uint32_t)(RT * tile_all));
            for (int i = 0; i < RT; ++i)
                for (int kb = 0; kb < a.kblocks; ++kb)
                    tma_load_2d(tileA + i * tile_all + (size_t)kb * kTileBytes, &mapZ, kb * kKB, (int)q0 + i * kTile, &bar_q);
            q_issued = true;
            for (int64_t t = 0; t < ntiles; ++t) {
                const int sl = (int)(t % S);
                const int64_t r = t / S;
                if (r >= 1 && !mbar_wait_or_fail(&bar_empty[sl], (uint32_t)((r - 1) & 1), fail)) {
                    ok = false;
                    break;
                }
                // the slot's last readers included the epilogue's generic loads
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                unsigned char *tb = tileB + (size_t)sl * tile_all;
                mbar_expect_tx(&bar_full[sl], (uint32_t)tile_all + 2 * kTile * 4);
                for (int kb = 0; kb < a.kblocks; ++kb)
                    tma_load_2d(tb + (size_t)kb * kTileBytes, &mapX, kb * kKB, (int)((tile0 + t) * kTile), &bar_full[sl]);
                bulk_load(s_xc[sl], a.xc + (tile0 + t) * kTile, kTile * 4, &bar_full[sl]);
                bulk_load(s_coef[sl], a.coef + (tile0 + t) * kTile, kTile * 4, &bar_full[sl]);
                issued = t + 1;
            }
        }
    } else if (warp == 1) {
        // ---- MMA issue: D[b] = Z_tile * X_tile^T over all K
        if (lane == 0) {
            ok = mbar_wait_or_fail(&bar_q, 0, fail);
            for (int64_t t = 0; ok && t < ntiles; ++t) {
                const int sl = (int)(t % S), b = (int)(t & 1);
                const int64_t r = t / S, u = t >> 1;
                if (!mbar_wait_or_fail(&bar_full[sl], (uint32_t)(r & 1), fail) ||
                    (u >= 1 && !mbar_wait_or_fail(&bar_acce[b], (uint32_t)((u - 1) & 1), fail))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const unsigned char *tb = tileB + (size_t)sl * tile_all;
                for (int i = 0; i < RT; ++i)
                for (int kb = 0; kb < a.kblocks; ++kb) {
                    const uint32_t dcol = tmem + (uint32_t)((b * RT + i) * kTile);
                    const uint32_t sa = smem_u32(tileA + i * tile_all + (size_t)kb * kTileBytes);
                    const uint32_t sb = smem_u32(tb + (size_t)kb * kTileBytes);
#pragma unroll
                    for (int ks = 0; ks < kKB / 16; ++ks) {
                        const uint64_t da = smem_desc_sw128(sa + ks * 32);
                        const uint64_t db = smem_desc_sw128(sb + ks * 32);
                        const uint32_t accum = (kb | ks) ? 1u : 0u;
                        asm volatile(
                            "{\n\t.reg .pred p;\n\t"
                            "setp.ne.b32 p, %4, 0;\n\t"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                            ::"r"(dcol), "l"(da), "l"(db), "r"(kIdesc), "r"(accum)
                            : "memory");
                    }
                }
                // both fire when these MMAs are done: the accumulator is
                // ready, and the MMA no longer reads the slot
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(&bar_accf[b])) : "memory");
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                             ::"r"(smem_u32(&bar_empty[sl])) : "memory");
            }
        }
    } else {
        // ---- epilogue
        // The row's scaled norm factors out of the sum:
        //   sum_j c_j 2^min(g2 dot_j + xc_j + zc, 0)
        //     = 2^zc sum_j c_j 2^min(g2 dot_j + xc_j, -zc),
        // one addition less per pair; 2^zc is applied once per tile. A warp
        // with a row whose 2^-zc would leave FP32 (-zc > 120) keeps the
        // per-pair form.
        const unsigned long long g2v = pack_f32x2(a.g2, a.g2);
        float nzc[RT];
        unsigned long long zc2[RT];
        bool factored[RT], all_factored = true;
        double row_scale[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
            const int64_t q = q0 + i * kTile + my_row;
            const float zc = (q < a.nq) ? a.zc[q] : 0.f;
            nzc[i] = -zc;
            zc2[i] = pack_f32x2(zc, zc);
            factored[i] = !__any_sync(0xffffffffu, nzc[i] > 120.f);
            all_factored &= factored[i];
            row_scale[i] = factored[i] ? exp2((double)zc) : 1.0;
        }
        for (int64_t t = turn; t < ntiles; t += RT) {
            const int sl = (int)(t % S), b = (int)(t & 1);
            const int64_t r = t / S, u = t >> 1;
            const bool w_ok = mbar_wait_or_fail(&bar_accf[b], (uint32_t)(u & 1), fail) &&
                              mbar_wait_or_fail(&bar_full[sl], (uint32_t)(r & 1), fail);
            if (!__all_sync(0xffffffffu, w_ok)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            unsigned long long part[RT][2];
#pragma unroll
            for (int i = 0; i < RT; ++i) part[i][0] = part[i][1] = pack_f32x2(0.f, 0.f);
            // 64 values per thread at once (one tile: the 64 columns of this
            // half; two: 32 columns of each), so that a wait for tensor memory
            // covers that many; the accumulator is free for the MMA once the
            // last of them are in registers
            constexpr int kCols = 64 / RT;
#pragma unroll
            for (int c0 = 0; c0 < kTile / 2; c0 += kCols) {
                uint32_t rr[64];
                const uint32_t addr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * RT * kTile + half * (kTile / 2) + c0);
                tmem_ld_x32(rr, addr);
                tmem_ld_x32(rr + 32, RT == 1 ? addr + 32 : addr + kTile);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (c0 + kCols == kTile / 2) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&bar_acce[b]);
                }
                const ulonglong2 *xs = reinterpret_cast<const ulonglong2 *>(&s_xc[sl][half * (kTile / 2) + c0]);
                const ulonglong2 *cs = reinterpret_cast<const ulonglong2 *>(&s_coef[sl][half * (kTile / 2) + c0]);
                if (all_factored) {
#pragma unroll
                    for (int v = 0; v < kCols / 4; ++v) {
                        const ulonglong2 x4 = xs[v], c4 = cs[v];   // the same address in every lane
#pragma unroll
                        for (int i = 0; i < RT; ++i)
                            epi_quad<true>(rr + i * kCols + 4 * v, x4, c4, g2v, zc2[i], nzc[i], part[i][0], part[i][1]);
                    }
                } else {
#pragma unroll
                    for (int v = 0; v < kCols / 4; ++v) {
                        const ulonglong2 x4 = xs[v], c4 = cs[v];
#pragma unroll
                        for (int i = 0; i < RT; ++i) {
                            if (factored[i])
                                epi_quad<true>(rr + i * kCols + 4 * v, x4, c4, g2v, zc2[i], nzc[i], part[i][0], part[i][1]);
                            else
                                epi_quad<false>(rr + i * kCols + 4 * v, x4, c4, g2v, zc2[i], nzc[i], part[i][0], part[i][1]);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                float pa0, pa1, pb0, pb1;
                unpack_f32x2(part[i][0], pa0, pa1);
                unpack_f32x2(part[i][1], pb0, pb1);
                acc[i] += (double)((pa0 + pa1) + (pb0 + pb1)) * row_scale[i];
            }
            // this warp is done with slot sl
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_empty[sl]);
        }
    }
    if (!ok && lane == 0) {
        s_fail = 1;
        atomicExch(a.err, 1);
    }
    __syncthreads();
    if (s_fail) {
        // let this CTA's outstanding asynchronous work finish (bounded)
        // before its shared and tensor memory are released
        if (warp == 1 && lane == 0) {
            // a commit tracks every earlier MMA of this thread
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         ::"r"(smem_u32(&bar_drain)) : "memory");
            (void)mbar_wait(&bar_drain, 0);
        }
        if (warp == 0 && lane == 0) {
            // loads in flight: at most the last `stages` tiles, one per slot
            for (int64_t t = issued > S ? issued - S : 0; t < issued; ++t)
                (void)mbar_wait(&bar_full[t % S], (uint32_t)((t / S) & 1));
            if (q_issued) (void)mbar_wait(&bar_q, 0);
        }
    } else {
        // a row's sums (by column half and tile turn) meet in shared memory, in
        // a fixed order; one epilogue thread per row then has its total
        if (warp >= 2) {
#pragma unroll
            for (int i = 0; i < RT; ++i) s_acc[2 * turn + half][i * kTile + my_row] = acc[i];
        }
        __syncthreads();
        const int row = tid - 64;                 // epilogue threads 0 .. RT kTile - 1
        const int64_t q = q0 + row;
        const bool owner = row >= 0 && row < RT * kTile;
        bool mine = owner && q < a.nq;
        double sum = 0.0;
        if (owner) {
            sum = s_acc[0][row];
#pragma unroll
            for (int k = 1; k < 2 * RT; ++k) sum += s_acc[k][row];
        }
        if (splits > 1) {
            if (mine) a.part[(size_t)blockIdx.y * a.nq + q] = sum;
            __threadfence();
            __syncthreads();
            if (tid == 0) s_last = atomicAdd(a.done + blockIdx.x, 1u) == (unsigned)splits - 1u;
            __syncthreads();
            if (s_last) {
                __threadfence();
                // the epilogue's two sets of threads add half of the splits each
                const int set = row >= RT * kTile, rw = set ? row - RT * kTile : row;
                const int64_t qq = q0 + rw;
                double v = 0.0;
                if (row >= 0 && qq < a.nq) {
                    const int k1 = set ? splits : splits / 2;
                    for (int k = set ? splits / 2 : 0; k < k1; ++k) v += __ldcg(a.part + (size_t)k * a.nq + qq);
                }
                if (row >= 0 && set) s_acc[0][rw] = v;
                __syncthreads();
                if (owner) sum = v + s_acc[0][row];
            } else {
                mine = false;
            }
        }
        if (mine) {
            const int32_t out_row = a.qrow[q];
            double v = sum + a.add_scalar;
            if (a.yq) v -= (double)a.yq[out_row];
            a.out[out_row] = v;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * RT * kTile)
                     : "memory");
    }
}

// ------------------------------------------------------------- preparation

// Dense BF16 rows (row-major, ld = d_pad, a multiple of 64) from CSR rows
// (list or all) and the scaled norms used by the epilogue; padding rows are
// zero. A warp per row, the row cleared with 16-byte stores (one CTA of 64
// threads per row: 29 us for 48,868 rows of 12 entries).
__global__ void k_densify(int64_t nrows, int64_t nrows_pad, int d_pad, const int32_t *list,
                          const int64_t *indptr, const int32_t *indices, const float *vmix,
                          const float *normf, float nscale, __nv_bfloat16 *dense, float *cnorm,
                          const double *coef_in, float *coef_out, int32_t *outrow, int out_by_row)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= nrows_pad) return;
    __nv_bfloat16 *dst = dense + (size_t)r * d_pad;
    for (int c = lane; c < d_pad / 8; c += 32) reinterpret_cast<uint4 *>(dst)[c] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    if (r < nrows) {
        const int64_t row = list ? list[r] : r;
        const int64_t p1 = indptr[row + 1];
        for (int64_t p = indptr[row] + lane; p < p1; p += 32) dst[indices[p]] = __float2bfloat16_rn(vmix[p]);
        if (lane == 0) {
            cnorm[r] = nscale * normf[row];
            if (coef_out) coef_out[r] = (float)coef_in[r];
            if (outrow) outrow[r] = out_by_row ? (int32_t)row : (int32_t)r;
        }
    } else if (lane == 0) {
        cnorm[r] = 0.f;
        if (coef_out) coef_out[r] = 0.f;
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

bool make_map(CUtensorMap *m, const void *base, int64_t rows, int d_pad)
{
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)d_pad, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)d_pad * 2};
    cuuint32_t box[2] = {(cuuint32_t)kKB, (cuuint32_t)kTile};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

}  // namespace

bool tc_rbf_supported(int d) { return d >= 1 && d <= kMaxKBlocks * kKB && encode_fn() != nullptr; }

namespace {

// consecutive 256-byte aligned pieces of a buffer (NULL base: sizes only)
struct Pieces {
    unsigned char *p;
    size_t used = 0;
    template <class T>
    T *take(size_t count)
    {
        T *r = reinterpret_cast<T *>(p + used);
        used += (count * sizeof(T) + 255) & ~(size_t)255;
        return p ? r : nullptr;
    }
};

int pad_cols(int d) { return (d + kKB - 1) / kKB * kKB; }
int64_t pad_rows(int64_t n) { return (std::max<int64_t>(n, 1) + kTile - 1) / kTile * kTile; }

// the support vectors' side: dense rows, scaled norms, coefficients
struct SvSide {
    __nv_bfloat16 *X;
    float *xc, *coef;
};
SvSide sv_side(Pieces &p, int64_t nsv, int d)
{
    const int64_t n = pad_rows(nsv);
    SvSide s;
    s.X = p.take<__nv_bfloat16>((size_t)n * pad_cols(d));
    s.xc = p.take<float>(n);
    s.coef = p.take<float>(n);
    return s;
}
struct QSide {
    __nv_bfloat16 *Z;
    float *zc;
    int32_t *qrow;
    int *err;
    unsigned *done;
    double *part;
    int splits, rt;
};
// Two CTAs share an SM: with fewer query tiles than that the support tiles are
// split (48,868 support vectors, 300 queries: 3 CTAs took 377 us), at least
// four tiles to a CTA and at most 64 CTAs to a query tile (the last one adds
// their sums, an FP64 addition of a warp per 64 cycles).
QSide q_side(Pieces &p, int64_t nq, int64_t nsv, int d, bool keep_order)
{
    int dev = 0, sms = 1;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 1;
    const int64_t n = pad_rows(nq), tiles = n / kTile, nt = pad_rows(nsv) / kTile;
    QSide s;
    // two query tiles per CTA once they give every SM one (d <= 128: their
    // shared memory)
    s.rt = !keep_order && (tiles + 1) / 2 >= sms && pad_cols(d) <= 2 * kKB ? 2 : 1;
    const int64_t ctas = (tiles + s.rt - 1) / s.rt, slots = (s.rt == 2 ? 1 : 2) * (int64_t)sms;
    s.splits = 1;
    if (!keep_order && ctas < slots) {
        s.splits = (int)std::max<int64_t>(1, std::min<int64_t>({slots / ctas, nt / 4, 64}));
    } else if (!keep_order) {
        // more CTAs than fit at once: the split, of at least 16 support tiles
        // a CTA, whose last wave is fullest (391 CTAs on 152 SMs, 2.6 waves:
        // 2.77 ms; split by 5, 12.9 waves: 2.52)
        double best = 1e9;
        for (int k = 1; k <= 8 && nt / k >= 16; ++k) {
            const double waves = (double)(ctas * k) / (double)slots;
            const double cost = std::ceil(waves) / waves + 0.005 * k;
            if (cost < best) {
                best = cost;
                s.splits = k;
            }
        }
    }
    s.Z = p.take<__nv_bfloat16>((size_t)n * pad_cols(d));
    s.zc = p.take<float>(n);
    s.qrow = p.take<int32_t>(n);
    s.err = p.take<int>(1 + (size_t)tiles);   // the error word, then the tiles' counters
    s.done = reinterpret_cast<unsigned *>(s.err) + 1;
    s.part = p.take<double>(s.splits > 1 ? (size_t)s.splits * nq : 0);
    return s;
}

}  // namespace

size_t tc_rbf_sv_bytes(int64_t nsv, int d)
{
    Pieces p{nullptr};
    sv_side(p, nsv, d);
    return p.used;
}

size_t tc_rbf_workspace_bytes(const RbfContract &c)
{
    Pieces p{nullptr};
    q_side(p, c.nq, c.nsv, c.d, c.keep_order != 0);
    return p.used;
}

// The support vectors' side of a contraction into `sv` (tc_rbf_sv_bytes).
cudaError_t tc_rbf_prepare_sv(const RbfContract &c, void *sv, cudaStream_t st)
{
    Pieces p{static_cast<unsigned char *>(sv)};
    const SvSide s = sv_side(p, c.nsv, c.d);
    const int64_t n = pad_rows(c.nsv);
    const float nscale = (float)(-c.gamma) * 1.4426950408889634f;
    k_densify<<<(unsigned)(n / 8), 256, 0, st>>>(c.nsv, n, pad_cols(c.d), c.sv, c.x_indptr, c.x_indices, c.x_values,
                                                 c.x_normf, nscale, s.X, s.xc, c.coef, s.coef, nullptr, 0);
    return cudaGetLastError();
}

// Same contract as launch_rbf_contract (MODE_MIXED inputs: vmix values and
// FP32 norms), on the tensor cores. `sv` was filled by tc_rbf_prepare_sv;
// `ws` must hold tc_rbf_workspace_bytes.
cudaError_t launch_rbf_contract_tc(const RbfContract &c, const void *sv, void *ws, int *err_host, cudaStream_t st)
{
    *err_host = 0;
    if (c.nq <= 0) return cudaSuccess;
    if (c.nsv <= 0) return cudaErrorInvalidValue;   // (no support vectors: every sum is zero)
    const int d_pad = pad_cols(c.d);
    const int kblocks = d_pad / kKB;
    if (kblocks > kMaxKBlocks) return cudaErrorInvalidValue;
    const int64_t nq_pad = pad_rows(c.nq), tiles = nq_pad / kTile;
    Pieces pw{static_cast<unsigned char *>(ws)}, ps{static_cast<unsigned char *>(const_cast<void *>(sv))};
    const QSide q = q_side(pw, c.nq, c.nsv, c.d, c.keep_order != 0);
    const SvSide x = sv_side(ps, c.nsv, c.d);
    const float L2E = 1.4426950408889634f;
    const float nscale = (float)(-c.gamma) * L2E;
    cudaError_t e = cudaMemsetAsync(q.err, 0, sizeof(int) * (1 + (size_t)tiles), st);
    if (e != cudaSuccess) return e;
    k_densify<<<(unsigned)(nq_pad / 8), 256, 0, st>>>(c.nq, nq_pad, d_pad, c.q, c.z_indptr, c.z_indices, c.z_values,
                                                      c.z_normf, nscale, q.Z, q.zc, nullptr, nullptr, q.qrow, c.out_by_row);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    CUtensorMap mz, mx;
    if (!make_map(&mz, q.Z, nq_pad, d_pad) || !make_map(&mx, x.X, pad_rows(c.nsv), d_pad)) return cudaErrorInvalidValue;
    TcArgs a;
    a.nq = c.nq;
    a.nsv = c.nsv;
    a.kblocks = kblocks;
    a.zc = q.zc;
    a.xc = x.xc;
    a.coef = x.coef;
    a.g2 = 2.0f * (float)c.gamma * L2E;
    a.qrow = q.qrow;
    a.yq = c.yq;
    a.add_scalar = c.add_scalar;
    a.out = c.out;
    a.err = q.err;
    a.part = q.part;
    a.done = q.done;
    if (q.rt == 2) {
        // two query tiles + 4 slots at d <= 64, 2 at d <= 128; one CTA per SM
        a.stages = kblocks == 1 ? 4 : 2;
        const size_t smem = std::max<size_t>((size_t)(2 + a.stages) * kblocks * kTileBytes + 1024, 120 * 1024);
        e = cudaFuncSetAttribute(tc_rbf_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        tc_rbf_kernel<2><<<dim3((unsigned)((tiles + 1) / 2), (unsigned)q.splits), tc_threads(2), smem, st>>>(mz, mx, a);
    } else {
        // query tile + a ring of support tiles: 4 slots at d <= 64, else 2; at
        // least 80 KiB so that at most 2 CTAs share an SM: their 2 x 256
        // tensor-memory columns then fit the SM's 512 without waiting
        a.stages = kblocks == 1 ? 4 : 2;
        const size_t smem = std::max<size_t>((size_t)(1 + a.stages) * kblocks * kTileBytes + 1024, 80 * 1024);
        e = cudaFuncSetAttribute(tc_rbf_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        tc_rbf_kernel<1><<<dim3((unsigned)tiles, (unsigned)q.splits), tc_threads(1), smem, st>>>(mz, mx, a);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return cudaMemcpyAsync(err_host, q.err, sizeof(int), cudaMemcpyDeviceToHost, st);
}


// SFU exp2 rate (microbenchmark for the contraction's roofline): every thread
// runs 8 independent chains of ex2.approx, the instruction of the epilogue.
__global__ void k_sfu_ex2(int iters, float seed, float *sink)
{
    float a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = seed * (float)(j + 1) * 1e-3f - (float)(threadIdx.x & 7) * 1e-4f;
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float r;
            asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a[j]));
            a[j] = r * -0.5f;   // stays in (-1, 1): no overflow, no denormals
        }
    }
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) acc += a[j];
    if (acc == 12345.f) sink[blockIdx.x] = acc;   // keeps the loop alive
}

cudaError_t measure_sfu_ex2(double *ops_per_s, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int blocks = sms * 8, threads = 256, iters = 4096;
    float *sink = nullptr;
    if ((e = cudaMallocAsync(&sink, sizeof(float) * blocks, st)) != cudaSuccess) return e;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    k_sfu_ex2<<<blocks, threads, 0, st>>>(iters / 8, 0.5f, sink);   // warm-up
    cudaEventRecord(e0, st);
    k_sfu_ex2<<<blocks, threads, 0, st>>>(iters, 0.5f, sink);
    cudaEventRecord(e1, st);
    e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFreeAsync(sink, st);
    if (e == cudaSuccess) *ops_per_s = (double)blocks * threads * iters * 8 / (ms * 1e-3);
    return e;
}

}  // namespace svmgb
