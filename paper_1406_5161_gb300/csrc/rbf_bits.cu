// Decision values of binary rows (every stored value 1.0, d <= 256):
//   out[q] = sum_k coef_k exp(-gamma |x_k xor z_q|) + add_scalar,
// the contraction of rbf_contract.cu with both sides as bit masks: the squared
// distance is the popcount of an XOR and K one of at most 257 table values.
//
// One FP64 multiply-add per pair would bound it (an operation of a warp takes
// 64 cycles of its scheduler's FP64 pipe: 217 us for 10,000 queries against
// 11,700 support vectors, and the masked column gather before this one took
// 561 us in all). Here the products are integers: K in Q63, |coef| scaled to
// 62 bits by the largest coefficient's exponent, the product's upper 96 bits
// added to a 128-bit sum. Each term is exact to 2^-61 of the largest
// coefficient and the sum is exact, so it does not depend on the order or on
// the split, and it is rounded once to a double. Per pair about 4 XORs, 3
// popcounts (three words of a row through one carry-save adder), a table read
// and 15 integer operations: bound by popcount and issue.
//
// A thread holds one support vector's mask at a time and kTQ sums; a CTA's
// sums meet by shuffles and shared memory, those of the CTAs that share a
// query tile in a workspace (the last CTA to finish adds them).
#include <algorithm>

#include <cuda_runtime.h>

#include "fp64_math.cuh"
#include "svm_internal.cuh"

namespace svmgb {
namespace {

constexpr int kBThreads = 256;
constexpr int kBWarps = kBThreads / 32;
constexpr int kTQ = 8;
constexpr int kTabMax = 257;   // d <= 256

// What the sum needs to know of the coefficients (zeroed).
struct CoefInfo {
    int emax;       // largest exponent field of a finite one (subnormals count as 1)
    int infinite;   // 1: a positive one is infinite, 2: a negative one
};

// Rows list[0 .. m) (or 0 .. m-1) as bit masks of W words; info: of coef
// (NULL: none).
__global__ void k_mask_rows(int64_t m, int W, const int32_t *list, const int64_t *indptr, const int32_t *indices,
                            uint32_t *bits, const double *coef, CoefInfo *info)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int e = 0;
    if (k < m) {
        const int64_t r = list ? list[k] : k;
        uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const int64_t p1 = indptr[r + 1];
        for (int64_t p = indptr[r]; p < p1; ++p) {
            const int c = indices[p];
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] |= (c >> 5) == j ? 1u << (c & 31) : 0u;
        }
        uint4 *dst = reinterpret_cast<uint4 *>(bits + (size_t)k * W);
        dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
        if (W == 8) dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        if (coef) {
            const uint64_t b = double_to_bits(coef[k]);
            e = max((int)(b >> 52) & 0x7ff, 1);
            if (e == 0x7ff) {
                atomicOr(&info->infinite, b >> 63 ? 2 : 1);
                e = 0;
            }
        }
    }
    if (coef) {
        e = __reduce_max_sync(0xffffffffu, e);
        if ((threadIdx.x & 31) == 0 && e > *(volatile int *)&info->emax) atomicMax(&info->emax, e);
    }
}

struct BitsArgs {
    int64_t nq, nsv;
    const uint32_t *xbits, *zbits;
    const double *coef;
    const CoefInfo *info;
    const double *ktab;
    int ktab_len;
    double add_scalar;
    double *out;
    uint4 *part;       // [splits][nq] partial sums (128 bits each)
    unsigned *done;    // per query tile (zeroed)
};

__device__ __forceinline__ XdAcc xd_of(uint4 v)
{
    XdAcc a;
    a.w0 = v.x; a.w1 = v.y; a.w2 = v.z; a.w3 = v.w;
    return a;
}

template <int N>
__device__ __forceinline__ int popc_words(const uint32_t *x)
{
    // three words: their bitwise sum and carry, two popcounts instead of three
    if constexpr (N >= 3) {
        const uint32_t s = x[0] ^ x[1] ^ x[2];
        const uint32_t c = (x[0] & x[1]) | (x[2] & (x[0] | x[1]));
        return __popc(s) + 2 * __popc(c) + popc_words<N - 3>(x + 3);
    } else if constexpr (N == 2) {
        return __popc(x[0]) + __popc(x[1]);
    } else if constexpr (N == 1) {
        return __popc(x[0]);
    } else {
        return 0;
    }
}

template <int W>
__global__ void __launch_bounds__(kBThreads) rbf_bits_kernel(BitsArgs a)
{
    __shared__ uint64_t tab[kTabMax];
    __shared__ __align__(16) uint32_t zq[kTQ][W];
    __shared__ uint4 red[kBWarps][kTQ];
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t q0 = (int64_t)blockIdx.x * kTQ;
    const int nt = (int)min((int64_t)kTQ, a.nq - q0);
    // K in Q63 (1 = 2^63; truncated below 2^-63)
    for (int k = tid; k < kTabMax; k += kBThreads) {
        uint64_t v = 0;
        if (k < a.ktab_len) {
            const uint64_t b = double_to_bits(a.ktab[k]);
            const int sh = (int)(b >> 52) - 1012;   // m 2^(e - 1075 + 63)
            const uint64_t m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
            v = (b >> 52) == 0 ? 0ull : (sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull));
        }
        tab[k] = v;
    }
    for (int k = tid; k < kTQ * W; k += kBThreads)
        zq[k / W][k % W] = k / W < nt ? a.zbits[(size_t)(q0 + k / W) * W + k % W] : 0u;
    __syncthreads();
    const int emax = a.info->emax;
    const int splits = gridDim.y;
    const int64_t k1 = a.nsv * (int64_t)(blockIdx.y + 1) / splits;
    XdAcc acc[kTQ];
#pragma unroll
    for (int q = 0; q < kTQ; ++q) acc[q] = xd_zero();
    for (int64_t k = a.nsv * (int64_t)blockIdx.y / splits + tid; k < k1; k += kBThreads) {
        uint32_t x[W];
        const uint4 *xs = reinterpret_cast<const uint4 *>(a.xbits + (size_t)k * W);
#pragma unroll
        for (int j = 0; j < W / 4; ++j) {
            const uint4 v = __ldg(xs + j);
            x[4 * j] = v.x; x[4 * j + 1] = v.y; x[4 * j + 2] = v.z; x[4 * j + 3] = v.w;
        }
        // |coef| 2^(1084 - emax), below 2^62 (infinite ones: see the end)
        const uint64_t cb = double_to_bits(a.coef[k]);
        const int field = (int)(cb >> 52) & 0x7ff, sh = emax - max(field, 1) - 9;
        const uint64_t m = (cb & 0x000fffffffffffffull) | (field ? 0x0010000000000000ull : 0ull);
        const uint64_t cq = field == 0x7ff ? 0ull : (sh <= 0 ? m << -sh : (sh < 64 ? m >> sh : 0ull));
        const uint32_t neg = (uint32_t)((int32_t)(uint32_t)(cb >> 32) >> 31);
#pragma unroll
        for (int q = 0; q < kTQ; ++q) {
            uint32_t y[W];
#pragma unroll
            for (int j = 0; j < W / 4; ++j) {
                const uint4 v = *reinterpret_cast<const uint4 *>(&zq[q][4 * j]);
                y[4 * j] = x[4 * j] ^ v.x;
                y[4 * j + 1] = x[4 * j + 1] ^ v.y;
                y[4 * j + 2] = x[4 * j + 2] ^ v.z;
                y[4 * j + 3] = x[4 * j + 3] ^ v.w;
            }
            const uint64_t kv = tab[popc_words<W>(y)];
            const unsigned __int128 p = (unsigned __int128)cq * kv;
            // the upper 96 bits, complemented for a negative coefficient: one
            // unit (2^-61 of the largest coefficient's K) below its negation
            xd_add4(acc[q], (uint32_t)(p >> 32) ^ neg, (uint32_t)(p >> 64) ^ neg, (uint32_t)(p >> 96) ^ neg, neg);
        }
    }
#pragma unroll
    for (int q = 0; q < kTQ; ++q) {
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            XdAcc b;
            b.w0 = __shfl_xor_sync(0xffffffffu, acc[q].w0, off);
            b.w1 = __shfl_xor_sync(0xffffffffu, acc[q].w1, off);
            b.w2 = __shfl_xor_sync(0xffffffffu, acc[q].w2, off);
            b.w3 = __shfl_xor_sync(0xffffffffu, acc[q].w3, off);
            xd_add(acc[q], b);
        }
        if (lane == 0) red[warp][q] = make_uint4(acc[q].w0, acc[q].w1, acc[q].w2, acc[q].w3);
    }
    __syncthreads();
    XdAcc sum = xd_zero();
    if (tid < nt) {
        for (int w = 0; w < kBWarps; ++w) xd_add(sum, xd_of(red[w][tid]));
    }
    if (splits > 1) {
        if (tid < nt) a.part[(size_t)blockIdx.y * a.nq + q0 + tid] = make_uint4(sum.w0, sum.w1, sum.w2, sum.w3);
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(a.done + blockIdx.x, 1u) == (unsigned)splits - 1u;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        // a warp per query: its lanes add the splits
        for (int q = warp; q < nt; q += kBWarps) {
            XdAcc v = xd_zero();
            for (int k = lane; k < splits; k += 32) xd_add(v, xd_of(__ldcg(a.part + (size_t)k * a.nq + q0 + q)));
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) {
                XdAcc b;
                b.w0 = __shfl_xor_sync(0xffffffffu, v.w0, off);
                b.w1 = __shfl_xor_sync(0xffffffffu, v.w1, off);
                b.w2 = __shfl_xor_sync(0xffffffffu, v.w2, off);
                b.w3 = __shfl_xor_sync(0xffffffffu, v.w3, off);
                xd_add(v, b);
            }
            if (lane == 0) red[0][q] = make_uint4(v.w0, v.w1, v.w2, v.w3);
        }
        __syncthreads();
        if (tid < nt) sum = xd_of(red[0][tid]);
    }
    // the sum counts units of 2^(emax - 1115) (rounded to 53 bits where no
    // exponent can leave the normal range, then scaled)
    if (tid < nt) {
        double v = ldexp(xd_round(sum, -64), emax - 1115 + 64);
        // (every K is positive, so infinite coefficients alone decide)
        if (const int inf = a.info->infinite)
            v = bits_to_double(inf == 1 ? 0x7ff0000000000000ull : (inf == 2 ? 0xfff0000000000000ull : 0x7ff8000000000000ull));
        a.out[q0 + tid] = v + a.add_scalar;
    }
}

struct Plan {
    int W, splits;
    int64_t tiles;
    size_t xbits, zbits, head, part;   // bytes of the pieces of the workspace
};
Plan plan_of(const RbfContract &c)
{
    int dev = 0, sms = 1;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 1;
    Plan p;
    p.W = c.d <= 128 ? 4 : 8;
    p.tiles = (c.nq + kTQ - 1) / kTQ;
    // as in rbf_contract.cu: every SM its three CTAs as long as each thread
    // has a support vector, eight waves of them while it keeps four
    const int64_t full = 3 * (int64_t)sms, chunks = std::max<int64_t>(1, (c.nsv + kBThreads - 1) / kBThreads);
    p.splits = (int)std::max(std::min((full + p.tiles - 1) / p.tiles, chunks),
                             std::min((8 * full + p.tiles - 1) / p.tiles, (chunks + 3) / 4));
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    p.xbits = up(4 * (size_t)p.W * std::max<int64_t>(c.nsv, 1));
    p.zbits = up(4 * (size_t)p.W * c.nq);
    p.head = up(sizeof(CoefInfo) + sizeof(unsigned) * (size_t)p.tiles);
    p.part = up(p.splits > 1 ? 16 * (size_t)p.splits * c.nq : 0);
    return p;
}

}  // namespace

// K in Q63 is as exact as a double down to 2^-11: only kernels whose smallest
// table value (the largest distance) is at least that.
bool rbf_bits_supported(const RbfContract &c)
{
    if (!(c.gamma * (double)(c.ktab_len - 1) <= 7.5)) return false;
    return c.mode == MODE_BINARY && c.d <= 256 && !c.keep_order && !c.out_by_row && !c.yq && !c.accumulate && !c.q;
}

size_t rbf_bits_workspace_bytes(const RbfContract &c)
{
    const Plan p = plan_of(c);
    return p.xbits + p.zbits + p.head + p.part;
}

cudaError_t launch_rbf_bits(const RbfContract &c, void *ws, cudaStream_t st)
{
    if (c.nq <= 0) return cudaSuccess;
    const Plan p = plan_of(c);
    unsigned char *w = static_cast<unsigned char *>(ws);
    uint32_t *xbits = reinterpret_cast<uint32_t *>(w);
    uint32_t *zbits = reinterpret_cast<uint32_t *>(w + p.xbits);
    CoefInfo *head = reinterpret_cast<CoefInfo *>(w + p.xbits + p.zbits);
    cudaError_t e = cudaMemsetAsync(head, 0, sizeof(CoefInfo) + sizeof(unsigned) * (size_t)p.tiles, st);
    if (e != cudaSuccess) return e;
    if (c.nsv > 0)
        k_mask_rows<<<(unsigned)((c.nsv + 127) / 128), 128, 0, st>>>(c.nsv, p.W, c.sv, c.x_indptr, c.x_indices, xbits,
                                                                     c.coef, head);
    k_mask_rows<<<(unsigned)((c.nq + 127) / 128), 128, 0, st>>>(c.nq, p.W, nullptr, c.z_indptr, c.z_indices, zbits,
                                                                nullptr, nullptr);
    BitsArgs a;
    a.nq = c.nq;
    a.nsv = c.nsv;
    a.xbits = xbits;
    a.zbits = zbits;
    a.coef = c.coef;
    a.info = head;
    a.ktab = c.ktab;
    a.ktab_len = c.ktab_len;
    a.add_scalar = c.add_scalar;
    a.out = c.out;
    a.done = reinterpret_cast<unsigned *>(head + 1);
    a.part = reinterpret_cast<uint4 *>(w + p.xbits + p.zbits + p.head);
    const dim3 grid((unsigned)p.tiles, (unsigned)p.splits);
    if (p.W == 4) rbf_bits_kernel<4><<<grid, kBThreads, 0, st>>>(a);
    else rbf_bits_kernel<8><<<grid, kBThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace svmgb
