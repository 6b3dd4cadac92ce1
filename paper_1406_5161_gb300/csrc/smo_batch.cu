// Batched SMO: many independent training jobs over one shared sample matrix
// in one persistent launch (one-vs-one subproblems, hyper-parameter grids).
//
// The grid is a set of thread-block clusters; each cluster takes the next
// job from a device work-list (an atomic counter), splits the job's rows
// over its CTAs and runs the job's SMO steps (Algorithm 1: Eqs. fup,
// bminmax, kktterm, alphaup) exactly as the single-job fused step does:
// target rows in shared memory, the FP64 pair step on warp 0 overlapped with
// the row sums of warps 1.., FP64 f updates, integer selection keys. The
// candidate exchange stays inside the cluster (asynchronous stores),
// so clusters never wait on one another and need no co-residency. When a
// job converges, the cluster reduces b (Section III-A) and the objective,
// writes the job's result and takes the next job.
//
// Rows of a job are ids into the shared matrix; the job's labels, alpha, f
// and index sets live in concatenated per-job arrays. Dense inputs in the
// mixed-precision mode are read from a BF16 row-major copy (2 bytes per
// value instead of 8 for index + value).
#include <cuda_bf16.h>

#include <type_traits>

#include "batch_status.cuh"
#include "smo_step.cuh"

namespace svmgb {
namespace smo {
namespace {

__device__ __forceinline__ unsigned ld_acquire_sys_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_volatile_i32(const int *p)
{
    return *reinterpret_cast<const volatile int *>(p);
}
__device__ __forceinline__ void st_release_sys_i32(int *p, int v)
{
    asm volatile("st.release.sys.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// bulk copy global -> this CTA's shared memory, counted on an mbarrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async;" ::: "memory"); }

struct __align__(16) BatchFinish {
    double sum_a, sum_ayfy, sum_f0;
    long long n0, nsv;
    int pad[2];
};

// limit of every wait of the kernel
constexpr int64_t kWaitNs = 10ll * 1000 * 1000 * 1000;

// 16 k-steps x 32 lanes of packed BF16 target pairs (uint2)
constexpr size_t kFragBytes = (size_t)16 * 32 * sizeof(uint2);

// What a step needs of a candidate: the first 48 bytes of its two sides.
struct __align__(16) SideHead {
    double f, a, nrm;
    int64_t p0;
    int32_t i, len, y, owner;
};
static_assert(sizeof(SideHead) == 48 && offsetof(SideHead, p0) == offsetof(Side, p0) && offsetof(SideHead, i) == offsetof(Side, i) &&
              offsetof(SideHead, len) == offsetof(Side, len) && offsetof(SideHead, y) == offsetof(Side, y), "SideHead is Side's head");
struct CandSlot {
    SideHead up, low;
};

struct BatchShared {
    Side wup[kWarps], wlow[kWarps];
    unsigned long long wkup[kWarps], wklow[kWarps];
    int wiup[kWarps], wilow[kWarps];
    CandSlot xc[2][kMaxCluster];   // every CTA's candidate, by epoch parity
    unsigned long long xbar[2];    // mbarriers of the two parities
    Side none[2];                  // empty I_up / I_low sides
    ResultArea res;
    BatchFinish fin[kMaxCluster];  // cluster leader: its CTAs' partial sums
    BatchFinish wfin[kWarps];
    double du, dl, au_new, al_new;
    unsigned char st_u, st_l;
    PairPre pre;
    unsigned long long stage_bar[kWarps];   // packed units: a row warp's unit has landed
    int bad;                                // a wait of the CTA, from the job's end on of the cluster, gave up
    int stop;                               // the gap is closed, the step is not taken
    int job;
};
// with the FP64 mode's table of the exponential, within what the launch plans
// (svm_api.cu) leave for static shared memory
static_assert(sizeof(BatchShared) + sizeof(uint64_t) * kExpfxTabLen <= 12288 - 64, "static shared memory of the batch kernel");

template <int MODE, int LPR>
__global__ void __launch_bounds__(kThreads, 1) smo_batch_kernel(BatchArgs B)
{
    using Tgt = typename RowMath<MODE>::Tgt;
    using Acc = typename RowMath<MODE>::Acc;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ BatchShared sh;
    // FP64: 2^(-j/256) in Q63 for the fixed-point exp
    __shared__ uint64_t expfx_s[MODE == MODE_FP64 ? kExpfxTabLen : 1];
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int csize = (int)cluster.num_blocks();
    const int crank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int dmax = B.d;   // target buffers hold this many columns
    const int maxnnz = B.maxnnz > 0 ? B.maxnnz : 1;
    const SmoLayout L = smo_layout(MODE, dmax, B.ktab_len, maxnnz, 0, 0, 0);
    Tgt *tbuf = reinterpret_cast<Tgt *>(dsm + L.tgt);
    int *tcol = reinterpret_cast<int *>(dsm + L.tcol);
    double *ktab = reinterpret_cast<double *>(dsm + L.ktab);
    const double *rtab = ktab + B.ktab_len;
    uint2 *frag = reinterpret_cast<uint2 *>(dsm + L.total);   // mixed: the tiles' target fragments
    uint32_t *kdir = reinterpret_cast<uint32_t *>(dsm + L.total + (MODE == MODE_MIXED ? kFragBytes : 0));
    if constexpr (MODE == MODE_FP64) {
        for (int c = tid; c < kExpfxTabLen; c += kThreads) expfx_s[c] = kExpfxTab[c];   // ordered by the cluster sync below
    }
    // packed rows (dense BF16 on the tensor cores): each row warp streams its
    // units of 32 rows through a stage of its own in shared memory
    constexpr bool PACK_MODE = MODE == MODE_MIXED && LPR == 16;
    unsigned char *stage0 = reinterpret_cast<unsigned char *>(
        ((uintptr_t)(kdir + B.kdir_words) + 127) & ~(uintptr_t)127);
    uint32_t stage_parity = 0;
    if (tid == 0) {
        for (int w = 0; w < kWarps; ++w) mbar_init(smem_u32(&sh.stage_bar[w]), 1);
        mbar_init(smem_u32(&sh.xbar[0]), 1);
        mbar_init(smem_u32(&sh.xbar[1]), 1);
        side_empty(sh.none[0], true);
        side_empty(sh.none[1], false);
        sh.bad = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_proxy();
    }
    cluster.sync();   // the barriers exist before any CTA of the cluster sends
    unsigned epoch = 0;

    for (;;) {
        // ---- next job from the work-list, broadcast to the cluster; none once
        //      a wait of this cluster gave up (agreed on at the end of that
        //      job): other clusters, or the host, take what is left
        if (crank == 0 && tid == 0) {
            int j = INT_MAX;
            if (sh.bad) {
            } else if (!B.ring) {
                j = atomicAdd(B.next_job, 1);
                if (j >= B.njobs) j = INT_MAX;
            } else {
                // server: wait (bounded by the idle limit) for a published slot
                const uint64_t t0 = global_ns();
                for (;;) {
                    const unsigned tail = ld_acquire_sys_u32(B.ring_tail);
                    const unsigned head = (unsigned)atomicAdd(B.next_job, 0);
                    if (head < tail) {
                        if ((unsigned)atomicCAS(B.next_job, (int)head, (int)(head + 1)) == head) {
                            j = ld_volatile_i32(B.ring + (head % (unsigned)B.ring_cap));
                            break;
                        }
                        continue;
                    }
                    if (ld_volatile_i32(B.shutdown)) break;
                    if (global_ns() - t0 > (uint64_t)B.idle_ns) break;
                    __nanosleep(2000);
                }
            }
            for (int r = 0; r < csize; ++r) *cluster.map_shared_rank(&sh.job, r) = j;
        }
        cluster.sync();
        const int job = sh.job;
        if (job == INT_MAX) break;
        const BatchJobDev J = B.jobs[job];
        // the job's matrix (shared by all jobs of a batch, own per served job)
        const int d = J.d;
        const bool dense = J.dense != 0;
        const int64_t *indptr = J.indptr;
        const int32_t *indices = J.indices;
        const float *values = J.values;
        const float *vmix = J.vmix;
        const __nv_bfloat16 *dmat = J.dmat;
        const double *norm = J.norm;
        const float *normf = J.normf;
        const int m = J.nrows;
        const int8_t *yj = J.y;
        double *aj = J.alpha;
        double *fj = J.f;
        uint8_t *sj = J.status;
        const int lo = (int)((int64_t)m * crank / csize);
        const int hi = (int)((int64_t)m * (crank + 1) / csize);
        const double C = J.C, gamma = J.gamma;
        const float gammaf = (float)gamma;
        const double snap = 1e-12 * C, c_snap = C - snap;
        const double thr = 2.0 * J.tau;
        const int32_t *rows = J.rows;
        // kernel-row cache of the cluster (FP64): row r's values at [r * kc_ld,
        // + m), each CTA its own rows' part; a bit per row that is stored,
        // kept alike in every CTA's shared memory
        constexpr bool KC_MODE = MODE == MODE_FP64;
        const int64_t kc_ld = ((int64_t)m + 31) & ~(int64_t)31;
        const bool kc_on = KC_MODE && B.kc && m <= 32 * B.kdir_words && (int64_t)m * kc_ld * 8 <= B.kc_stride;
        double *kc = kc_on ? reinterpret_cast<double *>(static_cast<unsigned char *>(B.kc) + (size_t)(blockIdx.x / csize) * B.kc_stride)
                       : nullptr;
        if (kc_on) {
            for (int w = tid; w < (m + 31) / 32; w += kThreads) kdir[w] = 0;
        }

        // FP64 with exact inner products (J.xd.on): target entries hold (m, b)
        // pairs as in the single-solve kernel; an absent value m = 0, b = tmin
        const bool xd = MODE == MODE_FP64 && J.xd.on;
        const int xd_tmin = J.xd.tmin, xd_bias = J.xd.bias, xd_unit = J.xd.unit;
        Tgt tclear;
        tgt_clear<MODE>(tclear);
        if constexpr (MODE == MODE_FP64) {
            if (xd) tclear = make_double2(__hiloint2double(xd_tmin, 0), __hiloint2double(xd_tmin, 0));
        }
        // ---- job set-up: tables, empty target buffers, and alpha = 0, f = -y
        //      unless an earlier launch left them after iter0 steps (the
        //      selection pass below then finds the pair that one had chosen)
        for (int c = tid; c < 2 * dmax; c += kThreads) tbuf[c] = tclear;
        if constexpr (MODE == MODE_BINARY) {
            for (int k = tid; k < B.ktab_len; k += kThreads) {
                const double kv = exp(-gamma * (double)k);
                const double eta = 2.0 - 2.0 * kv;
                ktab[k] = kv;
                ktab[B.ktab_len + k] = eta > 1e-12 ? 1.0 / eta : 0.0;
            }
        }
        for (int r = lo + tid; r < hi && (MODE != MODE_FP64 || J.iter0 == 0); r += kThreads) {
            const int8_t yr = yj[r];
            aj[r] = 0.0;
            fj[r] = -(double)yr;
            sj[r] = (uint8_t)(st_of(yr, 0.0, 1.0) | (yr > 0 ? 0x80 : 0));
        }
        // This CTA's rows in the order the tensor cores' fragments read them:
        // unit u (32 rows), tile q, 32-column block b, half h, lane: the 8
        // values of row 32 u + 16 q + 8 h + lane / 4 at columns 32 b + 8
        // (lane & 3). A unit is one bulk copy, and its reads have no bank
        // conflict; gathered row by row from the matrix in every step, the
        // warps waited for loads 57% of the time (long scoreboard) and a round
        // of 15 x 32 rows took 7 us.
        const int units = (hi - lo + 31) / 32;
        const uint32_t unit_bytes = 64u * (uint32_t)d;
        unsigned char *pk = nullptr;
        bool packed = false;
        if constexpr (PACK_MODE) {
            packed = dense && B.pack && (d & 31) == 0 && d <= 256 && (int64_t)units * unit_bytes <= B.pack_stride &&
                     unit_bytes <= (uint32_t)B.stage_bytes;
            if (packed) {
                pk = static_cast<unsigned char *>(B.pack) + (size_t)blockIdx.x * B.pack_stride;
                const int nb = d >> 5, per = nb * 128;   // 16-byte pieces of a unit
                for (int k = tid; k < units * per; k += kThreads) {
                    const int ln = k & 31, h = (k >> 5) & 1, qb = (k >> 6) % (2 * nb), u = k / per;
                    const int r = lo + 32 * u + 16 * (qb / nb) + 8 * h + (ln >> 2);
                    uint4 v = make_uint4(0, 0, 0, 0);
                    if (r < hi)
                        v = __ldg(reinterpret_cast<const uint4 *>(dmat + (size_t)rows[r] * d + 32 * (qb % nb) + 8 * (ln & 3)));
                    reinterpret_cast<uint4 *>(pk)[k] = v;
                }
                fence_async_proxy();   // the bulk copies read them
            }
        }
        __syncthreads();
        const int stage_warps = packed ? B.stage_warps : 0;
        unsigned char *stage = stage0 + (size_t)(warp - 1) * B.stage_bytes;
        const uint32_t stage_bar = smem_u32(&sh.stage_bar[warp]);
        bool in_flight = false;   // a unit is on its way into this warp's stage
        auto issue_unit = [&](int u) {
            if (lane == 0) {
                mbar_arrive_expect_tx(stage_bar, unit_bytes);
                bulk_load(smem_u32(stage), pk + (size_t)u * unit_bytes, unit_bytes, stage_bar);
            }
            in_flight = true;
        };
        auto wait_unit = [&]() {
            if (!in_flight) return;
            // (for the copy itself, whatever else failed: none is in flight
            // when the CTA leaves)
            const int bad = mbar_wait_bounded(stage_bar, stage_parity, kWaitNs, nullptr);
            if (__any_sync(0xffffffffu, bad) && lane == 0) sh.bad = 1;
            stage_parity ^= 1u;
            in_flight = false;
        };
        if (warp >= 1 && warp <= stage_warps && warp - 1 < units) issue_unit(warp - 1);

        Side up, low;
        side_empty(up, true);
        side_empty(low, false);
        bool first = true;
        int64_t iter = MODE == MODE_FP64 ? J.iter0 : 0;   // (only FP64 jobs are continued)
        int prev_valid = 0, prev_len_u = 0, prev_len_l = 0;
        int status_code = JOB_CONVERGED;
        for (;;) {
            const int buf = (int)(iter & 1);
            Tgt *T = tbuf + (size_t)buf * dmax;
            int *tcu = tcol + (size_t)(buf * 2 + 0) * maxnnz;
            int *tcl = tcol + (size_t)(buf * 2 + 1) * maxnnz;
            bool hu = false, hl = false;   // x_up's / x_low's kernel row is in the cache
            uint32_t kd_wu = 0, kd_wl = 0;
            if (!first) {
                // (the gap is tested beside the pair step, below)
                if (up.i == INT_MAX || low.i == INT_MAX) { status_code = JOB_CONVERGED; break; }
                if (iter >= J.max_iter) { status_code = dless(thr, low.f - up.f) ? JOB_ITER_LIMIT : JOB_CONVERGED; break; }
                if (kc_on) {
                    kd_wu = kdir[up.i >> 5];
                    kd_wl = kdir[low.i >> 5];
                    hu = (kd_wu >> (up.i & 31)) & 1u;
                    hl = (kd_wl >> (low.i & 31)) & 1u;
                }
                // ---- 1. targets into the shared-memory buffer
                if (dense) {
                    if constexpr (MODE == MODE_MIXED) {
                        const __nv_bfloat16 *ru = dmat + (size_t)up.p0 * d;
                        const __nv_bfloat16 *rl = dmat + (size_t)low.p0 * d;
                        for (int c = tid; c < d; c += kThreads) {
                            T[c].x = __bfloat162float(ru[c]);
                            T[c].y = __bfloat162float(rl[c]);
                        }
                    }
                } else {
                    // x_up by the first half of the threads, x_low by the
                    // second: both rows' loads in flight together
                    constexpr int kHalf = kThreads / 2;
                    if (tid < kHalf) {
                        for (int k = tid; k < up.len; k += kHalf) {
                            const int c = indices[up.p0 + k];
                            tcu[k] = c;
                            if constexpr (MODE == MODE_BINARY) reinterpret_cast<unsigned char *>(T + c)[0] = 1;
                            else if constexpr (MODE == MODE_FP64) xd_put<0>(T[c], values[up.p0 + k], xd, xd_tmin, 0);
                            else T[c].x = vmix[up.p0 + k];
                        }
                    } else {
                        for (int k = tid - kHalf; k < low.len; k += kHalf) {
                            const int c = indices[low.p0 + k];
                            tcl[k] = c;
                            if constexpr (MODE == MODE_BINARY) reinterpret_cast<unsigned char *>(T + c)[1] = 1;
                            else if constexpr (MODE == MODE_FP64) xd_put<1>(T[c], values[low.p0 + k], xd, xd_tmin, 0);
                            else T[c].y = vmix[low.p0 + k];
                        }
                    }
                }
                // the warps of the pair step's bounds only arrive; with both
                // kernel rows cached no row warp waits for the targets (warp
                // 0 does: its K(up, low) is computed from them)
                const bool both = hu && hl;
                if (warp >= kPre0 || (both && warp != 0)) fill_bar_arrive();
                else fill_bar_sync();
                if (warp == 0 && !both) filled_arrive();
                if (warp >= kPre0) {
                    // the pair step's part that K(up, low) does not enter
                    pair_pre<MODE == MODE_FP64>(&sh.pre, warp - kPre0, lane, up, low, C);
                    pre_bar_arrive();
                    if (!both) filled_sync();
                }
            }
            unsigned long long bku = kNoKey, bkl = kNoKey;
            int biu = INT_MAX, bil = INT_MAX, bru = 0, brl = 0;
            bool stop = false;   // the gap is closed: nothing of this step is taken
            if (warp == 0) {
                // ---- 2. pair step (Eq. alphaup with rho = -eta, Platt clip)
                if (!first) {
                    Acc s = 0;
                    if (dense) {
                        if constexpr (MODE == MODE_MIXED)
                            for (int c = lane; c < d; c += 32) s = fmaf(T[c].y, T[c].x, s);
                    } else if (xd) {
                        if constexpr (MODE == MODE_FP64) {
                            const int4 *T4 = reinterpret_cast<const int4 *>(T);
                            XdAcc a = xd_zero();
                            for (int k = lane; k < low.len; k += 32) {
                                const int4 t = T4[tcl[k]];
                                xd_add(a, t.z, t.x, t.w + t.y + xd_bias);
                            }
                            xd_lane_sum<32>(a);
                            s = xd_round(a, xd_unit);
                        }
                    } else {
                        for (int k = lane; k < low.len; k += 32) {
                            const Tgt t = T[tcl[k]];
                            if constexpr (MODE == MODE_BINARY) s += (int)(t & 1);
                            else if constexpr (MODE == MODE_FP64) s = fma(t.y, t.x, s);
                            else s = fmaf(t.y, t.x, s);
                        }
                    }
                    if (!xd) {
#pragma unroll
                        for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    }
                    pre_bar_sync();
                    const PairPre pre = sh.pre;
                    stop = !bits_less(thr, neg_if(pre.slope.x, low.y > 0));   // Eq. (kktterm)
                    bool curved;
                    double q;
                    if constexpr (MODE == MODE_BINARY) {
                        int dist = up.len + low.len - 2 * s;
                        dist = dist < 0 ? 0 : dist;
                        const double eta = 2.0 - 2.0 * ktab[dist], rinv = rtab[dist];
                        curved = bits_less(1e-12, eta);
                        const double q0 = pre.slope.x * rinv;
                        const double rr = fma(-eta, q0, pre.slope.x);
                        q = fma(rr, rinv, q0);
                    } else {
                        double kul;
                        if constexpr (MODE == MODE_FP64) {
                            kul = exp_neg_fx(gamma * dpos(fma(-2.0, s, pre.nsum)), expfx_s);
                        } else {
                            const float d2 = norm_f32(up.nrm) + norm_f32(low.nrm) - 2.0f * s;
                            kul = widen_f32(__expf(-gammaf * fmaxf(d2, 0.f)));
                        }
                        const double eta = 2.0 - 2.0 * kul;
                        curved = bits_less(1e-12, eta);
                        q = pair_quotient<true>(pre.slope, curved ? eta : 1.0);
                    }
                    const PairStep ps = pair_solve(pre, up, low, curved, q, C, snap, c_snap);
                    if (lane == 0) {
                        sh.stop = stop;
                        sh.du = ps.du;
                        sh.dl = ps.dl;
                        sh.au_new = ps.au;
                        sh.al_new = ps.al;
                        sh.st_u = status_of(up.y > 0, ps.au, C);
                        sh.st_l = status_of(low.y > 0, ps.al, C);
                    }
                    __syncwarp();
                    step_bar_arrive(kThreads);
                }
            } else {
                // ---- 3. row pass over this CTA's rows of the job
                constexpr int kRowWarps = kWarps - 1;
                double du = 0.0, dl = 0.0, au_new = 0.0, al_new = 0.0;
                unsigned char st_u = 0, st_l = 0;
                bool have_step = first;
                auto wait_step = [&]() {
                    if (!have_step) {
                        step_bar_sync(kThreads);
                        du = sh.du; dl = sh.dl;
                        st_u = sh.st_u; st_l = sh.st_l;
                        au_new = sh.au_new; al_new = sh.al_new;
                        stop = sh.stop != 0;
                        have_step = true;
                    }
                };
                double *kcu = kc_on && !first ? kc + (size_t)up.i * kc_ld : nullptr;
                double *kcl = kc_on && !first ? kc + (size_t)low.i * kc_ld : nullptr;
                // FP64 update of Eq. (fup) and selection keys of one row
                auto update_row = [&](int r, double ku, double kl, double fi, uint8_t sb) {
                    if (stop) return;
                    if (!first) {
                        fi = fma(dl, kl, fma(du, ku, fi));
                        fj[r] = fi;
                        if (r == up.i) {
                            sb = st_u;
                            sj[r] = sb;
                            aj[r] = au_new;
                        } else if (r == low.i) {
                            sb = st_l;
                            sj[r] = sb;
                            aj[r] = al_new;
                        }
                    }
                    const uint8_t set = set_bits(sb);
                    const unsigned long long kf = dkey(fi);
                    if (st_up(set) && ki_less(kf, r, bku, biu)) { bku = kf; biu = r; bru = r; }
                    if (st_low(set) && ki_less(~kf, r, bkl, bil)) { bkl = ~kf; bil = r; brl = r; }
                };
                // this row's kernel values from its inner products, or from the
                // cache; nv: the row's norm
                auto kernel_values = [&](int r, int len, Acc su, Acc sl, double nv, double &ku, double &kl) {
                    ku = kl = 0.0;
                    if (first) return;
                    if constexpr (MODE == MODE_BINARY) {
                        int du2 = up.len + len - 2 * su, dl2 = low.len + len - 2 * sl;
                        ku = ktab[du2 < 0 ? 0 : du2];
                        kl = ktab[dl2 < 0 ? 0 : dl2];
                    } else if constexpr (MODE == MODE_FP64) {
                        if (hu) ku = kcu[r];
                        else {
                            ku = exp_neg_fx(gamma * dpos(up.nrm + nv - 2.0 * su), expfx_s);
                            if (kc_on) kcu[r] = ku;
                        }
                        if (hl) kl = kcl[r];
                        else {
                            kl = exp_neg_fx(gamma * dpos(low.nrm + nv - 2.0 * sl), expfx_s);
                            if (kc_on) kcl[r] = kl;
                        }
                    } else {
                        // widened exactly by integer operations (a conversion
                        // instruction would take a slot of the FP64 pipe)
                        const float nf = norm_f32(nv);
                        ku = widen_f32(__expf(-gammaf * fmaxf(norm_f32(up.nrm) + nf - 2.0f * su, 0.f)));
                        kl = widen_f32(__expf(-gammaf * fmaxf(norm_f32(low.nrm) + nf - 2.0f * sl, 0.f)));
                    }
                };
                auto row_norm = [&](int g) -> double {
                    if constexpr (MODE == MODE_FP64) return norm[g];
                    else if constexpr (MODE == MODE_MIXED) return norm_bits(normf[g]);
                    else return 0.0;
                };
                auto finish_row = [&](int r, int g, int len, Acc su, Acc sl, double fi, uint8_t sb) {
                    double ku, kl;
                    kernel_values(r, len, su, sl, first ? 0.0 : row_norm(g), ku, kl);
                    update_row(r, ku, kl, fi, sb);
                };
                if (hu && hl) {
                    // both rows cached: a thread per row, coalesced
                    if constexpr (KC_MODE) {
                        for (int r0 = lo + tid - 32;; r0 += 4 * (kThreads - 32)) {
                            double ku[4], kl[4], fi[4];
                            uint8_t sb[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = r0 + j * (kThreads - 32);
                                ku[j] = kl[j] = fi[j] = 0.0;
                                sb[j] = 0;
                                if (r < hi) {
                                    ku[j] = kcu[r];
                                    kl[j] = kcl[r];
                                    fi[j] = fj[r];
                                    sb[j] = sj[r];
                                }
                            }
                            wait_step();
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int r = r0 + j * (kThreads - 32);
                                if (r < hi) update_row(r, ku[j], kl[j], fi[j], sb[j]);
                            }
                            if (r0 - (tid - 32) + 4 * (kThreads - 32) >= hi) break;   // uniform
                        }
                    }
                } else {
                bool blocked = false;
                if constexpr (LPR == 32) blocked = dense && d <= 256;
                bool tiles = false;   // dense BF16 rows on the tensor cores
                if constexpr (LPR == 16 && MODE == MODE_MIXED) tiles = dense && (d & 31) == 0 && d <= 256;
                if (tiles) {
                    if constexpr (LPR == 16 && MODE == MODE_MIXED) {
                        // Tiles of 16 rows x the two target rows on the
                        // tensor cores (mma m16n8k16, BF16 inputs, FP32
                        // accumulation; columns 2..7 of B are zero). Inside
                        // each 32-column block the K order is permuted so
                        // that a thread reads 8 consecutive values of a row
                        // with one 16-byte load: in k-step h of the block,
                        // logical k = 2t + i maps to column 8t + 4h + i and
                        // k = 2t + 8 + i to 8t + 4h + 2 + i; the targets use
                        // the same map, so the dot products are unchanged.
                        const int g = lane >> 2, t = lane & 3;
                        const int nblk = d >> 5;
                        // the target fragments, [k-step][lane], k-step = 2 * block + h,
                        // packed once per step by the row warps together
                        for (int ks = warp - 1; ks < 2 * nblk; ks += kRowWarps) {
                            uint32_t r0 = 0, r1 = 0;
                            if (!first && g < 2) {
                                const int c = 32 * (ks >> 1) + 8 * t + 4 * (ks & 1);
                                float e[4];
#pragma unroll
                                for (int x = 0; x < 4; ++x) e[x] = g == 0 ? T[c + x].x : T[c + x].y;
                                const __nv_bfloat162 p0 = __floats2bfloat162_rn(e[0], e[1]);
                                const __nv_bfloat162 p1 = __floats2bfloat162_rn(e[2], e[3]);
                                r0 = *reinterpret_cast<const uint32_t *>(&p0);
                                r1 = *reinterpret_cast<const uint32_t *>(&p1);
                            }
                            frag[ks * 32 + lane] = make_uint2(r0, r1);
                        }
                        rows_bar_sync();
                        // two tiles (32 rows, a unit) at a time: each row's two
                        // sums are handed to one lane, so that the exponentials
                        // and the FP64 updates run on whole warps
                        const int step_warps = packed ? stage_warps : kRowWarps;
                        // Packed units are walked forwards and backwards in
                        // turn: a step begins with the unit that its stage
                        // still holds, and the units read last are in L2 (76
                        // problems' rows, 152 MB, are more than L2 and came
                        // from HBM in every step when always walked forwards:
                        // 90 problems of 4,000 x 256, 104.6 -> 97.0 ms). The
                        // selection does not depend on the order.
                        const bool rev = packed && (iter & 1);
                        const int nu = warp <= step_warps && warp <= units ? (units - warp) / step_warps + 1 : 0;
                        for (int k = 0; k < nu; ++k) {
                            const int u = warp - 1 + (rev ? nu - 1 - k : k) * step_warps;
                            const int base = lo + 32 * u;
                            const int r = base + lane;
                            const bool valid = r < hi;
                            int grow = 0;
                            double fi = 0.0, nv = 0.0;
                            uint8_t sb = 0;
                            if (valid) {
                                grow = rows[r];
                                fi = fj[r];
                                sb = sj[r];
                                nv = row_norm(grow);
                            }
                            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
                            if (!first && packed) {
                                wait_unit();
                                const uint4 *sp = reinterpret_cast<const uint4 *>(stage) + lane;
#pragma unroll
                                for (int q = 0; q < 2; ++q) {
#pragma unroll 4
                                    for (int b = 0; b < nblk; ++b) {
                                        const uint4 x = sp[((q * nblk + b) * 2) * 32], z = sp[((q * nblk + b) * 2 + 1) * 32];
                                        const uint2 f0 = frag[(2 * b) * 32 + lane], f1 = frag[(2 * b + 1) * 32 + lane];
                                        mma_bf16_16816(acc[q], x.x, z.x, x.y, z.y, f0.x, f0.y);
                                        mma_bf16_16816(acc[q], x.z, z.z, x.w, z.w, f1.x, f1.y);
                                    }
                                }
                                // the next unit while this one's rows are
                                // finished
                                __syncwarp();
                                if (k + 1 < nu) {
                                    fence_async_proxy();
                                    issue_unit(rev ? u - step_warps : u + step_warps);
                                }
                            } else if (!first) {
#pragma unroll
                                for (int q = 0; q < 2; ++q) {
                                    const int ia = __shfl_sync(0xffffffffu, grow, 16 * q + g);
                                    const int ib = __shfl_sync(0xffffffffu, grow, 16 * q + g + 8);
                                    const __nv_bfloat16 *pa = base + 16 * q + g < hi ? dmat + (size_t)ia * d + 8 * t : nullptr;
                                    const __nv_bfloat16 *pb = base + 16 * q + g + 8 < hi ? dmat + (size_t)ib * d + 8 * t : nullptr;
#pragma unroll 4
                                    for (int b = 0; b < nblk; ++b) {
                                        const uint4 x = pa ? __ldg(reinterpret_cast<const uint4 *>(pa + 32 * b)) : make_uint4(0, 0, 0, 0);
                                        const uint4 z = pb ? __ldg(reinterpret_cast<const uint4 *>(pb + 32 * b)) : make_uint4(0, 0, 0, 0);
                                        const uint2 f0 = frag[(2 * b) * 32 + lane], f1 = frag[(2 * b + 1) * 32 + lane];
                                        mma_bf16_16816(acc[q], x.x, z.x, x.y, z.y, f0.x, f0.y);
                                        mma_bf16_16816(acc[q], x.z, z.z, x.w, z.w, f1.x, f1.y);
                                    }
                                }
                            }
                            // the sums of row base + lane: tile lane >> 4, row
                            // lane & 15, held by lane 4 (lane & 7) as (acc[2 s],
                            // acc[2 s + 1]), s = (lane >> 3) & 1
                            const int src = 4 * (lane & 7);
                            const int qq = lane >> 4, ss = (lane >> 3) & 1;
                            float su = 0.f, sl = 0.f;
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
#pragma unroll
                                for (int s2 = 0; s2 < 2; ++s2) {
                                    const float x = __shfl_sync(0xffffffffu, acc[q][2 * s2], src);
                                    const float z = __shfl_sync(0xffffffffu, acc[q][2 * s2 + 1], src);
                                    if (q == qq && s2 == ss) { su = x; sl = z; }
                                }
                            }
                            double ku = 0.0, kl = 0.0;
                            if (valid) kernel_values(r, d, su, sl, nv, ku, kl);
                            wait_step();
                            if (valid) update_row(r, ku, kl, fi, sb);
                        }
                        wait_step();
                    }
                } else if (blocked) {
                    if constexpr (LPR == 32 && MODE == MODE_MIXED) {
                        // 8 rows per warp at a time; lane l covers columns
                        // [8l, 8l+8) of all 8 rows with its target columns in
                        // registers; a butterfly transpose-reduction leaves
                        // each group of 4 lanes with one row's two sums
                        const int c8 = lane * 8;
                        const bool has_cols = c8 < d;
                        float tu[8], tl[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            tu[e] = 0.f;
                            tl[e] = 0.f;
                        }
                        if (!first && has_cols) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const float2 t = T[c8 + e];
                                tu[e] = t.x;
                                tl[e] = t.y;
                            }
                        }
                        const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0, h4 = (lane & 4) != 0;
                        const int ri = (h16 ? 4 : 0) + (h8 ? 2 : 0) + (h4 ? 1 : 0);
                        for (int base = lo + (warp - 1) * 8;; base += kRowWarps * 8) {
                            const bool round0 = base == lo + (warp - 1) * 8;
                            if (!round0 && base >= hi) break;
                            float pu[8], pl[8];
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                pu[j] = 0.f;
                                pl[j] = 0.f;
                                const int r = base + j;
                                if (!first && r < hi && has_cols) {
                                    const int g = rows[r];
                                    const uint4 raw = *reinterpret_cast<const uint4 *>(dmat + (size_t)g * d + c8);
                                    const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&raw);
#pragma unroll
                                    for (int e = 0; e < 4; ++e) {
                                        const float2 v = __bfloat1622float2(h2[e]);
                                        pu[j] = fmaf(v.x, tu[2 * e], pu[j]);
                                        pl[j] = fmaf(v.x, tl[2 * e], pl[j]);
                                        pu[j] = fmaf(v.y, tu[2 * e + 1], pu[j]);
                                        pl[j] = fmaf(v.y, tl[2 * e + 1], pl[j]);
                                    }
                                }
                            }
                            float au[4], al[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                au[k] = (h16 ? pu[k + 4] : pu[k]) + __shfl_xor_sync(0xffffffffu, h16 ? pu[k] : pu[k + 4], 16);
                                al[k] = (h16 ? pl[k + 4] : pl[k]) + __shfl_xor_sync(0xffffffffu, h16 ? pl[k] : pl[k + 4], 16);
                            }
                            float bu2[2], bl2[2];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                bu2[k] = (h8 ? au[k + 2] : au[k]) + __shfl_xor_sync(0xffffffffu, h8 ? au[k] : au[k + 2], 8);
                                bl2[k] = (h8 ? al[k + 2] : al[k]) + __shfl_xor_sync(0xffffffffu, h8 ? al[k] : al[k + 2], 8);
                            }
                            float su = (h4 ? bu2[1] : bu2[0]) + __shfl_xor_sync(0xffffffffu, h4 ? bu2[0] : bu2[1], 4);
                            float sl = (h4 ? bl2[1] : bl2[0]) + __shfl_xor_sync(0xffffffffu, h4 ? bl2[0] : bl2[1], 4);
                            su += __shfl_xor_sync(0xffffffffu, su, 2);
                            sl += __shfl_xor_sync(0xffffffffu, sl, 2);
                            su += __shfl_xor_sync(0xffffffffu, su, 1);
                            sl += __shfl_xor_sync(0xffffffffu, sl, 1);
                            const int r = base + ri;
                            double fi = 0.0;
                            uint8_t sb = 0;
                            int g = 0;
                            const bool lead = (lane & 3) == 0 && r < hi;
                            if (lead) {
                                g = rows[r];
                                fi = fj[r];
                                sb = sj[r];
                            }
                            wait_step();
                            if (lead) finish_row(r, g, d, su, sl, fi, sb);
                        }
                    }
                } else {
                    constexpr int RPW = 32 / LPR;
                    const int gl = lane & (LPR - 1);
                    const int gw = lane / LPR;
                    for (int kb = lo + (warp - 1) * RPW;; kb += kRowWarps * RPW) {
                        const bool round0 = kb == lo + (warp - 1) * RPW;
                        if (!round0 && kb >= hi) break;
                        const int r = kb + gw;
                        const bool valid = r < hi;
                        int g = 0;
                        int64_t p0 = 0, p1 = 0;
                        double fi = 0.0;
                        uint8_t sb = 0;
                        if (valid) {
                            g = rows[r];
                            if (!dense) {
                                p0 = indptr[g];
                                p1 = indptr[g + 1];
                            }
                            if (gl == 0) {
                                fi = fj[r];
                                sb = sj[r];
                            }
                        }
                        Acc su = 0, sl = 0;
                        XdAcc au = xd_zero(), al = xd_zero();   // FP64, exact inner products
                        if (!first && valid) {
                            if (dense) {
                                if constexpr (MODE == MODE_MIXED) {
                                const __nv_bfloat16 *xr = dmat + (size_t)g * d;
                                auto piece = [&](int c) {
                                    const uint4 raw = *reinterpret_cast<const uint4 *>(xr + c);
                                    const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&raw);
#pragma unroll
                                    for (int e = 0; e < 4; ++e) {
                                        const float2 v = __bfloat1622float2(h2[e]);
                                        const float2 t0 = T[c + 2 * e], t1 = T[c + 2 * e + 1];
                                        su = fmaf(v.x, t0.x, su);
                                        sl = fmaf(v.x, t0.y, sl);
                                        su = fmaf(v.y, t1.x, su);
                                        sl = fmaf(v.y, t1.y, sl);
                                    }
                                };
                                // long rows wait for loads: eight pieces'
                                // at a time (1,306 x 1,587, 2 lanes, 14.6 ->
                                // 13.1 us a step; 64 columns 3% slower so)
                                if (LPR <= 8 && d >= 16 * LPR * 8) {
#pragma unroll 8
                                    for (int c = gl * 8; c < d; c += LPR * 8) piece(c);
                                } else {
                                    for (int c = gl * 8; c < d; c += LPR * 8) piece(c);
                                }
                                }
                            } else if (xd) {
                                if constexpr (MODE == MODE_FP64) {
                                    // four entries' loads at a time, the rest of
                                    // the row one by one; a side whose row is
                                    // cached is left out. (Bound by issue: with a
                                    // bound check per entry and both forms in one
                                    // loop, 20 problems of 20,000 x 20 rows took
                                    // 39.5 ms for 500 steps, 36.4 with one entry
                                    // at a time, 35.6 so.)
                                    const int32_t *ip = indices + p0;
                                    const float *vp = values + p0;
                                    const int len = (int)(p1 - p0);
                                    const int4 *T4 = reinterpret_cast<const int4 *>(T);
                                    const int2 *T2 = reinterpret_cast<const int2 *>(T) + (hu ? 1 : 0);
                                    auto entry = [&](auto two, int c, uint32_t u) {
                                        const int32_t mx = xd_mant(u);
                                        const int e = xd_exp(u, xd_tmin) + xd_bias;
                                        if constexpr (two()) {
                                            const int4 t = T4[c];
                                            xd_add(au, mx, t.x, e + t.y);
                                            xd_add(al, mx, t.z, e + t.w);
                                        } else {
                                            const int2 t = T2[2 * c];
                                            xd_add(au, mx, t.x, e + t.y);
                                        }
                                    };
                                    auto sum_row = [&](auto two) {
                                        int k = gl;
#pragma unroll 1
                                        for (; k + 3 * LPR < len; k += 4 * LPR) {
                                            int cb[4];
                                            uint32_t ub[4];
#pragma unroll
                                            for (int j = 0; j < 4; ++j) {
                                                cb[j] = ip[k + j * LPR];
                                                ub[j] = __float_as_uint(vp[k + j * LPR]);
                                            }
#pragma unroll
                                            for (int j = 0; j < 4; ++j) entry(two, cb[j], ub[j]);
                                        }
#pragma unroll 1
                                        for (; k < len; k += LPR) entry(two, ip[k], __float_as_uint(vp[k]));
                                    };
                                    if (!hu && !hl) sum_row(std::true_type{});
                                    else sum_row(std::false_type{});
                                }
                            } else {
                                for (int64_t p = p0 + gl; p < p1; p += LPR) {
                                    const int c = indices[p];
                                    if constexpr (MODE == MODE_BINARY) {
                                        const unsigned short t = T[c];
                                        su += (int)(t & 0xff);
                                        sl += (int)(t >> 8);
                                    } else if constexpr (MODE == MODE_FP64) {
                                        const double v = (double)values[p];
                                        const double2 t = T[c];
                                        su = fma(v, t.x, su);
                                        sl = fma(v, t.y, sl);
                                    } else {
                                        const float v = vmix[p];
                                        const float2 t = T[c];
                                        su = fmaf(v, t.x, su);
                                        sl = fmaf(v, t.y, sl);
                                    }
                                }
                            }
                        }
                        if (!first && xd) {
                            if constexpr (MODE == MODE_FP64) {
                                xd_lane_sum<LPR>(au);
                                su = sl = xd_round(au, xd_unit);
                                if (!hu && !hl) {
                                    xd_lane_sum<LPR>(al);
                                    sl = xd_round(al, xd_unit);
                                }
                            }
                        } else if (!first) {
#pragma unroll
                            for (int o = LPR / 2; o >= 1; o >>= 1) {
                                su += __shfl_xor_sync(0xffffffffu, su, o);
                                sl += __shfl_xor_sync(0xffffffffu, sl, o);
                            }
                        }
                        double ku = 0.0, kl = 0.0;
                        if (valid && gl == 0) kernel_values(r, (int)(p1 - p0), su, sl, first ? 0.0 : row_norm(g), ku, kl);
                        wait_step();
                        if (valid && gl == 0) update_row(r, ku, kl, fi, sb);
                    }
                }
                }
            }
            if (stop) { status_code = JOB_CONVERGED; break; }   // (every CTA sees the same pair)
            // payload of a job row (job-local index r)
            auto make_side = [&](int r) {
                Side sd;
                const int g = rows[r];
                const uint8_t sb = sj[r];
                sd.f = fj[r];
                sd.a = aj[r];
                if constexpr (MODE == MODE_FP64) sd.nrm = norm[g];
                else if constexpr (MODE == MODE_MIXED) sd.nrm = norm_bits(normf[g]);
                else sd.nrm = 0.0;
                if (dense) {
                    sd.p0 = g;
                    sd.len = d;
                } else {
                    sd.p0 = indptr[g];
                    sd.len = (int)(indptr[g + 1] - sd.p0);
                }
                sd.i = r;
                sd.y = y_of(sb);
                sd.owner = 0;
                return sd;
            };
            {
                unsigned long long k1 = bku, k2 = bkl;
                int i1 = biu, i2 = bil;
                warp_min_ki(k1, i1);
                warp_min_ki(k2, i2);
                if (lane == 0) {
                    sh.wkup[warp] = k1; sh.wiup[warp] = i1;
                    sh.wklow[warp] = k2; sh.wilow[warp] = i2;
                }
                if (i1 != INT_MAX && biu == i1) sh.wup[warp] = make_side(bru);
                if (i2 != INT_MAX && bil == i2) sh.wlow[warp] = make_side(brl);
            }
            __syncthreads();
            // both rows are stored from here on (all threads have read this
            // step's bits; the barrier after the exchange orders the next step's reads)
            if (kc_on && !first && tid == 0) {
                const uint32_t bu = 1u << (up.i & 31), bl = 1u << (low.i & 31);
                const bool same = (up.i >> 5) == (low.i >> 5);
                kdir[up.i >> 5] = kd_wu | bu | (same ? bl : 0u);
                if (!same) kdir[low.i >> 5] = kd_wl | bl;
            }
            // ---- 4. candidate exchange inside the cluster: every CTA's
            //         candidate into every CTA's shared memory, as asynchronous
            //         stores counted on its mbarrier (lanes q and 16 + q send
            //         the first 48 bytes of the I_up and I_low sides to CTA q);
            //         every CTA reduces them in the same order. (Two cluster
            //         barriers a step before, 530 cycles each. With the gap
            //         test beside the pair step and row warps that do not
            //         wait for the target fill when both rows are cached, 45
            //         FP64 problems of 1,500 rows, d = 20, clusters of 4 CTAs,
            //         on one input: 35.0 -> 28.7 ms.)
            ++epoch;
            const int par = (int)(epoch & 1);
            if (warp == 0) {
                unsigned long long k1 = lane < kWarps ? sh.wkup[lane] : kNoKey;
                unsigned long long k2 = lane < kWarps ? sh.wklow[lane] : kNoKey;
                int i1 = lane < kWarps ? sh.wiup[lane] : INT_MAX;
                int i2 = lane < kWarps ? sh.wilow[lane] : INT_MAX;
                const int i1s = i1, i2s = i2;
                warp_min_ki(k1, i1);
                warp_min_ki(k2, i2);
                const int w1 = __ffs(__ballot_sync(0xffffffffu, i1s == i1)) - 1;
                const int w2 = __ffs(__ballot_sync(0xffffffffu, i2s == i2)) - 1;
                const bool side_low = lane >= 16;
                const int q = lane & 15;
                const Side *sd = side_low ? (i2 != INT_MAX ? &sh.wlow[w2] : &sh.none[1])
                                          : (i1 != INT_MAX ? &sh.wup[w1] : &sh.none[0]);
                if (q < csize) {
                    const uint4 *sv = reinterpret_cast<const uint4 *>(sd);
                    const uint32_t dst = cluster_addr(smem_u32(side_low ? &sh.xc[par][crank].low : &sh.xc[par][crank].up), q);
                    const uint32_t rbar = cluster_addr(smem_u32(&sh.xbar[par]), q);
#pragma unroll
                    for (int j = 0; j < 3; ++j) st_async_v4(dst + 16 * j, sv[j], rbar);
                }
                if (lane == 0) mbar_arrive_expect_tx(smem_u32(&sh.xbar[par]), (uint32_t)(csize * 2 * 48));
            }
            if (prev_valid && !dense && warp >= 8) {
                Tgt *P = tbuf + (size_t)(1 - buf) * dmax;
                const int *pcu = tcol + (size_t)((1 - buf) * 2 + 0) * maxnnz;
                const int *pcl = tcol + (size_t)((1 - buf) * 2 + 1) * maxnnz;
                for (int k = tid - 256; k < prev_len_u; k += kThreads - 256) P[pcu[k]] = tclear;
                for (int k = tid - 256; k < prev_len_l; k += kThreads - 256) P[pcl[k]] = tclear;
            }
            if (warp == 0) {
                const uint32_t parity = (uint32_t)((epoch - 1) >> 1) & 1u;
                int bad = mbar_wait_bounded(smem_u32(&sh.xbar[par]), parity, kWaitNs, nullptr);
                bad = __any_sync(0xffffffffu, bad || *(volatile int *)&sh.bad);
                unsigned long long k1 = kNoKey, k2 = kNoKey;
                int i1 = INT_MAX, i2 = INT_MAX;
                if (lane < csize && !bad) {
                    const CandSlot &cs = sh.xc[par][lane];
                    i1 = cs.up.i;
                    i2 = cs.low.i;
                    k1 = i1 == INT_MAX ? kNoKey : key_up(cs.up.f);
                    k2 = i2 == INT_MAX ? kNoKey : key_low(cs.low.f);
                }
                const int i1s = i1, i2s = i2;
                warp_min_ki(k1, i1);
                warp_min_ki(k2, i2);
                // (without any candidate lane 0 wins, whose side is the empty one)
                const int w1 = __ffs(__ballot_sync(0xffffffffu, i1s == i1)) - 1;
                const int w2 = __ffs(__ballot_sync(0xffffffffu, i2s == i2)) - 1;
                if (lane < 12) {
                    const bool u = lane < 6;
                    const int w = u ? lane : lane - 6;
                    reinterpret_cast<unsigned long long *>(u ? &sh.res.up : &sh.res.low)[w] =
                        reinterpret_cast<const unsigned long long *>(u ? &sh.xc[par][w1].up : &sh.xc[par][w2].low)[w];
                }
                if (lane == 0) sh.res.flag = bad;
            }
            __syncthreads();
            if (sh.res.flag) {
                if (tid == 0) sh.bad = 1;
                status_code = JOB_WAIT_GAVE_UP;
                break;
            }
            prev_valid = first ? 0 : 1;
            prev_len_u = up.len;
            prev_len_l = low.len;
            up = sh.res.up;
            low = sh.res.low;
            if (!first) ++iter;
            first = false;
        }

        wait_unit();   // the stage is free and the packed rows may be rewritten
        // ---- job results: b (Section III-A) and the objective from partial sums
        {
            BatchFinish pf = {0, 0, 0, 0, 0, {0, 0}};
            for (int r = lo + tid; r < hi; r += kThreads) {
                const double a = aj[r];
                const uint8_t sb = sj[r];
                const double yi = (sb & 0x80) ? 1.0 : -1.0;
                const double fi = fj[r];
                pf.sum_a += a;
                pf.sum_ayfy += a * yi * (fi + yi);
                if ((sb & 7) == ST_I0) { pf.sum_f0 += fi; pf.n0 += 1; }
                if (a > 0.0) pf.nsv += 1;
            }
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                pf.sum_a += __shfl_xor_sync(0xffffffffu, pf.sum_a, o);
                pf.sum_ayfy += __shfl_xor_sync(0xffffffffu, pf.sum_ayfy, o);
                pf.sum_f0 += __shfl_xor_sync(0xffffffffu, pf.sum_f0, o);
                pf.n0 += __shfl_xor_sync(0xffffffffu, pf.n0, o);
                pf.nsv += __shfl_xor_sync(0xffffffffu, pf.nsv, o);
            }
            if (lane == 0) sh.wfin[warp] = pf;
            __syncthreads();
            if (tid == 0) {
                BatchFinish t = sh.wfin[0];
                for (int w = 1; w < kWarps; ++w) {
                    t.sum_a += sh.wfin[w].sum_a;
                    t.sum_ayfy += sh.wfin[w].sum_ayfy;
                    t.sum_f0 += sh.wfin[w].sum_f0;
                    t.n0 += sh.wfin[w].n0;
                    t.nsv += sh.wfin[w].nsv;
                }
                *(cluster.map_shared_rank(sh.fin, 0) + crank) = t;
                if (sh.bad)
                    for (int r = 0; r < csize; ++r) *cluster.map_shared_rank(&sh.bad, r) = 1;
            }
            cluster.sync();
            if (crank == 0 && tid == 0) {
                BatchFinish t = sh.fin[0];
                for (int r = 1; r < csize; ++r) {
                    t.sum_a += sh.fin[r].sum_a;
                    t.sum_ayfy += sh.fin[r].sum_ayfy;
                    t.sum_f0 += sh.fin[r].sum_f0;
                    t.n0 += sh.fin[r].n0;
                    t.nsv += sh.fin[r].nsv;
                }
                BatchResultDev R;
                R.b_up = up.f;
                R.b_low = low.f;
                R.b = t.n0 > 0 ? t.sum_f0 / (double)t.n0 : 0.5 * (up.f + low.f);
                R.objective = t.sum_a - 0.5 * t.sum_ayfy;
                R.iters = iter;
                R.status = sh.bad ? JOB_WAIT_GAVE_UP : status_code;
                R.n_sv = (int32_t)t.nsv;
                B.results[job] = R;
                if (B.done) {
                    __threadfence_system();
                    st_release_sys_i32(B.done + job, 1);
                }
            }
            cluster.sync();   // shared memory of the cluster is reused by the next job
        }
    }
    cluster.sync();
}

template <int MODE>
void *batch_kernel_for(int lpr)
{
    switch (lpr) {
    case 1: return (void *)smo_batch_kernel<MODE, 1>;
    case 2: return (void *)smo_batch_kernel<MODE, 2>;
    case 4: return (void *)smo_batch_kernel<MODE, 4>;
    case 8: return (void *)smo_batch_kernel<MODE, 8>;
    case 16: return (void *)smo_batch_kernel<MODE, 16>;
    case 32: return (void *)smo_batch_kernel<MODE, 32>;
    default: return nullptr;
    }
}

void *batch_fn(int mode, int lpr)
{
    if (mode == MODE_MIXED) return batch_kernel_for<MODE_MIXED>(lpr);
    if (mode == MODE_FP64) return batch_kernel_for<MODE_FP64>(lpr);
    if (mode == MODE_BINARY) return batch_kernel_for<MODE_BINARY>(lpr);
    return nullptr;
}

}  // namespace
}  // namespace smo

size_t smo_batch_smem(int mode, int d, int ktab_len, int maxnnz, int kdir_words)
{
    // mixed mode: the target fragments of the tensor-core row tiles; then the
    // kernel-row cache's directory
    return smo_layout(mode, d, ktab_len, maxnnz, 0, 0, 0).total + (mode == MODE_MIXED ? smo::kFragBytes : 0) +
           4 * (size_t)kdir_words;
}

int smo_batch_max_clusters(int mode, int lpr, int dense, size_t smem, int cs)
{
    (void)dense;
    void *fn = smo::batch_fn(mode, lpr);
    if (!fn) return 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
    if (cs > 1 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cs;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t q = {};
    q.gridDim = dim3(cs);
    q.blockDim = dim3(smo::kThreads);
    q.dynamicSmemBytes = smem;
    q.attrs = &attr;
    q.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &q) != cudaSuccess) return 0;
    return n;
}

cudaError_t launch_smo_batch(int mode, int lpr, int dense, const BatchArgs &a, size_t smem, int cs,
                             int nclusters, cudaStream_t st)
{
    (void)dense;
    void *fn = smo::batch_fn(mode, lpr);
    if (!fn || cs < 1 || cs > smo::kMaxCluster || nclusters < 1) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (cs > 8) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    BatchArgs args = a;
    void *params[] = {&args};
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)cs;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cs * nclusters));
    cfg.blockDim = dim3(smo::kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace svmgb
