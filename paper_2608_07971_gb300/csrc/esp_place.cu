// Factored placement kernels of the ESP tatonnement (Sec. 3.2 with the placement expansion of
// Sec. 3.3): one pass over configurations x nodes per launch (k_place), and all rounds in one
// cooperative launch (k_place_res).

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "esp_barrier.h"
#include "esp_device.cuh"
#include "esp_kernels.h"
#include "esp_place.h"
#include "esp_warp.cuh"

namespace esp {

namespace {

// ---------------------------------------------------------------------------------------------
// Factored placement evaluation (esp_load_placement). A job's options are its KC configurations
// crossed with N nodes, and only the configurations are stored (Sec. 3.3's slowdown enters the
// value of (k, n) as the fp32 penalty sens_j * D[a_j][b_n]): a pass reads a few hundred bytes per
// job instead of KC * N options. One warp per job at a time; lane l takes nodes l and l + 32.
//
// Screen. G_k = the fp32 chain over the globally priced columns from -v32_k (v truncated as for a
// stored option), and candidate (k, n) scores q = the fp32 chain over the node's columns from
// fl(G_k + pen_n). Against the exact s (the fp64 chain from -(v_k - (double)pen_n)) this is one
// rounding more than the screen of a stored option; with M_s >= max|v_k| + max pen + sum_r max p_r
// max u_r the error stays within the same E (which has a factor of about 4 to spare), so the
// screen rule and the exact rule are those of the streaming kernel. Candidates are visited in
// increasing local index k * N + n on every lane, and configurations that repeat an earlier one
// of their job (marked at load) are skipped: their twins have lower indices and equal scores.

__host__ __device__ inline int place_warp_bytes(int R, int P, int KC)
{
    // configuration units, values, fp32 global parts, fp32 node-column units, fp32 prices
    return round16(KC * R * 4) + round16(KC * 8) + round16(KC * 4) + round16(KC * R * 4) + round16(P * 4);
}

// u: int32 units, or the same already converted (__int2float_rn)
template <int RT, typename U>
__device__ __forceinline__ float place_global_part(const U *u, double v, const ScenarioPrices &sp, int rg)
{
    float g = -screen_value(v);
#pragma unroll
    for (int r = 0; r < Cols<RT>::N; ++r) {
        if (r >= rg)
            break;
        g = __fmaf_rn(sp.pf[r], (float)u[r], g);
    }
    return g;
}

// uf: the configuration's units in fp32 (exact below 2^24, rounded above, as the stored screen does)
template <int RT>
__device__ __forceinline__ float place_node_part(const float *uf, float base, const float *p32s, int rg, int R, int n)
{
    float q = base;
    for (int r = rg; r < R; ++r)
        q = __fmaf_rn(p32s[rg + (R - rg) * n + (r - rg)], uf[r], q);
    return q;
}

// Shared-memory areas of one warp of the placement kernels: configuration units, values, fp32
// global parts, fp32 node-column units, fp32 prices.
struct PlaceWarpSmem {
    int32_t *us;
    double *vs;
    float *gs;
    float *ufs;
    float *p32s;
};

__device__ __forceinline__ PlaceWarpSmem place_warp_smem(unsigned char *smem, int wid, int R, int P, int KC)
{
    unsigned char *wbase = smem + (size_t)wid * place_warp_bytes(R, P, KC);
    PlaceWarpSmem w;
    w.us = reinterpret_cast<int32_t *>(wbase);
    w.vs = reinterpret_cast<double *>(wbase + round16(KC * R * 4));
    w.gs = reinterpret_cast<float *>(wbase + round16(KC * R * 4) + round16(KC * 8));
    w.ufs = reinterpret_cast<float *>(wbase + round16(KC * R * 4) + round16(KC * 8) + round16(KC * 4));
    w.p32s = reinterpret_cast<float *>(wbase + 2 * round16(KC * R * 4) + round16(KC * 8) + round16(KC * 4));
    return w;
}

// Best responses of the jobs [j_begin, j_end) (global job indices) over their configurations x
// nodes at the prices of c, the winners' demand into c's accumulators, then a flush.
template <int RT>
__device__ void place_jobs(WarpCtx<RT, true> &c, const DevPlace &pl, const PlaceWarpSmem &ws, int64_t j_begin,
                           int64_t j_end, int lane)
{
    const DevTable &t = c.t;
    const DevState &st = c.st;
    const int KC = pl.KC, N = pl.N, NT = pl.NT;
    const int R = c.R, rg = c.rg;
    int32_t *us = ws.us;
    double *vs = ws.vs;
    float *gs = ws.gs;
    float *ufs = ws.ufs;
    float *p32s = ws.p32s;
    for (int64_t j = j_begin; j < j_end; ++j) {
        const int sc = (int)(j / t.J);
        if (sc != c.s)
            enter_scenario<RT, true>(c, sc, p32s, lane);
        if (c.sp.skip)
            continue;
        __syncwarp();
        for (int i = lane; i < KC * R; i += 32)
            us[i] = __ldg(pl.cfg_units + j * KC * R + i);
        for (int k = lane; k < KC; k += 32)
            vs[k] = __ldg(pl.cfg_values + j * KC + k);
        const float sens = __ldg(pl.sens + j);
        const int aj = __ldg(pl.job_type + j);
        const uint32_t dup = __ldg(pl.cfg_dup + j);
        __syncwarp();
        // the global part of every configuration once (lane k), and the node columns' units in fp32;
        // a repeated configuration gets +inf and never survives the screen
        for (int k = lane; k < KC; k += 32)
            gs[k] = ((dup >> k) & 1u) ? INFINITY : place_global_part<RT>(us + k * R, vs[k], c.sp, rg);
        for (int i = lane; i < KC * R; i += 32)
            ufs[i] = __int2float_rn(us[i]);
        __syncwarp();

        const int n0 = lane, n1 = lane + 32;
        const bool h0 = n0 < N, h1 = n1 < N;
        const float pen0 = h0 ? __fmul_rn(sens, __ldg(pl.D + aj * NT + __ldg(pl.node_type + n0))) : 0.0f;
        const float pen1 = h1 ? __fmul_rn(sens, __ldg(pl.D + aj * NT + __ldg(pl.node_type + n1))) : 0.0f;
        float m1 = INFINITY, m2 = INFINITY;
        int i1 = kIdxNone;
        auto fold = [&](float q, int idx) {
            const bool better = q < m1;
            m2 = better ? m1 : fminf(m2, q);
            i1 = better ? idx : i1;
            m1 = fminf(m1, q);
        };
        for (int k = 0; k < KC; ++k) {
            const float g = gs[k];
            const float *uk = ufs + k * R;
            if (h0)
                fold(place_node_part<RT>(uk, __fadd_rn(g, pen0), p32s, rg, R, n0), k * N + n0);
            if (h1)
                fold(place_node_part<RT>(uk, __fadd_rn(g, pen1), p32s, rg, R, n1), k * N + n1);
        }
        const Best x = allreduce_best(Best{m1, i1, m2});
        const float thr = __fadd_ru(x.m1, c.sp.e2);
        int win = x.idx;
        double s_w = 0.0;
        bool has_s = false;
        if (c.sp.exact || !(x.m2 > thr)) {
            // survivors rescored in fp64: v_kn = v_k - (double)pen_n, then the chain of Eq. esp_score
            long long key = 0x7fffffffffffffffLL;
            int bi = kIdxNone;
            for (int k = 0; k < KC; ++k) {
                if ((dup >> k) & 1u)
                    continue;
                const int32_t *uk = us + k * R;
                int32_t u[Cols<RT>::N];
#pragma unroll
                for (int r = 0; r < Cols<RT>::N; ++r)
                    u[r] = (RT != 0 || r < R) ? uk[r] : 0;
                const float g = gs[k];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int n = h ? n1 : n0;
                    if (!(h ? h1 : h0))
                        continue;
                    const float pen = h ? pen1 : pen0;
                    const float q = place_node_part<RT>(ufs + k * R, __fadd_rn(g, pen), p32s, rg, R, n);
                    if (!c.sp.exact && !(q <= thr))
                        continue;
                    const double v = __dsub_rn(vs[k], (double)pen);
                    const long long kk = order_key(exact_score<RT, true>(u, v, n, c.sp, R, rg));
                    if (kk < key) {
                        key = kk;
                        bi = k * N + n;
                    }
                }
            }
#pragma unroll
            for (int dd = 16; dd >= 1; dd >>= 1) {
                const long long ok = __shfl_xor_sync(FULL, key, dd);
                const int oi = __shfl_xor_sync(FULL, bi, dd);
                if (ok < key || (ok == key && oi < bi)) {
                    key = ok;
                    bi = oi;
                }
            }
            win = bi;
            s_w = key_value(key);
            has_s = true;
            if (lane == 0)
                atomicAdd(st.stats, 1ull);
        }
        if (lane == 0) {
            const int k = win / N, n = win - k * N;
            int32_t u[Cols<RT>::N];
#pragma unroll
            for (int r = 0; r < Cols<RT>::N; ++r)
                u[r] = (RT != 0 || r < R) ? us[k * R + r] : 0;
            const double v = __dsub_rn(vs[k], (double)__fmul_rn(sens, __ldg(pl.D + aj * NT + __ldg(pl.node_type + n))));
            take_winner<RT, true>(c, j, win, u, v, n, has_s, s_w);
        }
    }
    flush<RT, true>(c, lane);
}

template <int RT, bool PLAIN>
__global__ void __launch_bounds__(kPlaceWarps * 32, 4) k_place(DevTable t, DevState st, DevPlace pl, SolveArgs a,
                                                            int round, int kind)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int R = RT ? RT : t.R, rg = t.r_global;
    const PlaceWarpSmem ws = place_warp_smem(smem, wid, R, t.P, pl.KC);
    const int w = blockIdx.x * kPlaceWarps + wid;
    if (w >= pl.n_warps)
        return;

    WarpCtx<RT, true> c;
    c.t = t;
    c.st = st;
    c.scen_warps = pl.scen_warps;
    c.a = a;
    c.round = round;
    c.R = R;
    c.rg = rg;
    c.kind = PLAIN ? (int)PASS_ROUND : kind;
    c.want_min = PLAIN ? false : ((kind == PASS_FINAL) || (st.dual_trace != nullptr));
    c.want_hash = PLAIN ? false : ((kind == PASS_ROUND) && (st.hash_trace != nullptr));
    c.uniform_k = 0;
    c.log2_k = 0;
    c.s = -1;
#pragma unroll
    for (int r = 0; r < Cols<RT>::N; ++r)
        c.acc[r] = 0;
    c.hacc = 0;
    place_jobs<RT>(c, pl, ws, pl.warp_job[w], pl.warp_job[w + 1], lane);
}

// Grid-wide barrier of a cooperative launch: every CTA adds 1 to the count of *bar (esp_barrier.h) and waits
// until it reaches target (= CTAs x barriers so far). Thread 0 waits, bounded (about 4 s); on expiry, or
// when another CTA gave up, the barrier fails for the whole CTA, the device error word is flagged and the word's
// abort bit set so that no CTA waits for it any longer. Every access of the word is 64 bits wide; the arrival
// releases (cumulatively, after the CTA barrier) what every thread of the CTA did before it.
__device__ bool grid_barrier(unsigned long long *bar, unsigned long long target, unsigned int *err, int *ok_s)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(bar), "l"(1ull) : "memory");
        uint64_t t0;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        bool ok = false;
        for (uint32_t it = 0;; ++it) {
            unsigned long long v;
            asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(bar) : "memory");
            if (bar_reached(v, target)) {
                ok = true;
                break;
            }
            if (bar_aborted(v))
                break;
            if (it > 64) {
                uint64_t t1;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
                if (t1 - t0 > 4000000000ull)
                    break;
                __nanosleep(200);
            }
        }
        if (!ok) {
            atomicOr(err, DEV_ERR_TIMEOUT);
            atomicOr(bar, kBarAbort);
        }
        *ok_s = ok ? 1 : 0;
    }
    __syncthreads();
    return *ok_s != 0;
}

// Exact score of Eq. esp_score (the chain of exact_score) with the prices in shared memory.
template <int RT>
__device__ __forceinline__ double exact_score_shared(const int32_t *u, double v, int g, const double *p64, int R,
                                                     int rg)
{
    double s = -v;
#pragma unroll
    for (int r = 0; r < Cols<RT>::N; ++r) {
        if (RT == 0 && r >= R)
            break;
        s = __fma_rn(p64[r >= rg ? rg + (R - rg) * g + (r - rg) : r], __int2double_rn(u[r]), s);
    }
    return s;
}

// All T rounds of a placement solve in one cooperative launch of one CTA (pr.warps warps, at most W) per SM. Each warp
// holds one job in shared memory for the whole solve:
// configuration units (int32 and fp32), values, and per lane the penalties of its two nodes. Each
// CTA holds the whole price state of every scenario in shared memory (S * P <= kPlaceResMaxPrices).
// A round: best responses of the CTA's jobs (the arithmetic of k_place), their demand summed in
// shared memory and added to buffer round % 3 of U3 with one atomic per column, a grid barrier,
// then Eq. price_update by the whole CTA from the same totals (one price per thread; per-scenario
// maxima and flags through shared atomics, which are order-independent), identical in every CTA.
// What bounds it is the chain of a round: best response, shared sums, atomics, grid barrier, update, bound. One
// job per warp: 9.6 us per round of 4096 jobs x 12 x 64, where two jobs one after the other in each of 16 warps,
// the sums as 64-bit shared atomics, two trips to L2 per poll of the barrier, two fp64 divides per price and the
// bound in fp64 took 15.0 (all but the first of these: 12.1). The jobs are spread over every SM, so that no more
// warps share one than they must; the bound W only sets the registers (64 per thread for 17 to 32 warps, which
// spills for R other than 8: 4096 jobs of R = 16 16.2 us per round, 20.6 before).
// CTA 0 writes the price and demand trajectories, clears the buffer that was last read before this
// round's barrier, and publishes the final state for the final pass. Hash and dual traces are not
// supported here (the host keeps the per-round launches for them).
template <int RT, int W>
__global__ void __launch_bounds__(W * 32, 1) k_place_res(DevTable t, DevState st, DevPlace pl,
                                                                   SolveArgs a, PlaceRes pr)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int ok_s;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int R = RT ? RT : t.R, rg = t.r_global;
    const int S = t.S, P = t.P, SP = S * P, T = a.T;
    const int KC = pl.KC, N = pl.N, NT = pl.NT;
    const PlaceResLayout L = place_res_layout(S, P, KC, R, pr.warps);

    // the CTA's demand of each price as two 32-bit sums, of the low 16 bits and of the rest of its winners' units:
    // an atomic add of 64 bits in shared memory is a loop of compare-and-swaps, which the columns that all
    // jobs share kept repeating
    uint32_t *Uc = reinterpret_cast<uint32_t *>(smem + L.u);
    static_assert(W <= 65536, "a sum of 16-bit parts fits 32 bits");
    double *lam_s = reinterpret_cast<double *>(smem + L.lam);
    double *p64_s = reinterpret_cast<double *>(smem + L.p64);
    double *rcp_s = reinterpret_cast<double *>(smem + L.rcp);
    long long *cap_s = reinterpret_cast<long long *>(smem + L.cap);
    float *p32_s = reinterpret_cast<float *>(smem + L.p32);
    float *eb_s = reinterpret_cast<float *>(smem + L.eb);
    int *frozen_s = reinterpret_cast<int *>(smem + L.flags);
    int *status_s = frozen_s + S, *conv_s = frozen_s + 2 * S, *rounds_s = frozen_s + 3 * S;
    int *bad_s = frozen_s + 4 * S;
    unsigned long long *dmax_s = reinterpret_cast<unsigned long long *>(smem + L.maxes);
    unsigned long long *amax_s = dmax_s + S;
    unsigned char *wb = smem + L.warps + (size_t)wid * L.warp_bytes;
    float *gs = reinterpret_cast<float *>(wb);

    // ---- the price state from k_init, and this warp's jobs
    for (int i = tid; i < SP; i += blockDim.x) {
        lam_s[i] = st.lam[i];
        p64_s[i] = st.p64[i];
        p32_s[i] = st.p32[i];
        cap_s[i] = t.cap[i];
        rcp_s[i] = st.rcp[i];
        Uc[2 * i] = Uc[2 * i + 1] = 0u;
    }
    for (int i = tid; i < S; i += blockDim.x) {
        eb_s[i] = st.ebound[i];
        frozen_s[i] = st.frozen[i];
        status_s[i] = 0;
        conv_s[i] = 0;
        rounds_s[i] = 0;
        bad_s[i] = 0;
        dmax_s[i] = 0ull;
        amax_s[i] = 0ull;
    }
    // of the scenario whose bound this warp computes (the first, when there are more scenarios than warps)
    const float own_umax = wid < S && lane < R ? __int2float_ru(st.umax[(size_t)wid * R + lane]) : 0.0f;
    const float own_vmax = wid < S ? __double2float_ru(st.vmax[wid]) : 0.0f;
    const int64_t j = (int64_t)blockIdx.x * pr.warps + wid;
    const bool has_job = j < pr.n_jobs;
    const int n0 = lane, n1 = lane + 32;
    const bool h0 = n0 < N, h1 = n1 < N;
    float pa = 0.0f, pb = 0.0f;   // penalties of the lane's nodes
    uint32_t dup = 0u;
    int sc = 0;
    int32_t *us = reinterpret_cast<int32_t *>(wb + L.job_units);
    float *ufs = reinterpret_cast<float *>(wb + L.job_ufs);
    double *vs = reinterpret_cast<double *>(wb + L.job_vals);
    float *pens = reinterpret_cast<float *>(wb + L.job_pens);
    if (has_job) {
        sc = (int)(j / t.J);
        for (int i = lane; i < KC * R; i += 32) {
            const int32_t u = __ldg(pl.cfg_units + j * KC * R + i);
            us[i] = u;
            ufs[i] = __int2float_rn(u);
        }
        for (int k = lane; k < KC; k += 32)
            vs[k] = __ldg(pl.cfg_values + j * KC + k);
        const float sens = __ldg(pl.sens + j);
        const int aj = __ldg(pl.job_type + j);
        dup = __ldg(pl.cfg_dup + j);
        pa = h0 ? __fmul_rn(sens, __ldg(pl.D + aj * NT + __ldg(pl.node_type + n0))) : 0.0f;
        pb = h1 ? __fmul_rn(sens, __ldg(pl.D + aj * NT + __ldg(pl.node_type + n1))) : 0.0f;
        pens[n0] = pa;
        pens[n1] = pb;
    }
    __syncthreads();

    for (int round = 0; round < T; ++round) {
        unsigned long long *Ub = pr.U3 + (size_t)(round % 3) * SP;

        // ---- best response of this warp's job at the CTA's prices
        if (has_job && !frozen_s[sc]) {
            const float *p32s = p32_s + (size_t)sc * P;
            const double *p64s = p64_s + (size_t)sc * P;
            ScenarioPrices sp;
#pragma unroll
            for (int r = 0; r < Cols<RT>::N; ++r)
                sp.pf[r] = (r < rg) ? p32s[r] : 0.0f;
            const float e = eb_s[sc];
            sp.exact = !(e < INFINITY);
            sp.e2 = sp.exact ? INFINITY : 2.0f * e;
            __syncwarp();
            for (int k = lane; k < KC; k += 32)
                gs[k] = ((dup >> k) & 1u) ? INFINITY : place_global_part<RT>(ufs + k * R, vs[k], sp, rg);
            __syncwarp();
            // this lane's node prices (columns r >= rg of nodes n0, n1) in registers
            const int nc = R - rg;
            float pn0[Cols<RT>::N], pn1[Cols<RT>::N];
#pragma unroll
            for (int c2 = 0; c2 < Cols<RT>::N; ++c2) {
                pn0[c2] = (c2 < nc && h0) ? p32s[rg + nc * n0 + c2] : 0.0f;
                pn1[c2] = (c2 < nc && h1) ? p32s[rg + nc * n1 + c2] : 0.0f;
            }
            // q of (k, n0) and (k, n1): the chain of place_node_part, same operations in the same order
            auto node_q = [&](int k, float &q0, float &q1) {
                const float g = gs[k];
                const float *uk = ufs + k * R + rg;
                q0 = __fadd_rn(g, pa);
                q1 = __fadd_rn(g, pb);
#pragma unroll
                for (int c2 = 0; c2 < Cols<RT>::N; ++c2) {
                    if (c2 >= nc)
                        break;
                    const float uf = uk[c2];
                    q0 = __fmaf_rn(pn0[c2], uf, q0);
                    q1 = __fmaf_rn(pn1[c2], uf, q1);
                }
            };
            float m1 = INFINITY, m2 = INFINITY;
            int i1 = kIdxNone;
            auto fold = [&](float qv, int idx) {
                const bool better = qv < m1;
                m2 = better ? m1 : fminf(m2, qv);
                i1 = better ? idx : i1;
                m1 = fminf(m1, qv);
            };
#pragma unroll 4
            for (int k = 0; k < KC; ++k) {
                float q0, q1;
                node_q(k, q0, q1);
                if (h0)
                    fold(q0, k * N + n0);
                if (h1)
                    fold(q1, k * N + n1);
            }
            // smallest, second smallest and holder over the warp by hardware reductions: the holder offers its
            // second smallest, the others their smallest; two holders make both equal (and the job ambiguous)
            const float g1 = warp_min_f32(m1);
            const unsigned holders = __ballot_sync(FULL, m1 == g1);
            const float o2 = warp_min_f32(m1 == g1 ? m2 : m1);
            const float g2 = (holders & (holders - 1u)) ? g1 : o2;
            const float thr = __fadd_ru(g1, sp.e2);
            int win = __shfl_sync(FULL, i1, __ffs((int)holders) - 1);
            if (sp.exact || !(g2 > thr)) {
                // survivors (q <= thr; all in exact mode; repeated configurations never), listed in
                // (k, node half, lane) order; up to 32 are rescored in fp64 one per lane
                int *cand = reinterpret_cast<int *>(wb + L.cand);
                int total = 0;
                for (int k = 0; k < KC && total <= 32; ++k) {
                    if ((dup >> k) & 1u)
                        continue;
                    float q0, q1;
                    node_q(k, q0, q1);
                    const unsigned b0 = __ballot_sync(FULL, h0 && (sp.exact || q0 <= thr));
                    const unsigned b1 = __ballot_sync(FULL, h1 && (sp.exact || q1 <= thr));
                    const unsigned below = (1u << lane) - 1u;
                    const int i0 = total + __popc(b0 & below), i1s = total + __popc(b0) + __popc(b1 & below);
                    if (((b0 >> lane) & 1u) && i0 < 32)
                        cand[i0] = k * N + n0;
                    if (((b1 >> lane) & 1u) && i1s < 32)
                        cand[i1s] = k * N + n1;
                    total += __popc(b0) + __popc(b1);
                }
                __syncwarp();
                long long key = 0x7fffffffffffffffLL;
                int bi = kIdxNone;
                if (total <= 32) {
                    if (lane < total) {
                        const int ci = cand[lane];
                        const int k = ci / N, n = ci - k * N;
                        int32_t u[Cols<RT>::N];
#pragma unroll
                        for (int r = 0; r < Cols<RT>::N; ++r)
                            u[r] = (RT != 0 || r < R) ? us[k * R + r] : 0;
                        const double v = __dsub_rn(vs[k], (double)pens[n]);
                        key = order_key(exact_score_shared<RT>(u, v, n, p64s, R, rg));
                        bi = ci;
                    }
                } else {
                    // many survivors: each lane rescores its own
                    for (int k = 0; k < KC; ++k) {
                        if ((dup >> k) & 1u)
                            continue;
                        float q0, q1;
                        node_q(k, q0, q1);
                        const int32_t *uk = us + k * R;
                        int32_t u[Cols<RT>::N];
#pragma unroll
                        for (int r = 0; r < Cols<RT>::N; ++r)
                            u[r] = (RT != 0 || r < R) ? uk[r] : 0;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int n = h ? n1 : n0;
                            if (!(h ? h1 : h0))
                                continue;
                            if (!sp.exact && !((h ? q1 : q0) <= thr))
                                continue;
                            const double v = __dsub_rn(vs[k], (double)(h ? pb : pa));
                            const long long kk = order_key(exact_score_shared<RT>(u, v, n, p64s, R, rg));
                            if (kk < key) {
                                key = kk;
                                bi = k * N + n;
                            }
                        }
                    }
                }
#pragma unroll
                for (int dd = 16; dd >= 1; dd >>= 1) {
                    const long long ok = __shfl_xor_sync(FULL, key, dd);
                    const int oi = __shfl_xor_sync(FULL, bi, dd);
                    if (ok < key || (ok == key && oi < bi)) {
                        key = ok;
                        bi = oi;
                    }
                }
                __syncwarp();
                win = bi;
                if (lane == 0)
                    atomicAdd(st.stats, 1ull);
            }
            // the winner's units into the CTA's demand (lane r: column r)
            const int kw = win / N, nw = win - kw * N;
            if (lane < R) {
                const uint32_t u = (uint32_t)us[kw * R + lane];
                const int col = lane >= rg ? rg + (R - rg) * nw + (lane - rg) : lane;
                uint32_t *dst = Uc + 2 * ((size_t)sc * P + col);
                if (u & 0xffffu)
                    atomicAdd(dst, u & 0xffffu);
                if (u >> 16)
                    atomicAdd(dst + 1, u >> 16);
            }
        }
        __syncthreads();
        // ---- the CTA's demand into the round's buffer; per-scenario reductions reset
        for (int i = tid; i < SP; i += blockDim.x) {
            const uint2 v = *reinterpret_cast<const uint2 *>(Uc + 2 * i);
            if ((v.x | v.y) != 0u) {
                atomicAdd(Ub + i, (unsigned long long)v.x + ((unsigned long long)v.y << 16));
                Uc[2 * i] = Uc[2 * i + 1] = 0u;
            }
        }
        for (int i = tid; i < S; i += blockDim.x) {
            bad_s[i] = 0;
            dmax_s[i] = 0ull;
            amax_s[i] = 0ull;
        }
        if (!grid_barrier(pr.bar, (unsigned long long)(round + 1) * gridDim.x, st.err, &ok_s))
            break;

        // ---- Eq. price_update of every scenario, one price per thread: the new prices are computed
        // into registers, and written once no price of the scenario became non-finite
        const double eta = step_size(a.eta0, a.step, round);
        const bool lead = blockIdx.x == 0;
        constexpr int kThreads = place_res_min_warps(W) * 32, kPrices = (kPlaceResMaxPrices + kThreads - 1) / kThreads;   // per thread
        double nl_r[kPrices], pe_r[kPrices];
#pragma unroll
        for (int m = 0; m < kPrices; ++m) {
            const int i = tid + m * (int)blockDim.x;
            nl_r[m] = pe_r[m] = 0.0;
            if (i >= SP)
                break;
            const int sc = i / P;
            if (frozen_s[sc])
                continue;
            const long long U = (long long)__ldcg(Ub + i);
            if (lead && st.dem_trace)
                st.dem_trace[((size_t)sc * T + round) * P + (i - sc * P)] = U;
            const double lam = lam_s[i];
            const double capd = (double)cap_s[i], rcp = rcp_s[i];
            const double nl = price_step_rcp(lam, U, cap_s[i], capd, rcp, eta, a.mode);
            nl_r[m] = nl;
            pe_r[m] = effective_price_rcp(nl, capd, rcp, a.mode);
            if (!isfinite(nl))
                atomicOr(bad_s + sc, 1);
            if (a.tol > 0.0) {   // maxima of the stopping rule (non-negative doubles order as integers)
                atomicMax(dmax_s + sc, (unsigned long long)__double_as_longlong(fabs(nl - lam)));
                atomicMax(amax_s + sc, (unsigned long long)__double_as_longlong(fabs(lam)));
            }
        }
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kPrices; ++m) {
            const int i = tid + m * (int)blockDim.x;
            if (i >= SP)
                break;
            const int sc = i / P;
            if (frozen_s[sc] || bad_s[sc])
                continue;
            lam_s[i] = nl_r[m];
            if (lead && st.lam_trace)
                st.lam_trace[((size_t)sc * (T + 1) + round + 1) * P + (i - sc * P)] = nl_r[m];
            p64_s[i] = pe_r[m];
            p32_s[i] = __double2float_rn(pe_r[m]);
        }
        __syncthreads();
        // stopping rule and screen bound, one warp per scenario. E only has to bound the screen's error from
        // above: it is computed in fp32 with every operation rounded up, from p <= p32 (1 + 2^-23) + 2^-149 and
        // M = max|v| + sum_r (largest p_r) max u_r; no fp64 operation, and one reduction per node column
        for (int sc = wid; sc < S; sc += pr.warps) {
            if (frozen_s[sc])
                continue;
            if (bad_s[sc]) {
                if (lane == 0) {
                    status_s[sc] = 2;
                    frozen_s[sc] = 1;
                }
                continue;
            }
            const double dmax = __longlong_as_double((long long)dmax_s[sc]);
            const double amax = __longlong_as_double((long long)amax_s[sc]);
            const bool conv = (a.tol > 0.0) && (dmax <= a.tol * fmax(1.0, amax));
            const float *p32s = p32_s + (size_t)sc * P;
            const float umax_up = sc == wid ? own_umax : lane < R ? __int2float_ru(st.umax[(size_t)sc * R + lane]) : 0.0f;
            const float vmax_up = sc == wid ? own_vmax : __double2float_ru(st.vmax[sc]);
            float p = lane < rg ? p32s[lane] : 0.0f;   // lane r: the largest price of column r
            for (int c2 = 0; c2 < R - rg; ++c2) {
                uint32_t pm = 0u;                      // prices are not negative: their bits order as they do
                for (int gi = lane; gi < t.n_groups; gi += 32)
                    pm = max(pm, __float_as_uint(p32s[rg + (R - rg) * gi + c2]));
                pm = __reduce_max_sync(FULL, pm);
                p = lane == rg + c2 ? __uint_as_float(pm) : p;
            }
            const float p_up = __fadd_ru(__fmul_ru(p, 1.0f + 0x1p-23f), 0x1p-149f);
            const bool huge = __any_sync(FULL, lane < R && !(p_up <= 0x1p100f));
            float term = lane < R ? __fmul_ru(p_up, umax_up) : 0.0f;
#pragma unroll
            for (int d = 8; d >= 1; d >>= 1)           // lanes 0 .. 15 hold the terms
                term = __fadd_ru(term, __shfl_xor_sync(FULL, term, d));
            const float M = __fadd_ru(vmax_up, term);
            if (lane == 0) {
                if (lead && st.time_trace)
                    st.time_trace[(size_t)sc * T + round] = global_ns();
                rounds_s[sc] = round + 1;
                if (conv) {
                    conv_s[sc] = 1;
                    frozen_s[sc] = 1;
                }
                eb_s[sc] = a.exact_only || huge || !(M <= 0x1p100f)
                               ? INFINITY
                               : __fadd_ru(__fmul_ru(M, (4.0f * R + 16.0f) * 0x1p-24f), 0x1p-99f);
            }
        }
        if (lead) {   // buffer (round + 2) % 3 was last read before this round's barrier
            unsigned long long *Uz = pr.U3 + (size_t)((round + 2) % 3) * SP;
            for (int i = tid; i < SP; i += blockDim.x)
                Uz[i] = 0ull;
        }
        __syncthreads();
    }
    // ---- CTA 0 publishes the final price state for the final pass and the objectives
    if (blockIdx.x == 0) {
        for (int i = tid; i < SP; i += blockDim.x) {
            st.lam[i] = lam_s[i];
            st.p64[i] = p64_s[i];
            st.p32[i] = p32_s[i];
        }
        for (int i = tid; i < S; i += blockDim.x) {
            st.ebound[i] = eb_s[i];
            st.frozen[i] = frozen_s[i];
            st.status[i] = status_s[i];
            st.converged[i] = conv_s[i];
            st.rounds_run[i] = rounds_s[i];
        }
    }
}

}  // namespace

int place_smem_bytes(int R, int P, int KC, int N, int NT)
{
    (void)N;
    (void)NT;
    return kPlaceWarps * place_warp_bytes(R, P, KC);
}

template <typename F>
static auto place_dispatch(int R, bool plain, F &&f)
{
    if (R == 8)
        return plain ? f(reinterpret_cast<const void *>(&k_place<8, true>)) : f(reinterpret_cast<const void *>(&k_place<8, false>));
    return plain ? f(reinterpret_cast<const void *>(&k_place<0, true>)) : f(reinterpret_cast<const void *>(&k_place<0, false>));
}

int place_ctas_per_sm(int R, int P, int KC, int N, int NT)
{
    const int smem = place_smem_bytes(R, P, KC, N, NT);
    int best = 1 << 30;
    for (int plain = 0; plain < 2; ++plain) {
        const int n = place_dispatch(R, plain != 0, [&](const void *fn) -> int {
            if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
                return 0;
            int m = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, fn, kPlaceWarps * 32, smem) != cudaSuccess)
                return 0;
            return m;
        });
        best = n < best ? n : best;
    }
    return best;
}

cudaError_t launch_place(const DevTable &t, const DevState &st, const DevPlace &pl, const SolveArgs &a, int round,
                         PassKind kind, int grid, cudaStream_t stream)
{
    const int smem = place_smem_bytes(t.R, t.P, pl.KC, pl.N, pl.NT);
    const bool plain = kind == PASS_ROUND && st.hash_trace == nullptr && st.dual_trace == nullptr;
    if (t.R == 8) {
        if (plain)
            k_place<8, true><<<grid, kPlaceWarps * 32, smem, stream>>>(t, st, pl, a, round, kind);
        else
            k_place<8, false><<<grid, kPlaceWarps * 32, smem, stream>>>(t, st, pl, a, round, kind);
    } else {
        if (plain)
            k_place<0, true><<<grid, kPlaceWarps * 32, smem, stream>>>(t, st, pl, a, round, kind);
        else
            k_place<0, false><<<grid, kPlaceWarps * 32, smem, stream>>>(t, st, pl, a, round, kind);
    }
    return cudaGetLastError();
}

int place_res_smem_bytes(int S, int P, int KC, int R, int warps)
{
    return place_res_layout(S, P, KC, R, warps).total;
}

static const void *place_res_kernel(int R, int warps)
{
    if (R == 8)
        return warps <= 8    ? reinterpret_cast<const void *>(&k_place_res<8, 8>)
               : warps <= 16 ? reinterpret_cast<const void *>(&k_place_res<8, 16>)
                             : reinterpret_cast<const void *>(&k_place_res<8, 32>);
    return warps <= 8    ? reinterpret_cast<const void *>(&k_place_res<0, 8>)
           : warps <= 16 ? reinterpret_cast<const void *>(&k_place_res<0, 16>)
                         : reinterpret_cast<const void *>(&k_place_res<0, 32>);
}

int place_res_ctas_per_sm(int S, int P, int KC, int R, int warps)
{
    const void *fn = place_res_kernel(R, warps);
    // the limit is the kernel's, not the table's: the device's largest for every one
    int m = 0, dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, fn, warps * 32, place_res_smem_bytes(S, P, KC, R, warps)) !=
            cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return m;
}

static cudaError_t place_res_launch(const DevTable &t, const DevState &st, const DevPlace &pl, const SolveArgs &a,
                                    const PlaceRes &pr, cudaStream_t stream, bool hold_barrier)
{
    cudaError_t e = cudaMemsetAsync(pr.bar, hold_barrier ? kBarHeldByte : 0, sizeof(*pr.bar), stream);
    if (e == cudaSuccess)   // the last rounds of the previous solve leave demand in two buffers
        e = cudaMemsetAsync(pr.U3, 0, 3 * (size_t)t.S * t.P * sizeof(unsigned long long), stream);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)pr.grid);
    cfg.blockDim = dim3((unsigned)pr.warps * 32);
    cfg.dynamicSmemBytes = (size_t)place_res_smem_bytes(t.S, t.P, pl.KC, t.R, pr.warps);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // every CTA co-resident: the grid barrier can complete
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&t, (void *)&st, (void *)&pl, (void *)&a, (void *)&pr};
    return cudaLaunchKernelExC(&cfg, place_res_kernel(t.R, pr.warps), args);
}

cudaError_t launch_place_res(const DevTable &t, const DevState &st, const DevPlace &pl, const SolveArgs &a,
                             const PlaceRes &pr, cudaStream_t stream)
{
    return place_res_launch(t, st, pl, a, pr, stream, false);
}

cudaError_t launch_place_res_held(const DevTable &t, const DevState &st, const DevPlace &pl, const SolveArgs &a,
                                  const PlaceRes &pr, cudaStream_t stream)
{
    return place_res_launch(t, st, pl, a, pr, stream, true);
}

}  // namespace esp
