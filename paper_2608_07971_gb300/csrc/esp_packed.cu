// Evaluation passes over the packed screen copy (esp_packed.h) of the ESP tatonnement (Sec. 3.2.2 and
// 3.2.3) for sm_103a: one launch per round with the price update fused in, and every round of a solve
// in one cooperative launch.
//
// What bounds them: a table larger than L2 streams from HBM every round. The passes this design
// replaced staged 4R + 8 bytes per option through shared memory, 128 options at a time; the what-if batch
// (R = 6, 32 bytes per option) ran at 0.995 of the copy bandwidth with 88% of the issue slots taken (668
// warp instructions per 128 options), so neither fewer bytes nor fewer instructions alone would have
// helped. Here an option takes 16 bytes, a warp screens 256 options per step, eight per lane, and a step is
// one bulk copy into one of the warp's two slots, two steps ahead.
//
// Screen. A lane screens eight consecutive options of a job. Unit fields become floats by inserting the
// exponent of 2^23 (one logic op for a low field, one funnel shift for a high field) and subtracting
// 2^23, exactly; the two fields of a word run as one packed fp32 pair (add.rn.f32x2, fma.rn.f32x2), the
// low fields accumulating from -v, the high fields from 0, and q is the sum of both chains. Against the
// exact score each chain has at most R roundings and the last sum one more, each within 2^-24 of
// M = |v| + sum_r p_r u_r, so |q - s| <= (R + 4) u M (1 + small) + 2^-99 holds as for the chain in column
// order, and the decision rule and its proof are those of esp_kernels.cu.
//
// Tables with a group column (G): the option's group slot is a field of one of its words, the columns priced
// per group are its last word, and their two prices come from a table in the warp's shared memory. The
// placement table of 4096 jobs x 768 options (R = 8, 64 groups; 20 bytes per option instead of 42) takes 28.2 us
// per round where the staged pass took 77.4; of the 28, 19 are the screen (63 MB, which L2 holds), the rest the
// chain of the slowest ambiguous job and of the update of 134 prices.
//
// The winner's units come from the words in the slot, and so do those of options that are scored exactly (the
// survivors of ambiguous jobs, every option in exact mode, the winners of the final pass): of the table itself only
// their fp64 values are read.

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "esp_device.cuh"
#include "esp_kernels.h"
#include "esp_ptx.cuh"
#include "esp_warp.cuh"

namespace esp {

namespace {

#ifndef ESP_PACK_CTAS
#define ESP_PACK_CTAS 5
#endif
constexpr int kPackWarps = 4;        // warps per CTA
constexpr int kPackSlots = 2;        // steps a warp holds: the one being screened and one on its way
// Winners a lane's 32-bit sums may take between flushes: each is below 2^23, so 511 fit; a tile adds at
// most 8 per step and kPackTileSteps (8) steps (a job of more steps counts once).
constexpr uint32_t kPackSpill = 511 - 8 * 8;

// Resident CTAs the register budget must allow (grouped with five: 44.1 us per round of the placement table
// of 4096 jobs x 768 options against 38.7, for the spills).
constexpr int pack_min_ctas(int nw, bool grouped = false)
{
    return grouped ? 4 : nw <= 3 ? ESP_PACK_CTAS : nw == 4 ? 5 : 4;
}

// Shared memory of a warp: the slots, their barriers, then the fp64 prices of the columns that every option shares.
constexpr int kPackPriceBytes = kMaxR * 8;
__host__ __device__ constexpr int pack_slot_bytes(int nw)
{
    return (nw + 1) * kPackStepVecs * 16;
}
__host__ __device__ constexpr int pack_warp_bytes(int nw)
{
    return kPackSlots * pack_slot_bytes(nw) + 16 + kPackPriceBytes;
}

__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The warp's state for the scenario it is in.
template <int NW>
struct Ctx {
    unsigned long long price[NW];   // fp32 prices of word k's (low, high) fields
    uint32_t lo[NW], hi[NW];        // the lane's demand since the last flush, per field
    uint32_t wins;                  // upper bound of the winners in them
    unsigned long long hash;
    const double *p64;              // fp64 prices of the scenario
    unsigned char *groups;          // shared memory behind the prices; grouped tables: two fp32 prices of each slot
    bool have64;                    // the fp64 prices below `groups` are this scenario's (fetch_prices)
    float e2;                       // 2E, +inf: exact evaluation
    bool exact, skip;
    int s;                          // scenario, -1: none
    int tiles;                      // tiles evaluated since the last arrival
    unsigned int resolved;
};

// Scores of the four options of vector `v` of plane 0; the other planes follow `plane` vectors apart.
template <int NW, bool G>
__device__ __forceinline__ void screen4(const uint4 *v, int plane, const PackFormat &f, const Ctx<NW> &c, float *q)
{
    const unsigned long long bias = pack2(-8388608.0f, -8388608.0f);
    const uint4 n = v[0];
    unsigned long long acc[4] = {pack2(__uint_as_float(n.x), 0.0f), pack2(__uint_as_float(n.y), 0.0f),
                                 pack2(__uint_as_float(n.z), 0.0f), pack2(__uint_as_float(n.w), 0.0f)};
    // the last word's prices are those of the option's group
    unsigned long long own[4];
    if (G) {
        const uint4 y = v[(f.g_word + 1) * plane];
        const uint32_t x[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int o = 0; o < 4; ++o)
            own[o] = *reinterpret_cast<const unsigned long long *>(c.groups + 8 * ((x[o] >> f.g_shift) & f.g_mask));
    }
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        const uint4 y = v[(k + 1) * plane];
        const uint32_t x[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const uint32_t lo = (x[o] & f.mask[k]) | 0x4b000000u;
            const uint32_t hi = __funnelshift_r(x[o], f.magic[k], f.shift[k]);
            acc[o] = fma2(G && k == NW - 1 ? own[o] : c.price[k], add2(pack2(__uint_as_float(lo), __uint_as_float(hi)), bias), acc[o]);
        }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
        const float2 t = unpack2(acc[o]);
        q[o] = t.x + t.y;
    }
}

// Smallest and second smallest of four.
__device__ __forceinline__ void two_smallest(const float *q, float &m1, float &m2)
{
    const float a0 = fminf(q[0], q[1]), a1 = fmaxf(q[0], q[1]);
    const float b0 = fminf(q[2], q[3]), b1 = fmaxf(q[2], q[3]);
    m1 = fminf(a0, b0);
    m2 = fminf(fmaxf(a0, b0), fminf(a1, b1));
}

// Everything a pass needs beyond the warp's own state.
struct Pass {
    const DevTable &t;
    const DevState &st;
    const DevPack &pk;
    const SolveArgs &a;
    int round, kind, lane;
    bool want_min, want_hash;   // minimal reduced costs; selection fingerprints
};

// The scenario's demand totals.
template <int NW>
__device__ __forceinline__ unsigned long long *totals(const Pass &ps, const Ctx<NW> &c)
{
    return (ps.kind == PASS_ROUND ? ps.st.U : ps.st.U_final) + (size_t)c.s * ps.t.P;
}

// Group columns of a winner: straight to the totals of its group (a scenario's winners spread over its groups).
template <int NW>
__device__ __forceinline__ void add_group(const Pass &ps, const Ctx<NW> &c, uint32_t x, uint32_t slot_word)
{
    const PackFormat &f = ps.pk.fmt;
    const uint32_t lo = x & f.mask[NW - 1], hi = f.col_hi[NW - 1] >= 0 ? x >> f.shift[NW - 1] : 0u;
    const int rg = ps.t.r_global;
    unsigned long long *dst =
        totals(ps, c) + rg + (ps.t.R - rg) * (int)pack_slot_group((slot_word >> f.g_shift) & f.g_mask);
    if (lo != 0u)
        atomicAdd(dst, (unsigned long long)lo);
    if (hi != 0u)
        atomicAdd(dst + 1, (unsigned long long)hi);
}

// Adds the units in the word at w (plane 0) to the lane's demand.
template <int NW, bool G>
__device__ __forceinline__ void add_option(const Pass &ps, Ctx<NW> &c, const uint32_t *w, int plane)
{
    const PackFormat &f = ps.pk.fmt;
#pragma unroll
    for (int k = 0; k < (G ? NW - 1 : NW); ++k) {
        const uint32_t x = w[(k + 1) * plane * 4];
        c.lo[k] += x & f.mask[k];
        c.hi[k] += x >> f.shift[k];
    }
    if (G)
        add_group(ps, c, w[NW * plane * 4], w[(f.g_word + 1) * plane * 4]);
}

// The scenario's fp64 prices into the warp's shared memory, once per scenario (the whole warp calls it). A pass of one
// round fetches them with the scenario's other prices; the persistent pass, which comes to a scenario for each tile,
// only before something is scored exactly.
template <int NW, bool G>
__device__ __forceinline__ void fetch_prices(const Pass &ps, Ctx<NW> &c)
{
    if (c.have64)
        return;
    c.have64 = true;
    if (ps.lane < (G ? ps.t.r_global : ps.t.R))   // through L2: a persistent pass sees them change between rounds
        reinterpret_cast<double *>(c.groups - kPackPriceBytes)[ps.lane] = __ldcg(c.p64 + ps.lane);
    __syncwarp();
}

// A whole number below 2^23 in fp64, by way of its fp32 bits: integer operations instead of a conversion, which would
// take as long a turn of the fp64 unit as the multiply-add that the number is for.
__device__ __forceinline__ double whole_f64(uint32_t u)
{
    const uint32_t b = __float_as_uint(__uint_as_float(0x4b000000u | u) - 8388608.0f);
    return __hiloint2double(b != 0u ? (int)((b >> 3) + (896u << 20)) : 0, (int)(b << 29));   // exponent bias 127 -> 1023
}

// The exact score (the chain of Eq. esp_score in column order) of the option of value v whose words are at w (plane
// 0). The units are whole numbers in the words, so only v is read from the table. (With units and prices read from the
// table and L2 column by column, exact mode took 254 us per round on 256 scenarios of 2048 x 16, R = 6, where the staged
// pass took 204 and this takes 130; the slowest ambiguous job is the end of every round, so a 2048-job cluster went
// from 10.0 to 8.7 us too, the what-if batch from 85 to 81 and the heavy-tailed table from 158 to 153.)
template <int NW, bool G>
__device__ __forceinline__ double exact_words(const Pass &ps, const Ctx<NW> &c, const uint32_t *w, int plane, double v)
{
    const PackFormat &f = ps.pk.fmt;
    const int R = ps.t.R, rg = G ? ps.t.r_global : R;
    const double *p = reinterpret_cast<const double *>(c.groups - kPackPriceBytes);
    double s = -v;
    auto unit = [&](int r) {
        const int at = f.field[r], k = at >> 1;
        const uint32_t x = w[(k + 1) * plane * 4];
        return whole_f64((at & 1) ? x >> f.shift[k] : x & f.mask[k]);
    };
    double pg[2] = {0.0, 0.0};
    if (G) {
        const double *own = c.p64 + rg + (R - rg) * (int)pack_slot_group((w[(f.g_word + 1) * plane * 4] >> f.g_shift) & f.g_mask);
        pg[0] = __ldcg(own);
        if (R - rg == 2)
            pg[1] = __ldcg(own + 1);
    }
#pragma unroll 4
    for (int r = 0; r < rg; ++r)
        s = __fma_rn(p[r], unit(r), s);
    if (G) {
        s = __fma_rn(pg[0], unit(rg), s);
        if (R - rg == 2)
            s = __fma_rn(pg[1], unit(rg + 1), s);
    }
    return s;
}

struct Exact {
    long long key;
    int idx;
};

// The value of the first option in `mask` (rescore's first one; loaded ahead of the prices, so that one trip to memory
// covers both).
__device__ __forceinline__ double first_value(const Pass &ps, int64_t first, uint32_t mask)
{
    return mask != 0u ? __ldg(ps.t.values + first + (__ffs((int)mask) - 1)) : 0.0;
}

// The lexicographic minimum of (s, index) in fp64 over the options first + i, i in the bits of `mask`: the words of
// options 0 .. 3 start at wa, those of 4 .. 7 at wb; v: the first one's value. Their indices are loc + i.
// (Ambiguous jobs only; out of line it made the row loops spill around the call.)
template <int NW, bool G>
__device__ __forceinline__ Exact rescore(const Pass &ps, const Ctx<NW> &c, const uint32_t *wa, const uint32_t *wb, int plane,
                                         int64_t first, uint32_t mask, int loc, double v)
{
    Exact x{0x7fffffffffffffffLL, kIdxNone};
    while (mask != 0u) {
        const int i = __ffs((int)mask) - 1;
        mask &= mask - 1;
        const double next = G ? first_value(ps, first, mask) : 0.0;   // (ungrouped: the registers it takes cost more)
        const long long k = order_key(exact_words<NW, G>(ps, c, (i < 4 ? wa : wb) + (i & 3), plane, v));
        v = G ? next : first_value(ps, first, mask);
        if (k < x.key) {   // increasing index: the first of equal scores stays
            x.key = k;
            x.idx = loc + i;
        }
    }
    return x;
}

// The minimum of (key, idx) over aligned groups of `lanes` lanes.
__device__ __forceinline__ Exact group_min(Exact x, int lanes)
{
    for (int d = 1; d < lanes; d <<= 1) {
        const long long ok = __shfl_xor_sync(FULL, x.key, d);
        const int oi = __shfl_xor_sync(FULL, x.idx, d);
        if (ok < x.key || (ok == x.key && oi < x.idx)) {
            x.key = ok;
            x.idx = oi;
        }
    }
    return x;
}

// Options of a vector that survive the screen (q <= thr; in exact mode every option but duplicates and
// padding); n: their -v32 words.
__device__ __forceinline__ uint32_t survivors(const uint4 &n, const float *q, bool exact, float thr)
{
    return ((n.x != kPackInf && (exact || q[0] <= thr)) ? 1u : 0u) |
           ((n.y != kPackInf && (exact || q[1] <= thr)) ? 2u : 0u) |
           ((n.z != kPackInf && (exact || q[2] <= thr)) ? 4u : 0u) |
           ((n.w != kPackInf && (exact || q[3] <= thr)) ? 8u : 0u);
}

// First option of packed job i. Of a table whose jobs have all the same number of options it is known without
// a load, else with one: an ambiguous job is a chain of trips to memory, and the round waits for the slowest.
__device__ __forceinline__ int64_t first_option(const Pass &ps, int i)
{
    return ps.pk.all_k > 0 ? (int64_t)i * ps.pk.all_k : __ldg(ps.pk.opt0 + i);
}

// Outputs of a winner beyond its demand: its packed job i, local index, value (read where it is wanted), words and,
// when known, exact score.
template <int NW, bool G>
__device__ __forceinline__ void extras(const Pass &ps, Ctx<NW> &c, int i, int local, double v, const uint32_t *w, int plane,
                                       bool have_s, long long key)
{
    const int64_t job = ps.pk.job ? __ldg(ps.pk.job + i) : i;
    if (ps.want_hash)
        c.hash += splitmix64_mix(((uint64_t)(uint32_t)(job - (int64_t)c.s * ps.t.J) << 32) | (uint32_t)local);
    if (ps.kind == PASS_FINAL) {
        ps.st.sel[job] = local;
        ps.st.job_val[job] = v;
    }
    if (ps.want_min)
        ps.st.job_min[job] = have_s ? key_value(key) : exact_words<NW, G>(ps, c, w, plane, v);
}

// Adds the lane's demand to the scenario's totals: every sum across the warp by two hardware reductions
// of 16-bit halves (each below 2^21), then one atomic per field, all fields in one instruction.
template <int NW, bool G>
__device__ __forceinline__ void add_demand(const Pass &ps, Ctx<NW> &c)
{
    constexpr int NU = G ? NW - 1 : NW;   // words of columns without groups
    unsigned long long *dst = totals(ps, c);
    unsigned long long mine = 0ull;
    int col = -1;
#pragma unroll
    for (int i = 0; i < 2 * NU; ++i) {
        const uint32_t v = (i & 1) ? c.hi[i >> 1] : c.lo[i >> 1];
        const unsigned long long x = (unsigned long long)__reduce_add_sync(FULL, v & 0xffffu) +
                                     ((unsigned long long)__reduce_add_sync(FULL, v >> 16) << 16);
        if (ps.lane == i) {
            mine = x;
            col = (i & 1) ? ps.pk.fmt.col_hi[i >> 1] : ps.pk.fmt.col_lo[i >> 1];
        }
    }
#pragma unroll
    for (int k = 0; k < NW; ++k)
        c.lo[k] = c.hi[k] = 0u;
    if (col >= 0 && mine != 0ull)
        atomicAdd(dst + col, mine);
    c.wins = 0;
}

// What an update records before the prices move: the dual value of the round, the fingerprint.
__device__ __forceinline__ void trace_round(const DevTable &t, const DevState &st, const SolveArgs &a, int s, int round,
                                            double lam_part, int lane)
{
    if (st.dual_trace) {   // g(lambda^t) from the minimal reduced costs of round t
        double part = 0.0;
        for (int j = lane; j < t.J; j += 32)
            part += -__ldcg(st.job_min + (size_t)s * t.J + j);
        const double g = warp_sum_fixed(part) + warp_sum_fixed(lam_part);
        if (lane == 0) {
            st.dual_trace[(size_t)s * (a.T + 1) + round] = g;
            if (g < st.best_dual[s])
                st.best_dual[s] = g;
        }
    }
    if (st.hash_trace && lane == 0) {
        st.hash_trace[(size_t)s * a.T + round] = __ldcg(st.hash + s);
        st.hash[s] = 0ull;
    }
}

// The end of an update (lane 0): the new prices' bound, the round's time and the stopping rule.
__device__ __forceinline__ void close_round(const DevTable &t, const DevState &st, const SolveArgs &a, int s, int round,
                                            double M, bool huge, bool conv)
{
    st.ebound[s] = screen_bound(M, t.R, a.exact_only || huge);
    if (st.time_trace)
        st.time_trace[(size_t)s * a.T + round] = global_ns();
    st.rounds_run[s] = round + 1;
    if (conv) {
        st.converged[s] = 1;
        st.frozen[s] = 1;
    }
}

// Eq. price_update for scenario s of a table without a group column after round `round` (one warp, lane k
// holds price k: P = R <= 16), as update_scenario does it, with every input loaded at once and the new
// prices and bound computed from registers. The chain of dependent trips to L2 is what this costs (it
// is the serial end of every round): one here, three when the new prices went through memory
// between the update, the effective prices and the bound.
__device__ __forceinline__ void update_flat(const DevTable &t, const DevState &st, const SolveArgs &a, int s, int round,
                                            int lane)
{
    const int P = t.P, T = a.T;
    const size_t sp = (size_t)s * P;
    const bool mine = lane < P;
    long long U = 0, C = 1;
    double lam = 0.0, rcp = 1.0;
    int umax = 0;
    if (mine) {
        U = (long long)__ldcg(st.U + sp + lane);
        C = __ldg(t.cap + sp + lane);
        lam = __ldcg(st.lam + sp + lane);
        rcp = __ldcg(st.rcp + sp + lane);
        umax = __ldg(st.umax + sp + lane);   // R = P
    }
    const double vmax = __ldg(st.vmax + s);
    const double Cd = (double)C;

    trace_round(t, st, a, s, round, mine ? ((a.mode == 1) ? lam : lam * Cd) : 0.0, lane);
    if (st.dem_trace && mine)
        st.dem_trace[((size_t)s * T + round) * P + lane] = U;
    if (mine)
        st.U[sp + lane] = 0ull;

    const double nl = mine ? price_step_rcp(lam, U, C, Cd, rcp, step_size(a.eta0, a.step, round), a.mode) : 0.0;
    if (__any_sync(FULL, mine && !isfinite(nl))) {
        if (lane == 0) {
            st.status[s] = 2;
            st.frozen[s] = 1;
        }
        return;
    }
    const double p = mine ? effective_price_rcp(nl, Cd, rcp, a.mode) : 0.0;
    if (mine) {
        st.lam[sp + lane] = nl;
        st.p64[sp + lane] = p;
        st.p32[sp + lane] = __double2float_rn(p);
        if (st.lam_trace)
            st.lam_trace[((size_t)s * (T + 1) + round + 1) * P + lane] = nl;
    }
    const bool huge = __any_sync(FULL, mine && !(p <= 0x1p100));
    const double M = vmax + warp_sum_fixed(mine ? p * (double)umax : 0.0);
    bool conv = false;
    if (a.tol > 0.0) {
        const double dmax = warp_max(mine ? fabs(nl - lam) : 0.0), amax = warp_max(mine ? fabs(lam) : 0.0);
        conv = dmax <= a.tol * fmax(1.0, amax);
    }
    if (lane == 0)
        close_round(t, st, a, s, round, M, huge, conv);
}

constexpr int kKeepAtOnce = 5;

// The same for a table with a group column: P prices, new ones kept in `keep` (P doubles of the warp's shared
// memory) until all are known to be finite.
__device__ __forceinline__ void update_grouped(const DevTable &t, const DevState &st, const SolveArgs &a, int s, int round,
                                               double *keep, int lane)
{
    const int P = t.P, T = a.T, R = t.R, rg = t.r_global, own = R - rg;   // own: 1 or 2 columns per group
    const size_t sp = (size_t)s * P;
    double lc = 0.0;
    if (st.dual_trace)
        for (int k = lane; k < P; k += 32) {
            const double lam = __ldcg(st.lam + sp + k);
            lc += (a.mode == 1) ? lam : lam * (double)__ldg(t.cap + sp + k);
        }
    trace_round(t, st, a, s, round, lc, lane);
    const double eta = step_size(a.eta0, a.step, round);
    const double vmax = __ldg(st.vmax + s);
    const int umax = lane < R ? __ldg(st.umax + (size_t)s * R + lane) : 0;
    bool bad = false;
    double dmax = 0.0, amax = 0.0;
    __syncwarp();   // every lane is done with the group prices in the same memory
    // five of a lane's prices at a time, their loads together (a loop whose last turn only some lanes take
    // ran one price after the other: 10 us for 134 prices)
    for (int k0 = lane; k0 < P + lane; k0 += 32 * kKeepAtOnce) {
        long long U[kKeepAtOnce], C[kKeepAtOnce];
        double lam[kKeepAtOnce], rcp[kKeepAtOnce];
#pragma unroll
        for (int i = 0; i < kKeepAtOnce; ++i) {
            const int k = k0 + 32 * i < P ? k0 + 32 * i : 0;
            U[i] = (long long)__ldcg(st.U + sp + k);
            C[i] = __ldg(t.cap + sp + k);
            lam[i] = __ldcg(st.lam + sp + k);
            rcp[i] = __ldg(st.rcp + sp + k);
        }
#pragma unroll
        for (int i = 0; i < kKeepAtOnce; ++i) {
            const int k = k0 + 32 * i;
            const double nl = price_step_rcp(lam[i], U[i], C[i], (double)C[i], rcp[i], eta, a.mode);
            if (k >= P)
                continue;
            if (st.dem_trace)
                st.dem_trace[((size_t)s * T + round) * P + k] = U[i];
            keep[k] = nl;
            bad |= !isfinite(nl);
            dmax = fmax(dmax, fabs(nl - lam[i]));
            amax = fmax(amax, fabs(lam[i]));
        }
    }
    __syncwarp();
    bad = __any_sync(FULL, bad);
    bool huge = false;
    double flat = 0.0, pm0 = 0.0, pm1 = 0.0;   // the lane's global price, its largest price of each group column
    for (int k0 = lane; k0 < P + lane; k0 += 32 * kKeepAtOnce) {
        double nl[kKeepAtOnce], p[kKeepAtOnce];
#pragma unroll
        for (int i = 0; i < kKeepAtOnce; ++i) {
            const int k = k0 + 32 * i < P ? k0 + 32 * i : lane < P ? lane : 0;
            nl[i] = keep[k];
            p[i] = effective_price_rcp(nl[i], (double)__ldg(t.cap + sp + k), __ldg(st.rcp + sp + k), a.mode);
        }
#pragma unroll
        for (int i = 0; i < kKeepAtOnce; ++i) {
            const int k = k0 + 32 * i;
            if (k >= P)
                continue;
            st.U[sp + k] = 0ull;
            if (bad)
                continue;
            st.lam[sp + k] = nl[i];
            st.p64[sp + k] = p[i];
            st.p32[sp + k] = __double2float_rn(p[i]);
            if (st.lam_trace)
                st.lam_trace[((size_t)s * (T + 1) + round + 1) * P + k] = nl[i];
            huge |= !(p[i] <= 0x1p100);
            if (k < rg)
                flat = p[i];   // k = lane
            else if (own == 1 || ((k - rg) & 1) == 0)
                pm0 = fmax(pm0, p[i]);
            else
                pm1 = fmax(pm1, p[i]);
        }
    }
    if (bad) {
        if (lane == 0) {
            st.status[s] = 2;
            st.frozen[s] = 1;
        }
        return;
    }
    huge = __any_sync(FULL, huge);
    pm0 = warp_max(pm0);
    if (own == 2)
        pm1 = warp_max(pm1);
    const double term = (lane < rg ? flat : lane == rg ? pm0 : pm1) * (double)umax;   // umax: 0 beyond column R - 1
    const double M = vmax + warp_sum_fixed(lane < R ? term : 0.0);
    bool conv = false;
    if (a.tol > 0.0)
        conv = warp_max(dmax) <= a.tol * fmax(1.0, warp_max(amax));
    if (lane == 0)
        close_round(t, st, a, s, round, M, huge, conv);
}

// The update of scenario s after `round`, by the warp whose arrival completed it; persist: then its
// version, which releases the scenario's next round (a stopped scenario releases every later one).
template <bool G>
__device__ __forceinline__ void finish_scenario(const DevTable &t, const DevState &st, const SolveArgs &a, int s, int round,
                                             unsigned char *groups, int lane, bool persist)
{
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    if (G)
        update_grouped(t, st, a, s, round, reinterpret_cast<double *>(groups), lane);
    else
        update_flat(t, st, a, s, round, lane);
    if (lane == 0)
        st.arrive[s] = 0u;   // every tile of the round has arrived
    if (persist) {
        // every lane's writes (prices, bound, cleared demand) before the version
        __threadfence();
        __syncwarp();
        if (lane == 0) {
            const unsigned int v = st.frozen[s] ? kVerStopped : (unsigned int)(round + 1);
            asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(st.ver + s), "r"(v) : "memory");
        }
    }
}

// The end of the warp's work on its scenario for now: demand and fingerprint, then (round passes with
// fused updates) the arrival of the tiles evaluated; the arrival that completes the scenario applies
// Eq. price_update. Every lane may have issued demand atomics or written reduced costs: the warp barrier
// orders them before lane 0's release-ordered (cumulative) arrival, which publishes them.
template <int NW, bool G, bool PERSIST>
__device__ __forceinline__ void leave(const Pass &ps, Ctx<NW> &c)
{
    if (c.s < 0 || c.skip)
        return;
    add_demand<NW, G>(ps, c);
    if (ps.want_hash) {
        unsigned long long h = c.hash;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1)
            h += __shfl_xor_sync(FULL, h, d);
        if (ps.lane == 0)
            atomicAdd(ps.st.hash + c.s, h);
        c.hash = 0ull;
    }
    if (ps.kind != PASS_ROUND || !ps.pk.fused)
        return;
    __syncwarp();
    unsigned int old = 0;
    if (ps.lane == 0)
        asm volatile("atom.add.release.gpu.u32 %0, [%1], %2;"
                     : "=r"(old)
                     : "l"(ps.st.arrive + c.s), "r"((unsigned int)c.tiles)
                     : "memory");
    old = __shfl_sync(FULL, old, 0);
    if (old + (unsigned int)c.tiles == (unsigned int)__ldg(ps.pk.scen_tiles + c.s))
        finish_scenario<G>(ps.t, ps.st, ps.a, c.s, ps.round, c.groups, ps.lane, PERSIST);
}

// Prices, bound and state of scenario s (through L2: another warp of this launch may have written them).
template <int NW, bool G, bool PERSIST>
__device__ __forceinline__ void enter(const Pass &ps, Ctx<NW> &c, int s)
{
    const DevState &st = ps.st;
    const size_t sp = (size_t)s * ps.t.P;
    const PackFormat &f = ps.pk.fmt;
    c.s = s;
    c.tiles = 0;
    const int frozen = __ldcg(st.frozen + s);
    const float e = __ldcg(st.ebound + s);
    c.p64 = st.p64 + sp;
    c.have64 = !PERSIST;
    double *const prices = reinterpret_cast<double *>(c.groups - kPackPriceBytes);
    const bool mine = !PERSIST && ps.lane < (G ? ps.t.r_global : ps.t.R);
    const double p64 = mine ? __ldcg(c.p64 + ps.lane) : 0.0;
#pragma unroll
    for (int k = 0; k < (G ? NW - 1 : NW); ++k) {
        const float pl = f.col_lo[k] >= 0 ? __ldcg(st.p32 + sp + f.col_lo[k]) : 0.0f;
        const float ph = f.col_hi[k] >= 0 ? __ldcg(st.p32 + sp + f.col_hi[k]) : 0.0f;
        c.price[k] = pack2(pl, ph);
    }
    if (G) {   // the slots' prices; an update of the scenario before may have used the memory
        const int rg = ps.t.r_global, own = ps.t.R - rg;
        __syncwarp();
        for (int g = ps.lane; g < ps.t.n_groups; g += 32) {
            const float *p = st.p32 + sp + rg + own * g;
            const float a = __ldcg(p), b = own == 2 ? __ldcg(p + 1) : 0.0f;
            *reinterpret_cast<unsigned long long *>(c.groups + 8 * pack_slot((uint32_t)g)) = pack2(a, b);
        }
        __syncwarp();
    }
    c.skip = ps.kind == PASS_ROUND && frozen != 0;
    c.exact = !(e < INFINITY);
    c.e2 = c.exact ? INFINITY : 2.0f * e;
    if (mine)
        prices[ps.lane] = p64;
    __syncwarp();
}

// A step of whole jobs of 3 .. 256 options: each job has 2^code lanes, its lane sub the options
// sub << per .. (per = 3: eight, per = 2: four) as vectors ia and ib of the slot (has_a, has_b: they exist; +inf past a job's end and in the
// jobs missing from a tile's last step). The lane's job is job jl of a tile of n_job jobs from packed job job0 on. An
// unambiguous job's winner is the one option that holds the smallest score.
template <int NW, bool G, bool PLAIN>
__device__ __forceinline__ void step_jobs(const Pass &ps, Ctx<NW> &c, const uint4 *slot, int V, int ia, int ib, bool has_a,
                                          bool has_b, bool any_b, int code, int per, int job0, int jl, int n_job)
{
    float qa[4], qb[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
    float a1, a2, b1 = INFINITY, b2 = INFINITY;
    screen4<NW, G>(slot + ia, V, ps.pk.fmt, c, qa);
    two_smallest(qa, a1, a2);
    if (any_b) {
        screen4<NW, G>(slot + ib, V, ps.pk.fmt, c, qb);
        two_smallest(qb, b1, b2);
    }
    a1 = has_a ? a1 : INFINITY;
    a2 = has_a ? a2 : INFINITY;
    b1 = has_b ? b1 : INFINITY;
    b2 = has_b ? b2 : INFINITY;
    const float l1 = fminf(a1, b1);
    float m1 = l1, m2 = fminf(fmaxf(a1, b1), fminf(a2, b2));
    if (code == 5) {
        // one job on all lanes: the lane that holds the smallest offers its second smallest, the others
        // their smallest; two lanes with the same smallest make both equal
        m1 = warp_min_f32(l1);
        const uint32_t holders = __ballot_sync(FULL, l1 == m1);
        const float o = warp_min_f32(l1 == m1 ? m2 : l1);
        m2 = (holders & (holders - 1u)) ? m1 : o;
    } else {
        for (int d = 1; d < (1 << code); d <<= 1) {
            const float o1 = __shfl_xor_sync(FULL, m1, d);
            const float o2 = __shfl_xor_sync(FULL, m2, d);
            m2 = fminf(fminf(m2, o2), fmaxf(m1, o1));
            m1 = fminf(m1, o1);
        }
    }
    const float thr = __fadd_ru(m1, c.e2);
    const bool amb = c.exact ? jl < n_job : (m1 < INFINITY && !(m2 > thr));
    bool mine = !amb && m1 < INFINITY && l1 == m1;   // held by one option only: a tie would make m2 = m1
    int o = a1 == m1 ? (qa[0] == m1 ? 0 : qa[1] == m1 ? 1 : qa[2] == m1 ? 2 : 3)
                     : (qb[0] == m1 ? 4 : qb[1] == m1 ? 5 : qb[2] == m1 ? 6 : 7);
    bool have_s = false;
    long long key = 0;
    if (__any_sync(FULL, amb)) {
        const int loc = (ps.lane & ((1 << code) - 1)) << per;
        Exact x{0x7fffffffffffffffLL, kIdxNone};
        uint32_t sv = 0u;
        int64_t first = 0;
        if (amb) {
            sv = (has_a ? survivors(slot[ia], qa, c.exact, thr) : 0u) | (has_b ? survivors(slot[ib], qb, c.exact, thr) << 4 : 0u);
            first = first_option(ps, job0 + jl) + loc;
        }
        const double v = first_value(ps, first, sv);
        fetch_prices<NW, G>(ps, c);
        if (sv != 0u)
            x = rescore<NW, G>(ps, c, reinterpret_cast<const uint32_t *>(slot + ia), reinterpret_cast<const uint32_t *>(slot + ib), V,
                               first, sv, loc, v);
        x = group_min(x, 1 << code);
        if (amb && x.idx >= loc && x.idx < loc + (1 << per)) {
            mine = have_s = true;
            o = x.idx - loc;
            key = x.key;
            ++c.resolved;
        }
    }
    if (mine) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(slot + (o < 4 ? ia : ib)) + (o & 3);
        add_option<NW, G>(ps, c, w, V);
        if (!PLAIN) {
            const int local = ((ps.lane & ((1 << code) - 1)) << per) + o;
            const double v = ps.want_min ? __ldg(ps.t.values + first_option(ps, job0 + jl) + local) : 0.0;
            extras<NW, G>(ps, c, job0 + jl, local, v, w, V, have_s, key);
        }
    }
}

// Four consecutive options of a tile whose jobs have one or two: jobs job0 + j0 .., `n` of them left in
// it (none or less: the lane has no job). v: the vector. The whole warp calls it.
template <int NW, bool G, bool PLAIN>
__device__ __forceinline__ void step_tiny(const Pass &ps, Ctx<NW> &c, const uint4 *v, int V, int K, int job0, int j0, int n)
{
    const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
    float q[4], thr[2] = {INFINITY, INFINITY};
    uint32_t amb = 0u, win = 0u;   // per pair of options: ambiguous; the second one wins
    if (K == 2) {
        screen4<NW, G>(v, V, ps.pk.fmt, c, q);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float qa = q[2 * p], qb = q[2 * p + 1];
            thr[p] = __fadd_ru(fminf(qa, qb), c.e2);
            win |= qb < qa ? 1u << p : 0u;
            amb |= p < n && (c.exact || !(fmaxf(qa, qb) > thr[p])) ? 1u << p : 0u;
        }
        if (__any_sync(FULL, amb != 0u))
            fetch_prices<NW, G>(ps, c);
    }
    // the jobs' values on their way together (one after the other, a trip to memory each, made the final pass of a
    // table with many such jobs several times as long as a round)
    int64_t first[4] = {0, 0, 0, 0};
    double val[4] = {0.0, 0.0, 0.0, 0.0};
    if (!PLAIN && ps.want_min) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < n && j * K < 4)
                first[j] = first_option(ps, job0 + j0 + j);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < n && j * K < 4 && !((amb >> j) & 1u))
                val[j] = __ldg(ps.t.values + first[j] + ((win >> j) & 1u));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j >= n || j * K >= 4)
            continue;
        int o = j * K + (int)((win >> j) & 1u);
        bool have_s = false;
        long long key = 0;
        if (j < 2 && ((amb >> j) & 1u)) {
            const uint32_t sv = (survivors(v[0], q, c.exact, thr[j]) >> (2 * j)) & 3u;
            const int64_t f = first_option(ps, job0 + j0 + j);
            const Exact x = rescore<NW, G>(ps, c, w + 2 * j, w, V, f, sv, 2 * j, first_value(ps, f, sv));
            o = x.idx;
            key = x.key;
            have_s = true;
            ++c.resolved;
            if (!PLAIN && ps.want_min)
                val[j] = __ldg(ps.t.values + first[j] + o - 2 * j);
        }
        add_option<NW, G>(ps, c, w + o, V);
        if (!PLAIN)
            extras<NW, G>(ps, c, job0 + j0 + j, o - j * K, val[j], w + o, V, have_s, key);
    }
}

// A job of more than 256 options, step by step: each lane keeps the best of its own options; the job's
// last step reduces across the warp, and the winner's words, read again from the packed copy, are added
// when the next job closes (or the tile ends), so that no job waits for them.
template <int NW>
struct Large {
    float m1, m2;
    int idx;
    uint32_t x[NW];   // words of the previous job's winner, zero on the other lanes
    uint32_t slot;    // the one of them that holds its group slot
};

template <int NW, bool G>
__device__ __forceinline__ void add_pending(const Pass &ps, Ctx<NW> &c, Large<NW> &b)
{
    const PackFormat &f = ps.pk.fmt;
    if (G && b.x[NW - 1] != 0u) {
        add_group(ps, c, b.x[NW - 1], b.slot);
        b.x[NW - 1] = 0u;
    }
#pragma unroll
    for (int k = 0; k < (G ? NW - 1 : NW); ++k) {
        c.lo[k] += b.x[k] & f.mask[k];
        c.hi[k] += b.x[k] >> f.shift[k];
        b.x[k] = 0u;
    }
}

// The packed vector (plane 0) that holds vector `vec` of a large job whose data start at `base`.
template <int NW>
__device__ __forceinline__ const uint4 *large_vec(const uint4 *base, const PackShape &sh, int vec)
{
    const int step = vec / sh.v, x = vec - step * sh.v;
    return base + (int64_t)step * sh.v * (NW + 1) + ((x & 1) ? sh.ca + (x >> 1) : x >> 1);
}

// Survivors of a large job in fp64 when a lane may hold several: its packed vectors are screened again (the
// same instructions give the same q).
template <int NW, bool G>
__device__ __forceinline__ Exact rescan_large(const Pass &ps, const Ctx<NW> &c, const uint4 *base, const PackShape &sh,
                                              int64_t opt0, float thr)
{
    Exact x{0x7fffffffffffffffLL, kIdxNone};
    for (int g = ps.lane; g < sh.m; g += 32) {
        const uint4 *v = large_vec<NW>(base, sh, g);
        float q[4];
        screen4<NW, G>(v, sh.v, ps.pk.fmt, c, q);
        const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
        const uint32_t sv = survivors(v[0], q, c.exact, thr);
        const Exact y = rescore<NW, G>(ps, c, w, w, sh.v, opt0 + 4 * g, sv, 4 * g, first_value(ps, opt0 + 4 * g, sv));
        if (y.key < x.key)
            x = y;
    }
    return x;
}

// The same of one lane's options, its vectors spread over the warp: one trip to memory, where rescan_large makes
// one per step of the job.
template <int NW, bool G>
__device__ __forceinline__ void rescan_lane(const Pass &ps, const Ctx<NW> &c, const uint4 *base, const PackShape &sh,
                                            int64_t opt0, float thr, int of, Exact &x)
{
    for (int i = ps.lane; i < 2 * sh.nch; i += 32) {
        const int step = i >> 1, at = 2 * of + (i & 1), g = step * sh.v + at;
        if (at >= sh.v || g >= sh.m)
            continue;
        const uint4 *v = large_vec<NW>(base, sh, g);
        float q[4];
        screen4<NW, G>(v, sh.v, ps.pk.fmt, c, q);
        const uint32_t *w = reinterpret_cast<const uint32_t *>(v);
        const uint32_t sv = survivors(v[0], q, c.exact, thr);
        const Exact y = rescore<NW, G>(ps, c, w, w, sh.v, opt0 + 4 * g, sv, 4 * g, first_value(ps, opt0 + 4 * g, sv));
        if (y.key < x.key || (y.key == x.key && y.idx < x.idx))
            x = y;
    }
}

template <int NW, bool G, bool PLAIN>
__device__ __forceinline__ void close_large(const Pass &ps, Ctx<NW> &c, const uint4 *base, const PackShape &sh, int job0,
                                            int jl, Large<NW> &b)
{
    add_pending<NW, G>(ps, c, b);
    const float m1 = warp_min_f32(b.m1);
    const bool first = b.m1 == m1;
    const uint32_t holders = __ballot_sync(FULL, first);
    const float o2 = warp_min_f32(first ? b.m2 : b.m1);
    const float m2 = (holders & (holders - 1u)) ? m1 : o2;
    const float thr = __fadd_ru(m1, c.e2);
    bool mine = first, have_s = false;
    int win = b.idx;
    long long key = 0;
    // words of option o of the job
    auto words = [&](int o) { return reinterpret_cast<const uint32_t *>(large_vec<NW>(base, sh, o >> 2)) + (o & 3); };
    if (c.exact || !(m2 > thr)) {
        const int64_t opt0 = first_option(ps, job0 + jl);
        Exact x{0x7fffffffffffffffLL, kIdxNone};
        const double own_value = first_value(ps, opt0 + b.idx, b.m1 <= thr && !c.exact ? 1u : 0u);
        auto own_best = [&]() {
            const uint32_t *w = words(b.idx);
            x = rescore<NW, G>(ps, c, w, w, sh.v, opt0 + b.idx, 1u, b.idx, own_value);
        };
        fetch_prices<NW, G>(ps, c);
        if (!c.exact && !__any_sync(FULL, b.m2 <= thr)) {   // every lane's own best at most
            if (b.m1 <= thr)
                own_best();
        } else {
            const uint32_t several = __ballot_sync(FULL, b.m2 <= thr);   // lanes with more than their own best
            if (!c.exact && __popc(several) <= sh.nch) {
                if (b.m1 <= thr && !(b.m2 <= thr))
                    own_best();
                for (uint32_t l = several; l != 0u; l &= l - 1u)
                    rescan_lane<NW, G>(ps, c, base, sh, opt0, thr, __ffs((int)l) - 1, x);
            } else {
                x = rescan_large<NW, G>(ps, c, base, sh, opt0, thr);
            }
        }
        const int own = x.idx;
        x = group_min(x, 32);
        win = x.idx;
        key = x.key;
        have_s = true;
        mine = own == win;
        if (mine)
            ++c.resolved;
    }
    if (mine) {
        const uint32_t *w = words(win);
#pragma unroll
        for (int i = 0; i < NW; ++i)
            b.x[i] = __ldg(w + (i + 1) * sh.v * 4);
        if (G)
            b.slot = __ldg(w + (ps.pk.fmt.g_word + 1) * sh.v * 4);
        if (!PLAIN) {
            const double v = ps.want_min ? __ldg(ps.t.values + first_option(ps, job0 + jl) + win) : 0.0;
            extras<NW, G>(ps, c, job0 + jl, win, v, w, sh.v, have_s, key);
        }
    }
    b.m1 = b.m2 = INFINITY;
    b.idx = kIdxNone;
}

template <int NW>
__device__ __forceinline__ void reset(Ctx<NW> &c)
{
    c.s = -1;
    c.skip = false;
    c.tiles = 0;
    c.wins = 0;
    c.hash = 0ull;
    c.resolved = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k)
        c.lo[k] = c.hi[k] = 0u;
}

// One warp's work: the tiles `next` hands out (its index, its round in *round; -1 when there are no
// more), evaluated in order. Lane 0 copies the step after the one in flight as soon as its slot is free,
// across tiles; a tile's record is loaded while the tile before it is evaluated. hold_tx: see SolveArgs.
template <int NW, bool G, bool PLAIN, bool PERSIST, typename Next>
__device__ __forceinline__ void run_warp(const DevTable &t, const DevState &st, const DevPack &pk, const SolveArgs &a,
                                         int round, int kind, unsigned char *smem, uint32_t hold_tx, Next &&next)
{
    const int lane = threadIdx.x & 31;
    Pass ps{t, st, pk, a, round, PLAIN ? (int)PASS_ROUND : kind, lane,
            PLAIN ? false : (kind == PASS_FINAL || st.dual_trace != nullptr),
            PLAIN ? false : (kind == PASS_ROUND && st.hash_trace != nullptr)};
    constexpr int kSlot = pack_slot_bytes(NW);
    const uint32_t slots_s = smem_u32(smem), bars = slots_s + kPackSlots * kSlot;
    int rt = 0, rn = 0;
    int kt = next(&rt);          // the tile being evaluated, its round, and the next tile
    if (kt < 0)
        return;
    int kn = next(&rn);
    auto load = [&](int k) {
        const uint4 x = __ldg(reinterpret_cast<const uint4 *>(pk.tiles + k));
        return PackTile{x.x, x.y, x.z, x.w};
    };
    PackTile T = load(kt), N = T;
    int job0 = __ldg(pk.job_begin + kt), jobn = 0;   // their first jobs
    if (kn >= 0) {
        N = load(kn);
        jobn = __ldg(pk.job_begin + kn);
    }
    if (lane == 0) {
        for (int s = 0; s < kPackSlots; ++s)
            mbar_init(bars + 8 * s, 1);
        fence_barrier_init();
    }
    __syncwarp();
    // the copies: source of the next step, its bytes, steps left in its tile; steps in flight
    const unsigned char *src;
    uint32_t bytes;
    int left, flying = 0, to = 0;
    bool in_next = false;
    auto start = [&](const PackTile &x) {
        const PackShape sh = pack_shape(x);
        src = reinterpret_cast<const unsigned char *>(pk.data) + (uint64_t)x.base * (16 * (NW + 1));
        bytes = (uint32_t)sh.v * (16 * (NW + 1));
        left = sh.steps;
    };
    auto issue = [&]() {
        if (left == 0) {
            if (in_next || kn < 0)
                return;
            start(N);
            in_next = true;
        }
        if (lane == 0) {
            fence_proxy_async();
            mbar_arrive_expect_tx(bars + 8 * to, bytes + hold_tx);
            bulk_g2s(slots_s + to * kSlot, src, bytes, bars + 8 * to);
        }
        hold_tx = 0u;
        src += bytes;
        --left;
        ++flying;
        to ^= 1;
    };
    start(T);
    issue();
    issue();
    // everything above reads only the packed table and the plan; prices, flags and the demand
    // accumulators were written by the previous kernel on the stream (a no-op for an ordinary launch)
    if (!PERSIST)
        asm volatile("griddepcontrol.wait;" ::: "memory");
    Ctx<NW> c;
    reset(c);
    c.have64 = !PERSIST;
    c.groups = smem + pack_warp_bytes(NW);
    int at = 0;                  // slot of the step to be screened
    uint32_t phases = 0;         // parity of each slot's next completion
    // the step in slot `at` has landed (bounded; warp-uniform)
    auto landed = [&]() {
        const bool ok = __all_sync(FULL, wait_stage(bars + 8 * at, (phases >> at) & 1u, st.err, a.wait_ms));
        if (ok) {
            phases ^= 1u << at;
            --flying;
        }
        return ok;
    };
    auto release = [&]() {       // every lane is done with slot `at`
        __syncwarp();
        at ^= 1;
        issue();
    };
    // an earlier launch's wait gave up: this warp does nothing (looked at after the first loads of prices)
    const unsigned int gave_up = __ldcg(st.err);
    bool ok = true;
    while (ok) {
        if (flying < kPackSlots)
            issue();             // a tile of one step left the copies waiting for this tile's successor
        const PackShape sh = pack_shape(T);
        if (PERSIST) {
            leave<NW, G, true>(ps, c);
            c.s = -1;
            if (!wait_version(st.ver, (int)T.scenario, rt, st.err, a.wait_ms, st.stats)) {
                ok = false;
                break;
            }
            ps.round = rt;
            enter<NW, G, true>(ps, c, (int)T.scenario);
        } else if ((int)T.scenario != c.s) {
            leave<NW, G, false>(ps, c);
            enter<NW, G, false>(ps, c, (int)T.scenario);
        }
        if (__any_sync(FULL, (gave_up & DEV_ERR_TIMEOUT) != 0u)) {
            ok = false;
            break;
        }
        if (c.wins >= kPackSpill)
            add_demand<NW, G>(ps, c);
        const int n_job = (int)T.n_job, steps = sh.steps;
        if (sh.code < (int)kPackTiny) {
            const int code = sh.code, sub = lane & ((1 << code) - 1), jl = lane >> code;
            const bool has_a = sub < sh.ca, has_b = sub < sh.cb, any_b = sh.cb > 0;
            const int ia = has_a ? jl * sh.ca + sub : 0, ib = has_b ? sh.per_step * sh.ca + jl * sh.cb + sub : 0;
            for (int st_i = 0; st_i < steps; ++st_i) {
                if (!(ok = landed()))
                    break;
                if (!c.skip)
                    step_jobs<NW, G, PLAIN>(ps, c, reinterpret_cast<const uint4 *>(smem + at * kSlot), sh.v, ia, ib, has_a, has_b,
                                         any_b, code, sh.narrow ? 2 : 3, job0, st_i * sh.per_step + jl, n_job);
                release();
            }
            c.wins += steps;
        } else if (sh.code == (int)kPackLarge) {
            Large<NW> big;
            big.m1 = big.m2 = INFINITY;
            big.idx = kIdxNone;
#pragma unroll
            for (int k = 0; k < NW; ++k)
                big.x[k] = 0u;
            int job = 0, ch = 0;
            for (int st_i = 0; st_i < steps; ++st_i) {
                if (!(ok = landed()))
                    break;
                if (!c.skip) {
                    const uint4 *slot = reinterpret_cast<const uint4 *>(smem + at * kSlot);
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        if (lane >= (h ? sh.cb : sh.ca))
                            break;
                        float q[4], r1, r2;
                        screen4<NW, G>(slot + (h ? sh.ca : 0) + lane, sh.v, pk.fmt, c, q);
                        two_smallest(q, r1, r2);
                        if (r1 < big.m1) {   // increasing index: earlier options keep ties
                            big.m2 = fminf(big.m1, r2);
                            big.idx = 4 * (ch * sh.v + 2 * lane + h) + (q[0] == r1 ? 0 : q[1] == r1 ? 1 : q[2] == r1 ? 2 : 3);
                            big.m1 = r1;
                        } else {
                            big.m2 = fminf(big.m2, r1);
                        }
                    }
                    __syncwarp();
                    if (++ch == sh.nch) {
                        close_large<NW, G, PLAIN>(ps, c,
                                               pk.data + ((uint64_t)T.base + (uint64_t)job * sh.nch * sh.v) * (NW + 1), sh, job0,
                                               job, big);
                        ch = 0;
                        ++job;
                    }
                }
                release();
            }
            add_pending<NW, G>(ps, c, big);
            c.wins += n_job;
        } else {
            for (int st_i = 0; st_i < steps; ++st_i) {
                if (!(ok = landed()))
                    break;
                if (!c.skip) {
                    const uint4 *slot = reinterpret_cast<const uint4 *>(smem + at * kSlot);
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        const int o0 = 4 * (64 * st_i + 32 * h + lane), j0 = o0 / sh.m;   // m = 1 or 2
                        step_tiny<NW, G, PLAIN>(ps, c, slot + 32 * h + lane, 64, sh.m, job0, j0, n_job - j0);
                    }
                }
                release();
            }
            c.wins += 8 * steps;
        }
        if (!ok)
            break;
        ++c.tiles;
        if (kn < 0) {
            leave<NW, G, PERSIST>(ps, c);
            break;
        }
        T = N;
        job0 = jobn;
        rt = rn;
        in_next = false;
        kn = next(&rn);
        if (kn >= 0) {
            N = load(kn);
            jobn = __ldg(pk.job_begin + kn);
        }
    }
    if (!ok) {   // a wait gave up: wait (bounded) for every copy still in flight, then leave
        for (; flying > 0; --flying, at ^= 1) {
            wait_stage(bars + 8 * at, (phases >> at) & 1u, st.err, a.wait_ms);
            phases ^= 1u << at;
        }
    }
    const unsigned int n = __reduce_add_sync(FULL, c.resolved);
    if (lane == 0 && n != 0u)
        atomicAdd(st.stats, (unsigned long long)n);
}

// One pass: warp w evaluates the tiles of its range. PLAIN: a round pass without traces. G: a table with a
// group column.
template <int NW, bool G, bool PLAIN>
__global__ void __launch_bounds__(kPackWarps * 32, pack_min_ctas(NW, G))
    k_packed(const __grid_constant__ DevTable t, const __grid_constant__ DevState st, const __grid_constant__ DevPack pk,
             const __grid_constant__ SolveArgs a, int round, int kind)
{
    extern __shared__ __align__(128) unsigned char smem[];
    // a pass launched as a programmatic dependent of this one may start its CTAs as slots free up; it
    // waits for this grid's completion before it reads state
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int wid = threadIdx.x >> 5, w = blockIdx.x * kPackWarps + wid;
    if (w >= pk.n_warps)
        return;
    int k = w, end = w + 1;
    if (pk.n_warps != pk.n_tiles) {
        const int32_t *begin = !PLAIN && kind == PASS_FINAL ? pk.final_begin : pk.warp_begin;
        k = __ldg(begin + w);
        end = __ldg(begin + w + 1);
    }
    run_warp<NW, G, PLAIN, false>(t, st, pk, a, round, kind,
                               smem + (size_t)wid * (pack_warp_bytes(NW) + (G ? pk.fmt.g_bytes : 0)),
                               (w == 0 && round == 0 && kind == PASS_ROUND) ? a.hold_tx : 0u,
                               [&](int *) { return k < end ? k++ : -1; });
}

// Rounds 0 .. n_rounds - 1 in one cooperative launch. Between two round passes a kernel boundary costs
// the whole GPU the slowest warp's tail, the next pass's ramp-up and the launch gap. Here the only
// dependence left is the true one: scenario s may be evaluated in round r once its r-th price update is
// done, published as ver[s] >= r by the warp whose arrival completed the round before.
// Work items are (round, tile) pairs, q = round * n_tiles + i, taken from one counter in increasing
// order by whichever warp is free; the tiles are listed by scenario, so a scenario's next-round items are
// handed out about a round after its current ones.
// Lane 0 asks the counter one item ahead of the one it hands out.
// Deadlock-free: every CTA is co-resident (cooperative launch); an item depends only on items of smaller
// index, a warp evaluates its items in the order it took them and publishes one before it waits for the
// next one's scenario, so the smallest unfinished item waits only for published work. Every wait is
// bounded.
template <int NW>
__global__ void __launch_bounds__(kPackWarps * 32, pack_min_ctas(NW))
    k_packed_persist(const __grid_constant__ DevTable t, const __grid_constant__ DevState st,
                     const __grid_constant__ DevPack pk, const __grid_constant__ SolveArgs a, int n_rounds)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned int Q = (unsigned int)n_rounds * (unsigned int)pk.n_tiles;   // below 2^31 (host)
    unsigned int pend = 0;
    if (lane == 0)
        pend = atomicAdd(st.work, 1u);
    run_warp<NW, false, true, true>(t, st, pk, a, 0, (int)PASS_ROUND, smem + (size_t)wid * pack_warp_bytes(NW),
                             blockIdx.x == 0 && wid == 0 ? a.hold_tx : 0u,
                             [&](int *round) {
                                 const unsigned int q = __shfl_sync(FULL, pend, 0);
                                 if (q >= Q)
                                     return -1;
                                 if (lane == 0)
                                     pend = atomicAdd(st.work, 1u);
                                 const unsigned int r = q / (unsigned int)pk.n_tiles;
                                 *round = (int)r;
                                 return (int)(q - r * (unsigned int)pk.n_tiles);
                             });
}

// The words of the packed copy (esp_packed.h): one block per step, one thread per option.
__global__ void __launch_bounds__(4 * kPackStepVecs) k_pack(DevTable t, const __grid_constant__ DevPack pk, uint32_t *data)
{
    const int R = t.R, words = pk.fmt.nw + 1;
    const PackTile T = pk.tiles[blockIdx.x];
    const PackShape sh = pack_shape(T);
    const int w = threadIdx.x;
    if (w >= 4 * sh.v)
        return;
    const int j0 = pk.job_begin[blockIdx.x], n_job = (int)T.n_job;
    // the job of word w of a plane and the option of it
    const int x = w >> 2, o = w & 3;
    for (int step = blockIdx.y; step < sh.steps; step += gridDim.y) {
        int jl, opt;
        if (sh.code == (int)kPackTiny) {
            const int at = 4 * (64 * step + x) + o;
            jl = at / sh.m;
            opt = at - jl * sh.m;
        } else if (sh.code == (int)kPackLarge) {
            jl = step / sh.nch;
            const int vec = x < sh.ca ? 2 * x : 2 * (x - sh.ca) + 1;
            opt = 4 * ((step - jl * sh.nch) * sh.v + vec) + o;
        } else {
            const int na = sh.per_step * sh.ca;
            const bool first = x < na;
            const int y = first ? x : x - na, per = first ? sh.ca : sh.cb;
            const int q = y / per, sub = y - q * per;
            jl = step * sh.per_step + q;
            opt = 4 * (sh.narrow ? sub : 2 * sub + (first ? 0 : 1)) + o;
        }
        uint32_t v = kPackInf, f[kPackMaxWords];
#pragma unroll
        for (int k = 0; k < kPackMaxWords; ++k)
            f[k] = 0u;
        if (jl < n_job) {
            const int64_t job = pk.job ? pk.job[j0 + jl] : j0 + jl;
            const int64_t a = t.job_off[job];
            if (opt == 0 && pk.opt0)
                pk.opt0[j0 + jl] = a;
            if (opt < t.job_off[job + 1] - a) {
                const int32_t *u = t.units + (a + opt) * R;
                if (u[0] >= 0) {   // not a duplicate
                    v = __float_as_uint(-screen_value(t.values[a + opt]));
                    if (v == kPackInf)   // beyond the screen's range (evaluated exactly): not padding
                        v = 0x7f7fffffu;
                }
#pragma unroll
                for (int k = 0; k < kPackMaxWords; ++k) {
                    if (k < pk.fmt.nw && pk.fmt.col_lo[k] >= 0)
                        f[k] = (uint32_t)(u[pk.fmt.col_lo[k]] & 0x7fffffff);
                    if (k < pk.fmt.nw && pk.fmt.col_hi[k] >= 0)
                        f[k] |= (uint32_t)(u[pk.fmt.col_hi[k]] & 0x7fffffff) << pk.fmt.shift[k];
                    if (pk.fmt.g_mask != 0u && k == pk.fmt.g_word)
                        f[k] |= pack_slot(t.group[a + opt]) << pk.fmt.g_shift;
                }
            }
        }
        uint32_t *out = data + ((uint64_t)T.base + (uint64_t)step * sh.v) * words * 4;
        out[w] = v;
#pragma unroll
        for (int k = 0; k < kPackMaxWords; ++k)
            if (k < pk.fmt.nw)
                out[(k + 1) * sh.v * 4 + w] = f[k];
    }
}

template <int NW, bool G>
struct PackKernels {
    static constexpr int kKernels = G ? 2 : 3;
    static const void *fn(int which)
    {
        if constexpr (!G)
            if (which == 2)
                return reinterpret_cast<const void *>(&k_packed_persist<NW>);
        return which == 0 ? reinterpret_cast<const void *>(&k_packed<NW, G, true>)
                          : reinterpret_cast<const void *>(&k_packed<NW, G, false>);
    }
};

template <typename F>
auto pack_dispatch(int nw, bool grouped, F &&f)
{
    if (grouped)
        switch (nw) {
        case 3: return f(PackKernels<3, true>());
        case 4: return f(PackKernels<4, true>());
        default: return f(PackKernels<6, true>());
        }
    switch (nw) {
    case 2: return f(PackKernels<2, false>());
    case 3: return f(PackKernels<3, false>());
    case 4: return f(PackKernels<4, false>());
    case 6: return f(PackKernels<6, false>());
    default: return f(PackKernels<8, false>());
    }
}

int pack_smem(int nw, int group_bytes)
{
    return kPackWarps * (pack_warp_bytes(nw) + group_bytes);
}

}  // namespace

int packed_ctas_per_sm(int nw, int group_bytes)
{
    return pack_dispatch(nw, group_bytes > 0, [&](auto k) -> int {
        int best = 0;
        // the limit is the kernel's, not the table's: the largest price table's for every one
        const int smem = pack_smem(nw, group_bytes);
        const int limit = pack_smem(nw, group_bytes > 0 ? pack_group_bytes(kPackMaxPrices, kPackMaxPrices) : 0);
        for (int i = 0; i < decltype(k)::kKernels; ++i) {
            int n = 0;
            if (cudaFuncSetAttribute(decltype(k)::fn(i), cudaFuncAttributeMaxDynamicSharedMemorySize, limit) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, decltype(k)::fn(i), kPackWarps * 32, smem) !=
                    cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
            best = i == 0 ? n : std::min(best, n);
        }
        return best;
    });
}

cudaError_t launch_pack(const DevTable &t, const DevPack &pk, uint4 *data, cudaStream_t stream)
{
    if (pk.n_tiles <= 0)
        return cudaSuccess;
    k_pack<<<dim3((unsigned)pk.n_tiles, 8), 4 * kPackStepVecs, 0, stream>>>(t, pk, reinterpret_cast<uint32_t *>(data));
    return cudaGetLastError();
}

cudaError_t launch_packed(const DevTable &t, const DevState &st, const DevPack &pk, const SolveArgs &a, int round,
                          PassKind kind, cudaStream_t stream, bool pdl)
{
    const bool plain = kind == PASS_ROUND && st.hash_trace == nullptr && st.dual_trace == nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((pk.n_warps + kPackWarps - 1) / kPackWarps));
    cfg.blockDim = dim3(kPackWarps * 32);
    const int group_bytes = t.group ? pk.fmt.g_bytes : 0;
    cfg.dynamicSmemBytes = (size_t)pack_smem(pk.fmt.nw, group_bytes);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    int k = kind;
    void *args[] = {(void *)&t, (void *)&st, (void *)&pk, (void *)&a, (void *)&round, (void *)&k};
    return pack_dispatch(pk.fmt.nw, group_bytes > 0,
                         [&](auto kk) { return cudaLaunchKernelExC(&cfg, decltype(kk)::fn(plain ? 0 : 1), args); });
}

cudaError_t launch_packed_persist(const DevTable &t, const DevState &st, const DevPack &pk, const SolveArgs &a,
                                  int n_rounds, int grid, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kPackWarps * 32);
    cfg.dynamicSmemBytes = (size_t)pack_smem(pk.fmt.nw, 0);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // every CTA co-resident: the version waits can end
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&t, (void *)&st, (void *)&pk, (void *)&a, (void *)&n_rounds};
    return pack_dispatch(pk.fmt.nw, false, [&](auto kk) { return cudaLaunchKernelExC(&cfg, decltype(kk)::fn(2), args); });
}

}  // namespace esp
