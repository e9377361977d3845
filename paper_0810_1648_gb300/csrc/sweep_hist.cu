// Pair sweep of PATH_HIST instances (common.cuh): Algorithm 2's round without
// stored messages.
//
// With H_ij(t+1) = -q (htilde_i - H_ji) / d_i and P_ij(t+1) = -q^2 / d_i (all of
// round t; d_i = Ptilde_i - P_ji), putting the same expression one round
// earlier in for H_ji gives exactly
//   H_ij(t+1) = -q mu_i(t) + P_ij(t+1) mu_j(t-1) + E_ij(t+1),
//   E_ij(t+1) = (q / d_i(t)) [(q^2 / d_j(t-1)) D_i(t) + E_ji(t)],
// D_x(t) = mu_x(t) - mu_x(t-2) (aggregates before round 0, and before a restart
// of H, are 0).  Summed over i, the first term is the sum that the residual
// needs anyway and the second is mu_j(t-1) times the sum of the P messages; E is
// of the order of z = q^2 / (d_i d_j) times what still changes.  What is left
// are sums over i of powers of q with weights of node i, times values of node
// j (r = 1 / Ptilde):
//   sum q mu_i                     residual and H
//   sum q^2k r_i^k = S2k, k = 1, 2, 3   sum P_ij = -(S2 - r S4 + 2 r^2 S6), and E's
//                                  even orders, r S4 D_j(t-1) + r^2 S6 (D_j(t-3) - 3 D_j(t-1))
//   sum q^3 r_i D_i                E, times r
//   sum q^5 r_i^2 (D_i(t-2) - 2 D_i)   E, times r^2
// with r = r_j(t-1); the terms of higher orders are below FP32 rounding on this
// path (choose_path).  Before round 0 there is no message: E(1) = 0 and P_ji(0) = 0,
// the factor of D_i(0) (which so counts as 0), and what P_ji(t) of later rounds
// adds to the expansions is missing from the first ones: round 1 has S2 - r S4 + r^2
// S6 and -D_i in place of -2 D_i, round 2 has -2 D_j(t-1) in place of -3.  Once no Ptilde changes, the P sums are known (Ptilde -
// Q_jj; S4 and S6 of the last live round), and E needs its sums only while it counts
// (e_terms): most rounds are one symmetric product Q mu.  Under the staged
// schedule mu in H is the mean of the stage and the P sums are the tile's own.
//
// Bound: Q streamed once a round (4 or 2 B a pair), or the Q epilogue of the
// recomputing kernel.  Measured, a frozen round's sweep: n = 20000, FP32 Q 823
// us with stored messages (28 B a pair), 123 us here (118 us for 4 B a pair at the
// copy bandwidth); n = 100000, BF16 Q and messages 10.6 ms and 1.60 ms (1.47).
#include "common.cuh"
#include "hist.cuh"
#include "ptx.cuh"
#include "qtile_epi.cuh"

#include <float.h>

namespace gabp {

namespace {

constexpr int HCW = 8;                         // consumer warps
constexpr int H_THREADS = (HCW + 1) * 32;      // and one producer warp
constexpr size_t H_CHUNK = 16384;              // ring stage: 32 rows of FP32 Q, 64 of BF16 Q
constexpr int H_STAGES = 4;
constexpr int H_GROUP = 64;                    // rows per row-sum reduction (four steps of 16)

// What a tile sums beside q mu.  Live P: q^2 (round 0, and where nothing else
// counts), with q^3, with q^3 and q^4, or everything; frozen P: nothing, q^3, or
// q^3 and q^5.
enum { K_LIVE0, K_LIVE1, K_LIVE4, K_LIVE, K_SUM, K_ONE, K_TWO };
// The sums of a wide tile, as rows of HTail::rs and cs; a small tile (sum_tile)
// has three at most, of q mu, mu of the stage, q^2 and q^3 in this order, and
// takes rows 0-2 and 3-5 in turn.
enum { S_R, S_M, S_2, S_4, S_6, S_W3, S_W5, S_COUNT };
constexpr int S_SMALL = 3;
__device__ __forceinline__ bool is_wide(int kind, bool staged)
{
    return kind == K_LIVE4 || kind == K_LIVE || kind == K_TWO || (kind == K_LIVE1 && staged);
}
// The node values, as rows of HTail::node: mean of the residual, the stage's
// mean (staged), and hnow's three.
enum { N_MU0, N_MU, N_R, N_W3, N_W5, N_COUNT };

struct HInfo {
    const float* ring;     // the stage's history
    float* part;
    float* s46;            // slots of S4, then of S6
    long long plen;
    Ctrl* ctrl;
    long long L;
    int npad, I, J, sR, sC, rows;   // (npad: n in the final pass)
    int t, kind, even, staged, end;
    float C;               // final pass: the box, and whether there is none (task)
    int task;
};

struct HTail {
    unsigned long long full[H_STAGES], empty[H_STAGES];
    unsigned long long tfull[2], tempty[2];
    int cabort, go;
    HInfo info[2];
    alignas(16) float node[2][2][N_COUNT][T];   // [slot][row, column block]
    alignas(16) float cs[S_COUNT][HCW][T];      // column sums of each warp
    float rs[S_COUNT][T];                       // row sums
};

__device__ __forceinline__ void hbar() { asm volatile("bar.sync 1, %0;" ::"n"(HCW * 32) : "memory"); }

template <typename QT>
__host__ __device__ constexpr int q_rows() { return (int)(H_CHUNK / (T * sizeof(QT))); }
template <>
__host__ __device__ constexpr int q_rows<void>() { return T; }

// Producer (one warp): publishes each tile's parameters with the values of its
// row and column nodes and, where Q is stored, streams its rows (whole:
// entries outside the pair set are stored as 0) in 16 KB copies, ahead across
// tiles.  QT = void: Q is recomputed elsewhere.  FINAL: for the final pass, the
// FP32 entries and the means ops[k].mu of every listed tile, whatever the
// instance's state.
template <typename QT, bool FINAL = false>
__device__ __forceinline__ void hist_producer(const Inst* __restrict__ tab, const int4* __restrict__ work,
                                              long long ntiles, HTail& sm, unsigned char* ring, volatile int* abort_flag,
                                              int lane, int st, const StopOp* __restrict__ ops, const Ctrl* ctrls, bool one,
                                              CtrlHead head)
{
    constexpr bool STREAM = q_rows<QT>() < T;
    const uint64_t pol = l2_evict_first_policy(), pol_keep = l2_evict_last_policy();
    int stage = 0, slot = 0;
    uint32_t phase = 0, tph = 0;
    auto stopped = [&]() { return abort_flag && __shfl_sync(0xffffffffu, *abort_flag, 0) != 0; };
    bool ok = true;
    auto give_up = [&](Ctrl* ctrl, long long L) {
        if (lane == 0) {
            record_error(ctrl, ST_ETIMEOUT, L);
            if (abort_flag) *abort_flag = 1;
        }
        ok = false;
    };
    // The round's settings of an instance do not change during a sweep: they
    // are read once per run of tiles of the same instance, and the next tile's
    // list entry ahead of its turn, so that no chain of loads stands between
    // the copies of two tiles.
    int inst = -1, t = 0, kind = 0, even = 0;
    bool done = true, staged = false;
    uint32_t use = 0;
    int4 wn = blockIdx.x < ntiles ? work[blockIdx.x] : make_int4(0, 0, 0, 0);
    for (long long L = blockIdx.x; L < ntiles && ok; L += gridDim.x) {
        const int4 w = wn;
        if (L + gridDim.x < ntiles) wn = work[L + gridDim.x];
        const Inst& p = tab[w.x];
        Ctrl* ctrl = p.ctrl;
        if (FINAL) {
            done = false;
            use = 1u << N_MU0;
        } else if (w.x != inst) {
            inst = w.x;
            if (!one) head = ctrl_head(ctrls + inst);
            done = head.done != 0;
            t = head.t;
            const int frozen = head.p_frozen, terms = head.terms;
            even = head.even;
            staged = p.nstages > 1;
            kind = frozen && t > 0                    ? (terms == 0 ? K_SUM : terms == 1 ? K_ONE : K_TWO)
                   : t == 0 || (!even && terms == 0)  ? K_LIVE0
                   : !even && terms == 1              ? K_LIVE1
                   : even <= 1 && terms <= 1          ? K_LIVE4
                                                      : K_LIVE;
            // node values of its tiles: bit a set where row a is copied
            use = 1u << N_MU0 | (staged ? 1u << N_MU : 0u) | (kind <= K_LIVE ? 1u << N_R : 0u) |
                  (kind == K_LIVE0 || kind == K_SUM ? 0u : 1u << N_W3) | (kind == K_LIVE || kind == K_TWO ? 1u << N_W5 : 0u);
        }
        if (done) continue;      // instance finished: tile skipped
        const int I = w.y, J = w.z, rows = min(T, p.n - I * T);
        if (stopped() || !mbar_wait_warp(&sm.tempty[slot], tph ^ 1u)) {
            give_up(ctrl, L);
            break;
        }
        if (lane == 0) {
            HInfo& ti = sm.info[slot];
            if (FINAL) {
                ti.C = p.C;
                ti.task = p.task;
            } else {
                ti.ring = p.hring + hist_offset(p.npad, st, 0);
                ti.s46 = p.hs46;
            }
            ti.part = p.part;
            ti.plen = (long long)part_len(p);
            ti.ctrl = ctrl;
            ti.L = L;
            ti.npad = FINAL ? p.n : p.npad; ti.I = I; ti.J = J;
            const int2 sl = tile_slots(p, w);
            ti.sR = sl.x; ti.sC = sl.y;
            ti.rows = rows;
            ti.t = t;
            ti.kind = kind;
            ti.even = even;
            ti.staged = staged;
            ti.end = 0;
            mbar_arrive_expect_tx(&sm.tfull[slot], (uint32_t)__popc(use) * 2 * T * (uint32_t)sizeof(float));
        }
        __syncwarp();
        const int a = lane >> 1;
        if ((use >> a) & 1u) {
            const size_t np = p.npad;
            const float* src = FINAL       ? ops[w.x].mu
                               : a == N_MU0 ? p.agg + (size_t)(t & 1) * 3 * np + 2 * np
                               : a == N_MU ? hist_slot(p, st, t) + 2 * np
                                           : p.hnow + (3 * (size_t)st + (a - N_R)) * np;
            bulk_load(&sm.node[slot][lane & 1][a][0], src + (size_t)((lane & 1) ? J : I) * T, T * sizeof(float),
                      &sm.tfull[slot], pol_keep);
        }
        if (++slot == 2) { slot = 0; tph ^= 1u; }
        if constexpr (STREAM) {
            constexpr int RC = q_rows<QT>();
            const void* store = FINAL ? p.qref : p.qstore;
            const unsigned char* qt = static_cast<const unsigned char*>(store) + (size_t)w.w * TT * sizeof(QT);
            const int nch = (rows + RC - 1) / RC;
            for (int c = 0; c < nch; ++c) {
                if (!mbar_wait_warp(&sm.empty[stage], phase ^ 1u)) {
                    give_up(ctrl, L);
                    break;
                }
                if (lane == 0) {
                    mbar_arrive_expect_tx(&sm.full[stage], (uint32_t)H_CHUNK);
                    bulk_load(ring + (size_t)stage * H_CHUNK, qt + (size_t)c * H_CHUNK, (uint32_t)H_CHUNK,
                              &sm.full[stage], pol);
                }
                if (++stage == H_STAGES) { stage = 0; phase ^= 1u; }
            }
        }
    }
    if constexpr (STREAM) await_copies<H_STAGES>(sm.full, stage, phase);
    await_copies<2>(sm.tfull, slot, tph);
    if (ok && !stopped() && mbar_wait_warp(&sm.tempty[slot], tph ^ 1u) && lane == 0) {
        sm.info[slot].end = 1;
        mbar_arrive(&sm.tfull[slot]);
    }
}

__device__ __forceinline__ void unpack_bf16(uint2 a, float2 (&q)[2])
{
    q[0] = make_float2(__uint_as_float(a.x << 16), __uint_as_float(a.x & 0xffff0000u));
    q[1] = make_float2(__uint_as_float(a.y << 16), __uint_as_float(a.y & 0xffff0000u));
}
// Tiles of few sums (at most q mu, mu of the stage and q^3): a consumer warp
// takes two rows at a time, one per half-warp: lane (half hf, hl = lane % 16)
// holds columns 4 hl .. 4 hl + 3 and 64 + 4 hl .. 64 + 4 hl + 3
// of row 2 cw + hf of each 16 rows, so that a half-warp's loads cover
// contiguous bytes and eight pairs share the row's values.
__device__ __forceinline__ void unpack_bf16(uint2 a, uint2 b, float2 (&q)[4])
{
    const uint32_t w[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = make_float2(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xffff0000u));
}

// Q streamed through the ring by the producer.
template <typename QT>
struct StreamedQ {
    static constexpr int ROWS = q_rows<QT>();
    unsigned char* ring;
    int stage;
    uint32_t phase;
    bool abort;
    __device__ __forceinline__ bool acquire(HTail& sm, const HInfo& ti, int lane, bool)
    {
        if (!abort && !mbar_wait_warp(&sm.full[stage], phase)) {
            abort = true;
            if (lane == 0) record_error(ti.ctrl, ST_ETIMEOUT, ti.L);
        }
        return !abort;
    }
    __device__ __forceinline__ void release(HTail& sm, int lane, bool)
    {
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.empty[stage]);
        if (++stage == H_STAGES) { stage = 0; phase ^= 1u; }
    }
    __device__ __forceinline__ void load(int lr, int hl, float2 (&q)[4]) const
    {
        const QT* row = reinterpret_cast<const QT*>(ring + (size_t)stage * H_CHUNK) + (size_t)(lr & (ROWS - 1)) * T;
        if constexpr (sizeof(QT) == 4) {
            const float4 a = *reinterpret_cast<const float4*>(row + 4 * hl), b = *reinterpret_cast<const float4*>(row + 64 + 4 * hl);
            q[0] = make_float2(a.x, a.y); q[1] = make_float2(a.z, a.w);
            q[2] = make_float2(b.x, b.y); q[3] = make_float2(b.z, b.w);
        } else {
            unpack_bf16(*reinterpret_cast<const uint2*>(row + 4 * hl), *reinterpret_cast<const uint2*>(row + 64 + 4 * hl), q);
        }
    }
    __device__ __forceinline__ void load_row(int lr, int lane, float2 (&q)[2]) const
    {
        const QT* row = reinterpret_cast<const QT*>(ring + (size_t)stage * H_CHUNK) + (size_t)(lr & (ROWS - 1)) * T;
        if constexpr (sizeof(QT) == 4) {
            const float4 a = *reinterpret_cast<const float4*>(row + 4 * lane);
            q[0] = make_float2(a.x, a.y); q[1] = make_float2(a.z, a.w);
        } else {
            unpack_bf16(*reinterpret_cast<const uint2*>(row + 4 * lane), q);
        }
    }
};

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }

// Sums of four values over the 16 lanes of a half-warp in a fixed order: lane
// hl holds the total of value hl / 4 (five shuffles).
__device__ __forceinline__ float half_sums4(const float (&x)[4], int hl)
{
    const bool b8 = (hl & 8) != 0, b4 = (hl & 4) != 0;
    float y[2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
        y[k] = (b8 ? x[k + 2] : x[k]) + __shfl_xor_sync(0xffffffffu, b8 ? x[k] : x[k + 2], 8);
    float v = (b4 ? y[1] : y[0]) + __shfl_xor_sync(0xffffffffu, b4 ? y[0] : y[1], 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    return v + __shfl_xor_sync(0xffffffffu, v, 1);
}
// The row sums of four steps -> dst[row].
__device__ __forceinline__ void put_rows(float* dst, float (&x)[4], int r0, int cw, int lane)
{
    const int hl = lane & 15;
    const float v = half_sums4(x, hl);
    if ((hl & 3) == 0) dst[r0 + 16 * (hl >> 2) + 2 * cw + (lane >> 4)] = v;
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = 0.f;
}
// The lane's column sums of both half-warps -> d (one row of cs).
__device__ __forceinline__ void put_cols(float* d, const float2 (&a)[4], int lane)
{
    const int hl = lane & 15;
    float2 m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        m[k].x = a[k].x + __shfl_xor_sync(0xffffffffu, a[k].x, 16);
        m[k].y = a[k].y + __shfl_xor_sync(0xffffffffu, a[k].y, 16);
    }
    if (lane < 16) *reinterpret_cast<float4*>(d + 4 * hl) = make_float4(m[0].x, m[0].y, m[1].x, m[1].y);
    else *reinterpret_cast<float4*>(d + 64 + 4 * hl) = make_float4(m[2].x, m[2].y, m[3].x, m[3].y);
}
__device__ __forceinline__ void ld_cols(const float* d, int hl, float2 (&v)[4])
{
    const float4 a = *reinterpret_cast<const float4*>(d + 4 * hl), b = *reinterpret_cast<const float4*>(d + 64 + 4 * hl);
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
    v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
}

// Runs `row(q, tile row, step of the group)` over the tile's rows of this
// lane's half-warp, 64 rows (four steps) at a time, and `group(first row)`
// after each.
template <class SRC, class ROW, class GROUP>
__device__ __forceinline__ void walk_tile(SRC& src, HTail& sm, const HInfo& ti, int cw, int lane, ROW row, GROUP group)
{
    constexpr int RC = SRC::ROWS < H_GROUP ? SRC::ROWS : H_GROUP, CPG = H_GROUP / RC, SPC = RC / 16;
    const int nch = (ti.rows + RC - 1) / RC, hf = lane >> 4, hl = lane & 15;
#pragma unroll 1
    for (int c0 = 0; c0 < nch; c0 += CPG) {
#pragma unroll
        for (int g = 0; g < CPG; ++g) {
            if (CPG > 1 && c0 + g >= nch) continue;
            if (src.acquire(sm, ti, lane, c0 + g == 0)) {
#pragma unroll
                for (int s = 0; s < SPC; ++s) {
                    const int r = (c0 + g) * RC + 16 * s + 2 * cw + hf;
                    float2 q[4];
                    src.load(r, hl, q);
                    row(q, r, g * SPC + s);
                }
            }
            src.release(sm, lane, c0 + g == nch - 1);
        }
        group(c0 * RC);
    }
}

// q mu, with q^2 (PTWO: live P) and q^3 (ONE) beside it.
template <bool PTWO, bool ONE, bool STAGED, class SRC>
__device__ __forceinline__ void sum_tile(SRC& src, HTail& sm, const HInfo& ti, int slot, int base, int cw, int lane)
{
    const int hl = lane & 15;
    const float (*R)[T] = sm.node[slot][0];
    const float (*C)[T] = sm.node[slot][1];
    float2 cm[4], cs[4], cr[4], cv[4], aR[4], aM[4], aP[4], aE[4];
    ld_cols(C[N_MU0], hl, cm);
    if (STAGED) ld_cols(C[N_MU], hl, cs);
    if (PTWO) ld_cols(C[N_R], hl, cr);
    if (ONE) ld_cols(C[N_W3], hl, cv);
    float xR[4], xM[4], xP[4], xE[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        aR[k] = aM[k] = aP[k] = aE[k] = f2(0.f);
        xR[k] = xM[k] = xP[k] = xE[k] = 0.f;
    }
    auto row = [&](const float2 (&q)[4], int r, int step) {
        const float2 am = f2(R[N_MU0][r]), as = f2(STAGED ? R[N_MU][r] : 0.f), ar = f2(PTWO ? R[N_R][r] : 0.f),
                     av = f2(ONE ? R[N_W3][r] : 0.f);
        float2 sR = f2(0.f), sM = f2(0.f), sP = f2(0.f), sE = f2(0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            aR[k] = fma2(q[k], am, aR[k]);
            sR = fma2(q[k], cm[k], sR);
            if (STAGED) {
                aM[k] = fma2(q[k], as, aM[k]);
                sM = fma2(q[k], cs[k], sM);
            }
            const float2 q2 = mul2(q[k], q[k]);
            if (PTWO) {
                aP[k] = fma2(q2, ar, aP[k]);
                sP = fma2(q2, cr[k], sP);
            }
            if (ONE) {
                const float2 q3 = mul2(q2, q[k]);
                aE[k] = fma2(q3, av, aE[k]);
                sE = fma2(q3, cv[k], sE);
            }
        }
        xR[step] = sR.x + sR.y;
        if (STAGED) xM[step] = sM.x + sM.y;
        if (PTWO) xP[step] = sP.x + sP.y;
        if (ONE) xE[step] = sE.x + sE.y;
    };
    auto group = [&](int r0) {
        put_rows(sm.rs[base], xR, r0, cw, lane);
        if (STAGED) put_rows(sm.rs[base + 1], xM, r0, cw, lane);
        if (PTWO) put_rows(sm.rs[base + 1 + STAGED], xP, r0, cw, lane);
        if (ONE) put_rows(sm.rs[base + 2], xE, r0, cw, lane);
    };
    walk_tile(src, sm, ti, cw, lane, row, group);
    put_cols(sm.cs[base][cw], aR, lane);
    if (STAGED) put_cols(sm.cs[base + 1][cw], aM, lane);
    if (PTWO) put_cols(sm.cs[base + 1 + STAGED][cw], aP, lane);
    if (ONE) put_cols(sm.cs[base + 2][cw], aE, lane);
}

__device__ __forceinline__ void ld_cols4(const float* d, int lane, float2 (&v)[2])
{
    const float4 a = *reinterpret_cast<const float4*>(d + 4 * lane);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
}

// Tiles of more sums: a warp takes two rows at a time (rows 16 s + cw and 8
// more), each lane four of their columns, which leaves room for all the weights
// and sums of a lane's columns (eight columns a lane did not fit 96 registers).
// A row's sums go through a warp reduction of eight values, of two rows where
// there are four at most.  What bounds it is arithmetic (10 to 21 paired
// instructions for two pairs, and the reductions), so a tile sums only what its
// instance's round needs: summing everything in every staged round with live P,
// 450 us a stage over 512 instances of 200 to 4000 points; now 190 (round 0)
// to 310.
template <bool LIVE, bool Q4, bool Q6, bool Q5, bool STAGED>
struct WideSums {
    static constexpr bool has(int s)
    {
        return s == S_R || s == S_W3 || (s == S_M && STAGED) || (s == S_2 && LIVE) || (s == S_4 && Q4) || (s == S_6 && Q6) ||
               (s == S_W5 && Q5);
    }
    static constexpr int index(int s)   // its place among the sums there are
    {
        int k = 0;
        for (int i = 0; i < s; ++i) k += has(i);
        return k;
    }
    static constexpr int count = index(S_COUNT);
    static constexpr int nth(int k)
    {
        for (int i = 0; i < S_COUNT; ++i)
            if (has(i) && index(i) == k) return i;
        return S_COUNT;
    }
};

template <bool LIVE, bool Q4, bool Q6, bool Q5, bool STAGED, class SRC>
__device__ __forceinline__ void wide_tile(SRC& src, HTail& sm, const HInfo& ti, int slot, int cw, int lane)
{
    using W = WideSums<LIVE, Q4, Q6, Q5, STAGED>;
    constexpr int NS = W::count, ROWS = NS <= 4 ? 2 : 1;   // rows per reduction
    const float (*R)[T] = sm.node[slot][0];
    const float (*C)[T] = sm.node[slot][1];
    float2 cm[2], cs[2], cr[2], c3[2], c5[2], a[NS][2];
    ld_cols4(C[N_MU0], lane, cm);
    if (STAGED) ld_cols4(C[N_MU], lane, cs);
    if (LIVE) ld_cols4(C[N_R], lane, cr);
    ld_cols4(C[N_W3], lane, c3);
    if (Q5) ld_cols4(C[N_W5], lane, c5);
#pragma unroll
    for (int s = 0; s < NS; ++s) a[s][0] = a[s][1] = f2(0.f);
    constexpr int RC = SRC::ROWS < H_GROUP ? SRC::ROWS : H_GROUP;
    const int nch = (ti.rows + RC - 1) / RC;
    // the row's sums -> x (in the order of W), the columns' -> a
    auto row = [&](int r, float2 (&x)[NS]) {
        constexpr int iR = W::index(S_R), iM = W::index(S_M), i2 = W::index(S_2), i4 = W::index(S_4), i6 = W::index(S_6),
                      i3 = W::index(S_W3), i5 = W::index(S_W5);
        float2 q[2];
        src.load_row(r, lane, q);
#pragma unroll
        for (int k = 0; k < NS; ++k) x[k] = f2(0.f);
        const float2 rm = f2(R[N_MU0][r]), rs = f2(STAGED ? R[N_MU][r] : 0.f), rr = f2(LIVE ? R[N_R][r] : 0.f),
                     r3 = f2(R[N_W3][r]), r5 = f2(Q5 ? R[N_W5][r] : 0.f);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            a[iR][k] = fma2(q[k], rm, a[iR][k]);
            x[iR] = fma2(q[k], cm[k], x[iR]);
            if constexpr (STAGED) {
                a[iM][k] = fma2(q[k], rs, a[iM][k]);
                x[iM] = fma2(q[k], cs[k], x[iM]);
            }
            const float2 q2 = mul2(q[k], q[k]), q3 = mul2(q2, q[k]);
            if constexpr (LIVE && !Q4) {
                a[i2][k] = fma2(q2, rr, a[i2][k]);
                x[i2] = fma2(q2, cr[k], x[i2]);
            }
            if constexpr (Q4) {
                const float2 wi = mul2(q2, rr), wj = mul2(q2, cr[k]);
                a[i2][k] = __fadd2_rn(a[i2][k], wi);
                x[i2] = __fadd2_rn(x[i2], wj);
                if constexpr (Q6) {
                    const float2 wi2 = mul2(wi, wi), wj2 = mul2(wj, wj);
                    a[i4][k] = __fadd2_rn(a[i4][k], wi2);
                    x[i4] = __fadd2_rn(x[i4], wj2);
                    a[i6][k] = fma2(wi2, wi, a[i6][k]);
                    x[i6] = fma2(wj2, wj, x[i6]);
                } else {
                    a[i4][k] = fma2(wi, wi, a[i4][k]);
                    x[i4] = fma2(wj, wj, x[i4]);
                }
            }
            a[i3][k] = fma2(q3, r3, a[i3][k]);
            x[i3] = fma2(q3, c3[k], x[i3]);
            if constexpr (Q5) {
                const float2 q5 = mul2(q3, q2);
                a[i5][k] = fma2(q5, r5, a[i5][k]);
                x[i5] = fma2(q5, c5[k], x[i5]);
            }
        }
    };
    const int k8 = (lane >> 2) & 7;   // the value that this lane has after a reduction
    float* put = sm.rs[W::nth(ROWS == 2 ? k8 & 3 : k8) % S_COUNT];
    const bool puts = (lane & 3) == 0 && (ROWS == 2 ? k8 & 3 : k8) < NS;
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
        if (src.acquire(sm, ti, lane, c == 0)) {
#pragma unroll(ROWS == 2 ? 1 : 2)
            for (int s = 0; s < RC / 8; s += ROWS) {
                const int r = c * RC + 8 * s + cw;
                float y[8];
#pragma unroll
                for (int u = 0; u < ROWS; ++u) {
                    float2 x[NS];
                    row(r + 8 * u, x);
#pragma unroll
                    for (int k = 0; k < 8 / ROWS; ++k) y[8 / ROWS * u + k] = k < NS ? x[k < NS ? k : 0].x + x[k < NS ? k : 0].y : 0.f;
                }
                const float v = reduce_scatter8x(y, lane);
                if (puts) put[r + (ROWS == 2 ? 8 * (k8 >> 2) : 0)] = v;
            }
        }
        src.release(sm, lane, c == nch - 1);
    }
#pragma unroll
    for (int s = 0; s < NS; ++s)
        *reinterpret_cast<float4*>(&sm.cs[W::nth(s)][cw][4 * lane]) = make_float4(a[s][0].x, a[s][0].y, a[s][1].x, a[s][1].y);
}

// Sum k of the thread's node: its row's (threads 0-127) and / or the eight
// warps' column sums (threads 128-255, and on a diagonal tile both).
__device__ __forceinline__ float node_sum(const HTail& sm, int k, int tid, int rows, bool diag)
{
    const int c = tid & (T - 1);
    float v = (tid < T && c < rows) ? sm.rs[k][c] : 0.f;
    if (tid >= T || diag) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < HCW; ++w) s += sm.cs[k][w][c];
        v += s;
    }
    return v;
}

// ---- final pass
// Sums q mu and q alpha, alpha = clip(mu, 0, C) (regression: mu), of a tile of
// stored FP32 entries, as sum_tile does it.  Means of nodes beyond n are not
// read as they are (nobody writes them): they count as 0.
template <class SRC>
__device__ __forceinline__ void final_tile(SRC& src, HTail& sm, const HInfo& ti, int slot, int base, int cw, int lane)
{
    const int hl = lane & 15, rows = ti.rows, cols = ti.npad - ti.J * T;
    const float* R = sm.node[slot][0][N_MU0];
    const float C = ti.C;
    const bool box = ti.task == 0;
    auto clip = [&](float v) { return box ? fminf(fmaxf(v, 0.f), C) : v; };
    float2 cm[4], ca[4], aR[4], aA[4];
    ld_cols(sm.node[slot][1][N_MU0], hl, cm);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = (k >= 2 ? 64 : 0) + 4 * hl + 2 * (k & 1);
        cm[k] = make_float2(c < cols ? cm[k].x : 0.f, c + 1 < cols ? cm[k].y : 0.f);
        ca[k] = make_float2(clip(cm[k].x), clip(cm[k].y));
        aR[k] = aA[k] = f2(0.f);
    }
    float xR[4] = {0.f, 0.f, 0.f, 0.f}, xA[4] = {0.f, 0.f, 0.f, 0.f};
    auto row = [&](const float2 (&q)[4], int r, int step) {
        const float m = r < rows ? R[r] : 0.f;
        const float2 am = f2(m), aa = f2(clip(m));
        float2 sR = f2(0.f), sA = f2(0.f);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            aR[k] = fma2(q[k], am, aR[k]);
            sR = fma2(q[k], cm[k], sR);
            aA[k] = fma2(q[k], aa, aA[k]);
            sA = fma2(q[k], ca[k], sA);
        }
        xR[step] = sR.x + sR.y;
        xA[step] = sA.x + sA.y;
    };
    auto group = [&](int r0) {
        put_rows(sm.rs[base], xR, r0, cw, lane);
        put_rows(sm.rs[base + 1], xA, r0, cw, lane);
    };
    walk_tile(src, sm, ti, cw, lane, row, group);
    put_cols(sm.cs[base][cw], aR, lane);
    put_cols(sm.cs[base + 1][cw], aA, lane);
}

// The eight consumer warps: tile after tile as the producer publishes them,
// each tile's sums to its slots in a fixed order.  One barrier a tile: a warp
// that has put its sums away waits for the next tile to be published, and the
// barrier then both completes the sums and makes the outcome of that wait (go
// on, end, give up) common.  Small tiles alternate between two sets of sums; a
// wide tile takes more.  (With two barriers a tile and every sum's code passed
// through by every tile: 144 us against 123 us a round at n = 20000.)
template <class SRC>
__device__ __forceinline__ void hist_consumers(SRC& src, HTail& sm, const Inst* __restrict__ tab,
                                               const int4* __restrict__ work, long long ntiles, int tid)
{
    const int cw = tid >> 5, lane = tid & 31;
    int slot = 0, base = 0;
    uint32_t tph = 0;
    auto await_tile = [&]() {
        if (!mbar_wait_warp(&sm.tfull[slot], tph) && lane == 0) {
            sm.cabort = 1;
            if (blockIdx.x < ntiles) record_error(tab[work[blockIdx.x].x].ctrl, ST_ETIMEOUT, -1);
        }
    };
    await_tile();
    hbar();
    for (;;) {
        if (*(volatile int*)&sm.cabort) break;
        if (sm.info[slot].end) break;
        const HInfo& ti = sm.info[slot];
        const int kind = ti.kind, rows = ti.rows;
        const bool diag = ti.I == ti.J, staged = ti.staged, wide = is_wide(kind, staged), live = kind <= K_LIVE, even = ti.even;
        float* part = ti.part;
        const long long plen = ti.plen;
        // this thread's node of the tile's sums: row block's for the first 128
        // threads, column block's for the others; its values of round t - 1
        const int c = tid & (T - 1);
        const size_t o = (size_t)(tid < T ? ti.sR : ti.sC) * T + c;
        float* s46 = nullptr;
        const float p6 = ti.t > 1 ? 2.f : 1.f, n6 = ti.t == 2 ? 2.f : 3.f;   // (of the first rounds: see above)
        float mu1 = 0.f, r1 = 0.f, D1 = 0.f, D3 = 0.f, S4 = 0.f, S6 = 0.f, P = 0.f;
        if (ti.t > 0 && (staged || kind != K_SUM)) {
            const size_t np = ti.npad;
            const float* node = ti.ring + (size_t)(tid < T ? ti.I : ti.J) * T + c;
            const float* old = node + ((unsigned)(ti.t - 1) % (unsigned)kHist) * 4 * np;
            mu1 = old[2 * np];
            if (kind != K_SUM) {
                r1 = 1.f / old[0];
                if (even) {
                    s46 = ti.s46 + o;
                    D1 = old[3 * np];
                    D3 = node[((unsigned)(ti.t + kHist - 3) % (unsigned)kHist) * 4 * np + 3 * np];
                    if (!live) { S4 = s46[0]; S6 = s46[plen]; }
                }
            }
            if (!live && staged) P = part[o];
        }
        if (kind == K_SUM) {
            if (staged) sum_tile<false, false, true>(src, sm, ti, slot, base, cw, lane);
            else sum_tile<false, false, false>(src, sm, ti, slot, base, cw, lane);
        } else if (kind == K_ONE) {
            if (staged) sum_tile<false, true, true>(src, sm, ti, slot, base, cw, lane);
            else sum_tile<false, true, false>(src, sm, ti, slot, base, cw, lane);
        } else if (kind == K_LIVE0) {
            if (staged) sum_tile<true, false, true>(src, sm, ti, slot, base, cw, lane);
            else sum_tile<true, false, false>(src, sm, ti, slot, base, cw, lane);
        } else if (!wide) {
            sum_tile<true, true, false>(src, sm, ti, slot, base, cw, lane);
        } else {
            hbar();   // the previous tile's sums are read out
            if (staged) {
                if (kind == K_LIVE1) wide_tile<true, false, false, false, true>(src, sm, ti, slot, cw, lane);
                else if (kind == K_LIVE4) wide_tile<true, true, false, false, true>(src, sm, ti, slot, cw, lane);
                else if (kind == K_LIVE) wide_tile<true, true, true, true, true>(src, sm, ti, slot, cw, lane);
                else wide_tile<false, false, false, true, true>(src, sm, ti, slot, cw, lane);
            } else {
                if (kind == K_LIVE4) wide_tile<true, true, false, false, false>(src, sm, ti, slot, cw, lane);
                else if (kind == K_LIVE) wide_tile<true, true, true, true, false>(src, sm, ti, slot, cw, lane);
                else wide_tile<false, false, false, true, false>(src, sm, ti, slot, cw, lane);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.tempty[slot]);   // its parameters are not read again
        if (++slot == 2) { slot = 0; tph ^= 1u; }
        await_tile();
        hbar();
        // (slot entries of nodes beyond n are written, and read by no one else)
        const bool mine = tid < T || !diag;
        float* d = part + o;
        if (!wide) {
            const float R = node_sum(sm, base, tid, rows, diag);
            if (mine) d[2 * plen] = R;
            if (kind != K_SUM || staged) {
                const float M = staged ? node_sum(sm, base + 1, tid, rows, diag) : 0.f;
                const float S2 = live ? node_sum(sm, base + 1 + staged, tid, rows, diag) : 0.f;
                const float W3 = (kind == K_ONE || kind == K_LIVE1) ? node_sum(sm, base + 2, tid, rows, diag) : 0.f;
                const float E = r1 * (fmaf(S4, D1, W3) + r1 * S6 * (D3 - n6 * D1));
                if (live) P = -S2;
                if (mine) {
                    if (live) d[0] = P;
                    if (staged) d[plen] = fmaf(P, mu1, E - M);
                    else if (kind != K_LIVE0) d[plen] = E;
                }
            }
        } else {
            const float R = node_sum(sm, S_R, tid, rows, diag);
            const float M = staged ? node_sum(sm, S_M, tid, rows, diag) : 0.f;
            if (live) {
                const float S2 = node_sum(sm, S_2, tid, rows, diag);
                if (even && s46) {
                    S4 = node_sum(sm, S_4, tid, rows, diag);
                    S6 = kind == K_LIVE ? node_sum(sm, S_6, tid, rows, diag) : 0.f;
                }
                P = fmaf(r1, fmaf(-p6 * r1, S6, S4), -S2);
            }
            const float W3 = node_sum(sm, S_W3, tid, rows, diag);
            const float W5 = kind == K_LIVE || kind == K_TWO ? node_sum(sm, S_W5, tid, rows, diag) : 0.f;
            const float E = r1 * (fmaf(S4, D1, W3) + r1 * fmaf(S6, D3 - n6 * D1, W5));
            if (mine) {
                d[2 * plen] = R;
                if (live) d[0] = P;
                if (live && s46) { s46[0] = S4; s46[plen] = S6; }
                d[plen] = staged ? fmaf(P, mu1, E - M) : E;
            }
            hbar();   // before the next tile writes its sums
        }
        base = S_SMALL - base;
    }
}

// The consumers of the final pass: as hist_consumers, sums to the slots 2 and 3.
template <class SRC>
__device__ __forceinline__ void final_consumers(SRC& src, HTail& sm, const Inst* __restrict__ tab,
                                                const int4* __restrict__ work, long long ntiles, int tid)
{
    const int cw = tid >> 5, lane = tid & 31;
    int slot = 0, base = 0;
    uint32_t tph = 0;
    auto await_tile = [&]() {
        if (!mbar_wait_warp(&sm.tfull[slot], tph) && lane == 0) {
            sm.cabort = 1;
            if (blockIdx.x < ntiles) record_error(tab[work[blockIdx.x].x].ctrl, ST_ETIMEOUT, -1);
        }
    };
    await_tile();
    hbar();
    while (!*(volatile int*)&sm.cabort && !sm.info[slot].end) {
        const HInfo& ti = sm.info[slot];
        const bool diag = ti.I == ti.J;
        const int rows = ti.rows;
        const long long plen = ti.plen;
        float* d = ti.part + (size_t)(tid < T ? ti.sR : ti.sC) * T + (tid & (T - 1));
        final_tile(src, sm, ti, slot, base, cw, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.tempty[slot]);
        if (++slot == 2) { slot = 0; tph ^= 1u; }
        await_tile();
        hbar();
        const float R = node_sum(sm, base, tid, rows, diag), A = node_sum(sm, base + 1, tid, rows, diag);
        if (tid < T || !diag) {
            d[2 * plen] = R;
            d[3 * plen] = A;
        }
        base = S_SMALL - base;
    }
}

__device__ __forceinline__ void init_htail(HTail& sm)
{
    for (int s = 0; s < H_STAGES; ++s) { mbar_init(&sm.full[s], 1); mbar_init(&sm.empty[s], HCW); }
    for (int s = 0; s < 2; ++s) { mbar_init(&sm.tfull[s], 1); mbar_init(&sm.tempty[s], HCW); }
    sm.cabort = 0;
}

// Read by the producer warp at the start of a sweep, beside the schedule: a
// handle's control block.  False where there is nothing to do: no tiles, or the
// instance has stopped (the rest of a captured chunk of rounds, which would
// otherwise pass through every tile: 640 us a round at n = 100000).
__device__ __forceinline__ bool sweep_head(const Sched* sched, const Ctrl* ctrls, bool one, CtrlHead& head)
{
    if (one) head = ctrl_head(ctrls);
    return sched->ntiles > 0 && !(one && head.done);
}

// Q stored (FP32 or BF16) and streamed.
template <typename QT>
__global__ void __launch_bounds__(H_THREADS, 2)
    k_sweep_hist(const Inst* __restrict__ tab, const int4* __restrict__ work, const Sched* __restrict__ sched, int stage_no,
                 const Ctrl* ctrls, int one)
{
    chain_next();
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = align_smem(smem_raw, 128);
    HTail& sm = *reinterpret_cast<HTail*>(ring + H_STAGES * H_CHUNK);
    const int tid = threadIdx.x;
    if (tid == 0) {
        init_htail(sm);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    chain_wait();
    const bool producer = tid >= HCW * 32;
    CtrlHead head{};
    if (producer) {
        const bool go = sweep_head(sched, ctrls, one != 0, head);
        if ((tid & 31) == 0) sm.go = go;
    }
    __syncthreads();
    if (!sm.go) return;
    const long long ntiles = sched->ntiles;
    work += sched->off;
    if (producer) {
        hist_producer<QT>(tab, work, ntiles, sm, ring, nullptr, tid & 31, stage_no, nullptr, ctrls, one != 0, head);
        return;
    }
    StreamedQ<QT> src{ring, 0, 0u, false};
    hist_consumers(src, sm, tab, work, ntiles, tid);
}

constexpr size_t hist_smem_bytes() { return 128 + H_STAGES * H_CHUNK + sizeof(HTail); }

// ---- Q recomputed in every sweep -------------------------------------------
// As the fused recompute of sweep.cu, without messages to stream: warps 0-7
// consume, warp 8 publishes the tiles, warp 9 copies the BF16 feature blocks,
// one thread of warp 10 issues the tcgen05 MMAs into a double-buffered TMEM
// accumulator, and warps 12-19 (two per TMEM lane quarter, one per column
// half) turn the Gram rows into BF16 Q values in a double-buffered shared
// tile, bitwise the values of the BF16 store.
constexpr int HR_XSTAGES = 2;
constexpr int HR_EPI = 8;
constexpr int HR_THREADS = (12 + HR_EPI) * 32;
constexpr uint32_t HR_TMEM_COLS = 256;
constexpr size_t HR_QTILE = (size_t)TT * sizeof(__nv_bfloat16);

struct HrExtra {
    unsigned long long xfull[HR_XSTAGES], xempty[HR_XSTAGES];
    unsigned long long accfull[2], accempty[2];
    unsigned long long qfull[2], qempty[2];
    unsigned long long drain;
    uint32_t tmem_base;
    int abort;
    ColTile cols[HR_EPI];
};
constexpr size_t hist_rc_smem_bytes()
{
    return 1024 + HR_XSTAGES * 2 * BLK_BYTES + 2 * HR_QTILE + sizeof(HTail) + sizeof(HrExtra);
}

// Q from the shared tile.  Its rows are stored with their 16-byte chunks
// permuted: chunk k of row r sits at chunk k ^ (r % 8), so that the epilogue's
// stores (one row per lane, the same chunk) spread over all banks.
struct TileQ {
    static constexpr int ROWS = T;
    const unsigned char* qtile;   // [2][T][T] BF16
    HrExtra* ex;
    int it;
    bool abort;
    __device__ __forceinline__ bool acquire(HTail& sm, const HInfo& ti, int lane, bool first)
    {
        if (first && !abort && !mbar_wait_warp(&ex->qfull[it & 1], (uint32_t)((it >> 1) & 1))) {
            abort = true;
            if (lane == 0) record_error(ti.ctrl, ST_ETIMEOUT, ti.L);
        }
        return !abort;
    }
    __device__ __forceinline__ void release(HTail&, int lane, bool last)
    {
        if (!last) return;
        __syncwarp();
        if (lane == 0) mbar_arrive(&ex->qempty[it & 1]);
        ++it;
    }
    __device__ __forceinline__ void load(int r, int hl, float2 (&q)[4]) const
    {
        const unsigned char* row = qtile + (size_t)(it & 1) * HR_QTILE + (size_t)r * T * 2;
        const int o = (((hl >> 1) ^ (r & 7)) << 4) + ((hl & 1) << 3);
        unpack_bf16(*reinterpret_cast<const uint2*>(row + o), *reinterpret_cast<const uint2*>(row + 128 + o), q);
    }
    __device__ __forceinline__ void load_row(int r, int lane, float2 (&q)[2]) const
    {
        const unsigned char* row = qtile + (size_t)(it & 1) * HR_QTILE + (size_t)r * T * 2;
        unpack_bf16(*reinterpret_cast<const uint2*>(row + (((lane >> 1) ^ (r & 7)) << 4) + ((lane & 1) << 3)), q);
    }
};

// A role's way through the CTA's tiles: list entries two tiles ahead of their
// turn, and whether an instance has stopped read once per run of its tiles, so that
// no role waits for either between two tiles.
struct TileWalk {
    const int4* work;
    long long ntiles;
    int4 w0, w1;      // the next tile and the one after
    int inst = -1;
    bool stopped = false;
    __device__ __forceinline__ TileWalk(const int4* list, long long n) : work(list), ntiles(n)
    {
        const long long L = blockIdx.x;
        w0 = L < ntiles ? work[L] : make_int4(0, 0, 0, 0);
        w1 = L + gridDim.x < ntiles ? work[L + gridDim.x] : w0;
    }
    __device__ __forceinline__ int4 next(long long L)
    {
        const int4 w = w0;
        w0 = w1;
        if (L + 2LL * gridDim.x < ntiles) w1 = work[L + 2LL * gridDim.x];
        return w;
    }
    __device__ __forceinline__ bool done(int k, const Ctrl* ctrls)
    {
        if (k != inst) {
            inst = k;
            stopped = *(volatile const int*)&ctrls[k].done != 0;
        }
        return stopped;
    }
};

__global__ void __launch_bounds__(HR_THREADS, 1)
    k_sweep_hist_rc(const Inst* __restrict__ tab, const int4* __restrict__ work, const Sched* __restrict__ sched,
                    int stage_no, const Ctrl* ctrls, int one)
{
    chain_next();
    chain_wait();
    extern __shared__ unsigned char smem_raw[];
    unsigned char* xops = align_smem(smem_raw, 1024);
    unsigned char* qtile = xops + HR_XSTAGES * 2 * BLK_BYTES;
    HTail& sm = *reinterpret_cast<HTail*>(qtile + 2 * HR_QTILE);
    HrExtra& ex = *reinterpret_cast<HrExtra*>(reinterpret_cast<unsigned char*>(&sm) + sizeof(HTail));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        init_htail(sm);
        for (int s = 0; s < HR_XSTAGES; ++s) { mbar_init(&ex.xfull[s], 1); mbar_init(&ex.xempty[s], 1); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ex.accfull[b], 1);
            mbar_init(&ex.accempty[b], HR_EPI);
            mbar_init(&ex.qfull[b], HR_EPI);
            mbar_init(&ex.qempty[b], HCW);
        }
        mbar_init(&ex.drain, 1);
        ex.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    CtrlHead head{};
    if (warp == 8) {
        const bool go = sweep_head(sched, ctrls, one != 0, head);
        if (lane == 0) sm.go = go;
    }
    __syncthreads();
    if (!sm.go) return;
    const long long ntiles = sched->ntiles;
    work += sched->off;
    if (warp == 10) tmem_alloc(&ex.tmem_base, HR_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = ex.tmem_base;
    volatile int* abort_flag = &ex.abort;

    if (warp < HCW) {
        TileQ src{qtile, &ex, 0, false};
        hist_consumers(src, sm, tab, work, ntiles, tid);
    } else if (warp == 8) {
        hist_producer<void>(tab, work, ntiles, sm, nullptr, abort_flag, lane, stage_no, nullptr, ctrls, one != 0, head);
    } else if (warp == 9) {
        if (lane == 0) {
            const uint64_t pol = l2_evict_last_policy();   // the features are read again by many tiles
            int xs = 0;
            uint32_t ph = 0;
            bool run = true;
            TileWalk walk(work, ntiles);
            for (long long L = blockIdx.x; L < ntiles && run; L += gridDim.x) {
                const int4 w = walk.next(L);
                const Inst& p = tab[w.x];
                if (walk.done(w.x, ctrls)) continue;
                const unsigned char* Xp = static_cast<const unsigned char*>(p.Xp);
                const int nkc = p.nkc;
                for (int kc = 0; kc < nkc; ++kc) {
                    if (*abort_flag || !mbar_wait(&ex.xempty[xs], ph ^ 1u)) {
                        *abort_flag = 1;
                        record_error(p.ctrl, ST_ETIMEOUT, L);
                        run = false;
                        break;
                    }
                    unsigned char* A = xops + (size_t)xs * 2 * BLK_BYTES;
                    mbar_arrive_expect_tx(&ex.xfull[xs], 2 * BLK_BYTES);
                    bulk_load(A, Xp + ((size_t)w.y * nkc + kc) * BLK_BYTES, BLK_BYTES, &ex.xfull[xs], pol);
                    bulk_load(A + BLK_BYTES, Xp + ((size_t)w.z * nkc + kc) * BLK_BYTES, BLK_BYTES, &ex.xfull[xs], pol);
                    if (++xs == HR_XSTAGES) { xs = 0; ph ^= 1u; }
                }
            }
            await_copies<HR_XSTAGES>(ex.xfull, xs, ph);
        }
    } else if (warp == 10) {
        if (lane == 0) {
            constexpr uint32_t IDESC = idesc_bf16_f32(T, T);
            int xs = 0, acc = 0;
            uint32_t ph = 0, aph = 0;
            TileWalk walk(work, ntiles);
            for (long long L = blockIdx.x; L < ntiles; L += gridDim.x) {
                const int inst = walk.next(L).x;
                const Inst& p = tab[inst];
                if (walk.done(inst, ctrls)) continue;
                const int nkc = p.nkc;
                bool ok = !*abort_flag && mbar_wait(&ex.accempty[acc], aph ^ 1u);
                tc_fence_after();
                const uint32_t d = tbase + (uint32_t)acc * T;
                for (int kc = 0; kc < nkc && ok; ++kc) {
                    if (*abort_flag || !mbar_wait(&ex.xfull[xs], ph)) { ok = false; break; }
                    tc_fence_after();
                    const unsigned char* A = xops + (size_t)xs * 2 * BLK_BYTES;
#pragma unroll
                    for (int s = 0; s < KCH / 16; ++s)
                        tc_mma_bf16(d, smem_desc(A + s * 256, 128, 1024), smem_desc(A + BLK_BYTES + s * 256, 128, 1024), IDESC,
                                    (kc | s) != 0);
                    tc_commit(&ex.xempty[xs]);
                    if (++xs == HR_XSTAGES) { xs = 0; ph ^= 1u; }
                }
                if (!ok) {
                    *abort_flag = 1;
                    record_error(p.ctrl, ST_ETIMEOUT, L);
                    break;
                }
                tc_commit(&ex.accfull[acc]);
                if (++acc == 2) { acc = 0; aph ^= 1u; }
            }
            tc_commit(&ex.drain);
            if (!mbar_wait(&ex.drain, 0u)) *abort_flag = 1;
        }
    } else if (warp >= 12) {
        const int ew = warp - 12, g = warp & 3, half = ew >> 2, r = 32 * g + lane;
        int it = 0;
        TileWalk walk(work, ntiles);
        TileCols<2> ahead{};
        if (blockIdx.x < ntiles) ahead = load_tile_cols<2>(tab[walk.w0.x], walk.w0.z, walk.w0.y * T + r, lane, 2 * half);
        for (long long L = blockIdx.x; L < ntiles; L += gridDim.x) {
            const int4 w = walk.next(L);
            const TileCols<2> cols = ahead;
            if (L + gridDim.x < ntiles)
                ahead = load_tile_cols<2>(tab[walk.w0.x], walk.w0.z, walk.w0.y * T + r, lane, 2 * half);
            const Inst& p = tab[w.x];
            Ctrl* ctrl = p.ctrl;
            if (walk.done(w.x, ctrls)) continue;
            const int n = p.n, I = w.y, J = w.z, acc = it & 1;
            const uint32_t par = (uint32_t)((it >> 1) & 1);
            const float gamma = p.gamma, lam2 = p.lam2;
            const float yi = cols.yi, si = cols.si;
            put_tile_cols(ex.cols[ew], cols, gamma, lane, 2 * half);
            const bool stop = __shfl_sync(0xffffffffu, *abort_flag, 0) != 0;
            if (stop || !mbar_wait_warp(&ex.accfull[acc], par) || !mbar_wait_warp(&ex.qempty[acc], par ^ 1u)) {
                if (lane == 0) {
                    *abort_flag = 1;
                    record_error(ctrl, ST_ETIMEOUT, L);
                }
                break;
            }
            tc_fence_after();
            const float ai = -gamma * kLog2e * si, c2 = 2.f * gamma * kLog2e;
            const uint32_t s1 = __float_as_uint(yi) & 0x80000000u, si2 = s1 | (s1 >> 16);
            uint4* qrow = reinterpret_cast<uint4*>(qtile + (size_t)acc * HR_QTILE + (size_t)r * T * 2);
            const int sw = r & 7;
#pragma unroll 1
            for (int cc = 2 * half; cc < 2 * half + 2; ++cc) {
                const uint32_t valid = chunk_valid(n, I, J, r, cc);
                float v[32];
                tmem_ld32(tbase + (uint32_t)acc * T + ((uint32_t)(32 * g) << 16) + (uint32_t)(32 * cc), v);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float vh[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) vh[u] = v[16 * h + u];
                    uint4 out[2];
                    q_half_bf16(vh, 32 * cc + 16 * h, ai, si2, ex.cols[ew], c2, lam2, (valid >> (16 * h)) & 0xffffu, out);
                    qrow[(4 * cc + 2 * h) ^ sw] = out[0];
                    qrow[(4 * cc + 2 * h + 1) ^ sw] = out[1];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&ex.accempty[acc]);
                mbar_arrive(&ex.qfull[acc]);
            }
            ++it;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 10) {
        tc_fence_after();
        tmem_dealloc(tbase, HR_TMEM_COLS);
    }
}

// Final pass over listed tiles of stored FP32 entries: off-diagonal sums
// sum_{j != i} Q_ij mu_j (the residual slots, which every round writes anew) and
// sum_{j != i} Q_ij alpha_j (slots 3): the P and H slots keep the sums of the
// current messages, which a staged round that goes on from here reads.
//
// What bounds it: one read of the entries, 4 bytes a pair, so it streams them as
// a round does.  With a CTA a tile that loaded its 64 KB at once: 178 us at n =
// 20000, 4.2 ms at n = 100000; now 121 us and 3.0 ms.
__global__ void __launch_bounds__(H_THREADS, 2)
    k_final_tiles_q(const Inst* __restrict__ tab, const StopOp* __restrict__ ops, const int4* __restrict__ work, long long ntiles)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = align_smem(smem_raw, 128);
    HTail& sm = *reinterpret_cast<HTail*>(ring + H_STAGES * H_CHUNK);
    const int tid = threadIdx.x;
    if (tid == 0) {
        init_htail(sm);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (tid >= HCW * 32) {
        hist_producer<float, true>(tab, work, ntiles, sm, ring, nullptr, tid & 31, 0, ops, nullptr, false, CtrlHead{});
        return;
    }
    StreamedQ<float> src{ring, 0, 0u, false};
    final_consumers(src, sm, tab, work, ntiles, tid);
}

// What choose_path() wants to know of the pairs, over listed tiles, for the
// instances whose margin leaves it open (the others cost a look at their
// control block).  From the FP32 entries, so that the forms with BF16 entries
// decide alike.
//
// What bounds it: one read of the entries, 4 bytes a pair.  A warp has its 16
// rows of a tile in flight at once and meets no barrier.  With four rows in
// flight and the check shared through a barrier: 38 us at n = 6238 (1225
// tiles); now 27; a batch of 18 instances: 167 -> 73 us.
//
// Other warps raise the maxima meanwhile, so whether an instance is still open
// is one lane's answer for its warp: all lanes take part in the shuffles below,
// or none.
__global__ void __launch_bounds__(256, 2) k_pair_z(const Inst* __restrict__ tab, const int4* __restrict__ work,
                                                  long long ntiles, bool single)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_agrees = [](bool mine) { return __shfl_sync(0xffffffffu, (int)mine, 0) != 0; };
    if (single && !warp_agrees(pair_z_open(tab[0]))) return;
    for (long long L = blockIdx.x; L < ntiles; L += gridDim.x) {
        const int4 w = work[L];
        for (int k = w.x; k >= 0; k = tab[k].form_next - 1) {
            const Inst& p = tab[k];
            if (!pair_z_asks(p)) continue;   // (what it reads is fixed by now)
            const float* q = p.qref + (size_t)w.w * TT + warp * T + 4 * lane;
            float4 a[T / 8];
#pragma unroll
            for (int r = 0; r < T / 8; ++r) a[r] = *reinterpret_cast<const float4*>(q + (size_t)r * 8 * T);
            if (!warp_agrees(orders_suffice(zu_pairs(p.ctrl)))) continue;   // settled by other tiles
            float rj[4], ri = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                rj[e] = __fdividef(1.f, p.qdiag[min(w.z * T + 4 * lane + e, p.n - 1)]);   // (entries beyond n are 0)
            if (lane < T / 8) ri = __fdividef(1.f, p.qdiag[min(w.y * T + 8 * lane + warp, p.n - 1)]);
            float best[2] = {0.f, FLT_MIN};   // the second never 0: the pass has run
#pragma unroll
            for (int r = 0; r < T / 8; ++r) {
                const float rr = __shfl_sync(0xffffffffu, ri, r);
                note_pair_z(a[r].x, rr, rj[0], best);
                note_pair_z(a[r].y, rr, rj[1], best);
                note_pair_z(a[r].z, rr, rj[2], best);
                note_pair_z(a[r].w, rr, rj[3], best);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                best[e] = warp_max_f(best[e]);
                if (lane == 0 && __float_as_uint(best[e]) > *(volatile unsigned*)&p.ctrl->zpair_bits[e])
                    atomicMax(&p.ctrl->zpair_bits[e], __float_as_uint(best[e]));
            }
        }
    }
}

}  // namespace

cudaError_t prepare_sweep_hist()
{
    cudaError_t e = cudaFuncSetAttribute(k_sweep_hist<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)hist_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep_hist<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)hist_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_final_tiles_q, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hist_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sweep_hist_rc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hist_rc_smem_bytes());
    return e;
}

void launch_sweep_hist(const Inst* tab, const int4* work, const Sched* sched, int stage_no, const RoundGrid& g, int q_mode,
                       bool chained, cudaStream_t s)
{
    if (q_mode == 2)
        launch_chained(chained, k_sweep_hist_rc, g.sweep, HR_THREADS, hist_rc_smem_bytes(), s, tab, work, sched, stage_no,
                       g.ctrls, g.one);
    else if (q_mode == 1)
        launch_chained(chained, k_sweep_hist<__nv_bfloat16>, g.sweep, H_THREADS, hist_smem_bytes(), s, tab, work, sched,
                       stage_no, g.ctrls, g.one);
    else
        launch_chained(chained, k_sweep_hist<float>, g.sweep, H_THREADS, hist_smem_bytes(), s, tab, work, sched, stage_no,
                       g.ctrls, g.one);
}

void launch_final_tiles_q(const Inst* tab, const StopOp* ops, const int4* tiles, long long ntiles, cudaStream_t s)
{
    const long long most = 2 * num_sms();
    k_final_tiles_q<<<(int)(ntiles < most ? ntiles : most), H_THREADS, hist_smem_bytes(), s>>>(tab, ops, tiles, ntiles);
}

void launch_pair_z(const Inst* tab, const int4* tiles, long long ntiles, int q_mode, bool single, cudaStream_t s)
{
    if (ntiles <= 0) return;
    if (q_mode == 2) {
        (void)launch_pair_z_gram(tab, tiles, ntiles, single, s);   // errors surface at the caller's cudaGetLastError
        return;
    }
    const long long most = 2 * num_sms();
    k_pair_z<<<(int)(ntiles < most ? ntiles : most), 256, 0, s>>>(tab, tiles, ntiles, single);
}

}  // namespace gabp
