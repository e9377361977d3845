// The node history of PATH_HIST (common.cuh): what a round appends to it, how
// many terms a round takes, and which instances keep it.
#pragma once

#include "common.cuh"

#include <cstddef>
#include "ptx.cuh"

namespace gabp {

// {Ptilde, htilde, mu, D} arrays (npad floats each) of round t as stage `st`
// saw them.
__host__ __device__ __forceinline__ size_t hist_offset(int npad, int st, int t)
{
    return ((size_t)st * kHist + (unsigned)t % (unsigned)kHist) * 4 * npad;
}
__device__ __forceinline__ float* hist_slot(const Inst& p, int st, int t) { return p.hring + hist_offset(p.npad, st, t); }

// Appends node x's aggregates of round t to stage st's history; mu2 and D2 are
// its mean and D two rounds earlier.  D(0) counts as 0, and D(1) once in the
// weight of q^5: no message precedes round 0 (sweep_hist.cu).
__device__ __forceinline__ void hist_push(const Inst& p, int st, int t, int x, float P, float h, float mu, float mu2,
                                          float D2)
{
    const size_t np = p.npad;
    float* s = hist_slot(p, st, t);
    const float D = t > 0 ? mu - mu2 : 0.f, ip = 1.f / P;
    s[x] = P;
    s[np + x] = h;
    s[2 * np + x] = mu;
    s[3 * np + x] = D;
    float* w = p.hnow + (size_t)3 * st * np;
    w[x] = ip;
    w[np + x] = D * ip;
    w[2 * np + x] = (D2 - (t > 1 ? 2.f : 1.f) * D) * ip * ip;
}

// Node x's means and htilde before round t: 0 (Step 1, or a restart of the H
// messages, whose P messages are kept).
__device__ __forceinline__ void hist_clear(const Inst& p, int x)
{
    for (int k = 0; k < p.nstages * kHist; ++k) {
        float* s = p.hring + (size_t)k * 4 * p.npad;
        for (int a = 1; a < 4; ++a) s[a * p.npad + x] = 0.f;
    }
}
// Step 1 (Algorithm 2; all messages 0): the aggregates of round 0.
__device__ __forceinline__ void hist_start(const Inst& p, int x, float P, float h, float mu)
{
    if (!p.hist) return;
    hist_clear(p, x);
    hist_push(p, 0, 0, x, P, h, mu, 0.f, 0.f);
}
// The H messages restart from 0 at round t with right-hand side h and the P
// messages kept.
__device__ __forceinline__ void hist_restart(const Inst& p, int t, int x, float P, float h, float mu)
{
    hist_clear(p, x);
    p.agg[(size_t)((t + 1) & 1) * 3 * p.npad + 2 * (size_t)p.npad + x] = 0.f;   // mu(t - 1)
    hist_push(p, 0, t, x, P, h, mu, 0.f, 0.f);
}
// Nodes x in [n, npad) that fill the last tile: their entries of Q are 0, and
// with finite values they add 0 to every sum, so that the sweep needs no
// masks.
__device__ __forceinline__ void hist_pad(const Inst& p, int x)
{
    if (!p.hist) return;
    for (int k = 0; k < 2; ++k) {
        float* a = p.agg + (size_t)k * 3 * p.npad;
        a[x] = 1.f;
        a[p.npad + x] = 0.f;
        a[2 * p.npad + x] = 0.f;
    }
    for (int k = 0; k < 3 * p.nstages; ++k) p.hnow[(size_t)k * p.npad + x] = 0.f;
    for (int k = 0; k < p.nstages * kHist; ++k) p.hring[(size_t)k * 4 * p.npad + x] = 1.f;
    hist_clear(p, x);
}

// What the kernels of a round read of an instance's control block, in two
// 16-byte loads.
struct CtrlHead {
    int t, done, p_frozen, path, terms, even;
};
__device__ __forceinline__ CtrlHead ctrl_head(const Ctrl* c)
{
    static_assert(offsetof(Ctrl, t) == 0 && offsetof(Ctrl, done) == 4 && offsetof(Ctrl, p_frozen) == 8 &&
                      offsetof(Ctrl, path) == 12 && offsetof(Ctrl, terms) == 16 && offsetof(Ctrl, even) == 20, "");
    CtrlHead h;
    int k, z;
    asm volatile("ld.volatile.global.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(h.t), "=r"(h.done), "=r"(h.p_frozen), "=r"(h.path) : "l"(c) : "memory");
    asm volatile("ld.volatile.global.v4.s32 {%0, %1, %2, %3}, [%4 + 16];"
                 : "=r"(h.terms), "=r"(h.even), "=r"(k), "=r"(z) : "l"(c) : "memory");
    return h;
}

// What a round leaves out (sweep_hist.cu) moves a mean by at most this
// fraction of the largest mean: the rounding of an FP32 mean.
constexpr float kLeftOut = 5.96e-8f;   // 2^-24
// Odd terms of E (q^3, q^5) a round needs.  `change` is the largest two-round
// change of a mean, relative to the largest mean (those of earlier rounds
// weighed in, next_change): without any every mean is off by at most z change,
// with the first by 3 z^2 change, with both by 10 z^3 change (<= kLeftOut on this
// path).
__device__ __forceinline__ int e_terms(float z, float change)
{
    if (z * change <= kLeftOut) return 0;
    return 3.f * z * z * change <= kLeftOut ? 1 : 2;
}
// Whether the even orders q^4, q^6 count: without them the P messages into a
// node are off by at most z u of Ptilde, E by z u change.
// (2: q^4 and q^6; 1: q^4 alone, where what q^6 adds is at most 2 z^2 u of Ptilde
// and 4 z^2 u change of a mean)
__device__ __forceinline__ int even_orders(float z, float u)
{
    return 4.f * z * z * u > kLeftOut ? 2 : 2.f * z * u > kLeftOut ? 1 : 0;
}
// Whether the tiles of a round after the first write E (live rounds with even
// orders always do).
__device__ __forceinline__ bool round_has_e(int terms, int even, bool frozen) { return terms > 0 || (!frozen && even); }
// The change of the round just done is `now`; u = |q| / d damps what earlier
// ones leave, and a round that happens to change little counts for at least
// half the one before.
__device__ __forceinline__ float next_change(float now, float before, float u)
{
    return fmaxf(now + fminf(u, 1.f) * before, 0.5f * before);
}

// Which instances keep a history (PATH_HIST) instead of their messages: those
// for which the orders the sweep sums, up to q^6, are all there is in FP32: 10
// z^3 <= 2^-24 over the pairs, z = q^2 / (d_i d_j) and u = |q| / d (z <= 1.8e-3;
// pairs beyond are near-duplicates with few neighbours).  z and u are
// known at Step 1, with d = Q_ii; later, with R_i <= Q_ii (strict dominance) and
// u0 = max |q_ij| / Q_jj <= 1/4, d_i >= Ptilde_i >= theta Q_ii for theta (1 -
// theta) = u0: if Ptilde_k >= theta Q_kk for every k, the P messages into i are
// at most sum_k |q_ik| (u0 / theta) <= (u0 / theta) Q_ii, so Ptilde_i >= (1 - u0
// / theta) Q_ii = theta Q_ii.  u0 <= max |q| max 1 / Q_ii and z <= u0^2 may settle
// it; else the pairs are looked at (k_pair_z).
struct ZU { float z, u; };
// Bounds for every round from those of Step 1.
__device__ __forceinline__ ZU zu_bounds(float z0, float u0)
{
    if (!(u0 <= 0.25f)) return ZU{1.f, 1.f};
    const float r = 2.f / (1.f + sqrtf(1.f - 4.f * u0));   // 1 / theta
    return ZU{z0 * r * r, u0 * r};
}
__device__ __forceinline__ bool orders_suffice(ZU b) { return 10.f * b.z * b.z * b.z <= kLeftOut; }
// From the instance's diagonal alone (z <= u^2); 1 where some row is not
// strictly dominant.
__device__ __forceinline__ ZU zu_diagonal(const Inst& p, const Ctrl* c)
{
    const double inv = __longlong_as_double((long long)c->inv_margin_bits);
    if (!p.hist || !(inv > 0.0 && inv < 1e30)) return ZU{1.f, 1.f};
    const float u = 1.01f * (1.f + p.lam2) * __uint_as_float(c->rq_bits);
    return zu_bounds(u * u, u);
}
// A pair's z and u of Step 1 into the running maxima (r = 1 / Q_ii).
__device__ __forceinline__ void note_pair_z(float q, float ri, float rj, float (&best)[2])
{
    const float u = q * ri, v = q * rj;
    best[0] = fmaxf(best[0], u * v);
    best[1] = fmaxf(best[1], fmaxf(fabsf(u), fabsf(v)));
}
// (a percent for entries rounded to BF16)
__device__ __forceinline__ ZU zu_pairs(const Ctrl* c)
{
    const volatile unsigned* b = c->zpair_bits;
    return zu_bounds(1.01f * __uint_as_float(b[0]), 1.01f * __uint_as_float(b[1]));
}
// Whether the pairs of an instance are to be looked at (further): they may
// admit it, or show a z so much smaller that its rounds take fewer terms
// (z from the diagonal above 2^-20: most instances of up to about 10000 points;
// the pass costs about as much as one round).
__device__ __forceinline__ bool pair_z_asks(const Inst& p)
{
    const Ctrl* c = p.ctrl;
    const double inv = __longlong_as_double((long long)c->inv_margin_bits);
    return p.hist && inv > 0.0 && inv < 1e30 && zu_diagonal(p, c).z > 9.5e-7f;
}
__device__ __forceinline__ bool pair_z_open(const Inst& p) { return pair_z_asks(p) && orders_suffice(zu_pairs(p.ctrl)); }
// At Step 1: the message path of an instance and the bounds its rounds go by.
__device__ __forceinline__ void choose_path(const Inst& p, Ctrl* c)
{
    ZU b = zu_diagonal(p, c);
    if (c->zpair_bits[1] != 0u) {
        const ZU q = zu_pairs(c);
        b = ZU{fminf(b.z, q.z), fminf(b.u, q.u)};
    }
    c->path = p.hist && orders_suffice(b) ? PATH_HIST : PATH_STORED;
    c->z = b.z;
    c->u = b.u;
    c->even = even_orders(b.z, b.u);
}

}  // namespace gabp
