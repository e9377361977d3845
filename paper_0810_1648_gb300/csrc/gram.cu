// The node sums of the final pass (residual r = 1 - Q mu and the dual objective
// from Q alpha; the tiles' parts come from sweep_hist.cu and gram_tc32.cu), Q read
// back, and decision values of callers without a handle (gabp_decision_noalloc):
// SIMT FP32 Gram tiles by FMAs, K-chunks of 16 double-buffered in shared memory, with
// an epilogue on the values that a thread holds: d^2 = max(0, s_i + s_j - 2 G), K =
// expf(-gamma d^2) + lambda^2.  The distances use the norm expansion with norms of
// the same FP32 rows, so d^2_ii is 0 up to rounding and is clamped at 0.  (Staging, Q
// tiles and decisions of a handle: gram_tc32.cu.)
#include "common.cuh"
#include "gabp_svm.h"
#include "ptx.cuh"

#include <float.h>
#include <mutex>
#include <string>

namespace gabp {

namespace {

constexpr int KC = 16;

// RBF entry from a Gram value (norm expansion, clamped distance).
__device__ __forceinline__ float rbf_from_gram(float g, float si, float sj, float gamma)
{
    const float d2 = fmaxf(0.f, si + sj - 2.f * g);
    return expf(-gamma * d2);
}

// Sums over the 16 tx-lanes that share a row (lanes differ in bits 0..3).
__device__ __forceinline__ float sum16(float v)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of FP32 values to more than FP64's bits without the FP64 pipe, which on
// this chip adds about two values a clock and SM: two error-free additions
// (Knuth) leave the rounding of a rounding error to the third word.  n = 100000
// (782 slots a node): 0.60 ms in FP64 additions, now 0.12.
struct Sum3 {
    float s = 0.f, e = 0.f, d = 0.f;
    __device__ __forceinline__ static float two_sum(float& a, float x)
    {
        const float t = a + x, b = t - a;
        const float err = (a - (t - b)) + (x - b);
        a = t;
        return err;
    }
    __device__ __forceinline__ void add(float x) { d += two_sum(e, two_sum(s, x)); }
    __device__ __forceinline__ double value() const { return isfinite(s) ? (double)s + ((double)e + (double)d) : (double)s; }
};

// Per node of a listed node block: r_i = b0_i - Q_ii mu_i - sum part0,
// (Q alpha)_i = Q_ii alpha_i + sum part1; writes alpha (and r in FP32 when
// requested); block partials {max |r_i|, sum b0_i alpha_i - 1/2 alpha_i
// (Q alpha)_i, #SV} into the instance's block buffer.  SVM: b0 = 1, alpha =
// clip(mu, 0, C), SV where alpha_i > threshold; KRR: b0 = the targets, alpha =
// mu, counted where |alpha_i| > threshold.
__global__ void __launch_bounds__(256) k_final_nodes(const Inst* __restrict__ tab,
                                                     const StopOp* __restrict__ ops,
                                                     const int2* __restrict__ nbl)
{
    const int2 nb = nbl[blockIdx.x];
    const Inst& p = tab[nb.x];
    const StopOp& op = ops[nb.x];
    const float* __restrict__ mu = op.mu;
    const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
    const int x = nb.y * 32 + lane, n = p.n;
    Sum3 s0, s1;
    if (x < n) {
        // the node's slots (see slot_begin)
        const int X = x / T, ns = slot_count(p, X);
        const float* p0 = p.part + 2 * part_len(p) + (size_t)slot_begin(p, X) * T + (x - X * T);
        const float* p1 = p0 + part_len(p);
#pragma unroll 4
        for (int k = g; k < ns; k += 8) {
            s0.add(p0[(size_t)k * T]);
            s1.add(p1[(size_t)k * T]);
        }
    }
    __shared__ double red[2][8][32];
    red[0][g][lane] = s0.value();
    red[1][g][lane] = s1.value();
    __syncthreads();
    if (g == 0) {
        double absr = 0.0, obj = 0.0, nsv = 0.0;
        if (x < n) {
            double a0 = 0.0, a1 = 0.0;
            for (int w = 0; w < 8; ++w) { a0 += red[0][w][lane]; a1 += red[1][w][lane]; }
            const double qd = p.qdiag[x], m = mu[x], bx = p.b0[x];
            const float af = p.task ? mu[x] : fminf(fmaxf(mu[x], 0.f), p.C);
            const double al = af;
            op.alpha[x] = af;
            const double r = bx - qd * m - a0;   // residual of the system Q mu = b0
            if (op.r_out) op.r_out[x] = (float)r;
            absr = fabs(r);
            if (!(absr <= DBL_MAX)) absr = INFINITY;
            const double qa = qd * al + a1;
            obj = bx * al - 0.5 * al * qa;
            nsv = (p.task ? fabsf(af) : af) > op.sv_threshold ? 1.0 : 0.0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            absr = fmax(absr, __shfl_xor_sync(0xffffffffu, absr, o));
            obj += __shfl_xor_sync(0xffffffffu, obj, o);
            nsv += __shfl_xor_sync(0xffffffffu, nsv, o);
        }
        if (lane == 0) {
            op.blockbuf[3 * nb.y + 0] = absr;
            op.blockbuf[3 * nb.y + 1] = obj;
            op.blockbuf[3 * nb.y + 2] = nsv;
        }
    }
}

// One CTA per listed instance: fixed-order reduction of its block partials
// -> final3 = {||r||_inf, objective, #SV}, also copied to f3_all[3 * slot].
__global__ void k_final_reduce(const Inst* __restrict__ tab, const StopOp* __restrict__ ops,
                               const int* __restrict__ members, double* __restrict__ f3_all)
{
    __shared__ double s[3][256];
    const int slot = members[blockIdx.x];
    const StopOp& op = ops[slot];
    const int nb = (tab[slot].n + 31) / 32;
    const int tid = threadIdx.x;
    double m = 0.0, o = 0.0, c = 0.0;
    for (int k = tid; k < nb; k += 256) {
        m = fmax(m, op.blockbuf[3 * k]);
        o += op.blockbuf[3 * k + 1];
        c += op.blockbuf[3 * k + 2];
    }
    s[0][tid] = m; s[1][tid] = o; s[2][tid] = c;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (tid < w) {
            s[0][tid] = fmax(s[0][tid], s[0][tid + w]);
            s[1][tid] += s[1][tid + w];
            s[2][tid] += s[2][tid + w];
        }
        __syncthreads();
    }
    if (tid == 0) {
        // tile sums that a bounded wait left out: no residual to go by
        if (tab[slot].ctrl->status == ST_ETIMEOUT) s[0][0] = INFINITY;
        for (int q = 0; q < 3; ++q) {
            op.final3[q] = s[q][0];
            if (f3_all) f3_all[3 * slot + q] = s[q][0];
        }
    }
}

// ---------------------------------------------------------------- inspection
__global__ void k_get_q(Inst p, const int4* __restrict__ work, int q_bf16, float* __restrict__ Qd)
{
    const long long L = work[blockIdx.x].w;
    const int I = work[blockIdx.x].y, J = work[blockIdx.x].z, n = p.n;
    for (int e = threadIdx.x; e < TT; e += blockDim.x) {
        const int r = e / T, c = e % T, i = I * T + r, j = J * T + c;
        if (i >= n || j >= n || (I == J && c <= r)) continue;
        const size_t o = (size_t)L * TT + e;
        const float q = q_bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(p.qstore)[o])
                               : static_cast<const float*>(p.qstore)[o];
        Qd[(size_t)i * n + j] = q;
        Qd[(size_t)j * n + i] = q;
    }
    if (I == J)
        for (int r = threadIdx.x; r < T; r += blockDim.x) {
            const int i = I * T + r;
            if (i < n) Qd[(size_t)i * n + i] = p.qdiag[i];
        }
}

}  // namespace

void launch_final(const Inst* tab, const StopOp* ops, const int4* tiles, long long ntiles, const int2* nbl,
                  int nblocks, const int* members, int nmembers, double* f3_all, int q_stored, cudaStream_t s)
{
    if (ntiles > 0) {
        if (q_stored)
            launch_final_tiles_q(tab, ops, tiles, ntiles, s);
        else
            (void)launch_final_tiles_gram(tab, ops, tiles, ntiles, s);   // errors surface at the caller's cudaGetLastError
    }
    if (nblocks > 0) k_final_nodes<<<nblocks, 256, 0, s>>>(tab, ops, nbl);
    if (nmembers > 0) k_final_reduce<<<nmembers, 256, 0, s>>>(tab, ops, members, f3_all);
}

void launch_get_q(const Inst& p, const int4* work, long long ntiles, int q_bf16, float* Qdense,
                  cudaStream_t s)
{
    k_get_q<<<(unsigned)ntiles, 256, 0, s>>>(p, work, q_bf16, Qdense);
}

}  // namespace gabp

// ---------------------------------------------------------------------------
// Decision values with no device allocation.
//
// Some callers cannot call cudaMalloc: plugins inside a host framework that
// owns all device memory through its own allocator, and latency-critical
// loops that cannot afford the implicit device-wide synchronisation of
// cudaMalloc/cudaFree.  gabp_decision_noalloc serves them:
// the caller passes every input and output as device memory, and the
// per-tile partial sums live in the file-scope array below, which every GPU that
// loads this library holds until the process exits.
namespace gabp {
namespace {

constexpr long long kNoAllocScratchFloats = 1LL << 20;   // 4 MiB

static __device__ __align__(256) float g_noalloc_scratch[kNoAllocScratchFloats];

// Partial decision values of a tile of 16 R test rows x 16 R training rows (I, J
// by the block index): f over the tile's training rows -> part[J t + s].  The
// squared norms come from the rows as the tile goes through them (one thread a
// row, features in order).
//
// What bounds it, on the few rows it is called with, is latency: so the norms
// have no launch of their own, and the tiles are small (64 x 64) until there are
// enough of 128 x 128, with half the operand loads, to fill the chip.  t = 64,
// n = 2000, m = 32: norms (two launches), 128 x 128 tiles and their sum took
// 24.0 us; now 11.2 (the call: 48 -> 32).
template <int R>
__global__ void __launch_bounds__(NTHREADS) k_decision_tiles_noalloc(
    const float* __restrict__ X, const float* __restrict__ y, const float* __restrict__ alpha, int n, int m,
    const float* __restrict__ Xt, int t, float gamma, float lam2, int NJ, float* __restrict__ part)
{
    constexpr int B = 16 * R, LD = B * KC / NTHREADS;
    struct Stage { float A[KC][B + 4], B_[KC][B + 4]; };
    __shared__ __align__(16) Stage sm[2];
    __shared__ float norm[2][B];
    chain_next();
    const long long L = blockIdx.x;
    const int s0 = (int)(L / NJ) * B, j0 = (int)(L % NJ) * B, J = (int)(L % NJ);
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    float acc[R][R];
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int b = 0; b < R; ++b) acc[a][b] = 0.f;
    float ra[LD], rb[LD];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < LD; ++u) {
            const int e = tid + NTHREADS * u, row = e / KC, k = k0 + e % KC;
            ra[u] = s0 + row < t && k < m ? Xt[(size_t)(s0 + row) * m + k] : 0.f;
            rb[u] = j0 + row < n && k < m ? X[(size_t)(j0 + row) * m + k] : 0.f;
        }
    };
    auto store = [&](Stage& st) {
#pragma unroll
        for (int u = 0; u < LD; ++u) {
            const int e = tid + NTHREADS * u, row = e / KC, kk = e % KC;
            st.A[kk][row] = ra[u];
            st.B_[kk][row] = rb[u];
        }
    };
    float wj[R];
#pragma unroll
    for (int b = 0; b < R; ++b) {
        const int j = j0 + tx * R + b;
        wj[b] = j < n ? alpha[j] * y[j] : 0.f;
    }
    const int nch = (m + KC - 1) / KC;
    float sq = 0.f;
    load(0);
    store(sm[0]);
    __syncthreads();
    for (int c = 0; c < nch; ++c) {
        const Stage& st = sm[c & 1];
        if (c + 1 < nch) load((c + 1) * KC);
#pragma unroll
        for (int kk = 0; kk < KC; ++kk) {
            float av[R], bv[R];
#pragma unroll
            for (int u = 0; u < R; u += 4) {
                *reinterpret_cast<float4*>(av + u) = *reinterpret_cast<const float4*>(&st.A[kk][ty * R + u]);
                *reinterpret_cast<float4*>(bv + u) = *reinterpret_cast<const float4*>(&st.B_[kk][tx * R + u]);
            }
#pragma unroll
            for (int a = 0; a < R; ++a)
#pragma unroll
                for (int b = 0; b < R; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
        }
        if (tid < 2 * B) {
            const float (*v)[B + 4] = tid < B ? st.A : st.B_;
#pragma unroll
            for (int kk = 0; kk < KC; ++kk) sq = fmaf(v[kk][tid & (B - 1)], v[kk][tid & (B - 1)], sq);
        }
        if (c + 1 < nch) store(sm[(c + 1) & 1]);
        __syncthreads();
    }
    if (tid < 2 * B) norm[tid / B][tid & (B - 1)] = sq;
    __syncthreads();
    float sj[R];
#pragma unroll
    for (int b = 0; b < R; ++b) sj[b] = norm[1][tx * R + b];
#pragma unroll
    for (int a = 0; a < R; ++a) {
        const int r = ty * R + a;
        const float si = norm[0][r];
        float f = 0.f;
#pragma unroll
        for (int b = 0; b < R; ++b) f = fmaf(wj[b], rbf_from_gram(acc[a][b], si, sj[b], gamma) + lam2, f);
        f = sum16(f);
        if (tx == 0 && s0 + r < t) part[(size_t)J * t + s0 + r] = f;
    }
}

__global__ void k_decision_sum(const float* __restrict__ part, int t, int NJ, float* __restrict__ out)
{
    chain_wait();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= t) return;
    double f = 0.0;
#pragma unroll 8
    for (int k = 0; k < NJ; ++k) f += (double)part[(size_t)k * t + s];
    out[s] = (float)f;
}

template <int R>
void launch_decision_noalloc(const float* X, const float* y, const float* alpha, int n, int m, const float* Xt, int t,
                             float gamma, float lam2, float* part, float* out, cudaStream_t s)
{
    constexpr int B = 16 * R;
    const int NI = (t + B - 1) / B, NJ = (n + B - 1) / B;
    k_decision_tiles_noalloc<R><<<(unsigned)((long long)NI * NJ), NTHREADS, 0, s>>>(X, y, alpha, n, m, Xt, t, gamma, lam2,
                                                                                    NJ, part);
    launch_chained(true, k_decision_sum, (t + 127) / 128, 128, 0, s, (const float*)part, t, NJ, out);
}

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
float* g_noalloc_dev_ptr[kMaxDevices] = {};

}  // namespace
}  // namespace gabp

extern "C" GABP_API gabp_status gabp_decision_noalloc(const float* X, const float* y, const float* alpha,
                                                      int64_t n, int64_t m, const float* Xtest, int64_t t,
                                                      double gamma, double lambda, float* out, void* stream)
{
    using namespace gabp;
    set_last_error("");
    auto fail = [](gabp_status st, const std::string& msg) { set_last_error(msg.c_str()); return st; };
    if (!X || !y || !alpha || (t > 0 && (!Xtest || !out)))
        return fail(GABP_EINVAL, "gabp_decision_noalloc: null pointer");
    if (n < 1 || m < 1 || t < 0 || n > (1LL << 30) || m > (1LL << 20) || t > (1LL << 30))
        return fail(GABP_EINVAL, "gabp_decision_noalloc: bad sizes");
    if (!(gamma > 0) || !(lambda >= 0)) return fail(GABP_EINVAL, "gabp_decision_noalloc: need gamma > 0, lambda >= 0");
    if (t == 0) return GABP_OK;
    const long long Nt = (n + T - 1) / T, Ntt = (t + T - 1) / T;
    const long long need = n + t + Nt * t;
    if (need > kNoAllocScratchFloats)
        return fail(GABP_EINVAL, "gabp_decision_noalloc: n + t + ceil(n/128)*t = " + std::to_string(need) +
                                     " floats of scratch exceeds the fixed maximum of " +
                                     std::to_string(kNoAllocScratchFloats) + "; split the test rows");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(GABP_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return fail(GABP_ECUDA, "gabp_decision_noalloc: device index out of range");
    float* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_dev_ptr[dev]) {
            // Once per device, with that device current: the device address of the
            // array (its name in host code is only a host-side stand-in).
            void* ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
            if (e != cudaSuccess)
                return fail(GABP_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            g_noalloc_dev_ptr[dev] = static_cast<float*>(ptr);
        }
        scratch = g_noalloc_dev_ptr[dev];
    }
    // Every scratch element read below is written earlier in the same call.  64 x
    // 64 tiles (up to where 128 x 128 ones fill the chip, see
    // k_decision_tiles_noalloc) take ceil(n / 64) t floats of it; the limit above,
    // which counts n + t floats more than 128 x 128 tiles need, is what callers
    // know.
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (Ntt * Nt < num_sms() && (n + 63) / 64 * t <= kNoAllocScratchFloats)
        launch_decision_noalloc<4>(X, y, alpha, (int)n, (int)m, Xtest, (int)t, (float)gamma, (float)(lambda * lambda),
                                   scratch, out, s);
    else
        launch_decision_noalloc<8>(X, y, alpha, (int)n, (int)m, Xtest, (int)t, (float)gamma, (float)(lambda * lambda),
                                   scratch, out, s);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(GABP_ECUDA, std::string("gabp_decision_noalloc: ") + cudaGetErrorString(e));
    return GABP_OK;
}
