// FP32-accurate Gram tiles on the 5th-generation tensor cores (tcgen05),
// fused with the RBF kernel, labels and bias: the FP32 Q tiles of the plain
// form, the FP32 copy the BF16 store keeps for its refinement residuals, and
// the |Q| row sums that set the weighted diagonal (Section 5 computes the
// kernel matrix once; Section 3.1 weights the diagonal by those sums;
// Section 1.1 defines D_ij = y_i y_j K(x_i, x_j)).
//
// Three BF16 planes.  Every FP32 feature is split as x = x1 + x2 + x3 with
// x1 = bf16(x), x2 = bf16(x - x1), x3 = bf16(x - x1 - x2) (both differences
// are exact in FP32), so x1 + x2 + x3 carries x to about 2^-27 of its size.
// The dot product keeps the six plane products with a + b <= 4,
//   x.y ~ x1.y3 + x2.y2 + x3.y1 + x1.y2 + x2.y1 + x1.y1,
// issued smallest first; the dropped ones are below 2^-26 of |x||y|.  The
// tensor cores multiply BF16 exactly; their FP32 accumulation drops low bits
// (toward zero), so each 64-feature chunk gets a fresh accumulator and the
// chunks are added on the CUDA cores (round to nearest).  The squared norms in
// d^2 = ||x_i||^2 + ||x_j||^2 - 2 x_i.x_j come from the same products (the
// diagonal of the diagonal tiles, a first pass): for near pairs, where K is
// large, the norms and the Gram value then carry the same truncation, which
// cancels in d^2 instead of shrinking every K by ~2 gamma ||x||^2 x 1e-8.
//
// k_gram_tc32 is persistent with warp roles: warp 0 streams the operand blocks
// of each (tile, chunk), two copies of three planes, into a two-stage
// shared-memory ring; warp 1 allocates 512 TMEM columns (four 128 x 128 FP32
// accumulators, one per K-step) and one thread issues the 24 MMAs of a chunk (6
// products x K = 64 in steps of 16); warp 2 prepares what the epilogue does next
// (T3Item and the labels, norms and means); warps 3-18 (four per TMEM lane
// quarter, one per 32 columns) add each chunk's accumulators into registers and
// run the epilogue of the mode:
//   formation   Q entries (norm expansion, clamp, expf, bias, labels), stored,
//               and |Q| over rows, over columns (in registers, then in shared
//               memory) and the tile maximum.  Instances
//               chained behind the listed one (the points of a parameter grid
//               over the same features) take their Q tiles from the same Gram
//               sums;
//   final pass  the same entries, not stored, times the means and the weights
//               (instances that recompute Q);
//   decision    entries of test rows against training rows, times the weights,
//               summed over a range of training tiles in registers;
//   pair pass   the largest z and |q| / d over the pairs (k_pair_z of
//               sweep_hist.cu) for instances that recompute Q.  The entries are
//               those that the other forms store, bit for bit, so that all of them
//               choose the same message path.  (From SIMT FP32 tiles, whose sums
//               round otherwise, refits of such handles took 1064 us at n = 6000, m
//               = 784 and 539 at n = 9000, m = 128.)
// Bound by the epilogue's latencies (the FMA pipe is 28 % busy, the LSU
// 14 %): with eight epilogue warps (64 columns each, all four accumulators
// handed over at once) two warps a scheduler left it waiting; with the epilogue
// looking up lists, tables and slots itself, formation took 522 us (n = 20000, m =
// 128) and 162 us (n = 12000, m = 64), now 350 and 104.
#include "common.cuh"
#include "hist.cuh"
#include "ptx.cuh"
#include "qtile_epi.cuh"

#include <float.h>

namespace gabp {

namespace {

constexpr int NPLANE = 3;
constexpr int T3_EPI_WARPS = 16;                     // four per TMEM lane quarter, one per 32 columns
constexpr int T3_CTL_WARPS = 3;                       // operand producer, MMA issuer, item preparer
constexpr int T3_THREADS = (T3_CTL_WARPS + T3_EPI_WARPS) * 32;
constexpr int T3_STAGES = 2;
constexpr size_t T3_STAGE_BYTES = (size_t)2 * NPLANE * BLK_BYTES;   // A planes, then B planes: 96 KB
// Accumulators per 64-feature chunk: one per K-step of 16 features, each
// receiving the step's five small products first and its x1.y1 product last,
// so that no x1.y1 partial sum passes through a truncating tensor-core
// addition; the chunk value is their sum on the CUDA cores (round to
// nearest).  Measured against the FP64 oracle (n = 2048, with the norms from
// the same products): mean relative error of K -2e-8 with four accumulators
// against +1.2e-6 with one (clustered data, gamma ||x||^2 ~ 24), +1.2e-7
// against +2.6e-7 (m = 128).  Each accumulator is handed over by itself, so the
// MMAs of the next chunk's first K-step run while the epilogue still reads the
// last ones.
constexpr int T3_NACC = KCH / 16;
constexpr uint32_t T3_TMEM_COLS = T3_NACC * T;
static_assert(T3_TMEM_COLS == 512, "all of TMEM");
constexpr uint32_t T3_IDESC = idesc_bf16_f32(T, T);
constexpr int T3_PRODUCTS = 6;

// Plane pairs (a, b) of the kept products, smallest first.
__device__ __forceinline__ int prod_a(int q) { return q == 0 ? 0 : q == 1 ? 1 : q == 2 ? 2 : q == 3 ? 0 : q == 4 ? 1 : 0; }
__device__ __forceinline__ int prod_b(int q) { return q == 0 ? 2 : q == 1 ? 1 : q == 2 ? 0 : q == 3 ? 1 : q == 4 ? 0 : 0; }

// The three BF16 planes of x.
__device__ __forceinline__ void split3(float x, __nv_bfloat16& b1, __nv_bfloat16& b2, __nv_bfloat16& b3)
{
    b1 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(b1);
    b2 = __float2bfloat16_rn(r1);
    const float r2 = r1 - __bfloat162float(b2);
    b3 = __float2bfloat16_rn(r2);
}

// Offset (in 16-byte units) of row rr's 8-feature group kg inside a packed
// 128 x 64 block: 8-row x 16-byte core matrices, K-adjacent ones 128 bytes
// apart, 8-row groups 1024 bytes apart (the canonical K-major layout).
__device__ __forceinline__ size_t core_off16(int rr, int kg)
{
    return (size_t)((rr / 8) * (KCH / 8) + kg) * 8 + (rr % 8);
}

// ---------------------------------------------------------------- staging
// Inputs to what the kernels read, in one pass: the FP32 rows (FP64 rounds,
// BF16 widens exactly) where a copy is kept, their three BF16 planes, the
// finiteness and label checks, the right-hand sides.
//
// What bounds it: 4 bytes read and 6 to 10 written per feature.  A thread takes 8
// features of a row (32 bytes of FP32, one 16-byte unit of each plane); 8
// consecutive threads take the 8 rows of a core matrix (row_position), so that
// they write its 128 bytes, and a warp reads 128 consecutive bytes of each row.
// With one thread a row for the checks and norms and a second pass for the
// planes: 107 + 14 us at n = 6238, m = 617; 40 + 10 us at n = 20000, m = 128;
// now 22 and 10 us.

// 8 consecutive features, in 16-byte loads where the rows are aligned to them.
template <class XT>
__device__ __forceinline__ void load8(const XT* __restrict__ x, float (&v)[8])
{
    constexpr int W = 16 / sizeof(XT);
#pragma unroll
    for (int u = 0; u < 8; u += W) {
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(x + u));
        XT e[W];
        memcpy(e, &q, 16);
#pragma unroll
        for (int t = 0; t < W; ++t) v[u + t] = (float)e[t];
    }
}

__device__ __forceinline__ bool rows_aligned(const void* X, size_t row_bytes)
{
    return ((reinterpret_cast<uintptr_t>(X) | row_bytes) & 15) == 0;
}

// Operand position of a row within its block: the rows 8 q + 2 j + b of each 32 (q,
// j < 4, b < 2) lie at 8 j + 2 q + b, so that the lane of the epilogue that holds
// positions 8 j + 2 q + {0, 1}, j = 0..3, of a tile row has eight consecutive
// columns, which it stores as 32 bytes.  Its own inverse is the same with q and j
// exchanged.
__host__ __device__ __forceinline__ int row_position(int r)
{
    return (r & ~31) | (r >> 1 & 3) << 3 | (r >> 3 & 3) << 1 | (r & 1);
}

// Row r (of Nt*T, zero beyond n) and 8-feature group gk -> Xf where it is kept
// and the three planes' blocks ((I nkc + kc) 3 + plane); false where a feature is
// not finite.
template <class XT>
__device__ __forceinline__ bool stage_group(const XT* __restrict__ X, bool vec, int n, int m, int nkc, int r, int gk,
                                            float* __restrict__ Xf, bool vecf, uint4* __restrict__ Xp3)
{
    const int kc = gk / (KCH / 8), kg = gk % (KCH / 8), k0 = gk * 8;
    const int I = r / T, rr = r % T;
    float x[8];
    bool ok = true;
    if (r < n && vec && k0 + 8 <= m) {
        load8(X + (size_t)r * m + k0, x);
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = r < n && k0 + u < m ? (float)X[(size_t)r * m + k0 + u] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) ok &= isfinite(x[u]);
    if (Xf && r < n) {
        float* d = Xf + (size_t)r * m + k0;
        if (vecf && k0 + 8 <= m) {
            reinterpret_cast<float4*>(d)[0] = make_float4(x[0], x[1], x[2], x[3]);
            reinterpret_cast<float4*>(d)[1] = make_float4(x[4], x[5], x[6], x[7]);
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k0 + u < m) d[u] = x[u];
        }
    }
    __align__(16) __nv_bfloat16 v[NPLANE][8];
#pragma unroll
    for (int u = 0; u < 8; ++u) split3(x[u], v[0][u], v[1][u], v[2][u]);
#pragma unroll
    for (int pl = 0; pl < NPLANE; ++pl) {
        const size_t blk = ((size_t)I * nkc + kc) * NPLANE + pl;
        Xp3[blk * (BLK_BYTES / 16) + core_off16(row_position(rr), kg)] = *reinterpret_cast<const uint4*>(v[pl]);
    }
    return ok;
}

// Row i's label (SVM: +-1, b = b0 = 1: the linear term 1'h of the dual) or
// target (KRR: (K + lambda_r I) c = y; the target moves to b and b0, the label
// becomes 1); false where it is not valid.
__device__ __forceinline__ bool stage_label(float* __restrict__ y, float* __restrict__ b, float* __restrict__ b0, int i,
                                            int task)
{
    const float yi = y[i];
    const float rhs = task ? yi : 1.f;
    if (task) y[i] = 1.f;
    b[i] = rhs;
    b0[i] = rhs;
    return task ? isfinite(yi) : yi == 1.f || yi == -1.f;
}

// Row (of 8 in consecutive operand positions) and group of thread e of a pass
// over whole rows.
__device__ __forceinline__ void stage_item(long long e, int groups, int& r, int& gk)
{
    const long long q = e >> 3;
    gk = (int)(q % groups);
    r = row_position((int)(q / groups) * 8 + (int)(e & 7));
}

// A caller's rows (FP32, FP64 or BF16).  Xf: where the FP32 rows are kept (null:
// nowhere, or X itself); y, b, b0: labels, null for test rows; diag: where the
// diagonal tile list goes, or null.  Errors go to check->status, bad_index =
// the first found row + row0.
template <class XT>
__global__ void k_stage_rows(const XT* __restrict__ X, int n, int m, int nkc, int Nt, float* __restrict__ Xf,
                             float* __restrict__ y, float* __restrict__ b, float* __restrict__ b0, int task,
                             uint4* __restrict__ Xp3, long long row0, Ctrl* __restrict__ check, int4* __restrict__ diag)
{
    const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int groups = nkc * (KCH / 8);
    if (diag && e < Nt) diag[e] = make_int4(0, (int)e, (int)e, (int)e);
    if (e >= (long long)Nt * T * groups) return;
    int r, gk;
    stage_item(e, groups, r, gk);
    bool ok = stage_group(X, rows_aligned(X, (size_t)m * sizeof(XT)), n, m, nkc, r, gk, Xf,
                          rows_aligned(Xf, (size_t)m * sizeof(float)), Xp3);
    if (y && gk == 0 && r < n) ok &= stage_label(y, b, b0, r, task);
    if (!ok && atomicCAS(&check->status, 0, (int)ST_EINVAL) == 0) check->bad_index = row0 + r;
}

// Listed node blocks (32 rows) of instances whose FP32 rows already sit in
// their X; the last block of an instance also writes the zero rows that pad its
// last tile.
__global__ void __launch_bounds__(256) k_stage_list(const Inst* __restrict__ tab, const int2* __restrict__ nbl)
{
    const int2 nb = nbl[blockIdx.x];
    const Inst& p = tab[nb.x];
    const int n = p.n, m = p.m, nkc = p.nkc, groups = nkc * (KCH / 8);
    const int rows = nb.y == (n - 1) / 32 ? p.Nt * T - nb.y * 32 : 32;
    const bool vec = rows_aligned(p.X, (size_t)m * sizeof(float));
    uint4* Xp3 = static_cast<uint4*>(const_cast<void*>(p.Xp3));
    for (int e = threadIdx.x; e < rows * groups; e += blockDim.x) {
        int r, gk;
        stage_item(e, groups, r, gk);
        r += nb.y * 32;
        bool ok = stage_group(p.X, vec, n, m, nkc, r, gk, nullptr, false, Xp3);
        if (gk == 0 && r < n)
            ok &= stage_label(const_cast<float*>(p.y), const_cast<float*>(p.b), const_cast<float*>(p.b0), r, p.task);
        if (!ok && atomicCAS(&p.ctrl->status, 0, (int)ST_EINVAL) == 0) p.ctrl->bad_index = r;
    }
}

// What the epilogue makes of the Gram tiles.
enum T3Mode {
    T3_FORM,     // Q tiles, |Q| sums (and, norms_only, the squared norms)
    T3_FINAL,    // sums q mu and q alpha of a tile's pairs, Q not stored
    T3_PAIRZ,    // the largest z and |q| / d of a tile's pairs, Q not stored (norms_only: one instance)
    T3_DECIDE    // decision values: rows = test rows, sums over the training columns
};

// The sums of a tile's epilogue (two in turn).
struct T3Sums {
    float col[2][4][T];     // per lane quarter: column sums over its 32 rows
    float row[2][4][T];     // per 32-column group: row sums
    float tmx[T3_EPI_WARPS];
};

// The columns' ([0]) and rows' ([1]) constants of an item (two in turn): label
// sign, norm and, in the final pass, mean and alpha; in a decision mu[0] holds
// the columns' weights y alpha.
struct T3Const {
    alignas(16) float y[2][T];
    float sq[2][T];
    float mu[2][T];
    float al[2][T];
};

// What the epilogue does next: a tile, or one of the instances that share its
// Gram.  One warp prepares it, with the constants, while the epilogue computes
// the item before (two in turn): looked up by the epilogue itself, work lists,
// instance tables and slots were a third of its time.
struct T3Item {
    int nkc;                 // chunks of accumulators to take in first; 0: the Gram at hand
    int end, diag, last;     // no item; a diagonal tile; decision: the entry's last tile, pair pass: to be looked at
    int rows, cols;          // rows and columns that there are (may exceed T)
    float gamma, lam2;
    float* store;            // where the entries go, or null
    float* tilemax;          // where the largest |q| goes, or null
    float* dst[2];           // the row's and the column's slot sums (FINAL: of q mu; those of q alpha plen behind)
    unsigned long long* fix[2];   // where set, fixed-point sums instead of slots
    int shift;
    long long plen;
    int4 w;                  // norms_only: the work entry
    Ctrl* ctrl;
};

struct T3Smem {
    unsigned long long xfull[T3_STAGES], xempty[T3_STAGES];
    unsigned long long accfull[T3_NACC], accempty[T3_NACC];
    unsigned long long drain;
    uint32_t tmem_base;
    int abort;
    T3Sums sums[2];
    T3Const cst[2];
    T3Item item[2];
    unsigned long long ifull[2], iempty[2], sync;
};


// ---- epilogue
// A warp has 32 rows (its lane quarter of TMEM) x 32 columns of the tile, in
// the layout of 16 x 256-bit loads: lane (lr = lane / 4, lq = lane % 4) holds
// positions 8 k + lr, k = 0..3, of the rows and 8 j + 2 lq and the next, j = 0..3,
// as pairs, of the columns: rows 8 (lr / 2) + 2 k + lr % 2 and columns 8 lq + 2 j and
// the next (row_position).  Four rows and eight columns a lane leave little to
// reduce across lanes (ten shuffles for the tile's row and column sums, where
// one row of 32 columns a lane took 31), the pairs go through two-wide arithmetic,
// and a row's eight entries are stored at once (in pairs, 8 bytes a lane, the
// stores took 11 passes each: 424 us against 350 at n = 20000, m = 128).
struct Frag {
    float2 v[4][4];   // [k][j]
};
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, Frag& f)
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
            "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(taddr + ((uint32_t)(16 * h) << 16))
            : "memory");
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 2; ++k)
                f.v[2 * h + k][j] = make_float2(__uint_as_float(r[4 * j + 2 * k]), __uint_as_float(r[4 * j + 2 * k + 1]));
    }
}

// exp(-gamma d2) + lam2 of two entries, d2 = max(0, si + sj - 2 g).
struct Rbf {
    float ngam, lam2;
};
__device__ __forceinline__ Rbf rbf_of(float gamma, float lam2) { return Rbf{-gamma, lam2}; }
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 rbf2(const Rbf& b, float2 g, float si, float2 sj)
{
    const float2 d = __ffma2_rn(f2(-2.f), g, __fadd2_rn(f2(si), sj));
    const float2 t = __fmul2_rn(f2(b.ngam), make_float2(fmaxf(0.f, d.x), fmaxf(0.f, d.y)));
    return __fadd2_rn(make_float2(expf(t.x), expf(t.y)), f2(b.lam2));
}
__device__ __forceinline__ float2 flip(float2 v, uint32_t sx, uint32_t sy)
{
    return make_float2(__uint_as_float(__float_as_uint(v.x) ^ sx), __uint_as_float(__float_as_uint(v.y) ^ sy));
}
__device__ __forceinline__ float2 ld2(const float* x) { return *reinterpret_cast<const float2*>(x); }

// Sums over the four lanes of a row: lane lq has that of value lq.
__device__ __forceinline__ float row_sums4(const float2 (&x)[4], int lane)
{
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = x[k].x + x[k].y;
    const bool b2 = (lane & 2) != 0, b1 = (lane & 1) != 0;
    float y[2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
        y[k] = (b2 ? v[k + 2] : v[k]) + __shfl_xor_sync(0xffffffffu, b2 ? v[k] : v[k + 2], 2);
    return (b1 ? y[1] : y[0]) + __shfl_xor_sync(0xffffffffu, b1 ? y[0] : y[1], 1);
}
// Sums over the eight lanes that share columns: lane lr has that of value lr of
// {x[0].x, x[0].y, x[1].x, ...}, column 8 lq + lr.
__device__ __forceinline__ float col_sums8(const float2 (&x)[4], int lane)
{
    const bool b16 = (lane & 16) != 0, b8 = (lane & 8) != 0, b4 = (lane & 4) != 0;
    float2 y[2], z;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float2 keep = b16 ? x[k + 2] : x[k], send = b16 ? x[k] : x[k + 2];
        y[k].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 16);
        y[k].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 16);
    }
    const float2 keep = b8 ? y[1] : y[0], send = b8 ? y[0] : y[1];
    z.x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, 8);
    z.y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, 8);
    return (b4 ? z.y : z.x) + __shfl_xor_sync(0xffffffffu, b4 ? z.x : z.y, 4);
}

// Running compensated sum s + c (+ e) += x + xc.
__device__ __forceinline__ void add_pair(float& s, float& c, float x, float xc)
{
    const float t = s + x, bp = t - s;
    c += (s - (t - bp)) + (x - bp) + xc;
    s = t;
}


// The decision's operands: tab[0] describes the test rows as an instance (n,
// Nt, nkc, Xp3, sq3), tab[1] is the training set; a work entry {0, I, J0, J1}
// sums test tile I over the training tiles [J0, J1).
struct DecideArgs {
    const float* alpha;
    float* part;      // [entries][T]
};

template <int MODE>
__global__ void __launch_bounds__(T3_THREADS, 1)
    k_gram_tc32(const Inst* __restrict__ tab, const int4* __restrict__ work, long long ntiles, int norms_only,
                const StopOp* __restrict__ ops, DecideArgs dec)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* oper = align_smem(smem_raw, 1024);
    T3Smem& sm = *reinterpret_cast<T3Smem*>(oper + T3_STAGES * T3_STAGE_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // (what pair_z_asks reads is fixed by now: every role finds the same)
    if (MODE == T3_PAIRZ && norms_only && !pair_z_asks(tab[0])) return;
    auto skipped = [&](int4 w) {
        if constexpr (MODE == T3_PAIRZ) {
            bool none = !norms_only;
            for (int k = none ? w.x : -1; k >= 0 && none; k = tab[k].form_next - 1) none = !pair_z_asks(tab[k]);
            return none;
        } else {
            return false;
        }
    };

    if (tid == 0) {
        for (int s = 0; s < T3_STAGES; ++s) { mbar_init(&sm.xfull[s], 1); mbar_init(&sm.xempty[s], 1); }
        for (int a = 0; a < T3_NACC; ++a) { mbar_init(&sm.accfull[a], 1); mbar_init(&sm.accempty[a], T3_EPI_WARPS); }
        for (int b = 0; b < 2; ++b) { mbar_init(&sm.ifull[b], 1); mbar_init(&sm.iempty[b], T3_EPI_WARPS); }
        mbar_init(&sm.sync, T3_EPI_WARPS);
        mbar_init(&sm.drain, 1);
        sm.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(&sm.tmem_base, T3_TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = sm.tmem_base;
    // (a decision's work entry covers several tiles)
    auto first_j = [&](int4 w) { return w.z; };
    auto last_j = [&](int4 w) { return MODE == T3_DECIDE ? w.w : w.z + 1; };

    if (warp == 0) {
        // ------------------------------------------------ operand producer
        if (lane == 0) {
            const uint64_t pol = l2_evict_last_policy();   // the planes are read again by many tiles
            int stage = 0;
            uint32_t ph = 0;
            bool run = true;
            for (long long L = blockIdx.x; L < ntiles && run; L += gridDim.x) {
                const int4 w = work[L];
                if (skipped(w)) continue;
                const Inst& p = tab[w.x];
                const unsigned char* A3 = static_cast<const unsigned char*>(p.Xp3);
                const unsigned char* B3 = MODE == T3_DECIDE ? static_cast<const unsigned char*>(tab[1].Xp3) : A3;
                const int I = w.y, nkc = p.nkc;
                for (int J = first_j(w); J < last_j(w) && run; ++J)
                    for (int kc = 0; kc < nkc; ++kc) {
                        if (*(volatile int*)&sm.abort || !mbar_wait(&sm.xempty[stage], ph ^ 1u)) {
                            sm.abort = 1;
                            record_error(p.ctrl, ST_ETIMEOUT, L);
                            run = false;
                            break;
                        }
                        unsigned char* S = oper + (size_t)stage * T3_STAGE_BYTES;
                        // a block's three planes lie behind one another
                        mbar_arrive_expect_tx(&sm.xfull[stage], (uint32_t)T3_STAGE_BYTES);
                        bulk_load(S, A3 + ((size_t)I * nkc + kc) * NPLANE * BLK_BYTES, NPLANE * BLK_BYTES, &sm.xfull[stage], pol);
                        bulk_load(S + (size_t)NPLANE * BLK_BYTES, B3 + ((size_t)J * nkc + kc) * NPLANE * BLK_BYTES,
                                  NPLANE * BLK_BYTES, &sm.xfull[stage], pol);
                        if (++stage == T3_STAGES) { stage = 0; ph ^= 1u; }
                    }
            }
            await_copies<T3_STAGES>(sm.xfull, stage, ph);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------ MMA issuer
        if (lane == 0) {
            int stage = 0;
            uint32_t ph = 0, aph = 0;
            bool run = true;
            for (long long L = blockIdx.x; L < ntiles && run; L += gridDim.x) {
                const int4 w = work[L];
                if (skipped(w)) continue;
                const Inst& p = tab[w.x];
                Ctrl* ctrl = p.ctrl;
                const int chunks = p.nkc * (last_j(w) - first_j(w));
                for (int kc = 0; kc < chunks && run; ++kc) {
                    if (*(volatile int*)&sm.abort || !mbar_wait(&sm.xfull[stage], ph)) run = false;
                    const unsigned char* S = oper + (size_t)stage * T3_STAGE_BYTES;
#pragma unroll
                    for (int a = 0; a < T3_NACC; ++a) {
                        if (run && !mbar_wait(&sm.accempty[a], aph ^ 1u)) run = false;
                        if (!run) break;
                        tc_fence_after();
                        const uint32_t d = tbase + (uint32_t)a * T;
#pragma unroll
                        for (int q = 0; q < T3_PRODUCTS; ++q)
                            tc_mma_bf16(d, smem_desc(S + (size_t)prod_a(q) * BLK_BYTES + a * 256, 128, 1024),
                                        smem_desc(S + (size_t)(NPLANE + prod_b(q)) * BLK_BYTES + a * 256, 128, 1024), T3_IDESC,
                                        q != 0 ? 1u : 0u);
                        tc_commit(&sm.accfull[a]);
                    }
                    if (!run) {
                        sm.abort = 1;
                        record_error(ctrl, ST_ETIMEOUT, L);
                        break;
                    }
                    tc_commit(&sm.xempty[stage]);
                    if (++stage == T3_STAGES) { stage = 0; ph ^= 1u; }
                    aph ^= 1u;
                }
            }
            // every MMA issued above must finish before the columns are freed
            tc_commit(&sm.drain);
            if (!mbar_wait(&sm.drain, 0u)) sm.abort = 1;
        }
    } else if (warp == 2) {
        // ----------------------------------------------- items and constants
        const bool consts = MODE != T3_FORM || !norms_only;
        int b = 0;
        uint32_t ph = 0;
        bool run = true;
        int4 wn = blockIdx.x < ntiles ? work[blockIdx.x] : make_int4(0, 0, 0, 0);
        for (long long L = blockIdx.x; L < ntiles && run; L += gridDim.x) {
            const int4 w = wn;
            if (L + gridDim.x < ntiles) wn = work[L + gridDim.x];
            if (skipped(w)) continue;
            const int I = w.y;
            for (int J = first_j(w); J < last_j(w) && run; ++J) {
                for (int k = w.x; k >= 0 && run;) {
                    const Inst& p = tab[k];                              // rows
                    const Inst& cp = MODE == T3_DECIDE ? tab[1] : p;     // columns
                    const int n = p.n, rows = n - I * T, cols = cp.n - J * T;
                    const int next = (MODE == T3_FORM && consts) || MODE == T3_PAIRZ ? p.form_next - 1 : -1;
                    // lane + 32 u of the tile's columns ([0]) and rows ([1])
                    float y[2][4], q[2][4], m[2][4];
                    if (consts) {
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const Inst& o = r ? p : cp;
                            const float* mu = MODE == T3_FINAL ? ops[k].mu : MODE == T3_DECIDE && r == 0 ? dec.alpha : nullptr;
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int x = (r ? I : J) * T + lane + 32 * u;
                                const bool in = x < o.n;
                                y[r][u] = in && MODE != T3_PAIRZ && (MODE != T3_DECIDE || r == 0) ? o.y[x] : 0.f;
                                q[r][u] = in ? o.sq3[x] : 0.f;
                                if (MODE == T3_PAIRZ) m[r][u] = in ? __fdividef(1.f, o.qdiag[x]) : 0.f;
                                else m[r][u] = in && mu ? mu[x] : 0.f;
                            }
                        }
                    }
                    const bool stop = __shfl_sync(0xffffffffu, *(volatile int*)&sm.abort, 0) != 0;
                    if (stop || !mbar_wait_warp(&sm.iempty[b], ph ^ 1u)) {
                        if (lane == 0) {
                            sm.abort = 1;
                            record_error(p.ctrl, ST_ETIMEOUT, L);
                        }
                        run = false;
                        break;
                    }
                    if (consts) {
                        T3Const& c = sm.cst[b];
#pragma unroll
                        for (int r = 0; r < 2; ++r)
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int x = lane + 32 * u;
                                c.sq[r][x] = q[r][u];
                                if (MODE == T3_DECIDE) {
                                    if (r == 0) c.mu[0][x] = m[0][u] * y[0][u];
                                    continue;
                                }
                                if (MODE == T3_PAIRZ) {
                                    c.mu[r][x] = m[r][u];
                                    continue;
                                }
                                c.y[r][x] = __uint_as_float(__float_as_uint(y[r][u]) & 0x80000000u);
                                if (MODE == T3_FINAL) {
                                    c.mu[r][x] = m[r][u];
                                    c.al[r][x] = p.task ? m[r][u] : fminf(fmaxf(m[r][u], 0.f), p.C);
                                }
                            }
                    }
                    if (lane == 0) {
                        T3Item& t = sm.item[b];
                        t.nkc = k == w.x ? p.nkc : 0;
                        t.end = 0;
                        t.diag = MODE != T3_DECIDE && I == J;
                        t.last = MODE == T3_PAIRZ ? pair_z_asks(p) : J + 1 == last_j(w);
                        t.rows = rows;
                        t.cols = cols;
                        t.gamma = cp.gamma;
                        t.lam2 = cp.lam2;
                        t.ctrl = p.ctrl;
                        t.w = w;
                        if (MODE == T3_DECIDE) {
                            t.dst[0] = dec.part + L * T;
                        } else if (consts && MODE != T3_PAIRZ) {
                            const int2 sl = p.rfix ? make_int2(0, 0) : tile_slots(p, w);
                            t.plen = (long long)part_len(p);
                            float* part = p.part + (MODE == T3_FINAL ? 2 * t.plen : 0);
                            t.dst[0] = part + (size_t)sl.x * T;
                            t.dst[1] = part + (size_t)sl.y * T;
                            t.store = MODE == T3_FORM && p.qref ? p.qref + (size_t)w.w * TT : nullptr;
                            t.tilemax = MODE == T3_FORM && p.tilemax ? p.tilemax + w.w : nullptr;
                            t.fix[0] = MODE == T3_FORM && p.rfix ? p.rfix + (size_t)I * T : nullptr;
                            t.fix[1] = MODE == T3_FORM && p.rfix ? p.rfix + (size_t)J * T : nullptr;
                            if (MODE == T3_FORM && p.rfix) t.shift = rsum_shift(n, p.lam2);
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.ifull[b]);
                    if ((b ^= 1) == 0) ph ^= 1u;
                    k = next;
                }
            }
        }
        if (run && mbar_wait_warp(&sm.iempty[b], ph ^ 1u) && lane == 0) {
            sm.item[b].end = 1;
            mbar_arrive(&sm.ifull[b]);
        }
    } else {
        // --------------------------------------------------------- epilogue
        // warp w reads TMEM lanes 32 (w % 4) ..: rows 32 g ..., columns [32 cg, 32 cg + 32)
        const int ew = warp - T3_CTL_WARPS, g = warp & 3, cg = ew >> 2;
        const int lr = lane >> 2, lq = lane & 3, c0 = 32 * cg;
        const int r0 = 32 * g + 8 * (lr >> 1) + (lr & 1), cq = c0 + 8 * lq;   // the lane's first row and column
        const int etid = tid - T3_CTL_WARPS * 32;
        uint32_t aph = 0, iph = 0, sph = 0;
        int b = 0, sb = 0;
        Frag G;
        // decision: the rows' compensated sums over the entry's training tiles
        float fs[4] = {0.f, 0.f, 0.f, 0.f}, fc[4] = {0.f, 0.f, 0.f, 0.f};
        // The epilogue's warps meet (bounded, like every wait): the item's sums are complete.
        auto meet = [&]() {
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.sync);
            const bool ok = mbar_wait_warp(&sm.sync, sph);
            sph ^= 1u;
            return ok;
        };
        bool ok = true;
        for (;;) {
            const bool stop = __shfl_sync(0xffffffffu, *(volatile int*)&sm.abort, 0) != 0;
            if (stop || !mbar_wait_warp(&sm.ifull[b], iph)) { ok = false; break; }
            const T3Item& it = sm.item[b];
            const T3Const& cc = sm.cst[b];
            if (it.end) break;
            const int nkc = it.nkc;
            for (int kc = 0; kc < nkc && ok; ++kc) {
                // the chunk's accumulators added to the running sums in order
#pragma unroll
                for (int a = 0; a < T3_NACC; ++a) {
                    if (!mbar_wait_warp(&sm.accfull[a], aph)) { ok = false; break; }
                    tc_fence_after();
                    Frag V;
                    tmem_ld_frag(tbase + (uint32_t)a * T + ((uint32_t)(32 * g) << 16) + (uint32_t)c0, V);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.accempty[a]);
                    if (kc == 0 && a == 0) {
                        G = V;
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int j = 0; j < 4; ++j) G.v[k][j] = __fadd2_rn(G.v[k][j], V.v[k][j]);
                    }
                }
                aph ^= 1u;
            }
            if (!ok) break;
            T3Sums& su = sm.sums[sb];
            if (MODE == T3_FORM && norms_only) {
                // diagonal tile: x_i . x_i is the Gram value at equal positions, of
                // the lanes with lr = 2 lq or 2 lq + 1
                const int4 w = it.w;
                if (cg == g && (lr >> 1) == lq) {
                    for (int k = w.x; k >= 0; k = tab[k].form_next - 1)
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int x = w.y * T + r0 + 2 * u;
                            if (x < tab[k].n) tab[k].sq3[x] = lr & 1 ? G.v[u][u].y : G.v[u][u].x;
                        }
                }
            } else if (MODE == T3_DECIDE) {
                const Rbf rb = rbf_of(it.gamma, it.lam2);
                float2 f[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 sj = ld2(&cc.sq[0][cq + 2 * j]), wj = ld2(&cc.mu[0][cq + 2 * j]);
#pragma unroll
                    for (int k = 0; k < 4; ++k) f[k] = __ffma2_rn(wj, rbf2(rb, G.v[k][j], cc.sq[1][r0 + 2 * k], sj), f[k]);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) add_pair(fs[k], fc[k], f[k].x + f[k].y, 0.f);
                if (it.last) {
                    // a row's four lanes: lane lq has row r0 + 2 lq
#pragma unroll
                    for (int o = 2; o > 0; o >>= 1) {
                        const bool up = (lane & o) != 0;
#pragma unroll
                        for (int k = 0; k < o; ++k) {
                            const float xs = __shfl_xor_sync(0xffffffffu, up ? fs[k] : fs[k + o], o);
                            const float xc = __shfl_xor_sync(0xffffffffu, up ? fc[k] : fc[k + o], o);
                            if (up) { fs[k] = fs[k + o]; fc[k] = fc[k + o]; }
                            add_pair(fs[k], fc[k], xs, xc);
                        }
                    }
                    su.row[0][cg][r0 + 2 * lq] = fs[0];
                    su.row[1][cg][r0 + 2 * lq] = fc[0];
#pragma unroll
                    for (int k = 0; k < 4; ++k) fs[k] = fc[k] = 0.f;
                    if (!meet()) { ok = false; break; }
                    if (etid < T) {
                        double v = 0.0;
                        for (int c = 0; c < 4; ++c) v += (double)su.row[0][c][etid] + (double)su.row[1][c][etid];
                        it.dst[0][etid] = (float)v;
                    }
                    sb ^= 1;
                }
            } else if (MODE == T3_PAIRZ) {
                if (it.last) {
                    const Rbf rb = rbf_of(it.gamma, it.lam2);
                    const int rows = it.rows, cols = it.cols;
                    float best[2] = {0.f, FLT_MIN};   // the second never 0: the pass has run
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = cq + 2 * j;
                        const float2 sj = ld2(&cc.sq[0][c]), rj = ld2(&cc.mu[0][c]);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int rk = r0 + 2 * k, least = it.diag ? rk : -1;
                            const float ri = cc.mu[1][rk];
                            const float2 e = rbf2(rb, G.v[k][j], cc.sq[1][rk], sj);
                            if (rk < rows && c < cols && c > least) note_pair_z(e.x, ri, rj.x, best);
                            if (rk < rows && c + 1 < cols && c + 1 > least) note_pair_z(e.y, ri, rj.y, best);
                        }
                    }
                    unsigned* const to = it.ctrl->zpair_bits;
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        best[u] = warp_max_f(best[u]);
                        if (lane == 0 && __float_as_uint(best[u]) > *(volatile unsigned*)&to[u])
                            atomicMax(&to[u], __float_as_uint(best[u]));
                    }
                }
            } else {
                const Rbf rb = rbf_of(it.gamma, it.lam2);
                const int rows = it.rows, cols = it.cols;
                const bool diag = it.diag != 0, full = !diag && rows >= T && cols >= T;   // every pair valid
                constexpr int NSUM = MODE == T3_FINAL ? 2 : 1;
                // FORM: |Q|; FINAL: q mu and q alpha, the row's over the columns and the columns' over the rows
                float2 rsum[NSUM][4], csum[NSUM][4];
#pragma unroll
                for (int s = 0; s < NSUM; ++s)
#pragma unroll
                    for (int k = 0; k < 4; ++k) rsum[s][k] = csum[s][k] = f2(0.f);
                float tmx = 0.f;
                float* const store = MODE == T3_FORM && it.store ? it.store + (size_t)r0 * T + cq : nullptr;
                const auto entry = [&](int k, float2 g2, float2 sj, int c) {
                    const int rk = r0 + 2 * k;
                    float2 e = rbf2(rb, g2, cc.sq[1][rk], sj);
                    if (!full) {
                        const int least = diag ? rk : -1;
                        if (!(rk < rows && c < cols && c > least)) e.x = 0.f;
                        if (!(rk < rows && c + 1 < cols && c + 1 > least)) e.y = 0.f;
                    }
                    return e;
                };
                if constexpr (MODE == T3_FORM) {
                    float2 sj[4], yj[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        sj[j] = ld2(&cc.sq[0][cq + 2 * j]);
                        yj[j] = ld2(&cc.y[0][cq + 2 * j]);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t si = __float_as_uint(cc.y[1][r0 + 2 * k]);
                        float2 q[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const float2 e = entry(k, G.v[k][j], sj[j], cq + 2 * j);
                            rsum[0][k] = __fadd2_rn(rsum[0][k], e);
                            csum[0][j] = __fadd2_rn(csum[0][j], e);
                            tmx = fmaxf(tmx, fmaxf(e.x, e.y));
                            q[j] = flip(e, si ^ __float_as_uint(yj[j].x), si ^ __float_as_uint(yj[j].y));
                        }
                        if (store)
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(store + 2 * k * T),
                                         "f"(q[0].x), "f"(q[0].y), "f"(q[1].x), "f"(q[1].y), "f"(q[2].x), "f"(q[2].y),
                                         "f"(q[3].x), "f"(q[3].y)
                                         : "memory");
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = cq + 2 * j;
                        const float2 sj = ld2(&cc.sq[0][c]), yj = ld2(&cc.y[0][c]), muj = ld2(&cc.mu[0][c]), alj = ld2(&cc.al[0][c]);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int rk = r0 + 2 * k;
                            const uint32_t si = __float_as_uint(cc.y[1][rk]);
                            const float2 q = flip(entry(k, G.v[k][j], sj, c), si ^ __float_as_uint(yj.x), si ^ __float_as_uint(yj.y));
                            rsum[0][k] = __ffma2_rn(q, muj, rsum[0][k]);
                            rsum[NSUM - 1][k] = __ffma2_rn(q, alj, rsum[NSUM - 1][k]);
                            csum[0][j] = __ffma2_rn(q, f2(cc.mu[1][rk]), csum[0][j]);
                            csum[NSUM - 1][j] = __ffma2_rn(q, f2(cc.al[1][rk]), csum[NSUM - 1][j]);
                        }
                    }
                }
#pragma unroll
                for (int s = 0; s < NSUM; ++s) {
                    su.row[s][cg][r0 + 2 * lq] = row_sums4(rsum[s], lane);
                    su.col[s][g][cq + lr] = col_sums8(csum[s], lane);
                }
                float* const tilemax = MODE == T3_FORM ? it.tilemax : nullptr;
                if (MODE == T3_FORM && tilemax) {
                    tmx = warp_max_f(tmx);
                    if (lane == 0) su.tmx[ew] = tmx;
                }
                if (!meet()) { ok = false; break; }
                // per-node slot partials (fixed order): row sums of the tile's rows,
                // column sums of its columns; both roles on a diagonal tile.  Where
                // fix is set they are added to the nodes' fixed-point sums instead.
                if (etid < 2 * T) {
                    const int off = etid & (T - 1), role = etid / T;
                    if (off < (role ? cols : rows) && !(diag && role)) {
#pragma unroll
                        for (int s = 0; s < NSUM; ++s) {
                            const float (*rw)[T] = su.row[s];
                            const float (*cl)[T] = su.col[s];
                            const float vr = (rw[0][off] + rw[1][off]) + (rw[2][off] + rw[3][off]);
                            const float vc = ((cl[0][off] + cl[1][off]) + cl[2][off]) + cl[3][off];
                            const float v = diag ? vr + vc : role ? vc : vr;
                            if (MODE == T3_FORM && it.fix[0]) atomicAdd(it.fix[role] + off, (unsigned long long)rsum_fix(v, it.shift));
                            else it.dst[role][s * it.plen + off] = v;
                        }
                    }
                }
                if (MODE == T3_FORM && etid == 0 && tilemax) {
                    float m2 = 0.f;
                    for (int e = 0; e < T3_EPI_WARPS; ++e) m2 = fmaxf(m2, su.tmx[e]);
                    *tilemax = m2;
                }
                sb ^= 1;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.iempty[b]);
            if ((b ^= 1) == 0) iph ^= 1u;
        }
        if (!ok && lane == 0) {
            sm.abort = 1;
            record_error(tab[work[blockIdx.x].x].ctrl, ST_ETIMEOUT, blockIdx.x);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tbase, T3_TMEM_COLS);
    }
}

constexpr size_t t3_smem_bytes() { return 1024 + T3_STAGES * T3_STAGE_BYTES + sizeof(T3Smem); }

// The opted-in shared memory, once per kernel and device.
template <int MODE>
cudaError_t launch_gram(const Inst* tab, const int4* work, long long ntiles, int norms_only, const StopOp* ops,
                        const DecideArgs& dec, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_gram_tc32<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)t3_smem_bytes());
    if (e != cudaSuccess) return e;
    const int sms = num_sms();
    k_gram_tc32<MODE><<<(int)(ntiles < sms ? ntiles : sms), T3_THREADS, t3_smem_bytes(), s>>>(tab, work, ntiles, norms_only,
                                                                                           ops, dec);
    return cudaGetLastError();
}

// The tiles of a decision (Ntt test tiles x Nt training tiles, row by row) in G
// even ranges, one per CTA: range c is [split_at(c), split_at(c + 1)), and the part of
// it in test tile I is its work entry I - (its first test tile), at index (that)
// G + c, which is how a grid of G CTAs takes them.  (In 4 ranges of each of 79
// test tiles, 316 entries on 152 CTAs, twelve CTAs had three of them and the
// others two: 376 us at t = 10000, n = 20000, m = 128; now 261.)
struct DecisionSplit {
    long long tiles;
    int G, Nt;
    __host__ __device__ long long split_at(int c) const { return (long long)c * tiles / G; }
    __host__ __device__ int first(int c) const { return (int)(split_at(c) / Nt); }
};

// out[s] of test row s of tile I: its entries' sums in order (FP64), unless a
// test row was refused.
__global__ void k_decision_out(const float* __restrict__ part, int t, DecisionSplit d, const Ctrl* __restrict__ check,
                               float* __restrict__ out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= t || check->status != 0) return;
    const int I = s / T;
    const long long lo = (long long)I * d.Nt, hi = lo + d.Nt;
    int c = (int)(lo * d.G / d.tiles);
    while (c > 0 && d.split_at(c) > lo) --c;
    while (d.split_at(c + 1) <= lo) ++c;
    double f = 0.0;
    for (; c < d.G && d.split_at(c) < hi; ++c) f += (double)part[((size_t)(I - d.first(c)) * d.G + c) * T + s % T];
    out[s] = (float)f;
}
__global__ void k_decision_work(int4* __restrict__ work, DecisionSplit d, int entries)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= entries) return;
    const int c = e % d.G, I = d.first(c) + e / d.G;
    const long long row = (long long)I * d.Nt, a = d.split_at(c), b = d.split_at(c + 1);
    const long long j0 = a > row ? a - row : 0, j1 = b < row + d.Nt ? b - row : d.Nt;
    work[e] = make_int4(0, I, (int)j0, (int)(j1 > j0 ? j1 : j0));   // (none: an empty range)
}

}  // namespace

size_t pack3_bytes(int Nt, int m) { return (size_t)NPLANE * Nt * bf16_chunks(m) * BLK_BYTES; }

cudaError_t launch_stage(const void* X, int x_dtype, int n, int m, int Nt, float* Xf, float* y, float* b, float* b0,
                         int task, void* Xp3, long long row0, Ctrl* check, int4* diag, cudaStream_t s)
{
    const int nkc = bf16_chunks(m);
    const unsigned grid = (unsigned)(((long long)Nt * T * nkc * (KCH / 8) + 255) / 256);
    uint4* out = static_cast<uint4*>(Xp3);
    if (Xf == X) Xf = nullptr;
    if (x_dtype == 1)
        k_stage_rows<<<grid, 256, 0, s>>>(static_cast<const double*>(X), n, m, nkc, Nt, Xf, y, b, b0, task, out, row0,
                                          check, diag);
    else if (x_dtype == 2)
        k_stage_rows<<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(X), n, m, nkc, Nt, Xf, y, b, b0, task, out,
                                          row0, check, diag);
    else
        k_stage_rows<<<grid, 256, 0, s>>>(static_cast<const float*>(X), n, m, nkc, Nt, Xf, y, b, b0, task, out, row0,
                                          check, diag);
    return cudaGetLastError();
}

cudaError_t launch_stage_list(const Inst* tab, const int2* nbl, int nblocks, cudaStream_t s)
{
    if (nblocks > 0) k_stage_list<<<nblocks, 256, 0, s>>>(tab, nbl);
    return cudaGetLastError();
}

cudaError_t launch_form_q_tc32(const Inst* tab, const int4* work, long long ntiles, int norms_only, cudaStream_t s)
{
    return launch_gram<T3_FORM>(tab, work, ntiles, norms_only, nullptr, DecideArgs{}, s);
}

cudaError_t launch_pair_z_gram(const Inst* tab, const int4* tiles, long long ntiles, bool single, cudaStream_t s)
{
    return launch_gram<T3_PAIRZ>(tab, tiles, ntiles, single, nullptr, DecideArgs{}, s);
}

cudaError_t launch_final_tiles_gram(const Inst* tab, const StopOp* ops, const int4* tiles, long long ntiles, cudaStream_t s)
{
    return launch_gram<T3_FINAL>(tab, tiles, ntiles, 0, ops, DecideArgs{}, s);
}

// (a range spans at most tiles / G + 1 + Nt - 1 of the row-major tiles' rows)
int decision_entries(int Ntt) { return 2 * num_sms() + Ntt; }

cudaError_t launch_decision_tc(const Inst* tab, const int4* diag, int4* work, int t, int Nt, const float* alpha, float* part,
                               const Ctrl* check, float* out, cudaStream_t s)
{
    const int Ntt = (t + T - 1) / T, sms = num_sms();
    DecisionSplit d;
    d.tiles = (long long)Ntt * Nt;
    d.G = (int)(d.tiles < sms ? d.tiles : sms);
    d.Nt = Nt;
    int deep = 1;   // the most test tiles of a range
    for (int c = 0; c < d.G; ++c) {
        const int rows = (int)((d.split_at(c + 1) - 1) / Nt) - d.first(c) + 1;
        deep = deep > rows ? deep : rows;
    }
    const int entries = deep * d.G;
    k_decision_work<<<(entries + 255) / 256, 256, 0, s>>>(work, d, entries);
    cudaError_t e = launch_gram<T3_FORM>(tab, diag, Ntt, 1, nullptr, DecideArgs{}, s);   // the test rows' norms
    if (e != cudaSuccess) return e;
    e = launch_gram<T3_DECIDE>(tab, work, entries, 0, nullptr, DecideArgs{alpha, part}, s);
    if (e != cudaSuccess) return e;
    k_decision_out<<<(t + 255) / 256, 256, 0, s>>>(part, t, d, check, out);
    return cudaGetLastError();
}

}  // namespace gabp
