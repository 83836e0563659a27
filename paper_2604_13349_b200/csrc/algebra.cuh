// Per-head dense algebra of Orthogonal BackFill (Eq. 2-6), one thread block per
// (cache, layer, KV head), everything in fp32.
//
// Inputs (from the streaming pass): Gram of the deleted values G_del, u = sum_del A_j v_j, the demand sums, and the
// retained rows themselves (read back from v_out).  The tuned streaming pass delivers G and u over ALL rows instead (it
// runs before the selection is known): P G_all P = P G_del P because P annihilates the retained rows; the retained
// rows' share of u and of the trace of G is subtracted here.
//
//   1. k_eff >= d: k_span_test has factorised G_keep (Cholesky).  If every pivot stayed above 1e-3 of its diagonal
//      entry the retained values span R^d, the residual of Eq. 3 is identically zero and delta = 0.
//   2. Otherwise the retained rows are reduced by Householder reflectors H_0 .. H_{m-1} (Eq. 2 as a QR factorisation:
//      reflector j maps row after row onto the coordinates 0 .. j); a row adds a reflector when what is left of it
//      beyond the coordinates reached so far exceeds 1e-4 of its own norm.  The same reflectors are then applied to G
//      from both sides.  With H = H_0 .. H_{m-1} the span of the retained values is the first m coordinates
//      of the rotated space, so the trailing block of H^T G H IS the residual's Gram matrix R^T R (Eq. 3 in Gram form,
//      App. H) in the d - m coordinates of the complement: no basis, no projector and no product P G P is formed, and
//      whatever is computed in those coordinates is orthogonal to the retained values to rounding.
//      r_bar (Eq. 4) is the tail of H^T u / (A_del + eps).
//   3. C = eigenvectors of the `rank` largest eigenvalues above 1e-5 of the largest.  For rank <= ALG_TRI_MAX_RANK the
//      reflectors simply go on: H_{m+1} .. H_{d-2} take the trailing block to tridiagonal form (so the basis and the
//      tridiagonal form together cost the d - 2 steps that the tridiagonal form of the full matrix would), the wanted
//      eigenvalues come from multisection on Sturm counts, their vectors from twisted factorisations (neighbours closer
//      than 1e-3 of the largest eigenvalue: from inverse iteration, kept orthogonal during it).  Heads of 128 channels stop as
//      soon as the first rows of the tridiagonal form provably hold the wanted eigenvalues and the next one, with their vectors, to
//      rounding: 24 to 36 rows of 96 where the spectrum falls off, and as many reflectors fewer on the way back.  For larger ranks: full
//      eigen-decomposition by parallel-order Jacobi rotations run to convergence.
//   4. Delta = C^T C r_bar (Eq. 5) in the rotated coordinates, taken back through the reflectors as ONE vector,
//      delta = A_del / (A_keep + eps) * Delta (Eq. 6), V_out = V_keep + delta on the head's retained rows (Eq. 7).
//
// What bounds it: the chain of d - 2 dependent reflectors, each a matrix-vector product, a reduction, a rank-two
// update and the norm of the next row.  The matrix therefore lives in REGISTERS (of every 32 rows half-warp g of 8 holds four,
// a lane pairs of columns for the two-wide FMA); only the reflector and the product cross warps, through shared memory,
// at one block barrier per reflector of a retained row and two per reflector of the tridiagonal form.  Steps run in
// stages of 32 so that finished rows and column pairs cost nothing and every register index is static.  128 threads of
// 255 registers and less than 113 KB per block: two blocks share a multiprocessor.  What is run once per head is written
// as small loops: a section's first pass costs about 130 cycles per 128 bytes of its code, more than its arithmetic.
// Measured on 36 x 8 heads, budget 32, rank 2, head_dim 128 (every head back-filled): 0.534 ms for the
// same algebra on a matrix in shared memory (Gram-Schmidt basis, M = P G P, then the reduction), 0.142 with all rows of the tridiagonal
// form, 0.110 (values whose channels fall off; how much the early end brings for other spectra stands at ALG_EXIT_FIRST).  Slower
// were: one barrier a row of the form, as for the retained rows (622 to 1400 cycles a row against 690 to 1210: more instructions),
// eight warps with half the registers, the chain of reflectors in a warp of its own beside the matrix warps (the registers it takes
// cost the others more), one copy of the step's code for all stages, the reflectors on G sixteen at a time in compact form (code
// that runs twice costs more to fetch than it saves), the auxiliary vector or the next row's norm in one warp only.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace obf {

constexpr int ALG_NW = 4;
constexpr int ALG_NT = 32 * ALG_NW;
constexpr int ALG_NG = 2 * ALG_NW;              // half-warps: the units that rows are dealt to
constexpr int ALG_BATCH = 32;                   // retained rows in registers at a time
constexpr float SPAN_ROW_TOL = 1e-4f;
constexpr float RCR_SKIP_TOL = 1e-6f;
constexpr float EIG_RANK_TOL = 1e-5f;
constexpr int JACOBI_MAX_SWEEPS = 30;
constexpr int ALG_TRI_MAX_RANK = 8;     // up to this rank only rank + 1 eigenvalues and rank eigenvectors are computed
static_assert(ALG_TRI_MAX_RANK + 1 < 32, "a lane for each of them and one more");
constexpr float EIG_CLUSTER_TOL = 1e-3f; // eigenvalues closer than this (relative to the largest): inverse iteration, kept orthogonal during it
// Rows of the tridiagonal form after which it is asked whether they suffice, and how many more at least before it is asked again (a
// quarter of them where that is more, half where the rest is far too large).  A question costs 400 cycles where the rest's bound exceeds
// all that the rows so far can hold, else 2000 to 4500 after 30 rows and twice that after 70; a row costs 850 to 1600.  So it is given up
// where the rest comes down too slowly: when a line through its last two bounds, half as far again, ends behind three quarters of all
// rows.  36 x 8 heads of 1024 positions, budget 32, ranks 1, 2 and 4, us a call:
//   values' channels             all rows         asked to the end   given up so
//   flat                         212  213  224    228  224  236      215  216  228
//   flat, three 8 times as large 211  213  222    198  207  234      199  207  226
//   0.985 each of the last       212  213  224    224  213  230      221  220  228
//   0.97 each of the last        212  213  225    201  203  213      199  203  212
//   inverse root of their number 211  213  222    182  187  199      181  187  199
constexpr int ALG_EXIT_FIRST = 18, ALG_EXIT_STEP = 6;
constexpr float ALG_EXIT_BEND = 1.5f, ALG_EXIT_SHARE = 0.75f;
constexpr float EIG_NEAR_TOL = 5e-2f;    // closer than this: one more step of inverse iteration on the twisted factors, then made orthogonal

// a where the mask is all ones, b where it is zero.  (A conditional between array elements would be a conditional
// address, and the array would have to live in memory.)
__device__ __forceinline__ f32x2 sel2(f32x2 mask, f32x2 a, f32x2 b) { return b ^ ((a ^ b) & mask); }
__device__ __forceinline__ f32x2 mask2(bool c) { return c ? ~0ull : 0ull; }
// Sums of N values per lane (a power of two) over runs of W lanes (W >= N): lane l of a run ends with the total of value
// l / (W / N).  Half as many values travel at every step: about N shuffles instead of N log2(W).
template <int N, int W>
__device__ __forceinline__ float transposed_sum(float (&a)[N], int lane)
{
    int off = W / 2;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? a[i] : a[i + n], keep = up ? a[i + n] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off >= 1; off >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off);
    return a[0];
}

__device__ __forceinline__ float half_sum(float v)
{
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The matrix in registers.  Of every 32 consecutive rows half-warp g (of ALG_NG = 8) holds the four 4 g .. 4 g + 3, lane c
// of its sixteen of each row the pairs of columns 32 q + 2 c, 32 q + 2 c + 1.  A reflector and the product with it meet the
// warps in shared memory: a lane reads its columns two by two and its rows four by four from the same array.
template <int D>
struct AlgShape {
    static constexpr int RW = D / ALG_NG;        // rows a lane holds
    static constexpr int NQ = D / 32;            // column pairs a lane holds per row
    static constexpr int RPS = 32 / ALG_NG;      // rows a lane holds of 32 consecutive ones
    __device__ static __forceinline__ int row(int grp, int r) { return 32 * (r / RPS) + RPS * grp + r % RPS; }
    __device__ static __forceinline__ int owner(int row) { return (row & 31) / RPS; }                    // its half-warp
    __device__ static __forceinline__ int slot(int row) { return RPS * (row / 32) + row % RPS; }         // and place there
};
static_assert(ALG_NG == 8, "rows are read four at a time");
template <int D>
using AlgMat = f32x2[AlgShape<D>::RW][AlgShape<D>::NQ];
template <int D>
using AlgRow = f32x2[AlgShape<D>::NQ];

// Column pairs from pair FROM on of a vector of D floats in shared memory.
template <int D, int FROM = 0>
__device__ __forceinline__ void alg_load(AlgRow<D> &x, const float *v, int c16)
{
#pragma unroll
    for (int q = FROM; q < AlgShape<D>::NQ; ++q) x[q] = *reinterpret_cast<const f32x2 *>(v + 32 * q + 2 * c16);
}
template <int D, int FROM = 0>
__device__ __forceinline__ float alg_dot(const AlgRow<D> &x, const AlgRow<D> &y)
{
    f32x2 a = mul2(x[FROM], y[FROM]);
#pragma unroll
    for (int q = FROM + 1; q < AlgShape<D>::NQ; ++q) a = fma2(x[q], y[q], a);
    return sum2(a);
}

// Stage S serves the reflectors 32 S .. 32 S + 31: their support starts at row and column 32 S or later.
// po = 2 M v on the rows of the stage (v in shared memory, its column pairs in v2).  With kp also this half-warp's share of
// v . p, in kp[grp]: formed from the lanes' partial sums, its reduction runs beside that of p.
template <int D, int S>
__device__ __forceinline__ void alg_product(const AlgMat<D> &M, const AlgRow<D> &v2, const float *v, float *po, float *kp, int grp, int c16)
{
    constexpr int RW = AlgShape<D>::RW, RPS = AlgShape<D>::RPS, R0 = RPS * S, NR = RW - R0;
    constexpr int NP = NR > 8 ? 16 : NR > 4 ? 8 : NR > 2 ? 4 : 2;
    float acc[NP];
#pragma unroll
    for (int r = 0; r < NP; ++r) acc[r] = r < NR ? alg_dot<D, S>(M[R0 + (r < NR ? r : 0)], v2) : 0.f;
    float ka = 0.f, kb = 0.f;
    if (kp) {
#pragma unroll
        for (int r = 0; r < NR; r += RPS) {
            const float4 w = *reinterpret_cast<const float4 *>(v + 32 * (S + r / RPS) + RPS * grp);
            ka = fmaf(w.x, acc[r], ka);
            kb = fmaf(w.y, acc[r + 1], kb);
            ka = fmaf(w.z, acc[r + 2], ka);
            kb = fmaf(w.w, acc[r + 3], kb);
        }
        ka = 2.f * half_sum(ka + kb);
    }
    const float s = 2.f * transposed_sum<NP, 16>(acc, c16);
    constexpr int LPR = 16 / NP;
    const int r = c16 / LPR;
    if ((c16 % LPR) == 0 && r < NR) po[AlgShape<D>::row(grp, R0 + r)] = s;
    if (kp && c16 == 0) kp[grp] = ka;
}

// M <- M - v w^T - w v^T with w = p - (v.p) v on the rows and columns of the stage.  x: row `xr` of the stage's first
// RPS rows as the update leaves it, formed first so that the next reflector need not wait.
template <int D, int S>
__device__ __forceinline__ void alg_update(AlgMat<D> &M, const AlgRow<D> &v2, const float *v, const float *p, const float *kp, int grp,
                                           int c16, int xr, AlgRow<D> &x)
{
    constexpr int RW = AlgShape<D>::RW, NQ = AlgShape<D>::NQ, RPS = AlgShape<D>::RPS, R0 = RPS * S;
    AlgRow<D> w2, nv2;
    alg_load<D, S>(w2, p, c16);
    float kq[ALG_NG / 4], kk = 0.f;
#pragma unroll
    for (int e = 0; e < ALG_NG / 4; ++e) {
        const float4 t = *reinterpret_cast<const float4 *>(kp + 4 * e);
        kq[e] = (t.x + t.y) + (t.z + t.w);
    }
#pragma unroll
    for (int e = 0; e < ALG_NG / 4; e += 2) kk += kq[e] + kq[e + 1];
    const f32x2 nk = pk(-kk, -kk), neg = pk(-1.f, -1.f);
#pragma unroll
    for (int q = S; q < NQ; ++q) {
        w2[q] = mul2(fma2(nk, v2[q], w2[q]), neg);
        nv2[q] = mul2(v2[q], neg);
    }
    {
        const int row = AlgShape<D>::row(grp, R0) + xr;
        const float v1 = v[row], w1 = fmaf(-kk, v1, p[row]);
        const f32x2 vx = pk(v1, v1), wx = pk(w1, w1);
        const f32x2 odd = mask2(xr & 1), high = mask2(xr & 2);
#pragma unroll
        for (int q = S; q < NQ; ++q) {
            const f32x2 m = sel2(high, sel2(odd, M[R0 + 3][q], M[R0 + 2][q]), sel2(odd, M[R0 + 1][q], M[R0][q]));
            x[q] = fma2(vx, w2[q], fma2(wx, nv2[q], m));
        }
    }
#pragma unroll
    for (int r = R0; r < RW; r += RPS) {
        const int row = AlgShape<D>::row(grp, r);
        const float4 va = *reinterpret_cast<const float4 *>(v + row), pa = *reinterpret_cast<const float4 *>(p + row);
        const float vv[4] = {va.x, va.y, va.z, va.w}, pp[4] = {pa.x, pa.y, pa.z, pa.w};
#pragma unroll
        for (int e = 0; e < RPS; ++e) {
            const float w = fmaf(-kk, vv[e], pp[e]);
#pragma unroll
            for (int q = S; q < NQ; ++q) M[r + e][q] = fma2(pk(vv[e], vv[e]), w2[q], fma2(pk(w, w), nv2[q], M[r + e][q]));
        }
    }
}

// Entry c (the same in every lane) of a row, given as column pairs, for both half-warps.
template <int D, int FROM = 0>
__device__ __forceinline__ float alg_entry(const AlgRow<D> &x, int c, int lane)
{
    f32x2 v = x[FROM];
#pragma unroll
    for (int q = FROM + 1; q < AlgShape<D>::NQ; ++q) v = sel2(mask2(c >> 5 == q), x[q], v);
    float a, b;
    upk(v, a, b);
    return __shfl_sync(0xffffffffu, (c & 1) ? b : a, (lane & 16) + ((c & 31) >> 1));
}

// Sum of squares of a row's entries from `from` on (pairs before FROM hold nothing of it).
template <int D, int FROM = 0>
__device__ __forceinline__ float alg_tail2(const AlgRow<D> &x, int from, int c16)
{
    float s = 0.f;
#pragma unroll
    for (int q = FROM; q < AlgShape<D>::NQ; ++q) {
        float a, b;
        upk(x[q], a, b);
        const int c = 32 * q + 2 * c16;
        a = c >= from ? a : 0.f;
        b = c + 1 >= from ? b : 0.f;
        s = fmaf(a, a, fmaf(b, b, s));
    }
    return half_sum(s);
}

// Writes the unit reflector of support >= j0 made of x: entry j0 is `first`, the others x, all scaled (a half-warp's lanes).
template <int D, int FROM = 0>
__device__ __forceinline__ void alg_store_reflector(const AlgRow<D> &x, int j0, float first, float rs, float *v, int c16)
{
#pragma unroll
    for (int q = 0; q < AlgShape<D>::NQ; ++q) {
        float a = 0.f, b = 0.f;
        if (q >= FROM) upk(x[q], a, b);
        const int c = 32 * q + 2 * c16;
        a = c < j0 ? 0.f : (c == j0 ? first : a) * rs;
        b = c + 1 < j0 ? 0.f : (c + 1 == j0 ? first : b) * rs;
        *reinterpret_cast<f32x2 *>(v + c) = pk(a, b);
    }
}

// Reflector j + 1 from row j of the trailing block (entries of x from j on), with the row's diagonal and off-diagonal
// entry of the tridiagonal form.  Every half-warp computes on its own row; the owner of row j stores.
template <int D, int FROM>
__device__ __forceinline__ void alg_row_done(const AlgRow<D> &x, int j, float tiny2, float *Y, float *ta, float *tb,
                                             int grp, int lane)
{
    const int c16 = lane & 15;
    const float below2 = alg_tail2<D, FROM>(x, j + 2, c16);          // squares right of the super-diagonal entry
    const float dg = alg_entry<D, FROM>(x, j, lane), x0 = alg_entry<D, FROM>(x, j + 1, lane);
    const float n2 = fmaf(x0, x0, below2), nrm = n2 * rsqrt_approx(fmaxf(n2, 1e-37f));
    const float al = x0 >= 0.f ? -nrm : nrm;
    const float vn2 = 2.f * fmaf(nrm, fabsf(x0), n2);                // |x - al e_0|^2
    const bool skip = !(below2 > tiny2) || !(vn2 > 1e-37f);          // nothing beyond the super-diagonal
    const float rs = skip ? 0.f : rsqrt_approx(vn2);
    if (grp == AlgShape<D>::owner(j)) {
        alg_store_reflector<D, FROM>(x, j + 1, x0 - al, rs, Y + (j + 1) * D, c16);
        if (c16 == 0) {
            ta[j] = dg;
            tb[j] = skip ? x0 : al;
        }
    }
}

// x with its entries before `from` zero.
template <int D, int FROM = 0>
__device__ __forceinline__ void alg_masked(AlgRow<D> &m, const AlgRow<D> &x, int from, int c16)
{
#pragma unroll
    for (int q = FROM; q < AlgShape<D>::NQ; ++q) {
        float a, b;
        upk(x[q], a, b);
        const int c = 32 * q + 2 * c16;
        m[q] = pk(c >= from ? a : 0.f, c + 1 >= from ? b : 0.f);
    }
}
// w: x from entry j0 + 1 on as it is (m, masked), entry j0 `first`, zeros before.
template <int D, int FROM = 0>
__device__ __forceinline__ void alg_with_first(AlgRow<D> &w, const AlgRow<D> &m, int j0, float first, int c16)
{
#pragma unroll
    for (int q = FROM; q < AlgShape<D>::NQ; ++q) {
        float a, b;
        upk(m[q], a, b);
        const int c = 32 * q + 2 * c16;
        w[q] = pk(c == j0 ? first : a, c + 1 == j0 ? first : b);
    }
}
// Half of |w|^2 and w's first entry, for a row of first entry x0 whose other squares sum to `below2`: w = x + sign(x0) |x| e_0.
__device__ __forceinline__ float alg_first(float x0, float below2, float &first, float &al)
{
    const float n2 = fmaf(x0, x0, below2), nrm = n2 * rsqrt_approx(fmaxf(n2, 1e-37f));
    al = x0 >= 0.f ? -nrm : nrm;
    first = x0 - al;
    return fmaf(nrm, fabsf(x0), n2);
}

// Sturm counts of the tridiagonal matrix (diagonal a, squared off-diagonals b2, scaled to a spectrum within [-1, 1]) at
// two shifts: the number of eigenvalues below each, as the sign changes of the leading principal minors'
// three-term recurrence p_i = (a_i - x) p_{i-1} - b2_{i-1} p_{i-2} (Givens' bisection).  No division: a step of the chain
// is one FMA.  Both values are rescaled by a power of two every four steps (a step grows them at most threefold; b2 is
// kept above 1e-14, so four steps shrink them by 1e-28 at most and two consecutive zeros cannot occur).
// n4: steps in groups of four; the arrays are padded to that with a = 2 (no sign change), b2 = 0.
__device__ __forceinline__ void sturm_count2(const float *a, const float *b2, int n4, float x0, float x1, int &c0, int &c1)
{
    float p0 = 1.f, q0 = 0.f, p1 = 1.f, q1 = 0.f;
    uint32_t n0 = 0u, n1 = 0u;
    float4 an = *reinterpret_cast<const float4 *>(a), bn = *reinterpret_cast<const float4 *>(b2);
#pragma unroll 1
    for (int i = 0; i < n4; ++i) {
        const float aa[4] = {an.x, an.y, an.z, an.w}, bb[4] = {-bn.x, -bn.y, -bn.z, -bn.w};
        // the next four steps' entries, ahead of the chain (the arrays have four floats to spare)
        an = *reinterpret_cast<const float4 *>(a + 4 * i + 4);
        bn = *reinterpret_cast<const float4 *>(b2 + 4 * i + 4);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float r0 = fmaf(aa[e] - x0, p0, bb[e] * q0), r1 = fmaf(aa[e] - x1, p1, bb[e] * q1);
            n0 += (__float_as_uint(r0) ^ __float_as_uint(p0)) >> 31;
            n1 += (__float_as_uint(r1) ^ __float_as_uint(p1)) >> 31;
            q0 = p0; p0 = r0;
            q1 = p1; p1 = r1;
        }
        // 2^-e of the larger one's exponent e (max 254 keeps the factor a normal number)
        const uint32_t e0 = max(__float_as_uint(p0) & 0x7F800000u, __float_as_uint(q0) & 0x7F800000u);
        const uint32_t e1 = max(__float_as_uint(p1) & 0x7F800000u, __float_as_uint(q1) & 0x7F800000u);
        const float f0 = __uint_as_float(0x7F000000u - min(e0, 0x7E800000u)), f1 = __uint_as_float(0x7F000000u - min(e1, 0x7E800000u));
        p0 *= f0; q0 *= f0;
        p1 *= f1; q1 *= f1;
    }
    c0 = (int)n0;
    c1 = (int)n1;
}

// Shared memory, in floats.  Y: the reflectors (all d of them on the tridiagonal route, else those of the retained rows).
template <int D>
__host__ __device__ constexpr int algebra_y_rows(int mcap, int rank, int fast_iters)
{
    return (fast_iters > 0 || rank > ALG_TRI_MAX_RANK) ? mcap : D;
}

// Workspace of the eigen-solvers: tridiagonal form (scaled diagonal and squared off-diagonals, per wanted vector six
// arrays), or two blocks of rows of the fixed-iteration route, or the trailing block and the eigenvector matrix of the
// Jacobi route.  At least the retained rows' share of u before it and the products among the reflectors after it.
template <int D>
__host__ __device__ constexpr int algebra_eig_floats(int rank, int fast_iters)
{
    const int r = rank < D ? rank : D;
    const int tri = 2 * (D + 8) + r * 6 * D;
    const int least = ALG_BATCH * D;
    const int eig = fast_iters > 0 ? 2 * r * D : (rank <= ALG_TRI_MAX_RANK ? tri : 2 * D * (D + 1));
    return eig > least ? eig : least;
}

template <int D>
constexpr size_t algebra_smem_bytes(int mcap, int rank, int fast_iters)
{
    return (size_t)(algebra_y_rows<D>(mcap, rank, fast_iters) * D +  2 * D + 6 * D + 96 +
                    algebra_eig_floats<D>(rank, fast_iters)) * sizeof(float) + 2 * D * sizeof(int);
}
// The most any call needs: the Jacobi route with d basis rows.
template <int D>
constexpr size_t ALG_SMEM_MAX = algebra_smem_bytes<D>(D, D, 0);
static_assert(ALG_SMEM_MAX<128> >= algebra_smem_bytes<128>(128, 128, 1) && ALG_SMEM_MAX<128> >= algebra_smem_bytes<128>(128, ALG_TRI_MAX_RANK, 0) &&
              ALG_SMEM_MAX<64> >= algebra_smem_bytes<64>(64, 64, 1) && ALG_SMEM_MAX<64> >= algebra_smem_bytes<64>(64, ALG_TRI_MAX_RANK, 0), "no route needs more");
static_assert(ALG_SMEM_MAX<128> <= 227 * 1024 - 1024, "a block has 227 KB, some of it static");

// 2. Reflectors of a head's k retained rows (Eq. 2), into Y (shared memory): how many there are.  A loop of its own and not one with
// that over G: together their code outgrows what a multiprocessor fetches at full speed.
// The next row passes through `next` (2 buffers of D + 4 floats) one reflector early, and every half-warp finds every reflector for
// itself; and as a reflector is its row but for one entry, which the row's norm decides, all products with it are formed while the
// norm is still being added up: one reduction and one barrier a row.  With the owner's reflector sent to the others, then their
// products, 1010 cycles a row of 128 channels, this way 660 (two heads on a multiprocessor 1070 and 900).
template <typename TIN, int D>
__device__ __forceinline__ int alg_reflectors(const TIN *vk, int k, float *Y, float *next)
{
    constexpr int NQ = AlgShape<D>::NQ;
    const int tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5), grp = tid >> 4, c16 = tid & 15;
    int m = 0;
    // a batch of rows in registers (G comes afterwards): row b0 + grp + ALG_NG s in slot s of the half-warp
    constexpr int NS = ALG_BATCH / ALG_NG;
    static_assert(NS == 4, "four slots to pick from");
    AlgRow<D> V[NS];
    float n0[NS] = {0.f, 0.f, 0.f, 0.f};                       // the rows' squared norms
    auto reflect_rows = [&](const AlgRow<D> &v) __attribute__((always_inline)) {
        float d4[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) d4[s] = alg_dot<D>(V[s], v);
        const float tot = -2.f * transposed_sum<NS, 16>(d4, c16);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const float f = __shfl_sync(0xffffffffu, tot, (lane & 16) + (16 / NS) * s);
#pragma unroll
            for (int q = 0; q < NQ; ++q) V[s][q] = fma2(pk(f, f), v[q], V[s][q]);
        }
    };
    // row i of the batch, as the reflectors so far leave it, for everybody, with its squared norm
    auto publish = [&](int i) __attribute__((always_inline)) {
        if (warp != (i % ALG_NG) / 2) return;
        const f32x2 odd = mask2(i / ALG_NG & 1), high = mask2(i / ALG_NG & 2);
        const float nn = i / ALG_NG & 2 ? (i / ALG_NG & 1 ? n0[3] : n0[2]) : (i / ALG_NG & 1 ? n0[1] : n0[0]);
        float *to = next + (i & 1) * (D + 4);
        if (grp != i % ALG_NG) return;
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            *reinterpret_cast<f32x2 *>(to + 32 * q + 2 * c16) = sel2(high, sel2(odd, V[3][q], V[2][q]), sel2(odd, V[1][q], V[0][q]));
        if (c16 == 0) to[D] = nn;
    };
#pragma unroll 1
    for (int b0 = 0; b0 < k && m < D; b0 += ALG_BATCH) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int i = b0 + grp + ALG_NG * s;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                V[s][q] = 0ull;
                if (i < k) {
                    const TIN *src = vk + (size_t)i * D + 32 * q + 2 * c16;
                    if constexpr (sizeof(TIN) == 4) V[s][q] = *reinterpret_cast<const f32x2 *>(src);
                    else {
                        const uint32_t w = *reinterpret_cast<const uint32_t *>(src);
                        V[s][q] = pk(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
                    }
                }
            }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            n0[s] = half_sum(alg_dot<D>(V[s], V[s]));
            // a reflector depends on its row's direction alone: rows whose squares leave the range of fp32's normal numbers
            // are brought back by a power of two.  A row that is not finite adds no direction and is a row of zeros from here on: it
            // meets the others with a factor of zero, which would not be zero
            const bool far = n0[s] != 0.f && !(n0[s] > 1e-24f && n0[s] < 1e24f);
            if (warp_uniform(far)) {                           // (any of them: the sum below takes the whole warp)
                const float f = !far ? 1.f : n0[s] < 1.f ? 1.8446744e19f : 5.421011e-20f;   // 2^64, 2^-64
#pragma unroll
                for (int q = 0; q < NQ; ++q) V[s][q] = mul2(V[s][q], pk(f, f));
                n0[s] = half_sum(alg_dot<D>(V[s], V[s]));
                const bool finite = n0[s] < INFINITY;
                n0[s] = finite ? n0[s] : 0.f;
#pragma unroll
                for (int q = 0; q < NQ; ++q) V[s][q] &= mask2(finite);
            }
        }
        // (the reflectors that earlier batches found, all published behind a barrier)
#pragma unroll 1
        for (int j = 0; j < m; ++j) {
            AlgRow<D> v;
            alg_load<D>(v, Y + j * D, c16);
            reflect_rows(v);
        }
        const int rows = min(ALG_BATCH, k - b0);
        publish(0);
        if (rows > 1) publish(1);
        __syncthreads();
        AlgRow<D> x;                                           // row i as all reflectors before it leave it (the same in every half-warp)
        alg_load<D>(x, next, c16);
        float nn = next[D];
        // Row i's buffer is written again with row i + 2, in iteration i, behind the barrier after its last read: that is the one that ends
        // iteration i - 1, where row i was read, and for row 0, read just now, this one.
        __syncthreads();
#pragma unroll 1
        for (int i = 0; i < rows; ++i) {
            AlgRow<D> r;
            const float *from = next + ((i + 1) & 1) * (D + 4);
            alg_load<D>(r, from, c16);
            const float nr = from[D];
            // The reflector of row i (zero unless the row adds a direction to the m there are) is the row but for its entry m: every product
            // with it is formed with the row's rest while the row's norm, which decides about that entry, is still being added up.
            AlgRow<D> w;
            alg_masked<D>(w, x, m + 1, c16);
            float d8[8] = {alg_dot<D>(w, w), alg_dot<D>(r, w), 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, f[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) d8[2 + s] = alg_dot<D>(V[s], w);
            const float tot = transposed_sum<8, 16>(d8, c16), below2 = __shfl_sync(0xffffffffu, tot, lane & 16);
            const float x0 = alg_entry<D>(x, m, lane);
            float first, al;
            const float h = alg_first(x0, below2, first, al), t2 = fmaf(x0, x0, below2);
            const bool add = warp_uniform(t2 > SPAN_ROW_TOL * SPAN_ROW_TOL * nn && t2 > 1e-37f);
            const float b = add ? -rcp_approx(h) : 0.f;
            alg_with_first<D>(w, w, m, first, c16);
            const float fr = b * fmaf(alg_entry<D>(r, m, lane), first, __shfl_sync(0xffffffffu, tot, (lane & 16) + 2));
#pragma unroll
            for (int s = 0; s < NS; ++s) f[s] = b * fmaf(alg_entry<D>(V[s], m, lane), first, __shfl_sync(0xffffffffu, tot, (lane & 16) + 4 + 2 * s));
            if (add && grp == i % ALG_NG) {
                // (to the last bit: the rows have met w, whose length is exact, G and the vectors will meet this)
                float rs = rsqrt_approx(2.f * h);
                rs *= fmaf(-h * rs, rs, 1.5f);
#pragma unroll
                for (int q = 0; q < NQ; ++q) *reinterpret_cast<f32x2 *>(Y + m * D + 32 * q + 2 * c16) = mul2(w[q], pk(rs, rs));
            }
            if (add && ++m >= D) break;                        // (the same everywhere)
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                x[q] = fma2(pk(fr, fr), w[q], r[q]);
#pragma unroll
                for (int s = 0; s < NS; ++s) V[s][q] = fma2(pk(f[s], f[s]), w[q], V[s][q]);
            }
            nn = nr;
            if (i + 2 < rows) publish(i + 2);
            __syncthreads();
        }
        // the reflectors are there, the buffers free
        __syncthreads();
    }
    return m;
}

// The reflectors of every head's retained rows, beside the pass over V where that waits for the selection (bf16 heads of 64 channels)
// and no budget reaches head_dim.  16 x 8 heads of 64 channels, 32 of 3001 rows: 126 -> 120 us a call.  Heads of 128 channels find
// theirs in k_obf_algebra: two of them share a multiprocessor there and hide it, and their call got slower (36 x 8 heads, 1024
// positions: 229 -> 233).
template <typename TIN, int D>
__global__ void __launch_bounds__(ALG_NT) k_obf_rows(const __grid_constant__ CallDev p)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    __shared__ __align__(16) float s_next[2 * (D + 4)];
    const int g = blockIdx.x;
    int ci, lh;
    locate(p, g, ci, lh);
    const CacheDev &c = p.c[ci];
    const int k = c.k_eff;
    if (c.T <= k) return;
    const int m = alg_reflectors<TIN, D>(reinterpret_cast<const TIN *>(c.v_out) + (size_t)lh * k * D, k, sm, s_next);
    float4 *dst = reinterpret_cast<float4 *>(p.rows_y + (size_t)g * p.alg_rows * D);
    for (int e = threadIdx.x; e < m * (D / 4); e += ALG_NT) dst[e] = reinterpret_cast<const float4 *>(sm)[e];
    if (threadIdx.x == 0) p.rows_m[g] = m;
}

template <typename TIN, int D>
__global__ void __launch_bounds__(ALG_NT, 2) k_obf_algebra(const __grid_constant__ CallDev p)
{
    pdl_wait();
    typedef AlgShape<D> SH;
    constexpr int RW = SH::RW, NQ = SH::NQ, LD = D + 1;
    extern __shared__ __align__(16) float sm[];
    float *Y = sm;                                                    // reflector j in row j, support >= j
    float *pl = Y + algebra_y_rows<D>(p.alg_rows, p.rank, p.fast_iters) * D;     // 2 buffers of D: the product with reflector j in j & 1
    float *ta = pl + 2 * D, *tb = ta + D;                             // tridiagonal form
    float *vu = tb + D, *vx = vu + D, *vc = vx + D, *vl = vc + D;     // vectors of d
    float *red = vl + D, *misc = red + 32, *tlam = misc + 32;         // 32 floats each
    int *ipq = reinterpret_cast<int *>(tlam + 32), *isel = ipq + D;   // Jacobi: pairs (p, q), selected columns
    float *rows_s = reinterpret_cast<float *>(isel + D);              // a batch of retained rows; then
    float *WS = rows_s;                                               // the workspace of the eigen-solvers
    __shared__ __align__(16) float kpart[2 * ALG_NG];                 // 2 buffers: the half-warps' shares of v . p

    const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5);
    const int grp = tid >> 4, c16 = tid & 15;                         // half-warp and the lane in it
    int ci, lh;
    locate(p, g, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff, S = p.gram_slots;
    const int n_del = gram_partial_count(p, c, lh);
    const float a_keep = p.sums[(size_t)g * 4], a_del = p.sums[(size_t)g * 4 + 1];
    const float alpha = a_del / (a_keep + p.eps);

    if (tid < D) {
        p.delta[(size_t)g * D + tid] = 0.f;
        if (c.delta_out) c.delta_out[(size_t)lh * D + tid] = 0.f;
    }
    if (T - k == 0 || p.rank <= 0) return;

    uint32_t status = 0u;
    int m = 0;
    float rcr = 0.f, lam1 = 0.f, lam_rho = 0.f, lam_next = 0.f, dnorm = 0.f, revr = 0.f, pc = 0.f;
    int rho = 0;
    bool done = false;

    // ---- 1. k_eff >= d: the span test kernel has already factorised G_keep --
    if (warp_uniform(k >= D && (p.hflag[g] & HFLAG_SPAN_FULL) != 0u)) { m = D; done = true; pc = 1.f; status |= OBF_DEV_SKIPPED | OBF_DEV_SPAN_FULL; }

    if (!done) {
        const TIN *vk = reinterpret_cast<const TIN *>(c.v_out) + (size_t)lh * k * D;
        const float *A = p.scores + c.tok_off + (size_t)lh * T;
        const int32_t *idx = c.idx_out + (size_t)lh * k;

        // ---- u (and, for the diagnostics, the plain sum of the deleted values) -------------------
        constexpr int NPART = ALG_NT / D;
        float sq = 0.f, us[U_LEVELS];                                  // us: what the pass over V added up, per level
#pragma unroll
        for (int l = 0; l < U_LEVELS; ++l) us[l] = 0.f;
        if (tid < D) {
#pragma unroll 1
            for (int sp = 0; sp < n_del; ++sp) {
                const float *uv = p.uvec + ((size_t)g * S + sp) * p.u_levels * D + tid;
#pragma unroll
                for (int l = 0; l < U_LEVELS; ++l)
                    if (l < p.u_levels) us[l] += uv[l * D];
            }
        }
        if (p.gram_all) {
            // the retained rows' share of u per mass level, and of the trace of G; a lane fetches one row's mass
            const int col = tid % D, part = tid / D;
            float uk[U_LEVELS];
#pragma unroll
            for (int l = 0; l < U_LEVELS; ++l) uk[l] = 0.f;
#pragma unroll 1
            for (int b0 = 0; b0 < k; b0 += 32) {
                // (the rows' loads are under way before the masses', which wait for the positions)
                constexpr int PR = 32 / NPART;
                float v[PR];
                const int at = b0 + lane < k ? idx[b0 + lane] : 0;
#pragma unroll
                for (int e = 0; e < PR; ++e) {
                    const int i = b0 + e * NPART + part;
                    v[e] = i < k ? to_f32(vk[(size_t)i * D + col]) : 0.f;
                }
                const float al = b0 + lane < k ? A[at] : 0.f;
#pragma unroll
                for (int e = 0; e < PR; ++e) {
                    const float a = __shfl_sync(0xffffffffu, al, e * NPART + part);
                    const int lev = u_level(a);
                    sq = fmaf(v[e], v[e], sq);
#pragma unroll
                    for (int l = 0; l < U_LEVELS; ++l) uk[l] = fmaf(l == lev ? a : 0.f, v[e], uk[l]);
                }
            }
#pragma unroll
            for (int l = 0; l < U_LEVELS; ++l) WS[(part * U_LEVELS + l) * D + col] = uk[l];
        }
        const float sq_keep = block_sum<ALG_NT>(sq, red);             // (its barriers also publish WS)
        if (tid < D) {
            // per level: what the pass over V added up minus the retained rows' share; smallest masses first
            float s = 0.f;
#pragma unroll
            for (int l = 0; l < U_LEVELS; ++l) {
                float kl = 0.f;
                if (p.gram_all)
                    for (int q = 0; q < NPART; ++q) kl += WS[(q * U_LEVELS + l) * D + tid];
                s += us[l] - kl;
            }
            vu[tid] = s;
            vx[tid] = c.diag ? p.svec[(size_t)g * D + tid] : 0.f;
        }
        __syncthreads();
        // one more vector per half-warp that the reflectors are applied to: u in the first, the sum of the deleted values
        // in the second
        AlgRow<D> aux;
        if (grp < 2) alg_load<D>(aux, grp == 0 ? vu : vx, c16);
        else {
#pragma unroll
            for (int q = 0; q < NQ; ++q) aux[q] = 0ull;
        }
        // x <- x - 2 (x.v) v
        auto reflect = [&](AlgRow<D> &x, const AlgRow<D> &v) __attribute__((always_inline)) {
            const float s = -2.f * half_sum(alg_dot<D>(x, v));
#pragma unroll
            for (int q = 0; q < NQ; ++q) x[q] = fma2(pk(s, s), v[q], x[q]);
        };
        // ---- 2. reflectors of the retained rows, unless k_obf_rows has found them ----
        if (p.rows_y) {
            m = warp_uniform(p.rows_m[g]);
            const float4 *src = reinterpret_cast<const float4 *>(p.rows_y + (size_t)g * p.alg_rows * D);
            for (int e = tid; e < m * (D / 4); e += ALG_NT) reinterpret_cast<float4 *>(Y)[e] = src[e];
            __syncthreads();
        } else {
            m = alg_reflectors<TIN, D>(vk, k, Y, WS);
        }
        // ---- G into registers, its trace, and the reflectors applied to it from both sides -----------------------
        AlgMat<D> M;
        {
            const float *G = p.gram_d + (size_t)g * S * D * D + 2 * c16;
#pragma unroll
            for (int r = 0; r < RW; ++r)
#pragma unroll
                for (int q = 0; q < NQ; ++q) M[r][q] = *reinterpret_cast<const f32x2 *>(G + SH::row(grp, r) * D + 32 * q);
#pragma unroll 1
            for (int sp = 1; sp < n_del; ++sp) {
                G += D * D;
#pragma unroll
                for (int r = 0; r < RW; ++r)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) M[r][q] = add2(M[r][q], *reinterpret_cast<const f32x2 *>(G + SH::row(grp, r) * D + 32 * q));
            }
        }
        // this thread's share of the diagonal from row `from` on
        auto diag_part = [&](int from) __attribute__((always_inline)) {
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const int i = SH::row(grp, r);
                float a, b;
                upk(M[r][r / SH::RPS], a, b);
                if (i >= from && c16 == (i & 31) >> 1) s += (i & 1) ? b : a;
            }
            return s;
        };

        // and of the squares of the trailing block from row and column `from` on
        auto square_part = [&](int from) __attribute__((always_inline)) {
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                AlgRow<D> x;
                alg_masked<D>(x, M[r], from, c16);
                const float t = sum2(fma2(x[0], x[0], NQ > 1 ? mul2(x[1], x[1]) : 0ull)), u = NQ > 2 ? sum2(fma2(x[NQ - 2], x[NQ - 2], mul2(x[NQ - 1], x[NQ - 1]))) : 0.f;
                if (SH::row(grp, r) >= from) s += t + u;
            }
            return s;
        };

        const float trAll = block_sum<ALG_NT>(diag_part(0), red);
        // squared Frobenius norm of the deleted values (the denominator of RCR).  As a difference of two fp32 traces
        // it is resolved down to about 1e-6 of the squared norm of all values: below 1e-5 of it the deleted values
        // count as negligible beside the retained ones and nothing is injected.
        const float trG = trAll - sq_keep;
        const bool del_negligible = p.gram_all && !(trG > 1e-5f * trAll);
        {
            auto apply_stage = [&](auto stage) __attribute__((always_inline)) {
                constexpr int ST = decltype(stage)::value;
                const int j1 = min(32 * ST + 32, m);
#pragma unroll 1
                for (int j = 32 * ST; j < j1; ++j) {
                    float *po = pl + (j & 1) * D, *kp = kpart + (j & 1) * ALG_NG;
                    AlgRow<D> v, x;
                    alg_load<D, ST>(v, Y + j * D, c16);
                    alg_product<D, ST>(M, v, Y + j * D, po, kp, grp, c16);
                    {
                        const float s = -2.f * half_sum(alg_dot<D, ST>(aux, v));
#pragma unroll
                        for (int q = ST; q < NQ; ++q) aux[q] = fma2(pk(s, s), v[q], aux[q]);
                    }
                    __syncthreads();                                   // p is there
                    alg_update<D, ST>(M, v, Y + j * D, po, kp, grp, c16, 0, x);
                }
            };
            if (m < D) {
                apply_stage(std::integral_constant<int, 0>{});
                apply_stage(std::integral_constant<int, 1>{});
                if constexpr (D > 64) {
                    apply_stage(std::integral_constant<int, D / 32 - 2>{});
                    apply_stage(std::integral_constant<int, D / 32 - 1>{});
                }
                __syncthreads();                                       // the buffers are used again
            }
        }
        if (m >= D) { done = true; pc = 1.f; status |= OBF_DEV_SKIPPED | OBF_DEV_SPAN_FULL; }

        if (!done) {
            if (c.diag) {
                // projection cosine: s = sum of the deleted values; its part inside span(V_keep) is the first m coordinates
                const float all = alg_tail2<D>(aux, 0, c16), out = alg_tail2<D>(aux, m, c16);
                if (grp == 1 && c16 == 0) misc[8] = all > 0.f ? sqrtf(fmaxf(all - out, 0.f) / all) : 0.f;
                __syncthreads();
                pc = misc[8];
            }
            float trM = block_sum<ALG_NT>(diag_part(m), red);
            rcr = del_negligible ? 0.f : trM / (trG + p.eps);
            if (warp_uniform(!(rcr >= RCR_SKIP_TOL))) { done = true; status |= OBF_DEV_SKIPPED; }
            // What follows squares the block's entries, so a trace far from one (values of 1e-11 or 1e9, say) is brought there by a
            // power of two: exact, and C does not depend on it.  misc[10]: what one stands for from here on (read behind barriers).
            if (tid == 0) misc[10] = 1.f;
            if (!done && warp_uniform(!(trM > 1e-6f && trM < 1e6f))) {
                const uint32_t e = min(max(__float_as_uint(trM) >> 23, 1u), 253u);
                const float f = __uint_as_float((254u - e) << 23);
#pragma unroll
                for (int r = 0; r < RW; ++r)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) M[r][q] = mul2(M[r][q], pk(f, f));
                trM *= f;
                if (tid == 0) misc[10] = __uint_as_float(e << 23);
            }

            int back = -1;                                         // the reflectors back .. m + 1 and m - 1 .. 0 lead back from the rotated coordinates
            const float inv_del = 1.f / (a_del + p.eps);

            // ---- 3a. few eigenpairs wanted: tridiagonal form, multisection, inverse iteration ----
            if (!done && p.fast_iters == 0 && p.rank <= ALG_TRI_MAX_RANK) {
                const float tiny2 = 1e-20f * trM * trM;
                int n = D - m;                                         // size of the trailing block, then of the tridiagonal form
                // Whether its first rows suffice is asked first after as many as spectra that fall off take, and never for the last few (heads
                // of 64 channels, not at all: the code costs them as much as it saves, 16 x 8 heads with 32 rows, rank 2, 116.3 -> 119.7 us).
                constexpr bool ASKS = D > 64;
                int last = ASKS ? m + ALG_EXIT_FIRST - 1 + (p.rank > 1 ? ALG_EXIT_STEP : 0) + (p.rank > 2 ? ALG_EXIT_STEP : 0) : D;
                float m2 = 0.f;                                        // squared Frobenius norm of the block
                if (ASKS && last <= D - 2 - 2 * ALG_EXIT_STEP) m2 = block_sum<ALG_NT>(square_part(m), red);
                if (n > 1) {
                    // reflector m + 1 from row m as it stands
                    AlgRow<D> x;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        x[q] = M[0][q];
#pragma unroll
                        for (int r = 1; r < RW; ++r) x[q] = sel2(mask2(r == SH::slot(m)), M[r][q], x[q]);
                    }
                    alg_row_done<D, 0>(x, m, tiny2, Y, ta, tb, grp, lane);
                }
                int J = m + 1;                                         // the next step's reflector
                auto reduce_stage = [&](auto stage, int last) __attribute__((always_inline)) {
                    constexpr int ST = decltype(stage)::value;
                    const int j1 = min(32 * ST + 31, last);
#pragma unroll 1
                    for (; J <= j1; ++J) {
                        const int j = J;
                        float *po = pl + (j & 1) * D, *kp = kpart + (j & 1) * ALG_NG;
                        AlgRow<D> v, x;
                        __syncthreads();                               // reflector j is there
                        alg_load<D, ST>(v, Y + j * D, c16);
                        alg_product<D, ST>(M, v, Y + j * D, po, kp, grp, c16);
                        {
                            const float s = -2.f * half_sum(alg_dot<D, ST>(aux, v));
#pragma unroll
                            for (int q = ST; q < NQ; ++q) aux[q] = fma2(pk(s, s), v[q], aux[q]);
                        }
                        __syncthreads();                               // p is there
                        alg_update<D, ST>(M, v, Y + j * D, po, kp, grp, c16, j & (SH::RPS - 1), x);
                        alg_row_done<D, ST>(x, j, tiny2, Y, ta, tb, grp, lane);
                    }
                };
                float *sa = WS, *sb2 = WS + D + 8, *vec = WS + 2 * (D + 8);   // vec: per wanted eigenvector dd, dl, du, du2, pv, y of D each
                // Whether the J - m rows of the tridiagonal form so far hold the wanted eigenpairs and the next one: 0, else in how many rows to
                // ask again (D: not at all).  With sigma just below the next one, M has as many eigenvalues above sigma as the leading part T
                // (Sylvester, block elimination of T - sigma) if the rest, R + b b^T / |d|, has none: b is the coupling to the rest, d < 0 the
                // last pivot of T - sigma.  The largest eigenvalue of R follows from its trace and Frobenius norm, which are those of M less T's:
                //   lambda <= t / N + sqrt((N - 1) / N (f^2 - t^2 / N)).
                // That is a count, and says nothing about which rows the vectors live in: a large eigenvalue may have come into the form after
                // smaller ones.  So the last entry of every wanted vector and of the next one, times the coupling, has to be nothing
                // beside rounding: from the recurrence for the vector upwards from its last entry, at both ends of the interval that holds
                // the eigenvalue, a lane for each.
                float *was = misc + 12 + 2 * warp;                     // a warp's: the rest's bound when last asked, and after how many rows
                if (lane == 0) was[1] = 0.f;
                auto leading_part_suffices = [&]() __attribute__((always_inline)) {
                    const int sz = warp_uniform(J - m), r = min(p.rank, D);
                    const float *da = ta + m, *db = tb + m;
                    __syncthreads();                                   // the entries are there
                    float s1 = 0.f, s2 = 0.f, gb = 0.f;
                    for (int i = lane; i < sz; i += 32) {
                        s1 += da[i];
                        s2 = fmaf(da[i], da[i], fmaf(2.f * db[i], db[i], s2));
                        gb = fmaxf(gb, fabsf(da[i]) + (i > 0 ? fabsf(db[i - 1]) : 0.f) + (i + 1 < sz ? fabsf(db[i]) : 0.f));
                    }
                    s1 = warp_sum(s1);
                    s2 = warp_sum(s2);
                    gb = fmaxf(warp_max(gb), 1e-30f);
                    const float scl = 1.f / gb, nr = (float)(D - J), t = trM - s1, f2 = m2 - s2 + 1e-5f * m2;
                    const float rest = (t / nr + sqrtf((nr - 1.f) / nr * fmaxf(f2 - t * t / nr, 0.f)) + 1e-5f * trM / nr) * scl, cb = fabsf(db[sz - 1]) * scl;
                    float *vb = vec + 4, *vi = vb + D + 4;             // couplings (a zero before and after them) and their reciprocals
                    bool suffice = false;
                    float sigma = 1.f;                                 // (T's eigenvalues are at most one, in units of gb)
                    if (warp_uniform(rest < 1.f)) {
                        const int n4 = (sz + 3) / 4;
                        if (tid < 4 * n4) {
                            const float b = (tid > 0 && tid < sz) ? db[tid - 1] * scl : 0.f;
                            sa[tid] = tid < sz ? da[tid] * scl : 2.f;
                            sb2[tid] = (tid > 0 && tid < sz) ? fmaxf(b * b, 1e-14f) : 0.f;
                            vb[tid - 1] = b;
                            if (tid > 0) vi[tid - 1] = 1.f / b;
                            if (tid + 1 == sz) vb[tid] = 0.f;
                        }
                        __syncthreads();
                        constexpr float STEP = 1.f / (2 * ALG_NT + 1);
                        uint16_t *cnt = reinterpret_cast<uint16_t *>(ipq);
                        int c0, c1;
                        sturm_count2(sa, sb2, n4, STEP * (2 * tid + 1), STEP * (2 * tid + 2), c0, c1);
                        cnt[tid] = (uint16_t)(c0 | c1 << 8);
                        __syncthreads();
                        // shifts not above eigenvalue e, the largest being number 0
                        auto shifts_up_to = [&](int e) __attribute__((always_inline)) {
                            int s = 0;
#pragma unroll
                            for (int i = 0; i < ALG_NW; ++i) {
                                const uint32_t two = cnt[lane + 32 * i];
                                s += ((int)(two & 255) < sz - e ? 1 : 0) + ((int)(two >> 8) < sz - e ? 1 : 0);
                            }
                            return __reduce_add_sync(0xffffffffu, s);
                        };
                        const int nx = shifts_up_to(r);
                        sigma = STEP * (float)nx;
                        if (warp_uniform(nx > 0 && rest * 1.0001f < sigma)) {
                            int at = nx;
#pragma unroll 1
                            for (int e = 0; e < r; ++e) {
                                const int s = shifts_up_to(e);
                                if (lane == e) at = s;
                            }
                            // Lanes 0 .. r: upwards, at both ends of their eigenvalue's interval, as far as the ends agree in sign: where they do not, an
                            // eigenvalue of the rows below lies between them and what follows says nothing (a form that falls apart, where the
                            // eigenvalue belongs to its lower part).  As far as they do, none lies there (from one row to the next their number
                            // changes by one at most), and an entry is nowhere between the ends smaller than at the smaller of them: a product of
                            // distances from points outside.  Last lane: downwards at sigma, for the last pivot.
                            const bool down = lane == 31;
                            const float sg = STEP * (float)at, sh = down ? sg : sg + STEP;
                            float y1 = 1.f, y0 = 0.f, z1 = 1.f, z0 = 0.f, top = 1.f;
                            bool live = true;
                            const int by = down ? 1 : -1;
                            const float *pa = down ? sa : sa + sz - 1, *pb = down ? vb - 1 : vb + sz - 1, *pi = down ? vi : vi + sz - 2;
#pragma unroll 4
                            for (int k = 1; k < sz; ++k, pa += by, pb += by, pi += by) {
                                const float a = *pa, b = *pb, ib = *pi;
                                const float y = -fmaf(a - sg, y1, b * y0) * ib, z = -fmaf(a - sh, z1, b * z0) * ib;
                                live = live && top < 1e25f && (y > 0.f ? z > 0.f : y < 0.f && z < 0.f);
                                const float f = down && fabsf(y) > 1e20f ? 1e-20f : 1.f;           // (downwards the quotient counts)
                                if (live) {
                                    y0 = y1 * f;
                                    y1 = y * f;
                                    z0 = z1 * f;
                                    z1 = z * f;
                                    top = fmaxf(top, fminf(fabsf(y1), fabsf(z1)));
                                }
                            }
                            const float d = (sa[sz - 1] - sg) + vb[sz - 2] * (y0 / y1);
                            const float d2 = __shfl_sync(0xffffffffu, live ? d : 1.f, 31);
                            const bool gone = lane < r ? cb <= 1e-9f * top : lane == r ? cb <= 1e-6f * top : true;
                            suffice = d2 < 0.f && (rest - cb * cb / d2) * 1.0001f < sigma && __all_sync(0xffffffffu, gone);
                        }
                    }
                    if (warp_uniform(suffice)) return 0;
                    // A line through the last two bounds of the rest, which comes down ever more slowly, tells when it will be down at sigma.
                    const float now = rest * gb, above = now - sigma * gb;
                    int rows = max(ALG_EXIT_STEP, rest > fminf(1.3f * sigma, 1.f) ? sz / 2 : sz / 4);
                    if (was[1] > 0.f && above > 0.f &&
                        (float)sz + ALG_EXIT_BEND * above * ((float)sz - was[1]) / fmaxf(was[0] - now, 1e-3f * now) > ALG_EXIT_SHARE * (float)(D - m)) rows = D;
                    __syncwarp();
                    if (lane == 0) {
                        was[0] = now;
                        was[1] = (float)sz;
                    }
                    return warp_uniform(rows);
                };
                int early = 0, more;
#pragma unroll 1
                do {
                    if (last > D - 2 - 2 * ALG_EXIT_STEP) last = D - 2;
                    reduce_stage(std::integral_constant<int, 0>{}, last);
                    reduce_stage(std::integral_constant<int, 1>{}, last);
                    if constexpr (D > 64) {
                        reduce_stage(std::integral_constant<int, D / 32 - 2>{}, last);
                        reduce_stage(std::integral_constant<int, D / 32 - 1>{}, last);
                    }
                    more = 0;
                    if (ASKS && last < D - 2) {
                        more = leading_part_suffices();
                        early = more ? 0 : 1;
                        last += more;
                    }
                    more = warp_uniform(more);
                } while (more);
                early = warp_uniform(early);
                const int through = warp_uniform(early ? J - 1 : D - 2);     // the last reflector of the form
                n = warp_uniform(early ? J - m : n);
                if (!early) {
                    // the last diagonal entry
                    float a, b;
                    upk(M[RW - 1][NQ - 1], a, b);
                    if (grp == SH::owner(D - 1) && c16 == 15) ta[D - 1] = b;
                }
                if (grp == 0) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) *reinterpret_cast<f32x2 *>(vu + 32 * q + 2 * c16) = aux[q];
                }
                __syncthreads();
                const int ne = min(min(p.rank, D) + 1, n);             // eigenvalues computed: the wanted ones and the next
                const int rmax = min(min(p.rank, D), n);
                const int n4 = (n + 3) / 4;
                const float *da = ta + m, *db = tb + m;                // db[i] couples i and i + 1, i < n - 1
                // bounds of the spectrum (Gershgorin); the recurrences run on the matrix scaled by their larger one
                float gb = 0.f;
                if (tid < n) gb = fabsf(da[tid]) + (tid > 0 ? fabsf(db[tid - 1]) : 0.f) + (tid < n - 1 ? fabsf(db[tid]) : 0.f);
                const float bound = fmaxf(block_max<ALG_NT>(gb, red), 1e-30f), scl = 1.f / bound;
                if (tid < 4 * n4) {
                    sa[tid] = tid < n ? da[tid] * scl : 2.f;
                    const float b = (tid > 0 && tid < n) ? db[tid - 1] * scl : 0.f;        // couples tid - 1 and tid
                    sb2[tid] = (tid > 0 && tid < n) ? fmaxf(b * b, 1e-14f) : 0.f;
                }
                __syncthreads();
                // eigenvalue e (largest first) by 65-way multisection, one warp each, two shifts per lane
                for (int e = warp; e < ne; e += ALG_NW) {
                    const int want = n - 1 - e;                        // it has exactly `want` eigenvalues below it
                    float lo = -0.001f, hi = 1.001f;                   // (R^T R has no negative eigenvalues beyond rounding)
#pragma unroll 1
                    for (int round = 0; round < 4; ++round) {          // 65^-4 of the interval: 5.6e-8 of the largest eigenvalue's bound
                        const float step = (hi - lo) * (1.f / 65.f);
                        const float x0 = fmaf(step, (float)(2 * lane + 1), lo), x1 = fmaf(step, (float)(2 * lane + 2), lo);
                        int c0, c1;
                        sturm_count2(sa, sb2, n4, x0, x1, c0, c1);
                        // shifts not above the eigenvalue: the counts are monotone in x
                        const int nl = __popc(__ballot_sync(0xffffffffu, c0 <= want)) + __popc(__ballot_sync(0xffffffffu, c1 <= want));
                        const float nlo = fmaf(step, (float)nl, lo), nhi = fmaf(step, (float)(nl + 1), lo);
                        if (nl > 0) lo = nlo;
                        if (nl < 64) hi = nhi;
                    }
                    if (lane == 0) tlam[e] = 0.5f * (lo + hi);         // in units of `bound`
                }
                __syncthreads();
                const float l1 = tlam[0];
                while (rho < rmax && tlam[rho] > EIG_RANK_TOL * l1 && tlam[rho] > 0.f) ++rho;
                rho = warp_uniform(rho);
                const float unit = misc[10];
                lam1 = l1 * bound * unit;
                lam_rho = rho > 0 ? tlam[rho - 1] * bound * unit : 0.f;
                lam_next = rho < ne ? fmaxf(tlam[rho] * bound, 0.f) * unit : 0.f;
                for (int t = 0; t < rho; ++t) revr += tlam[t];
                revr *= bound * unit / (trM * unit + p.eps);                         // trace of R^T R = sum of all its eigenvalues
                bool clustered = false;
                for (int t = 1; t < rho; ++t) clustered = clustered || tlam[t - 1] - tlam[t] <= EIG_CLUSTER_TOL * fabsf(l1);
                clustered = warp_uniform(clustered);
                // one warp, in order of the eigenvalues: orthogonal to the neighbours before it that are closer than tol, unit length
                auto orthogonal = [&](float tol) __attribute__((always_inline)) {
                    for (int j = 1; j < rho; ++j) {
                        float *y = vec + (j * 6 + 5) * D;
                        for (int i2 = 0; i2 < j; ++i2) {
                            if (warp_uniform(fabsf(tlam[i2] - tlam[j]) > tol * fabsf(l1))) continue;
                            const float *z = vec + (i2 * 6 + 5) * D;
                            float dsum = 0.f;
                            for (int cc = lane; cc < n; cc += 32) dsum = fmaf(y[cc], z[cc], dsum);
                            dsum = warp_sum(dsum);
                            for (int cc = lane; cc < n; cc += 32) y[cc] -= dsum * z[cc];
                            __syncwarp();
                        }
                        float n2 = 0.f;
                        for (int cc = lane; cc < n; cc += 32) n2 = fmaf(y[cc], y[cc], n2);
                        n2 = warp_sum(n2);
                        const float inv = n2 > 0.f ? rsqrtf(n2) : 0.f;
                        for (int cc = lane; cc < n; cc += 32) y[cc] *= inv;
                        __syncwarp();
                    }
                };
                // Close neighbours: inverse iteration on the scaled T: factor T - lambda I once (LU with row interchanges), three solves; the operands of four steps are fetched together, ahead of the chain that needs them
                constexpr float PERT = 4e-7f;
                if (!clustered) {
                    // Isolated eigenvalues: twisted factorisation.  Lane 0 eliminates from the top, lane 1 from the bottom, at
                    // the same time; where the two meet with the smallest remainder gamma the eigenvector has its largest
                    // entry, and its other entries follow outwards by multiplication alone (Fernando's method).  The residual
                    // is gamma over the vector's length; should it exceed 2e-7 of the spectrum's bound the inverse iteration
                    // below takes over.  gamma is about the shift's error, a few 1e-8 of the bound, and a neighbour's share of the
                    // vector is that over its distance (2e-5 of delta for one at 2e-3): with a neighbour, wanted or not, within
                    // EIG_NEAR_TOL one step of inverse iteration with the same factors squares that away, down to what T's own
                    // rounding leaves, at two multiply-adds per entry and no division, and wanted neighbours are made orthogonal.
                    // Farther ones leave less than 1e-6.  Each lane's operands lie in the order it needs them, four to a load.
                    // (Every lane computes, even ones the upper arm and odd ones the lower, and two of them store: a warp that enters a loop
                    // with two lanes only pays for it at every shuffle behind.)
                    constexpr float PIV = 1e-10f;
                    constexpr int PL = D / 32;                         // entries a lane holds
                    const bool lower = lane & 1;
                    if (tid == 0) misc[7] = 0.f;
                    __syncthreads();
                    for (int e = warp; e < rho; e += ALG_NW) {
                        float *pa = vec + e * 6 * D, *pb = pa + D, *qa = pb + D, *qb = qa + D, *y = pa + 5 * D;
                        const float lam = tlam[e];
#pragma unroll
                        for (int q = 0; q < PL; ++q) {
                            const int i = lane + 32 * q;
                            const bool on = i < n - 1;
                            const float bu = on ? db[i] * scl : 0.f, bd = on ? db[n - 2 - i] * scl : 0.f;
                            pa[i] = i < n ? sa[i] - lam : 1.f;
                            qa[i] = i < n ? sa[n - 1 - i] - lam : 1.f;
                            pb[i] = bu * bu;
                            qb[i] = bd * bd;
                        }
                        __syncwarp();
                        {
                            float *a = lower ? qa : pa;
                            const float *b = lower ? qb : pb;
                            float4 an = *reinterpret_cast<const float4 *>(a);
                            float d = an.x;
#pragma unroll 1
                            for (int t = 0; t < n4; ++t) {
                                const float4 ac = an, bc = *reinterpret_cast<const float4 *>(b + 4 * t);
                                an = *reinterpret_cast<const float4 *>(a + 4 * t + 4);
                                const float ax[4] = {ac.y, ac.z, ac.w, an.x}, bx[4] = {bc.x, bc.y, bc.z, bc.w};
                                float o[4];
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    d = copysignf(fmaxf(fabsf(d), PIV), d);
                                    o[q] = d;
                                    d = fmaf(-bx[q], rcp_approx(d), ax[q]);
                                }
                                if (lane < 2) *reinterpret_cast<float4 *>(a + 4 * t) = make_float4(o[0], o[1], o[2], o[3]);
                            }
                        }
                        __syncwarp();
                        float best = INFINITY;
                        int at = 0;
#pragma unroll
                        for (int q = 0; q < PL; ++q) {
                            const int i = lane + 32 * q;
                            const float gm = i < n ? fabsf(pa[i] + qa[n - 1 - i] - (sa[i] - lam)) : INFINITY;
                            if (gm < best) { best = gm; at = i; }
                        }
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) {
                            const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                            const int oa = __shfl_xor_sync(0xffffffffu, at, o);
                            if (ob < best || (ob == best && oa < at)) { best = ob; at = oa; }
                        }
                        // the multipliers along both arms and the pivots' reciprocals, from the twist outwards
                        const float gam = pa[at] + qa[n - 1 - at] - (sa[at] - lam);
                        float rt[PL], rb[PL];
#pragma unroll
                        for (int q = 0; q < PL; ++q) {
                            const int i = lane + 32 * q, u = at - 1 - i, w = at + 1 + i;
                            rt[q] = u >= 0 ? rcp_approx(pa[u]) : 0.f;
                            rb[q] = w < n ? rcp_approx(qa[n - 1 - w]) : 0.f;
                        }
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < PL; ++q) {
                            const int i = lane + 32 * q, u = at - 1 - i, w = at + 1 + i;
                            pa[i] = rt[q];
                            qa[i] = rb[q];
                            pb[i] = u >= 0 ? -db[u] * scl * rt[q] : 0.f;
                            qb[i] = w < n ? -db[w - 1] * scl * rb[q] : 0.f;
                        }
                        __syncwarp();
                        const float *mu = lower ? qb : pb, *rc = lower ? qa : pa;
                        float *x = lower ? y : pa + 4 * D;
                        // (both arms as far as the longer one: what lies behind an arm's end is zero)
                        const int len = warp_uniform(max(n - 1 - at, at));
                        float n1 = 0.f, z = 1.f;                       // n1: squares of the first vector's entries; z: the entry at the twist
                        {
                            float c = 1.f;
#pragma unroll 1
                            for (int t = 0; t < len; t += 4) {
                                const float4 mv = *reinterpret_cast<const float4 *>(mu + t);
                                float4 o;
                                o.x = mv.x * c; o.y = mv.y * o.x; o.z = mv.z * o.y; c = o.w = mv.w * o.z;
                                n1 = fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, fmaf(o.w, o.w, n1))));
                                if (lane < 2) *reinterpret_cast<float4 *>(x + t) = o;
                            }
                        }
                        const bool close = (e > 0 && tlam[e - 1] - lam < EIG_NEAR_TOL * l1) || (e + 1 < ne && lam - tlam[e + 1] < EIG_NEAR_TOL * l1);
                        if (warp_uniform(close)) {
                            // the step of inverse iteration: along both arms to the twist ..
                            float g = 0.f, mn = 0.f;
#pragma unroll 1
                            for (int t = (len + 3) / 4 * 4 - 4; t >= 0; t -= 4) {
                                const float4 xv = *reinterpret_cast<const float4 *>(x + t), mv = *reinterpret_cast<const float4 *>(mu + t);
                                float4 o;
                                o.w = fmaf(mn, g, xv.w); o.z = fmaf(mv.w, o.w, xv.z); o.y = fmaf(mv.z, o.z, xv.y); g = o.x = fmaf(mv.y, o.y, xv.x);
                                mn = mv.x;
                                if (lane < 2) *reinterpret_cast<float4 *>(x + t) = o;
                            }
                            g *= mn;
                            __syncwarp();
                            // .. across it and back
                            z = (1.f + __shfl_sync(0xffffffffu, g, 0) + __shfl_sync(0xffffffffu, g, 1)) * rcp_approx(copysignf(fmaxf(fabsf(gam), PIV), gam));
                            float c = z;
#pragma unroll 1
                            for (int t = 0; t < len; t += 4) {
                                const float4 xv = *reinterpret_cast<const float4 *>(x + t), mv = *reinterpret_cast<const float4 *>(mu + t);
                                const float4 rv = *reinterpret_cast<const float4 *>(rc + t);
                                float4 o;
                                o.x = fmaf(mv.x, c, xv.x * rv.x); o.y = fmaf(mv.y, o.x, xv.y * rv.y);
                                o.z = fmaf(mv.z, o.y, xv.z * rv.z); c = o.w = fmaf(mv.w, o.z, xv.w * rv.w);
                                if (lane < 2) *reinterpret_cast<float4 *>(x + t) = o;
                            }
                        }
                        __syncwarp();
                        n1 = 1.f + __shfl_sync(0xffffffffu, n1, 0) + __shfl_sync(0xffffffffu, n1, 1);
                        float yv[PL], n2 = 0.f;
                        // (z is about 1 / gamma: the entries are brought to the first vector's scale before they are squared)
                        const float zr = rcp_approx(z);
#pragma unroll
                        for (int q = 0; q < PL; ++q) {
                            const int i = lane + 32 * q;
                            yv[q] = i < n ? zr * (i == at ? z : i < at ? pa[4 * D + at - 1 - i] : y[i - at - 1]) : 0.f;
                            n2 = fmaf(yv[q], yv[q], n2);
                        }
                        n2 = warp_sum(n2);
                        const float inv = rsqrtf(n2);
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < PL; ++q)
                            if (lane + 32 * q < n) y[lane + 32 * q] = yv[q] * inv;
                        if (lane == 0 && !(best * rsqrtf(n1) <= 2e-7f)) misc[7] = 1.f;
                    }
                    __syncthreads();
                    clustered = warp_uniform(misc[7] != 0.f);
                    bool near = false;
                    for (int t = 1; t < rho; ++t) near = near || tlam[t - 1] - tlam[t] < EIG_NEAR_TOL * l1;
                    if (warp_uniform(near) && !clustered) {
                        if (warp == 0) orthogonal(EIG_NEAR_TOL);
                        __syncthreads();
                    }
                }
                for (int e = warp; clustered && e < rho; e += ALG_NW) {
                    float *dd = vec + e * 6 * D, *dl = dd + D, *du = dl + D, *du2 = du + D, *pv = du2 + D, *y = pv + D;
                    const float lam = tlam[e];
                    for (int i = lane; i < 4 * n4; i += 32) {
                        dd[i] = i < n ? sa[i] - lam : 1.f;
                        du[i] = i < n - 1 ? db[i] * scl : 0.f;         // entry (i, i + 1), and (i + 1, i)
                        // a start vector without structure
                        const uint32_t hsh = ((uint32_t)i * 2654435761u + (uint32_t)e * 40503u + 12345u) >> 8;
                        y[i] = i < n ? (float)(hsh & 0xFFFFu) * (1.f / 65536.f) - 0.5f : 0.f;
                    }
                    __syncwarp();
                    if (lane == 0) {
                        // the running pivot (di) and the entry right of it (ui)
                        float di = dd[0], ui = du[0];
                        float4 dn4 = *reinterpret_cast<const float4 *>(dd), un4 = *reinterpret_cast<const float4 *>(du);
#pragma unroll 1
                        for (int q = 0; q < n4; ++q) {
                            const float4 dc = dn4, uc = un4;
                            if (q + 1 < n4) {
                                dn4 = *reinterpret_cast<const float4 *>(dd + 4 * q + 4);
                                un4 = *reinterpret_cast<const float4 *>(du + 4 * q + 4);
                            }
                            const float li_[4] = {uc.x, uc.y, uc.z, uc.w};
                            const float dx[4] = {dc.y, dc.z, dc.w, dn4.x}, ux[4] = {uc.y, uc.z, uc.w, un4.x};
                            float o_d[4], o_l[4], o_u[4], o_u2[4], o_p[4];
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                const int i = 4 * q + t;
                                const float li = i < n - 1 ? li_[t] : 0.f;
                                const float dn = i < n - 1 ? dx[t] : 1.f, un = i < n - 2 ? ux[t] : 0.f;
                                const bool keep = fabsf(di) >= fabsf(li);
                                float den = keep ? di : li;
                                if (fabsf(den) < PERT) den = den < 0.f ? -PERT : PERT;
                                const float num = keep ? li : di;
                                const float rc = rcp_approx(den), f = num * rc;
                                o_d[t] = rc;                           // the solves multiply by the pivots' reciprocals
                                o_l[t] = f;
                                o_p[t] = keep ? 0.f : 1.f;
                                o_u[t] = keep ? ui : dn;
                                o_u2[t] = keep ? 0.f : un;
                                const float nd = keep ? fmaf(-f, ui, dn) : fmaf(-f, dn, ui);
                                ui = keep ? un : -f * un;
                                di = nd;
                            }
                            *reinterpret_cast<float4 *>(dd + 4 * q) = make_float4(o_d[0], o_d[1], o_d[2], o_d[3]);
                            *reinterpret_cast<float4 *>(dl + 4 * q) = make_float4(o_l[0], o_l[1], o_l[2], o_l[3]);
                            *reinterpret_cast<float4 *>(du + 4 * q) = make_float4(o_u[0], o_u[1], o_u[2], o_u[3]);
                            *reinterpret_cast<float4 *>(du2 + 4 * q) = make_float4(o_u2[0], o_u2[1], o_u2[2], o_u2[3]);
                            *reinterpret_cast<float4 *>(pv + 4 * q) = make_float4(o_p[0], o_p[1], o_p[2], o_p[3]);
                        }
                    }
                    __syncwarp();
                }
#pragma unroll 1
                for (int itn = 0; itn < (clustered ? 3 : 0); ++itn) {
                    for (int e = warp; e < rho; e += ALG_NW) {
                        float *dd = vec + e * 6 * D, *dl = dd + D, *du = dl + D, *du2 = du + D, *pv = du2 + D, *y = pv + D;
                        if (lane == 0) {
                            float yi = y[0];
                            float4 yn4 = *reinterpret_cast<const float4 *>(y), ln4 = *reinterpret_cast<const float4 *>(dl);
                            float4 pn4 = *reinterpret_cast<const float4 *>(pv);
#pragma unroll 1
                            for (int q = 0; q < n4; ++q) {
                                const float4 yc = yn4, lc = ln4, pc4 = pn4;
                                if (q + 1 < n4) {
                                    yn4 = *reinterpret_cast<const float4 *>(y + 4 * q + 4);
                                    ln4 = *reinterpret_cast<const float4 *>(dl + 4 * q + 4);
                                    pn4 = *reinterpret_cast<const float4 *>(pv + 4 * q + 4);
                                } else {
                                    yn4.x = 0.f;
                                }
                                const float yx[4] = {yc.y, yc.z, yc.w, yn4.x}, ll[4] = {lc.x, lc.y, lc.z, lc.w}, pp[4] = {pc4.x, pc4.y, pc4.z, pc4.w};
                                float o[4];
#pragma unroll
                                for (int t = 0; t < 4; ++t) {
                                    const float a0 = fmaf(-ll[t], yi, yx[t]), b0 = fmaf(-ll[t], yx[t], yi);
                                    o[t] = pp[t] == 0.f ? yi : yx[t];
                                    yi = pp[t] == 0.f ? a0 : b0;
                                }
                                *reinterpret_cast<float4 *>(y + 4 * q) = make_float4(o[0], o[1], o[2], o[3]);
                            }
                            float y0 = 0.f, y1 = 0.f;                  // y[i + 1], y[i + 2]
                            float4 yb = *reinterpret_cast<const float4 *>(y + 4 * n4 - 4), db4 = *reinterpret_cast<const float4 *>(dd + 4 * n4 - 4);
                            float4 ub = *reinterpret_cast<const float4 *>(du + 4 * n4 - 4), vb = *reinterpret_cast<const float4 *>(du2 + 4 * n4 - 4);
#pragma unroll 1
                            for (int q = n4 - 1; q >= 0; --q) {
                                const float yy[4] = {yb.x, yb.y, yb.z, yb.w}, iv[4] = {db4.x, db4.y, db4.z, db4.w};
                                const float uu[4] = {ub.x, ub.y, ub.z, ub.w}, u2[4] = {vb.x, vb.y, vb.z, vb.w};
                                if (q > 0) {
                                    yb = *reinterpret_cast<const float4 *>(y + 4 * q - 4);
                                    db4 = *reinterpret_cast<const float4 *>(dd + 4 * q - 4);
                                    ub = *reinterpret_cast<const float4 *>(du + 4 * q - 4);
                                    vb = *reinterpret_cast<const float4 *>(du2 + 4 * q - 4);
                                }
                                float o[4];
#pragma unroll
                                for (int t = 3; t >= 0; --t) {
                                    const float s = fmaf(-uu[t], y0, fmaf(-u2[t], y1, yy[t])) * iv[t];
                                    o[t] = s;
                                    y1 = y0;
                                    y0 = s;
                                }
                                *reinterpret_cast<float4 *>(y + 4 * q) = make_float4(o[0], o[1], o[2], o[3]);
                            }
                        }
                        __syncwarp();
                        // scaled to largest entry 1, then to unit length, by the whole warp (padding entries are zero)
                        float mx = 0.f;
                        for (int i = lane; i < n; i += 32) mx = fmaxf(mx, fabsf(y[i]));
                        mx = warp_max(mx);
                        const float sc1 = mx > 0.f ? 1.f / mx : 1.f;
                        float n2 = 0.f;
                        for (int i = lane; i < n; i += 32) { const float t = y[i] * sc1; n2 = fmaf(t, t, n2); }
                        n2 = warp_sum(n2);
                        const float inv = n2 > 0.f ? rsqrtf(n2) * sc1 : 0.f;
                        for (int i = lane; i < 4 * n4; i += 32) y[i] = i < n ? y[i] * inv : 0.f;
                        __syncwarp();
                    }
                    if (clustered) {
                        __syncthreads();
                        if (warp == 0) orthogonal(EIG_CLUSTER_TOL);
                        __syncthreads();
                    }
                }
                // r_bar's products with the eigenvectors, in the coordinates of the tridiagonal form
                for (int e = warp; e < rho; e += ALG_NW) {
                    const float *y = vec + (e * 6 + 5) * D;
                    float s = 0.f;
                    for (int i = lane; i < n; i += 32) s = fmaf(y[i], vu[m + i], s);
                    s = warp_sum(s);
                    if (lane == 0) vc[e] = s * inv_del;
                }
                __syncthreads();
                if (tid < D) {
                    float s = 0.f;
                    if (tid >= m && tid < m + n)
                        for (int t = 0; t < rho; ++t) s = fmaf(vc[t], vec[(t * 6 + 5) * D + tid - m], s);
                    vx[tid] = s;
                }
                back = through;
                done = true;
            }

            // r_bar in the rotated coordinates, for the other two routes
            if (!done) {
                if (grp == 0) {
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int cc = 32 * q + 2 * c16;
                        float a, b;
                        upk(aux[q], a, b);
                        vu[cc] = cc >= m ? a * inv_del : 0.f;
                        vu[cc + 1] = cc + 1 >= m ? b * inv_del : 0.f;
                    }
                }
                __syncthreads();
            }

            // ---- 3f. fast path of App. H: C <- orth(C M), a fixed number of times, from the first rows of the identity ----
            if (!done && p.fast_iters > 0) {
                int rho_f = min(min(p.rank, D), D - m);               // rank(R) <= d - m
                float *C = WS, *Yb = WS + min(p.rank, D) * D;         // row blocks; entries below m stay zero in C
                // the rows of the identity in the rotated coordinates: e_i H_0 .. H_{m-1} (what lies below m meets only zeros of M)
#pragma unroll 1
                for (int i0 = 0; i0 < rho_f; i0 += ALG_NG) {
                    const int i = i0 + grp;
                    AlgRow<D> x, v;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) x[q] = pk(32 * q + 2 * c16 == i ? 1.f : 0.f, 32 * q + 2 * c16 + 1 == i ? 1.f : 0.f);
#pragma unroll 1
                    for (int j = 0; j < m; ++j) { alg_load<D>(v, Y + j * D, c16); reflect(x, v); }
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int cc = 32 * q + 2 * c16;
                        float a, b;
                        upk(x[q], a, b);
                        if (i < rho_f) *reinterpret_cast<f32x2 *>(C + i * D + cc) = pk(cc >= m ? a : 0.f, cc + 1 >= m ? b : 0.f);
                    }
                }
                // Y = 2 C M from the registers (the factor drops out of the directions)
                auto times_m = [&](int rows) __attribute__((always_inline)) {
                    __syncthreads();
#pragma unroll 1
                    for (int i = 0; i < rows; ++i) {
                        AlgRow<D> v;
                        alg_load<D>(v, C + i * D, c16);
                        auto one = [&](auto stage) __attribute__((always_inline)) {
                            alg_product<D, decltype(stage)::value>(M, v, nullptr, Yb + i * D, nullptr, grp, c16);
                        };
                        if (D > 64 && m >= 96) one(std::integral_constant<int, D / 32 - 1>{});
                        else if (D > 64 && m >= 64) one(std::integral_constant<int, D / 32 - 2>{});
                        else if (m >= 32) one(std::integral_constant<int, 1>{});
                        else one(std::integral_constant<int, 0>{});
                    }
                    __syncthreads();
                };
#pragma unroll 1
                for (int itn = 0; itn < p.fast_iters; ++itn) {
                    times_m(rho_f);
                    // orth: Gram-Schmidt over the rows in order, twice; a row with nothing left is dropped (warp 0)
                    if (warp == 0) {
                        int kept = 0;
                        for (int i = 0; i < rho_f; ++i) {
                            // a lane's entries: lane, lane + 32, ..
                            float y[NQ], n0 = 0.f, n1 = 0.f;
#pragma unroll
                            for (int q = 0; q < NQ; ++q) { y[q] = 32 * q + lane >= m ? Yb[i * D + 32 * q + lane] : 0.f; n0 = fmaf(y[q], y[q], n0); }
                            n0 = warp_sum(n0);
                            for (int pass = 0; pass < 2; ++pass)
                                for (int j = 0; j < kept; ++j) {
                                    float dsum = 0.f;
#pragma unroll
                                    for (int q = 0; q < NQ; ++q) dsum = fmaf(y[q], C[j * D + 32 * q + lane], dsum);
                                    dsum = warp_sum(dsum);
#pragma unroll
                                    for (int q = 0; q < NQ; ++q) y[q] = fmaf(-dsum, C[j * D + 32 * q + lane], y[q]);
                                }
#pragma unroll
                            for (int q = 0; q < NQ; ++q) n1 = fmaf(y[q], y[q], n1);
                            n1 = warp_sum(n1);
                            if (warp_uniform(n1 > 1e-10f * n0 && n1 > 0.f)) {
                                const float inv = rsqrtf(n1);
#pragma unroll
                                for (int q = 0; q < NQ; ++q) C[kept * D + 32 * q + lane] = y[q] * inv;
                                ++kept;
                            }
                        }
                        if (lane == 0) misc[6] = (float)kept;
                    }
                    __syncthreads();
                    rho_f = warp_uniform((int)misc[6]);
                }
                rho = rho_f;
                // Rayleigh quotients of the rows (for the diagnostics), then Delta and delta
                if (c.diag) times_m(rho);
                for (int i = warp; i < rho; i += ALG_NW) {
                    float rq = 0.f, cu = 0.f;
                    for (int a = lane; a < D; a += 32) {
                        if (c.diag && a >= m) rq = fmaf(C[i * D + a], 0.5f * Yb[i * D + a], rq);
                        cu = fmaf(C[i * D + a], vu[a], cu);
                    }
                    rq = warp_sum(rq);
                    cu = warp_sum(cu);
                    if (lane == 0) { vl[i] = rq; vc[i] = cu; }
                }
                __syncthreads();
                for (int t = 0; t < rho; ++t) revr += vl[t];
                const float unit = misc[10];
                revr *= unit / (trM * unit + p.eps);
                lam1 = rho > 0 ? vl[0] * unit : 0.f; lam_rho = rho > 0 ? vl[rho - 1] * unit : 0.f; lam_next = 0.f;
                if (tid < D) {
                    float sacc = 0.f;
                    for (int t = 0; t < rho; ++t) sacc = fmaf(vc[t], C[t * D + tid], sacc);
                    vx[tid] = sacc;
                }
                back = 0;
                done = true;
            }

            // The last route works on the trailing block in shared memory (zero outside rows and columns >= m)
            float *B2 = WS;
            if (!done) {
#pragma unroll
                for (int r = 0; r < RW; ++r)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int i = SH::row(grp, r), cc = 32 * q + 2 * c16;
                        float a, b;
                        upk(M[r][q], a, b);
                        B2[i * LD + cc] = (i >= m && cc >= m) ? a : 0.f;
                        B2[i * LD + cc + 1] = (i >= m && cc + 1 >= m) ? b : 0.f;
                    }
                __syncthreads();
                for (int e = tid; e < D * D; e += ALG_NT) {            // symmetrise
                    const int a = e / D, bb = e % D;
                    if (a < bb) {
                        const float sy = 0.5f * (B2[a * LD + bb] + B2[bb * LD + a]);
                        B2[a * LD + bb] = sy;
                        B2[bb * LD + a] = sy;
                    }
                }
                __syncthreads();
            }

            // ---- 3b. Jacobi eigen-decomposition of the block (B2), eigenvectors in U -----
            if (!done) {
                float *vcs = vx;                                        // (c, s) of d / 2 pairs
                float *U = B2 + D * LD;                                 // d x d, starts as the identity
                for (int e = tid; e < D * D; e += ALG_NT) U[(e / D) * LD + (e % D)] = (e / D == e % D) ? 1.f : 0.f;
                __syncthreads();
                // rotations below the fp32 noise level of the largest eigenvalue never settle: stop there
                const float floor_abs = 2e-7f * block_max<ALG_NT>(tid < D ? B2[tid * LD + tid] : 0.f, red);
                bool converged = false;
#pragma unroll 1
                for (int sweep = 0; sweep < JACOBI_MAX_SWEEPS && !converged; ++sweep) {
                    if (tid == 0) misc[0] = 0.f;
                    __syncthreads();
#pragma unroll 1
                    for (int r = 0; r < D - 1; ++r) {
                        if (tid < D / 2) {
                            int pp, qq;
                            if (tid == 0) { pp = D - 1; qq = r; }
                            else { pp = (r + tid) % (D - 1); qq = (r - tid + (D - 1)) % (D - 1); }
                            if (pp > qq) { const int t = pp; pp = qq; qq = t; }
                            const float app = B2[pp * LD + pp], aqq = B2[qq * LD + qq], apq = B2[pp * LD + qq];
                            float cs = 1.f, sn = 0.f;
                            if (fabsf(apq) > 1e-7f * sqrtf(fabsf(app * aqq)) + floor_abs) {
                                const float theta = (aqq - app) / (2.f * apq);
                                const float t = (theta >= 0.f ? 1.f : -1.f) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                                cs = rsqrtf(t * t + 1.f);
                                sn = t * cs;
                                misc[0] = 1.f;
                            }
                            vcs[2 * tid] = cs; vcs[2 * tid + 1] = sn;
                            ipq[2 * tid] = pp; ipq[2 * tid + 1] = qq;
                        }
                        __syncthreads();
                        // What a thread meets in a row is one pair of columns, so its rotation is read once, and eight rows are
                        // in flight: 128 threads that took an entry at a time waited for shared memory (4 x 8 heads of 128,
                        // rank 9: 8.9 ms with an entry at a time, 2.6 so).
                        {
                            constexpr int STEP = ALG_NT / (D / 2), INF = 8;           // columns of M and U
                            const int t = tid % (D / 2);
                            const float cs = vcs[2 * t], sn = vcs[2 * t + 1];
                            const int pp = ipq[2 * t], qq = ipq[2 * t + 1];
                            if (sn != 0.f) {
#pragma unroll 1
                                for (int i0 = tid / (D / 2); i0 < D; i0 += INF * STEP) {
                                    float mp[INF], mq[INF], up[INF], uq[INF];
#pragma unroll
                                    for (int u = 0; u < INF; ++u) {
                                        const int i = i0 + u * STEP;
                                        mp[u] = B2[i * LD + pp]; mq[u] = B2[i * LD + qq];
                                        up[u] = U[i * LD + pp]; uq[u] = U[i * LD + qq];
                                    }
#pragma unroll
                                    for (int u = 0; u < INF; ++u) {
                                        const int i = i0 + u * STEP;
                                        B2[i * LD + pp] = cs * mp[u] - sn * mq[u];
                                        B2[i * LD + qq] = sn * mp[u] + cs * mq[u];
                                        U[i * LD + pp] = cs * up[u] - sn * uq[u];
                                        U[i * LD + qq] = sn * up[u] + cs * uq[u];
                                    }
                                }
                            }
                        }
                        __syncthreads();
                        {
                            constexpr int STEP = ALG_NT / D, INF = 8;                 // rows of M
                            const int j = tid % D;
#pragma unroll 1
                            for (int t0 = tid / D; t0 < D / 2; t0 += INF * STEP) {
                                float mp[INF], mq[INF], cs[INF], sn[INF];
                                int pp[INF], qq[INF];
#pragma unroll
                                for (int u = 0; u < INF; ++u) {
                                    const int t = t0 + u * STEP;
                                    cs[u] = vcs[2 * t]; sn[u] = vcs[2 * t + 1];
                                    pp[u] = ipq[2 * t]; qq[u] = ipq[2 * t + 1];
                                    mp[u] = B2[pp[u] * LD + j]; mq[u] = B2[qq[u] * LD + j];
                                }
#pragma unroll
                                for (int u = 0; u < INF; ++u) {
                                    if (sn[u] != 0.f) {
                                        B2[pp[u] * LD + j] = cs[u] * mp[u] - sn[u] * mq[u];
                                        B2[qq[u] * LD + j] = sn[u] * mp[u] + cs[u] * mq[u];
                                    }
                                }
                            }
                        }
                        __syncthreads();
                    }
                    converged = (misc[0] == 0.f);
                    __syncthreads();
                }
                if (!converged) status |= OBF_DEV_NO_CONVERGE;

                // ---- 5. top-rank eigenvectors, Delta, delta ----------------------
                if (tid < D) vl[tid] = B2[tid * LD + tid];
                __syncthreads();
                if (tid == 0) {
                    float l1 = 0.f;
                    for (int i = 0; i < D; ++i) l1 = fmaxf(l1, vl[i]);
                    int n = 0;
                    float last = 0.f, kept = 0.f;
                    const int rmax = min(p.rank, D);
                    while (n < rmax) {
                        int b = -1; float best = EIG_RANK_TOL * l1;
                        for (int i = 0; i < D; ++i) if (vl[i] > best) { best = vl[i]; b = i; }
                        if (b < 0) break;
                        isel[n++] = b; last = vl[b]; kept += vl[b]; vl[b] = -1.f;
                    }
                    float nxt = 0.f;
                    for (int i = 0; i < D; ++i) nxt = fmaxf(nxt, vl[i]);
                    misc[1] = l1; misc[2] = last; misc[3] = nxt; misc[4] = (float)n; misc[5] = kept;
                }
                __syncthreads();
                const float unit = misc[10];
                lam1 = misc[1] * unit; lam_rho = misc[2] * unit; lam_next = misc[3] * unit; rho = (int)misc[4];
                revr = misc[5] * unit / (trM * unit + p.eps);
                if (tid < rho) {
                    const int col = isel[tid];
                    float s = 0.f;
                    for (int cc = 0; cc < D; ++cc) s = fmaf(U[cc * LD + col], vu[cc], s);
                    vc[tid] = s;
                }
                __syncthreads();
                if (tid < D) {
                    float s = 0.f;
                    for (int t = 0; t < rho; ++t) s = fmaf(vc[t], U[tid * LD + isel[t]], s);
                    vx[tid] = s;
                }
                back = 0;
            }
            // Delta in the rotated coordinates (vx, all d of them, zero below m) -> delta, published and injected (Eq. 6-7)
            back = warp_uniform(back);
            if (back >= 0) {
                if (tid < D) pl[tid] = 0.f;
                __syncthreads();
                // (Four at a time, the products among them in the chain as well, 21000 cycles for 126 reflectors of 128 channels; so 17000.)
                // Sixteen reflectors at a time: H_0 .. H_15 x = x + sum_e s_e v_e with s = -2 (I + 2 L)^-1 V x, L the strictly lower
                // part of V V^T.  The triangular matrices of all groups first, a half-warp each; what is left in the chain of a
                // group are its products with x, sixteen multiply-adds and the sum.  v[0] is applied first; past the last one: zeros.
                const int count = (back > m ? back - m : 0) + m;
                const int zero = algebra_y_rows<D>(p.alg_rows, p.rank, p.fast_iters);       // (pl follows Y)
                auto reflector = [&](int l) __attribute__((always_inline)) { return Y + (l < 0 ? zero : l + (l >= m ? 1 : 0)) * D; };
                constexpr int GR = 16, GSZ = GR * GR;
                {
                    const int first = count - 1 - GR * grp;        // of this half-warp's group
                    float *Lg = WS + grp * GSZ;                    // product of v[e] and v[f], f < e, at [f][e]; then the inverse
#pragma unroll 1
                    for (int f0 = 0; f0 < GR && 2 * GR * warp < count; f0 += 8) {
                        AlgRow<D> vf[8];
#pragma unroll
                        for (int f = 0; f < 8; ++f) alg_load<D>(vf[f], reflector(first - f0 - f), c16);
#pragma unroll 1
                        for (int e = f0 + 1; e < GR; e += 2) {     // two rows at a time: their sums travel together
                            AlgRow<D> v, w;
                            float d[16];
                            alg_load<D>(v, reflector(first - e), c16);
                            alg_load<D>(w, reflector(first - e - 1), c16);
#pragma unroll
                            for (int f = 0; f < 8; ++f) {
                                d[f] = alg_dot<D>(v, vf[f]);
                                d[8 + f] = alg_dot<D>(w, vf[f]);
                            }
                            const float tot = transposed_sum<16, 16>(d, c16);
                            if (e + (c16 >> 3) < GR) Lg[(f0 + (c16 & 7)) * GR + e + (c16 >> 3)] = tot;
                        }
                    }
                    __syncwarp();
                    // column c16 of the inverse, by forward substitution
                    float t[GR];
#pragma unroll
                    for (int e = 0; e < GR; ++e) t[e] = e == c16 ? 1.f : 0.f;
#pragma unroll
                    for (int f = 0; f < GR; ++f) {
                        float g[GR];
#pragma unroll
                        for (int e = (f + 1) & ~3; e < GR; e += 4) {
                            const float4 u = *reinterpret_cast<const float4 *>(Lg + f * GR + e);
                            g[e] = u.x; g[e + 1] = u.y; g[e + 2] = u.z; g[e + 3] = u.w;
                        }
                        t[f] *= -2.f;
#pragma unroll
                        for (int e = f + 1; e < GR; ++e) t[e] = fmaf(t[f], g[e], t[e]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int e = 0; e < GR; ++e) Lg[e * GR + c16] = t[e];
                }
                __syncthreads();
                if (warp == 0) {
                    constexpr int PER = D / 32;                    // a lane's entries
                    typedef typename std::conditional<PER == 4, float4, float2>::type Vec;
                    float x[PER];
                    auto load = [&](float (&v)[PER], const float *from) __attribute__((always_inline)) {
                        *reinterpret_cast<Vec *>(v) = *reinterpret_cast<const Vec *>(from + PER * lane);
                    };
                    load(x, vx);
#pragma unroll 1
                    for (int g0 = 0; g0 * GR < count; ++g0) {
                        float v[GR][PER], d[GR], row[GR];
#pragma unroll
                        for (int e = 0; e < GR; ++e) load(v[e], reflector(count - 1 - GR * g0 - e));
#pragma unroll
                        for (int e = 0; e < GR; e += 4) {
                            const float4 t = *reinterpret_cast<const float4 *>(WS + g0 * GSZ + (lane >> 1) * GR + e);
                            row[e] = t.x; row[e + 1] = t.y; row[e + 2] = t.z; row[e + 3] = t.w;
                        }
#pragma unroll
                        for (int e = 0; e < GR; ++e) {
                            d[e] = 0.f;
#pragma unroll
                            for (int q = 0; q < PER; ++q) d[e] = fmaf(v[e][q], x[q], d[e]);
                        }
                        const float tot = transposed_sum<GR, 32>(d, lane);         // v[lane / 2] . x
                        float sa = 0.f, sb = 0.f;
#pragma unroll
                        for (int e = 0; e < GR; e += 2) {
                            sa = fmaf(row[e], __shfl_sync(0xffffffffu, tot, 2 * e), sa);
                            sb = fmaf(row[e + 1], __shfl_sync(0xffffffffu, tot, 2 * e + 2), sb);
                        }
                        sa += sb;
#pragma unroll
                        for (int e = 0; e < GR; ++e) {
                            const float f = __shfl_sync(0xffffffffu, sa, 2 * e);
#pragma unroll
                            for (int q = 0; q < PER; ++q) x[q] = fmaf(f, v[e][q], x[q]);
                        }
                    }
                    float dn = 0.f;
#pragma unroll
                    for (int q = 0; q < PER; ++q) {
                        x[q] *= alpha;
                        dn = fmaf(x[q], x[q], dn);
                    }
                    *reinterpret_cast<Vec *>(vx + PER * lane) = *reinterpret_cast<const Vec *>(x);
                    dn = warp_sum(dn);
                    if (lane == 0) misc[9] = dn;
                }
                __syncthreads();
                const float dn2 = misc[9];
                dnorm = sqrtf(dn2);
                if (!isfinite(dn2)) { status |= OBF_DEV_NONFINITE | OBF_DEV_SKIPPED; dnorm = 0.f; }
                else if (rho == 0 || dn2 == 0.f) status |= OBF_DEV_SKIPPED;
                else {
                    if (tid < D) {
                        p.delta[(size_t)g * D + tid] = vx[tid];
                        if (c.delta_out) c.delta_out[(size_t)lh * D + tid] = vx[tid];
                    }
                    // Eq. 7: V_out = V_keep + delta on every retained row; the fp32 sum is rounded once.  Attn-inject
                    // (App. D.2): row t takes k * A_t / (A_keep + eps) times delta instead
                    constexpr int EPT = 16 / (int)sizeof(TIN);
                    TIN *rows = reinterpret_cast<TIN *>(c.v_out) + (size_t)lh * k * D;
                    const float share = (float)k / (a_keep + p.eps);
                    // (four vectors a thread in flight)
#pragma unroll 1
                    for (int b0 = tid * EPT; b0 < k * D; b0 += 4 * ALG_NT * EPT) {
                        uint4 in[4];
                        float wgt[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int e0 = b0 + u * ALG_NT * EPT;
                            in[u] = e0 < k * D ? *reinterpret_cast<const uint4 *>(rows + e0) : make_uint4(0u, 0u, 0u, 0u);
                            wgt[u] = p.attn_inject && e0 < k * D ? share * A[idx[e0 / D]] : 1.f;
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int e0 = b0 + u * ALG_NT * EPT;
                            if (e0 >= k * D) break;
                            uint4 raw = in[u];
                            const float *dl = vx + e0 % D;
                            if constexpr (sizeof(TIN) == 4) {
                                raw.x = __float_as_uint(fmaf(wgt[u], dl[0], __uint_as_float(raw.x)));
                                raw.y = __float_as_uint(fmaf(wgt[u], dl[1], __uint_as_float(raw.y)));
                                raw.z = __float_as_uint(fmaf(wgt[u], dl[2], __uint_as_float(raw.z)));
                                raw.w = __float_as_uint(fmaf(wgt[u], dl[3], __uint_as_float(raw.w)));
                            } else {
                                uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const float lo = fmaf(wgt[u], dl[2 * q], __uint_as_float(w[q] << 16));
                                    const float hi2 = fmaf(wgt[u], dl[2 * q + 1], __uint_as_float(w[q] & 0xFFFF0000u));
                                    w[q] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
                                           ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi2)) << 16);
                                }
                                raw = make_uint4(w[0], w[1], w[2], w[3]);
                            }
                            *reinterpret_cast<uint4 *>(rows + e0) = raw;
                        }
                    }
                    // the int8 copy that was made with the gather is of the rows before; every thread reads back what it wrote
                    if (c.v_q8)
                        for (int e0 = tid * EPT; e0 < k * D; e0 += ALG_NT * EPT)
                            quantize16<TIN, D>(*reinterpret_cast<const uint4 *>(rows + e0), c.v_q8, c.v_scale, (size_t)lh * k + e0 / D, e0 % D / EPT);
                }
            }
            }
    }

    if (tid == 0) {
        if (status & (OBF_DEV_NONFINITE | OBF_DEV_NO_CONVERGE)) atomicOr(p.status, status & 0xFFu);
        if (c.diag) {
            obf_diag_t *dg = c.diag + lh;
            dg->rcr = rcr; dg->delta_norm = dnorm;
            dg->lam_1 = lam1; dg->lam_rho = lam_rho; dg->lam_next = lam_next;
            dg->span_rank = m; dg->rho_eff = rho; dg->status = status;
            dg->revr = revr; dg->pc = pc;
        }
    }
}

}  // namespace obf
