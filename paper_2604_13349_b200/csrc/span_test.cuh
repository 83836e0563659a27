// Span test of Orthogonal BackFill for budgets k_eff >= head_dim: does span(V_keep)
// (Eq. 2) fill all of R^d?  If it does, the residual of Eq. 3 is identically zero
// and delta = 0, whatever the deleted values are.
//
// The test is a Cholesky factorisation of G_keep = V_keep^T V_keep without
// pivoting: pivot j is the squared distance of value channel j from the span of
// channels 0..j-1 (over the retained rows); the span is declared full when every
// pivot stays above CHOL_PIVOT_TOL of the channel's own squared norm.  One block
// per (cache, layer, KV head).  Result: HFLAG_SPAN_FULL in hflag[head].
//
// FROM_ROWS (tuned path): G_keep is not read from the workspace but formed here from the first 2 d gathered rows of the
// head (any subset of the retained rows that spans R^d certifies the test), with warp-level mma (bf16 products are
// exact, fp32 accumulation) while the rows sit in the memory the matrix then passes through.
//
// What bounds it is the chain of d pivots and, as much, the code: it is run once per head, so it pays about 130 cycles
// for every 128 bytes of instructions it touches for the first time.  Hence the plainest form: the matrix in registers,
// laid out as in the dense algebra, and one rank-two update per pair of pivots, a small loop body with one block
// barrier: the owners of the next two rows update and publish them before the rest of their rows.  A blocked
// form (32-wide panels, the diagonal block in one warp's registers, 8 x 4 tiles behind it) took 33 us for eight heads; this
// one takes 26 (one pivot per barrier 36, entries doubled into pairs in shared memory 30, four pivots per barrier with the
// owners freeing their four rows of one another by shuffles 30).
#pragma once

#include "algebra.cuh"

namespace obf {

constexpr int ST_NT = 32 * ALG_NW;
constexpr float CHOL_PIVOT_TOL = 1e-3f;

template <int D>
struct SpanShape {
    static constexpr int ROWS = 2 * D;             // retained rows that enter G_keep with FROM_ROWS
    static constexpr int LD = D + 2;               // of the matrix on its way from the tensor cores to the registers
};

template <int D>
constexpr size_t span_smem_bytes(bool from_rows)
{
    return (from_rows ? (size_t)D * SpanShape<D>::LD : 0) * sizeof(float) + (size_t)(4 * D + D) * sizeof(float);
}

template <int D, bool FROM_ROWS = false>
__global__ void __launch_bounds__(ST_NT, 2) k_span_test(const __grid_constant__ CallDev p)
{
    pdl_wait();
    typedef AlgShape<D> SH;
    constexpr int RW = SH::RW, NQ = SH::NQ, LD = SpanShape<D>::LD;
    extern __shared__ __align__(16) float st_sm[];
    float *rows_s = st_sm;                                 // 2 buffers of 2 pivot rows
    float *dg = rows_s + 4 * D;                    // D original diagonal entries
    float *A = dg + D;                                     // FROM_ROWS: the rows, then the matrix

    const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = tid >> 4, c16 = tid & 15;
    int ci, lh;
    locate(p, g, ci, lh);
    const CacheDev &c = p.c[ci];
    const bool need = p.rank > 0 && c.T > c.k_eff && c.k_eff >= D;
    if (!need) {
        if (tid == 0) p.hflag[g] = 0u;
        return;
    }
    AlgMat<D> M;
    if constexpr (FROM_ROWS) {
        constexpr int ROWS = SpanShape<D>::ROWS, CH = D / 8;   // 16-byte chunks per row
        static_assert(ROWS * D * 2 <= D * LD * 4, "the rows are staged in the matrix's memory");
        // X: the first rows of the head's compacted values, [ROWS][D] bf16, rows past the end zero; the
        // 16-byte chunks of a row are permuted by the row number so that 8 x 8 matrix loads hit distinct banks
        uint8_t *X = reinterpret_cast<uint8_t *>(A);
        const int n_rows = c.k_eff < ROWS ? c.k_eff : ROWS;
        const uint4 *src = reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(c.v_out) + (size_t)lh * c.k_eff * D);
        // eight 16-byte loads in flight per thread
        static_assert(ROWS * CH % (8 * ST_NT) == 0, "whole passes");
#pragma unroll 1
        for (int i0 = tid; i0 < ROWS * CH; i0 += 8 * ST_NT) {
            uint4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * ST_NT, r = i / CH, ch = i % CH;
                v[u] = r < n_rows ? __ldg(src + (size_t)r * CH + ch) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * ST_NT, r = i / CH, ch = i % CH;
                *reinterpret_cast<uint4 *>(X + r * (2 * D) + (((ch & 8) | ((ch ^ r) & 7)) << 4)) = v[u];
            }
        }
        __syncthreads();
        // G = X^T X: warp w owns the 16-row blocks w, w + 4, .. of G (m16n8k16, A = X^T and B = X both read with
        // transposing 8 x 8 loads from the row-major X)
        constexpr int NB = D / 16 / ALG_NW;                // row blocks per warp
        const uint32_t xbase = (uint32_t)__cvta_generic_to_shared(X);
        const int mi = lane >> 3, rr = lane & 7;
        auto load4 = [&](uint32_t (&f)[4], int tok, int ch) __attribute__((always_inline)) {
            const uint32_t addr = xbase + tok * (2 * D) + (((ch & 8) | ((ch ^ tok) & 7)) << 4);
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(addr));
        };
        float acc[NB][D / 8][4];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int nt = 0; nt < D / 8; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[b][nt][e] = 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < ROWS; k0 += 16) {
            uint32_t a[NB][4];
            // matrices: (tokens k0.., dims i0..), (tokens k0.., dims i0 + 8..), (tokens k0 + 8.., dims i0..), (k0 + 8.., i0 + 8..)
#pragma unroll
            for (int b = 0; b < NB; ++b) load4(a[b], k0 + (mi >> 1) * 8 + rr, 2 * (warp + ALG_NW * b) + (mi & 1));
#pragma unroll
            for (int np = 0; np < D / 16; ++np) {
                // two 8-column tiles at once: (tokens k0.., dims n0..), (k0 + 8.., n0..), (k0.., n0 + 8..), (k0 + 8.., n0 + 8..)
                uint32_t bf[4];
                load4(bf, k0 + (mi & 1) * 8 + rr, 2 * np + (mi >> 1));
#pragma unroll
                for (int b = 0; b < NB; ++b)
#pragma unroll
                    for (int t2 = 0; t2 < 2; ++t2) {
                        float *d4 = acc[b][2 * np + t2];
                        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                                     : "+f"(d4[0]), "+f"(d4[1]), "+f"(d4[2]), "+f"(d4[3])
                                     : "r"(a[b][0]), "r"(a[b][1]), "r"(a[b][2]), "r"(a[b][3]), "r"(bf[2 * t2]), "r"(bf[2 * t2 + 1]));
                    }
            }
        }
        __syncthreads();                                   // every warp is done reading X: the matrix takes its place
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int nt = 0; nt < D / 8; ++nt) {
                float *dst = A + (16 * (warp + ALG_NW * b) + (lane >> 2)) * LD + nt * 8 + 2 * (lane & 3);
                *reinterpret_cast<f32x2 *>(dst) = pk(acc[b][nt][0], acc[b][nt][1]);
                *reinterpret_cast<f32x2 *>(dst + 8 * LD) = pk(acc[b][nt][2], acc[b][nt][3]);
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RW; ++r) alg_load<D>(M[r], A + SH::row(grp, r) * LD, c16);
    } else {
        const int n_part = gram_partial_count(p, c, lh);           // shape-generic path: one per token split
        const float *G = p.gram_k + (size_t)g * p.gram_slots * D * D + 2 * c16;
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int q = 0; q < NQ; ++q) M[r][q] = *reinterpret_cast<const f32x2 *>(G + SH::row(grp, r) * D + 32 * q);
#pragma unroll 1
        for (int sp = 1; sp < n_part; ++sp) {
            G += D * D;
#pragma unroll
            for (int r = 0; r < RW; ++r)
#pragma unroll
                for (int q = 0; q < NQ; ++q) M[r][q] = add2(M[r][q], *reinterpret_cast<const f32x2 *>(G + SH::row(grp, r) * D + 32 * q));
        }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int i = SH::row(grp, r);
        float a, b;
        upk(M[r][r / SH::RPS], a, b);
        if (c16 == (i & 31) >> 1) dg[i] = (i & 1) ? b : a;
    }
    // row `row`, one of the two of buffer `buf`, for everybody (a half-warp's lanes)
    auto publish = [&](int buf, int row, const AlgRow<D> &x) __attribute__((always_inline)) {
        float *ro = rows_s + (2 * buf + row) * D + 2 * c16;
#pragma unroll
        for (int q = 0; q < NQ; ++q) *reinterpret_cast<f32x2 *>(ro + 32 * q) = x[q];
    };
    if (grp == 0) { publish(0, 0, M[0]); publish(0, 1, M[1]); }
    bool ok = true;
    // the pivots 32 S .. 32 S + 31, two at a time: rows and columns before 32 S are finished
    auto pivots = [&](auto stage) __attribute__((always_inline)) {
        constexpr int S = decltype(stage)::value, R0 = SH::RPS * S;
#pragma unroll 1
        for (int j = 32 * S; ok && j < 32 * S + 32; j += 2) {
            const int buf = (j >> 1) & 1;
            const float *ra = rows_s + 2 * buf * D, *rb = ra + D;
            __syncthreads();                               // rows j and j + 1 are there, as the pivots before j have left them
            const float p0 = ra[j], e = ra[j + 1], i0 = -rcp_approx(p0), l = e * i0, p1 = fmaf(l, e, rb[j + 1]), i1 = -rcp_approx(p1);
            ok = p0 > CHOL_PIVOT_TOL * dg[j] && p0 > 0.f && p1 > CHOL_PIVOT_TOL * dg[j + 1] && p1 > 0.f;   // the same in every thread
            AlgRow<D> v0, v1;
            alg_load<D, S>(v0, ra, c16);
            alg_load<D, S>(v1, rb, c16);
#pragma unroll
            for (int q = S; q < NQ; ++q) {
                v1[q] = mul2(fma2(pk(l, l), v0[q], v1[q]), pk(i1, i1));        // row j + 1 without pivot j, over its pivot
                v0[q] = mul2(v0[q], pk(i0, i0));
            }
            if (j + 2 < D && grp == SH::owner(j + 2)) {
                // rows j + 2 and j + 3 before the others
                const float2 ea = *reinterpret_cast<const float2 *>(ra + j + 2), eb = *reinterpret_cast<const float2 *>(rb + j + 2);
                const float w0[2] = {ea.x, ea.y}, w1[2] = {fmaf(l, ea.x, eb.x), fmaf(l, ea.y, eb.y)};
                auto take = [&](auto cand) __attribute__((always_inline)) {
                    constexpr int R = decltype(cand)::value;
                    if (R < RW && SH::slot(j + 2) == R) {
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            AlgRow<D> x;
#pragma unroll
                            for (int q = 0; q < NQ; ++q) {
                                x[q] = M[R + e < RW ? R + e : 0][q];
                                if (q >= S) x[q] = fma2(pk(w1[e], w1[e]), v1[q], fma2(pk(w0[e], w0[e]), v0[q], x[q]));
                                // (keeps the compiler from merging the candidates' code into one that addresses the array)
                                asm volatile("// %1" : "+l"(x[q]) : "n"(R));
                            }
                            publish(buf ^ 1, e, x);
                        }
                    }
                };
                take(std::integral_constant<int, R0>{});
                take(std::integral_constant<int, R0 + 2>{});
                take(std::integral_constant<int, R0 + 4>{});
            }
#pragma unroll
            for (int r = R0; r < RW; r += 4) {
                const int row = SH::row(grp, r);
                const float4 a4 = *reinterpret_cast<const float4 *>(ra + row), b4 = *reinterpret_cast<const float4 *>(rb + row);
                const float aa[4] = {a4.x, a4.y, a4.z, a4.w}, bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float w1 = fmaf(l, aa[x], bb[x]);
#pragma unroll
                    for (int q = S; q < NQ; ++q) M[r + x][q] = fma2(pk(w1, w1), v1[q], fma2(pk(aa[x], aa[x]), v0[q], M[r + x][q]));
                }
            }
        }
    };
    static_assert(SH::RPS == 4, "three places for the next rows");
    pivots(std::integral_constant<int, 0>{});
    pivots(std::integral_constant<int, 1>{});
    if constexpr (D > 64) {
        pivots(std::integral_constant<int, D / 32 - 2>{});
        pivots(std::integral_constant<int, D / 32 - 1>{});
    }
    if (tid == 0) p.hflag[g] = ok ? HFLAG_SPAN_FULL : 0u;
}

}  // namespace obf
