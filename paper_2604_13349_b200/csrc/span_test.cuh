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
// exact, fp32 accumulation), 64 rows in shared memory at a time.
//
// The factorisation goes by panels of 16 channels.  The matrix (its lower blocks of 16 x 16, dealt so that every warp has as
// many) stays in the accumulator fragments that the tensor cores left it in; a panel passes through shared memory to one
// thread per row, which eliminates its 16 pivots without a block barrier: every warp holds the panel's diagonal block
// beside its own rows, a row of it per lane, and passes the pivot row round by shuffles.  What the panel takes from the blocks
// behind it is a product of 16 columns on the tensor cores: both operands as the sum of three bf16 parts, which is exact, and the six
// products of parts that fp32 sums can tell.
//
// What bounds it is the chain of d pivots (two at a time: shuffle, two reciprocals, multiply-adds, 1300 cycles a panel with the operands'
// parts and the barriers) and, beside the pass over V, how many blocks find room: 40 KB and at most 168 registers a thread let two of
// them stand beside a block of that pass.  Eight heads of 128 channels, 24.6 us as one rank-two update of a matrix in registers
// and one barrier per pair of pivots, now 13.0; of it forming G 2.8, the first panel 1.6, the last 0.7.  Calls: one layer of 2048
// positions 53.0 -> 40.8 us, 40 x 8 heads of 8192 472 -> 460, four ragged prompts of 36 x 8 935 -> 891.  Pivots against 64 bits,
// relative to the diagonal, 256 Gaussian rows: 1.1e-7 rms (1.5e-7 by rank-two updates; two TF32 parts and three products 1.4e-7).
#pragma once

#include "algebra.cuh"

namespace obf {

constexpr int ST_NT = 128;
constexpr float CHOL_PIVOT_TOL = 1e-3f;

template <int D>
struct SpanShape {
    static constexpr int ROWS = 2 * D;             // retained rows that enter G_keep with FROM_ROWS
    static constexpr int CHUNK = 64;               // of them in shared memory at a time, two chunks in turn
    static constexpr int NB = D / 16;              // blocks of 16 channels
    static constexpr int PAIRS = D == 128 ? NB + 1 : NB;   // 16 x 16 blocks a warp holds: of block rows w and NB - 1 - w, or of row w
    static constexpr int LD = 20;                  // floats between rows of a panel: fragment and row accesses without bank conflicts
    static constexpr int LS = 112;                 // bytes between rows of an operand: upper, middle and lower part of 16 values, and as many banks on
    static constexpr int CHUNK_BYTES = CHUNK * D * 2;
};
static_assert(ST_NT / 32 * 2 == SpanShape<128>::NB && ST_NT / 32 == SpanShape<64>::NB, "block rows are dealt to four warps");

template <int D>
constexpr size_t span_smem_bytes(bool from_rows)
{
    const size_t panels = D * SpanShape<D>::LD * sizeof(float) + 2 * D * SpanShape<D>::LS, rows = from_rows ? 2 * SpanShape<D>::CHUNK_BYTES : 0;
    return (panels > rows ? panels : rows) + D * sizeof(float);
}

// 16 values as upper, middle and lower bf16 parts (whose sum is the value), 32 bytes each.
__device__ __forceinline__ void store_parts(uint8_t *dst, const float (&x)[16])
{
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t w[3][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float a = x[8 * h + 2 * e], b = x[8 * h + 2 * e + 1];
#pragma unroll
            for (int part = 0; part < 3; ++part) w[part][e] = split_bf16x2(a, b);
        }
#pragma unroll
        for (int part = 0; part < 3; ++part)
            *reinterpret_cast<uint4 *>(dst + 32 * part + 16 * h) = make_uint4(w[part][0], w[part][1], w[part][2], w[part][3]);
    }
}

template <int D, bool FROM_ROWS = false>
__global__ void __launch_bounds__(ST_NT, 3) k_span_test(const __grid_constant__ CallDev p)
{
    pdl_wait();
    typedef SpanShape<D> SP;
    constexpr int NB = SP::NB, PAIRS = SP::PAIRS, LD = SP::LD;
    extern __shared__ __align__(16) float st_sm[];
    float *dg = st_sm;                                     // D original diagonal entries
    float *P = dg + D;                                     // a panel as the ones before it leave it
    uint8_t *Pl = reinterpret_cast<uint8_t *>(P + D * LD), *Pa = Pl + D * SP::LS;   // its rows over the pivots, negative, and its rows, in parts

    const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int fr = lane >> 2, fc = lane & 3;               // row and column of a lane in a fragment
    const int mi = lane >> 3, rr = lane & 7;               // 8 x 8 matrix, and row in it, whose address a lane gives
    int ci, lh;
    locate(p, g, ci, lh);
    const CacheDev &c = p.c[ci];
    const bool need = p.rank > 0 && c.T > c.k_eff && c.k_eff >= D;
    if (!need) {
        if (tid == 0) p.hflag[g] = 0u;
        return;
    }
    // This warp's blocks: block row and block column of pair i.
    auto block_row = [&](int i) __attribute__((always_inline)) { return D == 128 && i <= NB - 1 - warp ? NB - 1 - warp : warp; };
    auto block_col = [&](int i) __attribute__((always_inline)) { return D == 128 && i > NB - 1 - warp ? NB - i : i; };
    float acc[PAIRS][2][4];                                // two tiles of eight columns each
    if constexpr (FROM_ROWS) {
        constexpr int ROWS = SP::ROWS, CH = D / 8, CHUNK = SP::CHUNK, NC = ROWS / CHUNK;   // CH: 16-byte pieces per row
        // the first rows of the head's compacted values, bf16, rows past the end zero; the 16-byte pieces of a row are permuted by
        // the row number so that 8 x 8 matrix loads hit distinct banks
        uint8_t *X = reinterpret_cast<uint8_t *>(P);
        const uint32_t xbase = (uint32_t)__cvta_generic_to_shared(X);
        const int n_rows = c.k_eff < ROWS ? c.k_eff : ROWS;
        const uint4 *src = reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(c.v_out) + (size_t)lh * c.k_eff * D);
        auto fetch = [&](int chunk) __attribute__((always_inline)) {
            const uint32_t to = xbase + (chunk & 1) * SP::CHUNK_BYTES;
#pragma unroll
            for (int u = 0; u < CHUNK * CH / ST_NT; ++u) {
                const int i = tid + u * ST_NT, r = i / CH, ch = i % CH, row = chunk * CHUNK + r;
                const uint4 *from = src + (size_t)(row < n_rows ? row : 0) * CH + ch;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + r * (2 * D) + (((ch & 8) | ((ch ^ r) & 7)) << 4)),
                             "l"(from), "r"(row < n_rows ? 16 : 0) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
        fetch(1);
#pragma unroll
        for (int i = 0; i < PAIRS; ++i)
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][t][e] = 0.f;
        // G = X^T X (m16n8k16, A = X^T and B = X both read with transposing 8 x 8 loads from the row-major X)
#pragma unroll 1
        for (int chunk = 0; chunk < NC; ++chunk) {
            if (chunk + 1 < NC) asm volatile("cp.async.wait_group 1;" ::: "memory");
            else asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            const uint32_t xb = xbase + (chunk & 1) * SP::CHUNK_BYTES;
            auto load4 = [&](uint32_t (&f)[4], int tok, int ch) __attribute__((always_inline)) {
                const uint32_t addr = xb + tok * (2 * D) + (((ch & 8) | ((ch ^ tok) & 7)) << 4);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(addr));
            };
#pragma unroll 2
            for (int k0 = 0; k0 < CHUNK; k0 += 16) {
                // matrices of A: (tokens k0.., dims i0..), (k0.., i0 + 8..), (k0 + 8.., i0..), (k0 + 8.., i0 + 8..)
                uint32_t a[2][4];
                load4(a[0], k0 + (mi >> 1) * 8 + rr, 2 * warp + (mi & 1));
                load4(a[1], k0 + (mi >> 1) * 8 + rr, 2 * (D == 128 ? NB - 1 - warp : warp) + (mi & 1));
#pragma unroll
                for (int i = 0; i < PAIRS; ++i) {
                    if (D == 64 && i > warp) continue;
                    // B: (tokens k0.., dims n0..), (k0 + 8.., n0..), (k0.., n0 + 8..), (k0 + 8.., n0 + 8..)
                    uint32_t bf[4], f[4];
                    load4(bf, k0 + (mi & 1) * 8 + rr, 2 * block_col(i) + (mi >> 1));
#pragma unroll
                    for (int e = 0; e < 4; ++e) f[e] = D == 128 && i <= NB - 1 - warp ? a[1][e] : a[0][e];
#pragma unroll
                    for (int t = 0; t < 2; ++t) mma_bf16(acc[i][t], f, bf[2 * t], bf[2 * t + 1]);
                }
            }
            __syncthreads();                               // every warp is done reading the chunk
            if (chunk + 2 < NC) fetch(chunk + 2);
        }
    } else {
        const int n_part = gram_partial_count(p, c, lh);           // shape-generic path: one per token split
        const float *G = p.gram_k + (size_t)g * p.gram_slots * D * D;
#pragma unroll 1
        for (int sp = 0; sp < n_part; ++sp) {
#pragma unroll
            for (int i = 0; i < PAIRS; ++i) {
                // (heads of 64 channels read the blocks above the diagonal too, without a branch between their loads)
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float2 x = *reinterpret_cast<const float2 *>(G + (16 * block_row(i) + fr + 8 * h) * D + 16 * block_col(i) + 8 * t + 2 * fc);
                        acc[i][t][2 * h] = sp ? acc[i][t][2 * h] + x.x : x.x;
                        acc[i][t][2 * h + 1] = sp ? acc[i][t][2 * h + 1] + x.y : x.y;
                    }
            }
            G += D * D;
        }
    }
    // block i of column block `col` into P
    auto to_panel = [&](int i) __attribute__((always_inline)) {
        float *dst = P + (16 * block_row(i) + fr) * LD + 2 * fc;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            *reinterpret_cast<float2 *>(dst + 8 * t) = make_float2(acc[i][t][0], acc[i][t][1]);
            *reinterpret_cast<float2 *>(dst + 8 * t + 8 * LD) = make_float2(acc[i][t][2], acc[i][t][3]);
        }
    };
#pragma unroll
    for (int i = 0; i < PAIRS; ++i) {
        if (D == 64 && i > warp) continue;
        if (block_col(i) == 0) to_panel(i);
        if (block_col(i) == block_row(i)) {
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (fr == 2 * fc + e) {
                    dg[16 * block_row(i) + fr] = acc[i][0][e];
                    dg[16 * block_row(i) + 8 + fr] = acc[i][1][2 + e];
                }
        }
    }
    // where a lane's row of a block's fragments lies
    const uint32_t l_base = (uint32_t)__cvta_generic_to_shared(Pl) + ((mi & 1) * 8 + rr) * SP::LS + (mi >> 1) * 16;
    const uint32_t a_base = (uint32_t)__cvta_generic_to_shared(Pa) + ((mi >> 1) * 8 + rr) * SP::LS + (mi & 1) * 16;
    bool ok = true;
#pragma unroll 1
    for (int q = 0; q < NB; ++q) {
        __syncthreads();                                   // the panel is there
        {
            // d: row `lane mod 16` of the diagonal block, a: this thread's row, l: over the pivots
            const int row = tid < D ? tid : D - 1;
            float d[16], a[16], l[16], own = 0.f;
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 x = *reinterpret_cast<const float4 *>(P + (16 * q + (lane & 15)) * LD + e), y = *reinterpret_cast<const float4 *>(P + row * LD + e);
                d[e] = x.x; d[e + 1] = x.y; d[e + 2] = x.z; d[e + 3] = x.w;
                a[e] = y.x; a[e + 1] = y.y; a[e + 2] = y.z; a[e + 3] = y.w;
            }
            // two pivots at a time: their rows, x0 as it stands and x1 without pivot k
#pragma unroll
            for (int k = 0; k < 16; k += 2) {
                const float p0 = __shfl_sync(0xffffffffu, d[k], k), r = __shfl_sync(0xffffffffu, d[k + 1], k), i0 = -rcp_approx(p0), m = r * i0;
                const float p1 = fmaf(m, r, __shfl_sync(0xffffffffu, d[k + 1], k + 1)), i1 = -rcp_approx(p1);
                if ((lane & 14) == k) own = lane & 1 ? p1 : p0;
                const float f0 = d[k] * i0, f1 = fmaf(f0, r, d[k + 1]) * i1;
                l[k] = a[k] * i0;
                a[k + 1] = fmaf(l[k], r, a[k + 1]);
                l[k + 1] = a[k + 1] * i1;
#pragma unroll
                for (int j = k + 2; j < 16; ++j) {
                    const float x0 = __shfl_sync(0xffffffffu, d[j], k), x1 = fmaf(m, x0, __shfl_sync(0xffffffffu, d[j], k + 1));
                    d[j] = fmaf(f1, x1, fmaf(f0, x0, d[j]));
                    a[j] = fmaf(l[k + 1], x1, fmaf(l[k], x0, a[j]));
                }
            }
            // (the same in every warp)
            ok = __all_sync(0xffffffffu, own > CHOL_PIVOT_TOL * dg[16 * q + (lane & 15)] && own > 0.f);
            if (tid < D && row >= 16 * (q + 1)) {
                store_parts(Pl + row * SP::LS, l);
                store_parts(Pa + row * SP::LS, a);
            }
        }
        if (!ok || q + 1 == NB) break;
        __syncthreads();                                   // l and a are there, and every warp has read the panel
#pragma unroll
        for (int i = 0; i < PAIRS; ++i) {
            const int br = block_row(i), bc = block_col(i);
            if (bc <= q || bc > br) continue;              // (the same in every lane)
            uint32_t x[3][4], y[3][4];                     // parts of the block row's l (A), of the block column's a (B, two tiles)
#pragma unroll
            for (int part = 0; part < 3; ++part) {
                const uint32_t ax = l_base + 16 * br * SP::LS + 32 * part, ay = a_base + 16 * bc * SP::LS + 32 * part;
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(x[part][0]), "=r"(x[part][1]), "=r"(x[part][2]), "=r"(x[part][3]) : "r"(ax) : "memory");
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(y[part][0]), "=r"(y[part][1]), "=r"(y[part][2]), "=r"(y[part][3]) : "r"(ay) : "memory");
            }
            // the six products that count, small ones first
#pragma unroll
            for (int o = 0; o < 6; ++o) {
                constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                for (int t = 0; t < 2; ++t) mma_bf16(acc[i][t], x[pa[o]], y[pb[o]][2 * t], y[pb[o]][2 * t + 1]);
            }
            if (bc == q + 1) to_panel(i);
        }
    }
    if (tid == 0) p.hflag[g] = ok ? HFLAG_SPAN_FULL : 0u;
}

}  // namespace obf
