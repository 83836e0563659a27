// Cache-merging baseline (App. E of the paper, the comparison method "in the spirit of CaM"), per
// (cache, layer, KV head), after the usual selection and gather:
//   (ii)  every deleted position j is routed to the retained position whose key has the largest cosine
//         similarity with K_j (ties: the lowest position; a key of zero norm has similarity 0 with everything),
//   (iii) V*_t = V_t + sum over the j routed to t of A_j / (A_t + eps) * V_j;  keys unchanged.
#pragma once

#include "common.cuh"

namespace obf {

constexpr int MG_TILE = 64;                 // fp32 keys: deleted positions per block, retained positions per inner tile

template <int D>
constexpr size_t merge_smem_bytes() { return (size_t)(2 * MG_TILE * TD_LD<D> + 2 * MG_TILE) * sizeof(float); }

// Larger similarity wins, the lower slot among equals.
__device__ __forceinline__ void merge_better(float &best, int &best_r, float s, int r)
{
    if (s > best || (s == best && r < best_r)) { best = s; best_r = r; }
}

// Routing: assign[j] = slot (0 .. k_eff - 1) of the retained position most similar to position j, -1 for retained j.
// fp32 keys, on the CUDA cores.  grid = (ceil(T_max / MG_TILE), heads_total), 256 threads as 16 x 16: a thread holds
// 4 positions x 4 slots.
template <typename TIN, int D>
__global__ void __launch_bounds__(256) k_merge_assign(const __grid_constant__ CallDev p)
{
    pdl_wait();
    constexpr int LD = TD_LD<D>;
    extern __shared__ __align__(16) float mg_sm[];
    float *Kj = mg_sm, *Kt = Kj + MG_TILE * LD, *inv_j = Kt + MG_TILE * LD, *inv_t = inv_j + MG_TILE;
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff, j0 = blockIdx.x * MG_TILE;
    if (j0 >= T) return;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const TIN *Kh = reinterpret_cast<const TIN *>(c.k) + (size_t)lh * T * D;
    const TIN *Kr = reinterpret_cast<const TIN *>(c.k_out) + (size_t)lh * k * D;      // retained keys, compacted
    const uint8_t *keep = p.keep + c.tok_off + (size_t)lh * T;

    // 1 / norm of the rows of a tile (0 for a zero row or a row past the end): 4 threads per row
    auto inv_norms = [&](const float *rows, float *inv, int n_valid) {
        const int r = tid >> 2, part = tid & 3;
        float s = 0.f;
        for (int e = part; e < D; e += 4) s = fmaf(rows[r * LD + e], rows[r * LD + e], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (part == 0) inv[r] = (r < n_valid && s > 0.f) ? rsqrtf(s) : 0.f;
    };
    load_rows_f32<TIN, D, 256>(Kj, LD, Kh, j0, T, MG_TILE);
    __syncthreads();
    inv_norms(Kj, inv_j, T - j0);

    float best[4];
    int best_r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { best[i] = -INFINITY; best_r[i] = 0; }
    for (int r0 = 0; r0 < k; r0 += MG_TILE) {
        __syncthreads();
        load_rows_f32<TIN, D, 256>(Kt, LD, Kr, r0, k, MG_TILE);
        __syncthreads();
        inv_norms(Kt, inv_t, k - r0);
        __syncthreads();
        float acc[4][4];
        tile_dots<D>(Kj, Kt, ty, tx, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
                const int r = r0 + tx + 16 * jj;
                if (r < k) merge_better(best[i], best_r[i], acc[i][jj] * inv_j[ty + 16 * i] * inv_t[tx + 16 * jj], r);
            }
    }
    // the 16 threads of a position (consecutive lanes) agree on the best slot
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best[i], o);
            const int orr = __shfl_xor_sync(0xffffffffu, best_r[i], o);
            merge_better(best[i], best_r[i], ob, orr);
        }
        const int j = j0 + ty + 16 * i;
        if (tx == 0 && j < T) {
            const int a = keep[j] ? -1 : best_r[i];
            p.assign[c.tok_off + (size_t)lh * T + j] = a;
            if (c.assign_out) c.assign_out[(size_t)lh * T + j] = a;
        }
    }
}

// Routing for bf16 keys: the similarities on the tensor cores.  bf16 products are exact in fp32; their sums are rounded otherwise
// than a chain of fp32 multiply-adds, in the last place or two, so that of two slots whose similarities agree to 1e-6 either may
// be taken (equal keys have equal sums: the lowest slot).  Against 64 bits, 4 heads x 1500 positions, 40 slots: every position
// at its best slot, as in fp32.  A block takes MGT_ROWS positions of a head, 16 per warp and pass; the retained keys lie in
// shared memory, MGT_SLOTS at a time, in the 16-byte chunks of 8 x 8 matrix loads permuted by the row number.  Budgets of
// the merging method are small (tens of slots), so the kernel is a stream over K with a few tensor instructions per
// row: warp-level mma, which needs no staging of K (a lane reads the row fragments it multiplies straight from global
// memory, 16 bytes of a row at a time: the order of the channels inside the contraction is immaterial as long as both
// operands use the same one).  36 x 8 heads, T = 1024, 32 slots:
// 38 us against 239 us on the CUDA cores.
// grid = (ceil(T_max / MGT_ROWS), heads_total), 128 threads.
constexpr int MGT_ROWS = 256, MGT_SLOTS = 64, MGT_NT = 128;

template <int D>
__global__ void __launch_bounds__(MGT_NT) k_merge_assign_mma(const __grid_constant__ CallDev p)
{
    pdl_wait();
    constexpr int CH = D / 8;                                          // 16-byte chunks per row
    constexpr int KS = D / 16;                                         // k-steps of an mma
    __shared__ __align__(16) uint4 Rs[MGT_SLOTS * CH];
    __shared__ float inv_t[MGT_SLOTS];
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff, j0 = blockIdx.x * MGT_ROWS;
    if (j0 >= T) return;
    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31, gr = lane >> 2, gc = lane & 3;
    const uint4 *Kh = reinterpret_cast<const uint4 *>(c.k) + (size_t)lh * T * CH;
    const uint4 *Kr = reinterpret_cast<const uint4 *>(c.k_out) + (size_t)lh * k * CH;
    const uint8_t *keep = p.keep + c.tok_off + (size_t)lh * T;
    auto squares = [](const uint4 &v) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float a = __uint_as_float(w[e] << 16), b = __uint_as_float(w[e] & 0xFFFF0000u);
            s = fmaf(a, a, fmaf(b, b, s));
        }
        return s;
    };
    for (int pass = 0; pass < MGT_ROWS / (16 * (MGT_NT / 32)); ++pass) {
        // this lane's chunks of rows ja and ja + 8: gc, gc + 4, .. (its share of the contraction in that order of channels)
        const int jb = j0 + (pass * (MGT_NT / 32) + warp) * 16, ja = jb + gr;
        uint4 a[2][CH / 4];
        float inv_j[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < CH / 4; ++q) {
                a[h][q] = ja + 8 * h < T ? __ldg(Kh + (size_t)(ja + 8 * h) * CH + 4 * q + gc) : make_uint4(0u, 0u, 0u, 0u);
                s += squares(a[h][q]);
            }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            inv_j[h] = s > 0.f ? rsqrtf(s) : 0.f;
        }
        float best[2] = {-INFINITY, -INFINITY};
        int best_r[2] = {0, 0};
        for (int r0 = 0; r0 < k; r0 += MGT_SLOTS) {
            const int n_slots = min(MGT_SLOTS, k - r0);
            if (pass == 0 || k > MGT_SLOTS) {
                // (with one set of slots it is loaded once)
                __syncthreads();
                for (int i = tid; i < MGT_SLOTS * CH; i += MGT_NT) {
                    const int r = i / CH, ch = i % CH;
                    Rs[r * CH + (ch ^ (r & (CH - 1) & 7))] = r < n_slots ? __ldg(Kr + (size_t)(r0 + r) * CH + ch) : make_uint4(0u, 0u, 0u, 0u);
                }
                __syncthreads();
                if (tid < MGT_SLOTS) {
                    float s = 0.f;
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) s += squares(Rs[tid * CH + (ch ^ (tid & (CH - 1) & 7))]);
                    inv_t[tid] = s > 0.f ? rsqrtf(s) : 0.f;
                }
                __syncthreads();
            }
            if (jb < T) {
                for (int n0 = 0; n0 < n_slots; n0 += 8) {
                    // eight slots: slot n0 + gr in this lane's B fragments, the same chunks as of the rows
                    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int q = 0; q < CH / 4; ++q) {
                        const int r = n0 + gr;
                        const uint4 b = Rs[r * CH + ((4 * q + gc) ^ (r & (CH - 1) & 7))];
                        // a chunk of eight channels serves two k-steps of 16: four lanes x (2 + 2) channels each
                        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                                     : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
                                     : "r"(a[0][q].x), "r"(a[1][q].x), "r"(a[0][q].y), "r"(a[1][q].y), "r"(b.x), "r"(b.y));
                        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                                     : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3])
                                     : "r"(a[0][q].z), "r"(a[1][q].z), "r"(a[0][q].w), "r"(a[1][q].w), "r"(b.z), "r"(b.w));
                    }
                    // acc[0..1]: row gr, slots n0 + 2 gc, + 1; acc[2..3]: row gr + 8
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int r = n0 + 2 * gc + e;
                            if (r < n_slots) merge_better(best[h], best_r[h], acc[2 * h + e] * inv_j[h] * inv_t[r], r0 + r);
                        }
                }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const float ob = __shfl_xor_sync(0xffffffffu, best[h], o);
                const int orr = __shfl_xor_sync(0xffffffffu, best_r[h], o);
                merge_better(best[h], best_r[h], ob, orr);
            }
            const int j = ja + 8 * h;
            if (gc == 0 && j < T) {
                const int a2 = keep[j] ? -1 : best_r[h];
                p.assign[c.tok_off + (size_t)lh * T + j] = a2;
                if (c.assign_out) c.assign_out[(size_t)lh * T + j] = a2;
            }
        }
    }
    static_assert(KS % 2 == 0, "chunks are taken two k-steps at a time");
}

// Merge: WPS warps per retained slot; each walks its share of the head's routing in ascending position order and the
// warps' sums are added in that order (a fixed order: the result does not depend on scheduling); the fp32 sum is rounded
// once to the output type.
// A warp looks at 256 positions at a time (eight loads of the routing in flight), lists the hits in order, and fetches
// the values of eight of them together before it adds them up.  What bounds the kernel is the slot with the most hits, a
// heavy hitter's, and, with many slots, the walks themselves.  36 x 8 heads, T = 1024, 32 slots: one row at a time 115 us,
// eight rows in flight 44 us, the same with eight warps per slot 48 us, with two 35 us; 6 x 8 heads, T = 1500: one warp per
// slot 21 us, eight 11 us.  The warp's number is known to be the same in its lanes (88 -> 80 us a call, 36 x 8 heads of 64 channels; 126.9
// where 128.2) but for long walks over few slots, whose loads the compiler then puts in another order: 24 heads of 128 channels, T = 7585,
// 78.0 us a call without, 79.1 with it in all warps, 76.1 so.
// grid = (ceil(k_eff_max WPS / 8), heads_total), 256 threads.
template <typename TIN, int D, int WPS>
__global__ void __launch_bounds__(256) k_merge_apply(const __grid_constant__ CallDev p)
{
    pdl_wait();
    __shared__ int32_t hits_s[8][256];
    __shared__ float sum_s[8][D];
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff, lane = threadIdx.x & 31, warp = WPS == 8 && D == 128 ? (int)threadIdx.x >> 5 : warp_uniform((int)threadIdx.x >> 5);
    constexpr int SLOTS = 8 / WPS;                                      // slots of a block
    const int r0 = blockIdx.x * SLOTS, r = r0 + warp / WPS, part = warp % WPS;
    if (r0 >= k) return;
    constexpr int PER = D / 32;
    int32_t *hits = hits_s[warp];
    const TIN *Vh = reinterpret_cast<const TIN *>(c.v) + (size_t)lh * T * D + lane * PER;
    const float *A = p.scores + c.tok_off + (size_t)lh * T;
    const int32_t *assign = p.assign + c.tok_off + (size_t)lh * T;
    const float inv_at = 1.f / (A[c.idx_out[(size_t)lh * k + min(r, k - 1)]] + p.eps);
    float acc[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) acc[e] = 0.f;
    const int per = (T + 32 * WPS - 1) / (32 * WPS) * 32, j_end = r < k ? min(T, (part + 1) * per) : 0;   // positions of a warp: a multiple of 32
    for (int jb = part * per; jb < j_end; jb += 256) {
        int a[8], n = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) a[u] = jb + 32 * u + lane < j_end ? assign[jb + 32 * u + lane] : -1;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t hit = __ballot_sync(0xffffffffu, a[u] == r);
            if (a[u] == r) hits[n + __popc(hit & ((1u << lane) - 1u))] = jb + 32 * u + lane;
            n += __popc(hit);
        }
        __syncwarp();
        for (int h0 = 0; h0 < n; h0 += 8) {
            // a lane's PER elements of a row in one load of 4 to 16 bytes
            constexpr int W = PER * (int)sizeof(TIN) / 4;
            float w[8];
            uint32_t v[8][W];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int jj = hits[min(h0 + u, n - 1)];
                w[u] = A[jj];
                const void *src = Vh + (size_t)jj * D;
                if constexpr (W == 4) {
                    const uint4 t = *static_cast<const uint4 *>(src);
                    v[u][0] = t.x; v[u][1] = t.y; v[u][2] = t.z; v[u][3] = t.w;
                } else if constexpr (W == 2) {
                    const uint2 t = *static_cast<const uint2 *>(src);
                    v[u][0] = t.x; v[u][1] = t.y;
                } else {
                    v[u][0] = *static_cast<const uint32_t *>(src);
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (h0 + u < n) {
                    const float f = w[u] * inv_at;
#pragma unroll
                    for (int e = 0; e < PER; ++e) {
                        float x;
                        if constexpr (sizeof(TIN) == 4) x = __uint_as_float(v[u][e]);
                        else x = __uint_as_float((e & 1) ? v[u][e / 2] & 0xFFFF0000u : v[u][e / 2] << 16);
                        acc[e] = fmaf(f, x, acc[e]);
                    }
                }
            }
        }
        __syncwarp();
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) sum_s[warp][lane * PER + e] = acc[e];
    __syncthreads();
    for (int i = threadIdx.x; i < SLOTS * D; i += 256) {
        const int sl = i / D, e = i % D;
        if (r0 + sl >= k) break;
        TIN *out = reinterpret_cast<TIN *>(c.v_out) + ((size_t)lh * k + r0 + sl) * D + e;
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < WPS; ++w) sum += sum_s[sl * WPS + w][e];
        sum += to_f32(*out);
        if constexpr (sizeof(TIN) == 4) *out = sum;
        else *out = __float2bfloat16_rn(sum);
    }
}

}  // namespace obf
