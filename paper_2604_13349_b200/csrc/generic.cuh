// Shape-generic kernels (any n_q, T; head_dim 64 or 128; fp32 or bf16 inputs).
// All arithmetic is fp32 on the CUDA cores.  These kernels are the only path for
// fp32 caches and for shapes the tuned bf16 path does not cover.
#pragma once

#include "common.cuh"

namespace obf {

constexpr int SC_TILE = 64;           // queries x keys per score tile
constexpr int SC_NT = 256;
constexpr float LOG2E = 1.4426950408889634f;

// A row's statistics are folded over its keys in an order that T alone decides, whatever else is in the call: the key tiles are
// cut into up to 32 leaves of at least two tiles, the leaves are padded to a power of two, and neighbours are folded pair by
// pair.  The statistics kernel gives a block one aligned run of leaves, a power of two of them; the pooling kernel folds the
// runs' results.  However many blocks share a row, it is the same tree, so that a head's masses do not depend on the other
// heads of the call or on the scratch it was given.  (80 registers, three blocks on a multiprocessor.)
constexpr int SC_LEAVES = 32;
constexpr int SC_MAX_SPLITS = SC_LEAVES;
__host__ __device__ constexpr int sc_leaf_tiles(int T)
{
    const int tiles = (T + SC_TILE - 1) / SC_TILE, per = (tiles + SC_LEAVES - 1) / SC_LEAVES;
    return per < 2 ? 2 : per;
}
__host__ __device__ constexpr int sc_leaves(int T)
{
    const int n = ((T + SC_TILE - 1) / SC_TILE + sc_leaf_tiles(T) - 1) / sc_leaf_tiles(T);
    int p = 1;
    while (p < n) p *= 2;
    return p;
}

// (m, z) <- the fold of (m, z) and (m2, z2); (-inf, 0) is the empty one and changes nothing.
__device__ __forceinline__ void sc_fold(float &m, float &z, float m2, float z2)
{
    const float M = fmaxf(m, m2), Mf = fmaxf(M, -3e38f);                       // (-inf - -inf would be a NaN)
    z = fmaf(z2, exp2f(m2 - Mf), z * exp2f(m - Mf));
    m = M;
}

constexpr int SC_STACK = 5;                     // levels of a block's run of leaves (k_score_stats)
static_assert(1 << SC_STACK == SC_LEAVES && 2 * SC_STACK <= 18, "they lie where the pooling kernel has its 18 rows of 64");
template <int D>
constexpr size_t score_smem_bytes() { return 2 * SC_TILE * TD_LD<D> * sizeof(float) + 2 * SC_TILE * sizeof(float)
                                             + 16 * SC_TILE * sizeof(float); }

// Step a1, first pass (Eq. 1): for every query row the running maximum of the
// scaled logits (log2 domain) and the softmax normaliser over the keys of a split, an aligned run of leaves (above).
// grid = (ceil(n_q/64), heads_total, key splits); blocks beyond a cache's leaves exit.
template <typename TIN, int D>
__global__ void __launch_bounds__(SC_NT, 3) k_score_stats(const __grid_constant__ CallDev p)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    float *Qs = sm, *Ks = sm + SC_TILE * TD_LD<D>;
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, n_q = p.n_q;
    const int q0 = blockIdx.x * SC_TILE;
    const TIN *Kh = reinterpret_cast<const TIN *>(c.k) + (size_t)lh * T * D;
    const TIN *Qh = reinterpret_cast<const TIN *>(c.q) + (size_t)lh * n_q * D;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const float sc = LOG2E * rsqrtf((float)D);

    const int leaves = sc_leaves(T), splits = min(p.sc_splits, leaves), run = leaves / splits;     // all powers of two
    if ((int)blockIdx.z >= splits) return;
    load_rows_f32<TIN, D, SC_NT>(Qs, TD_LD<D>, Qh, q0, n_q, SC_TILE);
    const int leaf_keys = sc_leaf_tiles(T) * SC_TILE;
    // finished subtrees that wait for their right neighbour, one per level and row
    float *wait_m = Ks + SC_TILE * TD_LD<D>, *wait_z = wait_m + SC_STACK * SC_TILE;

    for (int leaf = 0; leaf < run; ++leaf) {
        const int j_begin = (blockIdx.z * run + leaf) * leaf_keys, j_end = min(T, j_begin + leaf_keys);
        float m[4], Z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { m[i] = -INFINITY; Z[i] = 0.f; }
        for (int j0 = j_begin; j0 < j_end; j0 += SC_TILE) {
            __syncthreads();
            load_rows_f32<TIN, D, SC_NT>(Ks, TD_LD<D>, Kh, j0, T, SC_TILE);
            __syncthreads();
            float acc[4][4];
            tile_dots<D>(Qs, Ks, ty, tx, acc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float tm = -INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] = (j0 + tx + 16 * j < T) ? acc[i][j] * sc : -INFINITY;
                    tm = fmaxf(tm, acc[i][j]);
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, o));
                const float nm = fmaxf(m[i], tm);
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) s += exp2f(acc[i][j] - nm);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                Z[i] = Z[i] * exp2f(m[i] - nm) + s;
                m[i] = nm;
            }
        }
        // the sixteen lanes of a row hold the same: the first four fold and store a row each
        const int slot = ty + 16 * tx, row = q0 + slot;
        if (tx < 4 && row < n_q) {
            float mi = tx == 0 ? m[0] : tx == 1 ? m[1] : tx == 2 ? m[2] : m[3];
            float zi = tx == 0 ? Z[0] : tx == 1 ? Z[1] : tx == 2 ? Z[2] : Z[3];
            // the keys outside the prompt go with the first leaf
            if (c.lse_extra && blockIdx.z == 0 && leaf == 0) fold_lse_extra(c.lse_extra[(size_t)lh * n_q + row], mi, zi);
            int level = 0;
#pragma unroll 1
            for (; (leaf >> level) & 1; ++level) {
                float M = wait_m[level * SC_TILE + slot], S = wait_z[level * SC_TILE + slot];
                sc_fold(M, S, mi, zi);
                mi = M;
                zi = S;
            }
            if (leaf + 1 < run) {
                wait_m[level * SC_TILE + slot] = mi;
                wait_z[level * SC_TILE + slot] = zi;
            } else {
                reinterpret_cast<float2 *>(p.stats)[((size_t)blockIdx.y * p.sc_splits + blockIdx.z) * n_q + row] = make_float2(mi, zi);
            }
        }
    }
}

// Step a1, second pass (Eq. 1): A_j = sum_t exp(s_tj - m_t) / Z_t for a tile of 64 keys.
// grid = (ceil(T_max/64), heads_total); blocks beyond a cache's T exit.
template <typename TIN, int D>
__global__ void __launch_bounds__(SC_NT, 3) k_score_pool(const __grid_constant__ CallDev p)
{
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    float *Qs = sm, *Ks = sm + SC_TILE * TD_LD<D>;
    float *rm = Ks + SC_TILE * TD_LD<D>, *rz = rm + SC_TILE, *red = rz + SC_TILE;
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, n_q = p.n_q;
    const int j0 = blockIdx.x * SC_TILE;
    if (j0 >= T) return;
    const TIN *Kh = reinterpret_cast<const TIN *>(c.k) + (size_t)lh * T * D;
    const TIN *Qh = reinterpret_cast<const TIN *>(c.q) + (size_t)lh * n_q * D;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const float sc = LOG2E * rsqrtf((float)D);

    load_rows_f32<TIN, D, SC_NT>(Ks, TD_LD<D>, Kh, j0, T, SC_TILE);
    float colsum[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q0 = 0; q0 < n_q; q0 += SC_TILE) {
        __syncthreads();
        load_rows_f32<TIN, D, SC_NT>(Qs, TD_LD<D>, Qh, q0, n_q, SC_TILE);
        {
            // a row's statistics over all keys, the upper levels of the tree: four threads per row, a run of splits each
            constexpr int PER = SC_MAX_SPLITS / 4;
            static_assert(SC_NT == 4 * SC_TILE && PER >= 1, "four threads per row");
            const int slot = threadIdx.x >> 2, part = threadIdx.x & 3, row = q0 + slot, splits = min(p.sc_splits, sc_leaves(T));
            const float2 *st = reinterpret_cast<const float2 *>(p.stats) + ((size_t)blockIdx.y * p.sc_splits + part * PER) * n_q + min(row, n_q - 1);
            float2 v[PER];
#pragma unroll
            for (int e = 0; e < PER; ++e) v[e] = part * PER + e < splits ? st[(size_t)e * n_q] : make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int w = 1; w < PER; w *= 2)
                if (w < splits) {
#pragma unroll
                    for (int e = 0; e < PER; e += 2 * w) sc_fold(v[e].x, v[e].y, v[e + w].x, v[e + w].y);
                }
            float M = v[0].x, Z = v[0].y;
            if (splits > PER) {
#pragma unroll
                for (int o = 1; o < 4; o *= 2) {
                    const float m2 = __shfl_xor_sync(0xffffffffu, M, o), z2 = __shfl_xor_sync(0xffffffffu, Z, o);
                    float ml = part & o ? m2 : M, zl = part & o ? z2 : Z;
                    sc_fold(ml, zl, part & o ? M : m2, part & o ? Z : z2);
                    M = ml;
                    Z = zl;
                }
            }
            if (part == 0) {
                rm[slot] = row < n_q ? M : 0.f;
                rz[slot] = row < n_q ? 1.0f / Z : 0.f;
            }
        }
        __syncthreads();
        float acc[4][4];
        tile_dots<D>(Qs, Ks, ty, tx, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float mi = rm[ty + 16 * i], zi = rz[ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) colsum[j] += exp2f(acc[i][j] * sc - mi) * zi;
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) red[ty * SC_TILE + tx + 16 * j] = colsum[j];
    __syncthreads();
    if (threadIdx.x < SC_TILE && j0 + threadIdx.x < T) {
        float a = 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r) a += red[r * SC_TILE + threadIdx.x];
        if (!isfinite(a)) atomicOr(p.status, OBF_DEV_NONFINITE);
        p.scores[c.tok_off + (size_t)lh * T + j0 + threadIdx.x] = a;
        if (c.scores_out) c.scores_out[(size_t)lh * T + j0 + threadIdx.x] = a;
    }
}

// What a selection leaves for its head: the demand sums and, where asked for, a fresh diagnostics record.
__device__ __forceinline__ void store_selection(const CallDev &p, const CacheDev &c, int g, int lh, float a_keep, float a_del, float next, uint32_t tau)
{
    float *sm = p.sums + (size_t)g * 4;
    const float kth = tau == 0xFFFFFFFFu ? INFINITY : key_score(tau);
    sm[0] = a_keep; sm[1] = a_del; sm[2] = kth; sm[3] = next;
    if (c.diag) {
        obf_diag_t dg;
        dg.a_keep = a_keep; dg.a_del = a_del; dg.alpha = a_del / (a_keep + p.eps);
        dg.rcr = 0.f; dg.delta_norm = 0.f; dg.kth_score = kth; dg.next_score = next;
        dg.lam_1 = dg.lam_rho = dg.lam_next = 0.f;
        dg.span_rank = -1; dg.rho_eff = 0; dg.status = OBF_DEV_SKIPPED; dg.revr = 0.f; dg.pc = 0.f;
        c.diag[lh] = dg;
    }
}

// Step a2: radix select of the k_eff largest masses on their order-preserving
// 32-bit keys (4 passes of 8 bits), then one ordered pass that emits the
// retained positions in ascending order; among masses equal to the k_eff-th
// largest, the lowest positions are taken.  One block per (cache, layer, head).
constexpr int SEL_NT = 1024;

__global__ void __launch_bounds__(SEL_NT) k_select(const __grid_constant__ CallDev p)
{
    pdl_wait();
    __shared__ uint32_t hist[256];
    __shared__ uint32_t s_prefix, s_want;
    __shared__ uint32_t wsum[32];
    __shared__ float red[32];
    int ci, lh;
    locate(p, blockIdx.x, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff;
    // the masses are handled as raw bit patterns so that every pass sees identical keys
    const uint32_t *A = reinterpret_cast<const uint32_t *>(p.scores + c.tok_off + (size_t)lh * T);
    uint8_t *keep = p.keep + c.tok_off + (size_t)lh * T;
    int32_t *idx = c.idx_out + (size_t)lh * k;
    const int tid = threadIdx.x;

    if (tid == 0) { s_prefix = 0u; s_want = (uint32_t)k; }
    uint32_t mask = 0u;
    for (int shift = 24; shift >= 0; shift -= 8) {
        if (tid < 256) hist[tid] = 0u;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        for (int j = tid; j < T; j += SEL_NT) {
            const uint32_t u = select_key(p, j, A[j]);
            if ((u & mask) == prefix) atomicAdd(&hist[(u >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (tid == 0) {
            uint32_t want = s_want, cum = 0u;
            int b = 255;
            for (; b > 0; --b) {
                if (cum + hist[b] >= want) break;
                cum += hist[b];
            }
            s_want = want - cum;
            s_prefix = prefix | ((uint32_t)b << shift);
        }
        mask |= 255u << shift;
        __syncthreads();
    }
    const uint32_t tau = s_prefix;       // key of the k-th largest mass
    const uint32_t want = s_want;        // how many positions with key == tau are retained (>= 1)

    uint32_t run_gt = 0u, run_eq = 0u;
    float sk = 0.f, sd = 0.f, nx = -1.0f;
    for (int base = 0; base < T; base += SEL_NT) {
        const int j = base + tid;
        const bool valid = j < T;
        const uint32_t abits = valid ? A[j] : 0u;
        const float a = __uint_as_float(abits);
        const uint32_t u = valid ? select_key(p, j, abits) : 0u;
        const bool gt = valid && u > tau, eq = valid && u == tau;
        uint32_t v = (gt ? 1u : 0u) | (eq ? 0x10000u : 0u);
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t n = __shfl_up_sync(0xffffffffu, inc, o);
            if ((tid & 31) >= o) inc += n;
        }
        if ((tid & 31) == 31) wsum[tid >> 5] = inc;
        __syncthreads();
        if (tid < 32) {
            uint32_t w = wsum[tid], winc = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t n = __shfl_up_sync(0xffffffffu, winc, o);
                if (tid >= o) winc += n;
            }
            wsum[tid] = winc - w;          // exclusive prefix of warp totals
            if (tid == 31) hist[0] = winc; // block total
        }
        __syncthreads();
        const uint32_t excl = inc - v + wsum[tid >> 5];
        const uint32_t gt_before = run_gt + (excl & 0xFFFFu), eq_before = run_eq + (excl >> 16);
        const bool kp = gt || (eq && eq_before < want);
        if (valid) {
            keep[j] = kp ? 1 : 0;
            if (kp) {
                const uint32_t pos = gt_before + min(eq_before, want);
                if (pos < (uint32_t)k) idx[pos] = j;
                else atomicOr(p.status, OBF_DEV_INTERNAL);
                sk += a;
            }
            else { sd += a; nx = fmaxf(nx, a); }
        }
        const uint32_t tot = hist[0];
        run_gt += tot & 0xFFFFu;
        run_eq += tot >> 16;
        __syncthreads();
    }
    const float a_keep = block_sum<SEL_NT>(sk, red);
    const float a_del = block_sum<SEL_NT>(sd, red);
    const float next = block_max<SEL_NT>(nx, red);
    if (tid == 0) {
        store_selection(p, c, blockIdx.x, lh, a_keep, a_del, next, tau);
    }
}

// Retained rows that the selection copies itself (k_select_smem): with this few a copy of its own costs a launch, 2 us, for
// what the head's block has in hand a moment after the positions; the block's threads fetch all of them at once.
constexpr int SEL_GATHER_MAX = 64;
// and this many where no multiprocessor has more than one head: its block of 1024 threads fetches them while the others would launch the
// copy: where a span test waits for the values beside the pass over V these only (8 heads, 205 of 2048 rows, 44.1 -> 42.2 us a call; 128 heads,
// 250 of 2000, 84.1 -> 82.5), without a span test keys and values up to half as many (32 heads, 100 of 1000 rows, 177 -> 173; with 200 rows
// eviction would go from 24.2 to 25.0).
constexpr int SEL_GATHER_FEW = 256;

constexpr int SEL_SMEM_MAX_T = 16384;               // keys of a head that fit in shared memory (k_select_smem)

// Layerwise selector, first half (Section 3.2, retention rule, second form): the masses of a layer's KV heads
// added up per position, head 0 first.  grid = (ceil(T_max / 256), layers of all caches).
__global__ void __launch_bounds__(256) k_layer_sum(const __grid_constant__ CallDev p)
{
    pdl_wait();
    int ci, lh;
    locate(p, blockIdx.y * p.kv_heads, ci, lh);
    const CacheDev &c = p.c[ci];
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j >= c.T) return;
    const float *A = p.scores + c.tok_off + (size_t)lh * c.T + j;
    float s = 0.f;
    for (int h = 0; h < p.kv_heads; ++h) s += A[(size_t)h * c.T];
    p.lscores[c.tok_off / p.kv_heads + (size_t)(lh / p.kv_heads) * c.T + j] = s;
}

// Step a2 for heads whose T keys fit in shared memory (the usual case): same result as k_select, bit for bit.
// What bounds it is the chain of barriers and serial steps, not the keys: four passes of 8 bits with their searches were
// 1500 cycles each before a key was looked at.  So the keys are counted by their upper 11 bits while they are loaded (four
// bins per octave: few equal ones in a warp), one search finds the bin of the k-th largest, and as it holds few keys as a
// rule (at most SEL_CAND_MAX) those are listed and ranked against one another, which ends the search; a fuller bin (many
// masses within a quarter of an octave, or equal) is split by the next 11 and the last 10 bits first.  Every warp has a
// contiguous run of positions for the listing and the ordered pass.
// Counters are 16 bits wide (T < 65536) so that, at T = 8192, two blocks find room beside a block of the pass over V.
// 8 heads, T = 2048: 8.5 -> 6.7 us; 288 heads, T = 4096: 16 -> 11.6; 320 heads, T = 8192, beside the pass over V: 56 -> 40.
// With LAYER every head's block selects on its layer's summed masses (the layer's heads repeat the same
// selection side by side rather than one block writing all of them in turn) and writes the demand sums of the head's own.
// gather_vecs != 0: the block copies its head's retained rows too (at most SEL_GATHER_FEW), that many 16-byte vectors each: of K and V, or, of
// V only where it is negative.
constexpr int SEL_CAND_MAX = 256, SEL_BINS = 2048;

template <int NT, bool LAYER = false>
__global__ void __launch_bounds__(NT, 2048 / NT) k_select_smem(const __grid_constant__ CallDev p, int gather_vecs)
{
    pdl_wait();
    extern __shared__ uint32_t sel_keys[];
    constexpr int NW = NT / 32, WPT = SEL_BINS / 2 / NT;                // words of two bins per thread
    static_assert(WPT >= 1 && SEL_BINS / 2 % NT == 0, "whole words per thread");
    __shared__ uint32_t hist[SEL_BINS / 2];
    __shared__ __align__(16) uint32_t cand[SEL_CAND_MAX];               // listed keys
    __shared__ uint8_t cand_warp[SEL_CAND_MAX];                         // the warp whose run a listed key lies in
    __shared__ uint32_t s_bin, s_want, s_count, s_listed, s_tau;
    __shared__ uint32_t wtot[32];
    __shared__ float red[3][32];
    __shared__ int s_idx[SEL_GATHER_FEW];
    int ci, lh;
    locate(p, blockIdx.x, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T, k = c.k_eff;
    const float *Af = p.scores + c.tok_off + (size_t)lh * T;
    const uint32_t *A = LAYER ? reinterpret_cast<const uint32_t *>(p.lscores + c.tok_off / p.kv_heads + (size_t)(lh / p.kv_heads) * T)
                              : reinterpret_cast<const uint32_t *>(Af);
    uint8_t *keep = p.keep + c.tok_off + (size_t)lh * T;
    int32_t *idx = c.idx_out + (size_t)lh * k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // adds the warp's keys to the bins; `in`: this lane's key counts
    auto count = [&](uint32_t digit, bool in) {
        const uint32_t ins = __ballot_sync(0xffffffffu, in);
        if (ins == 0u) return;
        // one digit for the whole warp (equal masses) is counted once
        const int first = __ffs(ins) - 1;
        const uint32_t d0 = __shfl_sync(0xffffffffu, digit, first);
        if (__all_sync(0xffffffffu, !in || digit == d0)) {
            if (lane == first) atomicAdd(&hist[d0 >> 1], (uint32_t)__popc(ins) << (16 * (d0 & 1u)));
        } else if (in) {
            atomicAdd(&hist[digit >> 1], 1u << (16 * (digit & 1u)));
        }
    };
    // the bin that holds the want-th largest key counted -> s_bin, s_count; what is still wanted of it -> s_want.  Thread 0
    // owns the highest bins.
    auto search = [&](uint32_t want) {
        __syncthreads();
        uint32_t h[WPT], own = 0u;
#pragma unroll
        for (int w = 0; w < WPT; ++w) {
            h[w] = hist[(NT - 1 - tid) * WPT + WPT - 1 - w];
            own += (h[w] >> 16) + (h[w] & 0xFFFFu);
        }
        uint32_t upto = own;                            // inclusive sum over the warp's lanes <= this one
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t n = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += n;
        }
        if (lane == 31) wtot[warp] = upto;
        __syncthreads();
        upto += __reduce_add_sync(0xffffffffu, lane < warp ? wtot[lane] : 0u);
        uint32_t above = upto - own;
        if (above < want && want <= upto) {
#pragma unroll
            for (int b = 0; b < 2 * WPT; ++b) {
                const uint32_t n = (b & 1) ? h[b / 2] & 0xFFFFu : h[b / 2] >> 16;
                if (above < want && want <= above + n) {
                    s_bin = (uint32_t)(((NT - 1 - tid) * WPT + WPT - 1 - b / 2) * 2 + 1 - (b & 1));
                    s_count = n;
                    s_want = want - above;
                }
                above += n;
            }
        }
        __syncthreads();
    };

    // keys into shared memory, counted by their upper 11 bits on the way; four loads in flight
    const int T_pad = (T + NT - 1) / NT * NT;
    bool clear = true;
    for (int j0 = tid; j0 < T_pad; j0 += 4 * NT) {
        uint32_t a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = j0 + u * NT < T ? A[j0 + u * NT] : 0u;
        if (clear) {
            // (while the first loads are on their way)
#pragma unroll
            for (int w = 0; w < WPT; ++w) hist[tid + w * NT] = 0u;
            if (tid == 0) { s_bin = 0u; s_count = 0u; s_want = 1u; s_listed = 0u; s_tau = 0u; }
            __syncthreads();
            clear = false;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + u * NT;
            const uint32_t key = select_key(p, j, a[u]);
            if (j < T) sel_keys[j] = key;
            count(key >> 21, j < T);
        }
    }
    search((uint32_t)k);
    uint32_t prefix = s_bin << 21, mask = 0xFFE00000u, want = s_want, n_in = s_count;
    // a full bin: the next 11 bits, then the last 10
    for (int shift = 10; shift >= 0 && n_in > (uint32_t)SEL_CAND_MAX; shift -= 10) {
#pragma unroll
        for (int w = 0; w < WPT; ++w) hist[tid + w * NT] = 0u;
        __syncthreads();
        for (int j = tid; j < T_pad; j += NT) {
            const uint32_t u = j < T ? sel_keys[j] : 0u;
            count((u >> shift) & (shift ? 0x7FFu : 0x3FFu), j < T && (u & mask) == prefix);
        }
        search(want);
        prefix |= s_bin << shift;
        mask |= (shift ? 0x7FFu : 0x3FFu) << shift;
        want = s_want;
        n_in = s_count;
    }

    // warp w owns positions [w * seg, (w + 1) * seg): its keys above the bin are counted, those in it listed
    const int seg = ((T + NW - 1) / NW + 31) / 32 * 32;
    const int j_begin = warp * seg, j_end = min(T, j_begin + seg);
    const uint32_t lt_mask = (1u << lane) - 1u;
    const bool listing = n_in <= (uint32_t)SEL_CAND_MAX;                // otherwise the bin is one value, all of its bits known
    uint32_t n_gt = 0u, n_eq = 0u;
#pragma unroll 4
    for (int j0 = j_begin; j0 < j_end; j0 += 32) {
        const int j = j0 + lane;
        const uint32_t u = j < j_end ? sel_keys[j] : 0u;
        const bool in = j < j_end && (u & mask) == prefix;
        const uint32_t m_in = __ballot_sync(0xffffffffu, in);
        n_gt += __popc(__ballot_sync(0xffffffffu, j < j_end && (u & mask) > prefix));
        n_eq += __popc(m_in);
        if (listing && in) {
            const uint32_t at = atomicAdd(&s_listed, 1u);
            if (at < (uint32_t)SEL_CAND_MAX) { cand[at] = u; cand_warp[at] = (uint8_t)warp; }
        }
    }
    if (lane == 0) wtot[warp] = n_gt | (listing ? 0u : n_eq << 16);
    __syncthreads();
    if (listing) {
        // every listed key against all of them (slots past the end, up to the next multiple of four, count as lower)
        const int n = (int)min(n_in, (uint32_t)SEL_CAND_MAX);
        const uint32_t mine = tid < n ? cand[tid] : 0u;
        uint32_t gt = 0u, eq = 0u;
        if (tid < n) {
            for (int i = 0; i < n; i += 4) {
                const uint4 q = *reinterpret_cast<const uint4 *>(cand + i);
                const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool there = i + e < n;
                    gt += there && v[e] > mine;
                    eq += there && v[e] == mine;
                }
            }
            if (gt < want && want <= gt + eq) { s_tau = mine; s_want = want - gt; }     // (equal keys write the same)
        }
        __syncthreads();
        if (tid < n && mine >= s_tau) atomicAdd(&wtot[cand_warp[tid]], mine > s_tau ? 1u : 0x10000u);
        __syncthreads();
    }
    const uint32_t tau = listing ? s_tau : prefix;       // key of the k-th largest mass
    want = listing ? s_want : want;                      // how many positions with key == tau are retained (>= 1)

    // positions before this warp's run: greater (low half), equal (high half).  (No half carries over: T < 65536.)
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? wtot[lane] : 0u);
    uint32_t run_gt = before & 0xFFFFu, run_eq = before >> 16;
    float sk = 0.f, sd = 0.f, nx = -1.0f;
    for (int j0 = j_begin; j0 < j_end; j0 += 128) {
        uint32_t key[4];
        float own[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u + lane;
            key[u] = j < j_end ? sel_keys[j] : 0u;
            // a protected position's key is not its mass; a layer's is not its heads'
            own[u] = j < j_end && (LAYER || j < p.n_sink) ? Af[j] : key_score(key[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u + lane;
            const bool valid = j < j_end, gt = valid && key[u] > tau, eq = valid && key[u] == tau;
            const uint32_t m_gt = __ballot_sync(0xffffffffu, gt), m_eq = __ballot_sync(0xffffffffu, eq);
            const uint32_t gt_before = run_gt + __popc(m_gt & lt_mask), eq_before = run_eq + __popc(m_eq & lt_mask);
            const bool kp = gt || (eq && eq_before < want);
            if (valid) {
                keep[j] = kp ? 1 : 0;
                if (kp) {
                    const uint32_t pos = gt_before + min(eq_before, want);
                    if (pos < (uint32_t)k) {
                        idx[pos] = j;
                        if (gather_vecs) s_idx[pos] = j;
                    }
                    else atomicOr(p.status, OBF_DEV_INTERNAL);
                    sk += own[u];
                } else { sd += own[u]; nx = fmaxf(nx, key_score(key[u])); }
            }
            run_gt += __popc(m_gt);
            run_eq += __popc(m_eq);
        }
    }

    // block totals of the retained and the deleted mass and the largest deleted one: the last warp, which has the least to
    // copy, adds up the warps' shares
    sk = warp_sum(sk); sd = warp_sum(sd); nx = warp_max(nx);
    if (lane == 0) { red[0][warp] = sk; red[1][warp] = sd; red[2][warp] = nx; }
    __syncthreads();
    if (gather_vecs) {
        // two vectors a thread in flight: of K and V, or two of V.  A row has 8, 16 or 32 vectors, and a head's rows of them fit 32 bits; with
        // divisions by that number 152 heads with 24 rows each took 27.3 us a call (so 25.5), 64 with 120 rows 26.6 (25.9).  Not unrolled it would be 24.9,
        // but the selection before it spills registers: 12 x 8 ragged heads that copy nothing here 328 -> 332
        const bool both = gather_vecs > 0;
        const int vecs = both ? gather_vecs : -gather_vecs, n = k * vecs, step = both ? NT : 2 * NT, sh = __ffs(vecs) - 1;
        const size_t to = (size_t)lh * n;
        const uint4 *vs = reinterpret_cast<const uint4 *>(c.v) + (size_t)lh * T * vecs, *ks = both ? reinterpret_cast<const uint4 *>(c.k) + (size_t)lh * T * vecs : vs;
        uint4 *vo = reinterpret_cast<uint4 *>(c.v_out) + to, *ko = both ? reinterpret_cast<uint4 *>(c.k_out) + to : vo;
        for (int e = tid; e < n; e += step) {
            const int e2 = both ? e : min(e + NT, n - 1), j = s_idx[e >> sh], j2 = s_idx[e2 >> sh];
            if ((unsigned)j >= (unsigned)T || (unsigned)j2 >= (unsigned)T) {       // never dereference a position outside the cache
                atomicOr(p.status, OBF_DEV_INTERNAL);
                continue;
            }
            const uint4 a = vs[(j << sh) + (e & (vecs - 1))], b = ks[(j2 << sh) + (e2 & (vecs - 1))];
            vo[e] = a;
            ko[e2] = b;
        }
    }
    if (warp == NW - 1) {
        sk = warp_sum(lane < NW ? red[0][lane] : 0.f);
        sd = warp_sum(lane < NW ? red[1][lane] : 0.f);
        nx = warp_max(lane < NW ? red[2][lane] : -1.0f);
        if (lane == 0) store_selection(p, c, blockIdx.x, lh, sk, sd, nx, tau);
    }
}

// Step a3: K_out = K[idx], V_out = V[idx] as 16-byte vectors.  A block copies GATHER_ROWS
// retained rows of one head; every thread moves one vector of four different rows of K
// and of V, with all eight loads in flight before the first store.
// grid = (ceil(k_eff_max / GATHER_ROWS), heads_total).
constexpr int GATHER_ROWS = 64;

// WHICH: 3 = keys and values, 1 = values only, 2 = keys only (the keys are needed by nothing that follows in
// the call, so their copy can run beside the later kernels).
// Where a cache wants the int8 copy of its relay, a row is quantised while it is in registers (an injection quantises its
// rows again, k_obf_algebra; values that are merged are quantised afterwards).  40 layers x 8 heads, 811 of 8192 rows: 511 us
// with a pass of its own over the compacted rows, 477 so (498 when the copy of the keys, which runs beside the span test,
// quantises the values too: the span test fills the register files).
template <typename TIN, int D, int WHICH = 3>
__global__ void __launch_bounds__(256) k_gather(const __grid_constant__ CallDev p)
{
    pdl_wait();
    constexpr int ROW_BYTES = D * (int)sizeof(TIN);
    constexpr int CH = ROW_BYTES / 16;             // vectors per row
    constexpr int RPP = 256 / CH;                  // rows per pass of the block
    constexpr int PASSES = GATHER_ROWS / RPP;
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int r0 = blockIdx.x * GATHER_ROWS;
    if (r0 >= c.k_eff) return;
    const int ch = threadIdx.x % CH, rr = threadIdx.x / CH;
    const char *kb = reinterpret_cast<const char *>(c.k) + (size_t)lh * c.T * ROW_BYTES;
    const char *vb = reinterpret_cast<const char *>(c.v) + (size_t)lh * c.T * ROW_BYTES;
    char *ko = reinterpret_cast<char *>(c.k_out) + (size_t)lh * c.k_eff * ROW_BYTES;
    char *vo = reinterpret_cast<char *>(c.v_out) + (size_t)lh * c.k_eff * ROW_BYTES;
    const int32_t *idx = c.idx_out + (size_t)lh * c.k_eff;
#pragma unroll 1
    for (int p0 = 0; p0 < PASSES; p0 += 4) {
        int r[4], j[4];
        uint4 kv[4], vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            r[u] = r0 + (p0 + u) * RPP + rr;
            j[u] = -1;
            if (p0 + u < PASSES && r[u] < c.k_eff) {
                j[u] = idx[r[u]];
                if ((unsigned)j[u] >= (unsigned)c.T) {     // never dereference a position outside the cache
                    atomicOr(p.status, OBF_DEV_INTERNAL);
                    j[u] = -1;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j[u] >= 0) {
                if (WHICH & 2) kv[u] = *reinterpret_cast<const uint4 *>(kb + (size_t)j[u] * ROW_BYTES + ch * 16);
                if (WHICH & 1) vv[u] = *reinterpret_cast<const uint4 *>(vb + (size_t)j[u] * ROW_BYTES + ch * 16);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j[u] >= 0) {
                if (WHICH & 2) *reinterpret_cast<uint4 *>(ko + (size_t)r[u] * ROW_BYTES + ch * 16) = kv[u];
                if (WHICH & 1) *reinterpret_cast<uint4 *>(vo + (size_t)r[u] * ROW_BYTES + ch * 16) = vv[u];
            }
        }
        if (c.k_q8) {
            const size_t head = (size_t)lh * c.k_eff;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (j[u] < 0) continue;                            // (the lanes of a row agree)
                if (WHICH & 2) quantize16<TIN, D>(kv[u], c.k_q8, c.k_scale, head + r[u], ch);
                if ((WHICH & 1) && !p.merge) quantize16<TIN, D>(vv[u], c.v_q8, c.v_scale, head + r[u], ch);
            }
        }
    }
}

// The int8 copy of the values of a merged cache, whose rows are final only then (quantize16 does the work).
// grid = (ceil(k_eff_max / QR_ROWS), heads_total), 256 threads.
constexpr int QR_ROWS = 64;

template <typename TIN, int D>
__global__ void __launch_bounds__(256) k_quantize_values(const __grid_constant__ CallDev p)
{
    pdl_wait();
    constexpr int CH = D * (int)sizeof(TIN) / 16;
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int r0 = blockIdx.x * QR_ROWS;
    if (!c.v_q8 || r0 >= c.k_eff) return;
    const size_t head = (size_t)lh * c.k_eff;
    for (int r = r0 + threadIdx.x / CH; r < min(r0 + QR_ROWS, c.k_eff); r += 256 / CH) {
        const uint4 raw = reinterpret_cast<const uint4 *>(c.v_out)[(head + r) * CH + threadIdx.x % CH];
        quantize16<TIN, D>(raw, c.v_q8, c.v_scale, head + r, threadIdx.x % CH);
    }
}

// Diagnostics only (projection cosine): s = sum of the deleted value rows of a head, for heads with a
// diagnostics record.  grid = (token splits, heads_total), 256 threads = 256 / D row groups x D columns.
template <typename TIN, int D>
__global__ void __launch_bounds__(256) k_vsum(const __grid_constant__ CallDev p)
{
    pdl_wait();
    __shared__ float part[256];
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    if (!c.diag || c.T <= c.k_eff) return;
    constexpr int RG = 256 / D > 0 ? 256 / D : 1;         // row groups
    const int col = threadIdx.x % D, rg = threadIdx.x / D;
    const int per = (c.T + gridDim.x - 1) / gridDim.x;
    const int r0 = blockIdx.x * per, r1 = min(c.T, r0 + per);
    const TIN *V = reinterpret_cast<const TIN *>(c.v) + (size_t)lh * c.T * D;
    const uint8_t *keep = p.keep + c.tok_off + (size_t)lh * c.T;
    float acc = 0.f;
    if (rg < RG)
        for (int r = r0 + rg; r < r1; r += RG)
            if (!keep[r]) acc += to_f32(V[(size_t)r * D + col]);
    part[threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.x < D) {
        float t = 0.f;
        for (int g2 = 0; g2 < RG; ++g2) t += part[g2 * D + threadIdx.x];
        atomicAdd(&p.svec[(size_t)blockIdx.y * D + threadIdx.x], t);
    }
}

// Step a4, streaming part: one pass over V accumulating, per head and token
// split, the Gram matrix of the deleted rows (for R^T R = P G_del P, App. H), the
// Gram matrix of the retained rows (only when k_eff >= d, for the span test) and
// u = sum over deleted j of A_j v_j (for r_bar, Eq. 4).
// grid = (splits, heads_total), 256 threads as a 16x16 grid of (D/16)^2 register tiles.
constexpr int GR_ROWS = 32;

template <typename TIN, int D>
__global__ void __launch_bounds__(256) k_gram(const __grid_constant__ CallDev p)
{
    pdl_wait();
    constexpr int NV = D / 64;               // float4 groups per thread along each axis
    constexpr int MT = 4 * NV;
    __shared__ __align__(16) float Vs[GR_ROWS * D];
    __shared__ float As[GR_ROWS];
    __shared__ int Fs[GR_ROWS];
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int T = c.T;
    const bool need_k = c.k_eff >= D;
    const TIN *Vh = reinterpret_cast<const TIN *>(c.v) + (size_t)lh * T * D;
    const float *A = p.scores + c.tok_off + (size_t)lh * T;
    const uint8_t *keep = p.keep + c.tok_off + (size_t)lh * T;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;

    const int tiles = (T + GR_ROWS - 1) / GR_ROWS;
    const int per = (tiles + p.splits - 1) / p.splits;
    const int t_begin = blockIdx.x * per, t_end = min(tiles, t_begin + per);

    // accumulators as pairs of columns for the two-wide multiply-add
    f32x2 accD[MT][MT / 2], accK[MT][MT / 2];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < MT / 2; ++j) { accD[i][j] = 0ull; accK[i][j] = 0ull; }
    float u = 0.f;

    // a tile's rows are on their way in registers while the tile before is worked on
    constexpr int VEC = 16 / (int)sizeof(TIN), CH = D / VEC, NPV = GR_ROWS * CH / 256;
    static_assert(NPV >= 1 && GR_ROWS * CH % 256 == 0, "whole passes");
    uint4 raw[NPV];
    float a_next = 0.f;
    int f_next = 2;
    auto fetch = [&](int t) {
        const int r0 = t * GR_ROWS;
#pragma unroll
        for (int u2 = 0; u2 < NPV; ++u2) {
            const int i = threadIdx.x + 256 * u2, r = i / CH, ch = i % CH;
            raw[u2] = r0 + r < T ? *reinterpret_cast<const uint4 *>(Vh + (size_t)(r0 + r) * D + ch * VEC) : make_uint4(0u, 0u, 0u, 0u);
        }
        if (threadIdx.x < GR_ROWS) {
            const int j = r0 + threadIdx.x;
            f_next = j < T ? (int)keep[j] : 2;
            a_next = j < T ? A[j] : 0.f;
        }
    };
    if (t_begin < t_end) fetch(t_begin);
    for (int t = t_begin; t < t_end; ++t) {
        __syncthreads();
#pragma unroll
        for (int u2 = 0; u2 < NPV; ++u2) {
            const int i = threadIdx.x + 256 * u2;
            float x[VEC];
            unpack16<TIN>(raw[u2], x);
            float4 *dst = reinterpret_cast<float4 *>(Vs + i * VEC);
#pragma unroll
            for (int e = 0; e < VEC / 4; ++e) dst[e] = make_float4(x[4 * e], x[4 * e + 1], x[4 * e + 2], x[4 * e + 3]);
        }
        if (threadIdx.x < GR_ROWS) { Fs[threadIdx.x] = f_next; As[threadIdx.x] = a_next; }
        __syncthreads();
        if (t + 1 < t_end) fetch(t + 1);
#pragma unroll 1
        for (int r = 0; r < GR_ROWS; ++r) {
            const int f = Fs[r];
            if (f == 2) break;
            if (f == 1 && !need_k) continue;
            float a[MT];
            f32x2 b[MT / 2];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const float4 fa = *reinterpret_cast<const float4 *>(&Vs[r * D + v * 64 + ty * 4]);
                const ulonglong2 fb = *reinterpret_cast<const ulonglong2 *>(&Vs[r * D + v * 64 + tx * 4]);
                a[4 * v] = fa.x; a[4 * v + 1] = fa.y; a[4 * v + 2] = fa.z; a[4 * v + 3] = fa.w;
                b[2 * v] = fb.x; b[2 * v + 1] = fb.y;
            }
            if (f == 0) {
#pragma unroll
                for (int i = 0; i < MT; ++i) {
                    const f32x2 ai = pk(a[i], a[i]);
#pragma unroll
                    for (int j = 0; j < MT / 2; ++j) accD[i][j] = fma2(ai, b[j], accD[i][j]);
                }
                if (threadIdx.x < D) u = fmaf(As[r], Vs[r * D + threadIdx.x], u);
            } else {
#pragma unroll
                for (int i = 0; i < MT; ++i) {
                    const f32x2 ai = pk(a[i], a[i]);
#pragma unroll
                    for (int j = 0; j < MT / 2; ++j) accK[i][j] = fma2(ai, b[j], accK[i][j]);
                }
            }
        }
    }
    const size_t slot = (size_t)blockIdx.y * p.splits + blockIdx.x;
    float *gd = p.gram_d + slot * D * D, *gk = p.gram_k + slot * D * D;
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        const int row = (i / 4) * 64 + ty * 4 + (i & 3);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int col = v * 64 + tx * 4;
            *reinterpret_cast<ulonglong2 *>(&gd[row * D + col]) = make_ulonglong2(accD[i][2 * v], accD[i][2 * v + 1]);
            if (need_k) *reinterpret_cast<ulonglong2 *>(&gk[row * D + col]) = make_ulonglong2(accK[i][2 * v], accK[i][2 * v + 1]);
        }
    }
    if (threadIdx.x < D) p.uvec[slot * D + threadIdx.x] = u;
}

}  // namespace obf
