// Tuned attention-mass kernel (step a1, Eq. 1 with the softmax of App. L.1) for bf16
// caches with head_dim 64 or 128 and up to 256 query rows per KV head (above 128 rows a head is
// worked on as two items of up to 128 rows per chunk, whose masses are added).
//
//   A_j = sum_t softmax_j(q_t . K_j / sqrt(d)),  t over the n_q query rows of the KV head.
//
// The softmax normaliser of a query is needed before any key's mass can be pooled, and it runs over all keys of the head, which
// many blocks share.  A key tile is nevertheless read once, multiplied once and exponentiated once: its weights wait in tensor
// memory, where the logits were, until the head's normalisers are known.
//
//   statistics  S = Q K_chunk^T on the tensor cores, queries on the tensor-memory lanes, 256 keys on the columns.  A thread owns
//       one query and 128 of the keys: their largest logit, rounded up to a whole number m of the log2 domain, then
//       P = exp2(s c - m) (c = log2(e)/sqrt(d)), written back over the logits, and their sum z.  The block publishes (m, z) of
//       the chunk per query and folds those of the head's other chunks as they appear into M_t and Z_t.  References that are whole
//       numbers make every change of reference a shift of the exponent: exact, and no work for the special-function unit.
//   pooling     A_j = sum_t P_tj 2^(m_t - M_t) / Z_t.  The weights are read back in the layout of a matrix fragment, four queries of
//       a pair of columns in a lane; what is left of the sum over queries is seven shuffles per 32 columns and one trip through
//       shared memory.
//
// A block has two slots, each with a chunk of 256 keys, its own half of the tensor memory, its own K and Q buffers, a control
// thread (TMA and MMA) and two groups of four warps, 128 columns each.  A slot works on one chunk after the other, load of the
// next one behind the arithmetic; while one slot waits for its head's other chunks the other one computes.  Chunks are dealt in
// the order of the heads over all slots of the grid, slot 0 of every block before slot 1, so that a block's two chunks are half a
// round apart.  A slot's chunks belong to heads in ascending order, the blocks are all resident (cooperative launch), so that the
// lowest unfinished head always makes progress.  Every wait is bounded (tc_common.cuh).
//
// What bounds it is the latency of a slot's chain, 14000 cycles per 256 keys at T = 8192 (logits 1500, statistics 4200, the
// exchange 4500, pooling 2900, last sum 1000), of which tensor memory allows two at a time; the special-function unit is a third
// busy, the issue slots half, DRAM a third.  Against the form before it (every tile visited twice, for the statistics and for the
// pooling: two exponentials, two MMAs and two trips from L2), calls in bursts of 10 ms and back to back for seconds, where the power
// limit counts what is done: 40 x 8 heads of 8192 positions 459 -> 464 us and 513 -> 481, 36 x 8 of 4096, eviction, 169 -> 169.5 and
// 185 -> 168; one layer of 2048 positions 57.4 -> 53.4, 16 x 8 heads of 64 channels 136 -> 120.  Slower in a burst: 36 x 8 heads of 4096
// with 160 queries 194 -> 214, 128 heads of 12000 171 -> 193 and of 16384 237 -> 268, 8 heads of up to 300 positions with 256
// queries 19 -> 20.5.  Chunks of 512 keys shared by clusters of two blocks, four slots of 128 keys, warps that pool three tiles behind
// the one they compute, and rounds of whole heads (each rank of slots its own, or one head across the ranks) were no faster.
#pragma once

#include "tc_common.cuh"

namespace obf {

constexpr int ST_CHUNK = 256;                       // keys of a chunk
constexpr int ST_SLOTS = 2;                         // chunks in work at a time
constexpr int ST_HALF = ST_CHUNK / 2;               // keys per consumer group
constexpr int ST_GROUPS = 2 * ST_SLOTS;             // consumer groups of four warps
constexpr int ST_PIECES = ST_HALF / 32;             // of 32 columns, each with a reference of its own
constexpr int ST_BOX_BYTES = 128 * 128;              // a 64-channel column block of the queries: 128 rows of 128 bytes
constexpr int ST_THREADS = 32 * ST_SLOTS + 128 * ST_GROUPS;
constexpr int ST_MAX_NQ = 256;                      // two query tiles of 128 rows
constexpr int ST_FLAT = 32;                         // chunks of a head whose statistics are folded in one step: sixteen words a group, all in flight at once
constexpr float ST_LOG2E = 1.4426950408889634f;
template <int D>
constexpr size_t score_tc_smem_bytes()
{
    return 1024 + (size_t)ST_SLOTS * (128 + ST_CHUNK) * D * 2 + (2 + 2 + ST_PIECES + 4) * ST_GROUPS * 128 * sizeof(float);
}

// An item with up to 32 (64) queries, the second one of a head with 160 for instance, would leave three (two) schedulers of
// four without work, as a group's warps own 32 rows of its operand each: the item's queries are loaded
// four times (twice), and the copies share the columns of a tile.  The tensor maps for that, of boxes of 32 rows and one column
// block, sit behind those of the first ST_PART_MAP caches (a third array of maps made every launch 1 to 2 us slower).  Calls with
// more caches have these maps only and load all their queries through them: a head's copies, and with them the order in which
// its statistics are added, never depend on how many caches a call has.
constexpr int ST_PART_MAP = OBF_MAX_CACHES / 2;

struct ScoreItem {
    int cache, lh, chunk;          // lh: KV head in the cache
    int keys;                      // of the chunk, at most ST_CHUNK
    int nq;                        // query rows of the item (at most 128)
    int copies;                    // of them in the operand: 1, 2 or 4
};

// What a block needs of a cache to find its work (kept in shared memory).
struct ScoreTab {
    int item_base, team, T;        // first (head, chunk) pair of the cache, chunks per head
};

// (Head, chunk) pair n of the call, query tile qt.
__device__ __forceinline__ void score_item(const CallDev &p, const ScoreTab *tab, int n, int qt, ScoreItem &it)
{
    int ci = 0;
#pragma unroll 1
    for (int i = 1; i < p.n_caches; ++i)
        if (n >= tab[i].item_base) ci = i;
    const ScoreTab c = tab[ci];
    const int rel = n - c.item_base;
    it.cache = ci;
    it.lh = rel / c.team;
    it.chunk = rel - it.lh * c.team;
    it.keys = min(ST_CHUNK, c.T - it.chunk * ST_CHUNK);
    it.nq = min(128, p.n_q - 128 * qt);
    // (the first term says no more than the second, but for the whole call: without it the consumers' code came out 1 to 3 % slower,
    // 36 x 8 heads of 4096 positions, 128 queries: 133.3 -> 136.7 us, 256 queries: 240 -> 247)
    it.copies = p.sc_single || it.nq > 64 ? 1 : it.nq > 32 ? 2 : 4;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 2^x for a whole number x <= 0 (below -126: zero).  Adding 1.5 * 2^23 + 127 leaves the biased exponent in the low bits.
__device__ __forceinline__ float exp2_whole(float x)
{
    return __uint_as_float(__float_as_uint(fmaxf(x, -127.f) + 12583039.f) << 23);
}

// (M, Z) <- the fold of (M, Z) and (m, z), references whole numbers; (-inf, 0) is the empty one and changes nothing.
__device__ __forceinline__ void score_fold(float &M, float &Z, float m, float z)
{
    const float Mn = fmaxf(M, m), Mf = fmaxf(Mn, -3e38f);                              // (-inf - -inf would be a NaN)
    Z = fmaf(z, exp2_whole(m - Mf), Z * exp2_whole(M - Mf));
    M = Mn;
}

__device__ __forceinline__ void st_relaxed_gpu_u64(unsigned long long *addr, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_relaxed_gpu_u64(const unsigned long long *addr)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(addr) : "memory");
    return v;
}

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Barrier of some of the block's warps.
__device__ __forceinline__ void named_barrier(int id, int threads)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ float logits_max(const uint32_t (&r)[32])
{
    float t[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) t[i] = fmaxf(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
#pragma unroll
    for (int e = 8; e < 32; e += 8)
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = max3(t[i], __uint_as_float(r[e + 2 * i]), __uint_as_float(r[e + 2 * i + 1]));
    return max3(fmaxf(t[0], t[1]), t[2], t[3]);
}

// 32 logits become their weights exp2(s c - m), whose sum is returned.
__device__ __forceinline__ float logits_to_weights(uint32_t (&r)[32], float sc, float nm)
{
    const f32x2 sc2 = pk(sc, sc), nm2 = pk(nm, nm);
    f32x2 z[2] = {0ull, 0ull};
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
        float a, b;
        upk(fma2(pk(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sc2, nm2), a, b);
        a = ex2_approx(a);
        b = ex2_approx(b);
        z[e / 2 % 2] = add2(z[e / 2 % 2], pk(a, b));
        r[e] = __float_as_uint(a);
        r[e + 1] = __float_as_uint(b);
    }
    return sum2(add2(z[0], z[1]));
}

// Weights of 64 keys (two pieces) under 32 queries, fragments of rows 0..15 (lo) and 16..31 (hi): the sums over the queries with
// the factors f (this lane's query, per piece), of this lane's two columns, score_col(lane) and the next one.
__device__ __forceinline__ void pool64(const uint32_t (&lo)[32], const uint32_t (&hi)[32], const float (&f)[2], int lane, float &s0, float &s1)
{
    float v[16];
#pragma unroll
    for (int pc = 0; pc < 2; ++pc) {
        // factors of the four rows of a fragment that this lane holds
        f32x2 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float t = __shfl_sync(0xffffffffu, f[pc], (lane >> 2) + 8 * i);
            w[i] = pk(t, t);
        }
#pragma unroll
        for (int b = 4 * pc; b < 4 * pc + 4; ++b) {
            f32x2 s = mul2(pk(__uint_as_float(lo[4 * b]), __uint_as_float(lo[4 * b + 1])), w[0]);
            s = fma2(pk(__uint_as_float(lo[4 * b + 2]), __uint_as_float(lo[4 * b + 3])), w[1], s);
            s = fma2(pk(__uint_as_float(hi[4 * b]), __uint_as_float(hi[4 * b + 1])), w[2], s);
            s = fma2(pk(__uint_as_float(hi[4 * b + 2]), __uint_as_float(hi[4 * b + 3])), w[3], s);
            upk(s, v[2 * b], v[2 * b + 1]);
        }
    }
    // over the eight lanes that share lane mod 4, half as many values at every step
#pragma unroll
    for (int n = 8, off = 16; n >= 2; n >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    s0 = v[0];
    s1 = v[1];
}
// Lane bit 4: piece, bits 3, 2: block of eight columns in it, bits 1, 0: pair of columns.
__device__ __forceinline__ int score_col(int lane) { return 8 * (lane >> 2) + 2 * (lane & 3); }

// LONG: some head of the call has more than ST_FLAT chunks (an instantiation of its own: with both ways of folding in one, heads of up
// to ST_FLAT chunks were 1 to 3 % slower).  Folding all chunks of a long head in every slot, sixteen words a sweep, cost 8 heads of 75000
// positions 165 us, this way 77 (the kernel that visited every tile twice: 91); 8 heads of 16384: 27.3, 25.4, 23.9; 128 heads of 12000: 189, 180, 157.
template <int D, bool LONG>
__global__ void __launch_bounds__(ST_THREADS, 1) k_score_tc(const __grid_constant__ CallDev p, const __grid_constant__ TcMaps tm)
{
    constexpr int Q_BYTES = 128 * D * 2, K_BYTES = ST_CHUNK * D * 2;
    extern __shared__ uint8_t st_smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(st_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *q_s = base;                                           // per slot [128 queries][d] bf16, 64-column blocks
    uint8_t *k_s = q_s + ST_SLOTS * Q_BYTES;                       // per slot [256 keys][d]
    float *s_m = reinterpret_cast<float *>(k_s + ST_SLOTS * K_BYTES);      // [group][128 rows] references of a group's columns
    float *s_z = s_m + ST_GROUPS * 128;                            // [group][128 rows] their sums
    float *s_fm = s_z + ST_GROUPS * 128;                           // [group][128 queries] references of the chunks the group folds
    float *s_fz = s_fm + ST_GROUPS * 128;
    float *s_pm = s_fz + ST_GROUPS * 128;                          // [group][piece][128 rows] references of a thread's pieces
    float *s_col = s_pm + ST_GROUPS * ST_PIECES * 128;             // [group][quarter][128 keys] pooled over a quarter's queries
    __shared__ uint64_t bar_full[ST_SLOTS], bar_t_full[ST_GROUPS], bar_t_empty[ST_GROUPS];
    __shared__ ScoreTab s_tab[OBF_MAX_CACHES];
    __shared__ uint32_t s_tmem, s_abort;

    const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
    const int n_items = p.sc_items, stride = ST_SLOTS * (int)gridDim.x;
    tc::WaitCtx wc{&s_abort, p.status, p.wait_limit_ns};

    if (tid == 0) {
        s_abort = 0u;
        for (int s = 0; s < ST_SLOTS; ++s) tc::mbar_init(&bar_full[s], 1);
        for (int g = 0; g < ST_GROUPS; ++g) {
            tc::mbar_init(&bar_t_full[g], 1);
            tc::mbar_init(&bar_t_empty[g], 4);                     // the group's warps
        }
        tc::mbar_init_fence();
    }
    if (tid >= 64 && tid < 64 + p.n_caches) {
        const CacheDev &c = p.c[tid - 64];
        ScoreTab e;
        e.item_base = c.sc_item_base;
        e.team = c.sc_team;
        e.T = c.T;
        s_tab[tid - 64] = e;
    }
    if (warp == 1) tc::tmem_alloc(&s_tmem, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp < ST_SLOTS) {
        // ---------------- control thread of a slot: TMA and MMA ----------------
        if (lane == 0) {
            const int slot = warp;
            const uint32_t q_addr = tc::smem_u32(q_s + slot * Q_BYTES), k_addr = tc::smem_u32(k_s + slot * K_BYTES);
            uint64_t *full = &bar_full[slot];
            // queries of an item, and its keys unless the item before had the same: both buffers are free
            auto load = [&](const ScoreItem &it, int qt, bool keys) {
                tc::mbar_expect_tx(full, Q_BYTES + (keys ? K_BYTES : 0));
                if (keys) tc::tma_load_rows(k_addr, &tm.a[it.cache], full, it.chunk * ST_CHUNK, it.lh);
                if (it.copies > 1 || p.n_caches > ST_PART_MAP) {
                    const CUtensorMap *boxes = &tm.b[(p.n_caches > ST_PART_MAP ? 0 : ST_PART_MAP) + it.cache];
                    for (int r = 0; r < 4; ++r)
                        for (int b = 0; b < D / 64; ++b)
                            tc::tma_load_block(q_addr + r * 32 * 128 + b * ST_BOX_BYTES, boxes, full,
                                               qt * 128 + 32 * (r % (4 / it.copies)), b, it.lh);
                } else {
                    tc::tma_load_rows(q_addr, &tm.b[it.cache], full, qt * 128, it.lh);          // rows past n_q read as zero
                }
            };
            int n = slot * (int)gridDim.x + (int)blockIdx.x, qt = 0;
            uint32_t u = 0, used[2] = {0u, 0u};                    // items of this slot so far, and the tiles handed to the tensor cores
            ScoreItem item;
            bool have = n < n_items;
            if (have) {
                score_item(p, s_tab, n, qt, item);
                load(item, qt, true);
            }
            while (have) {
                if (!tc::mbar_wait(full, u & 1u, wc, 20)) break;
                // operand descriptors: a step of 16 channels moves the start address by 32 bytes along the swizzled row, and to
                // the next column block after four
                const uint64_t dq = tc::smem_desc_sw128(q_addr, 16, 1024);
                const int halves = item.keys > ST_HALF ? 2 : 1;
                bool dead = false;
                // (one half after the other: the first group computes while the second half is multiplied)
                for (int h = 0; h < halves && !dead; ++h) {
                    const int g = 2 * slot + h;
                    if (!tc::mbar_wait(&bar_t_empty[g], (used[h] & 1u) ^ 1u, wc, 20)) { dead = true; break; }
                    tc::tc_fence_after();
                    const uint64_t dk = tc::smem_desc_sw128(k_addr + h * ST_HALF * 128, 16, 1024);
                    const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)(min(item.keys - h * ST_HALF, ST_HALF) + 31) & ~31u, 0, 0);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        tc::umma_bf16(tmem + g * ST_HALF, dq + (uint64_t)((kk >> 2) * (ST_BOX_BYTES >> 4) + (kk & 3) * 2),
                                      dk + (uint64_t)((kk >> 2) * (ST_CHUNK * 128 >> 4) + (kk & 3) * 2), idesc, kk > 0 ? 1u : 0u);
                    tc::umma_commit(&bar_t_full[g]);
                    ++used[h];
                }
                if (dead) break;
                // the next item's operands once the instructions have read this one's
                bool same = true;
                if (++qt == p.sc_qt) {
                    qt = 0;
                    n += stride;
                    same = false;
                }
                have = n < n_items;
                if (have) score_item(p, s_tab, n, qt, item);
                ++u;
                for (int h = 0; h < halves && !dead; ++h) dead = !tc::mbar_wait(&bar_t_full[2 * slot + h], (used[h] - 1) & 1u, wc, 20);
                if (dead) { have = false; break; }                 // (nothing more has been loaded)
                if (have) load(item, qt, !same);
            }
            // nothing this thread started may still be in flight when the block exits, also where a wait ran out
            const uint32_t loads = u + (have ? 1u : 0u);
            if (loads > 0) tc::mbar_drain(full, (loads - 1) & 1u, wc);
            for (int h = 0; h < 2; ++h)
                if (used[h] > 0) tc::mbar_drain(&bar_t_full[2 * slot + h], (used[h] - 1) & 1u, wc);
        }
    } else {
        // ---------------- consumers ----------------
        const int q = warp & 3;                        // tensor-memory lane quarter this warp may touch
        const int group = (warp - ST_SLOTS) >> 2, slot = group >> 1, half = group & 1;
        const int row = q * 32 + lane;                 // lane of the accumulators, and the key of the half this thread stores
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(group * ST_HALF);
        const float sc = ST_LOG2E * rsqrtf((float)D);
        float *col = s_col + (group * 4 + q) * 128, *pm = s_pm + group * ST_PIECES * 128 + row;
        uint32_t used = 0;                             // items with keys in this half so far
#pragma unroll 1
        for (int n = slot * (int)gridDim.x + (int)blockIdx.x; n < n_items; n += stride) {
            float pooled = 0.f;
#pragma unroll 1
            for (int qt = 0; qt < p.sc_qt; ++qt) {
                ScoreItem it;
                score_item(p, s_tab, n, qt, it);
                const CacheDev &c = p.c[it.cache];
                const int keys = it.keys - half * ST_HALF;             // of this group's columns (none: not more than 0)
                // An item costs by what it has: pieces of 32 columns that hold keys, quarters that hold queries.  With copies of
                // the queries a quarter walks its share of the pieces.
                const int share = 4 / it.copies, n_pc = min(4, (keys + 31) >> 5), n_quarters = min(share, (it.nq + 31) >> 5);
                const int first = it.copies > 1 ? q / share * share : 0;
                const int last = it.copies > 1 ? min(first + share, n_pc) : 32 * q < it.nq ? n_pc : 0;
                const int rows = 128 / it.copies, query = row & (rows - 1);
                const int lv = it.lh * p.sc_qt + qt;
                unsigned long long *words = reinterpret_cast<unsigned long long *>(p.sc_part) + (c.sc_part_off + (size_t)lv * c.sc_team * 128);
                const float extra = (c.lse_extra && query < it.nq) ? c.lse_extra[(size_t)it.lh * p.n_q + 128 * qt + query] : -INFINITY;
                if (keys > 0) {
                    tc::mbar_wait(&bar_t_full[group], used++ & 1u, wc, 20);
                    __syncwarp();
                    tc::tc_fence_after();
                }
                // ======== statistics: reference and sum of this thread's query over its columns, weights in place ========
                float m = -INFINITY, z = 0.f;
                if (keys < ST_HALF && first < last) {
                    // a head's ragged end: no such keys
#pragma unroll 1
                    for (int e = keys; e < 32 * n_pc; ++e) tc::tmem_st1(ta + e, 0xff800000u);
                    tc::tmem_st_wait();
                }
#pragma unroll 1
                for (int pc = first; pc < last; ++pc) {
                    uint32_t r[32];
                    tc::tmem_ld32(ta + 32u * pc, r);
                    tc::tmem_ld_wait32(r);
                    const float mp = ceilf(logits_max(r) * sc);
                    const float zp = logits_to_weights(r, sc, -fmaxf(mp, -3e38f));     // (no finite key: -inf - -inf would be a NaN)
                    tc::tmem_st32(ta + 32u * pc, r);
                    pm[128 * pc] = mp;
                    score_fold(m, z, mp, zp);
                }
                tc::tmem_st_wait();
                s_m[group * 128 + row] = m;
                s_z[group * 128 + row] = z;
                named_barrier(1 + slot, 256);
                // ======== the chunk's statistics out, the head's in ========
                // Per (head, chunk, query) one 64-bit word, (reference, sum): the sum's bits are zero (as cleared before the launch)
                // until it is published, never zero afterwards (the sum of a finite maximum's own weight is above a half; the sum
                // of a chunk without a finite logit is written as -0).  A word vouches for itself, so nothing is counted and
                // nothing fenced.  The two groups of the slot fold half of the head's chunks each, in ascending order.
                // In a head of more than ST_FLAT chunks every sixteenth chunk first folds the fifteen after it into its own (hop 0) and
                // publishes the sum of the sixteen; these sums come first among the head's words and are what everybody folds (hop 1).
                // Which way a head goes, and so the order of its sums, depends on its own length alone.
                {
                    float M = -INFINITY, Z = 0.f;
                    if (half == 0 && row < it.nq) {
#pragma unroll 1
                        for (int r = row; r < 128; r += rows) {
                            score_fold(M, Z, s_m[group * 128 + r], s_z[group * 128 + r]);
                            score_fold(M, Z, s_m[(group + 1) * 128 + r], s_z[(group + 1) * 128 + r]);
                        }
                    }
                    const bool flat = !LONG || c.sc_team <= ST_FLAT;
                    const int n_words = flat ? c.sc_team : (c.sc_team + 15) >> 4, per = (n_words + 1) >> 1;
                    const int behind = n_words + 15 * (it.chunk >> 4);             // where the fifteen words are
                    const int at = flat ? it.chunk : it.chunk & 15 ? behind + (it.chunk & 15) - 1 : it.chunk >> 4;
#pragma unroll 1
                    for (int hop = !flat && half == 0 && !(it.chunk & 15) ? 0 : 1; hop < 2; ++hop) {
                        if (hop == 1) {
                            if (half == 0 && row < it.nq && !p.debug_drop_publish) {
                                const uint32_t zb = Z == 0.f ? 0x80000000u : __float_as_uint(Z);
                                st_relaxed_gpu_u64(words + (size_t)at * 128 + row, ((unsigned long long)zb << 32) | __float_as_uint(M));
                            }
                            M = -INFINITY;
                            Z = 0.f;
                        }
                        const int c0 = hop == 0 ? behind : per * half;
                        const int c_end = hop == 0 ? min(behind + 15, c.sc_team) : min(n_words, per * (half + 1));
                        if (c0 < c_end && 32 * q < it.nq) {
                            // at most sixteen words, in flight together; a warp without queries has nothing to fetch
                            unsigned long long w[16];
                            const unsigned long long *from = words + (size_t)c0 * 128 + row;
#pragma unroll
                            for (int e = 0; e < 16; ++e) w[e] = (c0 + e < c_end && row < it.nq) ? 0ull : 0x80000000ff800000ull;   // (-inf, -0)
                            // From sixteen chunks on they are never there at once, and polls in vain hold up those who publish; with fewer
                            // the pause would be longer than the wait (36 x 8 heads of 3500 positions, 64 channels: 106.7 us without, 109.9
                            // with one of 400 ns).  600, 400 and no ns: 32 x 8 heads of 8192 positions with 32 queries 188.1, 190.6, 195.3 us,
                            // with 128 231.3, 229.0, 235.1, with 160 377.6, 370.2, 372.0, with 128 of 64 channels 220.0, 212.8, 211.0;
                            // 36 x 8 of 4096 with 128 131.4, 130.5, 133.6.
                            if (hop == 1 && c.sc_team >= 16) __nanosleep(600);
                            uint64_t t0 = 0ull;
                            for (;;) {
#pragma unroll
                                for (int e = 0; e < 16; ++e)
                                    if ((uint32_t)(w[e] >> 32) == 0u) w[e] = ld_relaxed_gpu_u64(from + e * 128);
                                uint32_t least = 0xFFFFFFFFu;
#pragma unroll
                                for (int e = 0; e < 16; ++e) least = min(least, (uint32_t)(w[e] >> 32));
                                // the warp leaves the loop as one: votes, not per-lane exits
                                if (__all_sync(0xffffffffu, least != 0u)) break;
                                const uint64_t now = tc::global_ns();
                                if (t0 == 0ull) t0 = now;
                                if (__any_sync(0xffffffffu, *(volatile uint32_t *)&s_abort != 0u || now - t0 > p.wait_limit_ns)) {
                                    if (lane == 0) {
                                        s_abort = 1u;
                                        atomicOr(p.status, OBF_DEV_TIMEOUT);
                                    }
                                    break;
                                }
                                __nanosleep(32);
                            }
                            float Mn = M;
#pragma unroll
                            for (int e = 0; e < 16; e += 2) Mn = max3(Mn, __uint_as_float((uint32_t)w[e]), __uint_as_float((uint32_t)w[e + 1]));
                            const float Mf = fmaxf(Mn, -3e38f);
                            Z *= exp2_whole(M - Mf);
#pragma unroll
                            for (int e = 0; e < 16; ++e) Z = fmaf(__uint_as_float((uint32_t)(w[e] >> 32)), exp2_whole(__uint_as_float((uint32_t)w[e]) - Mf), Z);
                            M = Mn;
                        }
                    }
                    s_fm[group * 128 + row] = M;
                    s_fz[group * 128 + row] = Z;
                }
                named_barrier(1 + slot, 256);
                // ======== pooling: the mass of every key over this item's queries ========
                float Mf = 0.f, rz = 0.f;                                  // padding rows count for nothing
                {
                    float M = s_fm[2 * slot * 128 + query], Z = s_fz[2 * slot * 128 + query];
                    score_fold(M, Z, s_fm[(2 * slot + 1) * 128 + query], s_fz[(2 * slot + 1) * 128 + query]);
                    if (query < it.nq) {
                        // the keys outside the prompt take their share of the normaliser
                        const float L = extra * ST_LOG2E;
                        if (L > -INFINITY) {
                            const float Mn = fmaxf(M, ceilf(L));
                            Z = Z * exp2_whole(fmaxf(M, -3e38f) - Mn) + exp2f(L - Mn);
                            M = Mn;
                        }
                        Mf = fmaxf(M, -3e38f);
                        rz = 1.f / Z;
                        if (!(Z > 0.f) || !isfinite(M) || !isfinite(rz)) {
                            if (it.chunk == 0 && !s_abort) atomicOr(p.status, OBF_DEV_NONFINITE);
                            rz = __int_as_float(0x7fc00000);
                        }
                        if (s_abort) { Mf = 3e38f; rz = 0.f; }
                    }
                }
#pragma unroll 1
                for (int pc = first; pc < last; pc += 2) {
                    // two pieces, the second of them perhaps one too many; the weights' way from tensor memory is behind the factors
                    uint32_t lo[32], hi[32];
                    const int p0 = min(pc, ST_PIECES - 2);
                    tc::tmem_ld_frag(ta + 32u * p0, lo);
                    tc::tmem_ld_frag(ta + 32u * p0 + (16u << 16), hi);
                    const float f[2] = {exp2_whole(pm[128 * p0] - Mf) * rz, exp2_whole(pm[128 * p0 + 128] - Mf) * rz};
                    tc::tmem_ld_wait64(lo, hi);
                    float s0, s1;
                    pool64(lo, hi, f, lane, s0, s1);
                    const int at = p0 + (lane >> 4);
                    if (at >= first && at < last) *reinterpret_cast<float2 *>(col + 32 * p0 + score_col(lane)) = make_float2(s0, s1);
                }
                if (keys > 0) tc::tc_fence_before();
                __syncwarp();
                if (lane == 0 && keys > 0) tc::mbar_arrive(&bar_t_empty[group]);
                named_barrier(1 + ST_SLOTS + group, 128);
                if (row < keys) {
                    const float *cs = s_col + (group * 4 + (row >> 5) / share * share) * 128 + row;
                    float a = 0.f;
                    for (int e = 0; e < n_quarters; ++e) a += cs[e * 128];
                    pooled += a;
                    if (qt + 1 == p.sc_qt) {
                        const int j = it.chunk * ST_CHUNK + half * ST_HALF + row;
                        if (!isfinite(pooled)) atomicOr(p.status, OBF_DEV_NONFINITE);
                        p.scores[c.tok_off + (size_t)it.lh * s_tab[it.cache].T + j] = pooled;
                        if (c.scores_out && p.sc_qt == 1) c.scores_out[(size_t)it.lh * s_tab[it.cache].T + j] = pooled;
                    }
                }
            }
        }
    }

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

// Heads with two query tiles whose masses the caller wants: a copy.
// grid = (ceil(T_max / 256), heads_total).
__global__ void __launch_bounds__(256) k_score_join(const __grid_constant__ CallDev p)
{
    pdl_wait();
    int ci, lh;
    locate(p, blockIdx.y, ci, lh);
    const CacheDev &c = p.c[ci];
    const int j = blockIdx.x * 256 + threadIdx.x;
    if (j < c.T && c.scores_out) c.scores_out[(size_t)lh * c.T + j] = p.scores[c.tok_off + (size_t)lh * c.T + j];
}

}  // namespace obf
