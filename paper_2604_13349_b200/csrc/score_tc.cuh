// Tuned attention-mass kernel (step a1, Eq. 1 with the softmax of App. L.1) for bf16
// caches with head_dim 64 or 128 and up to 256 query rows per KV head (above 128 rows a head is
// worked on as two items of up to 128 rows, which add their masses onto zeros).
//
//   A_j = sum_t softmax_j(q_t . K_j / sqrt(d)),  t over the n_q query rows of the KV head.
//
// The softmax normaliser of a query is needed before any key's mass can be pooled, so
// the keys are visited twice.  K comes from HBM once: the second visit follows the first
// closely enough to be served by the L2 cache.
//
//   pass A (statistics)  S = Q K_tile^T on the tensor cores with the QUERIES on the
//       tensor-memory lanes: a thread owns one query and keeps a reference m_t, its maximum
//       up to a margin (stats_update), and the sum z_t = sum_j exp2(s_tj c - m_t)
//       (c = log2(e)/sqrt(d)) over the block's
//       chunk of keys; nothing crosses lanes.  Per (head, chunk) the block publishes
//       (m_t, z_t); every block of the head's team folds all of them into
//       M'_t = M_t + log2(Z_t).
//   pass B (pooling)     S^T = K_tile Q^T with the KEYS on the lanes: a thread owns one
//       key and sums exp2(s_tj c - M'_t) = softmax_j over all queries of the tile;
//       again nothing crosses lanes, and a key's mass is complete in one thread.
//
// A head's T keys are cut into chunks of 4 tiles of 128 keys; a head's chunks are worked
// on by a team of blocks in the same round.  Rounds are dealt as
// (head, chunk) = (round * heads_per_round + block / team, block % team), and a block
// runs A(i), B(i - ST_LAG) for i = 0, 1, ..: a chunk's second visit comes one round after
// its first, when every block of its team has published (a longer lag pushes the chunk out
// of the L2 cache before its second visit).
// The wait for M' is bounded like every other wait (tc_common.cuh).
//
// Block = 23 warps: warp 0 TMA producer (K tiles through a 4-stage ring, asked into L2 one
// round ahead; Q of a pass is loaded while the pass before it runs, into the buffer of its
// kind: one for the statistics passes, one for the pooling passes, which read Q again),
// warps 1 and 22 MMA issuers, alternate tiles (accumulators in a 4-deep ring of 128 tensor-memory columns),
// warps 2..17 consumers in four groups of four, group g taking the tiles with index g (mod 4), so
// that every scheduler holds one warp of each group and the four are at different points of
// their tiles: a warp owns the 32 tensor-memory lanes of its quarter and walks the 128 columns
// of its tile 16 at a time, the next 16 on their way while it works (a rolled loop over two register
// sets: unrolled, with pieces of 32, that was slower than load, wait, work); the tile goes back to the
// MMA issuers when its last columns are in registers.  A key's pooled mass is complete in one thread.
// Measured alternatives that were slower: two groups (two warps per scheduler), a share of the
// exponentials evaluated as a polynomial on the FMA pipe (the special-function unit is busy two
// thirds of the time at most: it is not what the warps wait for).  With no arithmetic at all the
// kernel takes 0.202 of its 0.250 ms (40 x 8 heads, T = 8192): the supply of tiles bounds it.
// Warps 18..21 are the messengers, a query per lane: they publish the chunk statistics the consumers leave in
// shared memory and collect and fold the team's into the head's M' for the pooling pass a round later, so
// that the consumers never wait for global memory.
#pragma once

#include "tc_common.cuh"

namespace obf {

constexpr int ST_TILES = 4;                         // 128-key tiles per chunk
constexpr int ST_CHUNK = ST_TILES * 128;
constexpr int ST_STAGES = 4;                        // K tiles in flight in shared memory
constexpr int ST_TBUF = 4;                          // accumulator tiles in tensor memory
constexpr int ST_LAG = 1;                           // rounds between a chunk's statistics pass and its pooling pass
constexpr int ST_BOX_BYTES = 128 * 128;              // a 64-channel column block of a tile: 128 rows of 128 bytes
constexpr int ST_GROUPS = 4;                        // consumer groups of four warps, one accumulator tile each
constexpr int ST_CONSUMERS = ST_GROUPS * 128;
constexpr int ST_MESSENGERS = 4;                    // messenger warps, a query per lane
constexpr int ST_THREADS = 64 + ST_CONSUMERS + 32 * ST_MESSENGERS + 32;
constexpr int ST_MAX_NQ = 256;                      // two query tiles of 128 rows
constexpr float ST_LOG2E = 1.4426950408889634f;
// M' has the magnitude of the logits and its rounding, up to 2^-18 of a weight, is common to all keys of a query.  Heads of 64
// channels were computed without it and keep that precision: their references stay within 1 of the maximum (64 otherwise), and
// a weight is exp2(s c - M) times 1 / Z.  Sum of a row's weights at logits of 100: off by up to 4e-6 with M', 3e-7 so; masses
// against 64 bits, T = 1024, 160 queries, small logits: 2.1e-7 and 1.3e-7 (at large ones 4e-7 either way, from the tensor cores'
// sums).
template <int D>
constexpr bool ST_FINE = D == 64;
template <int D>
constexpr size_t score_tc_smem_bytes() { return 1024 + (size_t)(2 + ST_STAGES) * 128 * D * 2 + (2 * 2 * ST_GROUPS * 128 + (ST_FINE<D> ? 4 : 2) * 128) * sizeof(float) + 64; }
static_assert(ST_STAGES == ST_TBUF, "a ring stage is released by the accumulator barrier of the same index");

// An item with up to 32 (64) queries, the second one of a head with 160 for instance, would leave three (two) schedulers of
// four without work in a statistics pass, as a group's warps own 32 rows of its operand each: the item's queries are loaded
// four times (twice), and the copies share the columns of a tile.  The tensor maps for that sit behind those of the first
// ST_PART_MAP caches (a third array of maps made every launch 1 to 2 us slower); calls with more caches go without.
// 36 x 8 heads of 160 queries, T = 2048: 105 -> 97 us; 2 x 4 heads of 64 queries, T = 400: 10.2 -> 9.2.
constexpr int ST_PART_MAP = OBF_MAX_CACHES / 2;

struct ScoreItem {
    int r, cache, lh, chunk, nt;   // r: round; lh: KV head in the cache; nt: tiles of the chunk that hold at least one key
    int lv, qt;                    // lv = lh * query tiles + qt: the (head, query tile) pair; qt: which 128 query rows
    int nq;                        // query rows of the item (at most 128)
    int copies;                    // of them in the operand of its statistics pass: 1, 2 or 4
};

// What a block needs of a cache to find its work of a round (kept in shared memory).
struct ScoreTab {
    int round_base, hpr, hi, chunk, T;   // hi, chunk: this block's head slot and chunk inside a round of the cache
};

// Work of this block in round `r`; false when the block idles in that round.
__device__ __forceinline__ bool score_item(const CallDev &p, const ScoreTab *tab, int r, ScoreItem &it)
{
    int ci = 0;
#pragma unroll 1
    for (int i = 1; i < p.n_caches; ++i)
        if (r >= tab[i].round_base) ci = i;
    const ScoreTab c = tab[ci];
    if (c.hi >= c.hpr) return false;
    // a head with more than 128 query rows is dealt as two items, one per 128 rows: softmax rows are independent,
    // so the head's masses are the sum of the two items' masses
    const int lv = (r - c.round_base) * c.hpr + c.hi;
    if (lv >= p.heads_per_cache * p.sc_qt) return false;
    it.r = r;
    it.cache = ci;
    it.lv = lv;
    it.lh = p.sc_qt == 2 ? lv >> 1 : lv;
    // (a block that meets an even number of items a round would always get the same tile of a head, half of the blocks the
    // larger one: the two change places from round to round; T = 1024, teams of two blocks: 62 -> 54 us)
    it.qt = p.sc_qt == 2 ? (lv ^ ((c.hpr & 1) ? 0 : r - c.round_base)) & 1 : 0;
    it.nq = min(128, p.n_q - 128 * it.qt);
    it.copies = p.n_caches > ST_PART_MAP || it.nq > 64 ? 1 : it.nq > 32 ? 2 : 4;
    it.chunk = c.chunk;
    const int tiles = (c.T - c.chunk * ST_CHUNK + 127) >> 7;
    it.nt = tiles < ST_TILES ? tiles : ST_TILES;
    return true;
}

// The passes of a block in the order it runs them: A(i), B(i - ST_LAG) for i = 0, 1, ..
struct PassIter {
    int i = 0, ph = 0;
};

// Next pass with work for this block: kind 0 = statistics, 1 = pooling.
__device__ __forceinline__ bool next_pass(const CallDev &p, const ScoreTab *tab, int R, PassIter &s, ScoreItem &item, int &kind)
{
    while (s.i < R + ST_LAG) {
        const int ph = s.ph, r = ph == 0 ? s.i : s.i - ST_LAG;
        if (ph == 0) s.ph = 1;
        else { s.ph = 0; ++s.i; }
        if (r < 0 || r >= R) continue;
        if (!score_item(p, tab, r, item)) continue;
        kind = ph;
        return true;
    }
    return false;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
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

// Two logits at a time: exp2(s c + o), added to an accumulator pair.  The multiply-add and the sum are two-wide.
__device__ __forceinline__ void exp2_add(f32x2 &acc, uint32_t s0, uint32_t s1, f32x2 sc, f32x2 o)
{
    float a, b;
    upk(fma2(pk(__uint_as_float(s0), __uint_as_float(s1)), sc, o), a, b);
    acc = add2(acc, pk(ex2_approx(a), ex2_approx(b)));
}

// Two logits at a time: exp2(s c + o) w, added to an accumulator pair.
__device__ __forceinline__ void exp2_fma(f32x2 &acc, uint32_t s0, uint32_t s1, f32x2 sc, f32x2 o, f32x2 w)
{
    float a, b;
    upk(fma2(pk(__uint_as_float(s0), __uint_as_float(s1)), sc, o), a, b);
    acc = fma2(pk(ex2_approx(a), ex2_approx(b)), w, acc);
}

// Pass A on one thread's 16 logits of a piece: reference m (log2 domain) and sum z of exp2(s c - m) of one query.  The
// reference is the largest logit up to the last piece that exceeded it by MARGIN = 64: no more is needed for a sum that neither
// overflows nor loses its small terms, and the step that changes it is then a branch hardly ever taken.  (With 1 the terms that
// count lose no bits to the distance from the reference.)  z >= 1 wherever a finite logit was met.  With MASKED only the first
// n_valid columns are keys.
template <bool MASKED, int MARGIN>
__device__ __forceinline__ void stats_update(uint32_t (&rr)[16], int n_valid, float sc, float &m, float &z)
{
    if (MASKED) {
#pragma unroll
        for (int e = 0; e < 16; ++e)
            if (e >= n_valid) rr[e] = 0xff800000u;                                     // -inf: no such key
    }
    float t0 = fmaxf(__uint_as_float(rr[0]), __uint_as_float(rr[1])), t1 = fmaxf(__uint_as_float(rr[2]), __uint_as_float(rr[3]));
#pragma unroll
    for (int e = 4; e < 16; e += 4) {
        t0 = max3(t0, __uint_as_float(rr[e]), __uint_as_float(rr[e + 1]));
        t1 = max3(t1, __uint_as_float(rr[e + 2]), __uint_as_float(rr[e + 3]));
    }
    const float t = fmaxf(t0, t1) * sc;
    if (t > m + (float)MARGIN) {
        z *= ex2_approx(m - t);                                                        // (0 * exp2(-inf) at first)
        m = t;
    }
    const float mf = fmaxf(m, -3e38f);                                                 // (no key yet: -inf - -inf would be a NaN)
    const f32x2 sc2 = pk(sc, sc), o = pk(-mf, -mf);
    f32x2 z0 = 0ull, z1 = 0ull;
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
        exp2_add(z0, rr[e], rr[e + 1], sc2, o);
        exp2_add(z1, rr[e + 2], rr[e + 3], sc2, o);
    }
    z += sum2(add2(z0, z1));
}

// Pass B on one thread's 16 logits of a piece: the softmax weights of one key under 16 queries, added to a0, a1.
// mp: -M'_t of those queries (shared memory, the same address for every lane); with FINE -M_t, and 1 / Z_t behind it at rz.
template <bool FINE>
__device__ __forceinline__ void pool_piece(const uint32_t (&rr)[16], const float *mp, const float *rz, float sc, f32x2 &a0, f32x2 &a1)
{
    const f32x2 sc2 = pk(sc, sc);
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(mp + e);
        if constexpr (FINE) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(rz + e);
            exp2_fma(a0, rr[e], rr[e + 1], sc2, v.x, w.x);
            exp2_fma(a1, rr[e + 2], rr[e + 3], sc2, v.y, w.y);
        } else {
            exp2_add(a0, rr[e], rr[e + 1], sc2, v.x);
            exp2_add(a1, rr[e + 2], rr[e + 3], sc2, v.y);
        }
    }
}

template <int D>
__global__ void __launch_bounds__(ST_THREADS, 1) k_score_tc(const __grid_constant__ CallDev p, const __grid_constant__ TcMaps tm)
{
    constexpr int ST_TILE_BYTES = 128 * D * 2;
    extern __shared__ uint8_t st_smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(st_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t *q_s = base;                                           // 2 x [128 x 128] bf16: Q of a statistics pass, Q of a pooling pass; two 64-column halves each
    uint8_t *ring = q_s + 2 * ST_TILE_BYTES;                       // ST_STAGES x 32 KiB
    float *s_m = reinterpret_cast<float *>(ring + ST_STAGES * ST_TILE_BYTES);   // [2][tile of the chunk][128 queries] tile maxima
    float *s_z = s_m + 2 * ST_GROUPS * 128;                        // [2][tile of the chunk][128 queries] tile sums
    constexpr bool FINE = ST_FINE<D>;
    float *s_mp = s_z + 2 * ST_GROUPS * 128;                       // [2][128] -M'_t of the head being pooled
    float *s_rz = s_mp + 2 * 128;                                  // with FINE: -M_t there, [2][128] 1 / Z_t here
    __shared__ uint64_t bar_q_full[2], bar_q_free[2], bar_full[ST_STAGES];
    __shared__ uint64_t bar_t_full[ST_TBUF], bar_t_empty[ST_TBUF];
    __shared__ uint64_t bar_st_ready[2], bar_mp_ready[2];
    __shared__ ScoreTab s_tab[OBF_MAX_CACHES];
    __shared__ uint32_t s_tmem, s_abort;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = p.sc_rounds;
    tc::WaitCtx wc{&s_abort, p.status, p.wait_limit_ns};

    if (tid == 0) {
        s_abort = 0u;
        for (int b = 0; b < 2; ++b) { tc::mbar_init(&bar_q_full[b], 1); tc::mbar_init(&bar_q_free[b], 2); }
        for (int s = 0; s < ST_STAGES; ++s) tc::mbar_init(&bar_full[s], 1);
        for (int s = 0; s < ST_TBUF; ++s) {
            tc::mbar_init(&bar_t_full[s], 1);
            tc::mbar_init(&bar_t_empty[s], 4);                  // the four warps of the group that owns the tile
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&bar_st_ready[b], ST_CONSUMERS / 32);
            tc::mbar_init(&bar_mp_ready[b], ST_MESSENGERS);
        }
        tc::mbar_init_fence();
    }
    if (tid >= 64 && tid < 64 + p.n_caches) {
        const CacheDev &c = p.c[tid - 64];
        ScoreTab e;
        e.round_base = c.sc_round_base;
        e.hpr = c.sc_hpr;
        e.hi = (int)blockIdx.x / c.sc_team;
        e.chunk = (int)blockIdx.x - e.hi * c.sc_team;
        e.T = c.T;
        s_tab[tid - 64] = e;
    }
    if (warp == 1) tc::tmem_alloc(&s_tmem, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t it = 0, nq[2] = {0u, 0u};
            bool dead = false;
            // Q of a pass goes to the buffer of its kind once the MMAs of that buffer's last user are done
            auto load_q = [&](const ScoreItem &item, int kind) -> bool {
                if (nq[kind] > 0 && !tc::mbar_wait(&bar_q_free[kind], (nq[kind] - 1) & 1u, wc, 64)) return false;
                const uint32_t qdst = tc::smem_u32(q_s + kind * ST_TILE_BYTES);
                tc::mbar_expect_tx(&bar_q_full[kind], ST_TILE_BYTES);
                if (kind == 0 && item.copies > 1) {
                    for (int r = 0; r < 4; ++r)
                        for (int b = 0; b < D / 64; ++b)
                            tc::tma_load_block(qdst + r * 32 * 128 + b * ST_BOX_BYTES, &tm.b[ST_PART_MAP + item.cache], &bar_q_full[kind],
                                               item.qt * 128 + 32 * (r % (4 / item.copies)), b, item.lh);
                } else {
                    tc::tma_load_rows(qdst, &tm.b[item.cache], &bar_q_full[kind], item.qt * 128, item.lh);      // rows past n_q read as zero
                }
                ++nq[kind];
                return true;
            };
            PassIter pi;
            ScoreItem item, nxt;
            int kind = 0, nkind = 0;
            bool have = next_pass(p, s_tab, R, pi, item, kind);
            if (have) load_q(item, kind);
            while (have && !dead) {
                if (kind == 0) {
                    // the next statistics pass reads its tiles from HBM: ask for them now
                    ScoreItem nx;
                    if (item.r + 1 < R && score_item(p, s_tab, item.r + 1, nx)) {
                        for (int t = 0; t < nx.nt; ++t) tc::tma_prefetch_rows(&tm.a[nx.cache], nx.chunk * ST_CHUNK + t * 128, nx.lh);
                    }
                }
                for (int t = 0; t < item.nt; ++t, ++it) {
                    const int s = it % ST_STAGES;
                    // the stage is free once the MMAs of the tile that used it last are done: that is the
                    // same event that hands the accumulator tile to the consumers
                    if (it >= (uint32_t)ST_STAGES) {
                        const uint32_t j = it - ST_STAGES;
                        if (!tc::mbar_wait(&bar_t_full[j % ST_TBUF], (j / ST_TBUF) & 1u, wc, 64)) { dead = true; break; }
                    }
                    tc::mbar_expect_tx(&bar_full[s], ST_TILE_BYTES);
                    const uint32_t dst = tc::smem_u32(ring + s * ST_TILE_BYTES);
                    const int row0 = item.chunk * ST_CHUNK + t * 128;
                    tc::tma_load_rows(dst, &tm.a[item.cache], &bar_full[s], row0, item.lh);
                }
                if (dead) break;
                // Q of the next pass, while the tiles just asked for are worked on
                have = next_pass(p, s_tab, R, pi, nxt, nkind);
                if (have && !load_q(nxt, nkind)) dead = true;
                item = nxt;
                kind = nkind;
            }
            // nothing this thread started may still be in flight when the block exits
            for (uint32_t j = it > (uint32_t)ST_STAGES ? it - ST_STAGES : 0u; j < it; ++j)
                tc::mbar_wait(&bar_full[j % ST_STAGES], (j / ST_STAGES) & 1u, wc, 64);
            for (int b = 0; b < 2; ++b)
                if (nq[b] > 0) tc::mbar_wait(&bar_q_full[b], (nq[b] - 1) & 1u, wc, 64);
        }
    } else if (warp == 1 || warp == ST_THREADS / 32 - 1) {
        // ---------------- MMA issuers: two threads, alternate tiles ----------------
        // What an issuer does for a tile (two barrier tests, eight instructions that each hold the thread
        // for about 100 cycles, a commit) takes longer than the tensor cores need for the tile; two
        // issuers on separate warps overlap that.  Tiles are independent: different accumulators and ring
        // stages, and a commit only covers its own thread's instructions.
        if (lane == 0) {
            const uint32_t me = warp == 1 ? 0u : 1u;
            uint32_t it = 0, nq[2] = {0u, 0u};
            const uint32_t ring_addr = tc::smem_u32(ring);
            bool dead = false;
            PassIter pi;
            ScoreItem item;
            int kind = 0;
            while (!dead && next_pass(p, s_tab, R, pi, item, kind)) {
                if (!tc::mbar_wait(&bar_q_full[kind], nq[kind] & 1u, wc)) break;
                ++nq[kind];
                // operand descriptors: the k-step only moves the start address (in 16-byte units, low word)
                const uint64_t dq0 = tc::smem_desc_sw128(tc::smem_u32(q_s + kind * ST_TILE_BYTES), 16, 1024);
                // a pooling pass needs as many columns as the item has query rows, in pieces of 32
                const uint32_t idesc = tc::idesc_bf16(128, kind == 0 ? 128u : (uint32_t)(item.nq + 31) & ~31u, 0, 0);
                bool issued = false;
                for (int t = 0; t < item.nt; ++t) {
                    const uint32_t ti = it + t;
                    if ((ti & 1u) != me) continue;
                    // accumulator tile and ring stage share their index and the parity of their use
                    const uint32_t tb = ti % ST_TBUF, par = (ti / ST_TBUF) & 1u;
                    const bool e_ok = tc::mbar_test(&bar_t_empty[tb], par ^ 1u), f_ok = tc::mbar_test(&bar_full[tb], par);
                    if (!e_ok && !tc::mbar_wait(&bar_t_empty[tb], par ^ 1u, wc)) { dead = true; break; }
                    if (!f_ok && !tc::mbar_wait(&bar_full[tb], par, wc)) { dead = true; break; }
                    tc::tc_fence_after();
                    const uint64_t dk0 = tc::smem_desc_sw128(ring_addr + tb * ST_TILE_BYTES, 16, 1024);
                    const uint32_t acc = tmem + tb * 128u;
                    // pass A: queries on the lanes (S = Q K^T); pass B: keys on the lanes (S^T = K Q^T)
                    const uint64_t da0 = kind == 0 ? dq0 : dk0, db0 = kind == 0 ? dk0 : dq0;
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        // 16 channels per instruction: 32 bytes along the swizzled row, next column block after 4 steps
                        constexpr uint32_t HALF16 = ST_BOX_BYTES >> 4;
                        const uint64_t off16 = (uint64_t)((kk >> 2) * HALF16 + (kk & 3) * 2);
                        tc::umma_bf16(acc, da0 + off16, db0 + off16, idesc, kk > 0 ? 1u : 0u);
                    }
                    tc::umma_commit(&bar_t_full[tb]);
                    issued = true;
                }
                it += item.nt;
                // the Q buffer is free when both issuers' instructions of the pass are done
                if (!dead) {
                    if (issued) tc::umma_commit(&bar_q_free[kind]);
                    else tc::mbar_arrive(&bar_q_free[kind]);
                }
            }
        }
    } else if (warp < 2 + ST_CONSUMERS / 32) {
        // ---------------- consumers ----------------
        static_assert(ST_TBUF % ST_GROUPS == 0, "an accumulator tile must always belong to the same consumer group");
        const int q = warp & 3;                        // tensor-memory lane quarter this warp may touch
        const int grp = (warp - 2) >> 2;               // tiles with index == grp (mod ST_GROUPS) are this warp's
        const int row = q * 32 + lane;                 // lane of the accumulator tile: a query (pass A) or a key (pass B)
        const uint32_t tlane = tmem + ((uint32_t)(q * 32) << 16);
        const float sc = ST_LOG2E * rsqrtf((float)D);
        uint32_t it = 0, n_b[2] = {0u, 0u};

        // `pieces` 32-column pieces of an accumulator tile from piece `first` on, `work(half piece, registers)` on each 16
        // columns while the next 16 are on their way; the tile is handed back as soon as its last columns are in
        // registers.  An item with fewer than 128 query rows (the second one of a head with, say, 160) costs by what it
        // has: a warp whose lanes hold no query walks no piece of a statistics pass, and a pooling pass walks the columns
        // that hold queries.
        auto walk_tile = [&](uint32_t ti, int first, int pieces, auto &&work) {
            const uint32_t tb = ti % ST_TBUF;
            tc::mbar_wait(&bar_t_full[tb], (ti / ST_TBUF) & 1u, wc, 20);
            tc::tc_fence_after();
            const uint32_t ta = tlane + tb * 128u + 32u * first;
            uint32_t ra[16], rb[16];
            if (pieces > 0) tc::tmem_ld16(ta, ra);
#pragma unroll 1
            for (int pc = 0; pc < pieces; ++pc) {
                tc::tmem_ld_wait16(ra);
                tc::tmem_ld16(ta + 32u * pc + 16u, rb);
                work(2 * (first + pc), ra);
                tc::tmem_ld_wait16(rb);
                if (pc + 1 < pieces) {
                    tc::tmem_ld16(ta + 32u * pc + 32u, ra);
                } else {
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&bar_t_empty[tb]);
                }
                work(2 * (first + pc) + 1, rb);
            }
            if (pieces == 0) {
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&bar_t_empty[tb]);
            }
        };

        ScoreItem item, prev;
        bool have = false, have_prev = false;
        for (int i = 0; i < R + ST_LAG; ++i) {
            static_assert(ST_LAG == 1, "the item pooled is the one of the round before");
            prev = item;
            have_prev = have;
            // ======== pass A of round i: maximum and sum per query over the keys of this group's tiles ========
            have = i < R && score_item(p, s_tab, i, item);
            if (have) {
                const int T = s_tab[item.cache].T, buf = i & 1;
                // a chunk has at most as many tiles as there are groups: this group meets at most one of them
                static_assert(ST_GROUPS == ST_TILES, "one tile of a chunk per consumer group");
                const int my_t = (int)((uint32_t)(grp - (int)it) % ST_GROUPS);
                float m = -INFINITY, z = 0.f;
                if (my_t < item.nt) {
                    const int key0 = item.chunk * ST_CHUNK + my_t * 128;                  // key of column 0 of the tile
                    const int share = 4 / item.copies;           // pieces of 32 columns per copy
                    walk_tile(it + my_t, q / share * share, item.copies > 1 || 32 * q < item.nq ? share : 0, [&](int hp, uint32_t (&rr)[16]) {
                        // two copies of the update: the one that masks missing keys runs for a head's ragged last tile only
                        const int k0 = key0 + 16 * hp;
                        if (k0 + 16 > T) stats_update<true, FINE ? 1 : 64>(rr, T - k0, sc, m, z);
                        else stats_update<false, FINE ? 1 : 64>(rr, 16, sc, m, z);
                    });
                    // hand (m, z) of the tile to the messengers, filed under the tile's place in the chunk: they merge a
                    // chunk's tiles in that order whichever groups worked on them.  (The buffer is free: what the
                    // messengers made of its last contents has been waited for in the pooling pass since.)
                    s_m[(buf * ST_TILES + my_t) * 128 + row] = m;
                    s_z[(buf * ST_TILES + my_t) * 128 + row] = z;
                }
                it += item.nt;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&bar_st_ready[buf]);
            }
            // ======== pass B of the round before: pooled mass per key over all queries of the tile ========
            if (have_prev) {
                const CacheDev &c = p.c[prev.cache];
                const int T = s_tab[prev.cache].T, buf = (i - 1) & 1;
                tc::mbar_wait(&bar_mp_ready[buf], n_b[buf] & 1u, wc, 20);
                ++n_b[buf];
                const float *mp = s_mp + buf * 128, *rz = s_rz + buf * 128;
                const int my_t = (int)((uint32_t)(grp - (int)it) % ST_GROUPS);
                if (my_t < prev.nt) {
                    f32x2 a0 = 0ull, a1 = 0ull;
                    walk_tile(it + my_t, 0, (prev.nq + 31) >> 5, [&](int hp, uint32_t (&rr)[16]) { pool_piece<FINE>(rr, mp + 16 * hp, rz + 16 * hp, sc, a0, a1); });
                    const float a = sum2(add2(a0, a1));
                    const int j = prev.chunk * ST_CHUNK + my_t * 128 + row;
                    if (j < T) {
                        // with two query tiles per head the masses of both are added onto zeros: a sum of two terms, the
                        // same in either order
                        float *dst = p.scores + c.tok_off + (size_t)prev.lh * T;
                        if (!isfinite(a)) atomicOr(p.status, OBF_DEV_NONFINITE);
                        if (p.sc_qt == 1) {
                            dst[j] = a;
                            if (c.scores_out) c.scores_out[(size_t)prev.lh * T + j] = a;
                        } else {
                            atomicAdd(dst + j, a);
                        }
                    }
                }
                it += prev.nt;
            }
        }
    } else {
        // ---------------- messenger: the chunk's statistics out, the head's in, folded into M' ----------------
        // Per (head, chunk, query) one 64-bit word, (maximum, sum): zero (as cleared before the launch) until it is
        // published, never zero afterwards (the sum of a maximum's own exponential is one; a chunk without a finite logit
        // has the maximum -inf or a NaN).  A word vouches for itself, so nothing is counted and nothing fenced: every
        // block of a team polls the team's words and folds the head for itself, one trip through the L2 cache after the
        // last one is written.  (Counting the blocks in, folding in the last one and polling its result took 13000 cycles
        // a round, as long as the round's arithmetic.)
        uint32_t n_a[2] = {0u, 0u};
        const int t = (warp - 2 - ST_CONSUMERS / 32) * 32 + lane;                  // this lane's query
        for (int i = 0; i < R; ++i) {
            ScoreItem item;
            if (!score_item(p, s_tab, i, item)) continue;
            const CacheDev &c = p.c[item.cache];
            const int buf = i & 1, team = c.sc_team;
            const bool mine = t < item.nq;
            unsigned long long *words = reinterpret_cast<unsigned long long *>(p.sc_part) + (c.sc_part_off + (size_t)item.lv * team * 128) + t;
            const float extra = (c.lse_extra && mine) ? c.lse_extra[(size_t)item.lh * p.n_q + 128 * item.qt + t] : -INFINITY;
            tc::mbar_wait(&bar_st_ready[buf], n_a[buf] & 1u, wc, 20);
            float M = -INFINITY, Z = 0.f;
            {
                // tile by tile, and copy by copy of the queries in a tile
                const int rows = 128 / item.copies;
#pragma unroll 1
                for (int r = t; r < 128 && mine; r += rows) {
                    float m[ST_TILES], z[ST_TILES], Mn = M;
#pragma unroll
                    for (int e = 0; e < ST_TILES; ++e) {
                        const int at = (buf * ST_TILES + e) * 128 + r;
                        m[e] = e < item.nt ? s_m[at] : -INFINITY;
                        z[e] = e < item.nt ? s_z[at] : 0.f;
                        Mn = fmaxf(Mn, m[e]);
                    }
                    const float Mf = fmaxf(Mn, -3e38f);                        // (-inf - -inf would be a NaN)
                    Z *= ex2_approx(M - Mf);
#pragma unroll
                    for (int e = 0; e < ST_TILES; ++e) Z += z[e] * ex2_approx(m[e] - Mf);
                    M = Mn;
                }
                ++n_a[buf];
                if (mine && !p.debug_drop_publish)
                    st_relaxed_gpu_u64(words + (size_t)item.chunk * 128, ((unsigned long long)__float_as_uint(Z) << 32) | __float_as_uint(M));
            }
            M = -INFINITY;
            Z = 0.f;
            bool gave_up = false;
            // sixteen chunks in flight per sweep
#pragma unroll 1
            for (int c0 = 0; c0 < team && !gave_up; c0 += 16) {
                unsigned long long w[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) w[e] = (c0 + e < team && mine) ? 0ull : 0xff800000ull;   // (-inf, 0)
                uint64_t t0 = 0ull;
                for (;;) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (w[e] == 0ull) w[e] = ld_relaxed_gpu_u64(words + (size_t)(c0 + e) * 128);
                    bool all = true;
#pragma unroll
                    for (int e = 0; e < 16; ++e) all = all && w[e] != 0ull;
                    // the warp leaves the loop as one: votes, not per-lane exits
                    if (__all_sync(0xffffffffu, all)) break;
                    const uint64_t now = tc::global_ns();
                    if (t0 == 0ull) t0 = now;
                    if (__any_sync(0xffffffffu, *(volatile uint32_t *)&s_abort != 0u || now - t0 > p.wait_limit_ns)) {
                        if (lane == 0) {
                            s_abort = 1u;
                            atomicOr(p.status, OBF_DEV_TIMEOUT);
                        }
                        gave_up = true;
                        break;
                    }
                    __nanosleep(32);
                }
                float Mn = M;
#pragma unroll
                for (int e = 0; e < 16; ++e) Mn = fmaxf(Mn, __uint_as_float((uint32_t)w[e]));
                const float Mf = fmaxf(Mn, -3e38f);
                Z *= ex2_approx(M - Mf);
#pragma unroll
                for (int e = 0; e < 16; ++e) Z += __uint_as_float((uint32_t)(w[e] >> 32)) * ex2_approx(__uint_as_float((uint32_t)w[e]) - Mf);
                M = Mn;
            }
            // (the buffer is free: every consumer has pooled with its last contents before it handed in this round's statistics)
            float mp = INFINITY, rz = 0.f;                                     // exp2(-inf) = 0 for padding columns
            if (mine) {
                // the keys outside the prompt take their share of the normaliser
                fold_lse_extra(extra, M, Z);
                mp = FINE ? M : M + lg2_approx(Z);
                rz = FINE ? 1.f / Z : 1.f;
                if (gave_up) { mp = 0.f; rz = 1.f; }
                else if (!(Z > 0.f) || !isfinite(mp) || !isfinite(rz)) {
                    if (item.chunk == 0) atomicOr(p.status, OBF_DEV_NONFINITE);
                    mp = __int_as_float(0x7fc00000);
                }
            }
            s_mp[buf * 128 + t] = -mp;
            if (FINE) s_rz[buf * 128 + t] = rz;
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_mp_ready[buf]);
        }
    }

    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

// Heads with two query tiles (their masses are joined in the workspace) whose masses the caller wants: a copy.
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
