// ec_attend, skip step with FEW query rows (bf16, head_dim 128, at most 96 packed query rows per CTA column):
// ONE launch that refreshes the active rows' K/V in the cache, attends from the active rows over the whole
// cache and merges the key-range partials.  (Section 4.2 and Appendix A of the paper, partial branch:
// TransformerBlock(Q[M u R], K[I], V[I]) after the rows M u R got fresh K, V.)
//
// With 34 query rows a 128-row M tile would be three quarters padding, and a thread per query row would
// leave most softmax lanes idle.  Here the KEYS take the M axis of the tensor core and the query rows the N
// axis (N = 48, 64 or 96 slots):
//     S^T[128 keys x N]  = K_tile[128 keys x 128] . Q[N x 128]^T          (A = K tile, B = Q, both K-major)
//     O^T[128 d    x N] += V_tile^T[128 d x 128 keys] . P^T[128 keys x N]  (A = V tile MN-major, B = P^T MN-major)
// so a softmax thread owns one KEY (TMEM lane) and its scores against the query slots: all 128 lanes work, one
// exponential per (key, query), no padding rows, a pipeline step covers 128 keys.  A thread keeps its key lane's share of
// every row sum in registers; they are added up over the lanes once, at the end.  (Two auxiliary warps that read P^T back
// from shared memory took 1.2 us a tile and set the pace: 15.9 us a launch at L = 1983 with 96 rows, then 13.7.)  Two
// to four softmax warpgroups share the columns of a key, which shortens a thread's serial path (see soft_groups).
//   softmax  the references m[q] (log2 units) are shared by all keys of the CTA and live in shared memory.  The first
//            is the score of one valid key; p = 2^(s*scale*log2e - m[q]) needs no reduction as long as no score exceeds
//            its reference by more than 2^60 (bf16 and fp32 have room for that, and a reference is never above the true
//            maximum).  A barrier-wide OR tells: only then the column maxima are reduced, m is raised, and O^T and the
//            row sums are rescaled;
//   grid     (C, B*H_kv*n_sub) as clusters of C <= 8 CTAs (any count, not only powers of two) that split one
//            head's 128-key tiles, chosen so that the most-loaded SM streams the fewest tiles.  With grouped-query
//            attention the query heads of a kv head are packed into the N axis; when they exceed the slots the heads
//            (and, beyond 96 active rows, the rows) are spread over n_sub CTA columns that stream the same K/V (L2
//            serves the repeats);
//   K/V      the producer warp issues its TMA loads in key order through a ring of NS slots of 32 KB (K_0 V_0 K_1 V_1
//            ...: a K slot is free again as soon as the scores of its tile are computed, a V slot after the second
//            product, and an odd slot count is possible, which is what lets the 96-slot instantiation keep two and
//            a half tiles in flight); the loads depend on nothing, and the first fill of the ring is spaced in time
//            (one tile of every CTA per interval) so that the memory system always has requests queued while the
//            first tiles are consumed;
//   refresh  the active rows' fresh K/V reach the attention straight from k_new / v_new, not through the cache: one
//            CTA of every cluster (the last) attends to them as one or two EXTRA key tiles, fetched by TMA from the
//            fresh tensors (a [128 rows x 128] box of k_new is laid out exactly like a cache tile) after its cache
//            tiles (visited first they held a ring stage through the start of the stream and set that CTA two tile
//            times behind its peers), while every CTA masks the stale cached keys of the refreshed positions (a bit per key, built from
//            the index list).  The attention therefore never waits for the cache update: the auxiliary warps copy the
//            fresh rows to the cache in global memory, for later steps, ordered against nothing.  (Keys in a different
//            order, the same sum.)  When a CTA holds a single cache tile the extra tiles get a CTA of their own;
//   merge    CTA c of the cluster owns the output columns d in [c*DL, (c+1)*DL).  Every CTA leaves its O (un-normalised),
//            m and l in its own shared memory; after a cluster barrier the owners read their columns of all C partials out
//            of the peers (128-byte pieces: a warp whose lanes read different rows takes 2.1 us for what this does in 0.6),
//            combine, normalise and store; a second cluster barrier keeps every CTA's shared memory alive until its
//            peers have read it.
// What bounds it: HBM at long contexts (L = 4096, one sequence, 34 rows: 68.8 MB in 15.6 us), the serial path below that.
// Code that runs once is fetched about as slowly as it runs, so this path is kept short: index arithmetic before the
// wait, rolled loops in the merge.  (Q by TMA queues behind the K/V tiles of the first fill in the TMA unit: 0.6 us more at
// L = 768, 1.6 at 4096.  Parts sent to the owners instead of read by them, one cluster barrier less: 0.7 us more.)
// warp 0: TMA producer; warp 1: tcgen05.mma issue; the softmax warps: Q, softmax; two auxiliary warps: stale-key bits,
// cache update.  Launched with programmatic stream serialisation; what the previous kernel wrote is read only
// after griddepcontrol.wait.  Every mbarrier wait is bounded (EC_ERR_TIMEOUT in dev_status, CTA-wide abort flag: an
// aborted CTA stores no output); the CTA always frees its TMEM and exits.
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

#include <cstdio>
#include <mutex>
#include <type_traits>
#include <vector>

namespace ec {
namespace {

using namespace tc;

constexpr int BK = 128, HD = 128;
constexpr int kAuxThreads = 64;            // auxiliary warps: stale-key bits and cache update
// Softmax warpgroups: each takes an equal share of the query slots of every key, a multiple of 8.  us a pass by their number:
// 48 slots, 32 layers of 768 1: 273.8, 2: 247.2, 3: 249.7; 64 slots, 16 layers of 512 with k = 32 2: 153.5, 4: 149.9; 96
// slots, 32 layers of 1983 2: 453.2, 3: 448.2, 4: 460.1.
__host__ __device__ constexpr int soft_groups(int n) { return n == 48 ? 2 : n == 64 ? 4 : 3; }
__host__ __device__ constexpr int block_threads(int n) { return 64 + 128 * soft_groups(n) + kAuxThreads; }
constexpr uint32_t SUB = 128 * 128;        // [128 rows x 64 bf16], 128-byte swizzle: 16 KB
constexpr uint32_t TILE = 2 * SUB;         // [128 x 128] bf16
constexpr uint32_t STAGE = 2 * TILE;       // K tile + V tile: 64 KB
constexpr int kMaxStages = 6;              // ring slots of one tile (32 KB) each
constexpr int kMaxSlots = 96;              // query slots (packed rows) of one CTA column
constexpr int kMaxActive = 256;            // active rows of a sequence (refresh list, row chunks)
constexpr int kMaxTiles = 1024;            // key tiles of one CTA

enum { B_FULL = 0, B_EMPTY = kMaxStages, B_SFULL = 2 * kMaxStages, B_PFULL = B_SFULL + 2, B_PVDONE = B_PFULL + 1,
       B_QFULL = B_PVDONE + 1, B_LIST = B_QFULL + 1, B_DRY = B_LIST + 1, B_COUNT = B_DRY + 1 };

constexpr uint32_t kBarBytes = (B_COUNT * 8u + 15u) & ~15u;   // the barrier block, padded so that what follows is 16-byte aligned

// A probability may exceed its reference by this power of two before the references are raised: sums and products stay
// far from the fp32 range, and bf16 carries fp32's exponents, so nothing is lost.
constexpr float kRaise = 60.f;

// a CTA's partial for the merge: O, m and l
__host__ __device__ constexpr uint32_t partial_bytes(int n) { return (uint32_t)n * (HD * 4u + 8u); }

// the value is needed here: the compiler reads it now
template <typename V>
__device__ __forceinline__ void touch(V v) {
    if constexpr (sizeof(V) == 8) asm volatile("" ::"l"((unsigned long long)v) : "memory");
    else if constexpr (std::is_same_v<V, float>) asm volatile("" ::"f"(v) : "memory");
    else asm volatile("" ::"r"((uint32_t)v) : "memory");
}

// COLS consecutive 32-bit columns of this thread's TMEM lane -> registers
template <int COLS>
__device__ __forceinline__ void ld_row_part(uint32_t taddr, uint32_t* r) {
    static_assert(COLS % 8 == 0, "columns per thread");
#pragma unroll
    for (int c = 0; c < COLS; c += COLS % 16 ? 8 : 16)   // (accesses start at multiples of their width)
        if constexpr (COLS % 16) ld8(taddr + c, r + c);
        else ld16(taddr + c, r + c);
}
template <int COLS>
__device__ __forceinline__ void ld_row(uint32_t taddr, uint32_t* r) {
    ld_row_part<COLS>(taddr, r);
    wait_ld<COLS>(r);
}
struct KeysParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_new;   // nullptr: attend without refreshing
    const __nv_bfloat16* v_new;
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* active_idx;    // nullptr: identity
    __nv_bfloat16* out;
    int32_t* dev_status;
    int n_active, ctx_len, n_q_heads, n_kv_heads;
    int q_per_kv;     // H_q / H_kv
    int group;        // query heads of one kv head handled by one CTA column (the last one may have fewer: its packed
                      // rows keep the stride, the rows of the heads it lacks are empty)
    int group_inv;    // ceil(2^16 / group): r / group = (r * group_inv) >> 16 for packed rows r < 256
    int quads_inv;    // ceil(2^16 / (dl / 4)), for the items of the merge
    int rows_chunk;   // active rows handled by one CTA column (the last chunk may hold fewer)
    int n_sub_r;      // row chunks = ceil(n_active / rows_chunk)
    int n_sub;        // CTA columns per kv head = ceil(q_per_kv / group) * n_sub_r
    int n_splits, tiles_per_split, n_stages;
    int shift;        // 1: the first CTA of the cluster takes one cache tile more and the last, which also visits the
                      // fresh tiles, one less (ranges of the CTAs in between move up by one tile)
    int n_extra;      // key tiles of fresh rows attended by the last CTA of every cluster (0: nothing to refresh)
    int dl;           // output columns merged by one CTA of the cluster (a multiple of 8; the last CTAs may own fewer)
    uint32_t off_p, off_stage, off_list, off_bar;   // shared-memory carve (bytes from the 1024-aligned base); Q is at 0;
                                                    // off_list: the stale-key bits, 16 bytes per cache tile
    float scale_log2;
    // Nanoseconds the memory system needs for one stage of every CTA that streams its own K/V: the producer spaces
    // the first fill of its ring by this much per stage, so that the stages of the launch arrive one wave after the
    // other instead of all together (0: no spacing).
    uint32_t stagger_ns;
    // 1: the caller stated (EC_ATTN_CACHE_SETTLED) that nothing still running on the stream writes the caches, so the
    // first cache tile is asked for before the dependency wait
    int early_cache;
};

// words after the barrier block
struct alignas(16) KeysShared {
    uint32_t tmem;
    int abort_flag;
    int pad[2];
    alignas(16) float m[kMaxSlots];            // reference maxima of the query rows, log2 units (read as float2)
    alignas(16) float factor[2][kMaxSlots];    // [tile parity]: rescale factors of that tile's slow path
    float col[4][kMaxSlots];                   // per warp and column: maxima of the current slow path, at the end row sums
};

template <int N>
__global__ void __launch_bounds__(block_threads(N), 1)
attend_skip_keys_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                        const __grid_constant__ CUtensorMap map_kn, const __grid_constant__ CUtensorMap map_vn,
                        const KeysParams params) {
    static_assert(N == 48 || N == 64 || N == 96, "query-row slots per CTA");
    constexpr int NH = N / soft_groups(N);      // query slots of a softmax thread
    constexpr int kSoft = 128 * soft_groups(N), kThreads = block_threads(N);
    // tensor-memory columns: S^T x 2 and O^T at multiples of NP (the slots rounded up to 64 or 128)
    constexpr uint32_t NP = N <= 64 ? 64 : 128;
    constexpr uint32_t TM_S = 0, TM_O = 2 * NP;
    constexpr uint32_t TM_COLS = (3 * NP <= 256) ? 256 : 512;
    KeysParams p = params;
    keep_in_registers(p.k_new, p.active_idx, p.out, p.dev_status, p.scale_log2, p.n_active, p.ctx_len, p.n_q_heads, p.n_kv_heads,
                      p.group, p.group_inv, p.quads_inv, p.n_splits, p.tiles_per_split, p.n_stages, p.shift, p.n_extra, p.dl,
                      p.off_p, p.off_stage, p.off_list, p.off_bar);
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = (s2u(smem_raw) + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - s2u(smem_raw));
    const uint32_t bars = base + p.off_bar;
    KeysShared* sh = reinterpret_cast<KeysShared*>(gbase + p.off_bar + kBarBytes);
    volatile int* abort_flag = &sh->abort_flag;
    uint32_t* stale = reinterpret_cast<uint32_t*>(gbase + p.off_list);   // [cache tile][4]: a bit per stale key
    auto bar = [&](int idx) { return bars + idx * 8; };

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int split = blockIdx.x, bh = blockIdx.y / p.n_sub, sub = blockIdx.y % p.n_sub;
    const int b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads;
    const int hg = sub / p.n_sub_r * p.group;                                  // first query head of this CTA in its kv head
    const int hq0 = hk * p.q_per_kv + hg;                                      // ... and of all
    const int heads = min(p.group, p.q_per_kv - hg);                           // (the last column may have fewer)
    const int i0 = (sub % p.n_sub_r) * p.rows_chunk;                           // first active row of this CTA
    const int rows_total = min(p.rows_chunk, p.n_active - i0) * p.group;       // packed query rows of this CTA
    const int C = p.n_splits;
    const int DL = p.dl;
    const int n_tiles_total = (p.ctx_len + BK - 1) / BK;
    const int t_begin = split * p.tiles_per_split + (split > 0 ? p.shift : 0);
    const int t_end = min(n_tiles_total, (split + 1) * p.tiles_per_split + p.shift);
    const int TC = max(0, t_end - t_begin);                  // cache tiles of this CTA
    const int NS = p.n_stages;       // ring slots: tile j has K in slot 2j mod NS and V in slot (2j + 1) mod NS
    const bool refresh = p.k_new != nullptr;
    // the last CTA of the cluster attends to the fresh rows too, after its cache tiles, as XT extra key tiles read from
    // k_new / v_new: visits [0, TC) are cache tiles, visits [TC, T) fresh tiles
    const int XT = (refresh && split == p.n_splits - 1) ? p.n_extra : 0;
    const int T = XT + TC;           // tiles this CTA visits: >= 1 by construction of the plan
    const int key_lo = t_begin * BK, key_hi = min(p.ctx_len, t_end * BK);
    // partial of this CTA for the merge, over the (then dead) Q / P^T / stage memory: [query][PITCH] floats of O, then
    // (m, l)[N]; the peers read it from here
    constexpr uint32_t PITCH = HD;
    constexpr uint32_t ML_OFF = N * PITCH * 4;
    const int own_dl = max(0, min(DL, HD - split * DL));   // output columns this CTA owns (a multiple of 8)

    // ---- set-up ------------------------------------------------------------------------------
    // Under programmatic dependent launch this CTA starts while the tail of the previous kernel still runs.  Whatever
    // that kernel produces (q, k_new, v_new, the index list) is read after the dependency wait below.  The caches are
    // read before it only when the caller has stated that nothing in flight writes them: the producer thread then asks
    // for its first cache tile as soon as the barriers exist, and the memory system works through the rest of the
    // set-up, the previous kernel's tail and the wait.
    unsigned long long t_fill = 0;
    if (tid == 0) {
        for (int i = 0; i < B_COUNT; ++i) {
            uint32_t count = 1;
            if (i == B_PFULL || i == B_QFULL) count = kSoft / 32;
            if (i == B_LIST) count = kAuxThreads;
            mbar_init(bar(i), count);
        }
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (p.early_cache && TC > 0) {   // ring entry 0: the first cache tile
            t_fill = global_timer_ns();
            const uint32_t dst = base + p.off_stage;
            mbar_expect_tx(bar(B_FULL + 0), TILE);
            tma_load_4d(dst, &map_k, 0, t_begin * BK, 0, bh, bar(B_FULL + 0));
            mbar_expect_tx(bar(B_FULL + 1), TILE);
            tma_load_4d(dst + TILE, &map_v, 0, t_begin * BK, 0, bh, bar(B_FULL + 1));
        } else {
            prefetch_map(&map_k);
            prefetch_map(&map_v);
        }
        if (p.k_new) {
            prefetch_map(&map_kn);
            prefetch_map(&map_vn);
        }
    }
    if (refresh)
        for (int w = tid; w < TC * 4; w += kThreads) stale[w] = 0u;
    if (tid < N) sh->m[tid] = -INFINITY;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s2u(&sh->tmem)), "r"(TM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        fence_before();
    }
    __syncthreads();
    fence_after();
    const uint32_t tmem = sh->tmem;
    // Q: where this thread's 16-byte pieces of the packed rows come from (element offsets; -1: no such row).  Worked out
    // here, before the wait below, because what follows it is the serial path of a short launch.
    constexpr int kPieces = N * (HD / 8) / kSoft;
    int q_off[kPieces];
    if (warp >= 2 && warp < 2 + kSoft / 32) {
        const int stid = tid - 64;
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
            const int row = (stid >> 4) + u * (kSoft / 16);
            const int i = (row * p.group_inv) >> 16, jh = row - i * p.group;
            q_off[u] = (row < rows_total && jh < heads) ? ((i0 + i) * p.n_q_heads + hq0 + jh) * HD + (stid & 15) * 8 : -1;
            touch(q_off[u]);
        }
    }
    const __nv_bfloat16* q_seq = p.q + (long long)b * p.n_active * p.n_q_heads * HD;
    touch(q_seq);
    if (warp != 0) pdl_wait();     // the previous kernel of the stream has completed; its results may be read
    if (tid == 32) pdl_launch_dependents();
    __syncwarp();

    // First fill of the ring: cache tile j of every CTA is asked for j * stagger_ns after the first, so the first tiles of
    // all CTAs land before anybody's second, and requests stay queued while they are consumed.  (Asked for all at once,
    // the tiles of the whole launch arrive together after the time of all of them, and the memory system then idles
    // until the first slot is free again.)
    auto pace = [&](int j) {
        if (j == 0 || j >= TC || !p.stagger_ns) return;
        const unsigned long long due = t_fill + (unsigned long long)j * p.stagger_ns;
        while (global_timer_ns() < due) __nanosleep(64);
    };

    if (warp == 0) {
        // ================================ TMA producer ======================================
        if (lane == 0) {
            auto load = [&](int n) {   // ring entry n: K of tile n / 2 (even n) or its V (odd n)
                const int j = n >> 1, s = n % NS;
                const uint32_t dst = base + p.off_stage + s * TILE;
                mbar_expect_tx(bar(B_FULL + s), TILE);
                if (j >= TC) {   // active rows [128 x, 128 x + 128) of this kv head, fresh; rows past n_active read as zero
                    tma_load_5d(dst, (n & 1) ? &map_vn : &map_kn, 0, (j - TC) * BK, 0, hk, b, bar(B_FULL + s));
                } else {
                    tma_load_4d(dst, (n & 1) ? &map_v : &map_k, 0, (t_begin + j) * BK, 0, bh, bar(B_FULL + s));
                }
            };
            int n = 0;
            if (p.early_cache) {
                const int fill = min(NS, 2 * TC);
                for (n = TC > 0 ? 2 : 0; n < fill; ++n) {   // entries 0 and 1 are already on their way
                    if (!(n & 1)) pace(n >> 1);
                    load(n);
                }
                n = fill;
            }
            pdl_wait();
            if (n == 0) t_fill = global_timer_ns();
            for (; n < 2 * T; ++n) {
                if (n < NS) { if (!(n & 1)) pace(n >> 1); }
                else mbar_wait(bar(B_EMPTY + n % NS), (n / NS - 1) & 1, abort_flag, p.dev_status);
                load(n);
            }
        } else {
            pdl_wait();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================================ MMA issue (the whole warp, see elect_one) ==================
        const bool elected = elect_one();
        constexpr uint32_t IDESC_S = instr_desc2(N, 0, 0);    // A = K tile (K-major), B = Q (K-major)
        constexpr uint32_t IDESC_PV = instr_desc2(N, 1, 1);   // A = V tile (MN-major: d contiguous), B = P^T (MN-major)
        constexpr uint32_t QHALF = N * 128;                   // bytes of one 64-column half of the Q tile
        const uint64_t desc_q = smem_desc(base, 16, 1024), desc_p = smem_desc(base + p.off_p, SUB, 1024);
        auto products_s = [&](int slot, int buf) {
            const uint64_t desc_k = smem_desc(base + p.off_stage + slot * TILE, 16, 1024);
            fence_after();
            if (elected) {
#pragma unroll
                for (int k = 0; k < HD / 16; ++k)
                    mma_ss(tmem + TM_S + buf * NP, desc_k + ((k >> 2) * SUB + (k & 3) * 32) / 16,
                           desc_q + ((k >> 2) * QHALF + (k & 3) * 32) / 16, IDESC_S, k > 0);
            }
        };
        auto products_pv = [&](int slot, bool accumulate) {
            const uint64_t desc_v = smem_desc(base + p.off_stage + slot * TILE, SUB, 1024);
            fence_after();
            if (elected) {
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    mma_ss(tmem + TM_O, desc_v + k * 128, desc_p + k * 128, IDESC_PV, (accumulate || k > 0));
            }
        };
        // S of tile j needs the tile; P V of tile j needs P^T from the softmax.  Whichever is ready
        // is issued: P V of a tile does not wait for the next tile to land (its commit frees the stage for the
        // producer), S may run one tile ahead of P V (two S^T buffers).
        int next_s = 0, next_pv = 0;
        int ks = 0, vs = 1;               // ring slots of K of tile next_s and V of tile next_pv, and how often they were filled
        uint32_t k_turn = 0, v_turn = 0;
        auto step = [&](int& slot, uint32_t& turn) {
            slot += 2;
            if (slot >= NS) slot -= NS, turn ^= 1;
        };
        SpinGuard guard;
        // The first round is a dry one: both products on whatever shared memory holds (their results are overwritten: S of
        // tile 1, the first P V), so that the code of the loop has been fetched when the first tile needs it.
        bool dry = true;
        while (next_pv < T) {
            bool progressed = false;
            const bool s_ready = next_s < T && next_s <= next_pv + 1 && mbar_test_warp(bar(B_FULL + ks), k_turn);   // the tile has landed
            if (s_ready || dry) {
                products_s(ks, dry ? 1 : next_s & 1);
                if (elected) {
                    commit(bar(dry ? B_DRY : B_SFULL + (next_s & 1)));
                    commit(bar(dry ? B_DRY : B_EMPTY + ks));    // the K slot is free once these products have run
                }
                if (!dry) {
                    step(ks, k_turn);
                    ++next_s;
                    progressed = true;
                }
            }
            const bool p_ready = mbar_test_warp(bar(B_PFULL), next_pv & 1) && mbar_test_warp(bar(B_FULL + vs), v_turn);   // P^T is there, V has landed
            if (p_ready || dry) {
                products_pv(vs, next_pv > 0);
                if (elected) {
                    commit(bar(dry ? B_DRY : B_PVDONE));
                    commit(bar(dry ? B_DRY : B_EMPTY + vs));
                }
                if (!dry) {
                    step(vs, v_turn);
                    ++next_pv;
                    progressed = true;
                }
            }
            if (dry) {
                mbar_wait(bar(B_QFULL), 0, abort_flag, p.dev_status);
                dry = false;
                progressed = true;
            }
            if (progressed) guard.progress();
            else if (__any_sync(0xffffffffu, !guard.tick(abort_flag, p.dev_status))) break;
        }
    } else if (warp >= 2 + kSoft / 32) {
        // ===== auxiliary warps: stale-key bits; the fresh rows into the cache (for later steps) =====
        const int atid = tid - (64 + kSoft);
        if (refresh) {
            // which cached keys of this CTA's range are about to be refreshed: they are attended from k_new / v_new (as
            // extra tiles, by the last CTA of the cluster), so their cached copies must not count
            for (int i = atid; i < p.n_active; i += kAuxThreads) {
                const int r = (p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i) - key_lo;
                if (r >= 0 && r < key_hi - key_lo) atomicOr(&stale[r >> 5], 1u << (r & 31));
            }
            mbar_arrive(bar(B_LIST));   // release: the bits above are visible to whoever waits
        }
        if (refresh && sub == 0) {
            // The CTAs of one column also put the active rows' K/V into the cache, for later steps, each a share of the
            // rows: straight from the fresh tensors, eight 16-byte pieces in flight per thread.  Nothing in this launch
            // depends on these stores.
            const int pieces = p.n_active * 32;   // [row][K, V][16 pieces]
            for (int c0 = split * kAuxThreads + atid; c0 < pieces; c0 += 8 * C * kAuxThreads) {
                uint4 v[8];
                int pos[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int c = c0 + u * C * kAuxThreads, i = c >> 5;
                    pos[u] = -1;
                    if (c < pieces) {
                        pos[u] = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i;
                        const __nv_bfloat16* src = (c & 16) ? p.v_new : p.k_new;
                        v[u] = __ldg(reinterpret_cast<const uint4*>(
                            src + (((long long)b * p.n_active + i) * p.n_kv_heads + hk) * HD + (c & 15) * 8));
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int c = c0 + u * C * kAuxThreads;
                    if (pos[u] < 0 || pos[u] >= p.ctx_len) continue;
                    __nv_bfloat16* dst = (c & 16) ? p.v_cache : p.k_cache;
                    *reinterpret_cast<uint4*>(dst + ((long long)bh * p.ctx_len + pos[u]) * HD + (c & 15) * 8) = v[u];
                }
            }
        }
    } else {
        // ================================ Q, softmax (warps 2 ..) ===================================
        const int stid = tid - 64;
        const int wg = stid >> 7;                    // warpgroup: columns [wg * NH, (wg + 1) * NH) of every key
        const int c0 = wg * NH;
        const int st_w = stid & 127;
        constexpr uint32_t QHALF = N * 128;
        constexpr int W = NH % 16 ? 8 : 16;          // columns that are loaded together
        // Q rows of this kv head -> swizzled K-major tile of N rows (rows past rows_total are zero): all of a thread's
        // loads are issued before the first is stored
        {
            const int ch = stid & 15;
            uint4 v[kPieces];
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                ldg_nc_v4_pred(v[u], q_seq + q_off[u], q_off[u] >= 0);
            }
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                const int row = (stid >> 4) + u * (kSoft / 16);
                const uint32_t off = (ch >> 3) * QHALF + (row >> 3) * 1024 + (row & 7) * 128 + (((ch & 7) ^ (row & 7)) << 4);
                *reinterpret_cast<uint4*>(gbase + off) = v[u];
            }
            fence_async_smem();     // Q (generic proxy) -> visible to the tensor core (async proxy)
            mbar_arrive_warp(bar(B_QFULL));
        }

        const int quarter = warp & 3;
        const int kk = quarter * 32 + lane;          // key of the tile == TMEM lane == output column d later on
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const float sl2 = p.scale_log2;
        const f32x2 sl2_2 = pk(sl2, sl2);
        // P^T row of this key: [64-slot half][key][64 slots], 128-byte swizzle
        unsigned char* prow = gbase + p.off_p + (kk >> 3) * 1024 + (kk & 7) * 128;
        const int bar_or = 2 + 2 * wg, bar_sync = 3 + 2 * wg;   // named barriers of this warpgroup
        // which keys of the fresh tiles exist: active rows with a position inside the context (bit x: row 128 x + kk)
        uint32_t fresh_ok = 0;
        for (int x = 0; x < XT; ++x) {
            const int i = x * BK + kk;
            if (i < p.n_active) {
                const int pos = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i;
                if (pos >= 0 && pos < p.ctx_len) fresh_ok |= 1u << x;
            }
        }
        f32x2 lsum[NH / 2];   // this key lane's share of the row sums: probabilities as rounded for the second product
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) lsum[i] = pk(0.f, 0.f);
        bool masks_ready = !refresh;   // the stale-key bits are awaited once, before the first cache tile

        for (int j = 0; j < T; ++j) {
            mbar_wait(bar(B_SFULL + (j & 1)), (j >> 1) & 1, abort_flag, p.dev_status);
            fence_after();
            const uint32_t s_addr = tmem + lane_addr + TM_S + (j & 1) * NP + c0;
            // this thread's key does not count: a missing row of a fresh tile, a key past the end of the context (ragged
            // last tile), a cached key whose position is being refreshed (it is attended from the fresh tile instead)
            bool past_end;
            if (j >= TC) {
                past_end = !((fresh_ok >> (j - TC)) & 1u);
            } else {
                past_end = (t_begin + j) * BK + kk >= p.ctx_len;
                if (!masks_ready) {
                    mbar_wait(bar(B_LIST), 0, abort_flag, p.dev_status);
                    masks_ready = true;
                }
                if (refresh) past_end = past_end || ((stale[j * 4 + (kk >> 5)] >> (kk & 31)) & 1u);
            }
            if (j == 0) {
                // First reference: the scores of the first valid key among the first warp's 32 (any key that counts
                // will do: a reference is never above the true maximum, and probabilities may exceed it by 2^kRaise).
                if (quarter == 0) {
                    uint32_t sr[NH];
                    ld_row<NH>(s_addr, sr);
                    const uint32_t valid = __ballot_sync(0xffffffffu, !past_end);
                    if (lane == __ffs(valid) - 1) {
#pragma unroll
                        for (int c = 0; c < NH; c += 4)
                            *reinterpret_cast<float4*>(&sh->m[c0 + c]) =
                                make_float4(__uint_as_float(sr[c]) * sl2, __uint_as_float(sr[c + 1]) * sl2,
                                            __uint_as_float(sr[c + 2]) * sl2, __uint_as_float(sr[c + 3]) * sl2);
                    }
                }
                named_barrier(bar_sync, 128);
            }
            // d = s * scale * log2(e) - m[q], p = 2^d; does any score exceed its reference by more than 2^kRaise?
            uint32_t pw[NH / 2];
            while (true) {
                float dmx0 = -INFINITY, dmx1 = -INFINITY;
                uint32_t sr[2][W];
                ld_row_part<W>(s_addr, sr[0]);
#pragma unroll
                for (int q = 0; q < NH / W; ++q) {   // W columns at a time, the next ones on their way
                    wait_ld<W>(sr[q & 1]);
                    if (q + 1 < NH / W) ld_row_part<W>(s_addr + W * (q + 1), sr[(q + 1) & 1]);
#pragma unroll
                    for (int i = 0; i < W / 2; ++i) {
                        const float2 mm = *reinterpret_cast<const float2*>(&sh->m[c0 + W * q + 2 * i]);
                        f32x2 d2 = fma2(pk(__uint_as_float(sr[q & 1][2 * i]), __uint_as_float(sr[q & 1][2 * i + 1])), sl2_2,
                                        pk(-mm.x, -mm.y));
                        if (past_end) d2 = pk(-INFINITY, -INFINITY);   // probability 0 for every query
                        float d0, d1;
                        upk(d2, d0, d1);
                        if (i & 1) dmx1 = max3(dmx1, d0, d1); else dmx0 = max3(dmx0, d0, d1);
                        pw[W / 2 * q + i] = pack_bf16x2(fast_exp2(d0), fast_exp2(d1));
                    }
                }
                if (!named_barrier_or(bar_or, 128, fmaxf(dmx0, dmx1) > kRaise)) break;
                // ---- rare path: raise the references to the column maxima of this tile, rescale O^T and the row sums by
                //      the same factors, and once more ----
#pragma unroll
                for (int q = 0; q < NH / W; ++q) {
                    ld_row<W>(s_addr + W * q, sr[0]);
#pragma unroll
                    for (int c = 0; c < W; ++c) {
                        const float o = redux_max(past_end ? -INFINITY : __uint_as_float(sr[0][c]));
                        if (lane == (W * q + c) % 32) sh->col[quarter][c0 + W * q + c] = o;
                    }
                }
                named_barrier(bar_sync, 128);
                if (st_w < NH) {
                    const int c = c0 + st_w;
                    const float o = fmaxf(fmaxf(sh->col[0][c], sh->col[1][c]), fmaxf(sh->col[2][c], sh->col[3][c]));
                    const float m_old = sh->m[c];
                    const float m_new = fmaxf(m_old, o * sl2);
                    sh->factor[j & 1][c] = (m_old == -INFINITY) ? 0.f : fast_exp2(m_old - m_new);
                    sh->m[c] = m_new;
                }
                named_barrier(bar_sync, 128);
                if (j > 0) {   // O^T holds the tiles before j: P V of tile j - 1 must have completed
                    mbar_wait(bar(B_PVDONE), (j - 1) & 1, abort_flag, p.dev_status);
                    fence_after();
                    const uint32_t o_addr = tmem + lane_addr + TM_O + c0;
#pragma unroll
                    for (int q = 0; q < NH / W; ++q) {
                        ld_row<W>(o_addr + W * q, sr[0]);
#pragma unroll
                        for (int c = 0; c < W; ++c)
                            sr[0][c] = __float_as_uint(__uint_as_float(sr[0][c]) * sh->factor[j & 1][c0 + W * q + c]);
                        if constexpr (W == 8) st8(o_addr + W * q, sr[0]);
                        else st16(o_addr + W * q, sr[0]);
                    }
                    wait_st();
#pragma unroll
                    for (int i = 0; i < NH / 2; ++i) {
                        const float2 f = *reinterpret_cast<const float2*>(&sh->factor[j & 1][c0 + 2 * i]);
                        lsum[i] = mul2(lsum[i], pk(f.x, f.y));
                    }
                }
            }
            // the P^T buffer is free once P V of the previous tile has completed
            if (j > 0) mbar_wait(bar(B_PVDONE), (j - 1) & 1, abort_flag, p.dev_status);
#pragma unroll
            for (int ch = 0; ch < NH / 8; ++ch) {
                const int gch = (c0 >> 3) + ch;      // 16-byte chunk (8 slots) of the whole P^T row
                *reinterpret_cast<uint4*>(prow + (gch >> 3) * SUB + (((gch & 7) ^ (kk & 7)) << 4)) =
                    make_uint4(pw[4 * ch], pw[4 * ch + 1], pw[4 * ch + 2], pw[4 * ch + 3]);
            }
            fence_async_smem();
            fence_before();
            mbar_arrive_warp(bar(B_PFULL));
#pragma unroll
            for (int i = 0; i < NH / 2; ++i)   // (while the second product runs)
                lsum[i] = add2(lsum[i], pk(__uint_as_float(pw[i] << 16), __uint_as_float(pw[i] & 0xffff0000u)));
        }
        {   // row sums over the warp's 32 keys: the first steps halve the columns a lane holds, the last ones add neighbours
            constexpr int kHalve = NH % 16 ? 3 : 4;
            float v[NH];
#pragma unroll
            for (int i = 0; i < NH / 2; ++i) upk(lsum[i], v[2 * i], v[2 * i + 1]);
            int first = c0;
#pragma unroll
            for (int step = 1; step <= kHalve; ++step) {
                const int n = NH >> step, o = 32 >> step;
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
                first += up ? n : 0;
            }
#pragma unroll
            for (int i = 0; i < NH >> kHalve; ++i) {
#pragma unroll
                for (int o = 16 >> kHalve; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
                if (!(lane & ((32 >> kHalve) - 1))) sh->col[quarter][first + i] = v[i];
            }
        }
        named_barrier(bar_sync, 128);
        auto row_sum = [&](int c) { return (sh->col[0][c] + sh->col[1][c]) + (sh->col[2][c] + sh->col[3][c]); };
        if (C == 1) {
            if (st_w < NH) sh->factor[0][c0 + st_w] = 1.f / row_sum(c0 + st_w);
            named_barrier(bar_sync, 128);
        }
        mbar_wait(bar(B_PVDONE), (T - 1) & 1, abort_flag, p.dev_status);   // Q, P^T and the K/V stages are dead from here on
        fence_after();
        uint32_t o[NH];
        ld_row<NH>(tmem + lane_addr + TM_O + c0, o);
        fence_before();
        named_arrive(1, kSoft + 32);   // tensor memory has been read: the MMA warp may free it
        if (C == 1) {
            // ---- single CTA per (sequence, kv head): normalise and store column kk of every query row ----
            if (!*abort_flag) {
#pragma unroll
                for (int c = 0; c < NH; ++c) {
                    if (c0 + c < rows_total) {
                        const int i = ((c0 + c) * p.group_inv) >> 16, jh = c0 + c - i * p.group;
                        if (jh >= heads) continue;
                        __nv_bfloat16* dst = p.out + (((long long)b * p.n_active + i0 + i) * p.n_q_heads + hq0 + jh) * HD;
                        dst[kk] = __float2bfloat16_rn(__uint_as_float(o[c]) * sh->factor[0][c0 + c]);
                    }
                }
            }
        } else {
            // ---- this thread's O^T row (output column kk, its warpgroup's queries), m and l into this CTA's partial:
            //      consecutive lanes write consecutive words ----
            float* part = reinterpret_cast<float*>(gbase) + kk;
#pragma unroll
            for (int c = 0; c < NH; ++c)
                if (c0 + c < rows_total) part[(c0 + c) * PITCH] = __uint_as_float(o[c]);
            if (st_w < NH) {
                const int c = c0 + st_w;
                *reinterpret_cast<float2*>(gbase + ML_OFF + c * 8) = make_float2(sh->m[c], row_sum(c));
            }
        }
    }
    if (warp == 1) {
        __syncwarp();
        named_barrier(1, kSoft + 32);
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TM_COLS) : "memory");
    }
    if (C == 1) return;

    // ---- merge the C partials of the output columns this CTA owns: a thread takes a query row and four adjacent columns
    //      (consecutive threads read consecutive words), reads them out of the peers' shared memory and works out its row's
    //      weights 2^(m_s - m) / l itself: the few threads of a row repeat that, but nobody waits for a table.
    __syncwarp();
    cluster_arrive();
    cluster_wait();           // the partials of all CTAs are complete
    const int quads = DL / 4;
    if (!*abort_flag) {
#pragma unroll 1
        for (int idx = tid; idx < rows_total * quads; idx += kThreads) {
            const int qq = (idx * p.quads_inv) >> 16, d0 = (idx - qq * quads) * 4;
            const int i = (qq * p.group_inv) >> 16, jh = qq - i * p.group;
            if (d0 >= own_dl || jh >= heads) continue;
            const uint32_t at = base + ((uint32_t)qq * PITCH + (uint32_t)(split * DL + d0)) * 4u;
            float m = -INFINITY, l = 0.f, a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
            for (int s0 = 0; s0 < C; s0 += 4) {   // four sources at a time: their loads are in flight together
                float ms[4], ls[4], x[4][4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int s = min(s0 + k, C - 1);
                    ld_peer_v2(map_to_cta(base + ML_OFF + (uint32_t)qq * 8u, s), ms[k], ls[k]);
                    ld_peer_v4(map_to_cta(at, s), x[k]);
                }
                float mn = m;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (s0 + k >= C) ms[k] = -INFINITY;
                    mn = fmaxf(mn, ms[k]);
                }
                const float f = m == -INFINITY ? 0.f : fast_exp2(m - mn);
                m = mn;
                l *= f;
#pragma unroll
                for (int v = 0; v < 4; ++v) a[v] *= f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float e = fast_exp2(ms[k] - mn);
                    l = fmaf(e, ls[k], l);
#pragma unroll
                    for (int v = 0; v < 4; ++v) a[v] = fmaf(e, x[k][v], a[v]);
                }
            }
            const float inv = 1.f / l;
            __nv_bfloat16* dst = p.out + (((long long)b * p.n_active + i0 + i) * p.n_q_heads + hq0 + jh) * HD + split * DL + d0;
            *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(a[0] * inv, a[1] * inv), pack_bf16x2(a[2] * inv, a[3] * inv));
        }
    }
    // no CTA leaves while a peer may still read its partial
    __syncwarp();
    cluster_arrive_relaxed();
    cluster_wait();
}

// ---- host side ---------------------------------------------------------------------------
struct KeysPlan {
    bool ok;
    int group, rows_chunk, n_sub_r, n_sub;   // heads and active rows per CTA column, row chunks, CTA columns per kv head
    int n_slots, n_splits, tiles_per_split, n_stages, n_extra, dl, shift;
    uint32_t off_p, off_stage, off_list, off_bar, smem_bytes;
};

constexpr uint32_t kSmemMax = 232448;        // 227 KB: largest dynamic allocation of one CTA
constexpr uint32_t kSmemTwoPerSm = 115712;   // (228 KB per SM - 2 x 1 KB reserved) / 2

// tensor-memory columns the instantiation for n_slots allocates (see TM_COLS in the kernel)
constexpr int tm_columns(int n_slots) { return 3 * (n_slots <= 64 ? 64 : 128) <= 256 ? 256 : 512; }

// shared-memory carve for n_slots query slots and ns stages; `fresh`: room for the stale-key bits (16 bytes per
// cache tile of a CTA, of which it may hold one more than tiles_per_split)
void carve(KeysPlan& pl, int ns, bool fresh) {
    uint32_t off = (uint32_t)pl.n_slots * 256u;   // Q
    off = (off + 1023u) & ~1023u;
    pl.off_p = off;
    off += (uint32_t)((pl.n_slots + 63) / 64) * SUB;
    pl.off_stage = off;
    off += (uint32_t)ns * TILE;
    pl.off_list = off;
    off += fresh ? (uint32_t)(pl.tiles_per_split + 1) * 16u : 0u;
    pl.off_bar = off;
    off += kBarBytes + (uint32_t)sizeof(KeysShared) + 16u;
    pl.smem_bytes = off + 1024u;
    // an instantiation that allocates all 512 columns of tensor memory must never share an SM with a CTA of its own
    // cluster (the second allocation would wait for the first CTA, which waits for it at the cluster barrier): ask for
    // more than half an SM's shared memory
    if (tm_columns(pl.n_slots) > 256 && pl.smem_bytes <= kSmemTwoPerSm) pl.smem_bytes = kSmemTwoPerSm + 1024u;
    pl.n_stages = ns;
}

// How many clusters of c CTAs with this much dynamic shared memory the current device keeps resident at once (clusters
// are placed inside one GPC, so this can be fewer than SMs x CTAs per SM / c); -1 when it cannot be asked (no device).
// Asked once per (device, instantiation, cluster size, shared memory) and remembered.
template <int N>
int resident_clusters_of(int c, uint32_t smem) {
    static PerDeviceOnce attr_once;
    if (ensure_dynamic_smem(attr_once, attend_skip_keys_kernel<N>, (int)kSmemMax) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c, 1, 1);
    cfg.blockDim = dim3(block_threads(N), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attend_skip_keys_kernel<N>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    return n;
}

int resident_clusters(int n_slots, int c, uint32_t smem) {
    struct Entry { int dev, n_slots, c; uint32_t smem; int clusters; };
    static std::mutex mu;
    static std::vector<Entry> seen;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        return -1;
    }
    std::lock_guard<std::mutex> lock(mu);
    for (const Entry& e : seen)
        if (e.dev == dev && e.n_slots == n_slots && e.c == c && e.smem == smem) return e.clusters;
    const int n = n_slots == 48 ? resident_clusters_of<48>(c, smem) : n_slots == 64 ? resident_clusters_of<64>(c, smem)
                                                                                      : resident_clusters_of<96>(c, smem);
    seen.push_back({dev, n_slots, c, smem, n});
    return n;
}

// fresh: the call refreshes (k_new / v_new given), so the last CTA of every cluster also visits the fresh tiles
KeysPlan compute_keys_plan(const ec_attn_desc& d, int n_active, bool fresh) {
    KeysPlan pl{};
    const int g = d.n_q_heads / d.n_kv_heads;
    const int key_tiles = (d.ctx_len + BK - 1) / BK;
    const int sms = sm_count();
    long long best_cost = -1, best_ctas = 0;
    // A CTA column takes `group` query heads of a kv head; the columns of a kv head stream the same K/V (from L2).  Fewer
    // columns leave more CTAs for splitting the keys, but more packed rows make a tile dearer.
    for (int cols = 1; cols <= g; ++cols) {
        KeysPlan base = KeysPlan{};
        base.group = (g + cols - 1) / cols;
        if ((g + base.group - 1) / base.group != cols) continue;
        if (base.group > 1 && (long long)n_active * base.group > kMaxSlots) continue;
        // more active rows than slots: the rows are cut into equal chunks, one CTA column each
        base.n_sub_r = (n_active * base.group + kMaxSlots - 1) / kMaxSlots;
        base.rows_chunk = (n_active + base.n_sub_r - 1) / base.n_sub_r;
        base.n_sub_r = (n_active + base.rows_chunk - 1) / base.rows_chunk;
        base.n_sub = cols * base.n_sub_r;
        const int rows = base.rows_chunk * base.group;
        base.n_slots = rows <= 48 ? 48 : rows <= 64 ? 64 : 96;
        base.n_extra = fresh ? (n_active + BK - 1) / BK : 0;
        const long long columns = (long long)d.batch * d.n_kv_heads * base.n_sub;   // grid.y
        // Cluster shape: cs CTAs split the cache tiles (every one at least one tile); the fresh tiles go to the last of
        // them, or to one more CTA of their own (worth it when a CTA holds so few tiles that one more would be felt).
        // All CTAs resident at once; the most-loaded SM streams as few tiles as possible; among equals, more CTAs (more
        // SMs pulling).
        for (int cs = 1; cs <= 8 && cs <= key_tiles; ++cs) {
            const int tps = (key_tiles + cs - 1) / cs;
            if ((key_tiles + tps - 1) / tps != cs || tps > kMaxTiles) continue;   // this cs leaves a CTA empty
            for (int own = 0; own <= (fresh ? 1 : 0); ++own) {                     // own: the fresh tiles get their own CTA
                const int c = cs + own;
                if (c > 8) continue;
                const int dl = ((HD + c - 1) / c + 7) & ~7;                        // (the last CTAs may own fewer columns, or none)
                const int last_tiles = key_tiles - (cs - 1) * tps;
                const int visits = own ? (tps > base.n_extra ? tps : base.n_extra)
                                       : (tps > last_tiles + base.n_extra ? tps : last_tiles + base.n_extra);
                KeysPlan t = base;
                int ns = 2 * visits < kMaxStages ? 2 * visits : kMaxStages;   // ring slots: a K and a V slot per tile in flight
                t.tiles_per_split = tps;
                carve(t, ns, fresh);
                while (ns > 2 && t.smem_bytes > kSmemMax) carve(t, --ns, fresh);
                if (t.smem_bytes > kSmemMax || (ns < 4 && visits > 1)) continue;
                // the partial of the merge reuses the Q / P^T / stage memory
                if (c > 1 && partial_bytes(t.n_slots) > t.off_list) continue;
                const long long ctas = columns * c;
                if (ctas > sms) continue;   // one CTA per SM: registers
                // Cost in quarter tiles (about 0.25 us): the fresh tiles arrive early (they are small and mostly in L2), so
                // on a shared CTA they count a quarter of a cache tile.  96 slots: a tile takes 1.3 us where the memory
                // system does not set the pace (48, and 64 by the same price: 1.0), and the launch around the tiles up to 3
                // us more.  (Fitted when one softmax warpgroup, two with 96 slots, worked on a tile; the launches have become
                // up to 15 % shorter since, and the prices were not fitted again.)
                const long long cost = (t.n_slots == 96 ? 5LL * tps + 13 : 4LL * tps) + ((fresh && !own) ? t.n_extra : 0);
                if (best_cost >= 0 && (cost > best_cost || (cost == best_cost && ctas <= best_ctas))) continue;
                const int fit = resident_clusters(t.n_slots, c, t.smem_bytes);   // (-1: no device to ask, keep the estimate)
                if (fit >= 0 && columns > fit) continue;
                best_cost = cost;
                best_ctas = ctas;
                pl = t;
                pl.n_splits = c;
                // The CTA that also visits the fresh tiles has one visit more than its peers, and the cluster waits for
                // it at the merge.  The memory system serves whoever asks, so giving that CTA one cache tile less (and
                // the first CTA one more) lets it finish its stream early and spend the difference on the extra visit.
                pl.shift = (fresh && !own && cs >= 2 && tps >= 2 && last_tiles == tps) ? 1 : 0;
                pl.dl = dl;
                pl.ok = true;
            }
        }
    }
    return pl;
}

// The plan of the last geometry a thread asked for is kept: a layer loop asks for the same one at every call, twice (a
// plan takes 1 to 2 us of host time, a launch 3).
KeysPlan make_keys_plan(const ec_attn_desc& d, int n_active, bool fresh) {
    struct Key {
        int dev, batch, ctx_len, n_q_heads, n_kv_heads, n_active, fresh;
        bool operator==(const Key& o) const {
            return dev == o.dev && batch == o.batch && ctx_len == o.ctx_len && n_q_heads == o.n_q_heads &&
                   n_kv_heads == o.n_kv_heads && n_active == o.n_active && fresh == o.fresh;
        }
    };
    static thread_local Key last{-2, 0, 0, 0, 0, 0, 0};
    static thread_local KeysPlan plan;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    const Key key{dev, d.batch, d.ctx_len, d.n_q_heads, d.n_kv_heads, n_active, fresh ? 1 : 0};
    if (!(key == last)) {
        plan = compute_keys_plan(d, n_active, fresh);
        last = key;
    }
    return plan;
}

// bytes per nanosecond assumed for a streaming read when spacing the first ring fill: 0.7 of the nominal rate of the
// device (clock x bus width, double data rate; a spacing between 1.0 and 1.3 times the measured copy rate's stage
// time timed best), cached per device
double stream_bytes_per_ns() {
    static std::atomic<uint64_t> cached[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 5700.0;
    const bool slot = dev >= 0 && dev < kMaxDevices;
    if (slot) {
        const uint64_t v = cached[dev].load(std::memory_order_relaxed);
        if (v) return (double)v;
    }
    int khz = 0, bits = 0;
    if (cudaDeviceGetAttribute(&khz, cudaDevAttrMemoryClockRate, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&bits, cudaDevAttrGlobalMemoryBusWidth, dev) != cudaSuccess || khz <= 0 || bits <= 0) {
        (void)cudaGetLastError();
        return 5700.0;
    }
    const double rate = 0.7 * 2.0 * (double)khz * 1e3 * (bits / 8.0) * 1e-9;
    if (slot) cached[dev].store((uint64_t)rate, std::memory_order_relaxed);
    return rate;
}

template <int N>
cudaError_t launch_n(const KeysPlan& pl, const KeysParams& p, const CUtensorMap& mk, const CUtensorMap& mv,
                     const CUtensorMap& mkn, const CUtensorMap& mvn, int bh, cudaStream_t stream) {
    static PerDeviceOnce attr_once;
    if (const cudaError_t ea = ensure_dynamic_smem(attr_once, attend_skip_keys_kernel<N>, (int)kSmemMax); ea != cudaSuccess)
        return ea;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(pl.n_splits, bh, 1);
    cfg.blockDim = dim3(block_threads(N), 1, 1);
    cfg.dynamicSmemBytes = pl.smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = pl.n_splits;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // set-up may overlap the previous kernel's tail
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attend_skip_keys_kernel<N>, mk, mv, mkn, mvn, p);
}

}  // namespace

bool attend_skip_keys_supported(const ec_attn_desc& d, int n_active, bool fresh) {
    if (d.dtype != EC_BF16 || d.head_dim != HD || n_active < 1) return false;
    if (n_active > kMaxActive) return false;
    const KeysPlan pl = make_keys_plan(d, n_active, fresh);
    if (!pl.ok) return false;   // no cluster shape keeps all CTAs resident: the row-major skip kernel streams better
    if ((long long)d.batch * d.n_kv_heads * pl.n_sub > 65535) return false;   // grid.y
    // row chunks re-read the K/V of a head once per chunk: only worth it while the keys can still be split
    if (pl.n_sub_r > 1 && pl.n_splits < 2) return false;
    return true;
}

void attend_skip_keys_describe(const ec_attn_desc& d, int n_active, bool fresh, char* buf, size_t len) {
    const KeysPlan pl = make_keys_plan(d, n_active, fresh);
    snprintf(buf, len, "attend_skip_keys_kernel<%d> grid=(%d,%d) cluster=%d ring_slots=%d smem=%u ctas_per_sm=1 fresh_tiles=%d",
             pl.n_slots, pl.n_splits, d.batch * d.n_kv_heads * pl.n_sub, pl.n_splits, pl.n_stages, pl.smem_bytes, pl.n_extra);
}

cudaError_t launch_attend_skip_keys(const AttendArgs& a, const void* k_new, const void* v_new, const int32_t* active_idx,
                                    cudaStream_t stream) {
    const bool fresh = k_new != nullptr;
    const KeysPlan pl = make_keys_plan(a.d, a.n_active, fresh);
    if (!pl.ok) return cudaErrorInvalidConfiguration;
    const int bh = a.d.batch * a.d.n_kv_heads;
    CUtensorMap map_k, map_v;
    if (!make_cache_map(&map_k, a.k_cache, bh, a.d.ctx_len, BK) || !make_cache_map(&map_v, a.v_cache, bh, a.d.ctx_len, BK))
        return cudaErrorInvalidValue;
    KeysParams p{};
    CUtensorMap map_kn = map_k, map_vn = map_v;   // placeholders unless fresh
    if (fresh && (!make_fresh_map(&map_kn, k_new, a.d.batch, a.n_active, a.d.n_kv_heads, BK) ||
                  !make_fresh_map(&map_vn, v_new, a.d.batch, a.n_active, a.d.n_kv_heads, BK)))
        return cudaErrorInvalidValue;
    p.q = static_cast<const __nv_bfloat16*>(a.q);
    p.k_new = static_cast<const __nv_bfloat16*>(k_new);
    p.v_new = static_cast<const __nv_bfloat16*>(v_new);
    p.k_cache = static_cast<__nv_bfloat16*>(const_cast<void*>(a.k_cache));
    p.v_cache = static_cast<__nv_bfloat16*>(const_cast<void*>(a.v_cache));
    p.active_idx = active_idx;
    p.out = static_cast<__nv_bfloat16*>(a.out);
    p.dev_status = a.dev_status;
    p.n_active = a.n_active;
    p.ctx_len = a.d.ctx_len;
    p.n_q_heads = a.d.n_q_heads;
    p.n_kv_heads = a.d.n_kv_heads;
    p.group = pl.group;
    p.q_per_kv = a.d.n_q_heads / a.d.n_kv_heads;
    p.group_inv = (65536 + pl.group - 1) / pl.group;
    p.rows_chunk = pl.rows_chunk;
    p.n_sub_r = pl.n_sub_r;
    p.n_sub = pl.n_sub;
    p.n_splits = pl.n_splits;
    p.tiles_per_split = pl.tiles_per_split;
    p.shift = pl.shift;
    p.n_stages = pl.n_stages;
    p.n_extra = pl.n_extra;
    p.dl = pl.dl;
    p.quads_inv = (65536 + pl.dl / 4 - 1) / (pl.dl / 4);
    p.off_p = pl.off_p;
    p.off_stage = pl.off_stage;
    p.off_list = pl.off_list;
    p.off_bar = pl.off_bar;
    p.scale_log2 = a.scale * kLog2e;
    p.early_cache = (a.d.flags & EC_ATTN_CACHE_SETTLED) ? 1 : 0;
    p.stagger_ns = 0;
    if (pl.tiles_per_split > 1) {
        const double streams = (double)pl.n_splits * bh;   // CTAs with K/V of their own (columns of one head share it through L2)
        const double ns = streams * STAGE / stream_bytes_per_ns();
        p.stagger_ns = (uint32_t)(ns < 3000.0 ? ns : 3000.0);
    }
    const int cols = bh * pl.n_sub;
    return pl.n_slots == 48   ? launch_n<48>(pl, p, map_k, map_v, map_kn, map_vn, cols, stream)
           : pl.n_slots == 64 ? launch_n<64>(pl, p, map_k, map_v, map_kn, map_vn, cols, stream)
                              : launch_n<96>(pl, p, map_k, map_v, map_kn, map_vn, cols, stream);
}

}  // namespace ec
