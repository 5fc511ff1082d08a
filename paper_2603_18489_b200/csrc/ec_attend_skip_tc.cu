// ec_attend, skip step (bf16, head_dim 128, at most 256 packed query rows per kv head):
// ONE launch that refreshes the active rows' K/V in the cache, attends from the active
// rows over the whole cache and merges the key-range partials -- no workspace, no second
// kernel.  (Section 4.2 and Appendix A of the paper, partial branch:
// TransformerBlock(Q[M u R], K[I], V[I]) after the rows M u R got fresh K, V.)
//
// The step is HBM-bound (every K/V byte of the cache is read exactly once) and, at the
// context lengths of a diffusion LM block, latency-bound: the design keeps every
// global round trip off the path between kernel start and the first K/V tile, and off
// the path between the last tile and the output.
//   grid     (C, B*H_kv), launched as clusters of C CTAs: the C CTAs of a cluster share
//            one (sequence, kv head) and split its 64-key tiles into C contiguous ranges;
//   rows     the n_active x (H_q/H_kv) query rows that share the kv head are packed
//            into one or two 128-row M tiles (NT); the same K/V tile serves both;
//   warp 1   issues the tcgen05.mma (S = Q K^T, M128 N64 K16 x 8, into one of two TMEM S
//            buffers; O += P V, M128 N128 K16 x 4, P from shared memory, V MN-major), whichever
//            of the two is ready;
//   refresh  the fresh rows are attended straight from k_new / v_new, as extra key tiles that
//            the last CTA of a cluster visits after its cache tiles, while every CTA masks the
//            stale cached keys of the refreshed positions (a bit per key); softmax warps without
//            query rows build the masks and copy the fresh rows into the cache, ordered against
//            nothing.  (Waiting for that copy before the first tile that holds a refreshed
//            position, and for the list of positions before the first tile at all, cost 3 us a
//            launch);
//   warp 0   TMA producer: one 4-D box per operand tile ([2 halves][64 keys][64 columns],
//            128-byte swizzle), NS stages, full/empty mbarriers;
//   warps 2+ load Q into swizzled shared memory, then run the softmax: a query row (= TMEM lane)
//            has two threads, in warps that own the same lanes, each of which takes 32 of a
//            tile's 64 keys.  A reference in place of the running maximum: probabilities may
//            exceed it by 2^60 (fp32 and bf16 have room for that, and it is never above the
//            true maximum) before the two agree on a larger one and rescale O.  The chain of a
//            tile (scores, softmax, second product) is what bounds the kernel, not memory, as
//            long as there are fewer than about three CTAs for two SMs: 1.3 us with one thread
//            per row and a running maximum;
//   merge    the un-normalised rows (O, m, l) go from TMEM to a staging area grouped by
//            owner (row r belongs to CTA r mod C of the cluster) and from there with one
//            bulk shared-to-shared copy per owner into the owner's receive buffer,
//            completing on the owner's mbarrier; the owner combines the C partials,
//            normalises and writes out[b, i, h, :].
// Shared memory only holds the rows that exist: the tensor core always multiplies 128
// rows, and the rows past the last packed query row read whatever follows in the CTA's
// own allocation; rows of S, P and O are independent, so those values never reach a
// real row and are never stored.
// The kernel is launched with programmatic stream serialisation: set-up may overlap the
// previous kernel of the stream, and so may the first cache tiles when the caller has
// stated that nothing in flight writes the caches; all else is read after griddepcontrol.wait.
// Every mbarrier wait is bounded: a wait that runs out sets EC_ERR_TIMEOUT in the
// caller's dev_status word and a CTA-wide abort flag that makes all later waits fall
// through; the CTA still frees its TMEM and exits.
#include "ec_common.cuh"
#include "ec_skip_keys_pair.cuh"
#include "ec_tc_ptx.cuh"

#include <cuda.h>

#include <cstdio>

namespace ec {
namespace {

using namespace tc;

constexpr int BM = 128, BN = 64, HD = 128;
constexpr uint32_t KV_SUB = BN * 128;      // [64 keys x 64 bf16], 128-byte swizzle: 8 KB
constexpr uint32_t KV_TILE = 2 * KV_SUB;   // [64 keys x 128 bf16]
constexpr uint32_t STAGE = 2 * KV_TILE;    // K tile + V tile: 32 KB
constexpr int kMaxStages = 6;
constexpr int kRec = HD + 4;               // floats per exchanged row: O[128], m, l, pad (16-byte multiple)
constexpr int kMaxRows = 2 * BM;
constexpr int kMaxCluster = 8;
constexpr float kRaise = 60.f;             // a score may exceed its row's reference by this power of two

// barrier slots (8 bytes each)
enum {
    B_FULL = 0,                       // [kMaxStages] K/V tile landed
    B_EMPTY = kMaxStages,             // [kMaxStages] tile consumed
    B_SFULL = 2 * kMaxStages,         // [tile][2]
    B_PFULL = B_SFULL + 4,            // [tile]
    B_PVDONE = B_PFULL + 2,           // [tile]
    B_QFULL = B_PVDONE + 2,           // Q tiles staged
    B_LIST = B_QFULL + 1,             // key masks built
    B_RECV = B_LIST + 1,              // all partial rows this CTA owns have arrived
    B_COUNT = B_RECV + 1
};

// 32 columns of this thread's TMEM lane as floats
__device__ __forceinline__ void ld32f(uint32_t taddr, float* v) {
    uint32_t r[32];
    ld32(taddr, r);
    wait_ld<32>(r);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

struct SkipParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_new;   // nullptr: attend without refreshing
    const __nv_bfloat16* v_new;
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* active_idx;    // nullptr: identity
    __nv_bfloat16* out;
    int32_t* dev_status;
    int n_active, ctx_len, n_q_heads, n_kv_heads, group, rows_total;
    int n_splits, tiles_per_split, n_stages, rows_per_cta;
    int n_extra;      // key tiles of fresh rows attended by the last CTA of every cluster (0: nothing to refresh)
    int keys_on_m;    // 1: the CTA runs keys_pair::run
    int early_cache;  // 1: nothing still running on the stream writes the caches (EC_ATTN_CACHE_SETTLED)
    // shared-memory carve (bytes from the 1024-aligned base)
    uint32_t off_q[2], off_p[2], rows_pad[2], off_stage, off_recv, off_list, off_xch, off_bar;
    float scale_log2;
};

// words after the barrier block
struct SkipShared {
    uint32_t tmem;
    int abort_flag;
};

template <int NT>
__global__ void __launch_bounds__(64 + NT * 256, NT == 1 ? 2 : 1)
attend_skip_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                   const __grid_constant__ CUtensorMap map_kn, const __grid_constant__ CUtensorMap map_vn, const SkipParams p,
                   const keys_pair::Params kp) {
    constexpr int kThreads = 64 + NT * 256;
    constexpr int kSoftThreads = NT * 256;   // per row tile: (keys 0..31 / 32..63 of a key tile) x 128 rows
    constexpr uint32_t TM_COLS = NT * 256;   // per row tile: S0 [0,64), S1 [64,128), O [128,256)
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = s2u(smem_raw);
    unsigned char* gbase = smem_raw;
    if (base & 1023u) {   // never: the runtime puts dynamic shared memory on a 1024-byte boundary
        if (threadIdx.x == 0 && p.dev_status) atomicExch(p.dev_status, (int)EC_ERR_CUDA);
        return;
    }
    if constexpr (NT == 1) {
        if (p.keys_on_m) {   // few rows, a CTA per kv head: the maps hold 128-key boxes
            if (p.rows_total <= 48) keys_pair::run<48>(map_k, map_v, map_kn, map_vn, kp, smem_raw);
            else keys_pair::run<64>(map_k, map_v, map_kn, map_vn, kp, smem_raw);
            return;
        }
    }
    const uint32_t bars = base + p.off_bar;
    SkipShared* sh = reinterpret_cast<SkipShared*>(gbase + p.off_bar + B_COUNT * 8);
    volatile int* abort_flag = &sh->abort_flag;
    // [key tile of this CTA, cache tiles first][2]: a bit per key; of a cached key whose position is being refreshed (it does
    // not count: it is attended from the fresh tile instead), of a fresh key that exists
    uint32_t* bits = reinterpret_cast<uint32_t*>(gbase + p.off_list);
    auto bar = [&](int idx) { return bars + idx * 8; };

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int split = blockIdx.x, bh = blockIdx.y;
    const int b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads;
    const int C = p.n_splits;
    const int n_tiles_total = (p.ctx_len + BN - 1) / BN;
    const int t_begin = split * p.tiles_per_split;
    const int t_end = min(n_tiles_total, t_begin + p.tiles_per_split);
    const bool refresh = p.k_new != nullptr;
    const int TC = t_end - t_begin;  // cache tiles: >= 1 by construction of the plan
    const int XT = (refresh && split == p.n_splits - 1) ? p.n_extra : 0;   // fresh tiles, visited after them
    const int T = TC + XT;
    const int NS = p.n_stages;
    const int n_own = (p.rows_total - split + C - 1) / C;   // packed rows r = split + q * C merged by this CTA

    // softmax warps that own no query row copy the fresh rows; when every warp owns rows, all of them share it
    int n_idle = 0, my_idle = -1;
#pragma unroll
    for (int w = 2; w < 2 + NT * 8; ++w) {
        const int rows_w = min(BM, p.rows_total - ((w - 2) >> 3) * BM);
        if (!((w & 3) * 32 < rows_w)) {
            if (w == warp) my_idle = n_idle;
            ++n_idle;
        }
    }
    const int n_copy_threads = n_idle == 0 ? kSoftThreads : n_idle * 32;

    // ---- set-up (touches no global memory) -------------------------------------------------
    if (tid == 0) {
        prefetch_map(&map_k);
        prefetch_map(&map_v);
        for (int i = 0; i < B_COUNT; ++i) {
            uint32_t count = 1;
            if (i >= B_PFULL && i < B_PFULL + 2) {
                const int rows_t = min(BM, p.rows_total - (i - B_PFULL) * BM);
                count = rows_t > 0 ? 64u * ((rows_t + 31) / 32) : 1u;
            } else if (i == B_QFULL) {
                count = kSoftThreads;
            } else if (i == B_LIST) {
                count = (uint32_t)n_copy_threads;
            }
            mbar_init(bar(i), count);
        }
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (C > 1 && n_own > 0) mbar_expect_tx(bar(B_RECV), (uint32_t)(C * n_own * kRec * 4));
    }
    for (int w = tid; w < 2 * T; w += kThreads) bits[w] = 0u;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s2u(&sh->tmem)), "r"(TM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        fence_before();
    }
    __syncthreads();
    fence_after();
    const uint32_t tmem = sh->tmem;
    if (warp != 0) pdl_wait();     // the previous kernel of the stream has completed; its results may be read
    if (tid == 32) pdl_launch_dependents();
    __syncwarp();

    // softmax role: warp w >= 2 owns TMEM lanes 32 * (w % 4) of row tile (w - 2) / 8 and half ((w - 2) / 4) % 2 of the keys
    const int soft_tile = warp >= 2 ? (warp - 2) >> 3 : 0;
    const int half = warp >= 2 ? ((warp - 2) >> 2) & 1 : 0;
    const int soft_row = (warp & 3) * 32 + lane;
    const int soft_rows_t = min(BM, p.rows_total - soft_tile * BM);
    const bool soft_active = warp >= 2 && (warp & 3) * 32 < soft_rows_t;   // warp-uniform
    const bool valid = soft_active && soft_row < soft_rows_t;
    const uint32_t tm_t = tmem + ((uint32_t)((warp & 3) * 32) << 16) + soft_tile * 256;
    float m_used = -INFINITY, l_run = 0.f;
    const int key_lo = t_begin * BN, key_hi = min(p.ctx_len, t_end * BN);

    if (warp == 0) {
        // ================================ TMA producer ======================================
        if (lane == 0) {
            auto load = [&](int j) {
                const int s = j % NS;
                const uint32_t dst = base + p.off_stage + s * STAGE;
                mbar_expect_tx(bar(B_FULL + s), STAGE);
                if (j >= TC) {   // active rows [64 x, 64 x + 64) of this kv head, fresh; rows past n_active read as zero
                    tma_load_5d(dst, &map_kn, 0, (j - TC) * BN, 0, hk, b, bar(B_FULL + s));
                    tma_load_5d(dst + KV_TILE, &map_vn, 0, (j - TC) * BN, 0, hk, b, bar(B_FULL + s));
                } else {
                    tma_load_4d(dst, &map_k, 0, (t_begin + j) * BN, 0, bh, bar(B_FULL + s));
                    tma_load_4d(dst + KV_TILE, &map_v, 0, (t_begin + j) * BN, 0, bh, bar(B_FULL + s));
                }
            };
            int j = 0;
            if (p.early_cache)
                for (const int fill = min(NS, TC); j < fill; ++j) load(j);
            pdl_wait();
            for (; j < T; ++j) {
                if (j >= NS) mbar_wait(bar(B_EMPTY + j % NS), (j / NS - 1) & 1, abort_flag, p.dev_status);
                load(j);
            }
        } else {
            pdl_wait();
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================================ MMA issue (the whole warp, see elect_one) =====================
        const bool elected = elect_one();
        constexpr uint32_t IDESC_S = instr_desc(BN, 0), IDESC_PV = instr_desc(HD, 1);
        uint64_t desc_q[NT], desc_p[NT];
        uint32_t qh[NT];   // one 64-column half of the Q tile, in descriptor units
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            desc_q[t] = smem_desc(base + p.off_q[t], 16, 1024);
            desc_p[t] = smem_desc(base + p.off_p[t], 16, 1024);
            qh[t] = p.rows_pad[t] * 8u;
        }
        // S of a tile needs the tile, P V of a tile and row tile needs its P: whichever is ready is issued.  S may run
        // one tile ahead of P V (two S buffers).
        int next_s = 0, next_pv[NT], n_pv = 0;   // n_pv: tiles whose P V has been issued for every row tile
#pragma unroll
        for (int t = 0; t < NT; ++t) next_pv[t] = 0;
        mbar_wait(bar(B_QFULL), 0, abort_flag, p.dev_status);
        SpinGuard guard;
        while (n_pv < T) {
            bool progressed = false;
            if (next_s < T && next_s <= n_pv + 1 && mbar_test_warp(bar(B_FULL + next_s % NS), (next_s / NS) & 1)) {
                const uint64_t desc_k = smem_desc(base + p.off_stage + (next_s % NS) * STAGE, 16, 1024);
                fence_after();
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    if (elected) {
#pragma unroll
                        for (int k = 0; k < HD / 16; ++k)
                            mma_ss(tmem + t * 256 + (next_s & 1) * 64, desc_q[t] + (k >> 2) * qh[t] + (k & 3) * 2,
                                   desc_k + (k >> 2) * (KV_SUB / 16) + (k & 3) * 2, IDESC_S, k > 0);
                        commit(bar(B_SFULL + t * 2 + (next_s & 1)));
                    }
                }
                ++next_s;
                progressed = true;
            }
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                const int j = next_pv[t];
                if (j >= next_s || !mbar_test_warp(bar(B_PFULL + t), j & 1)) continue;
                const uint64_t desc_v = smem_desc(base + p.off_stage + (j % NS) * STAGE + KV_TILE, KV_SUB, 1024);
                fence_after();
                if (elected) {
#pragma unroll
                    for (int k = 0; k < BN / 16; ++k)
                        mma_ss(tmem + t * 256 + 128, desc_p[t] + k * 2, desc_v + k * 128, IDESC_PV, (j > 0 || k > 0));
                    commit(bar(B_PVDONE + t));
                }
                ++next_pv[t];
                progressed = true;
            }
            int done = next_pv[0];
#pragma unroll
            for (int t = 1; t < NT; ++t) done = min(done, next_pv[t]);
            for (; n_pv < done; ++n_pv)
                if (elected) commit(bar(B_EMPTY + n_pv % NS));
            if (progressed) guard.progress();
            else if (__any_sync(0xffffffffu, !guard.tick(abort_flag, p.dev_status))) break;
        }
    } else {
        // ================== Q staging, cache refresh, softmax (warps 2..) ========================
        const int stid = tid - 64;
        // Q rows of this kv head -> swizzled K-major tiles (rows past rows_total inside the padded tile are zero)
        for (int t = 0; t < NT; ++t) {
            const int rows_pad = (int)p.rows_pad[t];
            for (int c = stid; c < rows_pad * (HD / 8); c += kSoftThreads) {
                const int row = c >> 4, ch = c & 15;
                const int r = t * BM + row;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (r < p.rows_total) {
                    const int i = r / p.group, j = r % p.group;
                    v = __ldg(reinterpret_cast<const uint4*>(
                        p.q + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + j) * HD + ch * 8));
                }
                const uint32_t off = p.off_q[t] + (ch >> 3) * (uint32_t)rows_pad * 128u + (row >> 3) * 1024 + (row & 7) * 128 +
                                     (((ch & 7) ^ (row & 7)) << 4);
                *reinterpret_cast<uint4*>(gbase + off) = v;
            }
        }
        fence_async_smem();         // Q tiles (generic proxy) -> visible to the tensor core (async proxy)
        mbar_arrive(bar(B_QFULL));

        if (refresh && (n_idle == 0 || my_idle >= 0)) {
            const int wid = n_idle == 0 ? stid : my_idle * 32 + lane;
            // key masks: stale cached keys of this CTA's range, and the fresh keys that exist
            for (int i = wid; i < p.n_active; i += n_copy_threads) {
                const int pos = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i;
                if (pos >= key_lo && pos < key_hi) atomicOr(&bits[(pos - key_lo) >> 5], 1u << ((pos - key_lo) & 31));
                if (XT && pos >= 0 && pos < p.ctx_len) atomicOr(&bits[2 * TC + (i >> 5)], 1u << (i & 31));
            }
            mbar_arrive(bar(B_LIST));   // release: the bits above are visible to whoever waits
            // this CTA's share of the fresh rows -> cache in global memory, for later steps, four 16-byte pieces in flight
            // per thread; nothing in this launch depends on it
            const int pieces = p.n_active * 32;   // [row][K, V][16 pieces]
            for (int q0 = split * n_copy_threads + wid; q0 < pieces; q0 += 4 * C * n_copy_threads) {
                uint4 v[4];
                int pos[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = q0 + u * C * n_copy_threads, i = c >> 5;
                    pos[u] = -1;
                    if (c < pieces) {
                        pos[u] = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i;
                        const __nv_bfloat16* src = (c & 16) ? p.v_new : p.k_new;
                        v[u] = __ldg(reinterpret_cast<const uint4*>(
                            src + (((long long)b * p.n_active + i) * p.n_kv_heads + hk) * HD + (c & 15) * 8));
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = q0 + u * C * n_copy_threads;
                    if (pos[u] < 0 || pos[u] >= p.ctx_len) continue;
                    __nv_bfloat16* dst = (c & 16) ? p.v_cache : p.k_cache;
                    *reinterpret_cast<uint4*>(dst + ((long long)bh * p.ctx_len + pos[u]) * HD + (c & 15) * 8) = v[u];
                }
            }
        }

        // exchange between the two threads of a row: [half][row], rows that exist
        float* xch = reinterpret_cast<float*>(gbase + p.off_xch) + soft_tile * 2 * (int)p.rows_pad[0];
        const int rows_x = (int)p.rows_pad[soft_tile], soft_row_x = min(soft_row, rows_x - 1);
        if (soft_active) {
            const float sl2 = p.scale_log2;
            const f32x2 sl2_2 = pk(sl2, sl2);
            const int t = soft_tile;
            unsigned char* prow = gbase + p.off_p[t] + (soft_row >> 3) * 1024 + (soft_row & 7) * 128;
            const bool store_p = soft_row < (int)p.rows_pad[t];   // rows past the padded tile have no storage
            const int pair_bar = 1 + t * 4 + (warp & 3);          // named barrier of the two warps that share these rows

            for (int j = 0; j < T; ++j) {
                mbar_wait(bar(B_SFULL + t * 2 + (j & 1)), (j >> 1) & 1, abort_flag, p.dev_status);
                fence_after();
                uint32_t sc[32];
                ld32(tm_t + (j & 1) * 64 + half * 32, sc);
                wait_ld<32>(sc);
                uint32_t gone = 0;   // keys that do not count
                if (refresh) {
                    if (j == 0) mbar_wait(bar(B_LIST), 0, abort_flag, p.dev_status);
                    gone = j < TC ? bits[2 * j + half] : ~bits[2 * j + half];
                }
                const int left = p.ctx_len - (t_begin + j) * BN - half * 32;
                if (j < TC && left < 32) gone |= left <= 0 ? ~0u : ~0u << left;   // past the end of the context
                if (gone) {
#pragma unroll
                    for (int c = 0; c < 32; ++c)
                        if ((gone >> c) & 1u) sc[c] = 0xff800000u;   // -inf
                }
                float mx4[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) mx4[c] = __uint_as_float(sc[c]);
#pragma unroll
                for (int c = 4; c < 32; c += 2) mx4[(c >> 1) & 3] = max3(mx4[(c >> 1) & 3], __uint_as_float(sc[c]), __uint_as_float(sc[c + 1]));
                const float mx = valid ? fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * sl2 : -INFINITY;
                float factor = 1.f;
                const bool raise = named_barrier_or(pair_bar, 64, mx > m_used + kRaise);
                if (raise) {   // the first tile, and rarely later: the two threads of a row agree on a larger reference
                    if (soft_row < rows_x) xch[half * rows_x + soft_row] = mx;
                    named_barrier(pair_bar, 64);
                    const float m_new = fmaxf(m_used, fmaxf(mx, xch[(1 - half) * rows_x + soft_row_x]));
                    factor = m_used == -INFINITY ? 0.f : fast_exp2(m_used - m_new);
                    m_used = m_new;
                }
                const float mneg = valid && m_used != -INFINITY ? -m_used : 0.f;   // (no key has counted yet: every d is -inf)
                const f32x2 mneg2 = pk(mneg, mneg);
                f32x2 sum2[2] = {pk(0.f, 0.f), pk(0.f, 0.f)};
                uint32_t pw[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const f32x2 d2 = fma2(pk(__uint_as_float(sc[2 * c]), __uint_as_float(sc[2 * c + 1])), sl2_2, mneg2);
                    float d0, d1;
                    upk(d2, d0, d1);
                    const float e0 = fast_exp2(d0), e1 = fast_exp2(d1);
                    sum2[c & 1] = add2(sum2[c & 1], pk(e0, e1));
                    pw[c] = pack_bf16x2(e0, e1);
                }
                float a0, a1, b0, b1;
                upk(sum2[0], a0, a1);
                upk(sum2[1], b0, b1);
                l_run = fmaf(l_run, factor, (a0 + a1) + (b0 + b1));   // this half's share of the row sum

                // P buffer free and O stable once P V of the previous tile has completed
                if (j > 0) mbar_wait(bar(B_PVDONE + t), (j - 1) & 1, abort_flag, p.dev_status);
                if (store_p) {
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch)
                        *reinterpret_cast<uint4*>(prow + (((half * 4 + ch) ^ (soft_row & 7)) << 4)) =
                            make_uint4(pw[4 * ch], pw[4 * ch + 1], pw[4 * ch + 2], pw[4 * ch + 3]);
                }
                if (raise && j > 0) {   // each of the two threads scales its 64 columns
                    fence_after();
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        uint32_t o[32];
                        ld32(tm_t + 128 + half * 64 + c * 32, o);
                        wait_ld<32>(o);
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * factor);
                        st32(tm_t + 128 + half * 64 + c * 32, o);
                    }
                    wait_st();
                }
                fence_async_smem();
                fence_before();
                mbar_arrive(bar(B_PFULL + t));
            }
            if (soft_row < rows_x) xch[half * rows_x + soft_row] = l_run;
            named_barrier(pair_bar, 64);
            l_run += xch[(1 - half) * rows_x + soft_row_x];
            // all row tiles have finished their last P V: Q, P and the K/V stages are dead from here on
#pragma unroll
            for (int tt = 0; tt < NT; ++tt) mbar_wait(bar(B_PVDONE + tt), (T - 1) & 1, abort_flag, p.dev_status);
            fence_after();

            const int r = t * BM + soft_row;
            if (C == 1) {
                // ---- single CTA per (sequence, kv head): normalise and store -------------------
                const int i = valid ? r / p.group : 0, jh = valid ? r % p.group : 0;
                __nv_bfloat16* dst = p.out + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + jh) * HD + half * 64;
                const float inv = 1.f / l_run;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float o[32];
                    ld32f(tm_t + 128 + half * 64 + c * 32, o);
                    if (valid && !*abort_flag) {   // a CTA whose wait gave up stores nothing
#pragma unroll
                        for (int v4 = 0; v4 < 4; ++v4) {
                            uint4 w;
                            w.x = pack_bf16x2(o[v4 * 8 + 0] * inv, o[v4 * 8 + 1] * inv);
                            w.y = pack_bf16x2(o[v4 * 8 + 2] * inv, o[v4 * 8 + 3] * inv);
                            w.z = pack_bf16x2(o[v4 * 8 + 4] * inv, o[v4 * 8 + 5] * inv);
                            w.w = pack_bf16x2(o[v4 * 8 + 6] * inv, o[v4 * 8 + 7] * inv);
                            *reinterpret_cast<uint4*>(dst + c * 32 + v4 * 8) = w;
                        }
                    }
                }
            } else {
                // ---- un-normalised row -> staging, grouped by owner (CTA r mod C) -----------------
                float* rec = reinterpret_cast<float*>(gbase) +
                             (valid ? ((r % C) * p.rows_per_cta + r / C) : 0) * kRec;   // staging reuses the dead Q/P/stage memory
#pragma unroll
                for (int c = half * 2; c < half * 2 + 2; ++c) {
                    float o[32];
                    ld32f(tm_t + 128 + c * 32, o);
                    if (valid) {
#pragma unroll
                        for (int v4 = 0; v4 < 8; ++v4)
                            *reinterpret_cast<float4*>(rec + c * 32 + v4 * 4) =
                                make_float4(o[v4 * 4], o[v4 * 4 + 1], o[v4 * 4 + 2], o[v4 * 4 + 3]);
                    }
                }
                if (valid && half == 0) *reinterpret_cast<float4*>(rec + HD) = make_float4(m_used, l_run, 0.f, 0.f);
                fence_async_smem();   // staging (generic proxy) -> bulk copies (async proxy)
            }
        }
    }

    if (C > 1) {
        // every CTA of the cluster is past its main loop (its Q, P and K/V stages are dead, its barriers
        // initialised) and has staged its rows
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        // one bulk copy per owner into the owner's receive buffer, issued by the first C lanes of warp 0
        if (warp == 0 && lane < C) {
            const int owner = lane;
            const int n_rows_owner = (p.rows_total - owner + C - 1) / C;
            if (n_rows_owner > 0) {
                const uint32_t src = base + (uint32_t)(owner * p.rows_per_cta * kRec) * 4u;
                const uint32_t dst = map_to_cta(base + p.off_recv + (uint32_t)(split * p.rows_per_cta * kRec) * 4u, owner);
                bulk_copy_to_peer(dst, src, (uint32_t)(n_rows_owner * kRec) * 4u, map_to_cta(bar(B_RECV), owner));
            }
        }
        // ---- merge the C partials of the rows this CTA owns ------------------------------------
        if (n_own > 0) {
            mbar_wait(bar(B_RECV), 0, abort_flag, p.dev_status);
            const float* recv = reinterpret_cast<const float*>(gbase + p.off_recv);
            for (int qi = warp; qi < n_own; qi += kThreads / 32) {
                const int r = split + qi * C;
                // lane s < C holds (m_s, l_s); the weights are shared through shuffles
                float ms = -INFINITY, ls = 0.f;
                if (lane < C) {
                    const float2 ml = *reinterpret_cast<const float2*>(recv + (lane * p.rows_per_cta + qi) * kRec + HD);
                    ms = ml.x;
                    ls = ml.y;
                }
                float m = ms;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                m = __shfl_sync(0xffffffffu, m, 0);
                const float ws = lane < C ? fast_exp2(ms - m) : 0.f;
                float l = ws * ls;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                l = __shfl_sync(0xffffffffu, l, 0);
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < kMaxCluster; ++s) {
                    if (s < C) {
                        const float w = __shfl_sync(0xffffffffu, ws, s);
                        const float4 o = *reinterpret_cast<const float4*>(recv + (s * p.rows_per_cta + qi) * kRec + lane * 4);
                        acc.x = fmaf(w, o.x, acc.x);
                        acc.y = fmaf(w, o.y, acc.y);
                        acc.z = fmaf(w, o.z, acc.z);
                        acc.w = fmaf(w, o.w, acc.w);
                    }
                }
                const int i = r / p.group, jh = r % p.group;
                __nv_bfloat16* dst = p.out + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + jh) * HD;
                const float inv = 1.f / l;
                uint2 w2;
                w2.x = pack_bf16x2(acc.x * inv, acc.y * inv);
                w2.y = pack_bf16x2(acc.z * inv, acc.w * inv);
                if (!*abort_flag) *reinterpret_cast<uint2*>(dst + lane * 4) = w2;   // nothing from a CTA whose wait gave up
            }
        }
        // no CTA leaves while a peer may still copy out of or into its shared memory
        __syncwarp();
        cluster_arrive();
        cluster_wait();
    }

    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TM_COLS) : "memory");
    }
}

// ---- host side ---------------------------------------------------------------------------
struct SkipPlan {
    int nt, rows_total, n_splits, tiles_per_split, n_stages, rows_per_cta, n_extra;
    bool keys_on_m;   // at most 64 packed rows and a CTA per kv head: see ec_skip_keys_pair.cuh
    uint32_t off_q[2], off_p[2], rows_pad[2], off_stage, off_recv, off_list, off_xch, off_bar, smem_bytes;
};

constexpr uint32_t kSmemTwoPerSm = 115712;   // (228 KB per SM - 2 x 1 KB reserved) / 2
constexpr uint32_t kSmemMax = 232448;        // 227 KB: largest dynamic allocation of one CTA

SkipPlan make_skip_plan(const ec_attn_desc& d, int n_active) {
    SkipPlan pl{};
    const int g = d.n_q_heads / d.n_kv_heads;
    pl.rows_total = n_active * g;
    pl.nt = pl.rows_total > BM ? 2 : 1;
    const int key_tiles = (d.ctx_len + BN - 1) / BN;
    const int bh = d.batch * d.n_kv_heads;
    const int slots = (pl.nt == 1 ? 2 : 1) * sm_count();   // co-resident CTAs
    int c = slots / bh;
    if (c < 1) c = 1;
    if (c > kMaxCluster) c = kMaxCluster;
    if (c > key_tiles) c = key_tiles;
    pl.tiles_per_split = (key_tiles + c - 1) / c;
    pl.n_splits = (key_tiles + pl.tiles_per_split - 1) / pl.tiles_per_split;
    pl.rows_per_cta = (pl.rows_total + pl.n_splits - 1) / pl.n_splits;
    pl.n_extra = (n_active + BN - 1) / BN;
    uint32_t off = 0;
    for (int t = 0; t < 2; ++t) {
        const int rows_t = t < pl.nt ? (pl.rows_total - t * BM < BM ? pl.rows_total - t * BM : BM) : 0;
        pl.rows_pad[t] = (uint32_t)((rows_t + 7) / 8 * 8);
        pl.off_q[t] = off;
        off += pl.rows_pad[t] * 256u;
    }
    for (int t = 0; t < 2; ++t) {
        pl.off_p[t] = off;
        off += pl.rows_pad[t] * 128u;
    }
    pl.off_stage = off;   // multiple of 1024: every piece above is a multiple of 8 rows x 128 bytes
    // the exchange areas (staging, then receive buffer) reuse the memory below the list once the main loop is over
    const uint32_t recv = pl.n_splits > 1 ? (uint32_t)(pl.n_splits * pl.rows_per_cta * kRec * 4) : 0u;
    const uint32_t list = ((uint32_t)(pl.tiles_per_split + pl.n_extra) * 8u + 15u) & ~15u;   // key masks
    const uint32_t xch = (pl.rows_pad[0] + pl.rows_pad[1]) * 8u;   // two floats per row
    const uint32_t tail = list + xch + B_COUNT * 8u + 32u;   // + barrier block
    int ns = 0;
    if (pl.nt == 1) {   // two CTAs per SM when at least two stages fit in half an SM
        ns = off + tail < kSmemTwoPerSm ? (int)((kSmemTwoPerSm - off - tail) / STAGE) : 0;
        if (ns > 3) ns = 3;
    }
    if (ns < 2) {
        ns = off + tail < kSmemMax ? (int)((kSmemMax - off - tail) / STAGE) : 0;
        if (ns > kMaxStages) ns = kMaxStages;
    }
    const int visits = pl.tiles_per_split + pl.n_extra;
    if (ns > visits && ns > 2) ns = visits < 2 ? 2 : visits;
    pl.n_stages = ns;
    off += (uint32_t)ns * STAGE;
    pl.off_recv = recv;   // right behind the staging area, which starts at 0
    pl.off_list = off;
    off += list;
    pl.off_xch = off;
    off += xch;
    pl.off_bar = off;
    off += B_COUNT * 8u + 32u;
    pl.smem_bytes = off;
    // With at least a CTA per kv head and SM in flight, what counts is the time of a key tile; with fewer heads the keys
    // are split over a cluster, which needs the merge of this kernel.
    pl.keys_on_m = pl.nt == 1 && pl.n_splits == 1 && pl.rows_total <= keys_pair::kMaxSlots &&
                   keys_pair::smem_bytes(pl.rows_total, d.ctx_len) <= kSmemTwoPerSm;
    if (pl.keys_on_m) pl.smem_bytes = keys_pair::smem_bytes(pl.rows_total, d.ctx_len);
    return pl;
}

template <int NT>
cudaError_t launch_nt(const SkipPlan& pl, const SkipParams& p, const CUtensorMap& mk, const CUtensorMap& mv,
                      const CUtensorMap& mkn, const CUtensorMap& mvn, const keys_pair::Params& kp, int bh,
                      cudaStream_t stream) {
    static PerDeviceOnce attr_once;
    if (const cudaError_t ea = ensure_dynamic_smem(attr_once, attend_skip_kernel<NT>, (int)kSmemMax); ea != cudaSuccess) return ea;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(pl.n_splits, bh, 1);
    cfg.blockDim = dim3(64 + NT * 256, 1, 1);
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
    return cudaLaunchKernelEx(&cfg, attend_skip_kernel<NT>, mk, mv, mkn, mvn, p, kp);
}

}  // namespace

bool attend_skip_supported(const ec_attn_desc& d, int n_active) {
    if (d.dtype != EC_BF16 || d.head_dim != HD || n_active < 1) return false;
    const long long rows = (long long)n_active * (d.n_q_heads / d.n_kv_heads);
    if (rows > kMaxRows) return false;
    if ((long long)d.batch * d.n_kv_heads > 65535) return false;                       // grid.y
    const SkipPlan pl = make_skip_plan(d, n_active);
    const size_t exchange = pl.n_splits > 1 ? 2 * (size_t)pl.n_splits * pl.rows_per_cta * kRec * 4 : 0;
    return pl.n_stages >= 2 && pl.smem_bytes <= kSmemMax && exchange <= pl.off_list;
}

void attend_skip_describe(const ec_attn_desc& d, int n_active, char* buf, size_t len) {
    const SkipPlan pl = make_skip_plan(d, n_active);
    snprintf(buf, len, "attend_skip_kernel<%d> grid=(%d,%d) cluster=%d stages=%d smem=%u%s", pl.nt, pl.n_splits,
             d.batch * d.n_kv_heads, pl.n_splits, pl.keys_on_m ? 1 : pl.n_stages, pl.smem_bytes,
             pl.keys_on_m ? " keys_on_m" : "");
}

cudaError_t launch_attend_skip(const AttendArgs& a, const void* k_new, const void* v_new, const int32_t* active_idx,
                               cudaStream_t stream) {
    const SkipPlan pl = make_skip_plan(a.d, a.n_active);
    const int bh = a.d.batch * a.d.n_kv_heads;
    CUtensorMap map_k, map_v;
    const int box = pl.keys_on_m ? keys_pair::BK : BN;
    if (!make_cache_map(&map_k, a.k_cache, bh, a.d.ctx_len, box) || !make_cache_map(&map_v, a.v_cache, bh, a.d.ctx_len, box))
        return cudaErrorInvalidValue;
    CUtensorMap map_kn = map_k, map_vn = map_v;   // placeholders unless refreshing
    if (k_new && (!make_fresh_map(&map_kn, k_new, a.d.batch, a.n_active, a.d.n_kv_heads, box) ||
                  !make_fresh_map(&map_vn, v_new, a.d.batch, a.n_active, a.d.n_kv_heads, box)))
        return cudaErrorInvalidValue;
    SkipParams p{};
    p.n_extra = pl.n_extra;
    p.early_cache = (a.d.flags & EC_ATTN_CACHE_SETTLED) ? 1 : 0;
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
    p.group = a.d.n_q_heads / a.d.n_kv_heads;
    p.rows_total = pl.rows_total;
    p.n_splits = pl.n_splits;
    p.tiles_per_split = pl.tiles_per_split;
    p.n_stages = pl.n_stages;
    p.rows_per_cta = pl.rows_per_cta;
    for (int t = 0; t < 2; ++t) {
        p.off_q[t] = pl.off_q[t];
        p.off_p[t] = pl.off_p[t];
        p.rows_pad[t] = pl.rows_pad[t];
    }
    p.off_stage = pl.off_stage;
    p.off_recv = pl.off_recv;
    p.off_list = pl.off_list;
    p.off_xch = pl.off_xch;
    p.off_bar = pl.off_bar;
    p.scale_log2 = a.scale * kLog2e;
    p.keys_on_m = pl.keys_on_m ? 1 : 0;
    const keys_pair::Params kp{p.q, p.k_new, p.v_new, p.k_cache, p.v_cache, p.active_idx, p.out, p.dev_status, p.n_active,
                               p.ctx_len, p.n_q_heads, p.n_kv_heads, p.group, (65536 + p.group - 1) / p.group,
                               p.early_cache, p.scale_log2};
    return pl.nt == 1 ? launch_nt<1>(pl, p, map_k, map_v, map_kn, map_vn, kp, bh, stream)
                      : launch_nt<2>(pl, p, map_k, map_v, map_kn, map_vn, kp, bh, stream);
}

}  // namespace ec
