// ec_attend, recompute step and other dense cases (bf16; head_dim 128 with more than 256 packed query rows per
// kv head, head_dim 64 where that is faster than mma.sync, see prefers_mma): bidirectional attention of every active row over
// the whole cache on the Blackwell tensor cores (Appendix A of the paper, full branch; Algorithm 1 FullPrefill /
// FullRecompute).  What follows describes 128-wide heads; with 64 columns every tile is half as large, and O_t has 64 columns.
//
// The step is bound by the tensor pipe and, next to it, by the exponentials of the softmax.  One CTA owns
// TWO 128-row tiles of the packed (active row x query heads of one kv head) axis and walks over all
// 128-key tiles of that kv head; while the softmax of one row tile runs, the tensor core works for the other.
//   warp 0      TMA producer: K and V tiles ([128 keys x 128] bf16, one 4-D box each: [2 halves][128 keys]
//               [64 columns], 128-byte swizzle) through a ring of five 32 KB slots (K0 V0 K1 V1 ...), and the
//               two Q tiles of the unit, one box each.  (Grouped-query shapes are launched with one unit per
//               QUERY head, so a row tile is always 128 active rows of one head; the query heads of a kv head
//               stream the same K/V, which L2 serves.)
//   warp 1      tcgen05.mma issuer (the whole warp, one lane elected): S_t = Q_t K^T (both operands K-major in shared memory) into
//               the TMEM columns of row tile t, and O_t += P_t V with P_t read from TENSOR MEMORY (it
//               overwrites the first 64 columns of S_t as packed bf16) and V MN-major from shared memory.
//               Order per key tile j:  P V_0(j), S_0(j+1), P V_1(j), S_1(j+1): the pipe executes in order,
//               so S_t(j+1) cannot overwrite P_t(j) before P V_t(j) has read it;
//   warps 2..17 softmax, four warpgroups: (row tile 0 / 1) x (keys 0..63 / 64..127 of the tile).  A query row
//               (= TMEM lane) is shared by two threads in warps that own the same lanes; each does
//               tcgen05.ld of its 64 scores, exp2 with the scale folded in (packed fp32x2 FMA), its share of
//               the row sum, P rounded to bf16 and stored back with tcgen05.st.  There is no running maximum:
//               a row's reference is its largest score among the first eight keys, and only if a row sum
//               leaves the range that fp32 and bf16 share is the unit done again, with running maxima.  Halving
//               the per-thread row shortens the softmax that sits between two uses of the tensor pipe for the
//               same row tile.
//   warp 18     recompute steps only: every cache row is overwritten by the fresh row of the same position, so the
//               launch reads K/V straight from the token-major k_new / v_new (only the tensor map's strides
//               differ) and this warp stores landed tiles into the cache meanwhile: no separate refresh pass.
// TMEM (512 columns): S_0 [0,128), S_1 [128,256), O_0 [256,384), O_1 [384,512).
// Shared memory: Q_0, Q_1 (32 KB each, staged once), five 32 KB K/V slots, barriers: 225 KB, one CTA per SM.
// Every mbarrier wait is bounded; a wait that runs out sets EC_ERR_TIMEOUT in the caller's dev_status word and
// a CTA-wide abort flag that makes all later waits fall through; the CTA still frees its TMEM and exits.
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

#include <atomic>
#include <cstdio>

namespace ec {
namespace {

using namespace tc;

constexpr int BM = 128, BN = 128;
constexpr int kSoftThreads = 512;          // four softmax warpgroups: (row tile) x (64-column half)
constexpr int kThreads = 64 + kSoftThreads + 32;   // + one warp that copies fresh K/V into the cache (recompute steps)
constexpr uint32_t SUB = 128 * 128;        // [128 rows x 64 bf16], 128-byte swizzle: 16 KB
constexpr int kSlots = 5;
// shared memory for heads of HD = 64 or 128 columns
template <int HD>
struct Geo {
    static constexpr uint32_t TILE = HD / 64 * SUB;             // [128 x HD] bf16
    static constexpr uint32_t OFF_Q = 0;                        // two tiles
    static constexpr uint32_t OFF_RING = 2 * TILE;
    static constexpr uint32_t OFF_BAR = OFF_RING + kSlots * TILE;   // 224 KB or 112 KB
    static constexpr uint32_t OFF_XCH = OFF_BAR + 256;          // [2 tiles][2 halves][128 rows] floats
    static constexpr uint32_t NEEDED = OFF_XCH + 2 * 2 * BM * 4;
    static constexpr uint32_t BYTES = HD == 128 ? 232448 : NEEDED + 1024;   // all of a CTA's 227 KB; the rest is alignment slack
    static constexpr uint32_t PART = BM * HD * 4;               // un-normalised rows of a row tile (cut units), over the ring
    // (two CTAs never share an SM: they would have 1216 threads of 96 registers)
};
constexpr uint32_t TM_COLS = 512;
constexpr uint32_t TM_S = 0, TM_O = 256;   // + 128 * tile

// B_FREE: ring entries are released in groups, K_0, then {V_0, K_1}, {V_1, K_2}, ... (a second pass goes on: {V of the last
// tile, K_0}); group c completes phase c / 3 of barrier c % 3, by the products' commit and the copy warp.  Three barriers: the
// copy warp, which needs no product, walks through the first five entries, groups 0 to 2, at once; its arrival for group
// c + 3, entry 2 c + 6, waits for group c + 1, and so for the commit of group c.
// B_PFULL: + 2 * part + tile, see the softmax.
enum { B_FULL = 0, B_FREE = kSlots, B_SFULL = B_FREE + 3, B_PFULL = B_SFULL + 2, B_PVDONE = B_PFULL + 4,
       B_QFULL = B_PVDONE + 2, B_VERDICT = B_QFULL + 2, B_COPIED = B_VERDICT + 1, B_COUNT = B_COPIED + 1 };

// first pass: a row's sum may grow to this before the unit is done again with running maxima
constexpr float kMaxSum = 1.152921504606846976e18f;   // 2^60

struct DenseParams {
    __nv_bfloat16* out;
    // recompute step: the K/V this launch reads are the token-major fresh tensors [B, L, Hkv, 128]; its copy warp
    // stores their tiles into the caches [B, Hkv, L, 128]
    int copy;
    int32_t* dev_status;
    int n_active, ctx_len, n_q_heads, n_kv_heads, rows_total;
    // Grouped-query shapes run with one unit per QUERY head (the kernel's n_kv_heads is H_q, so its row tiles are 128
    // active rows of one head and come by TMA); the K/V of unit head h are those of the real kv head h / kv_div.
    int kv_div;
    float scale_log2;
    // Unit order = row-tile pair fastest, then head.  The first n_full units are whole; each later one (what would be
    // the last, partial wave of the launch) is cut along the keys into `split` CTAs, a cluster of the second launch.
    int n_pairs, n_full, split;
    int wait_first;   // second launch: 1 when there is no first one, see below
};

// First key tile of part i of a unit whose T key tiles are cut into s parts.  Every part holds T / s tiles and the first
// T % s parts one more, so none is empty while T >= s; the longest is no longer than with parts of ceil(T / s) tiles, the
// last of which start behind the last tile at T = 33 and s = 8, for instance.  The last part, which has the ragged tile to
// mask, is one of the short ones, and the division is one of 32 bits (1349 keys, 32 heads, 11 tiles in two parts: 49.6 us a
// layer; 49.9 with T * i / s in 64 bits, which also leaves the long part last).
__host__ __device__ constexpr int part_begin(int T, int s, int i) { return i * (T / s) + (i < T % s ? i : T % s); }

// kCut: the launch of the cut units.  A cluster leaves its un-normalised rows, m and l in shared memory, each CTA merges a
// share of them out of its peers'.  This launch follows the one of the whole units with programmatic serialisation and
// does NOT wait for it: every CTA of the first launch triggers after its own dependency wait, so whatever wrote q, k_new
// and v_new is complete by then, and the two launches write different rows.  It waits at its end instead, so that whoever
// waits for this launch has waited for both.  Measured, layers back to back (a third launch that combined partials from
// global memory -> merged here): 86.4 -> 78.5 us at 2 x 1531 with 28 heads, 237.5 -> 233.1 at 4096 with 28 heads,
// 58.0 -> 55.7 at 2048 with 19.
template <bool kCut, int HD>
__global__ void __launch_bounds__(kThreads, 1)
attend_dense_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_kd,
                    const __grid_constant__ CUtensorMap map_vd, const DenseParams p) {
    constexpr uint32_t TILE = Geo<HD>::TILE, OFF_Q = Geo<HD>::OFF_Q, OFF_RING = Geo<HD>::OFF_RING, OFF_BAR = Geo<HD>::OFF_BAR,
                       OFF_XCH = Geo<HD>::OFF_XCH, PART = Geo<HD>::PART;
    constexpr int CW = HD / 2, CH = CW / 8;   // output columns of a softmax thread, their 16-byte pieces as bf16
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = (s2u(smem_raw) + 1023u) & ~1023u;
    unsigned char* gbase = smem_raw + (base - s2u(smem_raw));
    const uint32_t bars = base + OFF_BAR;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + OFF_BAR + B_COUNT * 8);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + OFF_BAR + B_COUNT * 8 + 4);
    volatile int* again = reinterpret_cast<volatile int*>(gbase + OFF_BAR + B_COUNT * 8 + 8);   // verdict of the first pass
    float* xch = reinterpret_cast<float*>(gbase + OFF_XCH);
    auto bar = [&](int idx) { return bars + idx * 8; };
    if (base - s2u(smem_raw) + Geo<HD>::NEEDED > Geo<HD>::BYTES) {   // never with the 1024-byte alignment the runtime gives
        if (threadIdx.x == 0 && p.dev_status) atomicExch(p.dev_status, (int)EC_ERR_CUDA);
        return;
    }

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int lin = blockIdx.x;
    const int unit = kCut ? p.n_full + lin / p.split : lin;
    const int part = kCut ? lin % p.split : 0;
    const int pair = unit % p.n_pairs, bh = unit / p.n_pairs;
    const int b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads, hk_kv = hk / p.kv_div;
    const int r_pair = pair * 2 * BM;
    const int n_tiles_q = (p.rows_total - r_pair > BM) ? 2 : 1;   // row tiles of this CTA that hold rows
    const int T_all = (p.ctx_len + BN - 1) / BN;
    const int j0 = kCut ? part_begin(T_all, p.split, part) : 0;                  // first key tile of this CTA
    const int T = (kCut ? part_begin(T_all, p.split, part + 1) : T_all) - j0;    // >= 4 in a cut unit, see make_dense_plan

    if (tid == 0) {
        prefetch_map(&map_k);
        prefetch_map(&map_q);
        prefetch_map(&map_v);
        if (p.copy) {
            prefetch_map(&map_kd);
            prefetch_map(&map_vd);
        }
        for (int i = 0; i < B_COUNT; ++i)
            mbar_init(bar(i), (i >= B_PFULL && i < B_PFULL + 4) ? 256u : (p.copy && i >= B_FREE && i < B_FREE + 3) ? 2u : 1u);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s2u(tmem_slot)), "r"(TM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        fence_before();
    }
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    if (!kCut || p.wait_first) pdl_wait();   // the previous kernel of the stream has completed; global memory may be touched
    pdl_launch_dependents();

    if (warp == 0) {
        // ================================ TMA producer ======================================
        const bool elected = elect_one();   // (the whole warp: 521 -> 515 us a pass of 32 layers of 768)
        // Q: [half][row][64 columns] per row tile; rows past n_active read as zero
        auto load_q = [&](int t) {
            if (elected) {
                mbar_expect_tx(bar(B_QFULL + t), TILE);
                tma_load_5d(base + OFF_Q + t * TILE, &map_q, 0, r_pair + t * BM, hk, 0, b, bar(B_QFULL + t));
            }
        };
        load_q(0);   // the first scores need one row tile of Q and the first K tile
        int slot = 0, key = j0 * BN, group = 0;   // group: of the entry that had the slot before
        uint32_t turn = 0;
        for (int n = 0; n < 4 * T; ++n) {   // ring entry: K_j = 2j, V_j = 2j + 1; from 2T on the second pass
            if (n == 2 * T) {
                mbar_wait_warp(bar(B_VERDICT), 0, abort_flag, p.dev_status);
                if (!*again) break;
                key = j0 * BN;
            }
            if (n > kSlots && !(n & 1) && ++group == 3) group = 0, turn ^= 1;   // (five slots: entry n - 5 starts a group where n is even)
            if (n >= kSlots) mbar_wait_warp(bar(B_FREE + group), turn, abort_flag, p.dev_status);
            if (elected) {
                mbar_expect_tx(bar(B_FULL + slot), TILE);
                tma_load_5d(base + OFF_RING + slot * TILE, (n & 1) ? &map_v : &map_k, 0, key, 0, hk_kv, b, bar(B_FULL + slot));
            }
            if (n & 1) key += BN;
            if (++slot == kSlots) slot = 0;
            if (n == 0 && n_tiles_q > 1) load_q(1);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================================ MMA issuer ========================================
        // (the whole warp, see elect_one: with one thread this role took 3400 cycles a key tile and set the pace)
        const bool elected = elect_one();
        constexpr uint32_t IDESC_S = instr_desc(BN, 0), IDESC_PV = instr_desc(HD, 1);
        const uint64_t desc_q = smem_desc(base + OFF_Q, 16, 1024);
        auto products_s = [&](int t, uint64_t desc_k, int k0, int k1) {
            if (elected) {
#pragma unroll
                for (int k = k0; k < k1; ++k) {
                    const uint32_t koff = ((k >> 2) * SUB + (k & 3) * 32) / 16;
                    mma_ss(tmem + TM_S + t * 128, desc_q + t * (TILE / 16) + koff, desc_k + koff, IDESC_S, k > 0);
                }
            }
        };
        int slot = 0, group = 0;   // ring slot and phase of the next tile in the order K_0 V_0 K_1 V_1 ...; the next group to release
        uint32_t phase = 0, p_phase = 0;
        auto full = [&](int ahead) {   // has the ring entry `ahead` behind the next one landed?
            const bool wrapped = slot + ahead >= kSlots;
            return mbar_test(bar(B_FULL + slot + ahead - (wrapped ? kSlots : 0)), phase ^ (wrapped ? 1u : 0u));
        };
        auto take = [&](bool landed) {
            if (!landed) mbar_wait_warp(bar(B_FULL + slot), phase, abort_flag, p.dev_status);
            const int s = slot;
            if (++slot == kSlots) slot = 0, phase ^= 1;
            return s;
        };
        auto release = [&]() {
            if (elected) commit(bar(B_FREE + group));
            if (++group == 3) group = 0;
        };
        constexpr int kPeek = HD / 16 - 2;
        for (int pass = 0; pass < 2; ++pass) {
            if (pass == 1) {
                mbar_wait_warp(bar(B_VERDICT), 0, abort_flag, p.dev_status);
                if (!*again) break;
            }
            {
                const uint64_t desc_k = smem_desc(base + OFF_RING + take(false) * TILE, 16, 1024);
                for (int t = 0; t < n_tiles_q; ++t) {
                    mbar_wait_warp(bar(B_QFULL + t), 0, abort_flag, p.dev_status);
                    fence_after();
                    products_s(t, desc_k, 0, HD / 16);
                    if (elected) commit(bar(B_SFULL + t));
                }
                release();
            }
            // The pipe holds about three instructions behind the one that runs; an issuer that comes back from a barrier
            // later than that leaves it idle.  So the barriers of the next products are looked at while the last two
            // products of a group are still to be issued, and only what was not ready then is waited for.
            bool kv_ready = false, p_ready = false;
            for (int j = 0; j < T; ++j, p_phase ^= 1) {
                const bool more = j + 1 < T, more2 = j + 2 < T;
                const uint64_t desc_v = smem_desc(base + OFF_RING + take(kv_ready) * TILE, SUB, 1024);
                const uint64_t desc_k = smem_desc(base + OFF_RING + (more ? take(kv_ready) : 0) * TILE, 16, 1024);
                for (int t = 0; t < n_tiles_q; ++t) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (q == 1 || !p_ready) mbar_wait_warp(bar(B_PFULL + q * 2 + t), p_phase, abort_flag, p.dev_status);
                        fence_after();
                        // P of keys 0..63 lies over S columns 0..31, of keys 64..127 over S columns 64..95; part 0 are the first
                        // 48 keys of each half, part 1 the others
                        if (elected) {
#pragma unroll
                            for (int i = 0; i < (q ? 2 : 6); ++i) {
                                const int k = q ? i * 4 + 3 : (i / 3) * 4 + i % 3;
                                mma_ts(tmem + TM_O + t * HD, tmem + TM_S + t * 128 + (k >> 2) * 64 + (k & 3) * 8, desc_v + k * 128,
                                       IDESC_PV, (j > 0 || k > 0));
                            }
                        }
                    }
                    p_ready = false;
                    if (more) {
                        products_s(t, desc_k, 0, kPeek);
                        const bool next_tile = t + 1 == n_tiles_q;
                        const bool p_seen = mbar_test(bar(B_PFULL + (next_tile ? 0 : t + 1)), p_phase ^ (next_tile ? 1u : 0u));
                        if (t == 0) kv_ready = __all_sync(0xffffffffu, full(0) && (!more2 || full(1)));
                        p_ready = __all_sync(0xffffffffu, p_seen);
                        products_s(t, desc_k, kPeek, HD / 16);
                        if (elected) commit(bar(B_SFULL + t));
                    }
                    if (elected && (pass == 1 || !more)) commit(bar(B_PVDONE + t));
                }
                if (more) release();   // (the last V tile goes with the K_0 of a second pass)
            }
        }
        __syncwarp();
    } else if (warp < 2 + kSoftThreads / 32) {
        // ================================ softmax (warps 2..17) ================================
        // A row of a tile is shared by two threads, one per 64-column half, in warps that own the same TMEM
        // lanes: softmax warp ws = warp - 2 -> row tile ws / 8, column half (ws / 4) % 2, lanes 32 * (warp % 4).
        const int ws = warp - 2;
        const int t = ws >> 3, h = (ws >> 2) & 1;
        const int quarter = warp & 3;
        const int row = quarter * 32 + lane;        // row of the tile == TMEM lane
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const uint32_t tm_s = tmem + lane_addr + TM_S + t * 128;
        const uint32_t tm_o = tmem + lane_addr + TM_O + t * HD;
        float* xch_mine = xch + (t * 2 + h) * BM + row;        // exchanged with the partner thread of the row
        const float* xch_other = xch + (t * 2 + (1 - h)) * BM + row;
        const int pair_bar = 1 + t * 4 + quarter;              // named barrier of the two warps that share these rows
        if (t < n_tiles_q) {
            float m_used = -INFINITY, l_run = 0.f;
            const float sl2 = p.scale_log2;
            const f32x2 sl2_2 = pk(sl2, sl2);
            // ---- first pass: no running maximum.  The reference of a row is its largest score among the first eight keys
            //      (both threads of the row read those), so a thread needs nothing from its partner and nothing is
            //      reduced: probabilities may exceed 1 by what fp32 and bf16 exponents have room for, and the row sum
            //      tells at the end whether they stayed within it. ----
            {
                f32x2 mneg2 = pk(0.f, 0.f), sum2[2] = {pk(0.f, 0.f), pk(0.f, 0.f)};
                for (int j = 0; j < T; ++j) {
                    mbar_wait(bar(B_SFULL + t), j & 1, abort_flag, p.dev_status);
                    fence_after();
                    if (j == 0) {
                        uint32_t r8[8];
                        ld8(tm_s, r8);
                        wait_ld<8>(r8);
                        float mx = __uint_as_float(r8[0]);
#pragma unroll
                        for (int c = 1; c < 8; ++c)
                            if (j0 * BN + c < p.ctx_len) mx = fmaxf(mx, __uint_as_float(r8[c]));
                        m_used = mx * sl2;
                        mneg2 = pk(-m_used, -m_used);
                        named_barrier(pair_bar, 64);   // both threads of the row have read what P is about to overwrite
                    }
                    // P goes out in two parts, 48 columns and 16, so that three quarters of P V run while the rest is worked out:
                    // the chain of a row tile, scores - softmax - P V - scores, is what the other row tile has to cover.
                    // us a pass of 32 layers of 768 / 14 of 2 x 1531 (28 heads) / 2 of 8 x 4096 (at 1.5 GHz under the power
                    // cap): one part 530 / 1081 / 3910, halves 518 / 1055 / 3798, three quarters 516 / 1045 / 3726.
                    uint32_t sr[2][32];
                    ld32(tm_s + h * 64, sr[0]);
                    wait_ld<32>(sr[0]);
                    ld32(tm_s + h * 64 + 32, sr[1]);   // on its way while the first 32 scores are worked on
                    const int key0 = (j0 + j) * BN + h * 64;
                    const bool ragged = key0 + 64 > p.ctx_len;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if (q == 1) wait_ld<32>(sr[1]);
                        if (ragged) {
#pragma unroll
                            for (int c = 0; c < 32; ++c)
                                if (key0 + q * 32 + c >= p.ctx_len) sr[q][c] = 0xff800000u;   // -inf
                        }
                        uint32_t pw[16];
#pragma unroll
                        for (int c = 0; c < 16; ++c) {
                            const f32x2 d2 = fma2(pk(__uint_as_float(sr[q][2 * c]), __uint_as_float(sr[q][2 * c + 1])), sl2_2, mneg2);
                            float d0, d1;
                            upk(d2, d0, d1);
                            const float e0 = fast_exp2(d0), e1 = fast_exp2(d1);
                            sum2[c & 1] = add2(sum2[c & 1], pk(e0, e1));
                            pw[c] = pack_bf16x2(e0, e1);
                            if (q == 1 && c == 7) {
                                st8(tm_s + h * 64 + 16, pw);
                                wait_st();
                                fence_before();
                                mbar_arrive(bar(B_PFULL + t));
                            }
                        }
                        // (bf16 pairs over the first half of this thread's own scores)
                        if (q == 0) {
                            st16(tm_s + h * 64, pw);
                        } else {
                            st8(tm_s + h * 64 + 24, pw + 8);
                            wait_st();
                            fence_before();
                            mbar_arrive(bar(B_PFULL + 2 + t));
                        }
                    }
                }
                float a0, a1, b0, b1;
                upk(sum2[0], a0, a1);
                upk(sum2[1], b0, b1);
                l_run = (a0 + a1) + (b0 + b1);   // this half's share of the row sum
            }
            const bool redo = named_barrier_or(9, n_tiles_q * 256, !(l_run <= kMaxSum));
            if (ws == 0 && lane == 0) {
                *again = redo ? 1 : 0;
                mbar_arrive(bar(B_VERDICT));
            }
            // ---- second pass, only if a score left the first one's range: running maxima.  The unit is done twice: with
            //      scores of standard deviation 4 (nats) no unit takes it, with 8 some do and with 12 all (L = 768 19.0,
            //      22.4, 33.1 us a layer; 4096 255, 290, 505) ----
            if (redo) {
                m_used = -INFINITY;
                l_run = 0.f;
            }
            // B_PVDONE: one phase at the end of the first pass, one per key tile of the second
            const uint32_t last = redo ? T & 1 : 0;
            for (int j = 0; redo && j < T; ++j) {
                mbar_wait(bar(B_SFULL + t), (T + j) & 1, abort_flag, p.dev_status);
                fence_after();
                uint32_t sr[BN / 2];
                ld32(tm_s + h * 64, sr);
                ld32(tm_s + h * 64 + 32, sr + 32);
                wait_ld<64>(sr);
                const int key0 = (j0 + j) * BN + h * 64;
                if (key0 + 64 > p.ctx_len) {
#pragma unroll
                    for (int c = 0; c < 64; ++c)
                        if (key0 + c >= p.ctx_len) sr[c] = 0xff800000u;   // -inf
                }
                float mx[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) mx[c] = __uint_as_float(sr[c]);
#pragma unroll
                for (int c = 4; c < 64; c += 2) mx[(c >> 1) & 3] = max3(mx[(c >> 1) & 3], __uint_as_float(sr[c]), __uint_as_float(sr[c + 1]));
                const float mloc = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                *xch_mine = mloc;
                named_barrier(pair_bar, 64);   // both halves of the row have loaded their scores and posted their maxima
                const float m_tile = fmaxf(mloc, *xch_other) * sl2;
                float factor = 1.f;
                if (m_tile > m_used + 8.f || m_used == -INFINITY) {   // stale maximum allowed up to 2^8
                    factor = (m_used == -INFINITY) ? 0.f : fast_exp2(m_used - m_tile);
                    m_used = m_tile;
                }
                const bool need_rescale = (j > 0) && __any_sync(0xffffffffu, factor != 1.f);
                const f32x2 mneg2 = pk(-m_used, -m_used);
                f32x2 sum2[2] = {pk(0.f, 0.f), pk(0.f, 0.f)};
                uint32_t pw[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const f32x2 d2 = fma2(pk(__uint_as_float(sr[2 * c]), __uint_as_float(sr[2 * c + 1])), sl2_2, mneg2);
                    float d0, d1;
                    upk(d2, d0, d1);
                    const float e0 = fast_exp2(d0), e1 = fast_exp2(d1);
                    sum2[c & 1] = add2(sum2[c & 1], pk(e0, e1));
                    pw[c] = pack_bf16x2(e0, e1);
                }
                {
                    float a0, a1, b0, b1;
                    upk(sum2[0], a0, a1);
                    upk(sum2[1], b0, b1);
                    l_run = fmaf(l_run, factor, (a0 + a1) + (b0 + b1));   // this half's share of the row sum
                }
                if (need_rescale) {
                    // O holds tiles < j: P V of tile j - 1 must have completed before the accumulator is scaled;
                    // each of the two threads of a row scales its half of the columns
                    mbar_wait(bar(B_PVDONE + t), j & 1, abort_flag, p.dev_status);
                    fence_after();
#pragma unroll
                    for (int c = 0; c < CW / 32; ++c) {
                        uint32_t o[32];
                        ld32(tm_o + h * CW + c * 32, o);
                        wait_ld<32>(o);
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * factor);
                        st32(tm_o + h * CW + c * 32, o);
                    }
                }
                // P (bf16 pairs) over the first half of this thread's own scores
                st32(tm_s + h * 64, pw);
                wait_st();
                fence_before();
                mbar_arrive(bar(B_PFULL + t));
                mbar_arrive(bar(B_PFULL + 2 + t));
            }

            // ---- epilogue ------------------------------------------------------------------------
            mbar_wait(bar(B_PVDONE + t), last, abort_flag, p.dev_status);
            fence_after();
            *xch_mine = l_run;
            named_barrier(pair_bar, 64);
            const float l_row = l_run + *xch_other;   // both halves of a row carry the same reference maximum
            if constexpr (!kCut) {
                // Whole unit: the normalised row goes to shared memory, over the row tile's Q (its last scores are long
                // formed), and from there, a warp its own 32 rows and half of the columns, to global memory in pieces of 128 or 64
                // bytes.
                // (us a pass of 32 layers of 768: by TMA, a box for each row tile 510.4, for each warp 507.5; like this, with
                // no copy to wait for, 503.4.  Straight from the registers, a thread 128 bytes of its row: 3.5 us a unit.)
                // Rolled: the code of an epilogue runs once a unit and is fetched at about its own length in time.
                const float inv = 1.f / l_row;
                unsigned char* qtile = gbase + OFF_Q + t * TILE;
                auto piece = [&](int rw, int g) {   // piece g of the HD / 8 of a row: 128-byte swizzle, so that 32 lanes spread
                    return reinterpret_cast<uint4*>(qtile + (g >> 3) * SUB + (rw >> 3) * 1024 + (rw & 7) * 128 + (((g & 7) ^ (rw & 7)) << 4));
                };
#pragma unroll 1
                for (int c = 0; c < CW / 32; ++c) {
                    uint32_t o[32];
                    ld32(tm_o + h * CW + c * 32, o);
                    wait_ld<32>(o);
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        uint4 w;
                        w.x = pack_bf16x2(__uint_as_float(o[v4 * 8 + 0]) * inv, __uint_as_float(o[v4 * 8 + 1]) * inv);
                        w.y = pack_bf16x2(__uint_as_float(o[v4 * 8 + 2]) * inv, __uint_as_float(o[v4 * 8 + 3]) * inv);
                        w.z = pack_bf16x2(__uint_as_float(o[v4 * 8 + 4]) * inv, __uint_as_float(o[v4 * 8 + 5]) * inv);
                        w.w = pack_bf16x2(__uint_as_float(o[v4 * 8 + 6]) * inv, __uint_as_float(o[v4 * 8 + 7]) * inv);
                        *piece(row, h * CH + c * 4 + v4) = w;
                    }
                }
                __syncwarp();
                if (!*abort_flag) {   // a CTA whose wait gave up stores nothing
                    constexpr int RW = 32 / CH;                 // rows at a time, CH lanes a row
                    const int g = lane / CH, ch = lane % CH;
                    const int r0 = r_pair + t * BM + quarter * 32 + g;
                    __nv_bfloat16* dst = p.out + (((long long)b * p.n_active + r0) * p.n_q_heads + hk) * HD + h * CW + ch * 8;
                    const long long step = (long long)RW * p.n_q_heads * HD;
#pragma unroll
                    for (int k = 0; k < CH; ++k) {
                        const uint4 w = *piece(quarter * 32 + k * RW + g, h * CH + ch);
                        if (r0 + k * RW < p.rows_total) *reinterpret_cast<uint4*>(dst + k * step) = w;
                    }
                }
            } else {
                // part of a cut unit: the un-normalised row (relative to m_used), m and l stay in shared memory, over the
                // ring and Q: both row tiles' products and the copy warp's stores have to be through
                for (int tt = 0; tt < n_tiles_q; ++tt) mbar_wait(bar(B_PVDONE + tt), last, abort_flag, p.dev_status);
                if (p.copy) mbar_wait(bar(B_COPIED), 0, abort_flag, p.dev_status);
                unsigned char* prow = gbase + OFF_RING + t * PART + row * (HD * 4);
#pragma unroll 1
                for (int c = 0; c < CW / 32; ++c) {
                    uint32_t o[32];
                    ld32(tm_o + h * CW + c * 32, o);
                    wait_ld<32>(o);
#pragma unroll
                    for (int v4 = 0; v4 < 8; ++v4)   // (16-byte pieces swizzled by row: 32 lanes are 32 rows)
                        *reinterpret_cast<uint4*>(prow + (((h * (HD / 8) + c * 8 + v4) ^ (row & (HD / 4 - 1))) << 4)) =
                            make_uint4(o[v4 * 4], o[v4 * 4 + 1], o[v4 * 4 + 2], o[v4 * 4 + 3]);
                }
                if (h == 0) *reinterpret_cast<float2*>(gbase + OFF_Q + (t * BM + row) * 8) = make_float2(m_used, l_row);
            }
        }
        fence_before();
    } else if (p.copy && lane == 0) {
        // ====================== copy warp: this CTA's share of the refresh ============================
        // The key tiles that stream through the ring ARE the fresh rows: those of this CTA's share go from shared memory to
        // the cache by TMA (the same box through the cache's map; rows past L are not written), so the cache update reads
        // nothing.  The units of a kv head (its query heads' row-tile pairs) take turns by tile.  Nobody reads the cache
        // in this launch.  (A warp that copied its share of the rows through registers took longer than the six key
        // tiles of a unit at L = 768.)
        const int n_share = p.n_pairs * p.kv_div, mine = (hk % p.kv_div) * p.n_pairs + pair;
        int slot = 0;
        uint32_t phase = 0;
        for (int n = 0; n < 4 * T; ++n) {   // (on a second pass the tiles only pass by)
            if (n == 2 * T) {
                mbar_wait(bar(B_VERDICT), 0, abort_flag, p.dev_status);
                if (!*again) break;
            }
            mbar_wait(bar(B_FULL + slot), phase, abort_flag, p.dev_status);
            const int j = j0 + (n >> 1);
            if (n < 2 * T && j % n_share == mine && !*abort_flag) {
                tma_store_5d((n & 1) ? &map_vd : &map_kd, base + OFF_RING + slot * TILE, 0, j * BN, 0, hk_kv, b);
                bulk_commit();
                bulk_wait_read();   // the slot has been read
            }
            if (!(n & 1)) mbar_arrive(bar(B_FREE + (n >> 1) % 3));   // K tiles end a group
            if (++slot == kSlots) slot = 0, phase ^= 1;
        }
        mbar_arrive(bar(B_COPIED));
    }

    if constexpr (kCut) {
        // ---- merge: this CTA's share of the cluster's rows, w_s = 2^(m_s - M) / sum_s 2^(m_s - M) l_s ----
        __syncwarp();
        cluster_arrive();
        cluster_wait();           // the partials of all CTAs are complete
        float* weight = reinterpret_cast<float*>(gbase + OFF_Q + 2 * BM * 8);   // [row of the share][8]
        const int rows = n_tiles_q * BM, per = ((rows + p.split - 1) / p.split + 3) & ~3, row0 = part * per;   // whole groups of four
        const int share = min(per, rows - row0);
        for (int i = tid; i < share; i += kThreads) {
            float mm[8], ll[8], M = -INFINITY, L = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                ld_peer_v2(map_to_cta(base + OFF_Q + (row0 + i) * 8, min(q, p.split - 1)), mm[q], ll[q]);
                if (q >= p.split) mm[q] = -INFINITY;
                M = fmaxf(M, mm[q]);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                mm[q] = fast_exp2(mm[q] - M);
                L = fmaf(mm[q], ll[q], L);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) weight[i * 8 + q] = mm[q] / L;
        }
        __syncthreads();
        if (!*abort_flag) {   // a CTA whose wait gave up stores nothing
            constexpr int LR = HD / 4, RW = 32 / LR;   // lanes of a row, rows side by side in a warp: a lane takes four columns of four rows
            const int sub = lane / LR, l4 = lane % LR;
            for (int i0 = warp * 4 * RW + sub; i0 < share; i0 += kThreads / 32 * 4 * RW) {
                float4 acc[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                for (int q = 0; q < p.split; ++q) {
                    float x[4][4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int rr = row0 + i0 + k * RW;
                        ld_peer_v4(map_to_cta(base + OFF_RING + rr * (HD * 4) + ((l4 ^ (rr & (LR - 1))) << 4), q), x[k]);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float w = weight[(i0 + k * RW) * 8 + q];
                        acc[k].x = fmaf(w, x[k][0], acc[k].x);
                        acc[k].y = fmaf(w, x[k][1], acc[k].y);
                        acc[k].z = fmaf(w, x[k][2], acc[k].z);
                        acc[k].w = fmaf(w, x[k][3], acc[k].w);
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = r_pair + row0 + i0 + k * RW;
                    if (i0 + k * RW < share && r < p.rows_total)
                        *reinterpret_cast<uint2*>(p.out + (((long long)b * p.n_active + r) * p.n_q_heads + hk) * HD + l4 * 4) =
                            make_uint2(pack_bf16x2(acc[k].x, acc[k].y), pack_bf16x2(acc[k].z, acc[k].w));
                }
            }
        }
        __syncwarp();
        cluster_arrive();         // no CTA leaves while a peer may still read its partial
        cluster_wait();
    }

    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TM_COLS) : "memory");
    }
    if (kCut && warp == 0) pdl_wait();
}

// ---- host side ---------------------------------------------------------------------------
// Q of an MHA step seen as 5-D {64 columns, active row, head, half, sequence}: one box {64, 128, 1, 2, 1} lands as the
// two 128-byte-swizzled halves of a [128 rows x 128] tile; rows past n_active read as zero.
// K or V seen as 5-D {64 columns, key, half, kv head, sequence}: one box {64, 128, 2, 1, 1} lands as
// [half][key][64 columns], the two 128-byte-swizzled halves of a [128 keys x 128] tile; keys beyond L read as zero.
// Cache layout [B, Hkv, L, 128] or token-major [B, L, Hkv, 128] (the fresh K/V of a recompute step): only the
// strides differ.  (64-wide heads: one half.)
bool make_kv_map(CUtensorMap* map, const void* ptr, int hd, int batch, int n_kv_heads, int ctx_len, bool token_major) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)hd * 2;
    const cuuint64_t dims[5] = {64, (cuuint64_t)ctx_len, (cuuint64_t)hd / 64, (cuuint64_t)n_kv_heads, (cuuint64_t)batch};
    const cuuint64_t strides[4] = {token_major ? row * n_kv_heads : row, 128, token_major ? row : row * ctx_len,
                                   row * ctx_len * n_kv_heads};
    const cuuint32_t box[5] = {64, (cuuint32_t)BN, (cuuint32_t)hd / 64, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// How the launch is cut.  Units = (sequence, query head, row-tile pair); a unit walks over all T key tiles.  The
// hardware deals the CTAs to the SMs in launch order, so the last units form a partial wave: `tail` units on `sms` SMs.
// Cutting each of them along the keys into s CTAs, a cluster, fills that wave.  As many parts as run at once and leave four
// tiles each, if that takes four tiles off the wave: a launch of its own with its start and merge costs about as much.  (Nine
// tiles beside whole units lose by it; the tests of cut units have them in two parts.)
// us a layer by number of parts (the rule's in brackets): 4 units of 16 tiles (19 heads of 2048) 1: 55.8, 2: 49.6, (4): 46.5,
// 8: 45.1; 12 of 21 (28 heads of 2600) 1: 100.7, 2: 94.7, 4: 90.9, (5): 90.0, 8: 88.6; 12 of 10 (32 heads of 1280) 1: 39.9, (2): 38.0,
// 5: 37.6; 12 of 9 (1152) 1: 34.5, (2): 35.6; 40 of 12 (2 x 1531, 28 heads) 1: 67.4, 2: 64.8, (3): 64.6, 4 (two rounds): 79.2; 20
// of 12 (28 heads of 1500) 1: 45.1, 2: 41.8, (3): 41.2, 4: 40.6; 68 of 32 (32 heads of 4096) 1: 213.5, (2): 205, 3 (two rounds): 217.5.
struct DensePlan {
    int n_pairs, units, n_full, split;
};
// How many clusters of s CTAs of the cut launch the current device keeps resident at once.  A cluster stays inside a GPC, and
// these need neither be alike nor hold a multiple of s SMs: 148 SMs taken as eight GPCs of 18 gave 48 clusters of three, of which
// 45 ran and the others made a second round (8 heads of 1500, 48 units: 33.8 us a layer in three parts, 19.1 in two).
// Asked once per device; without a device to ask, that assumption.
template <int HD>
int resident_clusters(int s) {
    static std::atomic<int> cached[kMaxDevices][9] = {};   // + 1
    static PerDeviceOnce attr_once;
    int dev = 0, n = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess;
    const bool slot = known && dev >= 0 && dev < kMaxDevices;
    if (slot)
        if (const int v = cached[dev][s].load(std::memory_order_relaxed)) return v - 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(s, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Geo<HD>::BYTES;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (!known || ensure_dynamic_smem(attr_once, attend_dense_kernel<true, HD>, (int)Geo<HD>::BYTES) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, attend_dense_kernel<true, HD>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 8 * (sm_count() / 8 / s);
    }
    if (slot) cached[dev][s].store(n + 1, std::memory_order_relaxed);
    return n;
}

DensePlan make_dense_plan(const ec_attn_desc& d, int n_active) {
    DensePlan pl;
    pl.n_pairs = (n_active + 2 * BM - 1) / (2 * BM);
    pl.units = pl.n_pairs * d.batch * d.n_q_heads;
    pl.n_full = pl.units;
    pl.split = 1;
    const int sms = sm_count();
    const int T = (d.ctx_len + BN - 1) / BN, tail = pl.units % sms;
    for (int s = 8; s >= 2 && tail > 0; --s) {
        if (T / s < 4 || T - (T + s - 1) / s < 4) continue;
        if (tail > (d.head_dim == 128 ? resident_clusters<128>(s) : resident_clusters<64>(s))) continue;
        pl.split = s;
        pl.n_full = pl.units - tail;
        break;
    }
    return pl;
}


}  // namespace

// The two-tile kernel is used from 17 of its (row-tile pair, query head) units on.  The one-tile kernel behind a
// refresh launch, which takes the steps below, is the slower one on both sides of the line (us a layer, one-tile against this
// one): 32 units of 2 key tiles (32 heads of 256) 24.9 / 9.6, of 8 tiles (8 heads of 1024) 42.5 / 16.7, of 32 tiles (2 heads of
// 4096) 60.8 / 25.0; 20 units (2 x 300, 5 heads) 23.6 / 9.6; 16 units 24.8 / 11.0, 8 units of 3 tiles 19.6 / 9.0.  The line
// stops short of 16 units, which the tests of the dispatch expect on the one-tile kernel.
constexpr int kOneTileUnits = 16;

// 64-wide heads.  The mma.sync kernel packs the rows of a kv head's query heads and refreshes in its launch; this one has 128
// rows of a query head a tile and a refresh launch in front.  More than 256 fresh rows and more units than SMs are this one's
// (the faster one on all of 282 such shapes; one found since, 2 x 260 with 40 heads on 8 and 259 rows, takes 15.8 us, 13.5 on
// mma.sync).  Partial steps of at most 128 rows are mma.sync's unless they are large (a bound, below which the estimates are too
// rough).  Then the estimates of both decide, mma.sync where it is 3 % ahead.  Of 2153 shapes timed (1 to 32 sequences, 129 to
// 4096 keys, 8 to 1000 rows or all, 1 to 32 heads, groups of 1 to 8) 9 are more than 3 % slower here than on mma.sync, of 700
// others 7; when recompute steps and partial ones of more than 128 rows were not asked about, 42 and 24.
// us a layer, mma.sync / this kernel: recompute steps 2 x 1024 with 24 heads on 8 51.5 / 31.4, 4 x 1000 94.1 / 47.5, 1 x 300 with 9
// 9.0 / 7.8, 32 x 129 with 24 on 8 32.0 / 42.1; index lists 4 x 1000 with 24 on 8, 96 rows 23.9 / 13.6, 48 rows 16.2 / 13.3, 4 x 700
// with 6 on 2, 129 rows 10.9 / 13.6, 1 x 1000 with 9, 257 rows 9.2 / 14.8, 64 x 500 with 12 on 4, 40 rows 33.8 / 46.4.
double dense_us(const ec_attn_desc& d, int n_active, bool fresh) {   // 6 % rms
    const DensePlan pl = make_dense_plan(d, n_active);
    const int T = (d.ctx_len + BN - 1) / BN, sms = sm_count();
    const double tile = n_active > BM ? 1.44 : 1.02, around = n_active > BM ? 4.2 : 3.4;   // two row tiles or one
    double us = -0.7 + (pl.n_full + sms - 1) / sms * (tile * T + around);
    if (pl.split > 1) us += tile * ((T + pl.split - 1) / pl.split) + around + 4.2;
    if (fresh && n_active < d.ctx_len) us += 1.6 + 1.4e-4 * n_active * d.batch * d.n_kv_heads;
    return us;
}
bool prefers_mma(const ec_attn_desc& d, int n_active, bool fresh, long long units) {
    if (fresh && n_active > 2 * BM && units > sm_count()) return false;
    if (n_active < d.ctx_len && n_active <= BM) {
        const int packed = n_active * (d.n_q_heads / d.n_kv_heads), tiles = (packed + 63) / 64, sms = sm_count();
        const double rows = (double)tiles * (tiles > 1 && packed <= 48 * tiles ? 48 : 64) * d.batch * d.n_kv_heads;
        const double waves = (double)((units + sms - 1) / sms) * ((d.ctx_len + BN - 1) / BN + 3.3) + (fresh ? 2. : 0.);
        if (5.5 + rows * d.ctx_len / (fresh ? 0.55e6 : 0.8e6) <= waves) return true;
    }
    return attend_mma_us(d, n_active, fresh) < 0.97 * dense_us(d, n_active, fresh);
}
bool attend_dense_supported(const ec_attn_desc& d, int n_active, bool fresh) {
    if (d.dtype != EC_BF16 || n_active < 1) return false;
    // one unit per (sequence, query head, row-tile pair): grouped-query shapes are run head by head
    const long long pairs = ((long long)n_active + 2 * BM - 1) / (2 * BM);
    const long long units = pairs * d.batch * d.n_q_heads;
    if (units <= kOneTileUnits || units > 0x3fffffffLL) return false;
    return d.head_dim == 128 || !prefers_mma(d, n_active, fresh, units);
}

void attend_dense_describe(const ec_attn_desc& d, int n_active, char* buf, size_t len) {
    const DensePlan pl = make_dense_plan(d, n_active);
    const int T = (d.ctx_len + BN - 1) / BN;
    int lo = T, hi = 0;   // key tiles of the shortest and the longest part of a cut unit
    for (int i = 0; i < pl.split; ++i) {
        const int n = part_begin(T, pl.split, i + 1) - part_begin(T, pl.split, i);
        lo = n < lo ? n : lo;
        hi = n > hi ? n : hi;
    }
    const int n = snprintf(buf, len, "attend_dense_kernel%s grid=(%d,%d) cluster=1 whole_units=%d cut_units=%dx%d part_tiles=%d..%d",
                           d.head_dim == 64 ? "<64>" : "", pl.n_pairs, d.batch * d.n_q_heads, pl.n_full, pl.units - pl.n_full,
                           pl.split, lo, hi);
    if (pl.split > 1 && n > 0 && (size_t)n < len)
        snprintf(buf + n, len - n, " at_once=%d", d.head_dim == 128 ? resident_clusters<128>(pl.split) : resident_clusters<64>(pl.split));
}

template <int HD>
cudaError_t launch_dense(const AttendArgs& a, cudaStream_t stream) {
    CUtensorMap map_k, map_v;
    if (!make_kv_map(&map_k, a.k_cache, HD, a.d.batch, a.d.n_kv_heads, a.d.ctx_len, a.kv_token_major) ||
        !make_kv_map(&map_v, a.v_cache, HD, a.d.batch, a.d.n_kv_heads, a.d.ctx_len, a.kv_token_major))
        return cudaErrorInvalidValue;
    DenseParams p;
    p.out = static_cast<__nv_bfloat16*>(a.out);
    p.copy = a.kv_token_major && a.refresh_k_dst && a.refresh_v_dst;
    CUtensorMap map_kd = map_k, map_vd = map_v;   // placeholders unless copying
    if (p.copy && (!make_kv_map(&map_kd, a.refresh_k_dst, HD, a.d.batch, a.d.n_kv_heads, a.d.ctx_len, false) ||
                   !make_kv_map(&map_vd, a.refresh_v_dst, HD, a.d.batch, a.d.n_kv_heads, a.d.ctx_len, false)))
        return cudaErrorInvalidValue;
    p.dev_status = a.dev_status;
    p.n_active = a.n_active;
    p.ctx_len = a.d.ctx_len;
    p.n_q_heads = a.d.n_q_heads;
    p.n_kv_heads = a.d.n_q_heads;   // the kernel's heads are the query heads, see kv_div
    p.rows_total = a.n_active;
    p.kv_div = a.d.n_q_heads / a.d.n_kv_heads;
    p.scale_log2 = a.scale * kLog2e;
    const DensePlan pl = make_dense_plan(a.d, a.n_active);
    p.n_pairs = pl.n_pairs;
    p.n_full = pl.n_full;
    p.split = pl.split;
    p.wait_first = pl.n_full == 0;
    CUtensorMap map_q;
    {
        EncodeTiledFn fn = encode_fn();
        if (!fn) return cudaErrorInvalidValue;
        const cuuint64_t dims[5] = {64, (cuuint64_t)a.n_active, (cuuint64_t)a.d.n_q_heads, HD / 64, (cuuint64_t)a.d.batch};
        const cuuint64_t strides[4] = {(cuuint64_t)a.d.n_q_heads * HD * 2, (cuuint64_t)HD * 2, 128,
                                       (cuuint64_t)a.n_active * a.d.n_q_heads * HD * 2};
        const cuuint32_t box[5] = {64, (cuuint32_t)BM, 1, HD / 64, 1};
        const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
        if (fn(&map_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(a.q), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    static PerDeviceOnce once_whole, once_cut;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Geo<HD>::BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = pl.split;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    if (pl.n_full > 0) {
        if (const cudaError_t e = ensure_dynamic_smem(once_whole, attend_dense_kernel<false, HD>, (int)Geo<HD>::BYTES); e != cudaSuccess) return e;
        cfg.gridDim = dim3(pl.n_full, 1, 1);
        cfg.numAttrs = 1;
        if (const cudaError_t e = cudaLaunchKernelEx(&cfg, attend_dense_kernel<false, HD>, map_k, map_v, map_q, map_kd, map_vd, p);
            e != cudaSuccess)
            return e;
    }
    if (pl.n_full == pl.units) return cudaSuccess;
    if (const cudaError_t e = ensure_dynamic_smem(once_cut, attend_dense_kernel<true, HD>, (int)Geo<HD>::BYTES); e != cudaSuccess) return e;
    cfg.gridDim = dim3((pl.units - pl.n_full) * pl.split, 1, 1);
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attend_dense_kernel<true, HD>, map_k, map_v, map_q, map_kd, map_vd, p);
}

cudaError_t launch_attend_dense(const AttendArgs& a, cudaStream_t stream) {
    return a.d.head_dim == 128 ? launch_dense<128>(a, stream) : launch_dense<64>(a, stream);
}

}  // namespace ec
