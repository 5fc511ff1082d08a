// The many-head variant of the skip step with few rows, run by attend_skip_kernel<1> when one CTA takes a whole kv head
// and at most 64 packed query rows share it (bf16, head_dim 128): the KEYS take the M axis of the tensor core, as in
// attend_skip_keys_kernel,
//     S^T[128 keys x N] = K_tile . Q^T,   O^T[128 d x N] += V_tile^T . P^T   (N = 48 or 64 query slots),
// in a CTA small enough for two per SM.
//
// Why: with the query rows on M a batch of heads is bound by the softmax.  34 rows live in the TMEM lanes of two of the
// four warp quarters, so one SM sub-partition does 64 exponentials a lane and key tile of 64 for both CTAs (1.0 us a
// tile) while the others idle.  Here every lane of every quarter owns a key and half of its scores.  Eight sequences of
// 4096 with 32 heads and 34 rows: 85 us a layer (6.5 TB/s) against 107, five with 40 rows 68 against 87.
//   warp 0     TMA producer: one K slot and one V slot of 128 keys, each refilled as soon as its product has run (two
//              CTAs per SM keep each other's latency covered);
//   warp 1     tcgen05.mma issue, whichever product is ready, S one tile ahead (two S^T buffers);
//   warps 2-9  two softmax warpgroups, half the query slots each: Q, key masks and the cache update first, then
//              p = 2^(s*scale*log2e - m[q]) against references that only move when a score exceeds one by 2^60 (a
//              barrier-wide vote per tile), row sums per key lane in registers, added up once at the end.
// The fresh rows are attended as an extra key tile from k_new / v_new after the cache tiles, the stale cached keys masked;
// the cache update is ordered against nothing.
#pragma once

#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

namespace ec {
namespace keys_pair {

using namespace tc;

constexpr int BK = 128, HD = 128, kMaxSlots = 64;
constexpr int kThreads = 320, kSoft = 256;
constexpr uint32_t SUB = 128 * 128, TILE = 2 * SUB;
// shared-memory carve: Q, P^T, the K slot, the V slot, key masks
constexpr uint32_t OFF_Q = 0;
__host__ __device__ constexpr uint32_t off_p(int n) { return (uint32_t)n * 256u; }
__host__ __device__ constexpr uint32_t off_k(int n) { return off_p(n) + SUB; }
__host__ __device__ constexpr uint32_t off_v(int n) { return off_k(n) + TILE; }
__host__ __device__ constexpr uint32_t off_bits(int n) { return off_v(n) + TILE; }
__host__ __device__ constexpr int slots(int rows) { return rows <= 48 ? 48 : 64; }
constexpr uint32_t TM_COLS = 256, TM_S = 0, TM_O = 128;
constexpr float kRaise = 60.f;

enum { KB_KFULL = 0, KB_KEMPTY, KB_VFULL, KB_VEMPTY, KB_SFULL, KB_PFULL = KB_SFULL + 2, KB_PVDONE, KB_QFULL, KB_COUNT };

struct alignas(16) Shared {
    unsigned long long bars[KB_COUNT + (KB_COUNT & 1)];
    uint32_t tmem;
    int abort_flag;
    int pad[2];
    alignas(16) float m[kMaxSlots];          // references of the query rows, log2 units
    alignas(16) float factor[kMaxSlots];     // rescale factors of the rare path; at the end 1 / l
    float col[4][kMaxSlots];                 // per warp quarter: column maxima of the rare path; at the end row sums
};

struct Params {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_new;   // nullptr: attend without refreshing
    const __nv_bfloat16* v_new;
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* active_idx;
    __nv_bfloat16* out;
    int32_t* dev_status;
    int n_active, ctx_len, n_q_heads, n_kv_heads, group, group_inv;   // group_inv = ceil(2^16 / group)
    int early_cache;
    float scale_log2;
};

// key masks: 16 bytes per key tile, cache tiles first, then the fresh tile
__host__ __device__ constexpr uint32_t bits_bytes(int ctx_len) { return (uint32_t)((ctx_len + BK - 1) / BK + 1) * 16u; }
inline uint32_t smem_bytes(int rows, int ctx_len) { return off_bits(slots(rows)) + bits_bytes(ctx_len) + (uint32_t)sizeof(Shared); }

template <int COLS>
__device__ __forceinline__ void ld_cols(uint32_t taddr, uint32_t* r) {
#pragma unroll
    for (int c = 0; c < COLS; c += 8) ld8(taddr + c, r + c);
    wait_ld<COLS>(r);
}

template <int N>
__device__ __forceinline__ void run(const CUtensorMap& map_k, const CUtensorMap& map_v, const CUtensorMap& map_kn,
                                    const CUtensorMap& map_vn, const Params& p, unsigned char* gbase) {
    constexpr int NH = N / 2;
    // Who issues: the whole warp (see elect_one) with 48 slots, which is up to 3 % ahead from 768 keys on and with few rows, one
    // thread with 64, where the whole warp is the slower one (us a layer, 5 x 32 heads of 200 17.23 -> 17.60, of 768 26.4 -> 26.9).
    constexpr bool kWarpIssues = N == 48;
    constexpr uint32_t OFF_P = off_p(N), OFF_K = off_k(N), OFF_V = off_v(N), OFF_BITS = off_bits(N);
    const uint32_t base = s2u(gbase);
    uint32_t* bits = reinterpret_cast<uint32_t*>(gbase + OFF_BITS);
    Shared* sh = reinterpret_cast<Shared*>(gbase + OFF_BITS + bits_bytes(p.ctx_len));
    volatile int* abort_flag = &sh->abort_flag;
    const uint32_t bars = s2u(sh->bars);
    auto bar = [&](int i) { return bars + 8u * i; };

    const int tid = threadIdx.x, warp = kWarpIssues ? warp_index() : tid >> 5, lane = tid & 31;
    const int bh = blockIdx.y, b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads;
    const int rows_total = p.n_active * p.group;
    const bool refresh = p.k_new != nullptr;
    const int TC = (p.ctx_len + BK - 1) / BK, T = TC + (refresh ? 1 : 0);

    auto load_k = [&](int j) {
        mbar_expect_tx(bar(KB_KFULL), TILE);
        if (j < TC) tma_load_4d(base + OFF_K, &map_k, 0, j * BK, 0, bh, bar(KB_KFULL));
        else tma_load_5d(base + OFF_K, &map_kn, 0, 0, 0, hk, b, bar(KB_KFULL));   // rows past n_active read as zero
    };
    auto load_v = [&](int j) {
        mbar_expect_tx(bar(KB_VFULL), TILE);
        if (j < TC) tma_load_4d(base + OFF_V, &map_v, 0, j * BK, 0, bh, bar(KB_VFULL));
        else tma_load_5d(base + OFF_V, &map_vn, 0, 0, 0, hk, b, bar(KB_VFULL));
    };
    if (tid == 0) {
        for (int i = 0; i < KB_COUNT; ++i) mbar_init(bar(i), (i == KB_PFULL || i == KB_QFULL) ? kSoft : 1);
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (p.early_cache) {
            load_k(0);
            load_v(0);
        }
    }
    for (int w = tid; w < 4 * T; w += kThreads) bits[w] = 0u;
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
    pdl_wait();
    if (tid == 32) pdl_launch_dependents();
    __syncwarp();

    if (warp == 0) {
        if (lane == 0) {
            int jk = p.early_cache ? 1 : 0, jv = jk;
            SpinGuard guard;
            while (jk < T || jv < T) {
                bool progressed = false;
                if (jk < T && (jk == 0 || mbar_test(bar(KB_KEMPTY), (jk - 1) & 1))) {
                    load_k(jk++);
                    progressed = true;
                }
                if (jv < T && (jv == 0 || mbar_test(bar(KB_VEMPTY), (jv - 1) & 1))) {
                    load_v(jv++);
                    progressed = true;
                }
                if (progressed) guard.progress();
                else if (!guard.tick(abort_flag, p.dev_status)) break;
            }
        }
    } else if (warp == 1) {
        if (kWarpIssues || lane == 0) {
            const bool elected = kWarpIssues ? elect_one() : true;
            auto ready = [&](int i, int n) { return kWarpIssues ? mbar_test_lane(bar(i), n & 1) : mbar_test(bar(i), n & 1); };
            constexpr uint32_t IDESC_S = instr_desc2(N, 0, 0);    // A = K tile (K-major), B = Q (K-major)
            constexpr uint32_t IDESC_PV = instr_desc2(N, 1, 1);   // A = V tile (MN-major: d contiguous), B = P^T (MN-major)
            constexpr uint32_t QHALF = N * 128;
            const uint64_t desc_q = smem_desc(base + OFF_Q, 16, 1024), desc_p = smem_desc(base + OFF_P, SUB, 1024);
            const uint64_t desc_k = smem_desc(base + OFF_K, 16, 1024), desc_v = smem_desc(base + OFF_V, SUB, 1024);
            mbar_wait(bar(KB_QFULL), 0, abort_flag, p.dev_status);
            int next_s = 0, next_pv = 0;
            SpinGuard guard;
            while (next_pv < T) {
                bool progressed = false;
                if (next_s < T && next_s <= next_pv + 1 && ready(KB_KFULL, next_s)) {
                    fence_after();
                    if (elected) {
#pragma unroll
                        for (int k = 0; k < HD / 16; ++k)
                            mma_ss(tmem + TM_S + (next_s & 1) * 64, desc_k + ((k >> 2) * SUB + (k & 3) * 32) / 16,
                                   desc_q + ((k >> 2) * QHALF + (k & 3) * 32) / 16, IDESC_S, k > 0);
                        commit(bar(KB_SFULL + (next_s & 1)));
                        commit(bar(KB_KEMPTY));
                    }
                    ++next_s;
                    progressed = true;
                }
                if (next_pv < next_s && ready(KB_PFULL, next_pv) && ready(KB_VFULL, next_pv)) {
                    fence_after();
                    if (elected) {
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k)
                            mma_ss(tmem + TM_O, desc_v + k * 128, desc_p + k * 128, IDESC_PV, (next_pv > 0 || k > 0));
                        commit(bar(KB_PVDONE));
                        commit(bar(KB_VEMPTY));
                    }
                    ++next_pv;
                    progressed = true;
                }
                if (progressed) {
                    guard.progress();
                } else {
                    const bool go_on = guard.tick(abort_flag, p.dev_status);
                    if (kWarpIssues ? __any_sync(0xffffffffu, !go_on) : !go_on) break;
                }
            }
        }
    } else {
        const int stid = tid - 64, wg = stid >> 7, c0 = wg * NH, st_w = stid & 127;
        {   // Q rows -> swizzled K-major tile of N rows (rows past rows_total are zero), key masks, cache update
            constexpr int kPieces = N * (HD / 8) / kSoft;   // 16-byte pieces of Q per thread
            const int ch = stid & 15;
            uint4 v[kPieces];
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                const int row = (stid >> 4) + u * (kSoft / 16);
                const int i = (row * p.group_inv) >> 16, jh = row - i * p.group;
                v[u] = make_uint4(0u, 0u, 0u, 0u);
                ldg_nc_v4_pred(v[u], p.q + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + jh) * HD + ch * 8,
                               row < rows_total);
            }
            if (refresh && stid < p.n_active) {   // n_active <= rows_total <= N
                const int pos = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + stid) : stid;
                if (pos >= 0 && pos < p.ctx_len) {
                    atomicOr(&bits[pos >> 5], 1u << (pos & 31));                       // the cached key is stale
                    atomicOr(&bits[4 * TC + (stid >> 5)], 1u << (stid & 31));          // the fresh key exists
                }
            }
#pragma unroll
            for (int u = 0; u < kPieces; ++u) {
                const int row = (stid >> 4) + u * (kSoft / 16);
                const uint32_t off = OFF_Q + (ch >> 3) * (N * 128) + (row >> 3) * 1024 + (row & 7) * 128 + (((ch & 7) ^ (row & 7)) << 4);
                *reinterpret_cast<uint4*>(gbase + off) = v[u];
            }
            fence_async_smem();     // Q (generic proxy) -> visible to the tensor core (async proxy)
            mbar_arrive(bar(KB_QFULL));
            if (refresh) {
                const int pieces = p.n_active * 32;   // [row][K, V][16 pieces], at most N / 8 per thread
                uint4 w[N / 8];
                int pos[N / 8];
#pragma unroll
                for (int u = 0; u < N / 8; ++u) {
                    const int c = stid + u * kSoft, i = c >> 5;
                    pos[u] = -1;
                    if (c < pieces) {
                        pos[u] = p.active_idx ? __ldg(p.active_idx + (long long)b * p.n_active + i) : i;
                        w[u] = __ldg(reinterpret_cast<const uint4*>(
                            ((c & 16) ? p.v_new : p.k_new) + (((long long)b * p.n_active + i) * p.n_kv_heads + hk) * HD + (c & 15) * 8));
                    }
                }
#pragma unroll
                for (int u = 0; u < N / 8; ++u) {
                    const int c = stid + u * kSoft;
                    if (pos[u] < 0 || pos[u] >= p.ctx_len) continue;
                    *reinterpret_cast<uint4*>(((c & 16) ? p.v_cache : p.k_cache) + ((long long)bh * p.ctx_len + pos[u]) * HD +
                                              (c & 15) * 8) = w[u];
                }
            }
            named_barrier(6, kSoft);   // the masks are complete
        }
        const int quarter = warp & 3, kk = quarter * 32 + lane;   // key of the tile == TMEM lane == output column later on
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const float sl2 = p.scale_log2;
        const f32x2 sl2_2 = pk(sl2, sl2);
        unsigned char* prow = gbase + OFF_P + (kk >> 3) * 1024 + (kk & 7) * 128;   // P^T row of this key: 64 slots, swizzled
        const int bar_or = 2 + 2 * wg, bar_sync = 3 + 2 * wg;
        f32x2 lsum[NH / 2];
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) lsum[i] = pk(0.f, 0.f);
        for (int j = 0; j < T; ++j) {
            mbar_wait(bar(KB_SFULL + (j & 1)), (j >> 1) & 1, abort_flag, p.dev_status);
            fence_after();
            const uint32_t s_addr = tmem + lane_addr + TM_S + (j & 1) * 64 + c0;
            const bool bit = (bits[j * 4 + quarter] >> lane) & 1u;
            const bool gone = j < TC ? (bit || j * BK + kk >= p.ctx_len) : !bit;   // this key does not count
            uint32_t sr[NH];
            ld_cols<NH>(s_addr, sr);
            if (j == 0) {   // first reference: the scores of the first key that counts among the first warp's 32
                const uint32_t valid = __ballot_sync(0xffffffffu, !gone);
                if (quarter == 0 && lane == __ffs(valid) - 1) {
#pragma unroll
                    for (int c = 0; c < NH; c += 4)
                        *reinterpret_cast<float4*>(&sh->m[c0 + c]) =
                            make_float4(__uint_as_float(sr[c]) * sl2, __uint_as_float(sr[c + 1]) * sl2,
                                        __uint_as_float(sr[c + 2]) * sl2, __uint_as_float(sr[c + 3]) * sl2);
                }
                named_barrier(bar_sync, 128);
            }
            uint32_t pw[NH / 2];
            while (true) {
                float dmx0 = -INFINITY, dmx1 = -INFINITY;
#pragma unroll
                for (int i = 0; i < NH / 2; ++i) {
                    const float2 mm = *reinterpret_cast<const float2*>(&sh->m[c0 + 2 * i]);
                    f32x2 d2 = fma2(pk(__uint_as_float(sr[2 * i]), __uint_as_float(sr[2 * i + 1])), sl2_2, pk(-mm.x, -mm.y));
                    if (gone) d2 = pk(-INFINITY, -INFINITY);   // probability 0 for every query
                    float d0, d1;
                    upk(d2, d0, d1);
                    if (i & 1) dmx1 = max3(dmx1, d0, d1); else dmx0 = max3(dmx0, d0, d1);
                    pw[i] = pack_bf16x2(fast_exp2(d0), fast_exp2(d1));
                }
                if (!named_barrier_or(bar_or, 128, fmaxf(dmx0, dmx1) > kRaise)) break;
                // ---- rare: raise the references to this tile's column maxima, rescale O^T and the row sums, once more ----
#pragma unroll
                for (int c = 0; c < NH; ++c) {
                    const float o = redux_max(gone ? -INFINITY : __uint_as_float(sr[c]));
                    if (lane == c) sh->col[quarter][c0 + c] = o;
                }
                named_barrier(bar_sync, 128);
                if (st_w < NH) {
                    const int c = c0 + st_w;
                    const float o = fmaxf(fmaxf(sh->col[0][c], sh->col[1][c]), fmaxf(sh->col[2][c], sh->col[3][c]));
                    const float m_old = sh->m[c], m_new = fmaxf(m_old, o * sl2);
                    sh->factor[c] = (m_old == -INFINITY) ? 0.f : fast_exp2(m_old - m_new);
                    sh->m[c] = m_new;
                }
                named_barrier(bar_sync, 128);
                if (j > 0) {   // O^T holds the tiles before j: P V of tile j - 1 must have completed
                    mbar_wait(bar(KB_PVDONE), (j - 1) & 1, abort_flag, p.dev_status);
                    fence_after();
                    const uint32_t o_addr = tmem + lane_addr + TM_O + c0;
                    uint32_t o[8];
#pragma unroll
                    for (int q = 0; q < NH; q += 8) {
                        ld8(o_addr + q, o);
                        wait_ld<8>(o);
#pragma unroll
                        for (int c = 0; c < 8; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * sh->factor[c0 + q + c]);
                        st8(o_addr + q, o);
                    }
                    wait_st();
#pragma unroll
                    for (int i = 0; i < NH / 2; ++i) {
                        const float2 f = *reinterpret_cast<const float2*>(&sh->factor[c0 + 2 * i]);
                        lsum[i] = mul2(lsum[i], pk(f.x, f.y));
                    }
                }
                named_barrier(bar_sync, 128);   // the factors have been read
            }
            if (j > 0) mbar_wait(bar(KB_PVDONE), (j - 1) & 1, abort_flag, p.dev_status);   // the P^T buffer is free
#pragma unroll
            for (int ch = 0; ch < NH / 8; ++ch) {
                const int gch = (c0 >> 3) + ch;      // 16-byte chunk (8 slots) of the P^T row
                *reinterpret_cast<uint4*>(prow + ((gch ^ (kk & 7)) << 4)) =
                    make_uint4(pw[4 * ch], pw[4 * ch + 1], pw[4 * ch + 2], pw[4 * ch + 3]);
            }
            fence_async_smem();
            fence_before();
            mbar_arrive(bar(KB_PFULL));
#pragma unroll
            for (int i = 0; i < NH / 2; ++i)   // (while the second product runs)
                lsum[i] = add2(lsum[i], pk(__uint_as_float(pw[i] << 16), __uint_as_float(pw[i] & 0xffff0000u)));
        }
        {   // row sums over the warp's 32 keys: three steps halve the columns a lane holds, the last two add up
            float v[NH];
#pragma unroll
            for (int i = 0; i < NH / 2; ++i) upk(lsum[i], v[2 * i], v[2 * i + 1]);
            int first = c0;
#pragma unroll
            for (int step = 1; step <= 3; ++step) {
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
            for (int i = 0; i < NH / 8; ++i) {
                v[i] += __shfl_xor_sync(0xffffffffu, v[i], 2);
                v[i] += __shfl_xor_sync(0xffffffffu, v[i], 1);
                if (!(lane & 3)) sh->col[quarter][first + i] = v[i];
            }
        }
        named_barrier(bar_sync, 128);
        if (st_w < NH) {
            const int c = c0 + st_w;
            sh->factor[c] = 1.f / ((sh->col[0][c] + sh->col[1][c]) + (sh->col[2][c] + sh->col[3][c]));
        }
        named_barrier(bar_sync, 128);
        mbar_wait(bar(KB_PVDONE), (T - 1) & 1, abort_flag, p.dev_status);
        fence_after();
        uint32_t o[NH];
        ld_cols<NH>(tmem + lane_addr + TM_O + c0, o);
        if (!*abort_flag) {   // a CTA whose wait gave up stores nothing
#pragma unroll
            for (int c = 0; c < NH; ++c) {
                if (c0 + c >= rows_total) continue;
                const int i = ((c0 + c) * p.group_inv) >> 16, jh = c0 + c - i * p.group;
                p.out[(((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + jh) * HD + kk] =
                    __float2bfloat16_rn(__uint_as_float(o[c]) * sh->factor[c0 + c]);
            }
        }
        fence_before();
    }
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TM_COLS) : "memory");
    }
}

}  // namespace keys_pair
}  // namespace ec
