// ec_attend, bf16 storage, heads of 64, warp-level tensor-core path (mma.sync m16n8k16, fp32
// accumulation): refresh and active-row bidirectional attention over the full cache
// (Appendix A of the paper, partial branch; the full branch when n_active == L) in ONE launch.
//
// Work decomposition
//   - The query rows that share one kv head -- n_active rows x g = H_q/H_kv query
//     heads -- are flattened into one row axis r = i*g + j (GQA packing), cut into
//     64-row tiles; one CTA (4 warps x 16 rows) owns one tile.  Where as many tiles of
//     48 rows hold them (make_plan), the fourth warp only moves data.
//   - Keys are cut into 64-key tiles.  When there are few row tiles (skip step:
//     34 active rows) up to eight CTAs, a cluster, split the keys of a row tile; each leaves
//     (m, l, O) un-normalised in its shared memory and, after a cluster barrier, merges a share
//     of the rows out of its peers' (partials in global memory and a second launch took 5.4 us more).
//   - K/V tiles are staged in shared memory, XOR-swizzled so ldmatrix is bank-conflict free: by TMA, a box each, when
//     no index list sends keys elsewhere (the 128-byte swizzle of a 128-byte row is the same
//     XOR); else with 16-byte cp.async copies.  A key that is being refreshed is read from k_new / v_new (a table of
//     the CTA's keys, filled from the index list), so nothing waits for the cache update; the row
//     tiles of a kv head share the writing of the cache.
//   - Softmax is online (running max / sum per row, exp2 with the scale folded
//     in); P is re-packed from the S accumulators into A fragments in registers.
// What bounds it: latency on partial steps of 64-wide heads (four sequences of 1000 keys, 48 rows, 12 query heads on 4:
// 8.8 us a layer, against 14.9 with the refresh and the merge as launches of their own), the mma.sync rate (2048 flop
// per clock and SM, measured) and the instructions around it on larger ones (36 sequences of 1500, 64 rows, no refresh: 45.3 us
// when all threads issued the copies, 38.7 with TMA).  What prefers_mma gives away is attend_dense_kernel's.  Every wait
// is bounded: EC_ERR_TIMEOUT in dev_status, and a CTA whose wait gave up stores no output and no further cache rows.
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

#include <algorithm>
#include <cmath>

namespace ec {
namespace {

constexpr int BM = 64;   // query rows per CTA
constexpr int BN = 64;   // keys per tile
constexpr int kThreads = 128;
constexpr int D = 64;    // head_dim
// K/V stages in shared memory.  A tile computes in about half the time its data takes to arrive, so two tiles have to be
// on their way (9.5 us against 13.4 with one).
constexpr int ST = 3;
constexpr int kMaxMapKeys = 8192;   // keys of one CTA beyond which the refresh is a launch of its own

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    const int sz = valid ? 16 : 0;  // src-size 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// byte offset of 16-byte chunk `chunk` of row `row` in a swizzled [rows, D] bf16 tile
__device__ __forceinline__ uint32_t swz(int row, int chunk) {
    return (uint32_t)(row * (D * 2) + ((chunk ^ (row & 7)) << 4));
}

struct MmaParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k_new;   // nullptr: attend without refreshing
    const __nv_bfloat16* v_new;
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    const int32_t* active_idx;    // nullptr: identity
    __nv_bfloat16* out;
    int n_active, ctx_len, n_q_heads, n_kv_heads, group;  // group = H_q / H_kv
    int rows_total;   // n_active * group
    int row_tiles, tile_rows, n_splits, tiles_per_split;   // tile_rows: BM, or 48 (kSpare)
    float scale_log2;  // scale * log2(e)
    int32_t* dev_status;
};

// kSpare: the last warp has no rows.  kTma: K/V tiles come by TMA, one box each in the very layout that swz() describes
// (no index list, so no key is sent elsewhere; a row is the 128 bytes of the swizzle).
template <bool kSpare, bool kTma>
__global__ void __launch_bounds__(kThreads, 3) attend_mma_kernel(const MmaParams p, const __grid_constant__ CUtensorMap map_k,
                                                                  const __grid_constant__ CUtensorMap map_v) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = smem_raw + (kTma ? -smem_u32(smem_raw) & 1023u : 0u);
    constexpr int TILE_BYTES = BN * D * 2;
    constexpr int CHUNKS = D / 8;  // 16-byte chunks per row
    unsigned char* sQ = smem;                       // BM x D
    unsigned char* sK = smem + BM * D * 2;          // ST stages
    unsigned char* sV = sK + ST * TILE_BYTES;       // ST stages
    float2* s_ml = reinterpret_cast<float2*>(sV + ST * TILE_BYTES);   // (m, l) per row, for the merge
    uint64_t* full = reinterpret_cast<uint64_t*>(s_ml + BM);         // kTma: a barrier per stage
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + ST);
    int* map = reinterpret_cast<int*>(full + ST + 1);   // [key of this CTA]: active row that refreshes it, or -1
    float* part = reinterpret_cast<float*>(sK);     // the partial of the merge, over the stages: [BM][PP]
    constexpr int PP = D + 8;                       // row pitch: fragment stores of eight rows cover all banks

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = blockIdx.x % p.n_splits, unit = blockIdx.x / p.n_splits;
    const int row_tile = unit % p.row_tiles, bh = unit / p.row_tiles;
    const int b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads;
    const int r0 = row_tile * (kSpare ? p.tile_rows : BM);
    const int r_end = kSpare ? min(p.rows_total, r0 + p.tile_rows) : p.rows_total;   // no row of this CTA is beyond it

    const int n_tiles_total = (p.ctx_len + BN - 1) / BN;
    const int t_begin = split * p.tiles_per_split;
    const int t_end = min(n_tiles_total, t_begin + p.tiles_per_split);

    const __nv_bfloat16* kbase = p.k_cache + ((long long)bh * p.ctx_len) * D;
    const __nv_bfloat16* vbase = p.v_cache + ((long long)bh * p.ctx_len) * D;

    const int key_lo = t_begin * BN, n_keys = min(p.ctx_len, t_end * BN) - key_lo;
    const bool fresh = p.k_new != nullptr, mapped = fresh && p.active_idx != nullptr;
    if (mapped)
        for (int k = tid; k < n_keys; k += kThreads) map[k] = -1;
    // where this thread's pieces of Q are (two divisions each: before the wait, not behind it), -1: no such row
    constexpr int QN = BM * CHUNKS / kThreads;
    long long q_at[QN];
#pragma unroll
    for (int k = 0; k < QN; ++k) {
        const int c = tid + k * kThreads, r = r0 + c / CHUNKS, i = r / p.group, j = r - i * p.group;
        q_at[k] = r < r_end ? (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + j) * D + c % CHUNKS * 8 : -1;
    }
    if (kTma && tid == 0) {
        tc::prefetch_map(&map_k);
        tc::prefetch_map(&map_v);
        for (int s = 0; s < ST; ++s) tc::mbar_init(smem_u32(full + s), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    tc::pdl_wait();
    tc::pdl_launch_dependents();

    // keys that no table sends elsewhere: the cache's panel of this head, or (identity list) the fresh tensor's rows
    const bool identity = fresh && !mapped;
    const long long new0 = ((long long)b * p.n_active * p.n_kv_heads + hk) * D;
    const int new_stride = p.n_kv_heads * D, key_stride = identity ? new_stride : D;
    const __nv_bfloat16 *ksrc0 = identity ? p.k_new + new0 : kbase, *vsrc0 = identity ? p.v_new + new0 : vbase;
    auto load_kv = [&](int tile, int stage) {
        const int key0 = tile * BN;
        if constexpr (kTma) {   // (rows past the context read as zero)
            if (tid == 0) {
                const uint32_t bar = smem_u32(full + stage), k = smem_u32(sK) + stage * TILE_BYTES, v = smem_u32(sV) + stage * TILE_BYTES;
                tc::mbar_expect_tx(bar, 2 * TILE_BYTES);
                tc::tma_load_5d(k, &map_k, 0, key0, 0, hk, b, bar);
                tc::tma_load_5d(v, &map_v, 0, key0, 0, hk, b, bar);
            }
        } else {
            for (int c = tid; c < BN * CHUNKS; c += kThreads) {
                const int row = c / CHUNKS, ch = c % CHUNKS;
                const bool ok = key0 + row < p.ctx_len;
                const long long off = ok ? (long long)(key0 + row) * key_stride : 0;
                const __nv_bfloat16 *ks = ksrc0 + off, *vs = vsrc0 + off;
                if (mapped && ok) {
                    const int i = map[key0 + row - key_lo];
                    if (i >= 0) {
                        ks = p.k_new + new0 + (long long)i * new_stride;
                        vs = p.v_new + new0 + (long long)i * new_stride;
                    }
                }
                cp_async16(smem_u32(sK) + stage * TILE_BYTES + swz(row, ch), ks + ch * 8, ok);
                cp_async16(smem_u32(sV) + stage * TILE_BYTES + swz(row, ch), vs + ch * 8, ok);
            }
        }
    };
    if constexpr (kTma) {
        for (int s = 0; s < ST - 1; ++s)
            if (t_begin + s < t_end) load_kv(t_begin + s, s);
    }
    // ---- stage Q (rows beyond rows_total are zero-filled) --------------------------
#pragma unroll
    for (int k = 0; k < QN; ++k) {
        const int c = tid + k * kThreads;
        cp_async16(smem_u32(sQ) + swz(c / CHUNKS, c % CHUNKS), p.q + max(q_at[k], 0LL), q_at[k] >= 0);
    }
    if (mapped) {
        for (int i = tid; i < p.n_active; i += kThreads) {
            const int k = __ldg(p.active_idx + (long long)b * p.n_active + i) - key_lo;
            if (k >= 0 && k < n_keys) map[k] = i;
        }
        __syncthreads();
    }
    for (int s = 0; s < ST - 1; ++s) {
        if (!kTma && t_begin + s < t_end) load_kv(t_begin + s, s);
        cp_async_commit();
    }

    // ---- per-thread state ----------------------------------------------------------
    uint32_t qf[D / 16][4];
    float o[D / 8][4];
#pragma unroll
    for (int n = 0; n < D / 8; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};  // rows g and g+8 of the warp's 16

    bool q_loaded = false;
    for (int t = t_begin; t < t_end; ++t) {
        const int stage = (t - t_begin) % ST;
        if constexpr (kTma) {
            if (t == t_begin) cp_async_wait<0>();   // Q
            tc::mbar_wait(smem_u32(full + stage), ((t - t_begin) / ST) & 1, abort_flag, p.dev_status);
        } else {
            cp_async_wait<ST - 2>();
        }
        __syncthreads();   // the tile has landed, and everyone is done with the one before it, whose stage is refilled now
        if (t + ST - 1 < t_end) load_kv(t + ST - 1, (t - t_begin + ST - 1) % ST);
        cp_async_commit();

        const int key0 = t * BN;
        if (!kSpare || r0 + warp * 16 < r_end) {
            if (!q_loaded) {
                q_loaded = true;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    ldsm_x4(smem_u32(sQ) + swz(warp * 16 + (lane & 15), ks * 2 + (lane >> 4)), qf[ks]);
            }

            // ---- S = Q K^T --------------------------------------------------------------
            float s[BN / 8][4];
#pragma unroll
            for (int n = 0; n < BN / 8; ++n) { s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f; }
            const uint32_t kst = smem_u32(sK) + stage * TILE_BYTES;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
#pragma unroll
                for (int nb = 0; nb < BN / 16; ++nb) {
                    uint32_t kf[4];
                    const int key = nb * 16 + (lane & 7) + ((lane >> 4) << 3);
                    ldsm_x4(kst + swz(key, ks * 2 + ((lane >> 3) & 1)), kf);
                    mma_bf16(s[2 * nb], qf[ks], kf[0], kf[1]);
                    mma_bf16(s[2 * nb + 1], qf[ks], kf[2], kf[3]);
                }
            }
            // ---- mask keys beyond the context (ragged last tile) ------------------------
            if (key0 + BN > p.ctx_len) {
#pragma unroll
                for (int n = 0; n < BN / 8; ++n) {
                    const int kcol = key0 + n * 8 + 2 * (lane & 3);
                    if (kcol >= p.ctx_len) { s[n][0] = -INFINITY; s[n][2] = -INFINITY; }
                    if (kcol + 1 >= p.ctx_len) { s[n][1] = -INFINITY; s[n][3] = -INFINITY; }
                }
            }
            // ---- online softmax ---------------------------------------------------------
            float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int n = 0; n < BN / 8; ++n) {
                mx[0] = fmaxf(mx[0], fmaxf(s[n][0], s[n][1]));
                mx[1] = fmaxf(mx[1], fmaxf(s[n][2], s[n][3]));
            }
            float corr[2], mneg[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 1));
                mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], 2));
                const float m_new = fmaxf(m_run[h], mx[h] * p.scale_log2);
                corr[h] = (m_run[h] == -INFINITY) ? 0.f : fast_exp2(m_run[h] - m_new);
                m_run[h] = m_new;
                mneg[h] = -m_new;
            }
            float rs[2] = {0.f, 0.f};
#pragma unroll
            for (int n = 0; n < BN / 8; ++n) {
                s[n][0] = fast_exp2(fmaf(s[n][0], p.scale_log2, mneg[0]));
                s[n][1] = fast_exp2(fmaf(s[n][1], p.scale_log2, mneg[0]));
                s[n][2] = fast_exp2(fmaf(s[n][2], p.scale_log2, mneg[1]));
                s[n][3] = fast_exp2(fmaf(s[n][3], p.scale_log2, mneg[1]));
                rs[0] += s[n][0] + s[n][1];
                rs[1] += s[n][2] + s[n][3];
            }
            l_run[0] = fmaf(l_run[0], corr[0], rs[0]);
            l_run[1] = fmaf(l_run[1], corr[1], rs[1]);
#pragma unroll
            for (int n = 0; n < D / 8; ++n) {
                o[n][0] *= corr[0]; o[n][1] *= corr[0];
                o[n][2] *= corr[1]; o[n][3] *= corr[1];
            }
            // ---- O += P V ---------------------------------------------------------------
            const uint32_t vst = smem_u32(sV) + stage * TILE_BYTES;
#pragma unroll
            for (int ks = 0; ks < BN / 16; ++ks) {
                uint32_t pf[4];
                pf[0] = pack_bf16(s[2 * ks][0], s[2 * ks][1]);
                pf[1] = pack_bf16(s[2 * ks][2], s[2 * ks][3]);
                pf[2] = pack_bf16(s[2 * ks + 1][0], s[2 * ks + 1][1]);
                pf[3] = pack_bf16(s[2 * ks + 1][2], s[2 * ks + 1][3]);
#pragma unroll
                for (int db = 0; db < D / 16; ++db) {
                    uint32_t vf[4];
                    ldsm_x4_t(vst + swz(ks * 16 + (lane & 15), db * 2 + (lane >> 4)), vf);
                    mma_bf16(o[2 * db], pf, vf[0], vf[1]);
                    mma_bf16(o[2 * db + 1], pf, vf[2], vf[3]);
                }
            }
        }
        // refreshed keys into the cache, from the landed tile: the row tiles that walk over these keys take turns
        // (nothing from a stage whose wait gave up: it holds another tile, or none; unrolled by two, as the whole loop
        // unrolled cost a partial step without fresh rows 0.16 of 7.5 us a layer)
        if (fresh && t % p.row_tiles == row_tile && !(kTma && *abort_flag)) {
#pragma unroll 2
            for (int c = tid; c < BN * CHUNKS; c += kThreads) {
                const int row = c / CHUNKS, ch = c % CHUNKS, key = key0 + row;
                if (key >= p.ctx_len || (mapped && map[key - key_lo] < 0)) continue;
                const long long at = ((long long)bh * p.ctx_len + key) * D + ch * 8;
                *reinterpret_cast<uint4*>(p.k_cache + at) = *reinterpret_cast<const uint4*>(sK + stage * TILE_BYTES + swz(row, ch));
                *reinterpret_cast<uint4*>(p.v_cache + at) = *reinterpret_cast<const uint4*>(sV + stage * TILE_BYTES + swz(row, ch));
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();   // everyone is done with the stages before they become the partial

    const bool gave_up = kTma && *abort_flag;   // a CTA whose wait gave up stores nothing

    // ---- epilogue ------------------------------------------------------------------
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 1);
        l_run[h] += __shfl_xor_sync(0xffffffffu, l_run[h], 2);
    }
    auto out_row = [&](int r) {   // where packed row r goes
        const int i = r / p.group, j = r - i * p.group;
        return p.out + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + j) * D;
    };
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = warp * 16 + (lane >> 2) + 8 * h, r = r0 + row;
        if (p.n_splits == 1) {
            if (r >= r_end || gave_up) continue;
            __nv_bfloat16* dst = out_row(r);
            const float inv = 1.f / l_run[h];
#pragma unroll
            for (int n = 0; n < D / 8; ++n) {
                const uint32_t v = pack_bf16(o[n][2 * h] * inv, o[n][2 * h + 1] * inv);
                *reinterpret_cast<uint32_t*>(dst + n * 8 + 2 * (lane & 3)) = v;
            }
        } else if (!kSpare || r < r_end) {
#pragma unroll
            for (int n = 0; n < D / 8; ++n)
                *reinterpret_cast<float2*>(part + row * PP + n * 8 + 2 * (lane & 3)) = make_float2(o[n][2 * h], o[n][2 * h + 1]);
            if ((lane & 3) == 0) s_ml[row] = make_float2(m_run[h], l_run[h]);
        }
    }
    if (p.n_splits == 1) return;

    // ---- each CTA of the cluster merges a share of the rows: out = sum_s w_s O_s / sum_s w_s l_s, w_s = 2^(m_s - max m) ----
    tc::cluster_arrive();
    tc::cluster_wait();
    const int valid = min(BM, r_end - r0), per = (valid + p.n_splits - 1) / p.n_splits;
    const int rows_here = gave_up ? 0 : min(per, valid - split * per);
    for (int idx = tid; idx < rows_here * (D / 4); idx += kThreads) {
        const int row = split * per + idx / (D / 4), ch = idx % (D / 4);
        float mm[8], ll[8], x[8][4], M = -INFINITY, L = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int src = min(q, p.n_splits - 1);
            tc::ld_peer_v2(tc::map_to_cta(smem_u32(s_ml + row), src), mm[q], ll[q]);
            tc::ld_peer_v4(tc::map_to_cta(smem_u32(part + row * PP + ch * 4), src), x[q]);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (q >= p.n_splits) mm[q] = -INFINITY;
            M = fmaxf(M, mm[q]);
        }
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float w = fast_exp2(mm[q] - M);
            L = fmaf(w, ll[q], L);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = fmaf(w, x[q][e], acc[e]);
        }
        const float inv = 1.f / L;
        *reinterpret_cast<uint2*>(out_row(r0 + row) + ch * 4) =
            make_uint2(pack_bf16(acc[0] * inv, acc[1] * inv), pack_bf16(acc[2] * inv, acc[3] * inv));
    }
    tc::cluster_arrive_relaxed();   // no CTA leaves while a peer may still read its partial
    tc::cluster_wait();
}

struct Plan {
    int row_tiles, tile_rows, n_splits, tiles_per_split, rows_total;
};
// Keys of a row tile split over up to eight CTAs (a cluster; at least one tile each) while the launch stays within the
// three CTAs an SM holds: a CTA is a serial chain of tiles (about 1 us each when nothing hides their latency).
// Several row tiles of at most 48 rows (144 rows as 3 x 48 instead of 64 + 64 + 16): the padding of the last tile is not
// computed, and the tensor core (2048 flop per clock and SM) is shared by all tiles of an SM.  9.5 -> 9.0 us for four
// sequences of 1000 keys and 48 x 3 rows, 14.8 -> 13.8 for eight of 700.  A single tile gains nothing.
Plan make_plan(const ec_attn_desc& d, int n_active) {
    Plan pl;
    const int g = d.n_q_heads / d.n_kv_heads;
    pl.rows_total = n_active * g;
    pl.row_tiles = (pl.rows_total + BM - 1) / BM;
    pl.tile_rows = pl.row_tiles > 1 && pl.rows_total <= 48 * pl.row_tiles ? 48 : BM;
    const int key_tiles = (d.ctx_len + BN - 1) / BN;
    const long long base = (long long)pl.row_tiles * d.batch * d.n_kv_heads;
    int splits = (int)(3LL * sm_count() / base);
    if (splits < 1) splits = 1;
    if (splits > 8) splits = 8;
    if (splits > key_tiles) splits = key_tiles;
    pl.tiles_per_split = (key_tiles + splits - 1) / splits;
    pl.n_splits = (key_tiles + pl.tiles_per_split - 1) / pl.tiles_per_split;
    return pl;
}

// tile maps of the cache [B, Hkv, L, 64], or of token-major fresh rows [B, L, Hkv, 64]
bool make_tile_map(CUtensorMap* map, const void* ptr, const ec_attn_desc& d, bool token_major) {
    tc::EncodeTiledFn fn = tc::encode_fn();
    if (!fn) return false;
    const cuuint64_t row = 128, L = (cuuint64_t)d.ctx_len, H = (cuuint64_t)d.n_kv_heads;
    const cuuint64_t dims[5] = {64, L, 1, H, (cuuint64_t)d.batch};
    const cuuint64_t strides[4] = {token_major ? row * H : row, row, token_major ? row : row * L, row * L * H};
    const cuuint32_t box[5] = {64, (cuuint32_t)BN, 1, 1, 1}, estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool kSpare, bool kTma>
cudaError_t launch_d64(const AttendArgs& a, const Plan& pl, const void* k_new, const void* v_new, const int32_t* active_idx,
                     cudaStream_t stream) {
    MmaParams p;
    p.q = static_cast<const __nv_bfloat16*>(a.q);
    p.k_cache = static_cast<__nv_bfloat16*>(const_cast<void*>(a.k_cache));
    p.v_cache = static_cast<__nv_bfloat16*>(const_cast<void*>(a.v_cache));
    p.k_new = static_cast<const __nv_bfloat16*>(k_new);
    p.v_new = static_cast<const __nv_bfloat16*>(v_new);
    p.active_idx = active_idx;
    p.out = static_cast<__nv_bfloat16*>(a.out);
    p.n_active = a.n_active;
    p.ctx_len = a.d.ctx_len;
    p.n_q_heads = a.d.n_q_heads;
    p.n_kv_heads = a.d.n_kv_heads;
    p.group = a.d.n_q_heads / a.d.n_kv_heads;
    p.rows_total = pl.rows_total;
    p.row_tiles = pl.row_tiles;
    p.tile_rows = pl.tile_rows;
    p.n_splits = pl.n_splits;
    p.tiles_per_split = pl.tiles_per_split;
    p.scale_log2 = a.scale * kLog2e;
    p.dev_status = a.dev_status;
    const long long ctas = (long long)a.d.batch * a.d.n_kv_heads * pl.row_tiles * pl.n_splits;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    int map_keys = k_new && active_idx ? pl.tiles_per_split * BN : 0;
    if (map_keys > kMaxMapKeys) {   // no room for the table of keys
        if (const cudaError_t e = launch_refresh(a.d, p.k_cache, p.v_cache, k_new, v_new, active_idx, a.n_active, stream);
            e != cudaSuccess)
            return e;
        p.k_new = p.v_new = nullptr;
        map_keys = 0;
    }
    constexpr int smem = (BM + 2 * ST * BN) * D * 2 + BM * (int)sizeof(float2) + 8 * (ST + 1) + (kTma ? 1024 : 0);
    static_assert(BM * (D + 8) * 4 <= 4 * BN * D * 2, "the partial of the merge fits over the stages");
    static PerDeviceOnce attr_once;
    if (const cudaError_t ea = ensure_dynamic_smem(attr_once, attend_mma_kernel<kSpare, kTma>, smem + kMaxMapKeys * 4); ea != cudaSuccess) return ea;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem + (size_t)map_keys * 4;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = pl.n_splits;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    CUtensorMap map_k{}, map_v{};
    if (kTma && (!make_tile_map(&map_k, p.k_new ? k_new : a.k_cache, a.d, p.k_new) ||
                 !make_tile_map(&map_v, p.v_new ? v_new : a.v_cache, a.d, p.v_new)))
        return cudaErrorInvalidValue;
    return cudaLaunchKernelEx(&cfg, attend_mma_kernel<kSpare, kTma>, p, map_k, map_v);
}

}  // namespace

// Fitted to 850 shapes on which this kernel and attend_dense_kernel<64> are within a factor of 1.8 of each other: 8 % rms.
double attend_mma_us(const ec_attn_desc& d, int n_active, bool fresh) {
    const Plan pl = make_plan(d, n_active);
    const double ctas = (double)pl.row_tiles * d.batch * d.n_kv_heads * pl.n_splits;
    const bool refreshes = fresh && n_active < d.ctx_len;   // (a recompute step reads its keys out of k_new)
    double rounds, us = 3.8 + (fresh ? 1.3 : 0.) + (refreshes ? 9e-5 * n_active * d.batch * d.n_kv_heads : 0.);
    if (pl.n_splits == 1) {   // 3 CTAs run on an SM at once
        const double full = ctas / (3. * sm_count());
        rounds = full <= 1. ? 1. : 0.3 * full + 0.7 * std::ceil(full);
        us += 2. * (rounds - 1.);
    } else {   // of clusters, a few fewer
        rounds = std::max(1., std::ceil(ctas / (sm_count() * (pl.n_splits == 2 ? 3. : pl.n_splits < 8 ? 2.89 : 2.76))));
        us += 1.8 * (std::min(3., std::ceil(ctas / (0.81 * sm_count()))) * rounds * pl.rows_total / pl.row_tiles / BM - 1.);   // merge
    }
    return us + pl.tiles_per_split * rounds * (refreshes ? 1.9 : 1.45);
}

cudaError_t launch_attend_bf16(const AttendArgs& a, const void* k_new, const void* v_new, const int32_t* active_idx,
                               cudaStream_t stream) {
    if (a.n_active == 0) return cudaSuccess;
    const Plan pl = make_plan(a.d, a.n_active);
    const bool spare = pl.tile_rows < BM;
    if (k_new && active_idx)
        return spare ? launch_d64<true, false>(a, pl, k_new, v_new, active_idx, stream)
                     : launch_d64<false, false>(a, pl, k_new, v_new, active_idx, stream);
    return spare ? launch_d64<true, true>(a, pl, k_new, v_new, active_idx, stream)
                 : launch_d64<false, true>(a, pl, k_new, v_new, active_idx, stream);
}

}  // namespace ec
