// ec_attend, fp32 storage: refresh and active-row bidirectional attention over the full cache (Appendix A of the paper,
// partial branch; the full branch when every row is active) in ONE launch, entirely in fp32 on the FMA pipes (the
// tolerance that goes with fp32 tensors, 1e-5 relative, rules out tf32 tensor cores).
//
//   grid    a CTA of 128 threads takes 32 (16, 8) packed query rows (active row x query heads of one kv head) and a range of
//           32-key tiles; up to eight CTAs, a cluster, split the keys of a row tile when there are few row tiles, so
//           that a partial step of a small model still spreads over the chip.
//   tile    K and V tiles come by 16-byte asynchronous copies into one of two stages.  Thread (tr, tk) = (tid / 16,
//           tid % 16) holds rows R tr .. R tr + R - 1 (R = 4, 2 or 1): it forms their scores against keys tk and tk + 16 (packed fp32x2 over even
//           and odd columns: two partial sums), the 16 threads of a row exchange maxima and sums by shuffles, and
//           probabilities go through shared memory to the same warp, which accumulates D / 16 output columns a thread.
//   refresh a key that is being refreshed is read from k_new / v_new (a table of the CTA's keys, filled from the index
//           list), so nothing waits for the cache update; the row tiles of a kv head share the writing of the cache,
//           whose refreshed rows nobody reads.
//   merge   every CTA leaves O (un-normalised), m and l of its keys in shared memory; after a cluster barrier each
//           combines a share of the rows out of its peers' memory.
// What bounds it: latency at the sizes it is for.  34 rows x 4 heads of 64 over 256 keys: 4.9 us a call (a warp per query
// row that walks over all keys, behind a refresh launch, took 30.7).  At large sizes the FMA pipe: 438 rows x 8 heads of
// four sequences 80 us (511).
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

namespace ec {
namespace {

using namespace tc;

constexpr int kThreads = 128, BN = 32;
constexpr int kMaxMapKeys = 8192;   // keys of one CTA beyond which the refresh is a launch of its own

struct F32Params {
    const float *q, *k_new, *v_new;
    float *k_cache, *v_cache, *out;
    const int32_t* active_idx;
    int n_active, ctx_len, n_q_heads, n_kv_heads, group, rows_total, row_tiles, n_splits, tiles_per_split;
    float scale;
};

// shared memory, in floats (D-float rows padded by four: eight rows read as float4 then cover all banks)
template <int D, int R>
struct Carve {
    static constexpr int BM = 8 * R;
    static constexpr int P = D + 4;
    static constexpr int q = 0, kv = q + BM * P, stage = 2 * BN * P, p = kv + 2 * stage, pp = BN + 4;
    static constexpr int ml = p + BM * pp, map = ml + 2 * BM;
    static constexpr int part = kv;   // the partial of the merge, over the stages: [BM][D]
    static size_t bytes(int map_keys) { return (size_t)(map + map_keys) * 4; }
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    const int sz = valid ? 16 : 0;   // 0: the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}

// R: query rows of a thread, an eighth of the CTA's
template <int D, int R>
__global__ void __launch_bounds__(kThreads) attend_f32_kernel(const F32Params p) {
    using C = Carve<D, R>;
    constexpr int BM = 8 * R;
    constexpr int D4 = D / 4, OC = D / 16;   // float4 pieces of a row; output columns of a thread
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, tr = tid >> 4, tk = tid & 15;
    const int split = blockIdx.x % p.n_splits, unit = blockIdx.x / p.n_splits;
    const int row_tile = unit % p.row_tiles, bh = unit / p.row_tiles;
    const int b = bh / p.n_kv_heads, hk = bh % p.n_kv_heads;
    const int r0 = row_tile * BM;
    const int n_tiles = (p.ctx_len + BN - 1) / BN;
    const int t0 = split * p.tiles_per_split, t1 = min(n_tiles, t0 + p.tiles_per_split);
    const int key_lo = t0 * BN, key_hi = min(p.ctx_len, t1 * BN);
    const bool fresh = p.k_new != nullptr;
    const bool mapped = fresh && p.active_idx != nullptr;
    int* map = reinterpret_cast<int*>(sm + C::map);   // [key of this CTA]: active row that refreshes it, or -1
    if (mapped)
        for (int k = tid; k < key_hi - key_lo; k += kThreads) map[k] = -1;
    // where this thread's pieces of Q are (two divisions each: before the wait, not behind it), -1: no such row
    constexpr int QN = BM * D4 / kThreads;
    long long q_at[QN];
#pragma unroll
    for (int k = 0; k < QN; ++k) {
        const int c = tid + k * kThreads, r = r0 + c / D4, i = r / p.group, j = r - i * p.group;
        q_at[k] = r < p.rows_total ? (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + j) * D + c % D4 * 4 : -1;
    }
    const float *kc = p.k_cache + (long long)bh * p.ctx_len * D, *vc = p.v_cache + (long long)bh * p.ctx_len * D;
    const long long new0 = ((long long)b * p.n_active * p.n_kv_heads + hk) * D;
    const int new_stride = p.n_kv_heads * D;
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();

#pragma unroll
    for (int k = 0; k < QN; ++k) {
        const int c = tid + k * kThreads;
        cp_async16(s2u(sm + C::q + c / D4 * C::P + c % D4 * 4), p.q + max(q_at[k], 0LL), q_at[k] >= 0);
    }
    if (mapped) {
        for (int i = tid; i < p.n_active; i += kThreads) {
            const int k = __ldg(p.active_idx + (long long)b * p.n_active + i) - key_lo;
            if (k >= 0 && k < key_hi - key_lo) map[k] = i;
        }
        __syncthreads();
    }
    // the fresh row behind a key of this CTA, or -1
    auto fresh_row = [&](int key) { return !fresh ? -1 : mapped ? map[key - key_lo] : key; };
    auto load_kv = [&](int t, int stage) {
        float* ks = sm + C::kv + stage * C::stage;
        for (int c = tid; c < BN * D4; c += kThreads) {
            const int row = c / D4, ch = c % D4, key = t * BN + row;
            const bool ok = key < p.ctx_len;
            const float *ksrc = kc, *vsrc = vc;
            if (ok) {
                const int i = fresh_row(key);
                const long long at = i < 0 ? (long long)key * D : new0 + (long long)i * new_stride;
                ksrc = (i < 0 ? kc : p.k_new) + at + ch * 4;
                vsrc = (i < 0 ? vc : p.v_new) + at + ch * 4;
            }
            cp_async16(s2u(ks + row * C::P + ch * 4), ksrc, ok);
            cp_async16(s2u(ks + (BN + row) * C::P + ch * 4), vsrc, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (t0 < t1) load_kv(t0, 0);

    float m[R], l[R], o[R][OC];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        m[r] = -INFINITY;
        l[r] = 0.f;
#pragma unroll
        for (int c = 0; c < OC; ++c) o[r][c] = 0.f;
    }
    for (int t = t0; t < t1; ++t) {
        const int stage = (t - t0) & 1;
        if (t + 1 < t1) {
            load_kv(t + 1, stage ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float *ks = sm + C::kv + stage * C::stage, *vs = ks + BN * C::P;
        // ---- scores of R rows against two keys ----
        f32x2 acc[R][2];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = pk(0.f, 0.f);
#pragma unroll 4
        for (int ch = 0; ch < D4; ++ch) {
            const ulonglong2 k0 = *reinterpret_cast<const ulonglong2*>(ks + tk * C::P + ch * 4);
            const ulonglong2 k1 = *reinterpret_cast<const ulonglong2*>(ks + (tk + 16) * C::P + ch * 4);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(sm + C::q + (R * tr + r) * C::P + ch * 4);
                acc[r][0] = fma2(qv.y, k0.y, fma2(qv.x, k0.x, acc[r][0]));
                acc[r][1] = fma2(qv.y, k1.y, fma2(qv.x, k1.x, acc[r][1]));
            }
        }
        const bool in0 = t * BN + tk < p.ctx_len, in1 = t * BN + tk + 16 < p.ctx_len;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float a0, a1, b0, b1;
            upk(acc[r][0], a0, a1);
            upk(acc[r][1], b0, b1);
            const float s0 = in0 ? (a0 + a1) * p.scale : -INFINITY, s1 = in1 ? (b0 + b1) * p.scale : -INFINITY;
            float mx = fmaxf(s0, s1);
#pragma unroll
            for (int d = 8; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            const float m_new = fmaxf(m[r], mx);   // finite: every tile holds a key of the context
            const float corr = m[r] == -INFINITY ? 0.f : expf(m[r] - m_new);
            const float p0 = in0 ? expf(s0 - m_new) : 0.f, p1 = in1 ? expf(s1 - m_new) : 0.f;
            float sum = p0 + p1;
#pragma unroll
            for (int d = 8; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
            l[r] = fmaf(l[r], corr, sum);
            m[r] = m_new;
#pragma unroll
            for (int c = 0; c < OC; ++c) o[r][c] *= corr;
            sm[C::p + (R * tr + r) * C::pp + tk] = p0;
            sm[C::p + (R * tr + r) * C::pp + tk + 16] = p1;
        }
        __syncwarp();   // the probabilities of a row are written and read by the same warp
        // ---- O += P V: output columns 4 tk .. 4 tk + 3 (and 64 + 4 tk .. for D = 128) ----
#pragma unroll 2
        for (int k4 = 0; k4 < BN; k4 += 4) {
            float4 pr[R];
#pragma unroll
            for (int r = 0; r < R; ++r) pr[r] = *reinterpret_cast<const float4*>(sm + C::p + (R * tr + r) * C::pp + k4);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int c = 0; c < OC; c += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(vs + (k4 + k) * C::P + c * 16 + 4 * tk);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float pv = k == 0 ? pr[r].x : k == 1 ? pr[r].y : k == 2 ? pr[r].z : pr[r].w;
                        o[r][c] = fmaf(pv, v.x, o[r][c]);
                        o[r][c + 1] = fmaf(pv, v.y, o[r][c + 1]);
                        o[r][c + 2] = fmaf(pv, v.z, o[r][c + 2]);
                        o[r][c + 3] = fmaf(pv, v.w, o[r][c + 3]);
                    }
                }
            }
        }
        // refreshed keys into the cache, from the landed tile: the row tiles that walk over these keys take turns
        if (fresh && t % p.row_tiles == row_tile) {
            for (int c = tid; c < BN * D4; c += kThreads) {
                const int row = c / D4, ch = c % D4, key = t * BN + row;
                if (key >= p.ctx_len || fresh_row(key) < 0) continue;
                const long long at = ((long long)bh * p.ctx_len + key) * D + ch * 4;
                *reinterpret_cast<float4*>(p.k_cache + at) = *reinterpret_cast<const float4*>(ks + row * C::P + ch * 4);
                *reinterpret_cast<float4*>(p.v_cache + at) = *reinterpret_cast<const float4*>(vs + row * C::P + ch * 4);
            }
        }
        __syncthreads();   // everyone is done with this stage before it is refilled (or becomes the partial)
    }

    auto out_row = [&](int r) {   // where packed row r goes
        const int i = r / p.group, j = r - i * p.group;
        return p.out + (((long long)b * p.n_active + i) * p.n_q_heads + hk * p.group + j) * D;
    };
    if (p.n_splits == 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (r0 + R * tr + r >= p.rows_total) continue;
            float* dst = out_row(r0 + R * tr + r);
            const float inv = 1.f / l[r];
#pragma unroll
            for (int c = 0; c < OC; c += 4)
                *reinterpret_cast<float4*>(dst + c * 16 + 4 * tk) =
                    make_float4(o[r][c] * inv, o[r][c + 1] * inv, o[r][c + 2] * inv, o[r][c + 3] * inv);
        }
        return;
    }
    // ---- partial of this CTA, then each CTA of the cluster merges its share of the rows ----
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int c = 0; c < OC; c += 4)
            *reinterpret_cast<float4*>(sm + C::part + (R * tr + r) * D + c * 16 + 4 * tk) =
                make_float4(o[r][c], o[r][c + 1], o[r][c + 2], o[r][c + 3]);
        if (tk == 0) *reinterpret_cast<float2*>(sm + C::ml + 2 * (R * tr + r)) = make_float2(m[r], l[r]);
    }
    cluster_arrive();
    cluster_wait();
    const int per = (BM + p.n_splits - 1) / p.n_splits;   // rows merged by one CTA
    const int rows_here = min(per, min(BM, p.rows_total - r0) - split * per);
    for (int idx = tid; idx < rows_here * D4; idx += kThreads) {
        const int row = split * per + idx / D4, ch = idx % D4;
        float mm[8], ll[8], x[8][4], M = -INFINITY, L = 0.f;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int src = min(s, p.n_splits - 1);
            ld_peer_v2(map_to_cta(s2u(sm + C::ml + 2 * row), src), mm[s], ll[s]);
            ld_peer_v4(map_to_cta(s2u(sm + C::part + row * D + ch * 4), src), x[s]);
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            if (s >= p.n_splits) mm[s] = -INFINITY;
            M = fmaxf(M, mm[s]);
        }
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const float e = mm[s] == -INFINITY ? 0.f : expf(mm[s] - M);
            L = fmaf(e, ll[s], L);
            a.x = fmaf(e, x[s][0], a.x);
            a.y = fmaf(e, x[s][1], a.y);
            a.z = fmaf(e, x[s][2], a.z);
            a.w = fmaf(e, x[s][3], a.w);
        }
        const float inv = 1.f / L;
        *reinterpret_cast<float4*>(out_row(r0 + row) + ch * 4) = make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv);
    }
    cluster_arrive_relaxed();   // no CTA leaves while a peer may still read its partial
    cluster_wait();
}

template <int D, int R>
cudaError_t launch_d(const F32Params& p, int batch, cudaStream_t stream) {
    static PerDeviceOnce once;
    const size_t smem = Carve<D, R>::bytes(p.k_new && p.active_idx ? p.tiles_per_split * BN : 0);
    if (const cudaError_t e = ensure_dynamic_smem(once, attend_f32_kernel<D, R>, (int)Carve<D, R>::bytes(kMaxMapKeys)); e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((long long)batch * p.n_kv_heads * p.row_tiles * p.n_splits), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = p.n_splits;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attend_f32_kernel<D, R>, p);
}

}  // namespace

cudaError_t launch_attend_f32(const AttendArgs& a, const void* k_new, const void* v_new, const int32_t* active_idx,
                              cudaStream_t stream) {
    if (a.n_active == 0) return cudaSuccess;
    F32Params p{};
    p.q = static_cast<const float*>(a.q);
    p.k_new = static_cast<const float*>(k_new);
    p.v_new = static_cast<const float*>(v_new);
    p.k_cache = static_cast<float*>(const_cast<void*>(a.k_cache));
    p.v_cache = static_cast<float*>(const_cast<void*>(a.v_cache));
    p.out = static_cast<float*>(a.out);
    p.active_idx = active_idx;
    p.n_active = a.n_active;
    p.ctx_len = a.d.ctx_len;
    p.n_q_heads = a.d.n_q_heads;
    p.n_kv_heads = a.d.n_kv_heads;
    p.group = a.d.n_q_heads / a.d.n_kv_heads;
    p.rows_total = a.n_active * p.group;
    p.scale = a.scale;
    // The keys of a row tile are split over as many CTAs (at most eight, at least a tile each) as keep the launch within
    // four CTAs per SM, which is what shared memory leaves room for.  A row tile has 32 rows, or 16 while such a launch
    // has two CTAs per SM at most, or 8 while it has one: a CTA's time is its threads' rows times its key tiles, but every
    // row tile reads the keys again and waits for its SM's other ones.  (34 rows x 256 keys x 4 heads: 4.9 us with 16 rows,
    // 5.1 with 8, 160 CTAs, 5.8 with 32; 40 rows x 400 keys x 12 heads 8.5 with 16, 11.6 with 8, 10.9 with 32.)
    const int n_tiles = (a.d.ctx_len + BN - 1) / BN;
    const long long heads = (long long)a.d.batch * a.d.n_kv_heads;
    long long units = 0;
    int R = 1, splits = 1;
    for (;; R *= 2) {
        p.row_tiles = (p.rows_total + 8 * R - 1) / (8 * R);
        units = heads * p.row_tiles;
        splits = n_tiles < 8 ? n_tiles : 8;
        if (R == 4 || units * splits <= (long long)R * sm_count()) break;
    }
    if (units * splits > 4LL * sm_count()) splits = (int)(4LL * sm_count() / units);
    if (splits < 1) splits = 1;
    p.tiles_per_split = (n_tiles + splits - 1) / splits;
    p.n_splits = (n_tiles + p.tiles_per_split - 1) / p.tiles_per_split;
    if (units * p.n_splits > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    if (k_new && active_idx && p.tiles_per_split * BN > kMaxMapKeys) {   // no room for the table of keys
        if (const cudaError_t e = launch_refresh(a.d, p.k_cache, p.v_cache, k_new, v_new, active_idx, a.n_active, stream);
            e != cudaSuccess)
            return e;
        p.k_new = p.v_new = nullptr;
    }
    if (a.d.head_dim == 64)
        return R == 1 ? launch_d<64, 1>(p, a.d.batch, stream) : R == 2 ? launch_d<64, 2>(p, a.d.batch, stream) : launch_d<64, 4>(p, a.d.batch, stream);
    return R == 1 ? launch_d<128, 1>(p, a.d.batch, stream) : R == 2 ? launch_d<128, 2>(p, a.d.batch, stream) : launch_d<128, 4>(p, a.d.batch, stream);
}

}  // namespace ec
