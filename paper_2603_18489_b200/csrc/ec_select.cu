// ec_select_recent: decode history, recent-token selection and the skip_flag / dt bookkeeping of the cached
// denoising loop on the device (Eq. 2-3 and Appendix A of the paper), so that the row list of the next partial
// step never leaves the GPU.
//
// One CTA of 512 threads per sequence.  Thread i owns the contiguous positions [i*per, (i+1)*per), held in
// registers, so one block-wide scan of the per-thread counts (window rows and members of R packed into a word)
// yields both lists in ascending order.
//   tau_R = max(min over K, t - dt) without ever finding the k largest: the k-th largest value exceeds t - dt only if
//           at least k entries do, and is then one of the dt values t - dt + 1 .. t (one above t, if k entries are:
//           the first count tells), found by bisection (a probe is one block-wide count).  Fewer than k decoded
//           positions: the minimum is "-infinity" and t - dt stands.
// What bounds it: latency.  All global loads are issued in one round (two in sliding mode, whose window rows have to be
// checked against the mask), then about eight barriers.  Bisecting over all values that occur, behind dependent loads
// and with two scans, took 6.5 us a call at L = 4096 and 8.9 in sliding mode at L = 1983 under a serialised launch.  Back to
// back in a graph a call takes 2.1 us at L = 256, 3.1 (dt = 0) to 3.5 at 4096, 3.8 in sliding mode at 1983; searched in 64
// bits it is 0.1 longer in sliding mode.  The count of the entries above t is a barrier of its own where dt = 0: 0.15 us at
// 256, 0.25 at 4096.
// The kernel has no waits; an out-of-range window (block mode) or a window list that does not consist of masked
// positions (sliding mode) leaves the sequence untouched and reports n_active = -1.
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

namespace ec {
namespace {

constexpr int kSelThreads = 512, kSelWarps = kSelThreads / 32;
constexpr int kSelMaxPer = 32;   // positions per thread: ctx_len <= 16384

struct SelectParams {
    int32_t* history;
    ec_step_state* state;
    const uint8_t* decoded;
    const int32_t* window_start;
    const int32_t* decision;
    int32_t* active_idx;
    uint8_t* masked;   // sliding-window mode: [batch, ctx_len] positions still masked (in/out); nullptr: block mode
    int ctx_len, block, k, n_cap;
};

template <int PER>   // positions per thread held in registers: ctx_len <= PER * kSelThreads
__global__ void __launch_bounds__(kSelThreads) select_recent_kernel(const SelectParams p) {
    __shared__ uint32_t scratch[2][kSelWarps];
    __shared__ uint8_t s_mask[PER * kSelThreads];   // sliding mode: 1 masked, 2 decoded in this step
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t* H = p.history + (long long)b * p.ctx_len;
    const bool sliding = p.masked != nullptr;
    uint8_t* M = sliding ? p.masked + (long long)b * p.ctx_len : nullptr;
    int32_t* idx = p.active_idx + (long long)b * p.n_cap;
    const uint8_t* dec = p.decoded + (long long)b * p.block;
    const int per = (p.ctx_len + kSelThreads - 1) / kSelThreads;
    const int i0 = tid * per;
    int turn = 0;   // which half of the scratch the next sum uses: one barrier a sum is enough
    auto block_sum = [&](uint32_t v) {
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane == 0) scratch[turn][warp] = v;
        __syncthreads();
        const uint32_t total = __reduce_add_sync(0xffffffffu, lane < kSelWarps ? scratch[turn][lane] : 0u);
        turn ^= 1;
        return (int)total;
    };
    tc::pdl_wait();
    tc::pdl_launch_dependents();

    // ---- everything that depends on nothing -----------------------------------------------------------
    ec_step_state st = p.state[b];
    const int skip = p.decision[b] == EC_SKIP ? 1 : 0;
    const int w0 = sliding ? 0 : p.window_start[b];
    int32_t h[PER];
    uint32_t mbits = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) h[j] = (j < per && i0 + j < p.ctx_len) ? H[i0 + j] : EC_H_NEVER;
    if (sliding) {
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (j < per && i0 + j < p.ctx_len && M[i0 + j] != 0) mbits |= 1u << j;
    } else if (w0 < 0 || w0 > p.ctx_len - p.block) {   // uniform over the CTA
        if (tid == 0) p.state[b].n_active = -1;
        return;
    }
    // ---- Eq. 2: the positions decoded in this step get the step's index -----------------------------
    // block mode: window row r is position w0 + r; sliding mode: it is entry r of the row list of the previous call
    if (!sliding) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int r = i0 + j - w0;
            if (j < per && i0 + j < p.ctx_len && r >= 0 && r < p.block && dec[r]) {
                h[j] = st.t;
                H[i0 + j] = st.t;
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < PER; ++j)
            if (j < per) s_mask[i0 + j] = (mbits >> j) & 1u;
        // the current window holds min(block, masked positions left) rows; the list entries behind it are recent rows,
        // not window rows, whatever their flags say
        const int n_cur = min(p.block, block_sum(__popc(mbits)));   // (its barrier also publishes s_mask)
        // The window rows must be the list the previous call (or, before the first call, the caller) wrote: in range
        // and still masked.  Anything else would credit the decoded flags to the wrong positions, so the sequence is
        // left untouched and reports n_active = -1, as an out-of-range window does in block mode.
        uint32_t bad = 0;
        for (int r = tid; r < n_cur; r += kSelThreads) {
            const int pos = idx[r];
            bad += (pos < 0 || pos >= p.ctx_len || s_mask[pos] == 0) ? 1 : 0;
        }
        if (block_sum(bad)) {   // uniform over the CTA
            if (tid == 0) p.state[b].n_active = -1;
            return;
        }
        for (int r = tid; r < n_cur; r += kSelThreads) {
            if (dec[r]) {
                const int pos = idx[r];
                H[pos] = st.t;
                M[pos] = 0;
                s_mask[pos] = 2;
            }
        }
        __syncthreads();   // (also: the old list has been read, the new one may be written)
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (j < per && s_mask[i0 + j] == 2) {
                h[j] = st.t;
                mbits &= ~(1u << j);
            }
        }
    }
    // ---- Eq. 3 ----------------------------------------------------------------------------------------
    // (all values fit 32 bits: a t - dt below them is no limit, and nothing reaches one above them, see reached below)
    const long long since = (long long)st.t - st.dt_recompute;   // t - dt
    const bool reached = p.k > 0 && since <= INT32_MAX;          // k = 0: minimum over the empty set
    int tau = reached ? (int)(since > INT32_MIN ? since : (long long)INT32_MIN) : INT32_MAX;
    if (reached) {
        // the threshold is the largest value from tau to hi that k entries reach; tau itself needs no entry
        int hi = st.t;
        // one count: entries that exceed tau and, in the upper half word, entries that exceed t, which only a loop that sets
        // t back without its history leaves behind
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < PER; ++j) c += (h[j] > tau ? 1u : 0u) + (h[j] > st.t ? 0x10000u : 0u);
        const int counts = block_sum(c);
        if (counts >> 16 >= p.k) {
            tau = max(tau, st.t + 1);
            hi = INT32_MAX;
        } else if (tau < hi) {
            if ((counts & 0xffff) >= p.k) ++tau; else hi = tau;
        }
        while (tau < hi) {
            const uint32_t gap = (uint32_t)hi - (uint32_t)tau;
            const int mid = (int)((uint32_t)tau + (gap >> 1) + (gap & 1u));
            uint32_t n = 0;
#pragma unroll
            for (int j = 0; j < PER; ++j) n += (h[j] >= mid) ? 1 : 0;   // (EC_H_NEVER is below every mid)
            if (block_sum(n) >= p.k) tau = mid; else hi = mid - 1;
        }
        tau = max(tau, INT32_MIN + 1);   // never EC_H_NEVER
    }
    // ---- the window's rows and R (outside the block in block mode; a decoded position is never in a sliding window),
    //      ascending: one exclusive scan of both counts ----
    uint32_t rbits = 0;
    if (reached) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int r = i0 + j - w0;
            const bool in_r = h[j] >= tau;
            if (in_r && (sliding || r < 0 || r >= p.block)) rbits |= 1u << j;
        }
    }
    const uint32_t mine = (uint32_t)__popc(mbits) << 16 | (uint32_t)__popc(rbits);   // at most 16384 of each
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
    }
    if (lane == 31) scratch[turn][warp] = incl;
    __syncthreads();
    const uint32_t part = lane < kSelWarps ? scratch[turn][lane] : 0u;
    const uint32_t total = __reduce_add_sync(0xffffffffu, part);
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? part : 0u) + incl - mine;
    const int n_out = (int)(total & 0xffffu);
    int n_win = p.block;
    if (!sliding) {
        for (int r = tid; r < p.block; r += kSelThreads) idx[r] = w0 + r;   // block <= n_cap (checked on the host)
    } else {
        // sliding window: the first `block` positions that are still masked (fewer when fewer remain)
        n_win = min((int)(total >> 16), p.block);
        int at = (int)(before >> 16);
        for (uint32_t bits = mbits; bits && at < p.block; bits &= bits - 1) idx[at++] = i0 + __ffs(bits) - 1;
    }
    int at = n_win + (int)(before & 0xffffu);
    for (uint32_t bits = rbits; bits && at < p.n_cap; bits &= bits - 1) idx[at++] = i0 + __ffs(bits) - 1;
    for (int r = n_win + n_out + tid; r < p.n_cap; r += kSelThreads) idx[r] = -1;
    // ---- Appendix A: skip_flag, dt, t ------------------------------------------------------------------
    if (tid == 0) {
        st.skip_flag = skip;
        st.dt_recompute = skip ? st.dt_recompute + 1 : 0;
        st.t = st.t + 1;
        st.n_active = n_win + n_out;
        p.state[b] = st;
    }
}

}  // namespace

int select_recent_max_ctx() { return kSelMaxPer * kSelThreads; }

cudaError_t launch_select_recent(int32_t* history, int ctx_len, int batch, ec_step_state* state, const uint8_t* decoded,
                                 const int32_t* window_start, int block, const int32_t* decision, int k,
                                 int32_t* active_idx, int n_cap, uint8_t* masked, cudaStream_t stream) {
    SelectParams p{history, state, decoded, window_start, decision, active_idx, masked, ctx_len, block, k, n_cap};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(batch, 1, 1);
    cfg.blockDim = dim3(kSelThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (ctx_len <= 2 * kSelThreads) return cudaLaunchKernelEx(&cfg, select_recent_kernel<2>, p);
    if (ctx_len <= 8 * kSelThreads) return cudaLaunchKernelEx(&cfg, select_recent_kernel<8>, p);
    return cudaLaunchKernelEx(&cfg, select_recent_kernel<kSelMaxPer>, p);
}

}  // namespace ec
