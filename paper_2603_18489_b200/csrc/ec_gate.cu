// ec_entropy_gate: one streaming pass over the logits (Eq. 1 of the paper) that
// yields, per row, argmax / confidence / Shannon entropy, then the maximum
// entropy over the rows flagged "newly decoded" and its comparison with tau
// (Algorithm 1: E > tau -> recompute, else skip).
//
// R*V*sizeof(elem) bytes are read exactly once; the arithmetic is about seven instructions per element.
//   grid  : a CTA owns one chunk of columns of one row; rows have s or s + 1 chunks, so that the CTAs are one resident wave
//           without a place left over (4 CTAs of 256 threads per SM), see plan_chunks;
//   loop  : a thread takes the 16-byte vectors (bf16x8 / f32x4) t, t + 256, ... of the chunk in ascending
//           order through four rolling registers and keeps a running
//           (max, S, T) with S = sum 2^d, T = sum 2^d * d, d = x*log2(e) - base: one ex2.approx per element
//           and one packed fp32x2 FMA, add and FMA per pair of elements.  The base follows the maximum lazily: it moves, and S and T
//           are rescaled (S' = 2^dl S, T' = 2^dl (T + dl S), dl = old base - new base), only when a value
//           exceeds it by more than 2^64 (looked at once per pair of bf16 vectors), so the common path has one branch.  Logits are
//           clamped from below at -1e38 (packed bf16 max on the raw words), which keeps d finite:
//           -inf and finfo.min-style masks get probability 0 without a per-element special case;
//   argmax: the thread remembers the vector that raised its maximum; after the warp's maximum is
//           known, only the threads that attained it look at that vector again for the
//           first column (ties -> smallest index, through every reduction stage);
//   reduce: sums rescaled to the warp's base and added (shuffles), the warps' results merged behind one barrier;
//   merge : CTA partial (M, S, T, idx) -> workspace, one atomic ticket; the last CTA of a sequence
//           (no spinning: tickets only count arrivals) merges the partials of every row of the
//           sequence, writes H = ln S - ln2 * T / S, conf = 2^(M*log2e - base) / S and argmax, takes
//           the flagged maximum and the decision.  Sequences of more than 64 rows, or rows cut into more
//           than 32 splits, use two ticket levels instead (last CTA of a row, then last row of the sequence).
// The entropy identity used: with p_j = 2^{d_j} / S,  -sum p_j ln p_j = ln S - ln2 * T / S
// for any common base, so no partial ever needs the true row maximum.
// What bounds it: a call is about 5.5 us (launch, ramp, reduction, ticket, the finishing CTA) and its bytes at 6.1 TB/s for
// bf16, 7.4 for fp32 (from 288 and 576 rows, 256 rows of one and two chunks): [256, 126464] bf16 17.1 us, [32, 126464] 7.2;
// the decode mode, whose finishing CTA has the decoded set to form, 18.5 to 19.0.
// Of the 7.8 us above the 9.9 of its transfer (17.7, before pairs) 2.3 were arithmetic (16.9 without the exponentials, 15.4
// without any) and 5.5 the fixed part, whose pieces have not been timed apart.  Also timed at [256, 126464]: twelve vectors ahead through
// asynchronous copies 17.9 (fp32 26.6 against 24.2), two batches of four in registers 18.6, 3 to 21 CTAs a row 19.5 to
// 38, five CTAs per SM of 48 registers 20.4, sums of their own for the second vector of a pair 17.2, 592 equal shares
// that cross from row to row no better (224 rows 17.1 against 16.8, 160 rows 13.9 against 13.1); a ring of bulk copies
// with a producer warp 19.7, and 7.4 at [32, 126464].
// The kernel is launched with programmatic stream serialisation, touches global memory only after
// griddepcontrol.wait and waits for nothing else.
#include "ec_common.cuh"
#include "ec_tc_ptx.cuh"

#include <float.h>

#include <algorithm>

namespace ec {
namespace {

constexpr int kGateThreads = 256;
constexpr int kCtasPerSm = 4;
constexpr int kVec = 8;      // columns per thread in one slab of kGateThreads * kVec columns
constexpr int kPiece = 256;  // chunks of unequal rows are multiples of this many columns
constexpr int kMaxSplits = 96;
constexpr float kDClamp = -150.0f;  // 2^-150 flushes to 0 (ftz)
constexpr int kInFlight = 4;         // 16-byte vectors a thread keeps in flight
constexpr int kSingleLevelMaxRows = 64;
constexpr int kFinishSplits = 32;    // chunks of a row that the last CTA of a sequence finishes: eight threads a row, four each
constexpr float kRebase = 64.f;     // the base moves when a value exceeds it by more than 2^kRebase
constexpr unsigned int kXMinBf16x2 = 0xFE96FE96u;   // two bf16 of about -1e38: lower clamp of the logits
constexpr unsigned int kXMinF32 = 0xFE960000u;      // the same value as fp32 bits

struct Partial {
    float M;  // maximum of the chunk (clamped logits)
    float S;  // sum 2^(x*log2e - base(M))
    float T;  // sum 2^(..) * (x*log2e - base(M))
    int idx;  // first column attaining M
};

__device__ __forceinline__ float base_of(float M) { return fmaxf(M * kLog2e, -3.0e38f); }

__device__ __forceinline__ Partial merge(Partial a, Partial b) {
    const bool a_wins = (a.M > b.M) || (a.M == b.M && a.idx <= b.idx);
    Partial hi = a_wins ? a : b;
    const Partial lo = a_wins ? b : a;
    const float dl = base_of(lo.M) - base_of(hi.M);  // <= 0
    if (lo.S > 0.f && dl > kDClamp) {
        const float c = fast_exp2(dl);
        hi.S = fmaf(c, lo.S, hi.S);
        hi.T = fmaf(c, fmaf(dl, lo.S, lo.T), hi.T);
    }
    return hi;
}

// ticket: release (the partial written just before by this thread is visible to whoever sees the count) and
// acquire (whoever completes the count sees every earlier partial)
__device__ __forceinline__ int ticket_add(int* addr, int v) {
    int old;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(old) : "l"(addr), "r"(v) : "memory");
    return old;
}
// packed pairs of fp32 (one 64-bit register): two lanes per FMA / add issue slot
using tc::add2;
using tc::f32x2;
using tc::fma2;
using tc::pk;
using tc::upk;
__device__ __forceinline__ unsigned int max_bf16x2(unsigned int a, unsigned int b) {
    unsigned int d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// One 16-byte vector of a row: EPV elements, kept raw (packed) while in flight.
//   clamp()    lower clamp of all elements, on the raw words
//   vec_max()  maximum of the (clamped) vector as fp32
//   widen()    raw -> fp32
template <typename T>
struct Loader;

template <>
struct Loader<__nv_bfloat16> {
    static constexpr int EPV = 8;
    static __device__ __forceinline__ void clamp(uint4& u) {
        u.x = max_bf16x2(u.x, kXMinBf16x2); u.y = max_bf16x2(u.y, kXMinBf16x2);
        u.z = max_bf16x2(u.z, kXMinBf16x2); u.w = max_bf16x2(u.w, kXMinBf16x2);
    }
    static __device__ __forceinline__ unsigned int max_word(const uint4& u) {
        return max_bf16x2(max_bf16x2(u.x, u.y), max_bf16x2(u.z, u.w));
    }
    static __device__ __forceinline__ unsigned int max_words(unsigned int a, unsigned int b) { return max_bf16x2(a, b); }
    static __device__ __forceinline__ float word_max(unsigned int w) {
        return fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
    static __device__ __forceinline__ void widen(const uint4& u, float (&x)[8]) {
        const unsigned int w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            x[2 * i] = __uint_as_float(w[i] << 16);
            x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ void widen2(const uint4& u, f32x2 (&x)[4]) {
        const unsigned int w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = pk(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
    }
    static __device__ __forceinline__ float one(const __nv_bfloat16* p) {
        return fmaxf(__bfloat162float(*p), __uint_as_float(kXMinF32));
    }
};

template <>
struct Loader<float> {
    static constexpr int EPV = 4;
    static __device__ __forceinline__ void clamp(uint4& u) {
        const float lo = __uint_as_float(kXMinF32);
        u.x = __float_as_uint(fmaxf(__uint_as_float(u.x), lo)); u.y = __float_as_uint(fmaxf(__uint_as_float(u.y), lo));
        u.z = __float_as_uint(fmaxf(__uint_as_float(u.z), lo)); u.w = __float_as_uint(fmaxf(__uint_as_float(u.w), lo));
    }
    // "word" = one fp32 value here
    static __device__ __forceinline__ unsigned int max_word(const uint4& u) {
        return __float_as_uint(fmaxf(fmaxf(__uint_as_float(u.x), __uint_as_float(u.y)),
                                     fmaxf(__uint_as_float(u.z), __uint_as_float(u.w))));
    }
    static __device__ __forceinline__ unsigned int max_words(unsigned int a, unsigned int b) {
        return __float_as_uint(fmaxf(__uint_as_float(a), __uint_as_float(b)));
    }
    static __device__ __forceinline__ float word_max(unsigned int w) { return __uint_as_float(w); }
    static __device__ __forceinline__ void widen(const uint4& u, float (&x)[4]) {
        x[0] = __uint_as_float(u.x); x[1] = __uint_as_float(u.y);
        x[2] = __uint_as_float(u.z); x[3] = __uint_as_float(u.w);
    }
    static __device__ __forceinline__ void widen2(const uint4& u, f32x2 (&x)[2]) {
        x[0] = pk(__uint_as_float(u.x), __uint_as_float(u.y));
        x[1] = pk(__uint_as_float(u.z), __uint_as_float(u.w));
    }
    static __device__ __forceinline__ float one(const float* p) { return fmaxf(*p, __uint_as_float(kXMinF32)); }
};

struct GateParams {
    const void* logits;
    long long row_stride;
    int n_rows, vocab, rows_per_seq;
    // the first n_few rows are cut into `splits` chunks of chunk[0] columns, the others into one more, of chunk[1]
    int n_few, splits, chunk[2];
    unsigned int inverse[2];   // ceil(2^32 / splits), ceil(2^32 / (splits + 1)): quotients of a block index (below 2^23) by mulhi
    int pitch;          // partials of a row
    int single_level;   // 1: the last CTA of a sequence finishes all its rows; 0: per-row then per-sequence tickets
    const uint8_t* flags;
    float tau;
    int* argmax_out;
    float* conf_out;
    float* entropy_out;  // never null inside the kernel (workspace scratch if the caller gave none)
    float* max_entropy_out;
    int* decision_out;
    int* row_ticket;  // [n_rows], zero on entry, zero on exit
    int* seq_ticket;  // [n_seq],  zero on entry, zero on exit
    Partial* partials;  // [n_rows, pitch]
    // decode mode (masked != nullptr, single_level only): the decoded set comes from the confidences
    uint8_t* masked;       // in/out [n_rows]: rows still masked; cleared for the rows decoded here
    float conf_thr;
    uint8_t* decoded_out;  // [n_rows]
    int* tokens;           // [n_rows]: argmax written for the decoded rows
    // Section 5.3's other candidate metrics over the decoded rows (single_level only; either may be null)
    float* ent_sum_out;    // [n_seq]
    float* max_conf_out;   // [n_seq]
};

template <bool kUneven>
__device__ __forceinline__ int splits_of(const GateParams& p, int row) { return p.splits + (kUneven && row >= p.n_few ? 1 : 0); }
__device__ __forceinline__ const Partial* partials_of(const GateParams& p, int row) { return p.partials + (long long)row * p.pitch; }

// warp-collective: merge the split partials of one row, write the row's outputs, return its entropy (all lanes)
template <bool kUneven>
__device__ __forceinline__ float finish_row(const GateParams& p, int row, int lane) {
    Partial acc;
    acc.M = -INFINITY; acc.S = 0.f; acc.T = 0.f; acc.idx = 0x7fffffff;
    const int n = splits_of<kUneven>(p, row);
    for (int s = lane; s < n; s += 32) {
        const float4 f = __ldcg(reinterpret_cast<const float4*>(partials_of(p, row) + s));
        Partial q;
        q.M = f.x; q.S = f.y; q.T = f.z; q.idx = __float_as_int(f.w);
        acc = merge(acc, q);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Partial q;
        q.M = __shfl_xor_sync(0xffffffffu, acc.M, o);
        q.S = __shfl_xor_sync(0xffffffffu, acc.S, o);
        q.T = __shfl_xor_sync(0xffffffffu, acc.T, o);
        q.idx = __shfl_xor_sync(0xffffffffu, acc.idx, o);
        acc = merge(acc, q);
    }
    const float H = fmaxf(logf(acc.S) - kLn2 * acc.T / acc.S, 0.f);
    if (lane == 0) {
        const float conf = fast_exp2(fmaf(acc.M, kLog2e, -base_of(acc.M))) / acc.S;
        if (p.argmax_out) p.argmax_out[row] = acc.idx;
        if (p.conf_out) p.conf_out[row] = conf;
        p.entropy_out[row] = H;
    }
    return H;
}

// kUneven: rows of splits or splits + 1 chunks on a grid of one dimension; otherwise (splits, rows).  (One kernel for both cost
// the even launches 1 to 4 %.)
template <typename T, bool kUneven>
__global__ void __launch_bounds__(kGateThreads, kCtasPerSm) gate_kernel(const GateParams p) {
    constexpr int kWarps = kGateThreads / 32;
    __shared__ float4 s_part[kWarps];
    __shared__ float s_H[kSingleLevelMaxRows];
    __shared__ float s_conf[kSingleLevelMaxRows];
    __shared__ int s_arg[kSingleLevelMaxRows];
    __shared__ int s_last;

    using L = Loader<T>;
    constexpr int EPV = L::EPV;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the rows with fewer and larger chunks come first: the SMs are dealt the large chunks, then the small ones
    int row = blockIdx.y, split = blockIdx.x, n_splits = p.splits, chunk = p.chunk[0];
    if (kUneven && p.pitch > p.splits) {   // (always; without the second condition the instance spills and is 1 to 2 % slower)
        const int few = p.n_few * p.splits;
        const bool more = split >= few;
        const int at = more ? split - few : split;
        row = (int)__umulhi((unsigned)at, more ? p.inverse[1] : p.inverse[0]);
        if (n_splits == 1 && !more) row = at;
        if (more) ++n_splits, chunk = p.chunk[1];
        split = at - row * n_splits;
        if (more) row += p.n_few;
    }
    const T* rowp = reinterpret_cast<const T*>(p.logits) + (long long)row * p.row_stride;
    const int c0 = split * chunk;
    const int c_end = min(p.vocab, c0 + chunk);

    // Thread t owns the whole vectors t, t + 256, ... of the chunk.  They pass through a rolling set of kInFlight registers:
    // as soon as a vector has been consumed its register is given to the load kInFlight vectors ahead.  The ragged end
    // of a row (a vocabulary that is no multiple of the vector length) is handled by element below.
    constexpr int kVStride = kGateThreads * EPV;
    const int n_vec = (c_end - c0) / EPV;
    const int n_mine = n_vec > tid ? (n_vec - tid + kGateThreads - 1) / kGateThreads : 0;
    const T* mine = rowp + c0 + tid * EPV;
    uint4 raw[kInFlight];
    auto fetch = [&](int i, uint4& v) {
        if (i < n_mine) v = __ldcs(reinterpret_cast<const uint4*>(mine + (long long)i * kVStride));   // streamed once
    };
    tc::pdl_wait();                 // the previous kernel of the stream has completed: the logits are final
    tc::pdl_launch_dependents();
#pragma unroll
    for (int r = 0; r < kInFlight; ++r) fetch(r, raw[r]);

    // running state: maximum, exponent base, and S, T as two packed lanes each
    float m = -INFINITY, base = base_of(-INFINITY);
    f32x2 S2 = pk(0.f, 0.f), T2 = pk(0.f, 0.f);
    int mat = -1;               // the vector (the first of the pair) that raised the maximum last
    const f32x2 kL2 = pk(kLog2e, kLog2e);
    auto rebase_if_needed = [&](float vmax) {
        if (fmaf(vmax, kLog2e, -base) > kRebase) {   // rare
            const float nb = base_of(vmax);
            const float dl = fmaxf(base - nb, kDClamp);
            const float c = fast_exp2(dl);
            float s0, s1, t0, t1;
            upk(S2, s0, s1);
            upk(T2, t0, t1);
            t0 = s0 > 0.f ? c * fmaf(dl, s0, t0) : 0.f;
            t1 = s1 > 0.f ? c * fmaf(dl, s1, t1) : 0.f;
            S2 = pk(s0 * c, s1 * c);
            T2 = pk(t0, t1);
            base = nb;
        }
    };
    auto add = [&](const uint4& v) {
        const f32x2 nb2 = pk(-base, -base);
        f32x2 x2[EPV / 2];
        L::widen2(v, x2);
#pragma unroll
        for (int e = 0; e < EPV / 2; ++e) {
            const f32x2 d2 = fma2(x2[e], kL2, nb2);
            float d0, d1;
            upk(d2, d0, d1);
            const f32x2 e2 = pk(fast_exp2(d0), fast_exp2(d1));
            S2 = add2(S2, e2);
            T2 = fma2(e2, d2, T2);
        }
    };
    auto raise = [&](float vmax, int i) {
        rebase_if_needed(vmax);
        mat = vmax > m ? i : mat;   // strictly greater: the first vectors of a tie survive
        m = fmaxf(m, vmax);
    };
    // bf16: two vectors behind one look at the maximum, which is a branch that the exponentials of one vector and the
    // clamps and maxima of the next cannot cross ([256, 126464] 17.7 -> 17.1 us); fp32 waits for memory and for the
    // second of two vectors the longer (22.6 -> 23.2)
    constexpr bool kPairs = EPV == 8;
    auto consume2 = [&](uint4 v, uint4 w, int i) {   // vectors i and i + 1
        L::clamp(v);
        L::clamp(w);
        raise(L::word_max(L::max_words(L::max_word(v), L::max_word(w))), i);
        add(v);
        add(w);
    };
    auto consume = [&](uint4 v, int i) {             // (pairs: the last vector of an odd number)
        L::clamp(v);
        raise(L::word_max(L::max_word(v)), i);
        add(v);
    };
    int i0 = 0;
    for (; i0 + kInFlight <= n_mine; i0 += kInFlight) {
#pragma unroll
        for (int r = 0; r < kInFlight; r += 2) {
            if (kPairs) consume2(raw[r], raw[r + 1], i0 + r);
            else consume(raw[r], i0 + r);
            fetch(i0 + r + kInFlight, raw[r]);
            if (!kPairs) consume(raw[r + 1], i0 + r + 1);
            fetch(i0 + r + 1 + kInFlight, raw[r + 1]);
        }
    }
#pragma unroll
    for (int r = 0; r < kInFlight; r += 2) {
        if (kPairs && i0 + r + 1 < n_mine) {
            consume2(raw[r], raw[r + 1], i0 + r);
        } else {
            if (i0 + r < n_mine) consume(raw[r], i0 + r);
            if (!kPairs && i0 + r + 1 < n_mine) consume(raw[r + 1], i0 + r + 1);
        }
    }
    int tail_col = -1;
    {   // the ragged end of the chunk: fewer than EPV columns, one element per thread
        const int col = c0 + n_vec * EPV + tid;
        if (col < c_end) {
            const float x = L::one(rowp + col);
            rebase_if_needed(x);
            tail_col = x > m ? col : -1;
            m = fmaxf(m, x);
            float s0, s1, t0, t1;
            upk(S2, s0, s1);
            upk(T2, t0, t1);
            const float d = fmaf(x, kLog2e, -base);
            const float e = fast_exp2(d);
            S2 = pk(s0 + e, s1);
            T2 = pk(fmaf(e, d, t0), t1);
        }
    }

    // ---- warp maximum; the threads that attained it find its first column in the vector that raised it --------
    // (every thread asks again for that vector or pair: an L2 hit, in flight during the reduction)
    constexpr int kAgain = kPairs ? 2 : 1;
    uint4 again[kAgain];
    if (mat >= 0) {
#pragma unroll
        for (int k = 0; k < kAgain; ++k)
            again[k] = __ldg(reinterpret_cast<const uint4*>(mine + (long long)min(mat + k, n_mine - 1) * kVStride));
    }
    const float M = tc::redux_max(m);
    int idx = 0x7fffffff;
    if (m == M) {
        if (tail_col >= 0) {
            idx = tail_col;
        } else if (mat >= 0) {
#pragma unroll
            for (int k = kAgain - 1; k >= 0; --k) {   // descending: the smallest column survives
                float x[EPV];
                L::clamp(again[k]);
                L::widen(again[k], x);
#pragma unroll
                for (int e = EPV - 1; e >= 0; --e)
                    if (x[e] == M) idx = c0 + min(mat + k, n_mine - 1) * kVStride + tid * EPV + e;
            }
        }
    }
    // ---- sums against the warp's base, first column of the maximum --------------------------------------
    float S, Tt;
    {
        float s0, s1, t0, t1;
        upk(S2, s0, s1);
        upk(T2, t0, t1);
        S = s0 + s1;
        Tt = t0 + t1;
    }
    if (S > 0.f) {
        const float dl = fmaxf(base - base_of(M), kDClamp);
        const float c = fast_exp2(dl);
        Tt = c * fmaf(dl, S, Tt);
        S *= c;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, o);
        Tt += __shfl_xor_sync(0xffffffffu, Tt, o);
    }
    idx = __reduce_min_sync(0xffffffffu, idx);
    if (lane == 0) s_part[warp] = make_float4(M, S, Tt, __int_as_float(idx));
    __syncthreads();

    // ---- publish the CTA's partial; count arrivals (tickets only count, nothing spins) --------------------
    const int seq = row / p.rows_per_seq;
    if (warp == 0) {
        const float4 f = s_part[lane % kWarps];
        Partial acc;
        acc.M = f.x; acc.S = f.y; acc.T = f.z; acc.idx = __float_as_int(f.w);
#pragma unroll
        for (int o = kWarps / 2; o > 0; o >>= 1) {
            Partial q;
            q.M = __shfl_xor_sync(0xffffffffu, acc.M, o);
            q.S = __shfl_xor_sync(0xffffffffu, acc.S, o);
            q.T = __shfl_xor_sync(0xffffffffu, acc.T, o);
            q.idx = __shfl_xor_sync(0xffffffffu, acc.idx, o);
            acc = merge(acc, q);
        }
        if (lane == 0) {
            *reinterpret_cast<float4*>(p.partials + (long long)row * p.pitch + split) =
                make_float4(acc.M, acc.S, acc.T, __int_as_float(acc.idx));
            const int old = p.single_level ? ticket_add(&p.seq_ticket[seq], 1) : ticket_add(&p.row_ticket[row], 1);
            int all = p.rows_per_seq * p.splits;   // partials of the sequence
            if (kUneven) all = p.rows_per_seq * (p.splits + 1) - min(max(p.n_few - seq * p.rows_per_seq, 0), p.rows_per_seq);
            s_last = old == (p.single_level ? all : n_splits) - 1;
        }
    }
    __syncthreads();   // orders the ticket's acquire before the other threads' reads of the partials
    if (!s_last) return;

    if (p.single_level) {
        // ---- last CTA of the sequence: finish every row, then the masked maximum and the decision ----
        // eight threads per row (each merges up to four split partials, then three shuffle steps), 32 rows per pass
        for (int r0 = 0; r0 < p.rows_per_seq; r0 += kGateThreads / 8) {
            const int r = r0 + (tid >> 3), j = tid & 7;
            const bool ok = r < p.rows_per_seq;
            const int rr = seq * p.rows_per_seq + (ok ? r : 0);
            float4 f[4];
            const int n_part = splits_of<kUneven>(p, rr);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int sp = j + 8 * k;
                f[k] = make_float4(-INFINITY, 0.f, 0.f, __int_as_float(0x7fffffff));
                if (ok && sp < n_part) f[k] = __ldcg(reinterpret_cast<const float4*>(partials_of(p, rr) + sp));
            }
            Partial acc;
            acc.M = f[0].x; acc.S = f[0].y; acc.T = f[0].z; acc.idx = __float_as_int(f[0].w);
#pragma unroll
            for (int k = 1; k < 4; ++k) {
                Partial q;
                q.M = f[k].x; q.S = f[k].y; q.T = f[k].z; q.idx = __float_as_int(f[k].w);
                acc = merge(acc, q);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                Partial q;
                q.M = __shfl_xor_sync(0xffffffffu, acc.M, o);
                q.S = __shfl_xor_sync(0xffffffffu, acc.S, o);
                q.T = __shfl_xor_sync(0xffffffffu, acc.T, o);
                q.idx = __shfl_xor_sync(0xffffffffu, acc.idx, o);
                acc = merge(acc, q);
            }
            if (ok && j == 0) {
                const float H = fmaxf(logf(acc.S) - kLn2 * acc.T / acc.S, 0.f);
                const float conf = fast_exp2(fmaf(acc.M, kLog2e, -base_of(acc.M))) / acc.S;
                if (p.argmax_out) p.argmax_out[rr] = acc.idx;
                if (p.conf_out) p.conf_out[rr] = conf;
                p.entropy_out[rr] = H;
                if (p.masked) {
                    s_H[r] = H;
                    s_conf[r] = conf;
                    s_arg[r] = acc.idx;
                } else {
                    s_H[r] = p.flags[rr] ? H : -INFINITY;
                    s_conf[r] = p.flags[rr] ? conf : -INFINITY;
                }
            }
        }
        __syncthreads();
        if (warp == 0 && p.masked) {
            // ---- confidence-based parallel decoding (Section 2.1 of the paper; threshold 0.9 in its experiments):
            // every masked row above the threshold is decoded; if none is, the masked row of highest confidence
            // (smallest index on ties).  Lane l owns rows l and l + 32 (rows_per_seq <= 64).
            bool msk[2], dec[2];
            float best = -1.f;
            int best_r = 0x7fffffff;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int r = lane + 32 * q;
                msk[q] = r < p.rows_per_seq && p.masked[seq * p.rows_per_seq + r] != 0;
                dec[q] = msk[q] && s_conf[r] > p.conf_thr;
                if (msk[q] && s_conf[r] > best) { best = s_conf[r]; best_r = r; }   // rows ascend: the first maximum stays
            }
            if (!__any_sync(0xffffffffu, dec[0] || dec[1])) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int orow = __shfl_xor_sync(0xffffffffu, best_r, o);
                    if (ob > best || (ob == best && orow < best_r)) { best = ob; best_r = orow; }
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) dec[q] = msk[q] && (lane + 32 * q == best_r);
            }
            float E = -INFINITY, Hsum = 0.f, Cmax = -INFINITY;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int r = lane + 32 * q;
                if (r < p.rows_per_seq) {
                    const int rr = seq * p.rows_per_seq + r;
                    p.decoded_out[rr] = dec[q] ? 1 : 0;
                    if (dec[q]) {
                        p.tokens[rr] = s_arg[r];
                        p.masked[rr] = 0;
                        E = fmaxf(E, s_H[r]);
                        Hsum += s_H[r];
                        Cmax = fmaxf(Cmax, s_conf[r]);
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                E = fmaxf(E, __shfl_xor_sync(0xffffffffu, E, o));
                Hsum += __shfl_xor_sync(0xffffffffu, Hsum, o);
                Cmax = fmaxf(Cmax, __shfl_xor_sync(0xffffffffu, Cmax, o));
            }
            if (lane == 0) {
                if (p.ent_sum_out) p.ent_sum_out[seq] = Hsum;
                if (p.max_conf_out) p.max_conf_out[seq] = Cmax;
                p.max_entropy_out[seq] = E;
                p.decision_out[seq] = (E > p.tau) ? EC_RECOMPUTE : EC_SKIP;
                p.seq_ticket[seq] = 0;   // ready for the next call
            }
        } else if (warp == 0) {
            float E = -INFINITY, Hsum = 0.f, Cmax = -INFINITY;
            for (int r = lane; r < p.rows_per_seq; r += 32) {
                E = fmaxf(E, s_H[r]);
                Hsum += (s_H[r] == -INFINITY) ? 0.f : s_H[r];   // rows outside the decoded set carry -inf
                Cmax = fmaxf(Cmax, s_conf[r]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                E = fmaxf(E, __shfl_xor_sync(0xffffffffu, E, o));
                Hsum += __shfl_xor_sync(0xffffffffu, Hsum, o);
                Cmax = fmaxf(Cmax, __shfl_xor_sync(0xffffffffu, Cmax, o));
            }
            if (lane == 0) {
                if (p.ent_sum_out) p.ent_sum_out[seq] = Hsum;
                if (p.max_conf_out) p.max_conf_out[seq] = Cmax;
                p.max_entropy_out[seq] = E;
                p.decision_out[seq] = (E > p.tau) ? EC_RECOMPUTE : EC_SKIP;
                p.seq_ticket[seq] = 0;   // ready for the next call
            }
        }
        return;
    }

    // ---- last CTA of the row finishes the row; the last row of the sequence finishes the sequence ----
    if (warp != 0) return;
    finish_row<kUneven>(p, row, lane);
    int seq_last = 0;
    if (lane == 0) {
        p.row_ticket[row] = 0;
        seq_last = ticket_add(&p.seq_ticket[seq], 1) == p.rows_per_seq - 1;
    }
    seq_last = __shfl_sync(0xffffffffu, seq_last, 0);
    if (!seq_last) return;
    float E = -INFINITY;
    for (int r = lane; r < p.rows_per_seq; r += 32) {
        const int rr = seq * p.rows_per_seq + r;
        if (p.flags[rr]) E = fmaxf(E, __ldcg(&p.entropy_out[rr]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) E = fmaxf(E, __shfl_xor_sync(0xffffffffu, E, o));
    if (lane == 0) {
        p.max_entropy_out[seq] = E;
        p.decision_out[seq] = (E > p.tau) ? EC_RECOMPUTE : EC_SKIP;
        p.seq_ticket[seq] = 0;
    }
}

// workspace carving: [row_ticket: R i32][seq_ticket: R i32][entropy scratch: R f32][pad to 16][partials]
struct GateWs {
    size_t off_row, off_seq, off_ent, off_part, total;
};
GateWs carve(int n_rows) {
    GateWs w;
    const size_t r = (size_t)n_rows;
    w.off_row = 0;
    w.off_seq = r * 4;
    w.off_ent = r * 8;
    w.off_part = ((r * 12) + 15) & ~(size_t)15;
    w.total = w.off_part + r * kMaxSplits * sizeof(Partial);
    return w;
}

// How the rows are cut: one resident wave of 4 CTAs of 256 threads per SM, all its places taken.  Rows get `splits` chunks
// or one more, so that the CTAs are as many as the places: with equal splits, 400 CTAs of 200 rows on 592 places, 104 SMs had
// three CTAs, 44 two.  (Chunks are whole pieces of 256 columns, so where they are short the last ones of a row may be empty: 8
// rows of 153700 have 56 of 592 CTAs without work.)  us a call, equal -> as here, on logits that no call before has read, bf16
// [32, 126464] 6.91 -> 6.66, 128 rows 11.26 -> 10.29, 200 17.45 -> 14.38, 256 16.88 -> 16.80, 300 27.4 -> 19.3, fp32 32 rows
// 7.56 -> 7.36.  Equal chunks, whole 2048-column slabs, are the better ones where
//   - a row would have more than the 32 chunks that one CTA finishes, and no more of equal ones: 16 rows of 126464 as 37 or 38
//     chunks 6.53, as 31 5.29 (10 rows of 152064, 59 or 60 and 38 chunks: fp32 6.92 against 7.28 of equal ones);
//   - they are no longer than the longest chunk here (rounding them to slabs costs less than 5 %), and rows with one chunk more
//     are too few to spare every SM one of the long ones: 148 rows of 32000 2 % longer here, 592 of 4104 3 %; with whole rows as
//     the long chunks the line lies at two fifths, or one half below 48 K columns: 400 rows (192 cut) of 126464 28.5 -> 24.2, of
//     32000 11.8 -> 12.2, 425 and 450 rows (167, 142 cut) 0 to 3 % longer;
//   - fp32, which waits for memory rather than for its arithmetic, has large chunks: above 8192 columns [56, 126464], [64,
//     151936] and [80, 100352] took 1.6 to 2.2 % longer here, below [32, 50304] 8, [32, 126464] 5, [56, 64000] 5 % less.
void plan_chunks(GateParams& p, int max_splits, bool bf16) {
    const int slab = kGateThreads * kVec;
    const long long slots = (long long)kCtasPerSm * sm_count();
    long long want = slots / p.n_rows;
    p.n_few = p.n_rows;
    if (want >= (bf16 ? 1 : 6) && want + 1 <= max_splits && p.vocab / (want + 1) >= slab && (bf16 || p.vocab / want <= 8192)) {
        const int longest = (int)((p.vocab + want - 1) / want), more = (int)(slots - want * p.n_rows);
        const int even = std::min((longest + slab - 1) / slab * slab, p.vocab);
        const bool finish = want + 1 <= kFinishSplits || (p.vocab + even - 1) / even > kFinishSplits;
        const bool spares = want > 1 ? 8LL * more >= p.n_rows : (p.vocab < 49152 ? 4LL : 5LL) * more >= 2LL * p.n_rows;
        if (finish && (spares || longest * 20LL <= even * 19LL)) {
            p.splits = (int)want;
            p.pitch = p.splits + 1;
            p.n_few = p.n_rows - more;
            for (int k = 0; k < 2; ++k) {
                const int n = p.splits + k;
                p.inverse[k] = (unsigned int)((0x100000000LL + n - 1) / n);
                p.chunk[k] = ((p.vocab + n - 1) / n + kPiece - 1) / kPiece * kPiece;
            }
            return;
        }
    }
    if (want < 1) want = 1;
    if (want > max_splits) want = max_splits;
    const int per = (int)((p.vocab + want - 1) / want);
    p.chunk[0] = p.chunk[1] = (per + slab - 1) / slab * slab;
    p.splits = p.pitch = (p.vocab + p.chunk[0] - 1) / p.chunk[0];
    p.inverse[0] = p.inverse[1] = 0;
}

template <typename T, bool kUneven>
cudaError_t launch_t(const GateParams& p, cudaStream_t stream) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = kUneven ? dim3(p.n_few * p.splits + (p.n_rows - p.n_few) * p.pitch, 1, 1) : dim3(p.splits, p.n_rows, 1);
    cfg.blockDim = dim3(kGateThreads, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // launch latency may overlap the previous kernel's tail
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, gate_kernel<T, kUneven>, p);
}

}  // namespace

size_t gate_workspace_bytes(int n_rows, int vocab) {
    if (n_rows <= 0 || vocab <= 0) return 0;
    return carve(n_rows).total;
}

size_t gate_ticket_bytes(int n_rows) { return n_rows > 0 ? carve(n_rows).off_ent : 0; }   // row + sequence tickets

cudaError_t launch_gate(const GateArgs& a, cudaStream_t stream) {
    const GateWs w = carve(a.n_rows);
    char* ws = static_cast<char*>(a.workspace);
    GateParams p;
    p.logits = a.logits;
    p.row_stride = a.row_stride;
    p.n_rows = a.n_rows;
    p.vocab = a.vocab;
    p.rows_per_seq = a.rows_per_seq;
    p.single_level = 0;
    p.flags = a.flags;
    p.tau = a.tau;
    p.argmax_out = a.argmax_out;
    p.conf_out = a.conf_out;
    p.entropy_out = a.entropy_out ? a.entropy_out : reinterpret_cast<float*>(ws + w.off_ent);
    p.max_entropy_out = a.max_entropy_out;
    p.decision_out = a.decision_out;
    p.row_ticket = reinterpret_cast<int*>(ws + w.off_row);
    p.seq_ticket = reinterpret_cast<int*>(ws + w.off_seq);
    p.partials = reinterpret_cast<Partial*>(ws + w.off_part);
    p.masked = a.masked;
    p.conf_thr = a.conf_threshold;
    p.decoded_out = a.decoded_out;
    p.tokens = a.tokens;
    p.ent_sum_out = a.entropy_sum_out;
    p.max_conf_out = a.max_conf_out;
    // decode mode and the extra metrics need all rows of a sequence in one CTA's hands at the end: the single-level
    // finish (at most 32 splits)
    const bool one_cta_finish = a.masked || a.entropy_sum_out || a.max_conf_out;
    plan_chunks(p, one_cta_finish ? kFinishSplits : kMaxSplits, a.dtype == EC_BF16);
    p.single_level = (a.rows_per_seq <= kSingleLevelMaxRows && p.pitch <= kFinishSplits) ? 1 : 0;
    if (one_cta_finish && !p.single_level) return cudaErrorInvalidValue;   // rows_per_seq > 64 or vocab > 32 * 8192 * ...: rejected by the API layer
    if (p.pitch > p.splits) return a.dtype == EC_BF16 ? launch_t<__nv_bfloat16, true>(p, stream) : launch_t<float, true>(p, stream);
    return a.dtype == EC_BF16 ? launch_t<__nv_bfloat16, false>(p, stream) : launch_t<float, false>(p, stream);
}

}  // namespace ec
