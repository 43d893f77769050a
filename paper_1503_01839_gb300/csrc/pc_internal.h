// pc_internal.h -- host-side declarations shared by the library's .cu files.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <vector>
#include <cuda_runtime.h>

#include "picount.h"
#include "pc_common.cuh"

// ------------------------------------------------------------------ errors
// Every CUDA call goes through PC_CUDA; on failure the enclosing function
// returns PC_ECUDA after recording the message in the context.
void pc_set_error(pc_ctx* ctx, const char* fmt, ...);

#define PC_CUDA(ctx, call)                                                     \
    do {                                                                       \
        cudaError_t e_ = (call);                                               \
        if (e_ != cudaSuccess) {                                               \
            pc_set_error((ctx), "%s failed: %s (%s:%d)", #call,                \
                         cudaGetErrorString(e_), __FILE__, __LINE__);          \
            return PC_ECUDA;                                                   \
        }                                                                      \
    } while (0)

#define PC_TRY(expr)                                                           \
    do {                                                                       \
        int r_ = (expr);                                                       \
        if (r_ != PC_OK) return r_;                                            \
    } while (0)

// Launch check: a launch error (bad configuration) is reported at once.
#define PC_LAUNCHED(ctx) PC_CUDA(ctx, cudaGetLastError())

// --------------------------------------------------------------- buffers
// Grow-only device buffer owned by the context.
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    template <class T> T* as() const { return (T*)p; }
};

int buf_reserve(pc_ctx* ctx, DevBuf& b, size_t bytes);
void buf_free(DevBuf& b);

// ----------------------------------------------------------------- tables
struct Tables {
    // primes <= 65536 (bootstrap), u32, ascending, 0-based
    DevBuf small_primes;
    u32 n_small = 0;
    // pi table over [0, pi_limit]
    u64 pi_limit = 0;
    DevBuf pi_rec;   // PiRec per 240 numbers
    // primes[1..nprimes] (u32), primes[0] = 1, primes[nprimes+1] = next prime
    u64 prime_limit = 0;
    u64 nprimes = 0;
    DevBuf primes;
    DevBuf primes_rcp;   // floor((2^64 - 1) / p_k), same indexing as primes
    DevBuf primes_dv;    // p_k | floor((2^(32+s) - 1) / p_k) << 32, s = floor(log2 p_k) (pc_dv)
    // squarefree m-list over [2, ml_limit] with lpf > p_cmin
    u64 ml_limit = 0;
    u32 ml_cmin = 99;
    u64 ml_n = 0;
    DevBuf ml_m, ml_info, ml_gpf, ml_rcp, ml_rec, rank_bits, rank_cnt;
    // sub-lists of the m-list: entries with lpf index > sl_K[k] (ascending K), so
    // that the leaves of a prime p_b with b >= K need not skip entries with lpf <= p_K
    static constexpr int NSUB = 4;
    DevBuf sl_rec[NSUB], sl_rcp[NSUB], sl_bits[NSUB], sl_cnt[NSUB];   // MList::rec and rcp only
    u32 sl_K[NSUB] = {0, 0, 0, 0};
    u64 sl_n[NSUB] = {0, 0, 0, 0};
    u32 n_sl = 0;
    // sampled pi table (Section 2.1): samp[j] = pi(j * samp_s), covering every v <= samp_limit
    DevBuf samp;
    u32 samp_s = 0;
    u64 samp_limit = 0;
    // presieve pattern of the primes 7, 11, 13, 17, 19 (WHEEL19_PERIOD bytes of the mod-30
    // bitset, then a copy of its start so that any 128 KiB slice is contiguous)
    DevBuf wheel19;
    // patterns of the primes 7 .. 61 in the mod-30 bitset: entry (k - 4) PATTERN_P + r of p_k
    // holds the 16 bytes from byte index g = r mod p_k on, a bit clear where p_k divides
    DevBuf pat16;
    // odd-number pi table over [0, podd_limit] (pi_odd1): one uint2 per 64 integers
    DevBuf pi_odd;
    u64 podd_limit = 0;
    // phi(., c) residue tables for the primorial of c (c = 0..7)
    DevBuf phiT[8];
    bool phiT_ok[8] = {false, false, false, false, false, false, false, false};

    PiTable pi() const { return PiTable{pi_rec.as<PiRec>(), pi_limit}; }
    RankTable rank() const { return RankTable{rank_bits.as<u64>(), rank_cnt.as<u32>(), ml_limit}; }
    MList mlist() const
    {
        return MList{ml_m.as<u32>(), ml_info.as<u32>(), ml_gpf.as<u32>(), ml_rcp.as<u64>(),
                     ml_rec.as<uint4>(), ml_n, ml_limit, ml_cmin};
    }
    MList sublist(int k) const
    {
        return MList{nullptr, nullptr, nullptr, sl_rcp[k].as<u64>(), sl_rec[k].as<uint4>(), sl_n[k], ml_limit, sl_K[k]};
    }
    RankTable subrank(int k) const { return RankTable{sl_bits[k].as<u64>(), sl_cnt[k].as<u32>(), ml_limit}; }
};

// ---------------------------------------------------------------- context
struct pc_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;   // stream every kernel of this context uses
    cudaStream_t own_stream = nullptr;
    // Independent phases of one call run beside its stream: on side streams that wait for the
    // call's start and that its stream waits for before the results are read (pc_engine.cu).
    // While a phase is enqueued there, stream is the side stream and scan_sel its scan scratch.
    cudaStream_t side[2] = {nullptr, nullptr};
    cudaEvent_t ev_fork = nullptr, ev_join[2] = {nullptr, nullptr};
    int scan_sel = 0;
    pc_params params{};
    int sm_count = 0;
    size_t smem_optin = 0;
    Tables T;
    // scratch (grow-only)
    DevBuf seg_b, seg_off, counts, tallies, acc_seg, partials, result, misc, scan_tmp[3];
    DevBuf easy_rng[2], easy_chunk_off[2];   // of the easy pass, of the table leaves' pass
    DevBuf starts;
    DevBuf mq_q, mq_pref, mq_e, mq_h, mq_hq, mq_p;   // batched queries (pc_pi_count_batch)
    DevBuf p2_seg;   // P2: per-segment sums, counts and tallies
    DevBuf p2_bkt;   // P2 bucket sieve: the buckets of one wave of segments and their fill counts
    // pinned host staging for small results
    void* host_stage = nullptr;
    // the counters of pc_last_stats, and those with an entry point of their own
    struct Stats : pc_stats {
        u64 table_leaves;   // hard leaves read from the pi table (pc_table_leaves)
    };
    Stats stats{};
    char errmsg[512] = {0};
    cudaEvent_t ev[16];
    bool ev_ok = false;
    // A worker context borrows the tables of its parent (shallow copy of T):
    // it never grows or frees them.  Batched and served queries run on
    // workers, one host thread and one stream each, so that their kernels
    // overlap on the device.
    bool borrowed = false;
    std::vector<pc_ctx*> workers;
    // autotuned alpha and segment bytes per decimal digit count of x (0 = not tuned)
    u32 tuned_alpha[21] = {0};
    u32 tuned_seg[21] = {0};
    u32 seg_call = 0;   // hard-leaf segment bytes chosen for the running pi(x) call (0 = default)
    u32 tuned_ctas[21] = {0};   // autotuned resident CTAs per SM of the hard-leaf sieve (0 = most)
    u32 tuned_ctas_seg[21] = {0};   // segment bytes they were timed at: for another size they say nothing
    u32 ctas_call = 0;          // the value for the running call
    u32 ctas_seg_call = 0;      // and its segment bytes (0: any)
    // device counters of the running call (easy leaves, runs, their leaves, P2 crossings, table
    // leaves), beside the result slots; null outside a leaf-sum call
    unsigned long long* dstat = nullptr;
    bool hard_timed = false, easy_timed = false, p2_timed = false;   // ev[0..1] / ev[2..3] / ev[4..5] hold kernel times
    // the hard-leaf sieve's instantiation for the last (threads, shared memory, residency) asked for
    struct { int nt = 0, want = -1, per_sm = 0; size_t smem = 0; void* fn = nullptr; } hk;
    bool p2_smem_set = false;   // the P2 sieve's shared-memory limit has been raised
    // How the batched phases (mq_*) run: MQ_DIRECT launches as it goes; MQ_PREPARE reserves
    // scratch, uploads the arrays built on the host and reads back table values, with no
    // device work; MQ_CAPTURE then enqueues only device work (kernels, memsets), into a
    // CUDA graph, and must not grow any scratch
    int mq_mode = 0;
    u64 mq_p2_pv[2] = {0, 0};   // pi values mq_p2 needs, read in the prepare pass
    // hard-leaf sieve geometry of the batched schedule (pc_autotune_batch; 0 = default:
    // 16 KiB segments, as many resident CTAs per SM as fit)
    u32 batch_seg = 0, batch_ctas = 0;
    bool batch_builtin_alpha = false;   // the batch uses the built-in alphas, not pc_autotune's
    void* mq_hard_kern = nullptr;   // the batched sieve's instantiation and resident CTAs per SM,
    int mq_hard_per_sm = 0;         // chosen (and its shared-memory limit set) before any capture
};

enum { MQ_DIRECT = 0, MQ_PREPARE = 1, MQ_CAPTURE = 2 };
inline bool mq_device_work(const pc_ctx* c) { return c->mq_mode != MQ_PREPARE; }
inline bool mq_host_upload(const pc_ctx* c) { return c->mq_mode != MQ_CAPTURE; }

u32 default_alpha(u64 x);
int decimal_digits(u64 x);
u32 choose_alpha(const pc_ctx* ctx, u64 x);

// Worker contexts of ctx (created on first use, tables refreshed from ctx).
int workers_ensure(pc_ctx* ctx, int n);
void workers_destroy(pc_ctx* ctx);
// Build every table that queries up to x_max (pi(x) with the built-in alpha,
// and phi(x, a) for a <= a_max) need, so that workers never grow them.
int tables_for_queries(pc_ctx* ctx, const u64* xs, size_t n, u64 a_max);
int pi_count_impl(pc_ctx* ctx, u64 x, u32 alpha, u64* out);
int phi_impl(pc_ctx* ctx, u64 x, u64 a, u64* out);

// ------------------------------------------------------------------- util
// out[i] = sum_{j<i} in[j] for i < n, and out[n] = total (out has n+1 slots).
int scan_exclusive_u32_to_u32(pc_ctx* ctx, const u32* in, u32* out, u64 n);
int scan_exclusive_u32_to_u64(pc_ctx* ctx, const u32* in, u64* out, u64 n);
// *out = sum of n i128 values
int reduce_i128(pc_ctx* ctx, const I128Pair* in, u64 n, I128Pair* out);
int copy_to_host(pc_ctx* ctx, void* dst, const void* src, size_t bytes);  // synchronizes

// ----------------------------------------------------------------- tables
// Make sure tables cover pi lookups up to pi_limit, primes up to
// prime_limit (plus one sentinel prime), and the m-list up to ml_limit with
// lpf(m) > p_cmin.
int tables_ensure(pc_ctx* ctx, u64 pi_limit, u64 prime_limit, u64 ml_limit, u32 cmin);
// the presieve pattern of the primes 7..19 (Tables::wheel19), built once by a context that
// owns its tables (tables_ensure does); a no-op for one that borrows them
static constexpr u32 WHEEL19_PERIOD = 7u * 11u * 13u * 17u * 19u;   // bytes (30 integers each)
int tables_wheel19(pc_ctx* ctx);
static constexpr u32 PATTERN_P = 64;          // Tables::pat16 holds the primes below
static constexpr u32 PATTERN_PRIMES = 15;     // p_4 = 7 .. p_18 = 61
int tables_pat16(pc_ctx* ctx);
int tables_phi_c(pc_ctx* ctx, u32 c);   // phi(., c) residue table
// values of pi(v) for a handful of v (v <= pi_limit, at most PI_ASK_MAX), synchronizing
static constexpr int PI_ASK_MAX = 16;
int tables_pi_values(pc_ctx* ctx, const u64* v, u64* out, int n);
// pi(v) for any number of v (every v <= the table limit), synchronizing
int tables_pi_many(pc_ctx* ctx, const u64* v, u64* out, size_t n);

// The running call's result buffer, zeroed once per call and read back once at its end: eight
// I128Pair parts, then (as u64) the call's counters (dstat), the hard-leaf sieve's (HardArgs::stat)
// and the work queues, each on a line of its own.
static constexpr size_t RES_DSTAT = 128, RES_HARD = 256, RES_QUEUE = 384, RES_BYTES = 768;
enum { Q_EASY = 0, Q_HARD = 1, Q_P2 = 2, Q_TABLE = 3 };
inline unsigned long long* call_dstat(pc_ctx* c) { return (unsigned long long*)(c->result.as<unsigned char>() + RES_DSTAT); }
inline unsigned long long* call_hard_stat(pc_ctx* c) { return (unsigned long long*)(c->result.as<unsigned char>() + RES_HARD); }
inline unsigned long long* call_queue(pc_ctx* c, int q) { return (unsigned long long*)(c->result.as<unsigned char>() + RES_QUEUE + 64 * q); }

// ----------------------------------------------------------------- leaves
struct LeafProblem {
    u64 x, y, z;
    u32 c;        // ordinary-leaf wheel depth
    u64 a;        // leaves use primes p_b with c < b <= a
    bool trunc;   // a < pi(y): filter gpf(m) <= p_a
    u64 piy;      // pi(y)
    u64 B;        // pi(isqrt z)
    u64 R4;       // pi(x^(1/4)): a leaf with u >= p_b^2 and m > p_b has p_b^4 < x
    u64 E;        // pi(iroot3 x): a leaf with u >= p_b has p_b^3 < x
    // hard-leaf sieve over segments [shard_k * nseg / shard_n, (shard_k + 1) * nseg / shard_n) only
    // (shard_n = 0: all of them); the leaves' carries then start from phi(L - 1, b)
    u32 shard_k = 0, shard_n = 0;
    // the hard leaves with u < p_b^2 (read from the pi table, see easy_range) are added to the
    // easy sum by run_easy, not to the hard one by run_hard_sieve: for callers that want only
    // the total
    bool table_in_easy = false;
};

// phi(m, b) for every c <= b <= b_max (Section 4 starting values): out[b - c]
int phi_starts(pc_ctx* ctx, u64 m, u32 c, u64 b_max, u64* out);

// Each adds its sum to *out (device I128Pair) -- out must be zeroed first.
int run_s1_trivial(pc_ctx* ctx, const LeafProblem& P, I128Pair* out_s1, I128Pair* out_trivial);
// whether the easy leaves read pi(u) from the odd-number table (the fastest way; y < 2^29)
bool easy_odd_table(const pc_ctx* ctx, const LeafProblem& P);
int run_easy(pc_ctx* ctx, const LeafProblem& P, I128Pair* out);
int run_hard_smallb(pc_ctx* ctx, const LeafProblem& P, I128Pair* out);
int run_hard_sieve(pc_ctx* ctx, const LeafProblem& P, I128Pair* out);
// the hard leaves with y <= u < p_b^2, b > b_min, whose u lies in [u_lo, u_hi)
int run_hard_table(pc_ctx* ctx, const LeafProblem& P, u64 b_min, u64 u_lo, u64 u_hi, I128Pair* out);
// P2 takes the pi values it needs from the caller's one lookup: p2_ask writes the arguments (at
// most P2_ASK), run_p2 gets their pi values in the same order
static constexpr int P2_ASK = 5;
int p2_ask(pc_ctx* ctx, u64 x, u64 y, u64* v);
int run_p2(pc_ctx* ctx, u64 x, u64 y, u64 a, const u64* pv, I128Pair* out);

// ------------------------------------------------------- batched queries
// One pi(x) query of a batched launch (pc_pi_count_batch): its parameters, and the
// table values the batch reads back once for all queries.
struct MQ {
    u64 x, y, z;
    u64 a;      // pi(y)
    u64 B;      // pi(isqrt z)
    u64 K;      // pi(isqrt x)
    u64 nlim;   // m-list entries with m <= y
    u64 E;      // pi(iroot3 x): the easy leaves have b <= E
    u64 R4;     // pi(x^(1/4)): the leaves that need the sieve have b <= R4
    u32 c;
    u32 pad;
};

// The parts of every query of a batch, [q][0..4] = S1, trivial, easy, hard, P2, summed
// exactly by atomic_add_i128 (any order).
struct MQPlan {
    u32 Q = 0;
    const MQ* dq = nullptr;      // device copy of hq
    I128Pair* parts = nullptr;   // device, Q x 5
    std::vector<MQ> hq;
};

__device__ __forceinline__ void mq_atomic_add_i128(I128Pair* p, i128 v)
{
    // the low words add with wrap-around; every addition sends its own carry to the high word
    const unsigned long long lo = (unsigned long long)(u64)v;
    const unsigned long long old = atomicAdd((unsigned long long*)&p->lo, lo);
    const u64 carry = old + lo < old ? 1u : 0u;
    atomicAdd((unsigned long long*)&p->hi, (unsigned long long)((u64)(i64)(v >> 64) + carry));
}

// The last index k < n with pref[k] <= v (pref ascending, pref[0] <= v), by a whole warp: 32
// probes a round, so 10^5 entries take four dependent loads instead of seventeen.
__device__ __forceinline__ u64 warp_find(const u64* pref, u64 n, u64 v, u32 lane)
{
    u64 lo = 0;
    while (n > 1) {
        const u64 step = (n + 31) / 32, at = lane * step;
        const bool le = at < n && pref[lo + at] <= v;
        const u64 c = (u64)__popc(__ballot_sync(0xffffffffu, le)) - 1;   // lane 0's is true
        lo += c * step;
        n = pc_min(step, n - c * step);
    }
    return lo;
}

// The same for a v that never falls below the last call's, whose answer is hint: usually a
// little ahead, two loads away.
__device__ __forceinline__ u64 warp_find_from(const u64* pref, u64 n, u64 v, u32 lane, u64 hint)
{
    constexpr u64 step = 16;
    const u64 at = hint + lane * step;
    const u64 c = (u64)__popc(__ballot_sync(0xffffffffu, at < n && pref[at] <= v)) - 1;   // lane 0's is true
    const u64 lo = hint + c * step;
    if (c == 31) return lo + warp_find(pref + lo, n - lo, v, lane);   // past the window
    const u64 m = pc_min(step, n - lo);
    return lo + (u64)__popc(__ballot_sync(0xffffffffu, lane < m && pref[lo + lane] <= v)) - 1;
}

// the last index k < n with pref[k] <= v (pref ascending, pref[0] <= v)
__device__ __forceinline__ u64 mq_find(const u64* pref, u64 n, u64 v)
{
    u64 lo = 0, hi = n;
    while (hi - lo > 1) {
        const u64 mid = (lo + hi) >> 1;
        if (pref[mid] <= v) lo = mid; else hi = mid;
    }
    return lo;
}

int mq_info(pc_ctx* ctx, MQPlan& P);          // fills a, B, K, nlim, E, R4 (one read-back for the batch)
int mq_s1_trivial(pc_ctx* ctx, const MQPlan& P);
int mq_easy(pc_ctx* ctx, const MQPlan& P);
int mq_hard(pc_ctx* ctx, const MQPlan& P);
int mq_p2(pc_ctx* ctx, const MQPlan& P);

// segment bytes: the context's fixed size, else dflt
u32 pc_seg_bytes(pc_ctx* ctx, u32 dflt);
// default segment bytes of the hard-leaf sieve over [0, z]
u32 hard_seg_for(u64 z);
