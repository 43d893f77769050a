// pc_hard.cu -- the hard special leaves: the main sieve of Section 3 on the GPU.
//
// The interval [0, z] (z = x/y) is cut into segments; a segment is split
// into sub-ranges of sub_bytes bytes (30*sub_bytes integers, mod-30 wheel),
// one per warp of the CTA that owns the segment.  Each warp walks the primes
// p_b in order, b = k0+1 .. B_s, over its own sub-range only:
//
//   1. leaves of b (b > c): its bitset holds the integers of the sub-range
//      coprime to p_1..p_{b-1}, so for a hard leaf (b, m) with
//      u = x/(p_b m) in the sub-range, phi(u, b-1) = phi(L_w - 1, b-1) +
//      local(u), local(u) = set bits in [L_w, u].  The warp adds
//      -mu(m) * local(u) to its sum and -mu(m) to its tally for b: the unknown
//      phi(L_w - 1, b-1) is recorded, not needed, exactly as the tallies of
//      Section 3.
//   2. cross off the multiples of p_b in the sub-range, then record its count
//      of set bits.
//
// Warps never wait for one another inside a batch of primes (only
// __syncwarp); once per batch the CTA folds the warps' counts and tallies
// into segment rows and settles the carries between its own sub-ranges.
// Across segments, phi(L_s - 1, b - 1) = sum_{s' < s} count(s', b - 1) is an
// exclusive scan (the carries), and
//   S2_hard = sum (local sums) + sum_{s,b} tally(s, b) * phi(L_s - 1, b - 1).
// All segments are sieved at once, so the per-round synchronization of the
// blocks in Section 3 becomes one scan.
//
// A hard leaf (b, m) has u < x / p_b^2, so a segment starting at L only
// needs the primes p_b <= isqrt(x / L).  The hard leaves with u < p_b^2 are read
// from the pi table (easy_range in pc_leaves.cu), so it needs only those with
// p_b^2 <= L + span - 1 as well: B_s = pi(min(isqrt(x/L), isqrt(L + span - 1))),
// at most pi(x^(1/4)).  The segments with B_s >= b are thus consecutive,
// s >= p_b^2 / span; there the carry of b starts from phi(v, b-1) =
// pi(v) - b + 2, v = L - 1 < p_b^2, again from the pi table.
//
// Load balance: hard leaves crowd near u = y (their density falls like
// 1/u^2), so one segment can hold a large share of them.  A pre-pass counts
// the leaves of every segment; heavy segments are handed to several CTAs
// ("replicas"), each of which owns a run of consecutive steps and crosses off
// the primes before it with no counts; so is every segment while there are
// fewer than CTAs (Section 3 mentions dynamic block scheduling; here the
// schedule is a list of work items ordered by estimated cost, planned on the
// device).
#include <algorithm>
#include <cmath>
#include <vector>

#include "pc_internal.h"
#include "pc_sieve.cuh"

static constexpr u32 BATCH = 64;
// below this (PATTERN_P) a warp ANDs its sub-range with the prime's periodic pattern, 16 bytes a
// lane, and counts its blocks in the same pass; from here on lanes cross off (class, round) pairs
static_assert(PATTERN_P <= 64, "pattern primes are below 64");
// Block counters serve the leaves only.  A warp whose batch has few leaf steps lets them go
// stale and counts its blocks again at each leaf step (RECOUNT_COST: measured against the decrements),
// rather than decrement them at every crossing (about 5 instructions a pass of 32).
static constexpr u32 RECOUNT_COST = 160;
static constexpr u32 MAX_NW = 16;       // warps (sub-ranges) per segment
static constexpr u32 MAX_SUB = 8192;    // bytes per sub-range: up to 256 blocks of 256 bits
static constexpr u32 MAX_SEG = 131072;  // bytes per segment
// Steps of primes p >= sub-range bytes >> RUN_SHIFT (at most 2^RUN_SHIFT multiples per
// residue class in a sub-range) with p^3 above the segment are taken in runs (sparse_runs):
// (runs of 32 steps with up to 512 leaves measured fastest on GB300, against 32 to 256
// leaves and thresholds of 1, 1/4 and 1/8 of the sub-range)
static constexpr u32 RUN_SHIFT = 1;
static constexpr u32 RUN_LEAVES = 512;             // a run ends after the step that brings its leaves to this many
static constexpr u32 LOG_CAP = 512;                // hit log entries per warp (a run with leaves ends before more)
static_assert((8u << RUN_SHIFT) <= 32u && (8u << RUN_SHIFT) + 1 <= LOG_CAP, "a step's hits fit in a word and in the log");

// A work item: the steps b_lo <= b < b_hi (and b <= B_s) of segment s.  A light
// segment is one item with all its steps; a heavy one is split into replicas that
// each own a run of consecutive steps (see plan_bsplit_kernel).
struct HardItem {
    u32 s;      // segment
    u32 b_lo;   // first step
    u32 b_hi;   // one past the last step (~0: to the segment's last)
    u32 pad;
};

struct HardArgs {
    u64 x, y, z;
    u32 c, k0, kleaf, bmax;
    u64 a;
    bool trunc;
    u64 nseg;
    u64 s0, s1;   // the segments [s0, s1) of this run (a shard, or all of them)
    u32 seg_bytes, sub_bytes, nw, sub_shift;   // sub_bits = 1 << sub_shift
    u64 span;     // integers per segment
    u64 dspan;    // integers per sub-range
    PiTable pit;
    RankTable rk;
    MList ml;
    // sub-lists of the m-list (lpf index > slK[k]); a prime p_b reads its leaves
    // from the last one with slK <= b, else from ml
    MList sl[Tables::NSUB];
    RankTable srk[Tables::NSUB];
    u32 slK[Tables::NSUB];
    u32 nsl;
    const u32* primes;
    const u64* primes_rcp;
    const uint2* primes_dv;   // p_k and its 32-bit reciprocal (pc_dv)
    const uint4* pat;     // patterns of the primes 7 .. 61 (Tables::pat16)
    const u32* segB;
    const u64* off;
    const u32* rlo;     // first segment of row b (index b - k0): entry s of the row is off + s - rlo
    const u64* start;   // phi(L_{s0} - 1, b) for b = k0 .. bmax (index b - k0), or null for s0 = 0
    u32* counts;
    i32* tallies;
    const HardItem* items;
    const unsigned long long* nitems;   // number of items, written by the planner
    I128Pair* acc;                 // the hard sum
    u32* queue;
    unsigned long long* stat;      // [0] hard leaves, [1] multiples crossed off (from p >= PATTERN_P on)
};

struct __align__(16) StepInfo {
    u64 xp;        // x / p_b
    u64 q;         // L / p_b
    u64 mlo, mhi;  // leaf window m in (mlo, mhi]
    u64 vp;        // floor((2^64 - 1) / p_b)
    u32 p;
    u32 r0;        // L mod p_b
    u8 cbit[8];    // bit of class j inside its byte
    u32 flags;     // bit 0: leaves are primes, bit 1: step has leaves, bits 2-4: m-list (0 = all, k = sub-list k-1),
                   // bit 6: p^3 > the last integer of the segment and p >= the sub-range's bytes >> RUN_SHIFT
                   // (see sparse_runs)
    u32 pself;     // segment bit of p_b itself, or ~0
    u32 row;       // off - rlo of b, mod 2^32: the count / tally rows' entry of segment s is row + s
    u32 pad;
};

// leaf range of prime b in the segment [L, L + span): m in (mlo, mhi], u >= p_b^2.
// vp, vL, vLs: reciprocals of p, L (0 when L = 0) and L + span.
__device__ __forceinline__ bool leaf_window(const HardArgs& A, u64 p, u64 vp, u64 xp, u64 L, u64 vL, u64 vLs,
                                            u64& mlo, u64& mhi)
{
    // u >= p^2; xp / p^2 = floor(floor(xp / p) / p)
    mhi = pc_min(A.y, div_rcp(div_rcp(xp, p, vp), p, vp));
    if (L) mhi = pc_min(mhi, div_rcp(xp, L, vL));                        // u >= L
    mlo = pc_max(div_rcp(A.y, p, vp), div_rcp(xp, L + A.span, vLs));     // u < L + span, m > y / p
    return mhi > mlo;
}

// A warp owns its sub-range, so crossing off one prime needs no atomics on
// the bitset.  For p < PATTERN_P the lanes AND 16 bytes each with the prime's
// pattern; for larger p a lane takes one residue class in every fourth wheel
// round (30 p integers, p bytes) and reads and writes single bytes: two
// multiples of p with cofactors coprime to 30 differ by at least 2p > 30, so no
// two crossings share a byte.  Block counters take shared-memory atomics, since
// lanes of one pass may share a block.  (S2_hard(10^18), y = 2*10^7: this kernel 54.2 -> 45.9 ms
// against whole rounds per lane below 64, word accesses, counters decremented at every
// crossing and grouped steps of four primes; issue-bound, 59 % of cycles, 16 warps per SM.)
// Instantiated for several (threads, resident CTAs) launch bounds: fewer
// registers per thread buy more resident warps to hide shared-memory latency.
// A launch over the segments of many queries (the batched form): item g is segment
// g - qpref[q] of query q, qpref[q] <= g < qpref[q + 1], with arguments qargs[q] and its
// local sums added to qacc[q].  Queries keep their segments whole (no replicas).
struct MultiArgs {
    const HardArgs* qargs;
    const u32* qpref;   // nq + 1 entries
    u32 nq;
    unsigned long long items;
    I128Pair* qacc;     // query q's sum goes to qacc[q * qstride]
    u32 qstride;
};

template <int MAXT, int MINB, bool MULTI>
__global__ void __launch_bounds__(MAXT, MINB) hard_sieve_kernel(HardArgs A0, MultiArgs M)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // blocks of 256 bits (four 64-bit words); each lane owns bpl consecutive blocks
    const u32 nw = A0.nw, sub_bytes = A0.sub_bytes, sub_words = sub_bytes >> 2, nbw = sub_bytes >> 5, bpl = nbw >> 5;
    const u32 sub_bits = sub_bytes << 3;
    StepInfo* st = (StepInfo*)smem_raw;
    u32* bits = (u32*)(smem_raw + BATCH * sizeof(StepInfo));
    u16* blk = (u16*)(bits + (A0.seg_bytes >> 2));  // nw * nbw block counters
    u16* pre = blk + nw * nbw;                     // nw * nbw prefix counts
    u32* I = (u32*)(pre + nw * nbw);               // BATCH * (nw + 1)
    u32* cw = I + BATCH * (nw + 1);                // BATCH * nw
    i32* tw = (i32*)(cw + BATCH * nw);             // BATCH * nw
    u16* first = (u16*)(tw + BATCH * nw);          // BATCH * nw * 8: first byte of class j, or >= sub_bytes
    u16* hitlog = first + BATCH * nw * 8;          // nw * LOG_CAP

    __shared__ u32 patw[80];
    __shared__ u32 prev[MAX_NW];
    __shared__ u64 rLk[MAX_NW + 1];   // reciprocals of L + k * dspan, k = 0..nw
    __shared__ u32 s_item;
    __shared__ i128 red[32];
    // the m-lists a step may read its leaves from: index 0 the whole list, k the sub-list k-1
    __shared__ const uint4* lst_rec[1 + Tables::NSUB];
    __shared__ RankTable lst_rank[1 + Tables::NSUB];

    const u32 tid = threadIdx.x, lane = tid & 31, w = tid >> 5, NT = blockDim.x;
    make_pattern_words(patw, A0.k0);
    if (tid <= Tables::NSUB) {
        const MList& l = tid == 0 ? A0.ml : A0.sl[tid - 1];
        lst_rec[tid] = l.rec;
        lst_rank[tid] = tid == 0 ? A0.rk : A0.srk[tid - 1];
    }
    u32* my = bits + w * sub_words;
    u8* myb = (u8*)my;
    const u64* my64 = (const u64*)my;
    u16* myblk = blk + w * nbw;
    u32* myblk32 = (u32*)myblk;
    u16* mypre = pre + w * nbw;
    u16* lg = hitlog + w * LOG_CAP;

    // count the set bits of every 256-bit block of the sub-range into myblk;
    // returns this lane's share of the total.  Lanes read consecutive 16-byte
    // halves of blocks (no bank conflicts) and pairs of lanes add up a block.
    auto count_blocks = [&]() -> u32 {
        u32 tot = 0;
        const ulonglong2* h2 = (const ulonglong2*)my;
        for (u32 k = lane; k < 2 * nbw; k += 32) {
            const ulonglong2 v = h2[k];
            u32 c = __popcll(v.x) + __popcll(v.y);
            tot += c;
            c += __shfl_xor_sync(0xffffffffu, c, 1);
            if (!(k & 1)) myblk[k >> 1] = (u16)c;
        }
        return tot;
    };
    i64 acc = 0;
    unsigned long long nbusy = 0, nleafy = 0;
    u32 nleaves = 0, nclears = 0;   // a lane's share of a launch stays far below 2^32

    __shared__ __align__(16) unsigned char sA_raw[MULTI ? sizeof(HardArgs) : 16];
    __shared__ u32 s_q;
    u32 cur_q = ~0u;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(A0.queue, 1u);
        __syncthreads();
        const u64 item = s_item;
        u64 s;
        u32 it_lo, it_hi;
        if (MULTI) {
            if (item >= M.items) break;
            if (tid == 0) {   // the item's query: the last q with qpref[q] <= item
                u32 lo = 0, hi = M.nq;
                while (hi - lo > 1) {
                    const u32 mid = (lo + hi) >> 1;
                    if (M.qpref[mid] <= item) lo = mid; else hi = mid;
                }
                s_q = lo;
            }
            __syncthreads();
            const u32 q = s_q;
            if (q != cur_q) {   // the previous query's sums, then this query's arguments
                if (cur_q != ~0u) {
                    const i128 tq = block_sum_i128((i128)acc, red);
                    if (tid == 0) mq_atomic_add_i128(M.qacc + (u64)cur_q * M.qstride, tq);
                    acc = 0;
                }
                const u32* src = (const u32*)(M.qargs + q);
                for (u32 k = tid; k < sizeof(HardArgs) / 4; k += NT) ((u32*)sA_raw)[k] = src[k];
                cur_q = q;
                __syncthreads();
            }
            s = item - M.qpref[q];
            it_lo = ((const HardArgs*)sA_raw)->k0 + 1;
            it_hi = ~0u;
        } else {
            if (item >= *A0.nitems) break;
            const HardItem it = A0.items[item];
            s = it.s;
            it_lo = it.b_lo;
            it_hi = it.b_hi;
        }
        const HardArgs& A = MULTI ? *(const HardArgs*)sA_raw : A0;
        const u32 Bs = A.segB[s];
        const u32 b_first = it_lo, b_last = it_hi - 1 < Bs ? it_hi - 1 : Bs;   // this item's steps
        const u64 L = s * A.span;
        const u64 Lw = L + w * A.dspan;

        fill_pattern(bits, A.seg_bytes >> 2, L, patw, A.k0);
        if (tid <= nw) {
            const u64 Lk = L + tid * A.dspan;
            rLk[tid] = Lk ? ~0ull / Lk : 0;
        }
        if (b_first > A.k0 + 1 && b_first <= b_last) {
            // A replica that starts at step b_first needs the state after p_{b_first - 1}:
            // the primes before it are crossed off in any order, with no counts (the
            // replica that owns those steps records them), then the blocks are counted.
            __syncthreads();
            auto none = [](u32) {};
            u32 b = A.k0 + 1;
            for (; b < b_first; b++) {   // small primes: the whole CTA, lanes over wheel rounds
                const u32 p = A.primes[b];
                if (p >= 512) break;
                u64 ks = L ? div_rcp(L + p - 1, p, A.primes_rcp[b]) : 0;
                if (ks < p) ks = p;
                cross_off_coop(bits, A.seg_bytes, L, p, ks, tid, NT, none);
            }
            for (u32 task = tid; task < 8 * (b_first - b); task += NT) {   // one thread per (prime, class)
                const u32 bq = b + (task >> 3);
                const u64 p = A.primes[bq];
                u64 ks = L ? div_rcp(L + p - 1, p, A.primes_rcp[bq]) : 0;
                if (ks < p) ks = p;
                cross_off_class(bits, A.seg_bytes, L, (u32)p, ks, task & 7, none);
            }
            for (u32 bq = A.k0 + 1 + tid; bq < b_first; bq += NT) {   // the primes themselves (first segment)
                const u64 p = A.primes[bq];
                if (p >= L + A.span) break;
                if (p >= L) {
                    const u32 pos = seg_pos(p, L);
                    atomicAnd(&bits[pos >> 5], ~(1u << (pos & 31)));
                }
            }
        }
        __syncthreads();
        u32 cnt = __reduce_add_sync(0xffffffffu, count_blocks());
        if (lane == 0) prev[w] = cnt;
        bool stale = false;   // the warp's block counters lag behind its bitset
        __syncthreads();
        if (tid == 0 && b_first == A.k0 + 1) {
            u32 t = 0;
            for (u32 k = 0; k < nw; k++) t += prev[k];
            A.counts[A.off[0] + (s - A.s0)] = t;
        }

        for (u32 bb = b_first; bb <= b_last; bb += BATCH) {
            const u32 nb = b_last - bb + 1 < BATCH ? b_last - bb + 1 : BATCH;
            __syncthreads();
            // A: per-prime data of the batch
            for (u32 t = tid; t < nb; t += NT) {
                const u32 b = bb + t;
                StepInfo si;
                const u64 p = A.primes[b];
                const u64 vp = A.primes_rcp[b];
                si.p = (u32)p;
                si.vp = vp;
                si.xp = div_rcp(A.x, p, vp);
                si.q = div_rcp(L, p, vp);
                si.r0 = (u32)(L - si.q * p);
                si.row = (u32)A.off[b - A.k0] - A.rlo[b - A.k0];
                si.pad = 0;
                si.flags = 0;
                si.mlo = si.mhi = 0;
                si.pself = (p >= L && p < L + A.span) ? seg_pos(p, L) : ~0u;
                if (b > A.kleaf && b <= A.a && leaf_window(A, p, vp, si.xp, L, rLk[0], rLk[nw], si.mlo, si.mhi))
                {
                    u32 li = 0;
                    for (u32 k = 0; k < A.nsl; k++)
                        if (A.slK[k] <= b) li = k + 1;
                    si.flags = 2u | (p * p > A.y ? 1u : 0u) | (li << 2);
                }
                if (p >= (A.sub_bytes >> RUN_SHIFT) && p * p > div_rcp(L + A.span - 1, p, vp)) si.flags |= 64u;
                const u32 p30 = (u32)p % 30;
                for (int j = 0; j < 8; j++) si.cbit[j] = (u8)idx30(p30 * r8(j) % 30);
                st[t] = si;
            }
            __syncthreads();
            // B: leaf index boundaries of every sub-range, and the first multiples in it
            for (u32 idx = tid; idx < nb * (nw + 1); idx += NT) {
                const u32 t = idx / (nw + 1), k = idx - t * (nw + 1);
                const StepInfo& si = st[t];
                u32 v32 = 0;
                if (si.flags & 2u) {
                    u64 v;
                    if (k == 0) v = si.mhi;
                    else if (k == nw) v = si.mlo;
                    else v = pc_max(pc_min(div_rcp(si.xp, L + k * A.dspan, rLk[k]), si.mhi), si.mlo);
                    if (si.flags & 1u) {
                        const u64 b = bb + t;
                        v32 = (u32)(pc_min(pc_max(pi_lookup(A.pit, v), b), A.a) + 1);
                    } else {
                        v32 = (u32)rank_lookup(lst_rank[(si.flags >> 2) & 7u], v);
                    }
                }
                I[idx] = v32;
            }
            for (u32 idx = tid; idx < nb * nw; idx += NT) {
                const u32 t = idx / nw, k = idx - t * nw;
                const StepInfo& si = st[t];
                if (bb + t >= Bs || si.p < PATTERN_P) continue;
                const u64 p = si.p;
                u64 klo = si.q + div_rcp((u64)si.r0 + k * A.dspan + p - 1, p, si.vp);   // ceil(L_k / p)
                if (klo < p) klo = p;
                const u64 qa = klo / 30;
                const u32 kmod = (u32)(klo - 30 * qa);
                // the wheel round of klo starts at byte base of the sub-range (negative when it
                // began before it); every class's first multiple k p >= klo p is at or after 0
                const i64 base64 = (i64)(p * qa) - (i64)(L / 30 + (u64)k * sub_bytes);
                const i32 base = base64 > (i64)sub_bytes ? (i32)sub_bytes : (i32)base64;
                u32 f[8];
#pragma unroll
                for (u32 j = 0; j < 8; j++) {
                    const i32 fj = base + (i32)((u32)p * r8(j) / 30) + (r8(j) < kmod ? (i32)p : 0);
                    f[j] = (u32)min(fj, (i32)sub_bytes);
                }
                *(uint4*)(first + 8 * idx) = make_uint4(f[0] | f[1] << 16, f[2] | f[3] << 16, f[4] | f[5] << 16,
                                                        f[6] | f[7] << 16);
            }
            __syncthreads();
            // C: every warp runs the batch over its own sub-range.  It marks its steps with
            // leaves (and, for the counters, those with work at all) with ballots.
            auto leaf_range = [&](u32 t, u32& j0, u32& j1) {
                j0 = I[t * (nw + 1) + w + 1];
                j1 = I[t * (nw + 1) + w];
            };
            u64 busy = 0, leafy = 0, sparse = 0;
            u32 lj0[BATCH / 32], lj1[BATCH / 32];   // leaf range of step h*32 + lane
#pragma unroll
            for (u32 h = 0; h < BATCH / 32; h++) {
                const u32 t = h * 32 + lane;
                bool on = false, sq = false;
                lj0[h] = lj1[h] = 0;
                if (t < nb) {
                    const u32 b = bb + t, fl = st[t].flags, ps = st[t].pself;
                    sq = (fl & 64u) != 0;
                    if (b < Bs) {
                        if (st[t].p < PATTERN_P) {
                            on = true;
                        } else {
                            const uint4 f = *(const uint4*)(first + 8 * (t * nw + w));
                            const u32 m = __vminu2(__vminu2(f.x, f.y), __vminu2(f.z, f.w));
                            on = (m & 0xFFFFu) < sub_bytes || (m >> 16) < sub_bytes;
                        }
                        if (ps != ~0u && (ps >> A.sub_shift) == w) on = true;
                    }
                    if (b > A.kleaf && (fl & 2u)) {
                        leaf_range(t, lj0[h], lj1[h]);
                        if (lj1[h] > lj0[h]) on = true;
                    }
                    if (b > A.kleaf) tw[t * nw + w] = 0;
                }
                busy |= (u64)__ballot_sync(0xffffffffu, on) << (h * 32);
                leafy |= (u64)__ballot_sync(0xffffffffu, lj1[h] > lj0[h]) << (h * 32);
                sparse |= (u64)__ballot_sync(0xffffffffu, sq) << (h * 32);
            }
            // the sparse steps are a suffix of the batch (both of their conditions grow with p):
            // steps below t_sp go one by one, the rest in runs
            const u32 t_sp = sparse ? (u32)__ffsll((long long)sparse) - 1 : nb;
            const u64 lomask = t_sp >= 64 ? ~0ull : (1ull << t_sp) - 1;
            // Leaf data (m, its reciprocal, lpf index and mu) does not depend on the
            // sieve, so the first 32 leaves of the next leaf step are loaded ahead,
            // while the warp is still crossing off earlier primes.
            // A leaf's data is a record: m, its 32-bit reciprocal, lpf index << 1 | [mu = -1], gpf;
            // entry i of the list of a step with these flags (a prime m: lpf = itself, mu = -1)
            auto leaf_rec = [&](u32 fl, u32 i) -> uint4 {
                if (fl & 1u) {
                    const uint2 d = __ldg(A.primes_dv + i);
                    return make_uint4(d.x, d.y, ~0u, 0u);
                }
                return __ldg(lst_rec[(fl >> 2) & 7u] + i);
            };
            const uint4 no_leaf = make_uint4(1u, 0u, 0u, 0u);   // lpf index 0: no leaf of any b
            uint4 pf = no_leaf;
            auto leaf_bounds = [&](u32 t, u32& j0, u32& j1) {
                const u32 h = t >> 5;
                j0 = __shfl_sync(0xffffffffu, h ? lj0[1] : lj0[0], t & 31);
                j1 = __shfl_sync(0xffffffffu, h ? lj1[1] : lj1[0], t & 31);
            };
            auto prefetch = [&](u32 t) {
                u32 j0, j1;
                leaf_bounds(t, j0, j1);
                const u32 i = j0 + lane;
                pf = i < j1 ? leaf_rec(st[t].flags, i) : no_leaf;
            };
            // the count end of the leaf with record r of a step with x / p_b = xp: the bits of the
            // sub-range up to u = xp / m.  u - Lw = floor((xp - m Lw) / m) is below the sub-range's
            // length.  A lane without a leaf gets a small end (no_leaf: rel <= 1).
            const u64 negL = 0 - Lw;
            const bool m31 = !(A.y >> 31);
            const u32 gmax = A.trunc ? (u32)pc_min(A.a, 0xFFFFFFFFull) : ~0u;   // gpf(m) <= p_a
            auto leaf_end = [&](u64 xp, const uint4& r) -> u32 {
                const u32 rel = div_near(xp + r.x * negL, r.x, r.y, m31);
                const u32 q30 = rel / 30;
                return q30 * 8 + cntle30(rel - 30 * q30);
            };
            // prefix counts of the 256-bit blocks of the sub-range (from the block counters)
            auto block_prefix = [&]() {
                if (bpl == 8) {   // one 16-byte load and store per lane
                    const uint4 q = ((const uint4*)myblk)[lane];
                    const u32 c01 = (q.x & 0xFFFFu) + (q.x >> 16), c23 = (q.y & 0xFFFFu) + (q.y >> 16);
                    const u32 c45 = (q.z & 0xFFFFu) + (q.z >> 16), c67 = (q.w & 0xFFFFu) + (q.w >> 16);
                    const u32 own = c01 + c23 + c45 + c67;
                    u32 incl = own;
                    for (int o = 1; o < 32; o <<= 1) {
                        u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    const u32 r0 = incl - own, r2 = r0 + c01, r4 = r2 + c23, r6 = r4 + c45;
                    uint4 o4;
                    o4.x = r0 | ((r0 + (q.x & 0xFFFFu)) << 16);
                    o4.y = r2 | ((r2 + (q.y & 0xFFFFu)) << 16);
                    o4.z = r4 | ((r4 + (q.z & 0xFFFFu)) << 16);
                    o4.w = r6 | ((r6 + (q.w & 0xFFFFu)) << 16);
                    ((uint4*)mypre)[lane] = o4;
                } else {
                    u32 run = 0;
                    for (u32 k = 0; k < bpl; k++) run += myblk[lane * bpl + k];
                    u32 incl = run;
                    for (int o = 1; o < 32; o <<= 1) {
                        u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    run = incl - run;
                    for (u32 k = 0; k < bpl; k++) {
                        const u32 bi = lane * bpl + k;
                        mypre[bi] = (u16)run;
                        run += myblk[bi];
                    }
                }
                __syncwarp();
            };
            // set bits of the sub-range up to the count end e (0 < e <= sub_bits; other lanes
            // read clamped, in-bounds words and add what they like)
            auto count_to = [&](u32 e) -> u32 {
                u32 bi = e >> 8;
                if (bi >= nbw) bi = nbw - 1;
                // set bits of block bi below the end (0..256 of them), no data-dependent loop:
                // the whole words before the end's word, and that word's bits below the end
                const u32 rem = e - (bi << 8), wi = rem >> 6 < 3 ? rem >> 6 : 3;
                const ulonglong2 h0 = ((const ulonglong2*)my64)[2 * bi];
                const u64 h2 = my64[4 * bi + 2], hw = my64[4 * bi + wi];
                u32 n = mypre[bi] + __popcll(low_bits_top(hw, rem - 64 * wi));
                if (wi > 0) n += __popcll(h0.x);
                if (wi > 1) n += __popcll(h0.y);
                if (wi > 2) n += __popcll(h2);
                return n;
            };
            nbusy += __popcll(busy);
            nleafy += __popcll(leafy);
            // counting again at each leaf step against decrementing in each pass of each step (the
            // middle one of the batch has sub_bytes / 4p passes, at least one)
            const u32 mid4 = 4 * st[nb >> 1].p;
            const bool lazy = (u32)__popcll(leafy & lomask) * RECOUNT_COST * (mid4 < sub_bytes ? mid4 : sub_bytes) <
                              (u32)__popcll(lomask) * 5u * sub_bytes;
            auto fresh_blocks = [&]() {
                if (!stale) return;
                count_blocks();
                stale = false;
                __syncwarp();
            };
            if (leafy & lomask) prefetch(__ffsll((long long)(leafy & lomask)) - 1);
            __syncwarp();
            // Runs of sparse steps (p >= the sub-range's bytes >> RUN_SHIFT, so each residue
            // class has at most 2^RUN_SHIFT multiples in the sub-range, and p^3 above the
            // segment's last integer).  A bit still set when the run starts is 1, a prime, or a
            // product of primes that are all >= the run's first prime; below that prime cubed it
            // has at most two of them, so exactly one crossing of the run reaches it, that of its
            // least prime factor q, at the cofactor n / q >= q.  So every crossing of every step of
            // the run is found against the bitset as it is at the run's start, a step per lane (the
            // first bytes of its eight classes are one 16-byte load): no lane waits for another,
            // and 32 steps without leaves cost about what two did one after the other (four steps a
            // pass, lane = (step, class): S2_hard(10^18)'s sieve 45.9 ms, this 42.3).  The
            // crossings that hit a set bit are cleared at once in a run without leaves; otherwise
            // they go to a log, ordered by step.  A leaf of step t needs the count of set bits up
            // to u after the steps before t; that is the count on the run's starting bitset less
            // the logged hits of the run's steps before t below u.  So the leaves of all steps of a
            // run share 32-lane passes, one block prefix serves the whole run, and the logged bits
            // are cleared once at its end.  A run ends after the step that brings its leaves to
            // RUN_LEAVES, at 32 steps, or where the log is full, which keeps the log scans short.
            auto sparse_runs = [&](u32 t0) {
                while (t0 < nb) {
                    // the leaf ranges of the next (up to) 32 steps, one per lane
                    const u32 ts = t0 + lane;
                    u32 j0 = 0, j1 = 0;
                    {
                        const u32 src = ts & 31;
                        const u32 a0 = __shfl_sync(0xffffffffu, lj0[0], src), a1 = __shfl_sync(0xffffffffu, lj0[1], src);
                        const u32 c0 = __shfl_sync(0xffffffffu, lj1[0], src), c1 = __shfl_sync(0xffffffffu, lj1[1], src);
                        if (ts < nb) {
                            j0 = ts >= 32 ? a1 : a0;
                            j1 = ts >= 32 ? c1 : c0;
                        }
                    }
                    const u32 n = j1 - j0;   // 0 for steps without leaves in this sub-range (or share)
                    const u32 avail = nb - t0 < 32 ? nb - t0 : 32;
                    // crossings of step t0 + lane against the starting bitset: bit 8 m + j of hm is
                    // set when the m-th multiple of class j hits a set bit
                    const u16* fs = first + 8 * ((lane < avail ? ts : t0) * nw + w);
                    const StepInfo& ss = st[lane < avail ? ts : t0];
                    const u32 p = ss.p;
                    u32 hm = 0, self = ~0u, nx = 0;   // nx: the step's crossings
                    if (lane < avail && bb + ts < Bs) {
                        const uint4 f4 = *(const uint4*)fs;
                        const uint2 c8 = *(const uint2*)ss.cbit;
                        const u32 fw[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                        for (u32 j = 0; j < 8; j++) {
                            u32 by = (fw[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
                            const u32 bj = ((j < 4 ? c8.x : c8.y) >> (8 * (j & 3))) & 0xFFu;
#pragma unroll
                            for (u32 m = 0; m < (1u << RUN_SHIFT); m++, by += p) {
                                if (by < sub_bytes) {
                                    hm |= ((myb[by] >> bj) & 1u) << (8 * m + j);
                                    nx++;
                                }
                            }
                        }
                        if (s == 0) {   // p itself
                            const u32 ps = ss.pself;
                            if (ps != ~0u && (ps >> A.sub_shift) == w) {
                                const u32 pos = ps & (sub_bits - 1);
                                if ((my[pos >> 5] >> (pos & 31)) & 1u) self = pos;
                            }
                        }
                    }
                    const u32 h = __popc(hm) + (self != ~0u ? 1u : 0u);
                    u32 hin = h;   // hits of the steps up to t0 + lane
                    for (int o = 1; o < 32; o <<= 1) {
                        const u32 v = __shfl_up_sync(0xffffffffu, hin, o);
                        if (lane >= o) hin += v;
                    }
                    // the bit positions of this lane's hits, one after the other
                    auto each_hit = [&](auto&& f) {
                        for (u32 left = hm; left; left &= left - 1) {
                            const u32 q = __ffs(left) - 1;
                            f(((fs[q & 7] + (q >> 3) * p) << 3) + ss.cbit[q & 7]);
                        }
                        if (self != ~0u) f(self);
                    };
                    auto clear_hit = [&](u32 pos) {
                        atomicAnd(&my[pos >> 5], ~(1u << (pos & 31)));
                        if (!stale) atomicSub(&myblk32[pos >> 9], 1u << (16 * ((pos >> 8) & 1)));
                    };
                    if (!__any_sync(0xffffffffu, n)) {
                        __syncwarp();
                        each_hit(clear_hit);
                        nclears += nx;
                        if (lane < avail) cw[ts * nw + w] = cnt - hin;
                        cnt -= __shfl_sync(0xffffffffu, hin, 31);
                        __syncwarp();
                        t0 += avail;
                        continue;
                    }
                    u32 incl = n;
                    for (int o = 1; o < 32; o <<= 1) {
                        const u32 v = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += v;
                    }
                    // at least one step: a step has at most 8 << RUN_SHIFT hits and its own prime
                    const u32 fits = __popc(__ballot_sync(0xffffffffu, lane < avail && hin <= LOG_CAP));
                    const u32 enough = __ballot_sync(0xffffffffu, lane < fits && incl >= RUN_LEAVES);
                    const u32 len = enough ? (u32)__ffs(enough) : fits;   // steps t0 .. t0 + len - 1
                    const u32 TL = __shfl_sync(0xffffffffu, incl, len - 1);
                    const u32 loff = incl - n;                             // first leaf of step t0 + lane
                    if (lane < len) nclears += nx;   // the steps past the run are crossed again in the next one
                    // leaf g of the run: its step i (the last i < len with loff_i <= g) and its
                    // m-list data (nothing for g >= TL)
                    auto run_leaf = [&](u32 g, u32& i, uint4& r) {
                        i = 0;
                        for (u32 stp = 16; stp; stp >>= 1) {
                            const u32 cand = i + stp;
                            const u32 vv = __shfl_sync(0xffffffffu, loff, cand & 31);
                            if (cand < len && vv <= g) i = cand;
                        }
                        const u32 ji = __shfl_sync(0xffffffffu, j0, i);
                        const u32 li = __shfl_sync(0xffffffffu, loff, i);
                        const u32 fl = st[t0 + i].flags;
                        r = g < TL ? leaf_rec(fl, ji + (g - li)) : no_leaf;
                    };

                    const u32 nent = __shfl_sync(0xffffffffu, hin, len - 1), hoff = hin - h;   // log entries: all, before the step
                    if (lane < len) {
                        u32 off = hoff;
                        each_hit([&](u32 pos) { lg[off++] = (u16)pos; });
                    }
                    __syncwarp();
                    if (TL) {
                        fresh_blocks();
                        block_prefix();   // of the run's starting bitset
                        // each pass's m-list loads are issued one pass ahead (S2_hard(1e17) kernel
                        // 13.62 -> 13.30 ms with the same for steps taken one at a time)
                        u32 ci;
                        uint4 cr;
                        run_leaf(lane, ci, cr);
                        for (u32 g0 = 0; g0 < TL; g0 += 32) {
                            const u32 i = ci;
                            const uint4 r = cr;
                            if (g0 + 32 < TL) run_leaf(g0 + 32 + lane, ci, cr);   // next pass in flight
                            const u32 hi = __shfl_sync(0xffffffffu, hoff, i);
                            const u32 t = t0 + i, b = bb + t;
                            const u64 xp = st[t].xp;
                            const bool valid = r.z > 2 * b + 1 && r.w <= gmax;
                            const u32 e = leaf_end(xp, r);
                            u32 below = 0;   // hits of the run's earlier steps below the count end
                            for (u32 k = 0; k < hi; k++) below += lg[k] < e ? 1u : 0u;
                            const u32 cnt_u = count_to(e) - below;
                            const i32 sg = valid ? ((r.z & 1u) ? 1 : -1) : 0;
                            acc += (i64)sg * (i32)cnt_u;
                            if (valid) atomicAdd(&tw[t * nw + w], sg);
                            nleaves += valid;
                        }
                        __syncwarp();
                    }
                    // clear the logged bits; counts after every step of the run
                    for (u32 k = lane; k < nent; k += 32) clear_hit(lg[k]);
                    if (lane < len) cw[(t0 + lane) * nw + w] = cnt - hin;
                    cnt -= nent;
                    __syncwarp();
                    t0 += len;
                }
            };
            // Crosses off the steps t0 <= t < t1, one after the other (b < Bs): lane = (class j,
            // round offset o), four wheel rounds of p per pass, single bytes read and written.
            // The loop runs for every step of a run without a branch on its data, its passes are
            // counted by p alone, and the next step's data is loaded ahead: a step costs a few
            // dozen instructions, which is what bounds the sieve where leaves are few.  With upd
            // the block counters follow; byte y's is half (y >> 5) & 1 of word y >> 6.
            // nf, np, nbj: the data of step t0, loaded before its leaves.
            u32 nf = 0, np = 0, nbj = 0;
            auto load_step = [&](u32 t) {
                nf = first[8 * (t * nw + w) + (lane & 7)];
                np = st[t].p;
                nbj = st[t].cbit[lane & 7];
            };
            auto cross_steps = [&](u32 t0, u32 t1, bool upd) {
                const u32 j = lane & 7, o = lane >> 3;
                const u16* fp = first + 8 * (t0 * nw + w) + j;
                u32* cp = cw + t0 * nw + w;
                for (u32 t = t0; t < t1; t++, cp += nw) {
                    const u32 p = np, bj = nbj, bm = 1u << bj, step4 = 4 * p;
                    u32 by = nf + p * o;
                    fp += 8 * nw;
                    if (t + 1 < t1) {
                        nf = *fp;
                        np = st[t + 1].p;
                        nbj = st[t + 1].cbit[j];
                    }
                    if (step4 >= sub_bytes) {   // one pass: at most one crossing per lane
                        const bool in = by < sub_bytes;
                        u32 v = 0;
                        if (in) {
                            v = myb[by];
                            myb[by] = (u8)(v & ~bm);
                            nclears++;
                        }
                        const bool hit = (v & bm) != 0;
                        if (upd && hit) atomicSub(&myblk32[by >> 6], 1u << ((by >> 1) & 16));
                        cnt -= __popc(__ballot_sync(0xffffffffu, hit));
                    } else {
                        // two passes at a time, both bytes loaded before either is written (4p
                        // bytes apart).  dec: the hits times 2^bj below bit 16, the crossings above
                        u32 dec = 0;
                        for (u32 lim = 0; lim < sub_bytes; lim += 2 * step4, by += 2 * step4) {
                            const u32 bz = by + step4;
                            const bool ia = by < sub_bytes, ib = bz < sub_bytes;
                            u32 va = 0, vb = 0;
                            if (ia) va = myb[by];
                            if (ib) vb = myb[bz];
                            if (ia) myb[by] = (u8)(va & ~bm);
                            if (ib) myb[bz] = (u8)(vb & ~bm);
                            if (ia) dec += (va & bm) | 0x10000u;
                            if (ib) dec += (vb & bm) | 0x10000u;
                            if (upd) {
                                if (va & bm) atomicSub(&myblk32[by >> 6], 1u << ((by >> 1) & 16));
                                if (vb & bm) atomicSub(&myblk32[bz >> 6], 1u << ((bz >> 1) & 16));
                            }
                        }
                        nclears += dec >> 16;
                        cnt -= __reduce_add_sync(0xffffffffu, (dec & 0xFFFFu) >> bj);
                    }
                    __syncwarp();
                    if (s == 0) {   // p itself (p^2 is below the segment's end: in segment 0 only)
                        const u32 ps = st[t].pself;
                        u32 own = 0;
                        if (lane == 0 && ps != ~0u && (ps >> A.sub_shift) == w) {
                            const u32 pos = ps & (sub_bits - 1), mask = 1u << (pos & 31), old = my[pos >> 5];
                            my[pos >> 5] = old & ~mask;
                            own = (old & mask) ? 1u : 0u;
                            if (upd) atomicSub(&myblk32[pos >> 9], own << (16 * ((pos >> 8) & 1)));
                        }
                        cnt -= __shfl_sync(0xffffffffu, own, 0);
                        __syncwarp();
                    }
                    if (lane == 0) *cp = cnt;
                }
            };
            // Step t of a prime below PATTERN_P: AND with its pattern (p itself included), 16 bytes
            // a lane, counting the blocks on the way: lanes 2i, 2i + 1 hold the halves of a block
            auto pattern_step = [&](u32 t) {
                const u32 p = st[t].p;
                const u64 g = L / 30 + (u64)w * sub_bytes + 16 * lane;
                u32 ph = (u32)(g - div_rcp(g, p, st[t].vp) * p);
                const u32 dph = 512 % p;
                const uint4* pat = A.pat + (bb + t - 4) * PATTERN_P;   // p_4 = 7
                uint4* h4 = (uint4*)my;
                u32 tot = 0;
                for (u32 k = lane; k < 2 * nbw; k += 32) {
                    uint4 v = h4[k];
                    const uint4 m = __ldg(pat + ph);
                    v.x &= m.x, v.y &= m.y, v.z &= m.z, v.w &= m.w;
                    h4[k] = v;
                    u32 c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
                    tot += c;
                    c += __shfl_xor_sync(0xffffffffu, c, 1);
                    if (!(k & 1)) myblk[k >> 1] = (u16)c;
                    ph += dph;
                    if (ph >= p) ph -= p;
                }
                cnt = __reduce_add_sync(0xffffffffu, tot);
                stale = false;
                if (lane == 0) cw[t * nw + w] = cnt;
                __syncwarp();
            };
            // the steps below t_sp: the leaves of each step, then its crossings together with those
            // of the leaf-free steps after it
            const u32 t_x = Bs - bb < t_sp ? Bs - bb : t_sp;   // steps that cross off: b < Bs
            u64 lf = leafy & lomask;
            if (t_x) load_step(0);
            for (u32 t = 0;;) {
                const u32 tn = lf ? (u32)__ffsll((long long)lf) - 1 : t_sp;
                const u32 te = tn < t_x ? tn : t_x;
                if (t < te && np < PATTERN_P) {
                    for (; t < te && st[t].p < PATTERN_P; t++) pattern_step(t);
                    if (t < te) load_step(t);
                }
                if (t < te) {
                    const bool upd = !(lazy || stale);
                    stale = !upd;
                    cross_steps(t, te, upd);
                }
                t = tn;
                if (tn >= t_sp) break;
                lf &= lf - 1;
                if (t < t_x) load_step(t);
                const u32 b = bb + t, fl = st[t].flags;
                int tl = 0;
                u32 j0, j1;
                leaf_bounds(t, j0, j1);
                fresh_blocks();
                block_prefix();
                const u64 xp = st[t].xp;
                auto one_leaf = [&](const uint4& r) {
                    // no early exit: a lane without a leaf of b (no entry, lpf <= p_b, or
                    // gpf > p_a) runs the same code and adds 0; its block index is clamped
                    // in count_to, so its reads stay inside the sub-range
                    const bool valid = r.z > 2 * b + 1 && r.w <= gmax;
                    const u32 c = count_to(leaf_end(xp, r));
                    const i32 sg = valid ? ((r.z & 1u) ? 1 : -1) : 0;
                    acc += (i64)sg * (i32)c;
                    tl += sg;
                    nleaves += valid;
                };
                uint4 nr = no_leaf;
                if (j0 + 32 + lane < j1) nr = leaf_rec(fl, j0 + 32 + lane);           // second 32 in flight
                one_leaf(pf);                                                         // first 32, loaded ahead
                if (lf) prefetch(__ffsll((long long)lf) - 1);                         // next leaf step
                for (u32 base = j0 + 32; base < j1; base += 32) {                     // the rest
                    const uint4 r = nr;
                    nr = base + 32 + lane < j1 ? leaf_rec(fl, base + 32 + lane) : no_leaf;   // next 32 in flight
                    one_leaf(r);
                }
                tl = __reduce_add_sync(0xffffffffu, (u32)tl);
                if (lane == 0) tw[t * nw + w] = tl;   // steps without leaves keep the 0 set above
                __syncwarp();   // its reads before the next step's crossings
            }
            if (t_x < t_sp && lane == 0) cw[t_x * nw + w] = cnt;   // b = B_s: leaves only
            __syncwarp();
            if (t_sp < nb) sparse_runs(t_sp);
            __syncthreads();
            // D: segment rows, and the carries between the CTA's sub-ranges
            for (u32 t = tid; t < nb; t += NT) {
                const u32 b = bb + t;
                u32 C = 0;
                for (u32 k = 0; k < nw; k++) C += cw[t * nw + k];
                const u32 at = st[t].row + (u32)s;
                if (b < Bs) A.counts[at] = C;
                if (b > A.kleaf) {
                    const u32* cp = t ? cw + (t - 1) * nw : prev;
                    i32 T = 0;
                    i64 intra = 0, run = 0;
                    for (u32 k = 0; k < nw; k++) {
                        const i32 tk = tw[t * nw + k];
                        T += tk;
                        intra += (i64)tk * run;
                        run += cp[k];
                    }
                    A.tallies[at] = T;   // one item owns the step
                    acc += intra;
                }
            }
            __syncthreads();
            if (tid < nw) prev[tid] = cw[(nb - 1) * nw + tid];
        }
    }
    i128 tot = block_sum_i128((i128)acc, red);
    if (MULTI) {
        if (tid == 0 && cur_q != ~0u) mq_atomic_add_i128(M.qacc + (u64)cur_q * M.qstride, tot);
    } else {
        if (tid == 0 && tot != 0) mq_atomic_add_i128(A0.acc, tot);
    }
    unsigned long long nleaves64 = nleaves, nclears64 = nclears;
    for (int o = 16; o; o >>= 1) {
        nleaves64 += __shfl_xor_sync(0xffffffffu, nleaves64, o);
        nclears64 += __shfl_xor_sync(0xffffffffu, nclears64, o);
    }
    if (lane == 0 && nleaves64) atomicAdd(A0.stat, nleaves64);
    if (lane == 0 && nclears64) atomicAdd(A0.stat + 1, nclears64);
    if (lane == 0 && nbusy) atomicAdd(A0.stat + 2, nbusy);     // busy (warp, step) pairs
    if (lane == 0 && nleafy) atomicAdd(A0.stat + 3, nleafy);   // of which with leaves
}

// ---------------------------------------------------------- schedule
// B_s of segment s: the primes p_b, b <= bmax, with p_b^2 <= x / L and p_b^2 <= L + span - 1
__device__ __forceinline__ u32 seg_b(u64 x, u64 s, u64 span, u32 bmax, const PiTable& pit)
{
    const u64 L = s * span;
    u64 n = L + span - 1;
    if (s) n = pc_min(n, x / L);
    const u64 r = pc_isqrt(n);   // at most x^(1/4) when L > 0
    return r > pit.limit ? bmax : (u32)pc_min(pi_lookup(pit, r), (u64)bmax);
}

// The segments of row b in [s0, s1), those with B_s >= b: first segment and number.
// p_b^2 <= L + span - 1 from segment p_b^2 / span on, p_b^2 <= x / L up to L = x / p_b^2.
PC_HD u32 row_range(u64 x, u64 p, u64 span, u64 nseg, u64 s0, u64 s1, u32* first)
{
    const u64 lo = pc_max(p * p / span, s0);
    const u64 hi = pc_min(pc_min(x / (p * p) / span + 1, nseg), s1);
    *first = (u32)lo;
    return hi > lo ? (u32)(hi - lo) : 0u;
}

// phi(L - 1, b - 1) at the first segment of row b: L <= p_b^2, so only 1 and the primes from
// p_b on are left (a shard that starts later has it in start)
__device__ __forceinline__ u64 row_start(const HardArgs& A, u32 b)
{
    const u64 p = A.primes[b], lo = p * p / A.span;
    if (lo < A.s0) return A.start[b - 1 - A.k0];
    if (lo == 0) return 0;
    const u64 n = pi_lookup(A.pit, lo * A.span - 1);   // below p_b^2 <= isqrt(x)
    return n >= b ? n - b + 2 : 1;
}

// The run's schedule in one launch.  The first segblocks blocks take a warp per segment s in
// [s0, s1): B_s, and an upper bound of its hard leaves (the lpf filter of the m-list is not
// applied), its lanes over the segment's leaf primes b (kleaf < b <= min(B_s, a)).  The others
// take a thread per row b: its segments.
__global__ void __launch_bounds__(256) hard_prep_kernel(HardArgs A, u32 segblocks, u32* segB, unsigned long long* est,
                                                        u32* len, u32* rlo)
{
    if (blockIdx.x >= segblocks) {
        const u32 t = (blockIdx.x - segblocks) * blockDim.x + threadIdx.x, b = A.k0 + t;
        if (b <= A.bmax) len[t] = row_range(A.x, A.primes[b], A.span, A.nseg, A.s0, A.s1, rlo + t);
        return;
    }
    const u64 s = A.s0 + ((u64)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    const u32 lane = threadIdx.x & 31;
    if (s >= A.s1) return;   // the whole warp
    const u64 L = s * A.span;
    u32 B = 0;
    u64 v = 0;
    if (lane == 0) B = seg_b(A.x, s, A.span, A.bmax, A.pit);
    if (lane < 2) v = L + lane * A.span;
    v = v ? ~0ull / v : 0;   // reciprocals of L (0 for L = 0) and L + span
    B = __shfl_sync(0xffffffffu, B, 0);
    const u64 vL = __shfl_sync(0xffffffffu, v, 0), vLs = __shfl_sync(0xffffffffu, v, 1);
    const u64 bhi = pc_min((u64)B, A.a);
    u64 n = 0;
    for (u64 b = A.kleaf + 1 + lane; b <= bhi; b += 32) {
        const u64 p = A.primes[b];
        const u64 vp = A.primes_rcp[b];
        const u64 xp = div_rcp(A.x, p, vp);
        u64 mlo, mhi;
        if (!leaf_window(A, p, vp, xp, L, vL, vLs, mlo, mhi)) continue;
        if (p * p > A.y) {
            const u64 k0 = pc_min(pc_max(pi_lookup(A.pit, mlo), b), A.a);
            const u64 k1 = pc_min(pc_max(pi_lookup(A.pit, mhi), b), A.a);
            n += k1 - k0;
        } else {
            n += rank_lookup(A.rk, mhi) - rank_lookup(A.rk, mlo);
        }
    }
    for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) {
        segB[s] = B;
        est[s] = n;
    }
}

// S2_hard carries: for each leaf prime b, the exclusive scan over segments
// of count(., b-1) dotted with tally(., b).
template <int NT>
__global__ void __launch_bounds__(NT) hard_combine_kernel(HardArgs A, I128Pair* out)
{
    __shared__ u64 wsum[NT / 32];
    __shared__ u64 s_carry;
    __shared__ i128 red[32];
    const u32 lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    i128 dot = 0;
    for (u32 b = A.kleaf + 1 + blockIdx.x; b <= A.bmax; b += gridDim.x) {
        const u64 row = A.off[b - A.k0];
        const u64 Sb = A.off[b - A.k0 + 1] - row;
        if (Sb == 0) continue;
        // row b - 1 holds every segment of row b
        const u64 prow = A.off[b - 1 - A.k0] + (A.rlo[b - A.k0] - A.rlo[b - 1 - A.k0]);
        if (threadIdx.x == 0) s_carry = row_start(A, b);
        __syncthreads();
        for (u64 base = 0; base < Sb; base += NT) {
            const u64 s = base + threadIdx.x;
            const u64 v = s < Sb ? (u64)A.counts[prow + s] : 0;
            u64 incl = v;
            for (int o = 1; o < 32; o <<= 1) {
                u64 t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) wsum[wid] = incl;
            __syncthreads();
            if (wid == 0) {
                u64 w = lane < NT / 32 ? wsum[lane] : 0, wi = w;
                for (int o = 1; o < 32; o <<= 1) {
                    u64 t = __shfl_up_sync(0xffffffffu, wi, o);
                    if (lane >= o) wi += t;
                }
                if (lane < NT / 32) wsum[lane] = wi - w;
            }
            __syncthreads();
            const u64 c0 = s_carry;
            const u64 carry = c0 + wsum[wid] + incl - v;
            if (s < Sb) {
                const i32 tl = A.tallies[row + s];
                if (tl) dot += (i128)tl * (i128)carry;
            }
            __syncthreads();
            if (threadIdx.x == NT - 1) s_carry = c0 + wsum[wid] + incl;
            __syncthreads();
        }
    }
    dot = block_sum_i128(dot, red);
    if (threadIdx.x == 0 && dot != 0) mq_atomic_add_i128(out, dot);
}

// ---------------------------------------------------------------- host
u32 pc_seg_bytes(pc_ctx* ctx, u32 dflt)
{
    u32 sb = ctx->params.seg_bytes ? ctx->params.seg_bytes : dflt;
    if (sb < 1024) sb = 1024;
    if (sb > MAX_SEG) sb = MAX_SEG;
    if (sb > 4096) sb = sb / 4096 * 4096;
    else if (sb > 2048) sb = 4096 > sb ? 2048 : 4096;   // sub-ranges are powers of two
    else sb = sb / 1024 * 1024;
    return sb;
}

// Geometry of the hard-leaf sieve over [0, z] for one query: segment bytes and warp sub-range
// bytes.  A warp walks its steps one after the other (a microsecond each), so while the
// sub-ranges are fewer than the warps the chip holds (152 x 16), smaller ones shorten the
// chain; once they are many, larger ones do fewer steps per integer.  The lines lie where the
// sieve's time crosses on GB300 (8 KiB / 1 KiB against 32 KiB / 8 KiB: 0.088 / 0.223 ms at
// z = 8e5, 0.193 / 0.324 at 6e6, 0.375 / 0.565 at 9e7; 16 KiB / 2 KiB 0.51 / 0.67 at 1.4e8;
// 16 KiB / 4 KiB 0.825 / 1.03 at 3.3e8, 2.67 / 2.75 at 1.5e9, 4.91 / 4.65 at 3e9).
static u32 hard_sub_for(u64 z)
{
    return z < 120000000ull ? 1024 : z < 280000000ull ? 2048 : z < 2000000000ull ? 4096 : 8192;
}

static constexpr u32 HARD_SEG_TOP = 32768;
u32 hard_seg_for(u64 z)
{
    return z < 400000ull ? 2048 : z < 120000000ull ? 8192 : z < 2000000000ull ? 16384 : HARD_SEG_TOP;
}

// bytes per warp sub-range: a power of two dividing seg_bytes, at most 16 warps
static u32 pc_sub_bytes(pc_ctx* ctx, u32 seg_bytes, u32 dflt)
{
    u32 wb = ctx->params.warp_bytes ? ctx->params.warp_bytes : dflt;
    if (wb > MAX_SUB) wb = MAX_SUB;
    if (wb > seg_bytes) wb = seg_bytes;
    while (seg_bytes % wb) wb >>= 1;
    while (seg_bytes / wb > MAX_NW) wb <<= 1;
    return wb;
}

// The sieve's geometry from the two defaults.  Above 16 x 4096 bytes only 8192-byte sub-ranges
// are few enough, so a segment of an odd multiple of 4096 there is rounded down to a multiple
// of 8192: the sub-ranges have to tile it, or its last bytes belong to no warp.
static int set_geometry(pc_ctx* ctx, HardArgs& A, u32 seg_dflt, u32 sub_dflt)
{
    A.seg_bytes = pc_seg_bytes(ctx, seg_dflt);
    if (A.seg_bytes > MAX_NW * (MAX_SUB / 2)) A.seg_bytes = A.seg_bytes / MAX_SUB * MAX_SUB;
    A.sub_bytes = pc_sub_bytes(ctx, A.seg_bytes, sub_dflt);
    A.nw = A.seg_bytes / A.sub_bytes;
    if (A.nw * A.sub_bytes != A.seg_bytes) {
        pc_set_error(ctx, "hard-leaf sieve: sub-ranges of %u bytes do not tile a segment of %u", A.sub_bytes, A.seg_bytes);
        return PC_EINVAL;
    }
    A.sub_shift = 3;
    while ((1u << A.sub_shift) < A.sub_bytes * 8) A.sub_shift++;
    A.span = 30ull * A.seg_bytes;
    A.dspan = 30ull * A.sub_bytes;
    return PC_OK;
}

// Work items, planned on the device: segments, heavy ones split into replicas.  Cost of a
// segment (seg_cost, in units of one leaf): 128 for each of its (segment, prime) steps, 0.08
// for each crossing (by Mertens' theorem span * 8/30 * sum_{13 <= p <= P} 1/p ~
// span * 8/30 * (ln ln P - 1.0056), P the largest prime the segment sieves with) and its
// estimated hard leaves.  A segment whose leaves outweigh both its sieve and a fair share of
// the launch (total / (4 * resident CTAs)) becomes R replicas that share its
// leaves.  Items are handed out largest first from an atomic counter, ordered
// by cost in buckets of a quarter octave (the order only balances the load).
static constexpr int PLAN_BUCKETS = 128;

struct PlanScratch {
    double total;                 // cost of every segment of the run
    unsigned long long nitems;    // items planned
    u32 cnt[PLAN_BUCKETS];        // items per cost bucket
    u32 cur[PLAN_BUCKETS];        // next free slot of each bucket
    u32 nheavy;                   // segments split into replicas
    u32 pad;
};

struct HeavySeg {
    u32 s;     // segment
    u32 pos;   // its first item
    u32 R;     // its replicas (items pos .. pos + R - 1)
    u32 pad;
};

struct PlanArgs {
    const u32* segB;
    const unsigned long long* est;
    u32 k0;
    float x, z;
    u64 span, s0, s1;
    double inv_ctas4;           // 1 / (4 * resident CTAs)
    u32 ctas;
    u64 cap;                    // slots in items
    PlanScratch* scr;
    u32* split;                 // per segment: R | bucket << 16 (R = 0: no item)
    HardItem* items;
    HeavySeg* heavy;            // the segments with R > 1
    unsigned long long* stat;   // [4] items, [5] item steps, [6] set when cap was too small,
                                // [7] steps replicas cross off before their own
};

__device__ __forceinline__ float seg_cost(const PlanArgs& P, u64 s)
{
    const float steps = (float)(P.segB[s] - P.k0);
    const float sz = sqrtf(P.z);
    const float top = fminf(sqrtf((float)(s + 1) * (float)P.span), sz);
    const float pm = s ? fminf(sqrtf(P.x / ((float)s * (float)P.span)), top) : top;
    const float ll = pm > 16.0f ? logf(logf(pm)) - 1.0056f : 0.0f;
    return 128.0f * steps + 0.08f * (float)P.span * (8.0f / 30.0f) * (ll > 0.0f ? ll : 0.0f);
}

// R and the cost bucket of segment s: R | bucket << 16, or 0 for a segment without steps
__device__ __forceinline__ u32 seg_split(const PlanArgs& P, u64 s, float target)
{
    if (P.segB[s] <= P.k0) return 0;
    const float base = seg_cost(P, s), e = (float)P.est[s];
    u32 R = 1;
    if (base + e > target && e > base) {
        const float room = fmaxf(target - base, base);
        R = (u32)fminf(1024.0f, ceilf(e / fmaxf(room, 1.0f)));
        if (R < 1) R = 1;
    }
    const int k = (int)floorf(4.0f * log2f((base + e) / R));   // a replica's share
    const u32 key = (u32)(k < 0 ? 0 : (k >= PLAN_BUCKETS ? PLAN_BUCKETS - 1 : k));
    return R | (key << 16);
}

__global__ void plan_cost_kernel(PlanArgs P)
{
    __shared__ double part[32];
    double t = 0;
    for (u64 s = P.s0 + (u64)blockIdx.x * blockDim.x + threadIdx.x; s < P.s1; s += (u64)gridDim.x * blockDim.x)
        if (P.segB[s] > P.k0) t += seg_cost(P, s) + (double)P.est[s];
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0;
        for (u32 k = 0; k < blockDim.x / 32; k++) b += part[k];
        atomicAdd(&P.scr->total, b);
    }
}

// the split of every segment, decided once and stored
__global__ void plan_split_kernel(PlanArgs P)
{
    const float target = fmaxf((float)(P.scr->total * P.inv_ctas4), 1.0f);
    for (u64 s = P.s0 + (u64)blockIdx.x * blockDim.x + threadIdx.x; s < P.s1; s += (u64)gridDim.x * blockDim.x) {
        const u32 v = seg_split(P, s, target);
        if (v) {
            atomicAdd(&P.scr->cnt[v >> 16], v & 0xFFFFu);
            atomicAdd(&P.stat[5], (unsigned long long)(P.segB[s] - P.k0));
        }
        P.split[s] = v;
    }
}

// first slot of every bucket, the most costly bucket first (one block)
__global__ void plan_offsets_kernel(PlanArgs P)
{
    if (threadIdx.x != 0) return;
    unsigned long long run = 0;
    for (int k = PLAN_BUCKETS - 1; k >= 0; k--) {
        P.scr->cur[k] = (u32)run;
        run += P.scr->cnt[k];
    }
    if (run > P.cap) {   // cannot happen with cap = segments + 8 * CTAs; the run reports it
        P.stat[6] = 1;
        run = 0;
    }
    P.scr->nitems = run;
    P.stat[4] = run;
}

__global__ void plan_scatter_kernel(PlanArgs P)
{
    if (P.stat[6]) return;
    for (u64 s = P.s0 + (u64)blockIdx.x * blockDim.x + threadIdx.x; s < P.s1; s += (u64)gridDim.x * blockDim.x) {
        const u32 v = P.split[s], R = v & 0xFFFFu;
        if (!R) continue;
        const u32 pos = atomicAdd(&P.scr->cur[v >> 16], R);
        // replica 0 starts at the first step; the others get their steps in plan_bsplit_kernel
        for (u32 r = 0; r < R; r++) P.items[pos + r] = HardItem{(u32)s, r ? ~0u : P.k0 + 1, ~0u, 0u};
        if (R > 1) P.heavy[atomicAdd(&P.scr->nheavy, 1u)] = HeavySeg{(u32)s, pos, R, 0u};
    }
}

// The planner in one launch (one CTA) for up to PLAN_ONE segments: the same decisions, with the
// buckets in shared memory.  When the items are fewer than the launch's CTAs, every segment is
// split further, to at least FILL_STEPS steps a replica: the steps of an item are a serial chain,
// and the crossings a replica repeats are done by the whole CTA at once (pi(10^9) 0.125 -> 0.11 ms,
// pi(10^11) 0.21 -> 0.155, pi(10^12) 0.256 -> 0.19; with 8, 16, 32 steps pi(10^11) 0.169, 0.167, 0.195).
// (Four launches and their gaps cost more than the work: pi(10^12) plans 26 segments.)
static constexpr u64 PLAN_ONE = 8192;
static constexpr u32 FILL_STEPS = 4;
__global__ void __launch_bounds__(1024) plan_one_kernel(PlanArgs P)
{
    __shared__ double part[32];
    __shared__ u32 cnt[PLAN_BUCKETS], cur[PLAN_BUCKETS];
    __shared__ u32 nheavy, ok, n0;
    __shared__ unsigned long long steps;
    const u32 tid = threadIdx.x;
    if (tid < PLAN_BUCKETS) cnt[tid] = 0;
    if (tid == 0) nheavy = n0 = 0, steps = 0;
    double t = 0;
    unsigned long long st = 0;
    for (u64 s = P.s0 + tid; s < P.s1; s += 1024)
        if (P.segB[s] > P.k0) {
            t += seg_cost(P, s) + (double)P.est[s];
            st += P.segB[s] - P.k0;
        }
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((tid & 31) == 0) part[tid >> 5] = t;
    __syncthreads();
    if (st) atomicAdd(&steps, st);
    double total = 0;
    for (u32 k = 0; k < 32; k++) total += part[k];
    const float target = fmaxf((float)(total * P.inv_ctas4), 1.0f);
    for (u64 s = P.s0 + tid; s < P.s1; s += 1024) {
        const u32 v = seg_split(P, s, target);
        P.split[s] = v;
        if (v) atomicAdd(&n0, v & 0xFFFFu);
    }
    __syncthreads();
    const u32 fill = n0 && n0 < P.ctas ? P.ctas / n0 : 1;   // items grow to at most the CTAs
    for (u64 s = P.s0 + tid; s < P.s1; s += 1024) {
        u32 v = P.split[s];
        if (fill > 1 && v) {
            const u32 R = v & 0xFFFFu, most = (P.segB[s] - P.k0) / FILL_STEPS;
            const u32 R2 = R * fill < most ? R * fill : (most > R ? most : R);
            // the share's bucket falls by four per halving, as in seg_split
            const int key = (int)(v >> 16) - (int)(4.0f * log2f((float)R2 / (float)R));
            P.split[s] = v = R2 | (u32)(key < 0 ? 0 : key) << 16;
        }
        if (v) atomicAdd(&cnt[v >> 16], v & 0xFFFFu);
    }
    __syncthreads();
    if (tid == 0) {   // first slot of every bucket, the most costly bucket first
        unsigned long long run = 0;
        for (int k = PLAN_BUCKETS - 1; k >= 0; k--) {
            cur[k] = (u32)run;
            run += cnt[k];
        }
        ok = run <= P.cap;   // always, with cap = segments + 8 * CTAs; the run reports it if not
        P.scr->nitems = P.stat[4] = ok ? run : 0;
        P.stat[5] = steps;
        P.stat[6] = ok ? 0 : 1;
    }
    __syncthreads();
    if (ok)
        for (u64 s = P.s0 + tid; s < P.s1; s += 1024) {
            const u32 v = P.split[s], R = v & 0xFFFFu;
            if (!R) continue;
            const u32 pos = atomicAdd(&cur[v >> 16], R);
            for (u32 r = 0; r < R; r++) P.items[pos + r] = HardItem{(u32)s, r ? ~0u : P.k0 + 1, ~0u, 0u};
            if (R > 1) P.heavy[atomicAdd(&nheavy, 1u)] = HeavySeg{(u32)s, pos, R, 0u};
        }
    __syncthreads();
    if (tid == 0) P.scr->nheavy = nheavy;
}

// Estimated cost of step b of the segment [L, L + span), in the units of seg_cost (one
// leaf = 1): 128 for the step, 0.08 per crossing, plus its hard leaves (upper bound, as in
// hard_prep_kernel).  Integer, so that prefix sums are exact.
__device__ __forceinline__ unsigned long long step_cost(const HardArgs& A, u32 b, u64 L, u64 vL, u64 vLs)
{
    const u64 p = A.primes[b], vp = A.primes_rcp[b];
    unsigned long long c = 128 + (16ull * A.seg_bytes / p) / 25;
    if (b > A.kleaf && b <= A.a) {
        const u64 xp = div_rcp(A.x, p, vp);
        u64 mlo, mhi;
        if (leaf_window(A, p, vp, xp, L, vL, vLs, mlo, mhi)) {
            if (p * p > A.y) {
                const u64 k0 = pc_min(pc_max(pi_lookup(A.pit, mlo), b), A.a);
                const u64 k1 = pc_min(pc_max(pi_lookup(A.pit, mhi), b), A.a);
                c += k1 - k0;
            } else {
                c += rank_lookup(A.rk, mhi) - rank_lookup(A.rk, mlo);
            }
        }
    }
    return c;
}

// The steps of a heavy segment's replicas: replica r owns the steps from the first b
// whose cost before it reaches r / R of the segment's total (one CTA per segment; a
// prefix sum of exact integer costs, so every step goes to exactly one replica).
__global__ void __launch_bounds__(256) plan_bsplit_kernel(HardArgs A, PlanArgs P)
{
    __shared__ unsigned long long wsum[8];
    __shared__ unsigned long long s_tot;
    const u32 tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (P.stat[6]) return;
    const u32 nh = P.scr->nheavy;
    for (u32 h = blockIdx.x; h < nh; h += gridDim.x) {
        const HeavySeg hs = P.heavy[h];
        const u64 s = hs.s, L = s * A.span, R = hs.R;
        const u32 Bs = A.segB[s];
        const u64 vL = L ? ~0ull / L : 0, vLs = ~0ull / (L + A.span);
        const u32 nsteps = Bs - A.k0, per = (nsteps + 255) / 256;
        const u32 b0 = pc_min((u64)A.k0 + 1 + (u64)tid * per, (u64)Bs + 1), b1 = pc_min((u64)b0 + per, (u64)Bs + 1);
        unsigned long long mine = 0;
        for (u32 b = b0; b < b1; b++) mine += step_cost(A, b, L, vL, vLs);
        unsigned long long incl = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        if (tid == 0) {
            unsigned long long run = 0;
            for (u32 k = 0; k < 8; k++) {
                const unsigned long long v = wsum[k];
                wsum[k] = run;
                run += v;
            }
            s_tot = run;
        }
        __syncthreads();
        const unsigned long long T = s_tot;
        unsigned long long before = wsum[wid] + incl - mine;
        for (u32 b = b0; b < b1; b++) {
            const unsigned long long after = before + step_cost(A, b, L, vL, vLs);
            // replicas r with R * before < r * T <= R * after start right after step b
            u64 r_hi = R * after / T;
            if (r_hi > R - 1) r_hi = R - 1;
            for (u64 r = R * before / T + 1; r <= r_hi; r++) {
                P.items[hs.pos + r].b_lo = b + 1;
                P.items[hs.pos + r - 1].b_hi = b + 1;
                if (b + 1 <= Bs) atomicAdd(&P.stat[7], (unsigned long long)(b - A.k0));
            }
            before = after;
        }
        __syncthreads();
    }
}

static size_t hard_smem(const HardArgs& A)
{
    static_assert(sizeof(StepInfo) % 16 == 0, "StepInfo must keep 16-byte alignment");
    return BATCH * sizeof(StepInfo) + A.seg_bytes + (size_t)A.nw * (A.sub_bytes >> 5) * 4 +
           (size_t)BATCH * (A.nw + 1) * 4 + 2 * (size_t)BATCH * A.nw * 4 + (size_t)BATCH * A.nw * 16 +
           (size_t)A.nw * LOG_CAP * sizeof(u16);
}

// The instantiation: the most resident warps (registers and shared memory permitting), or
// at least ctas_per_sm resident CTAs when that is set; *per_sm its resident CTAs (<= 8).
template <bool MULTI>
static int choose_hard_kernel(pc_ctx* ctx, const HardArgs& A, size_t smem, void (**out)(HardArgs, MultiArgs),
                              int* out_per_sm)
{
    struct Variant {
        void (*fn)(HardArgs, MultiArgs);
        int maxt, minb;
    };
    static const Variant variants[] = {{hard_sieve_kernel<512, 1, MULTI>, 512, 1},
                                       {hard_sieve_kernel<256, 3, MULTI>, 256, 3},
                                       {hard_sieve_kernel<512, 2, MULTI>, 512, 2},
                                       {hard_sieve_kernel<256, 4, MULTI>, 256, 4}};
    const int nt = 32 * (int)A.nw;
    const bool other_seg = ctx->ctas_seg_call && ctx->ctas_seg_call != A.seg_bytes;   // tuned at another size
    const int want = (int)(ctx->params.ctas_per_sm ? ctx->params.ctas_per_sm : other_seg ? 0 : ctx->ctas_call);
    if (!MULTI && ctx->hk.fn && ctx->hk.nt == nt && ctx->hk.smem == smem && ctx->hk.want == want) {
        *out = (void (*)(HardArgs, MultiArgs))ctx->hk.fn;
        *out_per_sm = ctx->hk.per_sm;
        return PC_OK;
    }
    void (*kern)(HardArgs, MultiArgs) = nullptr;
    int per_sm = 0;
    for (const Variant& v : variants) {
        if (nt > v.maxt) continue;
        // The limit is a property of the kernel, shared by every host thread of the
        // process: always raise it to the device maximum (never to this call's size),
        // so that a concurrent query with larger segments is not cut short.
        cudaFuncAttributes fa;
        PC_CUDA(ctx, cudaFuncGetAttributes(&fa, v.fn));
        const size_t dyn_max = ctx->smem_optin - fa.sharedSizeBytes;
        if (smem > dyn_max) {
            pc_set_error(ctx, "hard-leaf sieve: %zu bytes of shared memory per CTA", smem);
            return PC_EINVAL;
        }
        cudaError_t ea = cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn_max);
        if (ea != cudaSuccess) {
            pc_set_error(ctx, "cudaFuncSetAttribute(smem=%zu): %s", dyn_max, cudaGetErrorString(ea));
            return PC_ECUDA;
        }
        int fit = 0;   // resident CTAs the SM can hold (registers and shared memory)
        PC_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, v.fn, nt, smem));
        if (fit < 1) continue;
        if (want) {
            // the least register-constrained variant reaching the requested residency
            if (!kern || (per_sm < want && fit > per_sm)) {
                kern = v.fn;
                per_sm = fit;
            }
        } else if (fit > per_sm) {
            kern = v.fn;
            per_sm = fit;
        }
    }
    if (!kern) {
        pc_set_error(ctx, "hard-leaf sieve: no launch configuration fits (smem=%zu, threads=%d)", smem, nt);
        return PC_EINVAL;
    }
    if (want && per_sm > want) per_sm = want;
    if (per_sm > 8) per_sm = 8;   // 32 KiB segments fit 4; smaller ones (autotuned, or set) up to 8
    *out = kern;
    *out_per_sm = per_sm;
    if (!MULTI) {
        ctx->hk.nt = nt, ctx->hk.smem = smem, ctx->hk.want = want;
        ctx->hk.fn = (void*)kern, ctx->hk.per_sm = per_sm;
    }
    return PC_OK;
}

// primes below 2^16 (a run's sieving primes are at most x^(1/4) < 55109), p_1 at index 1
static const std::vector<u32>& host_primes()
{
    static const std::vector<u32> ps = [] {
        std::vector<u32> v(1, 1);
        std::vector<char> comp(65536, 0);
        for (u32 i = 2; i < 65536; i++) {
            if (comp[i]) continue;
            v.push_back(i);
            for (u64 j = (u64)i * i; j < 65536; j += i) comp[j] = 1;
        }
        return v;
    }();
    return ps;
}

int run_hard_sieve(pc_ctx* ctx, const LeafProblem& P, I128Pair* out)
{
    HardArgs A{};
    A.x = P.x;
    A.y = P.y;
    A.z = P.z;
    A.c = P.c;
    A.k0 = P.c >= 5 ? 5 : (P.c == 4 ? 4 : 3);
    A.kleaf = P.c > A.k0 ? P.c : A.k0;
    A.a = P.a;
    A.trunc = P.trunc;
    // A shard's bounds, and with them its value, are counted in segments: shards keep 32 KiB
    // whatever z, so that parts summed from several processes do not hang on the rule by z.
    // One tuned size serves a whole decade of x, over which z grows more than fourfold: sizes up to
    // the rule's largest are limits on the rule's, so that the tuner can keep the rule (32 KiB)
    // and small z keep their segments (tuned 16 KiB as a limit and as the size itself: pi(7e12)
    // 0.31 and 0.38 ms, pi(3e11) 0.156 and 0.182).
    const u32 rule = hard_seg_for(P.z), tuned = ctx->seg_call;
    const u32 seg = tuned > HARD_SEG_TOP || (tuned && tuned < rule) ? tuned : rule;
    PC_TRY(set_geometry(ctx, A, P.shard_n ? 32768 : seg, P.shard_n ? 8192 : hard_sub_for(P.z)));
    A.nseg = P.z / A.span + 1;
    A.s0 = 0;
    A.s1 = A.nseg;
    if (P.shard_n) {
        A.s0 = A.nseg * P.shard_k / P.shard_n;
        A.s1 = A.nseg * (P.shard_k + 1) / P.shard_n;
        if (A.s1 <= A.s0) return PC_OK;   // an empty shard
    }
    const u64 bmax = pc_min(pc_min(P.B, P.a), P.R4);
    std::vector<u64> hstart;
    if (P.shard_n && A.s0 && bmax > A.kleaf) {
        // carries into the shard: phi(L - 1, b) for every b (Section 4), computed before
        // this run launches anything (the queries may grow the tables) or claims scratch
        hstart.resize(bmax - A.k0 + 1);
        PC_TRY(phi_starts(ctx, A.s0 * A.span - 1, A.k0, bmax, hstart.data()));
    }
    if (!P.table_in_easy) PC_TRY(run_hard_table(ctx, P, A.kleaf, A.s0 * A.span, A.s1 * A.span, out));
    if (bmax <= A.kleaf) return PC_OK;   // no hard leaf needs the sieve
    A.bmax = (u32)bmax;
    A.pit = ctx->T.pi();
    A.rk = ctx->T.rank();
    A.ml = ctx->T.mlist();
    A.nsl = ctx->T.n_sl;
    for (int k = 0; k < Tables::NSUB; k++) {
        A.sl[k] = ctx->T.sublist(k);
        A.srk[k] = ctx->T.subrank(k);
        A.slK[k] = k < (int)A.nsl ? ctx->T.sl_K[k] : ~0u;
    }
    A.primes = ctx->T.primes.as<u32>();
    A.primes_rcp = ctx->T.primes_rcp.as<u64>();
    A.primes_dv = ctx->T.primes_dv.as<uint2>();
    A.pat = ctx->T.pat16.as<uint4>();

    const u64 nrows = bmax - A.k0 + 1;
    const u64 ns = A.s1 - A.s0;
    PC_TRY(buf_reserve(ctx, ctx->seg_b, A.nseg * sizeof(u32) + 2 * (nrows + 1) * sizeof(u32)));
    PC_TRY(buf_reserve(ctx, ctx->seg_off, (nrows + 1) * sizeof(u64) + A.nseg * sizeof(u64) + A.nseg * sizeof(u32) +
                                              A.nseg * sizeof(HeavySeg) + 16));
    u32* segB = ctx->seg_b.as<u32>();
    u32* rowlen = segB + A.nseg;
    u32* rlo = rowlen + nrows + 1;
    u64* off = ctx->seg_off.as<u64>();
    unsigned long long* est = (unsigned long long*)(off + nrows + 1);
    u32* split = (u32*)(est + A.nseg);   // the work-item split of every segment
    HeavySeg* heavy = (HeavySeg*)(((uintptr_t)(split + A.nseg) + 15) & ~(uintptr_t)15);
    const u32 segblocks = (u32)((ns + 7) / 8);
    hard_prep_kernel<<<segblocks + (unsigned)((nrows + 255) / 256), 256, 0, ctx->stream>>>(A, segblocks, segB, est,
                                                                                          rowlen, rlo);
    PC_LAUNCHED(ctx);
    ctx->stats.kernel_launches++;
    PC_TRY(scan_exclusive_u32_to_u64(ctx, rowlen, off, nrows));
    A.segB = segB;
    A.off = off;
    A.rlo = rlo;
    A.start = nullptr;
    if (!hstart.empty()) {
        PC_TRY(buf_reserve(ctx, ctx->starts, hstart.size() * sizeof(u64)));
        PC_CUDA(ctx, cudaMemcpyAsync(ctx->starts.p, hstart.data(), hstart.size() * sizeof(u64),
                                     cudaMemcpyHostToDevice, ctx->stream));
        A.start = ctx->starts.as<u64>();
        PC_CUDA(ctx, cudaStreamSynchronize(ctx->stream));   // hstart is pageable memory of this call
    }
    // entries of the count and tally rows, as the device lays them out
    u64 total = 0;
    const std::vector<u32>& hp = host_primes();
    for (u64 b = A.k0; b <= bmax; b++) {
        u32 first;
        total += row_range(P.x, hp[b], A.span, A.nseg, A.s0, A.s1, &first);
    }
    ctx->stats.steps = total;
    if (total >> 32) {
        pc_set_error(ctx, "hard-leaf sieve: %llu count rows exceed 32-bit offsets", (unsigned long long)total);
        return PC_EOVERFLOW;
    }

    const size_t smem = hard_smem(A);
    void (*kern)(HardArgs, MultiArgs) = nullptr;
    int per_sm = 0;
    PC_TRY(choose_hard_kernel<false>(ctx, A, smem, &kern, &per_sm));
    int ctas = ctx->sm_count * per_sm;

    // the work items, planned on the device
    const u64 cap = ns + 8ull * (u64)ctas + 64;
    const size_t items_bytes = (cap * sizeof(HardItem) + 15) / 16 * 16;
    PC_TRY(buf_reserve(ctx, ctx->counts, total * sizeof(u32)));
    PC_TRY(buf_reserve(ctx, ctx->tallies, total * sizeof(i32)));
    PC_TRY(buf_reserve(ctx, ctx->acc_seg, items_bytes + sizeof(PlanScratch)));
    HardItem* ditems = ctx->acc_seg.as<HardItem>();
    PlanScratch* scr = (PlanScratch*)(ctx->acc_seg.as<unsigned char>() + items_bytes);
    A.counts = ctx->counts.as<u32>();
    A.tallies = ctx->tallies.as<i32>();
    A.items = ditems;
    A.nitems = &scr->nitems;
    A.acc = out;
    A.queue = (u32*)call_queue(ctx, Q_HARD);
    A.stat = call_hard_stat(ctx);
    PlanArgs PA{segB, est, A.k0, (float)P.x, (float)P.z, A.span, A.s0, A.s1, 1.0 / (4.0 * ctas), (u32)ctas, cap,
                scr, split, ditems, heavy, A.stat};
    if (ns <= PLAN_ONE) {
        plan_one_kernel<<<1, 1024, 0, ctx->stream>>>(PA);
        PC_LAUNCHED(ctx);
        ctx->stats.kernel_launches++;
    } else {
        const unsigned pg = (unsigned)pc_min((ns + 255) / 256, (u64)ctx->sm_count * 4);
        PC_CUDA(ctx, cudaMemsetAsync(scr, 0, sizeof(PlanScratch), ctx->stream));
        plan_cost_kernel<<<pg, 256, 0, ctx->stream>>>(PA);
        PC_LAUNCHED(ctx);
        plan_split_kernel<<<pg, 256, 0, ctx->stream>>>(PA);
        PC_LAUNCHED(ctx);
        plan_offsets_kernel<<<1, 32, 0, ctx->stream>>>(PA);
        PC_LAUNCHED(ctx);
        plan_scatter_kernel<<<pg, 256, 0, ctx->stream>>>(PA);
        PC_LAUNCHED(ctx);
        ctx->stats.kernel_launches += 4;
    }
    plan_bsplit_kernel<<<(unsigned)pc_min(ns, (u64)ctx->sm_count * 2), 256, 0, ctx->stream>>>(A, PA);
    PC_LAUNCHED(ctx);
    ctx->stats.kernel_launches++;

    PC_CUDA(ctx, cudaEventRecord(ctx->ev[0], ctx->stream));
    kern<<<ctas, 32 * A.nw, smem, ctx->stream>>>(A, MultiArgs{});
    PC_LAUNCHED(ctx);
    PC_CUDA(ctx, cudaEventRecord(ctx->ev[1], ctx->stream));
    ctx->hard_timed = true;
    hard_combine_kernel<256><<<(int)pc_min(bmax - A.kleaf, 4096), 256, 0, ctx->stream>>>(A, out);
    PC_LAUNCHED(ctx);
    ctx->stats.kernel_launches += 2;
    ctx->stats.segments = A.nseg;
    ctx->stats.seg_bytes = A.seg_bytes;
    return PC_OK;
}

// ------------------------------------------------------- many queries at once
// The hard leaves of every pi(x) query of a batch in one sieve launch over all their
// segments (largest queries first, since the batch sorts them so), with the segment
// schedule and the count rows of every query built by one launch each.

// B_s for segment g - pref[q] of query q
__global__ void mq_seg_b_kernel(const HardArgs* qa, const u64* pref, u32 Q, u32* segB)
{
    const u64 g = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= pref[Q]) return;
    const u64 q = mq_find(pref, Q + 1, g);
    const HardArgs& A = qa[q];
    const u64 s = g - pref[q];
    segB[g] = seg_b(A.x, s, A.span, A.bmax, A.pit);
}

// row b = k0 + g - rpref[q] of query q: its segments with B_s >= b
__global__ void mq_row_len_kernel(const HardArgs* qa, const u64* rpref, u32 Q, u32* len, u32* rlo)
{
    const u64 g = (u64)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= rpref[Q]) return;
    const u64 q = mq_find(rpref, Q + 1, g);
    const HardArgs& A = qa[q];
    const u32 b = A.k0 + (u32)(g - rpref[q]);
    len[g] = row_range(A.x, A.primes[b], A.span, A.nseg, 0, A.nseg, rlo + g);
}

// the carries: a warp per (query, b), kleaf < b <= bmax: the exclusive scan over
// segments of count(., b - 1) dotted with tally(., b), into the query's hard part
__global__ void mq_combine_kernel(const HardArgs* qa, const u64* cpref, u32 Q, I128Pair* parts)
{
    const u32 lane = threadIdx.x & 31;
    const u64 gw = ((u64)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = ((u64)gridDim.x * blockDim.x) >> 5;
    for (u64 g = gw; g < cpref[Q]; g += nwarps) {
        const u64 q = mq_find(cpref, Q + 1, g);
        const HardArgs& A = qa[q];
        const u32 b = A.kleaf + 1 + (u32)(g - cpref[q]);
        const u64 row = A.off[b - A.k0], Sb = A.off[b - A.k0 + 1] - row;
        if (Sb == 0) continue;
        const u64 prow = A.off[b - 1 - A.k0] + (A.rlo[b - A.k0] - A.rlo[b - 1 - A.k0]);
        u64 carry = row_start(A, b);
        i128 dot = 0;
        for (u64 base = 0; base < Sb; base += 32) {
            const u64 s = base + lane;
            const u64 v = s < Sb ? (u64)A.counts[prow + s] : 0;
            u64 incl = v;
            for (int o = 1; o < 32; o <<= 1) {
                const u64 t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (s < Sb) {
                const i32 tl = A.tallies[row + s];
                if (tl) dot += (i128)tl * (i128)(carry + incl - v);
            }
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        dot = warp_sum_i128(dot);
        if (lane == 0 && dot != 0) mq_atomic_add_i128(parts + 5 * q + 3, dot);
    }
}

int mq_hard(pc_ctx* ctx, const MQPlan& P)
{
    const u32 Q = P.Q;
    HardArgs T{};   // what every query of the batch shares: tables, geometry, queue, counters
    T.k0 = 5;
    T.kleaf = 5;
    PC_TRY(set_geometry(ctx, T, ctx->batch_seg ? ctx->batch_seg : 16384, 8192));
    T.pit = ctx->T.pi();
    T.rk = ctx->T.rank();
    T.ml = ctx->T.mlist();
    T.nsl = ctx->T.n_sl;
    for (int k = 0; k < Tables::NSUB; k++) {
        T.sl[k] = ctx->T.sublist(k);
        T.srk[k] = ctx->T.subrank(k);
        T.slK[k] = k < (int)T.nsl ? ctx->T.sl_K[k] : ~0u;
    }
    T.primes = ctx->T.primes.as<u32>();
    T.primes_rcp = ctx->T.primes_rcp.as<u64>();
    T.primes_dv = ctx->T.primes_dv.as<uint2>();
    T.pat = ctx->T.pat16.as<uint4>();
    // per query: segments, count rows b = k0 .. bmax, carried rows b = kleaf + 1 .. bmax
    std::vector<u64> spref(Q + 1, 0), rpref(Q + 1, 0), cpref(Q + 1, 0);
    std::vector<u32> ipref(Q + 1, 0);
    u64 bound = 0;   // count-row entries: at most segments x rows per query
    for (u32 q = 0; q < Q; q++) {
        const MQ& m = P.hq[q];
        const u64 bmax = pc_min(pc_min(m.B, m.a), m.R4);
        const bool work = m.c == 5 && bmax > T.kleaf;
        const u64 nseg = work ? m.z / T.span + 1 : 0;
        const u64 nrows = work ? bmax - T.k0 + 1 : 0;
        spref[q + 1] = spref[q] + nseg;
        rpref[q + 1] = rpref[q] + nrows;
        cpref[q + 1] = cpref[q] + (work ? bmax - T.kleaf : 0);
        bound += nseg * nrows;
    }
    const u64 S = spref[Q], R = rpref[Q];
    if (S == 0) return PC_OK;
    if (bound >> 32 || S >> 32) {
        pc_set_error(ctx, "batch: %llu count-row entries exceed 32-bit offsets", (unsigned long long)bound);
        return PC_EOVERFLOW;
    }
    for (u32 q = 0; q <= Q; q++) ipref[q] = (u32)spref[q];
    // mq_h: spref | rpref | cpref (Q+1 u64 each) | ipref (Q+1 u32) | segB (S u32) |
    // rowlen (R u32) | rlo (R u32) | off (R+1 u64) | queue + counters (128 B)
    auto al = [](size_t v) { return (v + 15) / 16 * 16; };
    const size_t o_r = al((Q + 1) * 8), o_c = o_r + al((Q + 1) * 8), o_i = o_c + al((Q + 1) * 8);
    const size_t o_sb = o_i + al((Q + 1) * 4), o_rl = o_sb + al(S * 4);
    const size_t o_ro = o_rl + al(R * 4), o_off = o_ro + al(R * 4), o_q = o_off + al((R + 1) * 8), total = o_q + 128;
    PC_TRY(buf_reserve(ctx, ctx->mq_h, total));
    PC_TRY(buf_reserve(ctx, ctx->mq_hq, Q * sizeof(HardArgs)));
    PC_TRY(buf_reserve(ctx, ctx->counts, bound * sizeof(u32)));
    PC_TRY(buf_reserve(ctx, ctx->tallies, bound * sizeof(i32)));
    unsigned char* base = ctx->mq_h.as<unsigned char>();
    u64* d_spref = (u64*)base;
    u64* d_rpref = (u64*)(base + o_r);
    u64* d_cpref = (u64*)(base + o_c);
    u32* d_ipref = (u32*)(base + o_i);
    u32* d_segB = (u32*)(base + o_sb);
    u32* d_rowlen = (u32*)(base + o_rl);
    u32* d_rlo = (u32*)(base + o_ro);
    u64* d_off = (u64*)(base + o_off);
    u32* d_queue = (u32*)(base + o_q);
    HardArgs* d_qa = ctx->mq_hq.as<HardArgs>();
    std::vector<HardArgs> qa(Q, T);
    for (u32 q = 0; q < Q; q++) {
        const MQ& m = P.hq[q];
        HardArgs& A = qa[q];
        A.x = m.x;
        A.y = m.y;
        A.z = m.z;
        A.c = m.c;
        A.a = m.a;
        A.trunc = false;
        const u64 bmax = pc_min(pc_min(m.B, m.a), m.R4);
        A.bmax = (u32)pc_max(bmax, T.k0);
        A.nseg = spref[q + 1] - spref[q];
        A.s0 = 0;
        A.s1 = A.nseg;
        A.segB = d_segB + spref[q];
        A.off = d_off + rpref[q];
        A.rlo = d_rlo + rpref[q];
        A.start = nullptr;
        A.counts = ctx->counts.as<u32>();
        A.tallies = ctx->tallies.as<i32>();
        A.queue = d_queue;
        A.stat = (unsigned long long*)(d_queue + 2);
    }
    cudaStream_t st = ctx->stream;
    if (mq_host_upload(ctx)) {
        PC_CUDA(ctx, cudaMemcpyAsync(d_qa, qa.data(), Q * sizeof(HardArgs), cudaMemcpyHostToDevice, st));
        PC_CUDA(ctx, cudaMemcpyAsync(d_spref, spref.data(), (Q + 1) * 8, cudaMemcpyHostToDevice, st));
        PC_CUDA(ctx, cudaMemcpyAsync(d_rpref, rpref.data(), (Q + 1) * 8, cudaMemcpyHostToDevice, st));
        PC_CUDA(ctx, cudaMemcpyAsync(d_cpref, cpref.data(), (Q + 1) * 8, cudaMemcpyHostToDevice, st));
        PC_CUDA(ctx, cudaMemcpyAsync(d_ipref, ipref.data(), (Q + 1) * 4, cudaMemcpyHostToDevice, st));
    }
    // the sieve's instantiation (its shared-memory attribute set outside any capture)
    T.queue = d_queue;
    T.stat = (unsigned long long*)(d_queue + 2);
    const size_t smem = hard_smem(T);
    if (ctx->mq_mode != MQ_CAPTURE) {
        void (*kern)(HardArgs, MultiArgs) = nullptr;
        int per_sm = 0;
        ctx->ctas_call = ctx->batch_ctas;   // the batch's tuned residency (0: as many as fit)
        const int rc = choose_hard_kernel<true>(ctx, T, smem, &kern, &per_sm);
        ctx->ctas_call = 0;
        PC_TRY(rc);
        ctx->mq_hard_kern = (void*)kern;
        ctx->mq_hard_per_sm = per_sm;
    }
    if (!mq_device_work(ctx)) return scan_exclusive_u32_to_u64(ctx, d_rowlen, d_off, R);   // its scratch only
    PC_CUDA(ctx, cudaMemsetAsync(d_queue, 0, 128, st));
    mq_seg_b_kernel<<<(unsigned)((S + 255) / 256), 256, 0, st>>>(d_qa, d_spref, Q, d_segB);
    PC_LAUNCHED(ctx);
    mq_row_len_kernel<<<(unsigned)((R + 255) / 256), 256, 0, st>>>(d_qa, d_rpref, Q, d_rowlen, d_rlo);
    PC_LAUNCHED(ctx);
    PC_TRY(scan_exclusive_u32_to_u64(ctx, d_rowlen, d_off, R));
    // the sieve: items are the segments of every query, handed out in order
    void (*kern)(HardArgs, MultiArgs) = (void (*)(HardArgs, MultiArgs))ctx->mq_hard_kern;
    const int per_sm = ctx->mq_hard_per_sm;
    const u64 ctas = pc_min((u64)ctx->sm_count * per_sm, S);
    MultiArgs M{d_qa, d_ipref, Q, (unsigned long long)S, P.parts + 3, 5u};
    kern<<<(unsigned)ctas, 32 * T.nw, smem, st>>>(T, M);
    PC_LAUNCHED(ctx);
    if (cpref[Q]) {
        mq_combine_kernel<<<ctx->sm_count * 8, 256, 0, st>>>(d_qa, d_cpref, Q, P.parts);
        PC_LAUNCHED(ctx);
    }
    ctx->stats.kernel_launches += 4;
    return PC_OK;
}
