// hr_runs.cu - the per-wave checker of single traces (sm_103a): variants 0 to 3,
// and every-epoch regions whose waves suit it (hr_single_route()).
//
// Like hr_check_kernel (hr_kernels.cu) it applies the trace wave by wave to the
// shadow in HBM, after the same pre-pass, and orders the waves with a completion
// count per stage.  It differs in what keeps a long wave busy:
//
//   - Independent warps.  A work item is one step of a warp, 32 x RPL consecutive
//     records of one wave (or HR_RUN_CLEAR_WORDS shadow words to clear).  A warp
//     claims items in ticket order (the CTA's first claim is one atomic for all its
//     warps; later ones are per warp, a run of up to MAX_CLAIM items at a time when
//     the check has many) and loads their records straight into registers, the next
//     step's while the current one is applied.
//   - One publication per stage and warp.  An item of wave w may only touch the
//     shadow once every item of the previous stage is done; a warp adds its finished
//     items to its stage's count when it leaves the stage, not tile by tile: the
//     release that orders its shadow updates before the count waits for all of them.
//   - Absorbed accesses end early.  Whether an access leaves its word's value as it
//     is follows from the FSM table's index alone (absorbs()), so most accesses need
//     one table look-up after their load and no fold.  The others go into a queue
//     of the warp in shared memory and are folded and CASed a full warp at a time:
//     the long part of the code runs on full warps instead of on the one lane in ten
//     that needs it.  (An access that is absorbed stays absorbed under any other
//     access of its wave, so the order does not matter.)
//   - Words every thread touches.  A word whose state absorbs an op from any thread
//     is noted in a table of the CTA, and later accesses skip their load: on a
//     power-law graph the hub words otherwise keep one L2 slice at 77 % of its tag
//     rate while the average slice is at 11 %.
//
// Measured on the power-law push (2^22 vertices, 537M records, 4 waves): 9.95 ms
// with hr_check_kernel's best shape, 4.53 ms here (variant 3; 118 G accesses/s at
// 1.9 TB/s of records: limited by the latency of the loads and CASes).  Short waves are bound by the hand-over from stage to stage, which
// hr_check_kernel's tiles, claimed and copied ahead by a producer warp, do better:
// batches of many traces (64 uneven traces: 2.4 ms there, 2.7 ms here) and variants
// 4 and 5 stay with it (tree reduction, 1.03M records in 8 waves: 87 us there,
// 94 to 128 us here).
#include <cuda_runtime.h>

#include "hr_check.cuh"
#include "hr_launch.cuh"
#include "hr_per_device.h"

namespace {

constexpr int CONS = 8;                        // warps per CTA
constexpr int CHECK_THREADS = CONS * 32;
constexpr unsigned KNOWN = 64;                 // slots of the CTA's table of finished stages
constexpr unsigned SEEN = 2048;                // entries of the CTA's table of absorbed accesses
constexpr unsigned FLIGHT = 1024;              // entries of the CTA's table of accesses being CASed
constexpr unsigned MAX_CLAIM = 16;             // items a warp claims at a time, at most

// WarpItem::last of a stage whose wait ran out.  (Taking the items off the warp's count
// of finished ones instead kept their number in a register: variant 3 spilled, and the
// power-law push below took 4.86 instead of 4.55 ms.)
constexpr unsigned LEFT = 2;

// What a warp keeps of its current stage and region, in shared memory: it is
// the same for all lanes and read once an item, so it costs no registers.
struct alignas(16) WarpItem {
    unsigned s, begin, end, type;         // stage, its items [begin, end), its type
    unsigned dep, dep_need, last, skip;   // previous stage of the job and its items; 1: the job's last; region failed
    const hr_record* first;               // the wave's records
    unsigned long long n;
    unsigned long long key;               // its key (rebased)
    unsigned kb, filtering;               // kernel base; the region's filter selects only part of the accesses
    unsigned stamp, lookup;               // job and kernel, for the table of absorbed accesses; whether it is used
    unsigned long long* shadow;
    unsigned last_word, region;           // the region's n_words - 1 and number
    hr_geom geom;
    hr_filter filter;
};

__device__ __forceinline__ unsigned ld_acquire_cta(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];"
                 : "=r"(v)
                 : "r"((uint32_t)__cvta_generic_to_shared(p))
                 : "memory");
    return v;
}

__device__ __forceinline__ void st_release_cta(unsigned* p, unsigned v)
{
    asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v)
                 : "memory");
}

// one record, read once (evict-first)
__device__ __forceinline__ uint4 ld_record(const hr_record* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }

// CTAs per SM (the launch bounds below): 2 for the 4-record shapes, 3 for the
// 2-record ones.  More warps hide more of a long wave's latency but make more
// warps that wait and poll at each stage's end.  Power-law push / 1.57M-record
// pieces of a global-memory trace (three), with 2, 3, 4 CTAs per SM: variant 1
// 5.49, 5.72, 7.77 ms / 374, 495, 595 us; variant 3 5.92, 4.89, 4.73 ms / 359,
// 446, 521 us.  Every-epoch regions (16.8M accesses): 1.43 ms with
// hr_check_kernel; here 1.17 ms with 2 records a lane, 1.07 ms with 4 (one fence
// serves a lane's records), 1.62 ms with 4 at 3 CTAs per SM (spills).

// One lane's bounded wait until a stage's completion count reaches `need`.
// s_known[dep % KNOWN] holds 1 + the last stage a warp of the CTA saw complete
// in that slot.  (No warp polls on behalf of the others: a lock for that starved
// warps whose stage shared its slot, for as long as the wait's bound.)
__device__ __forceinline__ bool stage_wait(const unsigned* done, unsigned need, unsigned dep, unsigned* s_known,
                                           unsigned* abort_flag, unsigned* err, unsigned long long wait_ns)
{
    unsigned* known = &s_known[dep % KNOWN];
    const unsigned long long t0 = globaltimer();
    unsigned ns = 64;
    for (unsigned n = 0;; ++n) {
        if (ld_acquire_cta(known) == dep + 1u) return true;
        if (ld_acquire_u32(done) >= need) {
            st_release_cta(known, dep + 1u);
            return true;
        }
        if ((n & 7u) == 7u) {
            if (*(volatile unsigned*)abort_flag) return false;
            if (globaltimer() - t0 > wait_ns) {
                atomicExch(abort_flag, 1u);
                hr_set_error(err, HR_ERR_TIMEOUT);
                return false;
            }
        }
        __nanosleep(ns);
        if (ns < HR_WAIT_SLEEP_MAX_NS) ns <<= 1;
    }
}

// The CTA's table of absorbed accesses: an entry says that word's state, in
// this job's current kernel, absorbs this op from any thread (every block reads,
// every block does atomics, or RACE; such a state only ever moves to RACE, which
// absorbs everything, until the kernel ends).  A later access of that kind skips
// its shadow load: without that, the words all threads touch keep one L2 slice
// busy while the others idle.  64-bit entries, written and read whole.
//
// Until such a state is seen, a stage's first accesses of a hub word all CAS it: a
// quarter of a 1.3M-record stage is in flight at once, and CASes of one word pass
// one after the other.  A table of the accesses (word, op) the CTA has a CAS out
// for lets one of them go; the others load the word again afterwards and mostly
// find themselves absorbed.  Power-law pushes, variants 0 and 3, without and with it:
// 40,000 vertices (2.56M records, 2 waves) 194 and 290 us, 157 and 160 us; 2^22
// vertices 5.49 and 4.83 ms (variants 1 and 3), 5.47 and 4.53 ms.
__device__ __forceinline__ unsigned flight_key(unsigned word, unsigned op) { return ((word << 2) | op) + 1u; }
__device__ __forceinline__ unsigned flight_slot(unsigned word) { return word % FLIGHT; }
__device__ __forceinline__ unsigned seen_slot(unsigned word) { return word % SEEN; }
__device__ __forceinline__ unsigned long long seen_key(unsigned word, unsigned stamp)
{
    return ((unsigned long long)stamp << 32) | word;
}
// For each index of the FSM table: 0 if the transition changes the shadow value,
// ABSORBED if it leaves it as it is, ABSORBED | ANY if it does so for every thread.
// The index decides that alone: a value keeps only the fields its level needs, and
// equal fields are what the thread relation and the sync status say.
constexpr unsigned ABSORBED = 1, ANY = 2;
__device__ __forceinline__ unsigned absorbs(const unsigned char* table, unsigned idx)
{
    const unsigned e = table[idx], trel = (idx >> 2) & 3u, srel = idx & 3u;
    if ((e & 31u) != idx >> 6) return 0u;
    switch (e >> 5) {
    case HR_LVL_THREAD: return trel == HR_TREL_SAME && srel == HR_SREL_UNSYNC ? ABSORBED : 0u;
    case HR_LVL_WARP: return trel <= HR_TREL_WARP && srel == HR_SREL_UNSYNC ? ABSORBED : 0u;
    case HR_LVL_BLOCK: return trel <= HR_TREL_BLOCK && srel != HR_SREL_BLOCK ? ABSORBED : 0u;
    case HR_LVL_GRID:
    case HR_LVL_RACE: return ABSORBED | ANY;
    }
    return 0u;
}

// Result of folding accesses into a shadow value: the new value, 1 + the
// prior state when the fold entered RACE (else 0), and the lane whose access
// did it.  Returned by value so the callers' state stays in registers.
struct Fold {
    unsigned long long n;
    unsigned raced, who;
};

// Fold the accesses of one lane group (lanes in `grp`, in lane order) into o.
__device__ __forceinline__ Fold fold_group(unsigned long long o, unsigned grp, const unsigned* tids,
                                        const unsigned char* ops, unsigned bc, unsigned wc,
                                        unsigned ktag, const hr_geom& g, const unsigned char* table)
{
    Fold f{o, 0u, threadIdx.x & 31};
    unsigned last_tid = ~0u, last_op = ~0u;
    while (grp) {
        const unsigned l = __ffs(grp) - 1;
        grp &= grp - 1;
        // the summary depends on the set of accesses: a repeat of the access
        // just applied (same thread, same op, same wave) changes nothing
        if (tids[l] == last_tid && ops[l] == last_op) continue;
        last_tid = tids[l];
        last_op = ops[l];
        unsigned r = 0;
        f.n = hr_fsm_step(f.n, last_tid, last_op, bc, wc, ktag, g, table, &r);
        if (r && !f.raced) {
            f.raced = r;
            f.who = l;
        }
    }
    return f;
}


// compareTids of two threads by the xor of their ids (power-of-two geometry)
__device__ __forceinline__ unsigned rel_pow2(unsigned x, unsigned bd_shift, unsigned ws_shift)
{
    return x == 0u ? HR_TREL_SAME : (x >> bd_shift) ? HR_TREL_GRID : (x >> ws_shift) ? HR_TREL_BLOCK : HR_TREL_WARP;
}

// A warp's accesses that their words' values do not absorb, until a step's
// worth of them is there (shared memory).
template <unsigned CAP>
struct alignas(16) Queue {
    unsigned long long o[CAP];  // the shadow value loaded
    unsigned word[CAP];
    unsigned tid[CAP];
    unsigned char op[CAP];
};

template <bool AGG, int RPL, bool EVERY>
__global__ void __launch_bounds__(CHECK_THREADS, RPL >= 4 ? 2 : 3)
    hr_run_kernel(hr_region_dev* __restrict__ regions, hr_work w, const unsigned char* __restrict__ gtable)
{
    constexpr unsigned ITEM = 32 * RPL;
    constexpr unsigned QCAP = ITEM + 32;
    __shared__ __align__(16) unsigned char s_table[2048];
    __shared__ WarpItem s_item[CONS];
    __shared__ unsigned char s_abs[EVERY ? 16 : 2048];
    __shared__ Queue<EVERY ? 1 : QCAP> s_queue[EVERY ? 1 : CONS];
    __shared__ unsigned s_known[KNOWN];
    __shared__ unsigned long long s_seen[EVERY ? 1 : SEEN];
    __shared__ unsigned s_flight[EVERY ? 1 : FLIGHT];  // flight_key() of an access, or 0
    __shared__ unsigned s_first;

    const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the tables, while the kernel before this one ends
    for (unsigned i = threadIdx.x; i < 128; i += CHECK_THREADS)
        reinterpret_cast<uint4*>(s_table)[i] = reinterpret_cast<const uint4*>(gtable)[i];
    for (unsigned i = threadIdx.x; i < KNOWN; i += CHECK_THREADS) s_known[i] = 0u;
    if (!EVERY) {
        for (unsigned i = threadIdx.x; i < SEEN; i += CHECK_THREADS) s_seen[i] = ~0ull;
        for (unsigned i = threadIdx.x; i < 2048; i += CHECK_THREADS) s_abs[i] = (unsigned char)absorbs(gtable, i);
        for (unsigned i = threadIdx.x; i < FLIGHT; i += CHECK_THREADS) s_flight[i] = 0u;
    }
    hr_grid_wait();
    const unsigned total = hr_bin_taken(w.ctl) ? 0u : w.ctl->run_items;  // binned: the work is done already
    if (total == 0) return;
    // items per claim: enough to keep the ticket counter out of the way, few
    // enough that a stage's items spread over all warps
    const unsigned claim =
        (unsigned)max(1ull, min((unsigned long long)MAX_CLAIM,
                                total / ((unsigned long long)w.ctl->n_stages * gridDim.x * (CONS * 2u))));
    if (threadIdx.x == 0) s_first = atomicAdd(&w.ctl->ticket, CONS * claim);
    WarpItem& it = s_item[wid];
    if (lane == 0) {
        it.region = ~0u;  // (nothing is counted before the first region is set)
        it.s = it.begin = it.end = it.skip = 0u;
        it.dep = HR_NO_DEP;
    }
    __syncthreads();

    const hr_geom& g = it.geom;
    const hr_filter& filt = it.filter;
    auto& q = s_queue[EVERY ? 0 : wid];
    unsigned known = HR_NO_DEP;  // last dependency this warp has seen complete
    unsigned lc_acc = 0, lc_cas = 0, lc_retry = 0, lc_merged = 0;  // this lane's counts since the last flush
    auto flush = [&]() {
        unsigned long long v[4] = {lc_acc, lc_cas, lc_retry, lc_merged};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            for (int o2 = 16; o2 > 0; o2 >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o2);
            if (lane == 0 && v[i]) atomicAdd(&regions[it.region].counters[i], v[i]);
        }
        lc_acc = lc_cas = lc_retry = lc_merged = 0;
    };
    unsigned finished = 0;   // items of this stage finished but not published
    auto publish = [&]() {
        __syncwarp();
        if (lane == 0 && finished) {
            hr_stage* st = &w.stages[it.s];
            if (it.last == LEFT) {  // its wait ran out: what was not applied is not done, and no later stage may start
            } else if (it.last) {   // the job's last stage: the item that completes it stamps the job's end
                const unsigned prev = atom_add_release(&st->done, finished);
                if (prev + finished == it.end - it.begin) w.jobs[st->job].done_ns = globaltimer();
            } else {
                red_release_add(&st->done, finished);
            }
        }
        finished = 0;
        __syncwarp();
    };

    unsigned t = s_first + wid * claim, t_end = t + claim, ahead = HR_NO_DEP;
    for (unsigned n_claims = 1;; ++n_claims) {
        if (t == t_end) {  // the next claim
            unsigned c = ahead;
            if (lane == 0 && c == HR_NO_DEP) c = atomicAdd(&w.ctl->ticket, claim);
            t = __shfl_sync(0xffffffffu, c, 0);
            t_end = t + claim;
            ahead = HR_NO_DEP;
            if ((n_claims & 7u) == 0u) {
                unsigned stop = 0;
                if (lane == 0) {
                    stop = *(volatile unsigned*)&w.ctl->abort;
                    if (it.end && *(volatile unsigned*)&regions[it.region].error) it.skip = 1u;
                }
                __syncwarp();
                if (__shfl_sync(0xffffffffu, stop, 0)) break;
            }
        }
        if (t >= total) break;
        if (t >= it.end) {  // move to the stage holding item t
            publish();
            const unsigned n_st = w.ctl->n_stages;
            unsigned s = it.s;
            for (;;) {  // 32 stages at a time: the last one that starts at or before t
                const unsigned q = s + 1 + lane;
                const bool before = q <= n_st && w.stages[q].item_begin <= t;
                const unsigned m = __ballot_sync(0xffffffffu, before);
                s += __popc(m);
                if (m != 0xffffffffu) break;
            }
            const unsigned r = w.jobs[w.stages[s].job].region;
            if (r != it.region) {
                flush();
                __syncwarp();
                if (lane == 0) {
                    const hr_region_dev& rg = regions[r];
                    it.geom = rg.geom;
                    it.filter = rg.filter;
                    it.filtering = hr_filter_active(rg.filter);
                    it.shadow = rg.shadow;
                    it.last_word = (unsigned)(rg.n_words - 1ull);
                    it.region = r;
                }
            }
            if (lane == 0) {
                const hr_stage& st = w.stages[s];
                const hr_jobd& jb = w.jobs[st.job];
                it.s = s;
                it.begin = st.item_begin;
                it.end = w.stages[s + 1].item_begin;
                it.type = st.type;
                it.dep = st.dep;
                it.dep_need = st.dep_need;
                it.last = st.last;
                it.kb = (unsigned)(jb.kb >> 32);
                it.first = jb.trace + w.wave_start[st.wave];
                it.n = w.wave_end[st.wave] - w.wave_start[st.wave];
                it.key = w.wave_key[st.wave];  // already rebased by the pre-pass
                it.stamp = (st.job << 18) | ((unsigned)(w.wave_key[st.wave] >> 32) << 2);
                // words met again and again are worth looking up in the CTA's table
                it.lookup = !EVERY && jb.n / 8 >= regions[r].n_words;
                it.skip = *(volatile unsigned*)&regions[r].error != 0;
            }
            __syncwarp();
        }
        // this claim's items of this stage: one run of consecutive records
        const unsigned e = min(t_end, it.end);
        const unsigned item = t - it.begin, n_items = e - t;
        t = e;
        finished += n_items;
        // the next claim, while this stage has plenty of items left
        if (t == t_end && it.end - t > 2u * CONS * gridDim.x * claim)
            ahead = lane == 0 ? atomicAdd(&w.ctl->ticket, claim) : 0u;
        if (it.skip) continue;
        const unsigned dep = it.dep;
        const bool ready = dep == HR_NO_DEP || dep == known;
        auto wait_dep = [&]() {
            unsigned ok = 1;
            if (lane == 0)
                ok = stage_wait(&w.stages[dep].done, it.dep_need, dep, s_known, &w.ctl->abort,
                                &regions[it.region].error, w.wait_ns);
            if (!ok) it.last = LEFT;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            __syncwarp();
            known = dep;
            return ok != 0;
        };
        const bool sb4 = g.shadow_bytes == 4;
        unsigned long long* const shadow = it.shadow;
        const unsigned last_word = it.last_word;
        if (it.type == HR_STAGE_CLEAR) {
            if (!ready && !wait_dep()) break;
            const unsigned long long sb = g.shadow_bytes;
            const unsigned long long span = w.clear_words * sb;
            const unsigned long long bb = item * span;
            const unsigned long long be = min(((unsigned long long)last_word + 1ull) * sb, bb + n_items * span);
            clear_bytes(shadow, bb, be, lane);
            continue;
        }
        const unsigned kern = (unsigned)(it.key >> 32), bcwc = (unsigned)it.key;
        const unsigned bc = bcwc >> 16, wc = bcwc & 0xFFFFu, ktag = kern & 7u;
        const unsigned kern16 = kern - it.kb;  // the records' own kernel ordinal
        const hr_record* rec = it.first + (unsigned long long)item * ITEM + lane;
        unsigned n_rec = (unsigned)min((unsigned long long)n_items * ITEM, it.n - (unsigned long long)item * ITEM);
        // the wave's clocks fit the region's shadow packing (else every access overflows it)
        const bool clk_fit = hr_fits(0u, bc, wc, g);
        const bool plain = !it.filtering && !sb4 && clk_fit;  // no filter, every tid and clock fits
        const bool lookup = it.lookup != 0;
        const unsigned bds = g.bd_shift, wss = g.ws_shift;
        const unsigned wave_hi = (ktag << (HR_SH_KTAG_SHIFT - 32)) | (bc << (HR_SH_BC_SHIFT - 32)) | (wc & 0xFFu);
        auto step = [&](unsigned long long o, unsigned a_tid, unsigned a_op, unsigned* r) -> unsigned long long {
            return bds != ~0u ? hr_fsm_step_pow2(o, a_tid, a_op, bc, wc, ktag, bds, wss, s_table, r)
                              : hr_fsm_step(o, a_tid, a_op, bc, wc, ktag, g, s_table, r);
        };

        // Apply the queue's last n accesses (n <= ITEM), RPL to a lane: fold each into
        // the value it was queued with and send out every CAS before reading any of
        // their results.
        unsigned queued = 0;
        auto apply = [&](unsigned n) {
            __syncwarp();
            queued -= n;
            unsigned long long seen[RPL];
            unsigned casm = 0;   // bit k: a CAS went out for slot k
            unsigned defer = 0;  // bit k: the CTA has a CAS out for this access already
            unsigned own = 0;    // bit k: slot k's CAS is entered in the table of those
            unsigned race = 0;   // a byte per slot: 0, or 1 + the prior state of a word this fold moves into RACE
            unsigned whose = 0;  // a byte per slot: the lane whose access does
            unsigned grp[RPL];   // AGG: the lanes whose accesses this slot folds, in lane order
#pragma unroll
            for (int k = 0; k < RPL; ++k) {
                const unsigned i = queued + k * 32 + lane;
                bool a = k * 32 + lane < n;
                grp[k] = 1u << lane;
                if (AGG && (unsigned)(k * 32) < n) {
                    // lanes of this slot applying the same word
                    const unsigned am = __ballot_sync(0xffffffffu, a);
                    const unsigned mw = __match_any_sync(0xffffffffu, a ? q.word[i] : 0u) & am;
                    if (__any_sync(0xffffffffu, a && mw != (1u << lane))) {
                        // an exact repeat (same word, thread, op, wave) of a lower lane's
                        // access adds nothing to the summary: drop it
                        const unsigned same =
                            __match_any_sync(0xffffffffu, a ? ((unsigned long long)q.tid[i] << 32) | q.op[i] : 0ull) & mw;
                        if (a && (unsigned)(__ffs(same) - 1) != lane) {
                            a = false;
                            lc_merged++;
                        }
                        // distinct accesses to one word: the lowest lane folds them
                        const unsigned m = mw & __ballot_sync(0xffffffffu, a);
                        if (a) {
                            grp[k] = m;
                            if ((unsigned)(__ffs(m) - 1) != lane) {
                                a = false;  // folded by the group leader
                                lc_merged++;
                            }
                        }
                    }
                }
                if (!a) continue;
                unsigned r = 0, who = lane;
                const unsigned long long o = q.o[i];
                unsigned long long nv;
                if (AGG && grp[k] != (1u << lane)) {
                    const Fold f = fold_group(o, grp[k], q.tid + queued + k * 32, q.op + queued + k * 32, bc, wc, ktag, g, s_table);
                    nv = f.n;
                    r = f.raced;
                    who = f.who;
                } else {
                    nv = step(o, q.tid[i], q.op[i], &r);
                }
                if (nv != o && lookup) {
                    const unsigned key = flight_key(q.word[i], q.op[i]);
                    const unsigned out = atomicCAS(&s_flight[flight_slot(q.word[i])], 0u, key);
                    if (out == key) {
                        defer |= 1u << k;
                        continue;
                    }
                    own |= (unsigned)(out == 0u) << k;
                }
                if (nv != o) {
                    seen[k] = hr_shadow_cas(shadow, q.word[i], o, nv, g);
                    casm |= 1u << k;
                    race |= r << (8 * k);
                    if (AGG) whose |= who << (8 * k);
                }
            }
            // A CAS that returned the value it expected stuck.  One that lost folds
            // again into what it saw (mostly an equal transition by another lane,
            // which already absorbs this access), until a CAS sticks or the retry cap
            // is reached.
            unsigned lost = 0, todo = 0;
#pragma unroll
            for (int k = 0; k < RPL; ++k) {
                if (!((casm >> k) & 1u)) continue;
                lc_cas++;
                const unsigned i = queued + k * 32 + lane;
                if (seen[k] != q.o[i]) {
                    lc_retry++;
                    lost |= 1u << k;
                    todo |= 1u << k;
                    q.o[i] = seen[k];
                } else if ((race >> (8 * k)) & 0xFFu) {
                    todo |= 1u << k;
                }
                if ((own >> k) & 1u) *(volatile unsigned*)&s_flight[flight_slot(q.word[i])] = 0u;
            }
            if (defer) {  // look again, every word's load before the first result
#pragma unroll
                for (int k = 0; k < RPL; ++k)
                    if ((defer >> k) & 1u) seen[k] = hr_shadow_load(shadow, q.word[queued + k * 32 + lane], g);
#pragma unroll
                for (int k = 0; k < RPL; ++k)
                    if ((defer >> k) & 1u) q.o[queued + k * 32 + lane] = seen[k];
                lost |= defer;
                todo |= defer;
            }
            while (todo) {
                const unsigned k = __ffs(todo) - 1;
                todo &= todo - 1;
                const unsigned i = queued + k * 32 + lane, wd = q.word[i], a_tid = q.tid[i], a_op = q.op[i];
                unsigned m = 1u << lane;
                if (AGG) {
#pragma unroll
                    for (int j = 0; j < RPL; ++j) m = k == (unsigned)j ? grp[j] : m;
                }
                unsigned raced = (race >> (8 * k)) & 0xFFu, who = AGG ? (whose >> (8 * k)) & 0xFFu : lane;
                if ((lost >> k) & 1u) {
                    unsigned long long sv = q.o[i];
                    bool done = false;
                    raced = 0;
                    for (unsigned tries = 0;; ++tries) {
                        unsigned r = 0;
                        unsigned long long nv;
                        if (AGG && m != (1u << lane)) {
                            const Fold f = fold_group(sv, m, q.tid + queued + k * 32, q.op + queued + k * 32, bc, wc, ktag, g, s_table);
                            nv = f.n;
                            r = f.raced;
                            who = f.who;
                        } else {
                            nv = step(sv, a_tid, a_op, &r);
                            who = lane;
                        }
                        if (nv == sv) {  // no change: this access moved nothing into RACE
                            done = true;
                            break;
                        }
                        // (a deferred access has not tried yet: one CAS beside the cap's)
                        if (tries > w.cas_cap || (tries == w.cas_cap && !((defer >> k) & 1u))) break;
                        lc_cas++;
                        const unsigned long long x = hr_shadow_cas(shadow, wd, sv, nv, g);
                        if (x == sv) {
                            raced = r;
                            done = true;
                            break;
                        }
                        sv = x;
                    }
                    if (!done) hr_set_error(&regions[it.region].error, HR_ERR_CONTENTION);
                }
                if (raced) {
                    const unsigned j = queued + k * 32 + who;
                    hr_region_dev* region = regions + it.region;
                    hr_append_race(region->ring, region->ring_cap, &region->n_races, &region->flags,
                                   wd + (it.filtering ? (unsigned)filt.word_lo : 0u), q.tid[j], kern, bc, region->region,
                                   q.op[j], raced - 1u);
                }
            }
            __syncwarp();  // the queue's slots may be written again
        };

        uint4 v[RPL];
        auto load = [&]() {
#pragma unroll
            for (int k = 0; k < RPL; ++k)
                v[k] = k * 32 + lane < n_rec ? ld_record(rec + k * 32) : make_uint4(0u, 0u, 0u, 0u);
        };
        load();  // (while a wait for the previous stage runs)
        if (!ready && !wait_dep()) break;
        for (;;) {
            // Decode the records
            unsigned word[RPL], tid[RPL];
            unsigned ops = 0;   // 2 bits per slot
            unsigned err = 0;
            unsigned actm = 0;  // bit k: slot k holds an access to look at
#pragma unroll
            for (int k = 0; k < RPL; ++k) {
                const bool in = k * 32 + lane < n_rec;
                const unsigned op = (v[k].w >> 16) & 0xFFu;
                // record key (kernel + kernel base, bc, wc) against the wave's
                const bool same_wave = v[k].z == bcwc && (v[k].w & 0xFFFFu) == kern16;
                unsigned widx = v[k].x, tidf = v[k].y;
                bool a = in && op <= HR_A && same_wave;
                if (!plain) {
                    // selective monitoring: unmonitored accesses are skipped, a word window
                    // maps words to shadow indices, a symmetric group folds the access onto
                    // its representative (tidf, widx)
                    bool mon = true;
                    if (it.filtering && a) {
                        unsigned long long ix = v[k].x;
                        mon = hr_monitored(filt, g, &tidf, v[k].x, &ix);
                        widx = (unsigned)ix;
                    }
                    if (a && mon && widx > last_word) err = HR_ERR_RANGE;
                    a = a && mon && widx <= last_word;
                    if (a && (!clk_fit || (sb4 && (tidf >> g.tid_bits)))) {
                        err = HR_ERR_CLOCK_OVERFLOW;  // tid, bc or wc wider than the shadow packing
                        a = false;
                    }
                } else if (a && widx > last_word) {
                    err = HR_ERR_RANGE;
                    a = false;
                }
                if (in && !(same_wave && op <= HR_A)) {  // a barrier record, or an error
                    if (!same_wave) err = HR_ERR_ORDER;
                    else if (op > HR_SYNCWARP || (op == HR_SYNCWARP && ((v[k].w >> 24) & HR_RECFLAG_PARTIAL_MASK)))
                        err = HR_ERR_UNSUPPORTED;
                }
                lc_acc += a;
                // an access that its word's state absorbs from any thread (a table entry
                // made below): nothing to do
                if (lookup && a && s_seen[seen_slot(widx)] == seen_key(widx, it.stamp | op)) {
                    a = false;
                    lc_merged++;
                }
                word[k] = widx;
                tid[k] = tidf;
                ops |= (op & 3u) << (2 * k);
                actm |= (unsigned)a << k;
            }
            if (err) hr_set_error(&regions[it.region].error, err);
            unsigned long long o[RPL];
            if constexpr (!EVERY) {
#pragma unroll
                for (int k = 0; k < RPL; ++k) {
                    o[k] = 0ull;
                    if ((actm >> k) & 1u)
                        o[k] = sb4 ? hr_expand32(hr_ld_relaxed32((unsigned*)shadow + word[k]), g)
                                   : hr_ld_relaxed(shadow + word[k]);
                }
            }
            // the next step's records travel while this one's accesses are looked at
            const bool more = n_rec > ITEM;
            if (more) {
                rec += ITEM;
                n_rec -= ITEM;
                load();
            }
            if constexpr (EVERY) {
                unsigned rw[RPL], ov[RPL];
#pragma unroll
                for (int k = 0; k < RPL; ++k) {
                    rw[k] = word[k] + (it.filtering ? (unsigned)filt.word_lo : 0u);
                    ov[k] = (ops >> (2 * k)) & 3u;
                }
                const unsigned st = every_epoch_slots<RPL>(shadow, (unsigned long long)last_word + 1ull, actm, word, rw,
                                                           tid, ov, bc, wc, kern, g, regions + it.region, w.cas_cap);
                if (st) hr_set_error(&regions[it.region].error, st);
            } else {
                // Queue the accesses that change their word's value
#pragma unroll
                for (int k = 0; k < RPL; ++k) {
                    const unsigned op = (ops >> (2 * k)) & 3u;
                    bool a = (actm >> k) & 1u;
                    const unsigned ohi = (unsigned)(o[k] >> 32), olo = (unsigned)o[k];
                    const unsigned d = ohi ^ wave_hi;  // kernel tag, bc and wc against the wave's
                    if (a && (d & (7u << (HR_SH_KTAG_SHIFT - 32))) == 0u) {
                        const unsigned trel = bds != ~0u ? rel_pow2(tid[k] ^ olo, bds, wss) : hr_thread_rel(tid[k], olo, g);
                        const unsigned srel = (d & (0xFFFFu << (HR_SH_BC_SHIFT - 32))) ? HR_SREL_BLOCK
                                              : (d & 0xFFu)                            ? HR_SREL_WARP
                                                                                       : HR_SREL_UNSYNC;
                        const unsigned ab = s_abs[((ohi >> (HR_SH_STATE_SHIFT - 32)) << 6) | (op << 4) | (trel << 2) | srel];
                        a = ab == 0u;
                        if (lookup && (ab & ANY)) s_seen[seen_slot(word[k])] = seen_key(word[k], it.stamp | op);
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, a);
                    if (a) {
                        const unsigned i = queued + __popc(m & ((1u << lane) - 1u));
                        q.o[i] = o[k];
                        q.word[i] = word[k];
                        q.tid[i] = tid[k];
                        q.op[i] = (unsigned char)op;
                    }
                    queued += __popc(m);
                }
                while (queued > QCAP - ITEM || (!more && queued)) apply(min(queued, ITEM));
            }
            if (!more) break;
        }
    }
    publish();
    flush();
}

template <bool AGG, int RPL, bool EVERY>
cudaError_t launch(hr_region_dev* d_regions, const hr_work& w, unsigned long long n, const unsigned char* d_table,
                   cudaStream_t stream)
{
    struct Fit {
        int sms, per_sm;
    };
    static hr_per_device<Fit> fits;
    int dev = 0;
    cudaGetDevice(&dev);
    const Fit fit = fits.get(dev, [dev] {
        Fit f{0, 0};
        cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f.per_sm, hr_run_kernel<AGG, RPL, EVERY>, CHECK_THREADS, 0);
        if (f.per_sm < 1) f.per_sm = 1;
        return f;
    });
    // no more warps than the records give items to (one CTA per SM at least, for
    // shadow clears): others would only start, take a ticket and leave
    const unsigned long long items = (n + w.tile - 1) / w.tile, ctas = (items + CONS - 1) / CONS;
    const unsigned long long full = (unsigned long long)fit.sms * fit.per_sm;
    const unsigned grid = (unsigned)(ctas > full ? full : ctas < (unsigned)fit.sms ? (unsigned)fit.sms : ctas);
    return hr_launch(hr_run_kernel<AGG, RPL, EVERY>, grid, CHECK_THREADS, 0, stream, d_regions, w, d_table);
}

}  // namespace

cudaError_t hr_launch_runs(hr_region_dev* d_regions, const hr_work& w, unsigned long long n,
                           const unsigned char* d_table, unsigned variant, cudaStream_t stream)
{
    switch (variant) {
    case 0: return launch<true, 4, false>(d_regions, w, n, d_table, stream);
    case 1: return launch<false, 4, false>(d_regions, w, n, d_table, stream);
    case 2: return launch<true, 2, false>(d_regions, w, n, d_table, stream);
    case 3: return launch<false, 2, false>(d_regions, w, n, d_table, stream);
    case HR_EVERY_EPOCH_VARIANT: return launch<false, HR_RUN_EVERY_RPL, true>(d_regions, w, n, d_table, stream);
    }
    return cudaErrorInvalidValue;
}
