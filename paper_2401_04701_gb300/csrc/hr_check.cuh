// hr_check.cuh - device code the per-wave checkers share (hr_kernels.cu, hr_runs.cu).
#pragma once

#include "hr_internal.h"

namespace {

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long globaltimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned atom_add_release(unsigned* p, unsigned v)
{
    unsigned old;
    asm volatile("atom.release.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bytes [bb, be) of a shadow to zero (one warp; bb a multiple of 16): 16-byte stores and a
// 4-byte tail.  hr_check_trace_noalloc takes a shadow at any multiple of 8: 8-byte stores
// then (its values are 8 bytes).
__device__ __forceinline__ void clear_bytes(void* shadow, unsigned long long bb, unsigned long long be, unsigned lane)
{
    unsigned char* const p = static_cast<unsigned char*>(shadow);
    if (reinterpret_cast<unsigned long long>(p) & 15ull) {
        for (unsigned long long i = bb + 8ull * lane; i < be; i += 256ull)
            *reinterpret_cast<unsigned long long*>(p + i) = 0ull;
        return;
    }
    for (unsigned long long i = bb + 16ull * lane; i < be; i += 512ull) {
        if (i + 16 <= be)
            *reinterpret_cast<ulonglong2*>(p + i) = make_ulonglong2(0ull, 0ull);
        else
            for (unsigned long long j = i; j < be; j += 4) *reinterpret_cast<unsigned*>(p + j) = 0u;
    }
}

// Every-epoch mode for a lane's RPL accesses at once (bit k of `act`: slot k
// holds one): the steps of hr_ep_apply, each over every slot before the next,
// so each step costs one round trip for all of them and one fence serves them
// all.  Per access: fold it into the summaries of the conflict kinds it holds
// (CAS loops), then a sequentially consistent fence, then read the summaries
// of the kinds it conflicts with; a conflicting holder is reported once per
// (word, kernel, epoch) through a CAS on the stamp word.  Of two concurrent
// conflicting accesses at least one therefore sees the other.  Returns 0 or
// HR_ERR_CONTENTION when a CAS loop reached `cap` tries.
template <int RPL>
__device__ __forceinline__ unsigned every_epoch_slots(unsigned long long* shadow, unsigned long long n_words,
                                                      unsigned act, const unsigned* idx, const unsigned* report_word,
                                                      const unsigned* tid, const unsigned* op, unsigned bc,
                                                      unsigned wc, unsigned kernel, const hr_geom& g,
                                                      hr_region_dev* region, unsigned cap)
{
    const unsigned ktag = kernel & 7u;
    unsigned err = 0;
    auto holds = [&](int k) { return op[k] == HR_R ? 1u : (op[k] == HR_A ? 2u : 3u); };
    auto against = [&](int k) { return op[k] == HR_R ? 2u : (op[k] == HR_A ? 1u : 3u); };
    // 1. the held kinds' summaries, all loaded at once, then every first CAS
    unsigned long long o[RPL][2], seen[RPL][2];
    unsigned casm = 0;  // bit 2k+b: a CAS went out on summary b of slot k
#pragma unroll
    for (int k = 0; k < RPL; ++k)
#pragma unroll
        for (int b = 0; b < 2; ++b)
            if (((act >> k) & 1u) && ((holds(k) >> b) & 1u)) o[k][b] = hr_ld_relaxed(shadow + b * n_words + idx[k]);
#pragma unroll
    for (int k = 0; k < RPL; ++k)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            if (!((act >> k) & 1u) || !((holds(k) >> b) & 1u)) continue;
            const unsigned long long n = hr_ep_update(o[k][b], tid[k], bc, wc, ktag, g);
            if (n == o[k][b]) continue;
            seen[k][b] = atomicCAS(shadow + b * n_words + idx[k], o[k][b], n);
            casm |= 1u << (2 * k + b);
        }
    // a CAS that lost: fold again into what it saw
#pragma unroll
    for (int k = 0; k < RPL; ++k)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            if (!((casm >> (2 * k + b)) & 1u) || seen[k][b] == o[k][b]) continue;
            unsigned long long* p = shadow + b * n_words + idx[k];
            unsigned long long cur = seen[k][b];
            bool ok = false;
            for (unsigned tries = 1; tries < cap; ++tries) {
                const unsigned long long n = hr_ep_update(cur, tid[k], bc, wc, ktag, g);
                if (n == cur) { ok = true; break; }
                const unsigned long long sv = atomicCAS(p, cur, n);
                if (sv == cur) { ok = true; break; }
                cur = sv;
            }
            if (!ok) {
                err = HR_ERR_CONTENTION;
                act &= ~(1u << k);  // this access is not applied: it reports nothing
            }
        }
    if (!act) return err;
    asm volatile("fence.sc.gpu;" ::: "memory");
    // 2. the conflicting kinds' summaries, all loaded at once
    unsigned long long sv[RPL][2];
#pragma unroll
    for (int k = 0; k < RPL; ++k)
#pragma unroll
        for (int b = 0; b < 2; ++b)
            if (((act >> k) & 1u) && ((against(k) >> b) & 1u)) sv[k][b] = hr_ld_relaxed(shadow + b * n_words + idx[k]);
    // 3. a conflicting holder: claim the (kernel, epoch) of the report
#pragma unroll
    for (int k = 0; k < RPL; ++k) {
        if (!((act >> k) & 1u)) continue;
        unsigned prior = 0;
#pragma unroll
        for (int b = 0; b < 2; ++b)
            if (!prior && ((against(k) >> b) & 1u) && hr_ep_pred(sv[k][b], tid[k], bc, wc, ktag, g))
                prior = hr_ep_level(sv[k][b], ktag);
        if (!prior) continue;
        unsigned long long* st = shadow + 2 * n_words + idx[k];
        const unsigned long long mine = ((((unsigned long long)kernel) << 16) | bc) + 1ull;
        unsigned long long cur = hr_ld_relaxed(st);
        bool claimed = false;
        for (unsigned tries = 0; cur < mine && tries < cap; ++tries) {
            const unsigned long long x = atomicCAS(st, cur, mine);
            if (x == cur) { claimed = true; break; }
            cur = x;
        }
        if (claimed)
            hr_append_race(region->ring, region->ring_cap, &region->n_races, &region->flags, report_word[k], tid[k],
                           kernel, bc, region->region, op[k], prior);
        else if (cur < mine)
            err = HR_ERR_CONTENTION;
    }
    return err;
}

}  // namespace
