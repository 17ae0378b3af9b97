// hr_internal.h - device-side data structures shared by the kernels and the API.
#pragma once

#include <cstdint>

#include "../../include/hirace.h"
#include "../../include/hirace_device.cuh"

// Geometry with exact reciprocals and, when both sizes are powers of two,
// shifts; plus the shadow packing (8 bytes, or 4 with a tid_bits-wide tid).
inline hr_geom hr_make_geom(uint32_t block_dim, uint32_t warp_size, uint32_t shadow_bytes = 8, uint32_t tid_bits = 0,
                            uint32_t report_mode = HR_REPORT_FIRST)
{
    auto magic = [](uint32_t d) { return d <= 1 ? 0ull : (~0ull) / d + 1ull; };
    auto log2_exact = [](uint32_t d) -> uint32_t {
        if (d == 0 || (d & (d - 1))) return ~0u;
        uint32_t s = 0;
        while ((1u << s) < d) ++s;
        return s;
    };
    hr_geom g{};
    g.block_dim = block_dim;
    g.warp_size = warp_size;
    g.bd_magic = magic(block_dim);
    g.ws_magic = magic(warp_size);
    const uint32_t bs = log2_exact(block_dim), ws = log2_exact(warp_size);
    g.bd_shift = (bs != ~0u && ws != ~0u) ? bs : ~0u;
    g.ws_shift = (bs != ~0u && ws != ~0u) ? ws : ~0u;
    g.report_mode = report_mode;
    g.shadow_bytes = report_mode == HR_REPORT_EVERY_EPOCH ? 24u : (shadow_bytes == 4 ? 4u : 8u);
    g.tid_bits = g.shadow_bytes == 4 ? (tid_bits ? tid_bits : 16u) : 0u;
    return g;
}

// Bytes per shadow word and tid width of a region descriptor (defaults applied):
// 8, 4 for the compact packing, 24 (three 8-byte arrays) in every-epoch mode.
inline uint32_t hr_desc_shadow_bytes(const hr_region_desc& d)
{
    return d.report_mode == HR_REPORT_EVERY_EPOCH ? 24u : (d.shadow_bytes == 4 ? 4u : 8u);
}
inline uint32_t hr_desc_tid_bits(const hr_region_desc& d)
{
    return d.shadow_bytes == 4 ? (d.tid_bits ? d.tid_bits : 16u) : 0u;
}
inline hr_geom hr_desc_geom(const hr_region_desc& d)
{
    return hr_make_geom(d.block_dim, d.warp_size, d.shadow_bytes == 4 ? 4u : 8u, hr_desc_tid_bits(d), d.report_mode);
}

// What hr_report and hr_counters tell of a region, kept in page-locked host memory
// that the device writes: at the end of every check and in every reset, so a
// report needs no copy once the region's work is done.  (A region with a device
// view is read from the device: instrumented kernels write its state themselves.)
struct hr_told {
    unsigned long long n_races;
    unsigned long long counters[4];
    unsigned int error, flags;
};

// Per-region state in device memory.
struct hr_region_dev {
    unsigned long long* shadow;   // n_words shadow values
    hr_race* ring;                // ring_cap race records
    unsigned long long n_words;
    unsigned long long ring_cap;
    // (an hr_told, which hr_report copies from a region with a device view)
    unsigned long long n_races;   // races found (may exceed ring_cap)
    unsigned long long counters[4];  // accesses, CAS attempts, CAS retries, accesses without a shadow access
    unsigned int error;           // sticky first error (hr_status)
    unsigned int flags;           // HR_FLAG_* bits
    unsigned long long group_waves;  // waves of the record group a host-memory check is in (hr_work::cont)
    unsigned long long last_key;  // wave key after the region's last processed record
    unsigned int used;            // 1: a record was processed since init/reset; 2: the shadow's
                                  // contents are unknown (cleared before the first wave)
    unsigned int region;
    hr_geom geom;
    hr_filter filter;             // monitored words, blocks, lanes (hr_set_filter)
    hr_told* told;                // the host's copy of the report
};

// the filter that monitors every access
__host__ __device__ inline hr_filter hr_filter_all()
{
    hr_filter f{};
    f.lane_mask = 0xFFFFFFFFu;
    return f;
}

// One job = one trace checked on one region.  A single-trace check is a batch
// of one job; a batch interleaves the jobs' stages wave-major.
struct hr_jobd {
    const hr_record* trace;
    unsigned long long n;         // records
    unsigned long long kb;        // kernel base added to every record's kernel, shifted left by 32
    unsigned region;
    unsigned G;                   // records per pre-pass interval
    unsigned int_begin;           // first global pre-pass interval of this job
    unsigned n_int;
    unsigned wave_begin;          // first global wave index (written on the device)
    unsigned n_waves;             // waves of this job (written on the device)
    unsigned long long done_ns;   // device clock when the job's last stage completed (0: no stages)
};

// Work stages: per wave an optional shadow clear (when the kernel-tag group
// changes) followed by the wave's record tiles.  A stage waits for `dep`, the
// previous stage of the same job, to reach `dep_need` per-warp completions.
enum { HR_STAGE_RECORDS = 0, HR_STAGE_CLEAR = 1 };
constexpr unsigned HR_NO_DEP = 0xFFFFFFFFu;

struct hr_stage {
    unsigned item_begin;  // first global work-item index of the stage
    unsigned wave;        // global wave index
    unsigned type;
    unsigned done;        // per-warp completions of this stage's items
    unsigned dep;
    unsigned dep_need;
    unsigned job;
    unsigned last;        // 1: the job's last stage (its completion time is recorded)
};

constexpr unsigned HR_BIN_SKEW = 256;           // a segment with more than 1/this of the accesses ...
constexpr unsigned HR_BIN_SKEW_MIN = 1u << 22;  // ... of a check this large goes to the per-wave checker

struct hr_ctl {
    unsigned ticket;       // next work item
    unsigned abort;        // set when a bounded wait expired
    unsigned n_waves;
    unsigned n_stages;
    unsigned total_items;
    unsigned n_jobs;
    unsigned n_intervals;
    unsigned binned;       // 1: the binned checker took this check (the per-wave checker then has no items)
    unsigned long long t0_ns;  // device clock when the check's first kernel started
    unsigned bin_parts;    // binned checker: (slice, wave) parts of the trace
    unsigned bin_total;    // binned checker: accesses moved into buckets
    unsigned fresh;        // 1: every shadow value reads as INIT for this check's first wave (the region
                           // is new or reset, or its last record came from an older kernel and no device
                           // view writes it), so a shadow segment need not be read
    unsigned bin_max_tid;  // binned checker: largest thread id of an applied access
    unsigned bin_pack4;    // binned checker: bucketed accesses are 4 bytes (tid < 2^(30 - HR_BIN_SEG_SHIFT))
    unsigned bin_tbits;    // binned checker: 0, or the tid width of a 4-byte working shadow in shared memory
                           // (fresh checks whose tids and clocks fit it)
    unsigned seg_ticket;   // binned checker: next segment a thread group of the segment pass takes
    unsigned bin_max_seg;  // binned checker: accesses of the fullest segment
    unsigned bin_count;    // binned checker: accesses counted into buckets
    unsigned bin_skip;     // automatic route: 1: the pre-pass left this check to the per-wave checker
    unsigned bin_every;    // 1: every-epoch region (binned only in the 4-byte working form)
    unsigned run_items;    // total_items, or 0 where both per-wave checkers are launched and hr_check_kernel has them
    unsigned check_items;  // total_items, or 0 where both are and hr_run_kernel has them
    unsigned bin_err;      // automatic route: 1: the count pass met an error (the per-wave checker then
                           // does the check, and reports it)
};

// Whether the binned checker applies this check (the flag, and the skew guard:
// one thread group applies a segment's accesses, so a large check whose fullest
// segment holds more than 1/HR_BIN_SKEW of them - the hub words of a power-law
// graph - goes to the per-wave checker instead, which is launched after the
// binned kernels).  Read by the kernels after the count and scan passes.
__host__ __device__ inline bool hr_bin_taken(const hr_ctl* c)
{
    return c->binned && !c->bin_err && !(c->bin_every && !c->bin_tbits) && !(c->bin_count >= HR_BIN_SKEW_MIN && (unsigned long long)c->bin_max_seg * HR_BIN_SKEW > c->bin_count);
}

// The automatic route: a check for which no variant was chosen takes the binned
// checker when its pre-pass expects that to be faster, and the count pass meets no
// error.  The expectation, in picoseconds: the per-wave checker needs 20 us, 9 us a
// wave and 28 ps a record; the binned one 75 us, 18 ps a record, 2.4 ps a word of the
// region (its shadow is written, and read unless nothing in it is live) and 1.6 ns an
// access of the fullest segment (one thread group applies it), which a sample of the
// records estimates.  The per-wave figures are those of variant 0 with ordinary
// launches; the shapes that run now take about 6 us a wave, so near break-even the
// binned checker is taken a little early.  Measured on global-memory traces (us a call,
// pre-pass included, per-wave variants 1 and 3 / binned / what the rule gives): 32 waves,
// 0.29M records on 2^20 words 234 and 201 / 102 / 94, 4.7M on 2^22 words 330 and 407 /
// 148 / 143, 75.2M on 2^26 words 1,967 and 2,135 / 1,315 / 1,291; 8 waves, 0.26M on
// 2^22 words 92 and 82 / 80 / 71; 4 waves, 0.57M on 2^22 words 66 and 72 / 79 / 75; one
// wave, 0.26M on 2^22 words 34 and 38 / 72 / 43.  A check that the pre-pass leaves to the
// per-wave checker pays about 6 us for the binned kernels that find nothing to do;
// smaller checks and regions never get there.
// Every-epoch regions take it when nothing in their shadow is live: there the
// per-wave checker needs 40 ps a record and the binned one 30 ps (pre-pass and check,
// 32 waves: 4.7M records 565 and 245 us, 18.8M 1043 and about 620 us).
constexpr unsigned long long HR_BIN_AUTO_MIN_N = 1ull << 18;     // records
constexpr unsigned long long HR_BIN_AUTO_MAX_N = 1ull << 27;     // (1 GiB of bucketed accesses)
constexpr unsigned long long HR_BIN_AUTO_BYTES = 3ull << 30;     // scratch a context allocates for it, at most
constexpr unsigned HR_BIN_AUTO_SEGS = 256;
constexpr unsigned HR_BIN_SAMPLES = 4096;                        // records sampled
constexpr unsigned long long HR_BIN_AUTO_PS_WAVE = 9000000, HR_BIN_AUTO_PS_REC = 28, HR_BIN_AUTO_PS_SKIP = 20000000,
                             HR_BIN_AUTO_PS_BIN = 75000000,
                             HR_BIN_AUTO_PS_BIN_REC = 18, HR_BIN_AUTO_PS_BIN_5_WORDS = 12,
                             HR_BIN_AUTO_PS_BIN_FULLEST = 1600, HR_BIN_AUTO_PS_REC_EVERY = 40,
                             HR_BIN_AUTO_PS_BIN_REC_EVERY = 30, HR_BIN_AUTO_PS_BIN_FULLEST_EVERY = 4000;

// Records of a piece of a trace in host memory, for `n` of them (at most HR_HOST_GROUP,
// which count together against the wave limit).  The copy of a piece hides the check of
// the one before, so only the last piece's check adds to the copies, while a piece is
// checked in less time than it is copied (16 B a record at 211 GB/s: 76 ps).  The
// per-wave checker touches the words a piece accesses: 2^21 records (0.16 ms of copy)
// are enough.  So are they where the library picks the checker for each piece.  The
// chosen binned checker reads and writes the whole shadow with every piece, as only the
// first one can find it fresh: about 75 us, 18 ps a record and 2.5 ps a word (4.5 ps on
// the 4-byte shadow).  Its pieces are the smallest equal parts that keep a quarter of the
// copy's time to spare, in whole MB (copies that start at an odd multiple of 16 B are
// slower: 6,428 us instead of 6,131 for the first of these traces).  Measured (us a call from page-locked memory; pieces of 2^21,
// 2^22, 2^23, 2^24): 75.2M records on 2^26 words 10,135, 6,206, 6,124, 6,105 (4-byte
// shadow 14,721, 8,540, 6,277, 6,357); 37.6M on 2^25 3,707, 3,116, 3,118, 3,251; 9.4M on
// 2^25 1,190, 1,114, 1,156, 1,071; 18.8M on 2^24 1,668, 1,660, 1,730, 1,808.  By this
// rule: 6,131 (4-byte 6,277), 3,112, 1,019 and 1,630.
constexpr unsigned long long HR_HOST_GROUP = 1ull << 24, HR_HOST_PIECE = 1ull << 21;
constexpr unsigned long long hr_host_piece(unsigned long long n, bool binned, unsigned long long n_words,
                                           unsigned shadow_bytes)
{
    if (!binned) return HR_HOST_PIECE;
    const unsigned long long check_ps = 75000000ull + n_words * (shadow_bytes == 4 ? 9 : 5) / 2;
    const unsigned long long least = check_ps * 5 / 4 / (76 - 18);
    const unsigned long long parts = n / (least > HR_HOST_PIECE ? least : HR_HOST_PIECE);
    return parts > 1 ? ((n + parts - 1) / parts + 0xFFFFull) & ~0xFFFFull : n;
}

// Scratch of the binned checker (hr_binned.cu), one per region.  The region's
// shadow is cut into segments of HR_BIN_SEG words.  The trace is cut into one
// contiguous slice per streaming CTA, and a slice into parts, one per wave it
// meets; parts are numbered in trace order, so their waves ascend.  The table
// holds, for segment s and part p at s * n_parts + p, first the part's number
// of accesses to the segment, then (after an exclusive scan in that order) where
// they go in the bucketed access array: segment-major, waves ascending.
#ifndef HR_BIN_SEG_SHIFT_BITS
#define HR_BIN_SEG_SHIFT_BITS 12
#endif
constexpr unsigned HR_BIN_SEG_SHIFT = HR_BIN_SEG_SHIFT_BITS;
constexpr unsigned HR_BIN_SEG = 1u << HR_BIN_SEG_SHIFT;  // shadow words per segment (4 or 8 B each in shared memory)
static_assert(HR_BIN_SEG_SHIFT >= 10 && HR_BIN_SEG_SHIFT <= 13, "the packed access keeps 16 bits for the word");
constexpr unsigned HR_BIN_MAX_SEGS = 16384;              // larger regions take the per-wave checker
constexpr unsigned HR_BIN_MAX_WAVES = 256;               // checks with more waves take the per-wave checker
constexpr unsigned HR_BIN_SCAN = 4096;                   // table entries per scan block
constexpr unsigned HR_BIN_CLUSTER = 4;                   // CTAs sharing bucket cursors in the scatter ...
constexpr unsigned HR_BIN_CLUSTER_FEW = 2;               // ... for regions of at most HR_BIN_FEW_SEGS segments
constexpr unsigned HR_BIN_FEW_SEGS = 2048;
constexpr unsigned HR_BIN_MAX_SUB = 16;                  // count slices per cluster slice, at most
struct hr_bin {
    unsigned* table;         // [seg_cap * part_cap] counts, then offsets
    unsigned* sums;          // [seg_cap * part_cap / HR_BIN_SCAN + 1] per scan block
    unsigned* part_wave;     // [part_cap] wave of each part (ascending)
    unsigned char* clear;    // [HR_BIN_MAX_WAVES] 1: the shadow is cleared before this wave
    uint2* out;              // [out_cap] bucketed accesses {tid, op << 16 | word within the segment}, or
                             // when ctl->bin_pack4 as unsigned tid << (SEG_SHIFT + 2) | op << SEG_SHIFT | word
    unsigned long long out_cap;
    unsigned n_seg;          // segments of this check's region
    unsigned seg_cap;        // segments the table holds
    unsigned part_cap;       // parts the table holds: HR_BIN_MAX_WAVES + slices - 1
    unsigned cluster;        // CTAs of a scatter cluster (hr_bin_shape())
    unsigned clusters;       // scatter clusters
    unsigned sub;            // count slices per cluster slice
    unsigned slices;         // count slices (CTAs of the count pass): clusters * sub
    unsigned every;          // 1: the region reports every epoch
    unsigned automatic;      // 1: no variant was chosen; the check takes this route where it is faster
    unsigned pow2;           // 1: block size and warp size are powers of two (bit-operation FSM step)
};

// Scratch of one check (device memory): job table, pre-pass counts, wave
// table, stage list and control block.
struct hr_work {
    hr_jobd* jobs;                   // [max_jobs]
    unsigned* counts;                // [max_intervals] boundaries per interval, then offsets among the job's waves
    unsigned long long* wave_start;  // [max_waves] first record (index into the job's trace)
    unsigned long long* wave_end;    // [max_waves] one past the last record
    unsigned long long* wave_key;    // [max_waves] rebased wave key
    hr_stage* stages;                // [2 * max_waves + 1]
    hr_ctl* ctl;
    unsigned max_waves;
    unsigned max_intervals;
    unsigned max_jobs;
    unsigned tile;                   // records per work item (set per kernel variant)
    unsigned check_tile;             // 0, or both per-wave checkers are launched: hr_check_kernel's records per item
    unsigned long long clear_words;  // shadow words per clear item (likewise)
    unsigned long long n_words;      // single traces: words of the region
    unsigned pow2;                   // single traces: 1: block size and warp size are powers of two
    unsigned consumers;              // per-warp completions per work item
    unsigned cas_cap;                // CAS retries before HR_ERR_CONTENTION
    unsigned long long wait_ns;      // bound of every device-side wait
    unsigned test_flags;             // HR_TEST_* hooks (tests only)
    unsigned views;                  // 1: a device view of the checked region exists (inline writes may
                                     // carry kernel ordinals the region's last key does not know)
    unsigned tell;                   // 1: the regions have hr_told copies
    unsigned cont;                   // 1: goes on with the record group of the region's last check, whose
                                     // waves count together against max_waves (single-trace checks only)
    hr_bin bin;                      // binned checker scratch (variant HR_BIN_VARIANT and the automatic route)
};

constexpr unsigned long long HR_DEFAULT_WAIT_NS = 4000000000ull;  // 4 s
constexpr unsigned HR_DEFAULT_CAS_CAP = 4096;

// bytes of an hr_work scratch block for the given capacities (256-B aligned parts)
inline size_t hr_work_bytes(unsigned max_jobs, unsigned max_intervals, unsigned max_waves)
{
    auto a = [](size_t x) { return (x + 255) & ~size_t(255); };
    return a(sizeof(hr_ctl)) + a((size_t)max_jobs * sizeof(hr_jobd)) + a((size_t)max_intervals * 4) +
           3 * a((size_t)max_waves * 8) + a((size_t)(2 * max_waves + 1) * sizeof(hr_stage));
}

// carve an hr_work out of `mem` (hr_work_bytes(...) bytes, 256-B aligned)
inline hr_work hr_work_at(void* mem, unsigned max_jobs, unsigned max_intervals, unsigned max_waves)
{
    auto a = [](size_t x) { return (x + 255) & ~size_t(255); };
    char* p = (char*)mem;
    hr_work w{};
    w.ctl = (hr_ctl*)p;
    p += a(sizeof(hr_ctl));
    w.jobs = (hr_jobd*)p;
    p += a((size_t)max_jobs * sizeof(hr_jobd));
    w.counts = (unsigned*)p;
    p += a((size_t)max_intervals * 4);
    w.wave_start = (unsigned long long*)p;
    p += a((size_t)max_waves * 8);
    w.wave_end = (unsigned long long*)p;
    p += a((size_t)max_waves * 8);
    w.wave_key = (unsigned long long*)p;
    p += a((size_t)max_waves * 8);
    w.stages = (hr_stage*)p;
    w.max_waves = max_waves;
    w.max_intervals = max_intervals;
    w.max_jobs = max_jobs;
    w.cas_cap = HR_DEFAULT_CAS_CAP;
    w.wait_ns = HR_DEFAULT_WAIT_NS;
    w.test_flags = 0;
    return w;
}

constexpr unsigned HR_MAX_BATCH = 512;  // jobs per batched launch

// Kernel variants (chosen by hr_set_variant / hr_autotune): consumer warps per
// CTA, records per consumer lane, warp aggregation.  Even ids aggregate; the
// odd id after each is the same shape without aggregation.
struct hr_variant {
    int aggregate;
    int rpl;         // records per consumer lane per tile
    int consumers;   // consumer warps per CTA (plus one producer warp)
};
constexpr hr_variant HR_VARIANTS[] = {{1, 4, 8}, {0, 4, 8}, {1, 2, 8}, {0, 2, 8}, {1, 1, 8}, {0, 1, 8}};
constexpr unsigned HR_N_SHAPES = sizeof(HR_VARIANTS) / sizeof(HR_VARIANTS[0]);
// The binned checker (hr_binned.cu): single-trace checks of first-race regions
// only; batches, and checks it cannot take, run the per-wave checker of shape 3.
constexpr unsigned HR_BIN_VARIANT = HR_N_SHAPES;
constexpr unsigned HR_BIN_FALLBACK = 3;
constexpr unsigned HR_N_VARIANTS = HR_N_SHAPES + 1;  // ids a caller may choose
// Internal id of the checkers that carry the every-epoch path (hr_check_kernel in
// variant 3's shape, hr_run_kernel); checks on regions in that report mode use it.
constexpr unsigned HR_EVERY_EPOCH_VARIANT = HR_N_VARIANTS;
// Batches for which no variant was chosen: four records a lane without aggregation,
// the fastest shape of every batch measured.  Variants 0, 1, 2, 3: 64 uneven
// traces (tree reductions and global-memory mixes, 110M records) 3.00, 2.20, 2.72,
// 2.39 ms; 16 power-law pushes (38M) 2.27, 1.60, 1.68, 1.70 ms.
constexpr unsigned HR_BATCH_DEFAULT = 1;
// Single traces for which none was chosen: two records a lane (variant 3) when words
// are met again and again (the accesses mostly end early, and more warps hide more
// latency) or the trace is small (its waves then reach more warps), else four
// (variant 1).  Calls with variants 0, 1, 2, 3: tree reductions of 0.1M, 1M and 10M
// records 129, 104, 99, 80 us, 137, 106, 110, 92 us and 273, 219, 230, 194 us; power-law
// pushes of 2.6M, 9.6M and 48M records 204, 209, 195, 204 us, 229, 215, 190, 181 us and
// 961, 886, 778, 727 us; global-memory traces of 0.29M, 4.7M and 75M records
// (variants 0, 1, 3) 285, 253, 214 us, 364, 324, 378 us and 2212, 1913, 1972 us.
constexpr unsigned long long HR_SMALL_TRACE = 1ull << 19;
constexpr unsigned hr_default_variant(unsigned long long n, unsigned long long n_words)
{
    return n / 8 >= n_words || n < HR_SMALL_TRACE ? 3u : 1u;
}
constexpr unsigned hr_variant_consumers(unsigned v)
{
    return v == HR_EVERY_EPOCH_VARIANT ? 8u
                                       : (unsigned)HR_VARIANTS[v == HR_BIN_VARIANT ? HR_BIN_FALLBACK : v].consumers;
}
constexpr unsigned hr_variant_tile(unsigned v)
{
    return v == HR_EVERY_EPOCH_VARIANT ? 8u * 32u * 2u
           : v == HR_BIN_VARIANT       ? hr_variant_tile(HR_BIN_FALLBACK)
                                       : HR_VARIANTS[v].consumers * 32u * HR_VARIANTS[v].rpl;
}
// The checker of a single trace: hr_run_kernel (hr_runs.cu) for variants 0 to 3 and
// every-epoch regions, hr_check_kernel for variants 4 and 5, or the one that the trace's
// waves are better for.  The host does not know the waves, so both are launched then and
// the pre-pass leaves one of them no items (about 1 us).
//
// Every-epoch regions (us, hr_check_kernel with 2 records a lane / hr_run_kernel with 4;
// waves of n records): 0.29M records in 32 waves 335 / 457, 1.03M in 32 307 / 390, 2.35M
// in 32 447 / 512; 3.5M in 32 587 / 539, 18.8M in 32 1,446 / 1,055, 37.6M in 32 2,072 /
// 1,900; 9.2M in 4 512 / 633, 75.2M in 32 3,650 / 3,928; 0.57M in 4 87 / 104, 2.3M in 4
// 211 / 192.
constexpr unsigned HR_RUN_EVERY_RPL = 4;  // records per lane in every-epoch regions
enum hr_route { HR_ROUTE_RUNS, HR_ROUTE_TILES, HR_ROUTE_BY_WAVES };
constexpr unsigned long long HR_EVERY_RUNS_MIN_N = 1ull << 21;  // records, and of a wave:
constexpr unsigned long long HR_EVERY_RUNS_MIN_WAVE = 98304, HR_EVERY_RUNS_MAX_WAVE = 1250000;
// First-race regions: a single block's shared array, met again and again between
// barriers, changes state with nearly every access, so looking for absorbed accesses
// first only adds to them: most where a block of odd size makes every look three
// divisions, and where lanes are aggregated.  A launch on as few words (a small graph)
// has one wave or a few, and there hr_run_kernel is ahead by 1.1 to 1.8.  Reductions of 6
// to 10 waves, hr_check_kernel / hr_run_kernel, variants 1, 2, 3: 0.63M records of
// 352-thread blocks 132 / 132, 117 / 132, 91 / 103; 2.1M of 352-thread blocks 138 / 156,
// 146 / 167, 115 / 139; 7.1M of 736-thread blocks 232 / 269, 251 / 283, 210 / 238; 10.1M of
// 96-thread blocks 208 / 201, 269 / 222, 201 / 191; 1.06M of 256-thread blocks 115 / 104,
// 107 / 118, 91 / 92; 10.3M of 1,024-thread blocks 238 / 263, 271 / 258, 228 / 220.
// Where each word is met thousands of times in all, most are absorbed again and
// hr_run_kernel is ahead: 2.8M records of 768-thread blocks on 1,536 words 207 / 186.
constexpr unsigned long long HR_SMALL_WORDS = 1ull << 14, HR_SMALL_MEETINGS = 1536;  // words, records a word
constexpr unsigned HR_SMALL_RUNS_WAVES = 4;  // waves that stay with hr_run_kernel
constexpr hr_route hr_single_route(unsigned v, unsigned long long n, unsigned long long n_words, bool pow2)
{
    if (v == HR_EVERY_EPOCH_VARIANT) return n < HR_EVERY_RUNS_MIN_N ? HR_ROUTE_TILES : HR_ROUTE_BY_WAVES;
    if (v >= 4) return HR_ROUTE_TILES;
    const bool large = n >= 1ull << 23, odd = !pow2 && n >= 1ull << 19;
    const bool tiles = v == 1 ? odd || large : v == 2 ? n >= 1ull << 18 && !large : v == 3 && odd && !large;
    return tiles && n_words <= HR_SMALL_WORDS && n <= n_words * HR_SMALL_MEETINGS ? HR_ROUTE_BY_WAVES : HR_ROUTE_RUNS;
}
// HR_ROUTE_BY_WAVES: whether hr_check_kernel takes a trace of n records in `waves` waves
__host__ __device__ constexpr bool hr_waves_tiled(bool every, unsigned long long n, unsigned waves)
{
    return every ? n < waves * HR_EVERY_RUNS_MIN_WAVE || n > waves * HR_EVERY_RUNS_MAX_WAVE
                 : waves > HR_SMALL_RUNS_WAVES;
}
constexpr unsigned hr_run_tile(unsigned v)
{
    return 32u * (v == HR_EVERY_EPOCH_VARIANT ? HR_RUN_EVERY_RPL : (unsigned)HR_VARIANTS[v].rpl);
}
constexpr unsigned HR_RUN_CLEAR_WORDS = 1u << 13;  // shadow words per clear item, at least
#ifndef HR_RING_DEPTH
#define HR_RING_DEPTH 2
#endif
#ifndef HR_BATCH
#define HR_BATCH 1
#endif
#ifndef HR_WAIT_SLEEP_MAX_NS
#define HR_WAIT_SLEEP_MAX_NS 1024  // longest back-off between polls of a stage counter
#endif
#ifndef HR_MIN_CTAS
#define HR_MIN_CTAS 3
#endif
constexpr int HR_RING = HR_RING_DEPTH;                   // tiles in flight in shared memory
constexpr unsigned HR_TICKET_BATCH = HR_BATCH;           // tiles a producer claims per ticket
constexpr unsigned HR_CLEAR_WORDS = 1u << 16;  // shadow words per clear item
// Words of a clear item: `step`, or as many more as leave a clear of n_words words at
// most HR_CLEAR_ITEMS items.  A check's items are numbered in 32 bits: its clears (one
// per kernel-tag group, 2^13 at most) then take 2^29 numbers of them; 2^32 words in
// items of 2^13 would take all 2^32.  (Found by the host: the division in hr_run_kernel
// cost its main loop registers, 3 % of the power-law push.)
constexpr unsigned HR_CLEAR_ITEMS = 1u << 16;
__host__ __device__ constexpr unsigned long long hr_clear_words(unsigned long long n_words, unsigned step)
{
    const unsigned long long least = (n_words + HR_CLEAR_ITEMS - 1) / HR_CLEAR_ITEMS;
    return least <= step ? step : (least + step - 1) / step * step;
}
static_assert(hr_clear_words(1ull << 32, HR_CLEAR_WORDS) == HR_CLEAR_WORDS, "hr_check_kernel's clear items");
constexpr unsigned HR_MAX_INTERVALS = 1u << 16;      // pre-pass intervals of a single-trace check
constexpr unsigned HR_BATCH_INTERVALS = 1u << 18;    // pre-pass intervals of a batch
constexpr unsigned long long HR_KEY_MASK = 0xFFFFFFFFFFFFull;

// kernel launch helpers (hr_kernels.cu)
// Check n_jobs jobs (1..HR_MAX_BATCH) on the regions of d_regions with the
// scratch w.  Jobs must name distinct regions and hold n > 0 records.
// *launches (if not NULL) receives the kernels launched: 3 for a single trace (one more
// with both per-wave checkers, five with the binned one), 5 for a batch; one fewer
// without w.tell.
cudaError_t hr_launch_jobs(hr_region_dev* d_regions, const hr_work& w, const hr_jobd* jobs, unsigned n_jobs,
                           const unsigned char* d_table, unsigned variant, cudaStream_t stream,
                           cudaEvent_t before_check, unsigned* launches = nullptr);
// hr_run_kernel for a single trace of n records, after the pre-pass (hr_runs.cu)
cudaError_t hr_launch_runs(hr_region_dev* d_regions, const hr_work& w, unsigned long long n,
                           const unsigned char* d_table, unsigned variant, cudaStream_t stream);
// interval size and count for a job of n records when it may use up to budget intervals
void hr_plan_intervals(unsigned long long n, unsigned budget, unsigned* G, unsigned* n_int);
int hr_check_grid_size(unsigned variant);
constexpr unsigned HR_SMALL_INTERVALS = 4096;  // pre-pass intervals of a trace, at most (one CTA finds its waves)
constexpr unsigned long long HR_RESET_FUSED = 4ull << 20;  // shadow bytes that a reset's one kernel clears itself
// The binned checker's five launches (hr_binned.cu), queued after the pre-pass
// of a single-job check; the per-wave checker queued after them finds no items
// when they took the check.
cudaError_t hr_launch_binned(hr_region_dev* d_regions, const hr_work& w, const unsigned char* d_table,
                             cudaStream_t stream);
// The binned checker's streaming shape for a region of n_seg segments (cluster,
// clusters, sub and slices of *bin).
void hr_bin_shape(unsigned n_seg, hr_bin* bin);
// bytes of a region's binned-checker tables (without the access buffer)
inline size_t hr_bin_table_bytes(unsigned seg_cap, unsigned part_cap)
{
    auto a = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t e = (size_t)seg_cap * part_cap;
    return a(e * 4) + a((e / HR_BIN_SCAN + 1) * 4) + a((size_t)part_cap * 4) + a(HR_BIN_MAX_WAVES);
}
cudaError_t hr_launch_sync_kernel(hr_region_dev* d_region, cudaStream_t stream);
cudaError_t hr_launch_reset(hr_region_dev* d_region, unsigned long long* shadow, unsigned long long shadow_bytes,
                            cudaStream_t stream);
cudaError_t hr_launch_reconfigure(hr_region_dev* d_region, unsigned long long n_words, hr_geom geom,
                                  cudaStream_t stream);
cudaError_t hr_launch_set_filter(hr_region_dev* d_region, hr_filter filter, cudaStream_t stream);
