// word_engine.cuh -- Algorithm 1 (Sec. IV-A) on bitmap words, for abstractions
// whose every box is its plane's entry (plane shape table without mismatch):
// all passes of a solve in one cooperative kernel.
//
// Of the pairs (x, u) whose box holds a cell changed in the previous pass (the
// per-input frontier) most still have a cell of infinite value in their box,
// so their candidate is +inf and they change nothing: on the fire model
// 100 x 100 x 36 x 8 x 15 110 M such pairs are met over a solve, 34 M of them
// with a finite box.  Both tests -- a changed cell in the box, no infinite
// cell in the box -- are answered for 32 cells of one input at once, from
// bitmaps over the cells whose entry says "the window of cells here holds a
// changed (an infinite) cell".  The windows are those of the value tables (one
// cell, 2 and 3 cells along dim 0, 3 x 3 cells on dims 0-1), each also over
// two planes along dims 2 and 3, so a box takes a few unaligned 32-bit reads.
// Only the pairs that pass both tests gather values.
//
// Bitmaps hold every plane (the cells with equal coordinates on dims >= 2) in
// whole words, so a word's cells share their boxes' offsets, and a unit -- up
// to 32 consecutive words of a plane, one per lane -- shares its lists.
//
// One pass, two phases with a grid barrier after each:
//   relax   the units none of whose lookups can meet a changed entry are
//           skipped (the planes' lookups as spans of words against one bit per
//           word); of the others a warp takes one input at a time, lane per
//           word, and the pairs of the masks go to a queue in shared memory; a
//           thread takes a pair (its lookups and its cost in flight together),
//           the smallest candidate of a cell wins, the lowest input among
//           equals.
//   tables  the windows of the units that hold a changed cell nearby; the
//           value tables are recomputed at entries whose window holds a
//           changed cell and no infinite one (entries with an infinite cell
//           are never gathered), a thread per entry.
// Boxes that differ from cell to cell (imported ones, the double integrator):
// the whole grid is one plane, a lane takes a cell and reads its record, the
// same tests go cell by cell, and a unit's spans are those of its own boxes.
//
// V, the tables and the bitmaps stay in the L2; the costs are read in the
// caller's layout [C][U], only by the pairs that pass the tests.
//
// What bounds it: latency.  A pass is two grid barriers (2.4 us each) and a chain
// of about 17 dependent L2 trips; on the fire model's busiest pass the relax phase
// issues in 40% of the cycles and DRAM is at 9%, tables 35% and 8%.  Solves, list
// forms in a graph (tuned where noted) -> this, on one GB300 and the inputs of seed
// 77 of perf/cases.py (another target, obstacles or fires move a case by 2 to 7
// times, both forms alike):
//   double integrator    64 x 64 x 5                    0.96 -> 0.50 ms
//   unicycle             100 x 100 x 32 x 10            2.68 -> 1.28 ms
//   unicycle             200 x 200 x 64 x 10 (tuned)    3.71 -> 1.89 ms
//   fire                 61 x 57 x 24 x 6 x 15          1.54 -> 0.48 ms
//   fire                 100 x 100 x 36 x 8 x 15 (tuned) 6.29 -> 2.93 ms
//   fire, class cost     60 x 60 x 24 x 6 x 15          1.33 -> 0.40 ms
//   fire, hybrid boxes   60 x 60 x 24 x 6 x 15          6.58 -> 0.48 ms
//   16 unicycles in one batch                           11.3 -> 5.0 ms
#pragma once
#include <cstring>

#include "solve_core.cuh"

namespace bfk {

constexpr int kWordThreads = 1024;
constexpr int kWordWarps = kWordThreads / 32;
constexpr int kWordSpans = 32;        // spans of a plane's lookups
constexpr int kWordUnits = 32;        // units a block relaxes at a time (a batch), at most
constexpr int kWordRows = 288;        // ... and (unit, input) rows
constexpr int kWordSlots = 208;       // words of a batch whose cells' candidates are kept at a time
constexpr int kWordPer = 4;           // pairs of a thread at a time
constexpr int kWordPairs = 4096;      // pair queue of a block
constexpr int kWordHead = 8;          // value lookups of a list kept in shared memory
constexpr int kWordEntries = 4096;    // table entries queued by a block
constexpr int kWordMaxU = 32;
constexpr int kWordTest = 128;        // units tested at a time
constexpr unsigned kWordSpinMax = 1u << 28;     // polls of a wait at a barrier
// Forms of the engine's functions.
constexpr int kWordOne = 0;           // one instance
constexpr int kWordMany = 1;          // several instances, each at its own pass
constexpr int kWordClass = 2;         // one instance with a successor class
constexpr int kWordBox = 3;           // one instance whose boxes differ from cell to cell
constexpr int kWordInsts = 128;       // instances of one batched launch
constexpr long long kNoCand = 0x7FFFFFFFFFFFFFFFLL;

// List of a (plane, input): int 0 = bit lookups | bit table << 8, ints 1 .. 31
// their offsets in bits of the bitmaps; int 32 = value lookups | value table
// << 8, ints 36 .. 95 their offsets in cells (padded to a multiple of 4 with
// the first).  A count of 0: no pair of the plane has a box.  Bit table = value
// table (0..3 = cell, 2 and 3 cells along dim 0, 3 x 3) + 4 when over two
// planes along dim 2 + 8 when along dim 3.
constexpr int kWordBits = 31;
constexpr int kWordVals = 60;
constexpr int kWordHdr = kWordBits + 1;          // the value lookups' header
constexpr int kWordVal = kWordHdr + 4;           // their first offset
constexpr int kWordEnt = kWordVal + kWordVals;

struct WordCtr {
    unsigned bar;                     // arrivals at the barrier after the set-up and the tables phases
    int err;                          // invalid input seen during set-up
    int fault;                        // a block gave up waiting at a barrier
    int status;
    int done;
    int ready;                        // batched form: the set-up was run
    long long round;                  // passes completed
    unsigned long long gate[4];       // barrier after the relax phase of pass r: gate[r & 3] = blocks arrived |
                                      // blocks with frontier cells << 16 | blocks with changed cells << 32
    unsigned long long sums[4];       // pass r: frontier cells << 32 | changed cells in sums[r & 3]
    unsigned long long total_relaxed, total_changed, total_pairs;
};

struct WordInst {
    GridDesc g;
    int planes, plane_cells;          // P, cells of a plane
    int plane_words;                  // words of a plane: bit b of word p plane_words + k = cell 32 k + b of plane p
    int unit_words, plane_units;      // words of a unit (the last of a plane may have fewer), units of a plane
    int units;                        // P plane_units
    int S;                            // P plane_words
    // quotients without a divide: by plane_units and unit_words as grid_div, i / U
    // of a row index (< 512) by a 16-bit product
    unsigned pu_mul, uw_mul, u_mul, nb_mul;
    int pu_shr, uw_shr, nb_shr;       // (nb: by the blocks of the launch)
    int vtabs;                        // bit t: some list gathers from value table t
    int btabs;                        // bit t: some list tests bit table t
    const int* lists;                 // [P][U][kWordEnt]
    const unsigned* vbits;            // [U][S] bit = the pair has a box
    const int4* spans;                // [P] (kWordBox: [units]) [kWordSpans] {plane q, first, last word relative to the reader's, 0}: the
                                      // words of q the plane's bit lookups read; q = -1: none, -2: anything
    const void* boxes;                // kWordBox: [U][C] records, compact or wide
    int box_fmt;
    const double* G;                  // [C][U] the caller's costs
    const double* terminal;           // [C] or NULL
    const unsigned char* target;
    const unsigned char* avoid;       // or NULL
    long long* Vnew;                  // [C] keys
    double* gmin;                     // [C] smallest cost of a cell's inputs
    // successor class (K = kWordClass): the cells, their running cost, and the value
    // tables over class cells; tab then holds those over the other cells (kKeyMin:
    // a window without one)
    const unsigned char* cls;         // [C]
    const double* Gc;                 // [C][U]
    long long* tabc[4];
    long long* tab[4];                // V at the start of the pass (kept when lists gather it), M2, M3, M33
    uint2* raw[2];                    // [S] by pass parity: {cells changed in the pass, cells of infinite value}
    unsigned char* flags[2];          // [units] by pass parity: some cell of the unit changed
    unsigned* act;                    // [S] cells that are not avoid cells
    uint2* bt[16];                    // [-1 .. S] {window holds a changed cell, ... an infinite cell}
    unsigned* live;                   // [units] bit = some window of the word holds a changed cell
    unsigned char* mu;                // [C]
    double* V;                        // [C] output
    WordCtr* ctr;
    long long* trace;                 // [trace_cap][4] or NULL
    long long trace_cap;
    long long cap;                    // most passes
};

struct WordSmem {
    long long best[kWordSlots * 32];          // smallest candidate of a slot's cells (kNoCand between windows)
    unsigned bu[kWordSlots * 32];             // its lowest input
    union {
        struct {
            unsigned pair[kWordPairs];        // slot of the window << 13 | bit << 8 | input, ~0: none
            int4 list[kWordRows][1 + kWordHead / 4];    // (unit, input) rows: the value list's head
            unsigned mask[kWordRows][32];     // ... the pairs to relax, by word
            short over[kWordRows];            // rows whose pairs did not fit the queue, -1: queued since
            unsigned f1[kWordUnits * 32];     // frontier cells of the batch's words
            unsigned short slot[kWordUnits * 32];       // words with pairs: their slot in the batch, 0xFFFF: none
            unsigned short word[kWordUnits * 32];       // slots: unit of the batch << 5 | word
            int4 at[kWordSlots];              // slots of the window: {first cell, word, first row, plane | instance << 24}
            int4 unit[kWordTest];             // units to relax {unit, plane | words << 24, first word, first cell}
            // batched form: the units' instances; of the batch's units the first
            // row and the counts, of its rows the unit
            unsigned char inst[kWordTest], of_row[kWordRows];
            int row0[kWordUnits + 1];
            unsigned nf1[kWordUnits], nchg[kWordUnits];
        } r;
        struct {
            int cell[kWordEntries];           // entries to recompute, -1: none
            unsigned char inst[kWordEntries];
        } t;
    };
    // batched form: units of this block before an instance's, its pass, active
    // (one instance: before[0] = the block's units)
    int before[kWordInsts + 1];
    long long round[kWordInsts];
    unsigned char active[kWordInsts];
    int nu;
    unsigned queued;                          // queue length
    int nover;                                // rows that did not fit
    int nslots;
    int nlive;
    int flag;
    unsigned long long gate;
    // of the relax phase (32-bit: the 64-bit shared-memory add is a compare-and-
    // swap loop, which cost a microsecond a pass)
    unsigned nf1, nchg, npairs;               // frontier cells, changed cells, pairs relaxed
    unsigned long long pairs;                 // relaxed since the kernel began (thread 0)
};

// Host: the geometry of an abstraction's bitmaps, and the bytes of an instance's
// engine state: [counters][changed and infinite, by parity][not avoid][windows]
// [live words][changed units, by parity][smallest costs], the windows with room
// for a word before and after.
inline size_t word_up(size_t n) { return (n + 255) / 256 * 256; }

// box: the form for boxes that differ from cell to cell, about a unit per block
// of `blocks` or more.
inline void word_geometry(WordInst& v, const bf_abstraction* a, bool box = false, int blocks = 1) {
    memset(&v, 0, sizeof v);
    v.g = a->g;
    v.planes = box ? 1 : (int)(a->g.C / a->g.stride[2]);
    v.plane_cells = (int)(box ? a->g.C : a->g.stride[2]);
    v.plane_words = box ? (int)((a->g.C + 31) / 32) : a->word_plane_words;
    v.plane_units = (v.plane_words + 31) / 32;
    if (box && v.plane_units < blocks) v.plane_units = blocks < v.plane_words ? blocks : v.plane_words;
    v.unit_words = (v.plane_words + v.plane_units - 1) / v.plane_units;     // even units
    if (box) v.plane_units = (v.plane_words + v.unit_words - 1) / v.unit_words;
    v.boxes = a->d_boxes;
    v.box_fmt = a->box_fmt;
    v.units = v.planes * v.plane_units;
    v.S = v.planes * v.plane_words;
    GridDesc q;
    memset(&q, 0, sizeof q);
    q.n[0] = v.plane_units;
    q.n[1] = v.unit_words;
    grid_divisors(q);
    v.pu_mul = q.dmul[0];
    v.pu_shr = q.dshr[0];
    v.uw_mul = q.dmul[1];
    v.uw_shr = q.dshr[1];
    v.u_mul = (65536u + (unsigned)v.g.U - 1u) / (unsigned)v.g.U;
    v.vtabs = a->word_vtabs;
    v.btabs = a->word_btabs;
    v.lists = a->d_wlists;
    v.vbits = a->d_vbits;
    v.spans = a->d_spans;
}

inline size_t word_state_bytes(const WordInst& v) {
    int nt = 0;
    for (int t = 0; t < 16; ++t) nt += (v.btabs >> t) & 1;
    const size_t words = word_up(4 * (size_t)v.S), units = word_up((size_t)v.units);
    return word_up(sizeof(WordCtr)) + 5 * words + (size_t)nt * (2 * words + 512) + word_up(4 * (size_t)v.units) +
           2 * units + word_up(8 * (size_t)v.g.C);
}

// Carve the state from p (word_state_bytes, zeroed).
inline void word_state(WordInst& v, void* mem) {
    unsigned char* p = (unsigned char*)mem;
    auto take = [&](size_t n) { unsigned char* q = p; p += n; return q; };
    const size_t words = word_up(4 * (size_t)v.S), units = word_up((size_t)v.units);
    v.ctr = (WordCtr*)take(word_up(sizeof(WordCtr)));
    v.raw[0] = (uint2*)take(2 * words);
    v.raw[1] = (uint2*)take(2 * words);
    v.act = (unsigned*)take(words);
    for (int t = 0; t < 16; ++t)
        if ((v.btabs >> t) & 1) v.bt[t] = (uint2*)(take(2 * words + 512) + 256);
    v.live = (unsigned*)take(word_up(4 * (size_t)v.units));
    v.flags[0] = take(units);
    v.flags[1] = take(units);
    v.gmin = (double*)take(word_up(8 * (size_t)v.g.C));
}

// Host: a caller whose launches by the engine are on the device, from before its
// first until it has waited for its last (solve_word.cu).  A block of the engine
// fills an SM and a launch starts when all its blocks fit, so launches at full
// width run one after the other: callers at the same time share the SMs.
struct WordTurn {
    WordTurn();
    ~WordTurn();
    WordTurn(const WordTurn&) = delete;
    WordTurn& operator=(const WordTurn&) = delete;
    int width(int blocks) const;      // blocks of this caller's launches that take `blocks` alone
private:
    int dev = 0, callers = 1, sms = 0;
};

// ---------------------------------------------------------------------------
// grid barrier (cooperative launch: every block is resident)
// ---------------------------------------------------------------------------
// Both barriers: every thread's writes before are visible to every thread
// after (block barrier, releasing arrival of thread 0; acquiring polls, block
// barrier).  2.4 us for 152 blocks of 1024 threads; a relaxed add and polls between
// fences take 2.7.  A wait that gives up (Spin polls) sets `fault` and the block
// leaves the kernel.  kWordSpinMax polls are about 40 s (0.15 us each): a block may
// work for long between two barriers while the others wait, up to 1e10 table lookups
// (10 s) on boxes of a million cells.  (A limit read from memory costs 0.06 us a
// barrier: 1103 -> 1116 us on a unicycle 100 x 100 x 32 x 10.)

// After the set-up and the tables phases; `target` counts arrivals over the
// kernel's life.
template <unsigned Spin = kWordSpinMax>
__device__ __forceinline__ bool word_barrier(WordCtr* k, unsigned& target, WordSmem& sm) {
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&k->bar) : "memory");
        unsigned v, n = 0;
        int ok = 1;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&k->bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if (++n > Spin) { ok = 0; atomicExch(&k->fault, 1); break; }
        }
        sm.flag = ok;
    }
    __syncthreads();
    return sm.flag != 0;
}

// After the relax phase of pass r: the arrivals carry whether any block saw a
// frontier cell and whether any cell changed, so the loop condition costs no
// further read (a line that every warp reads takes microseconds).  Returns the
// gate's value, 0 when the wait gave up.
template <unsigned Spin = kWordSpinMax>
__device__ __forceinline__ unsigned long long word_gate(WordCtr* k, int r, WordSmem& sm) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long s = (unsigned long long)sm.nf1 << 32 | sm.nchg;
        sm.pairs += sm.npairs;
        if (s) atomicAdd(&k->sums[r & 3], s);
        unsigned long long* g = &k->gate[r & 3];
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(g),
                     "l"(1ull + ((s >> 32) ? 1ull << 16 : 0ull) + ((s & 0xFFFFFFFFull) ? 1ull << 32 : 0ull))
                     : "memory");
        unsigned long long v;
        unsigned n = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(g) : "memory");
            if ((v & 0xFFFFull) >= gridDim.x) break;
            if (++n > Spin) { v = 0ull; atomicExch(&k->fault, 1); break; }
        }
        sm.gate = v;
    }
    __syncthreads();
    return sm.gate;
}

// Exclusive prefix sum of n over the warp; *tot the total.
__device__ __forceinline__ unsigned word_scan(unsigned n, unsigned& tot) {
    const int lane = threadIdx.x & 31;
    unsigned pre = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(0xFFFFFFFFu, pre, o);
        if (lane >= o) pre += x;
    }
    tot = __shfl_sync(0xFFFFFFFFu, pre, 31);
    return pre - n;
}

// ---------------------------------------------------------------------------
// set-up: lines 1-9 of Algorithm 1
// ---------------------------------------------------------------------------

// Bit pattern test of clean_cost: NaN, -inf and |finite| > 2^64 are errors.
__device__ __forceinline__ bool bad_cost(long long b) {
    return (unsigned long long)(b & 0x7FFFFFFFFFFFFFFFLL) > 0x43F0000000000000ULL && b != kKeyInf;
}

// Costs staged by a warp at a time: its cells' rows, padded to an odd stride so
// that a lane per cell reads its row without bank conflicts.
constexpr int kWordSlab = 544;

// W = terminal cost, mu = U (hand over), the bitmaps, and one pass over the
// costs: checked, and the smallest of a cell kept (a bound that spares most
// pairs their cost and their other lookups).  A stream at the HBM rate: 345 MB
// on the fire model.
template <int K>
__device__ __forceinline__ void word_init(const WordInst& w, double* slabs) {
    const int lane = threadIdx.x & 31;
    const int U = w.g.U;
    const double inf = __longlong_as_double(kKeyInf);
    double* slab = slabs + (threadIdx.x >> 5) * kWordSlab;
    const unsigned per = w.u_mul;                                        // i / U = i per >> 16 for i < 512
    const unsigned pad = (U & 1) ? 0u : 1u;
    const int nc = U <= 16 ? 32 : 16;                                    // cells staged at a time
    bool bad = false;
    for (int wd = blockIdx.x * kWordWarps + (int)(threadIdx.x >> 5); wd < w.S; wd += gridDim.x * kWordWarps) {
        const int p = wd / w.plane_words;
        const int i0 = (wd - p * w.plane_words) * 32;
        const int nv = min(32, w.plane_cells - i0);
        const long long c0 = (long long)p * w.plane_cells + i0;
        bool fin = false, av = false;
        if (lane < nv) {
            const long long c = c0 + lane;
            double x;
            if (w.terminal) {
                if (!clean_cost(w.terminal[c], x)) { bad = true; x = inf; }
            } else {
                x = w.target[c] ? 0.0 : inf;
            }
            av = w.avoid && w.avoid[c];
            if (av) x = inf;
            const long long k = key_of(x);
            fin = k != kKeyInf;
            w.Vnew[c] = k;
            w.mu[c] = kHandover;
        }
        const unsigned im = __ballot_sync(0xFFFFFFFFu, lane < nv);
        const unsigned f = __ballot_sync(0xFFFFFFFFu, fin);
        const unsigned a = __ballot_sync(0xFFFFFFFFu, av);
        if (lane == 0) {
            w.raw[1][wd] = make_uint2(f, im & ~f);  // "changed" before pass 0
            w.act[wd] = im & ~a;
        }
        for (int h = 0; h < nv; h += nc) {
            const int n = min(nc, nv - h);
            double m = inf;
#pragma unroll 1
            for (int cost = 0; cost < (K == kWordClass ? 2 : 1); ++cost) {
                const long long* src = reinterpret_cast<const long long*>(cost ? w.Gc : w.G) + (c0 + h) * U;
                long long v[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = q * 32 + lane < n * U ? __ldcs(src + q * 32 + lane) : 0ll;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const unsigned i = (unsigned)(q * 32 + lane);
                    bad |= bad_cost(v[q]);
                    if ((int)i < n * U) slab[i + ((i * per) >> 16) * pad] = __longlong_as_double(v[q]);
                }
                __syncwarp();
                if (lane < n) {
                    const double* row = slab + lane * (U + (int)pad);
                    for (int u = 0; u < U; ++u) m = row[u] < m ? row[u] : m;
                }
                __syncwarp();
            }
            if (lane < n) w.gmin[c0 + h + lane] = m;
        }
    }
    if (bad) atomicOr(&w.ctr->err, 1);
}

__device__ __forceinline__ int word_quot(unsigned x, unsigned mul, int shr) { return (int)((__umulhi(mul, x) + x) >> shr); }

// Batched form: instance i's units of this block are first + j gridDim.x
// (rotated from instance to instance: small instances spread over the blocks).
__device__ __forceinline__ int word_first(int i) { return (int)((blockIdx.x + 53u * (unsigned)i) % gridDim.x); }

// One instance: the block's j-th unit.  The blocks are rotated from one round of
// units to the next: planes and bands of rows (a plane's units) of every kind
// come to every block, and the frontier's work with them (without the rotation
// 1262 instead of 1202 us on a unicycle 100 x 100 x 32 x 10, 1302 / 1240 on a fire
// model 61 x 57 x 24 x 6 x 15; inputs of another seed than above).  61 and 53: primes
// that divide neither the 152 SMs nor a share of them (a width they divide is not
// rotated, nothing else).
__device__ __forceinline__ int word_mine(const WordInst& w, int j) {
    const unsigned x = blockIdx.x + 61u * (unsigned)j;
    return j * (int)gridDim.x + (int)(x - (unsigned)word_quot(x, w.nb_mul, w.nb_shr) * gridDim.x);
}

__device__ __forceinline__ int word_share(int units, int first) {
    return first < units ? (units - 1 - first) / (int)gridDim.x + 1 : 0;
}

// ... and how many it has: whole rounds, and one of the last round's.
__device__ __forceinline__ int word_count(const WordInst& w) {
    const int whole = w.units / (int)gridDim.x;
    return whole + (word_mine(w, whole) < w.units ? 1 : 0);
}

// No candidates yet (once per kernel; word_commit restores it).
// w: the instance, where there is one.
__device__ __forceinline__ void word_start(WordSmem& sm, const WordInst* w) {
    for (int i = threadIdx.x; i < kWordSlots * 32; i += kWordThreads) {
        sm.best[i] = kNoCand;
        sm.bu[i] = 0xFFu;
    }
    if (threadIdx.x == 0) {
        sm.pairs = 0ull;
        sm.before[0] = w ? word_count(*w) : 0;
    }
}

// ---------------------------------------------------------------------------
// relax
// ---------------------------------------------------------------------------

// Words of unit un: its plane, its first word in the plane, its word count.
__device__ __forceinline__ void word_unit(const WordInst& w, int un, int& p, int& k, int& n) {
    p = word_quot((unsigned)un, w.pu_mul, w.pu_shr);
    k = (un - p * w.plane_units) * w.unit_words;
    n = min(w.unit_words, w.plane_words - k);
}

// before[] of the active instances (whole block); the total.
__device__ __forceinline__ int word_split(const WordInst* insts, int n, WordSmem& sm) {
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        unsigned sum = 0u;
        for (int i = lane; i - lane < n; i += 32) {
            unsigned tot;
            const unsigned own = i < n && sm.active[i] ? (unsigned)word_share(insts[i].units, word_first(i)) : 0u;
            const unsigned pre = word_scan(own, tot);
            if (i < n) sm.before[i] = (int)(sum + pre);
            sum += tot;
        }
        if (lane == 0) sm.before[n] = (int)sum;
    }
    __syncthreads();
    return sm.before[n];
}

// The instance of the block's c-th unit: the last with before <= c that has units.
__device__ __forceinline__ int word_find(const WordSmem& sm, int n, int c) {
    int a = 0, b = n;
    while (b - a > 1) {
        const int h = (a + b) >> 1;
        if (sm.before[h] <= c) a = h;
        else b = h;
    }
    return a;
}

// Can a lookup of the words k .. k + n - 1 of plane p meet a changed entry?
// (whole warp; lanes take the plane's spans)
// at: the plane, or (kWordBox) the unit.
__device__ __forceinline__ bool word_live(const WordInst& w, int at, int k, int n) {
    const int lane = threadIdx.x & 31;
    const int4 sp = __ldg(w.spans + (long long)at * kWordSpans + lane);
    unsigned hit = sp.x == -2 ? 1u : 0u;
    if (sp.x >= 0) {
        const int a = max(k + sp.y, 0), b = min(k + n - 1 + sp.z, w.plane_words - 1);
        if (a <= b) {
            const int ua = word_quot((unsigned)a, w.uw_mul, w.uw_shr), ub = word_quot((unsigned)b, w.uw_mul, w.uw_shr);
            const unsigned* l = w.live + (long long)sp.x * w.plane_units;
#pragma unroll 4
            for (int j = ua; j <= ub; ++j) {
                const int lo = max(a - j * w.unit_words, 0), hi = min(b - j * w.unit_words, 31);
                hit |= l[j] & bit_range(lo, hi);
            }
        }
    }
    return __any_sync(0xFFFFFFFFu, hit != 0u);
}

// One lookup of word wd: the 32 bits from its first on, moved by off.
__device__ __forceinline__ void word_lookup(const uint2* at, int off, unsigned& chg, unsigned& inf) {
    const uint2* q = at + (off >> 5);
    const uint2 x = q[0], y = q[1];
    chg |= __funnelshift_r(x.x, y.x, off);
    inf |= __funnelshift_r(x.y, y.y, off);
}

// Masks of a word's cells for one input (vb: the pairs with a box): f1 those
// whose box holds a changed cell, the result those whose box holds no infinite
// cell either.
__device__ __forceinline__ unsigned word_mask(const WordInst& w, const int* list, int wd, unsigned vb,
                                              unsigned& f1) {
    const int4 e0 = __ldg(reinterpret_cast<const int4*>(list)), e1 = __ldg(reinterpret_cast<const int4*>(list) + 1);
    const int L = e0.x & 0xFF;
    f1 = 0u;
    if (vb == 0u) return 0u;
    const uint2* at = w.bt[e0.x >> 8] + wd;
    unsigned chg = 0u, inf = 0u;
    word_lookup(at, e0.y, chg, inf);
    if (L > 1) word_lookup(at, e0.z, chg, inf);
    if (L > 2) word_lookup(at, e0.w, chg, inf);
    if (L > 3) word_lookup(at, e1.x, chg, inf);
    if (L > 4) {
        word_lookup(at, e1.y, chg, inf);
        if (L > 5) word_lookup(at, e1.z, chg, inf);
        if (L > 6) word_lookup(at, e1.w, chg, inf);
        for (int j = 7; j < L; ++j) word_lookup(at, __ldg(list + 1 + j), chg, inf);
    }
    f1 = vb & chg;
    return f1 & ~inf;
}

// kWordBox: the box of (c, u): first cell and width per dim; false: blocked.
__device__ __forceinline__ bool word_box(const WordInst& w, int c, int u, int lo[4], int wd[4]) {
    const GridDesc& g = w.g;
    const long long at = (long long)u * g.C + c;
#pragma unroll
    for (int d = 0; d < 4; ++d) { lo[d] = 0; wd[d] = 1; }
    if (w.box_fmt == kBoxCompact) {
        const unsigned long long r = g.D <= 2 ? (unsigned long long)__ldg(reinterpret_cast<const unsigned*>(w.boxes) + at)
                                              : __ldg(reinterpret_cast<const unsigned long long*>(w.boxes) + at);
        if ((rec_byte(r, 1) & 0x7F) == 0) return false;
        int k[4] = {0, 0, 0, 0};
        cell_coords(g, c, k);
#pragma unroll
        for (int d = 0; d < 4; ++d)
            if (d < g.D) {
                wd[d] = rec_byte(r, 2 * d + 1) & 0x7F;
                int l = k[d] + rec_sbyte(r, 2 * d);
                if (g.periodic[d]) {
                    if (l < 0) l += g.n[d];
                    else if (l >= g.n[d]) l -= g.n[d];
                }
                lo[d] = l;
            }
        return true;
    }
    const short* q = reinterpret_cast<const short*>(w.boxes) + at * (2 * g.D);
    if (__ldg(q) == kBlocked) return false;
#pragma unroll
    for (int d = 0; d < 4; ++d)
        if (d < g.D) {
            lo[d] = __ldg(q + d);
            wd[d] = __ldg(q + g.D + d) - lo[d] + 1;
        }
    return true;
}

// The lookups that cover a box, four at a time: f(table, cells e0 .. e3), some of
// them the same.  3 x 3 windows where the box is that large and wraps neither dim
// 0 nor dim 1; else row by row, a row that wraps in two parts.
template <typename F>
__device__ __forceinline__ void word_cover(const GridDesc& g, const int lo[4], const int wd[4], F f) {
    const int n0 = g.n[0], n1 = g.n[1];
    const bool wrap0 = lo[0] + wd[0] > n0;
    const bool big = wd[0] >= 3 && wd[1] >= 3 && !wrap0 && lo[1] + wd[1] <= n1;
    const int step = big ? 6 : 2, top1 = big ? wd[1] - 3 : wd[1] - 1;
    for (int part = 0; part < (wrap0 ? 2 : 1); ++part) {
        const int a = part ? 0 : lo[0], len = part ? lo[0] + wd[0] - n0 : min(wd[0], n0 - lo[0]);
        const int tab = big ? 3 : min(len, 3) - 1, top0 = max(len - 3, 0);
        for (int j3 = 0; j3 < wd[3]; ++j3) {
            int x3 = lo[3] + j3;
            if (x3 >= g.n[3]) x3 -= g.n[3];
            for (int j2 = 0; j2 < wd[2]; j2 += 2) {
                int x2 = lo[2] + j2, y2 = lo[2] + min(j2 + 1, wd[2] - 1);
                if (x2 >= g.n[2]) x2 -= g.n[2];
                if (y2 >= g.n[2]) y2 -= g.n[2];
                const int bx = (x3 * g.n[2] + x2) * n1, by = (x3 * g.n[2] + y2) * n1;
                for (int j1 = 0;; j1 += step) {
                    int x1 = lo[1] + min(j1, top1), y1 = lo[1] + min(j1 + (big ? 3 : 1), top1);
                    if (x1 >= n1) x1 -= n1;
                    if (y1 >= n1) y1 -= n1;
                    for (int q = 0;; q += 3) {
                        const int x0 = a + min(q, top0);
                        f(tab, (bx + x1) * n0 + x0, (bx + y1) * n0 + x0, (by + x1) * n0 + x0, (by + y1) * n0 + x0);
                        if (q >= top0) break;
                    }
                    if (j1 + (big ? 3 : 1) >= top1) break;
                }
            }
        }
    }
}

// kWordBox: a word's masks for input u, lane per cell: f1 the cells whose box
// holds a changed cell, the result those whose box holds no infinite cell either.
__device__ __forceinline__ unsigned word_box_mask(const WordInst& w, int wd, int u, unsigned& f1) {
    const int c = wd * 32 + (threadIdx.x & 31);
    unsigned chg = 0u, inf = 0u;
    int lo[4], wid[4];
    if (c < w.g.C && word_box(w, c, u, lo, wid))
        word_cover(w.g, lo, wid, [&](int t, int e0, int e1, int e2, int e3) {
            const uint2* bt = w.bt[t];
            const uint2 x0 = bt[e0 >> 5], x1 = bt[e1 >> 5], x2 = bt[e2 >> 5], x3 = bt[e3 >> 5];
            chg |= (x0.x >> (e0 & 31)) | (x1.x >> (e1 & 31)) | (x2.x >> (e2 & 31)) | (x3.x >> (e3 & 31));
            inf |= (x0.y >> (e0 & 31)) | (x1.y >> (e1 & 31)) | (x2.y >> (e2 & 31)) | (x3.y >> (e3 & 31));
        });
    f1 = __ballot_sync(0xFFFFFFFFu, chg & 1u);
    return __ballot_sync(0xFFFFFFFFu, (chg & ~inf) & 1u);
}

// Queue the pairs of a row's masks m (whole warp; tag: the lane's word's slot and
// the input).  False: they do not fit.
__device__ __forceinline__ bool word_queue(WordSmem& sm, unsigned m, unsigned tag) {
    if (!__any_sync(0xFFFFFFFFu, m != 0u)) return true;
    const int lane = threadIdx.x & 31;
    unsigned tot, at = 0u;
    unsigned pos = word_scan((unsigned)__popc(m), tot);
    if (lane == 0) at = atomicAdd(&sm.queued, tot);
    at = __shfl_sync(0xFFFFFFFFu, at, 0);
    if (at + tot > (unsigned)kWordPairs) {           // the queue's last places hold nothing
        for (unsigned i = at + lane; i < (unsigned)kWordPairs; i += 32) sm.r.pair[i] = ~0u;
        return false;
    }
    for (pos += at; m; m &= m - 1u) sm.r.pair[pos++] = tag + ((unsigned)(__ffs(m) - 1) << 8);
    return true;
}

// Work the queued pairs off (whole block): a thread per pair, the smallest
// candidate of a cell so far and its lowest input.  A pair whose cell's smallest
// cost plus two of its lookups already reaches W cannot lower it: three of four
// pairs go that way on the fire model (two of three on the unicycle), without
// their own cost (from HBM) and their other lookups; the rest move together,
// warp by warp.  A queue that gives a thread one pair at most skips the test:
// it only adds a round of loads then.
template <int K>
__device__ __forceinline__ void word_pairs(const WordInst& w0, const WordInst* insts, WordSmem& sm) {
    constexpr bool M = K == kWordMany;
    const int np = (int)min(sm.queued, (unsigned)kWordPairs);
    const int lane = threadIdx.x & 31;
    for (int k0 = 0; k0 < np; k0 += kWordPer * kWordThreads) {
        // this thread's places: own[j kWordThreads]
        unsigned* own = sm.r.pair + k0 + threadIdx.x;
        int n = 0;                                         // the warp's pairs that are left
        if (np <= kWordThreads) {
            n = __popc(__ballot_sync(0xFFFFFFFFu, (int)threadIdx.x < np));
        } else if (K == kWordBox) {
            // every pair: there is no list to take two lookups from
#pragma unroll
            for (int j = 0; j < kWordPer; ++j)
                n += __popc(__ballot_sync(0xFFFFFFFFu, k0 + j * kWordThreads + (int)threadIdx.x < np));
        } else {
#pragma unroll
            for (int j0 = 0; j0 < kWordPer; j0 += 2) {
                unsigned e[2];
                long long v[2], a[2], b[2];
                double gm[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    e[j] = k0 + (j0 + j) * kWordThreads + (int)threadIdx.x < np ? own[(j0 + j) * kWordThreads] : ~0u;
                    v[j] = kKeyMin;                        // no pair: W below every candidate
                    gm[j] = 0.0;
                    a[j] = b[j] = kKeyInf;
                    if (e[j] != ~0u) {
                        const int4 at = sm.r.at[e[j] >> 13];
                        const WordInst& w = M ? insts[at.w >> 24] : w0;
                        const int c = at.x + (int)((e[j] >> 8) & 31u);
                        const int* l = reinterpret_cast<const int*>(sm.r.list[at.z + (int)(e[j] & 0xFFu)]);
                        const long long* tb = w.tab[l[0] >> 8] + c;
                        const int o0 = l[4], o1 = l[3 + min(l[0] & 0xFF, kWordHead)];
                        v[j] = w.Vnew[c];
                        gm[j] = w.gmin[c];
                        a[j] = tb[o0];
                        b[j] = tb[o1];
                        if (K == kWordClass) {
                            const long long* tc = w.tabc[l[0] >> 8] + c;
                            a[j] = max(a[j], tc[o0]);
                            b[j] = max(b[j], tc[o1]);
                        }
                    }
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const bool left = key_of(gm[j] + val_of(max(a[j], b[j]))) < v[j];
                    const unsigned m = __ballot_sync(0xFFFFFFFFu, left);
                    if (left) {
                        const int s = n + __popc(m & ((1u << lane) - 1u));
                        // place s of the warp: every place up to it was read
                        sm.r.pair[k0 + (s >> 5) * kWordThreads + ((int)threadIdx.x & ~31) + (s & 31)] = e[j];
                    }
                    n += __popc(m);
                }
            }
            __syncwarp();
        }
        long long d[kWordPer];
#pragma unroll
        for (int j = 0; j < kWordPer; ++j) {
            d[j] = kNoCand;
            if (j * 32 + lane < n) {
                const unsigned e = own[j * kWordThreads];
                if (e != ~0u) {
                    const int4 at = sm.r.at[e >> 13];
                    const WordInst& w = M ? insts[at.w >> 24] : w0;
                    d[j] = __double_as_longlong(
                        __ldcs(w.G + (long long)(at.x + (int)((e >> 8) & 31u)) * w.g.U + (e & 0xFFu)));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kWordPer; ++j) {
            const unsigned e = j * 32 + lane < n ? own[j * kWordThreads] : ~0u;
            if (e == ~0u) continue;
            const int i = (int)(e >> 8), u = (int)(e & 0xFFu);
            const int4 at = sm.r.at[i >> 5];
            const WordInst& w = M ? insts[at.w >> 24] : w0;
            if (K == kWordBox) {
                long long mb = kKeyMin;
                int lo[4], wid[4];
                word_box(w, at.x + (i & 31), u, lo, wid);
                word_cover(w.g, lo, wid, [&](int t, int e0, int e1, int e2, int e3) {
                    const long long* tb = w.tab[t];
                    mb = max(mb, max(max(tb[e0], tb[e1]), max(tb[e2], tb[e3])));
                });
                d[j] = key_of(__longlong_as_double(d[j]) + val_of(mb));
                if (d[j] < *(volatile long long*)&sm.best[i] && d[j] < atomicMin(&sm.best[i], d[j])) sm.bu[i] = 0xFFu;
                continue;
            }
            const int4* l = sm.r.list[at.z + u];
            const int hdr = l[0].x;
            const int L = hdr & 0xFF;
            const long long* tb = w.tab[hdr >> 8] + (at.x + (i & 31));
            const long long* tc = nullptr;
            double gc = 0.0;
            if (K == kWordClass) {
                tc = w.tabc[hdr >> 8] + (at.x + (i & 31));
                gc = __ldcs(w.Gc + (long long)(at.x + (i & 31)) * w.g.U + u);
            }
            long long m = kKeyMin, mc = kKeyMin;
            auto look = [&](const int4& o) {
                m = max(m, max(max(tb[o.x], tb[o.y]), max(tb[o.z], tb[o.w])));
                if (K == kWordClass) mc = max(mc, max(max(tc[o.x], tc[o.y]), max(tc[o.z], tc[o.w])));
            };
            look(l[1]);
            if (L > 4) {
                look(l[2]);
                if (L > kWordHead) {
                    const int4* rest = reinterpret_cast<const int4*>(
                        w.lists + ((long long)(at.w & 0xFFFFFF) * w.g.U + u) * kWordEnt + kWordVal + kWordHead);
                    for (int t = kWordHead; t < L; t += 4) look(__ldg(rest++));
                }
            }
            const double gv = __longlong_as_double(d[j]);
            if (K == kWordClass) {
                // the sup over the box of g(x,y,u) + V(y): each part that has cells
                // is its cost + its max (fl(g + .) is monotone)
                d[j] = kKeyMin;
                if (m != kKeyMin) d[j] = key_of(gv + val_of(m));
                if (mc != kKeyMin) d[j] = max(d[j], key_of(gc + val_of(mc)));
            } else {
                d[j] = key_of(gv + val_of(m));                            // the one FP64 add
            }
            // a smaller candidate: inputs found for the one before are stale
            if (d[j] < *(volatile long long*)&sm.best[i] && d[j] < atomicMin(&sm.best[i], d[j])) sm.bu[i] = 0xFFu;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kWordPer; ++j)
            if (d[j] < kKeyInf) {
                const unsigned e = own[j * kWordThreads];
                if (d[j] == sm.best[e >> 8]) atomicMin(&sm.bu[e >> 8], e & 0xFFu);
            }
        __syncthreads();
    }
}

// The window's cells whose smallest candidate is below W (whole block).
template <int K>
__device__ __forceinline__ void word_commit(const WordInst& w0, const WordInst* insts, int par0, const int4* unit,
                                            int first, int ns, WordSmem& sm) {
    constexpr bool M = K == kWordMany;
    constexpr int R = 3;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int j0 = wid; j0 < ns; j0 += kWordWarps * R) {
        long long b[R], old[R];
        uint2 x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int j = j0 + q * kWordWarps;
            b[q] = kNoCand;
            if (j < ns) {
                const int4 at = sm.r.at[j];
                const WordInst& w = M ? insts[at.w >> 24] : w0;
                const int par = M ? (int)sm.round[at.w >> 24] & 1 : par0;
                b[q] = sm.best[j * 32 + lane];
                if (b[q] != kNoCand) {
                    x[q] = w.raw[par][at.y];
                    old[q] = w.Vnew[at.x + lane];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int j = j0 + q * kWordWarps;
            if (j >= ns) continue;
            const int4 at = sm.r.at[j];
            const WordInst& w = M ? insts[at.w >> 24] : w0;
            bool changed = false;
            if (b[q] != kNoCand) {
                changed = b[q] < old[q];
                if (changed) {
                    w.Vnew[at.x + lane] = b[q];
                    w.mu[at.x + lane] = (unsigned char)sm.bu[j * 32 + lane];
                }
                sm.best[j * 32 + lane] = kNoCand;
                sm.bu[j * 32 + lane] = 0xFFu;
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, changed);
            if (changed && lane == __ffs(m) - 1) {                    // (a lane that has read the word)
                const int par = M ? (int)sm.round[at.w >> 24] & 1 : par0;
                const int ui = sm.r.word[first + j] >> 5;
                w.raw[par][at.y] = make_uint2(m, x[q].y & ~m);
                w.flags[par][unit[ui].x] = 1;
                atomicAdd(M ? &sm.r.nchg[ui] : &sm.nchg, (unsigned)__popc(m));
            }
        }
    }
}

// The relax phase of one pass over this block's share of the units.  count_only:
// the frontier is counted and nothing is relaxed (at the pass cap).  par: the
// pass's parity.  The block's counts go to sm.nf1, sm.nchg and sm.npairs.
// kWordMany: the active ones of n instances, each at
// its own pass (sm.round) and cap, its counts into its own sums.
template <int K>
__device__ __forceinline__ void word_relax(const WordInst& w0, const WordInst* insts, int n_insts, int par,
                                           bool count_only0, WordSmem& sm) {
    constexpr bool M = K == kWordMany;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int U0 = M ? 1 : w0.g.U;
    if (threadIdx.x == 0) sm.nf1 = sm.nchg = sm.npairs = 0u;
    // consecutive units go to different blocks: the frontier is uneven
    const int mine = M ? sm.before[n_insts] : sm.before[0];
    for (int t0 = 0; t0 < mine; t0 += kWordTest) {
        if (threadIdx.x == 0) { sm.nlive = 0; sm.nslots = 0; }
        if (threadIdx.x < kWordUnits * 32) sm.r.f1[threadIdx.x] = 0u;
        __syncthreads();
        for (int i = t0 + wid; i < min(mine, t0 + kWordTest); i += kWordWarps) {
            const int inst = M ? word_find(sm, n_insts, i) : 0;
            const WordInst& w = M ? insts[inst] : w0;
            const int un = M ? word_first(inst) + (i - sm.before[inst]) * (int)gridDim.x : word_mine(w0, i);
            int p, k, n;
            word_unit(w, un, p, k, n);
            if (word_live(w, K == kWordBox ? un : p, k, n) && lane == 0) {         // P < 2^24: checked at build
                const int at = atomicAdd(&sm.nlive, 1);
                sm.r.unit[at] = make_int4(un, p | n << 24, p * w.plane_words + k, p * w.plane_cells + k * 32);
                if (M) sm.r.inst[at] = (unsigned char)inst;
            }
        }
        __syncthreads();
        const int nlive = sm.nlive;
        for (int l0 = 0, nu; l0 < nlive; l0 += nu) {
            const int4* unit = sm.r.unit + l0;
            int rows;
            if (M) {
                if (wid == 0) {
                    // as many units as fit: their first rows
                    const int U = l0 + lane < nlive ? insts[sm.r.inst[l0 + lane]].g.U : 0;
                    unsigned tot;
                    const int r0 = (int)word_scan((unsigned)U, tot);
                    const bool fits = U > 0 && lane < kWordUnits && r0 + U <= kWordRows;
                    const unsigned fm = __ballot_sync(0xFFFFFFFFu, fits);
                    const int cnt = __popc(fm);                          // r0 grows: the first lanes
                    if (fits) {
                        sm.r.row0[lane] = r0;
                        sm.r.nf1[lane] = sm.r.nchg[lane] = 0u;
                        for (int q = 0; q < U; ++q) sm.r.of_row[r0 + q] = (unsigned char)lane;
                        if (lane == cnt - 1) {
                            sm.r.row0[cnt] = r0 + U;
                            sm.nu = cnt;
                        }
                    }
                }
                __syncthreads();
                nu = sm.nu;
                rows = sm.r.row0[nu];
            } else {
                nu = min(min(kWordUnits, kWordRows / U0), nlive - l0);
                rows = nu * U0;
            }
            // few units: every word has its slot from the start and the rows' pairs are
            // queued as they are found; else the words that have pairs get slots first
            const bool direct = nu * 32 <= kWordSlots;
            if (direct) {
                if ((int)threadIdx.x < nu * 32) {
                    const int4 un = unit[threadIdx.x >> 5];
                    const int inst = M ? sm.r.inst[l0 + (threadIdx.x >> 5)] : 0, j = threadIdx.x & 31;
                    sm.r.at[threadIdx.x] = make_int4(un.w + j * 32, un.z + j,
                                                     M ? sm.r.row0[threadIdx.x >> 5] : (int)(threadIdx.x >> 5) * U0,
                                                     (int)((unsigned)(un.y & 0xFFFFFF) | (unsigned)inst << 24));
                    sm.r.slot[threadIdx.x] = (unsigned short)threadIdx.x;
                    sm.r.word[threadIdx.x] = (unsigned short)threadIdx.x;
                }
                if (threadIdx.x == 0) { sm.queued = 0u; sm.nover = 0; sm.nslots = nu * 32; }
                __syncthreads();
            }
            // (unit, input) rows over the warps: the pairs to relax
            if (K == kWordBox) {
                // word by word: lanes take its cells
                for (int x = wid; x < rows * w0.unit_words; x += kWordWarps) {
                    const int it = word_quot((unsigned)x, w0.uw_mul, w0.uw_shr), j = x - it * w0.unit_words;
                    const int ui = (int)((unsigned)it * w0.u_mul >> 16);
                    const int4 un = unit[ui];
                    unsigned f1 = 0u, m = 0u;
                    if (j < (un.y >> 24)) m = word_box_mask(w0, un.z + j, it - ui * U0, f1) & w0.act[un.z + j];
                    if (lane == 0) {
                        if (f1) atomicOr(&sm.r.f1[ui * 32 + j], f1);
                        sm.r.mask[it][j] = m;
                    }
                }
                for (int x = threadIdx.x; x < rows * 32; x += kWordThreads)
                    if ((x & 31) >= w0.unit_words) sm.r.mask[x >> 5][x & 31] = 0u;
            } else {
                for (int it = wid; it < rows; it += kWordWarps) {
                    const int ui = M ? sm.r.of_row[it] : (int)((unsigned)it * w0.u_mul >> 16);
                    const WordInst& w = M ? insts[sm.r.inst[l0 + ui]] : w0;
                    const int U = M ? w.g.U : U0;
                    const int u = it - (M ? sm.r.row0[ui] : ui * U);
                    const int4 un = unit[ui];
                    const int wd = un.z + lane;
                    const int* list = w.lists + ((long long)(un.y & 0xFFFFFF) * U + u) * kWordEnt;
                    unsigned vb = 0u, act = 0u;
                    if (lane < (un.y >> 24)) {
                        vb = __ldg(w.vbits + (long long)u * w.S + wd);
                        act = w.act[wd];
                    }
                    int4 head = make_int4(0, 0, 0, 0);
                    if (lane < 1 + kWordHead / 4) head = __ldg(reinterpret_cast<const int4*>(list + kWordHdr) + lane);
                    unsigned f1;
                    unsigned m = word_mask(w, list, wd, vb, f1) & act;
                    if (f1) atomicOr(&sm.r.f1[ui * 32 + lane], f1);
                    if (lane < 1 + kWordHead / 4) sm.r.list[it][lane] = head;
                    sm.r.mask[it][lane] = m;
                    if (direct) {
                        if (M ? sm.round[sm.r.inst[l0 + ui]] >= w.cap : count_only0) m = 0u;
                        const unsigned n = __reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(m));
                        if (n && lane == 0) atomicAdd(&sm.npairs, n);
                        if (n && !word_queue(sm, m, (unsigned)(ui * 32 + lane) << 13 | (unsigned)u) && lane == 0)
                            sm.r.over[atomicAdd(&sm.nover, 1)] = (short)it;
                    }
                }
            }
            __syncthreads();
            // frontier cells; slots of the words that have pairs
            for (int ui = wid; ui < nu; ui += kWordWarps) {
                const unsigned f1 = sm.r.f1[ui * 32 + lane];
                sm.r.f1[ui * 32 + lane] = 0u;
                const unsigned nf = __reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(f1));
                if (nf && lane == 0) atomicAdd(M ? &sm.r.nf1[ui] : &sm.nf1, nf);
                if (direct) continue;
                unsigned any = 0u, n = 0u;
                const int r1 = M ? sm.r.row0[ui + 1] : (ui + 1) * U0;
                bool count_only = count_only0;
                if (M) count_only = sm.round[sm.r.inst[l0 + ui]] >= insts[sm.r.inst[l0 + ui]].cap;
                for (int it = M ? sm.r.row0[ui] : ui * U0; it < r1; ++it) {
                    const unsigned m = sm.r.mask[it][lane];
                    any |= m;
                    n += (unsigned)__popc(m);
                }
                n = __reduce_add_sync(0xFFFFFFFFu, n);
                const unsigned have = count_only ? 0u : __ballot_sync(0xFFFFFFFFu, any != 0u);
                int s = 0;
                if (lane == 0 && have) {
                    if (!M) atomicAdd(&sm.npairs, n);
                    s = atomicAdd(&sm.nslots, __popc(have));
                }
                s = __shfl_sync(0xFFFFFFFFu, s, 0) + __popc(have & ((1u << lane) - 1u));
                const bool mine_ = (have >> lane) & 1u;
                sm.r.slot[ui * 32 + lane] = mine_ ? (unsigned short)s : (unsigned short)0xFFFFu;
                if (mine_) sm.r.word[s] = (unsigned short)(ui << 5 | lane);
            }
            if (!direct) __syncthreads();
            const int nslots = sm.nslots;
            const bool found = direct && K != kWordBox;      // the pairs are queued already
            // the slots a window at a time
            for (int s0 = 0; s0 < nslots; s0 += kWordSlots) {
                const int ns = min(kWordSlots, nslots - s0);
                if (!direct) {
                    if ((int)threadIdx.x < ns) {
                        const int x = sm.r.word[s0 + threadIdx.x];
                        const int4 un = unit[x >> 5];
                        const int inst = M ? sm.r.inst[l0 + (x >> 5)] : 0;
                        sm.r.at[threadIdx.x] =
                            make_int4(un.w + (x & 31) * 32, un.z + (x & 31), M ? sm.r.row0[x >> 5] : (x >> 5) * U0,
                                      (int)((unsigned)(un.y & 0xFFFFFF) | (unsigned)inst << 24));
                    }
                    if (threadIdx.x == 0) { sm.queued = 0u; sm.nover = 0; }
                    __syncthreads();
                }
                if (!found && !(K == kWordBox && direct && count_only0)) {
                    for (int it = wid; it < rows; it += kWordWarps) {
                        const int ui = M ? sm.r.of_row[it] : (int)((unsigned)it * w0.u_mul >> 16);
                        const int u = it - (M ? sm.r.row0[ui] : ui * U0);
                        const unsigned s = (unsigned)sm.r.slot[ui * 32 + lane] - (unsigned)s0;
                        const unsigned m = s < (unsigned)ns ? sm.r.mask[it][lane] : 0u;
                        if (K == kWordBox && direct) {
                            const unsigned n = __reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(m));
                            if (n && lane == 0) atomicAdd(&sm.npairs, n);
                        }
                        if (!word_queue(sm, m, s << 13 | (unsigned)u) && lane == 0)
                            sm.r.over[atomicAdd(&sm.nover, 1)] = (short)it;
                    }
                    __syncthreads();
                }
                word_pairs<K>(w0, insts, sm);
                // rows that did not fit, until every one was queued
                const int nover = sm.nover;
                for (int more = nover; more;) {
                    __syncthreads();
                    if (threadIdx.x == 0) sm.queued = 0u;
                    __syncthreads();
                    bool again = false;
                    for (int i = wid; i < nover; i += kWordWarps) {
                        const int it = sm.r.over[i];
                        if (it < 0) continue;
                        const int ui = M ? sm.r.of_row[it] : (int)((unsigned)it * w0.u_mul >> 16);
                        const int u = it - (M ? sm.r.row0[ui] : ui * U0);
                        const unsigned s = (unsigned)sm.r.slot[ui * 32 + lane] - (unsigned)s0;
                        const unsigned m = s < (unsigned)ns ? sm.r.mask[it][lane] : 0u;
                        if (word_queue(sm, m, s << 13 | (unsigned)u)) {
                            __syncwarp();
                            if (lane == 0) sm.r.over[i] = -1;
                        } else {
                            again = true;
                        }
                    }
                    more = __syncthreads_or(again ? 1 : 0);
                    word_pairs<K>(w0, insts, sm);
                }
                word_commit<K>(w0, insts, par, unit, s0, ns, sm);
                __syncthreads();
            }
            if (M && (int)threadIdx.x < nu && sm.r.nf1[threadIdx.x]) {
                const int inst = sm.r.inst[l0 + threadIdx.x];
                atomicAdd(&insts[inst].ctr->sums[sm.round[inst] & 3],
                          (unsigned long long)sm.r.nf1[threadIdx.x] << 32 | sm.r.nchg[threadIdx.x]);
            }
            if (threadIdx.x == 0) sm.nslots = 0;
            __syncthreads();
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// tables
// ---------------------------------------------------------------------------

__device__ __forceinline__ void word_or(uint2& a, const uint2& b) {
    a.x |= b.x;
    a.y |= b.y;
}

// The six words of a unit's word that its windows reach: row r (0..2) from word
// k + (r n0 >> 5) of the plane, two words a row.  z: the third word of a row
// whose first bit is bit 31 (34 bits are used), ORed in by the caller's shift.
struct WordRows {
    uint2 a[3], b[3], z[3];
    __device__ __forceinline__ void load(const WordInst& w, const uint2* plane, int k, bool in, bool m33, bool add) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (r && !m33) break;
            const int i = k + ((r * w.g.n[0]) >> 5);
            const uint2 none = make_uint2(0u, 0u);
            const uint2 x = in && i < w.plane_words ? plane[i] : none;
            const uint2 y = in && i + 1 < w.plane_words ? plane[i + 1] : none;
            const uint2 t = ((r * w.g.n[0]) & 31) == 31 && in && i + 2 < w.plane_words ? plane[i + 2] : none;
            if (add) {
                word_or(a[r], x);
                word_or(b[r], y);
                word_or(z[r], t);
            } else {
                a[r] = x;
                b[r] = y;
                z[r] = t;
            }
        }
    }
    // windows over 1, 2, 3 cells along dim 0 and 3 x 3 cells, of one component
    __device__ __forceinline__ void windows(const WordInst& w, bool m33, uint2 out[4]) const {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            if (r && !m33) break;
            const int s = (r * w.g.n[0]) & 31;
            const unsigned lx = __funnelshift_r(a[r].x, b[r].x, s), hx = __funnelshift_r(b[r].x, z[r].x, s);
            const unsigned ly = __funnelshift_r(a[r].y, b[r].y, s), hy = __funnelshift_r(b[r].y, z[r].y, s);
            const uint2 w2 = make_uint2(lx | __funnelshift_r(lx, hx, 1), ly | __funnelshift_r(ly, hy, 1));
            const uint2 w3 = make_uint2(w2.x | __funnelshift_r(lx, hx, 2), w2.y | __funnelshift_r(ly, hy, 2));
            if (r == 0) {
                out[0] = make_uint2(lx, ly);
                out[1] = w2;
                out[2] = w3;
                out[3] = w3;
            } else {
                word_or(out[3], w3);
            }
        }
    }
};

// The planes one step along dims 2 and 3 of plane p, relative in planes (0:
// none).
__device__ __forceinline__ void word_steps(const GridDesc& g, int p, int& s2, int& s3) {
    const int k3 = (int)grid_div(g, 2, (unsigned)p), k2 = p - k3 * g.n[2];
    s2 = g.D < 3 ? 0 : (k2 + 1 < g.n[2] ? 1 : (g.periodic[2] ? -k2 : 0));
    s3 = g.D < 4 ? 0 : (k3 + 1 < g.n[3] ? g.n[2] : (g.periodic[3] ? -k3 * g.n[2] : 0));
}

// Did a cell change that a window of the unit holds (words k .. k + n - 1 of
// plane p)?  One flag per unit; lanes take the planes the windows reach (own,
// along dim 2, dim 3, both) and the units of their words.
__device__ __forceinline__ bool word_touched(const WordInst& w, const unsigned char* flags, int p, int k, int n) {
    const int lane = threadIdx.x & 31;
    int s2 = 0, s3 = 0;
    if (w.btabs & 0xFFF0) word_steps(w.g, p, s2, s3);         // else no window reaches another plane
    const int q = p + ((lane & 8) ? s2 : 0) + ((lane & 16) ? s3 : 0);
    const int last = min(k + n - 1 + ((2 * w.g.n[0] + 33) >> 5), w.plane_words - 1);
    bool hit = false;
    for (int j = word_quot((unsigned)k, w.uw_mul, w.uw_shr) + (lane & 7); j * w.unit_words <= last; j += 8)
        hit |= flags[q * w.plane_units + j] != 0;
    return __any_sync(0xFFFFFFFFu, hit);
}

// Write the bit tables first .. first + 3 at word wd; changed bits of the tables
// in use into any.
__device__ __forceinline__ void word_put(const WordInst& w, int wd, int first, const uint2 x[4], unsigned& any) {
#pragma unroll
    for (int t = 0; t < 4; ++t)
        if ((w.btabs >> (first + t)) & 1) {
            any |= x[t].x;
            w.bt[first + t][wd] = x[t];
        }
}

// The windows of the unit's words (lane: word k + lane of plane p; in: the lane
// has a word) into the bit tables; the result: the cells whose value-table
// entries are to be recomputed.  The windows over two planes are the windows of
// the planes' words ORed.
// r: the unit's own rows, loaded.
__device__ __forceinline__ unsigned word_tables_at(const WordInst& w, const uint2* raw, int p, int k, bool in,
                                                   WordRows& r, unsigned& any) {
    const bool m33 = ((w.btabs | w.vtabs) & 0x8888) != 0;
    const int wd = p * w.plane_words + k;
    const uint2* own = raw + (long long)p * w.plane_words;
    int s2 = 0, s3 = 0;
    if (w.btabs & 0xFFF0) word_steps(w.g, p, s2, s3);
    const long long d2 = (long long)s2 * w.plane_words, d3 = (long long)s3 * w.plane_words;
    uint2 x[4];
    unsigned need = 0u;
    r.windows(w, m33, x);
#pragma unroll
    for (int t = 0; t < 4; ++t)
        if ((w.vtabs >> t) & 1) {
            need |= x[t].x & ~x[t].y;
            any |= x[t].x;
        }
    if (in && (w.btabs & 0x000F)) word_put(w, wd, 0, x, any);
    if (w.btabs & 0xF0F0) {
        r.load(w, own + d2, k, in && s2 != 0, m33, true);
        if (w.btabs & 0x00F0) {
            r.windows(w, m33, x);
            if (in) word_put(w, wd, 4, x, any);
        }
        if (w.btabs & 0xF000) {
            r.load(w, own + d3, k, in && s3 != 0, m33, true);
            r.load(w, own + d2 + d3, k, in && s2 != 0 && s3 != 0, m33, true);
            r.windows(w, m33, x);
            if (in) word_put(w, wd, 12, x, any);
        }
    }
    if (w.btabs & 0x0F00) {
        r.load(w, own, k, in, m33, false);
        r.load(w, own + d3, k, in && s3 != 0, m33, true);
        r.windows(w, m33, x);
        if (in) word_put(w, wd, 8, x, any);
    }
    return need;
}

// One value table family at cell c: windows of val(x) over 1, 2, 3 and 3 x 3
// cells.  Windows that reach past a row's or the grid's end are never gathered;
// their cells are clamped to the array.
template <typename F>
__device__ __forceinline__ void word_windows_at(const WordInst& w, long long* const* tab, int c, F val) {
    const int n0 = w.g.n[0], last = (int)(w.g.C - 1);
    const long long v0 = val(c);
    if (w.vtabs & 14) {
        const long long m2 = max(v0, val(min(c + 1, last)));
        const long long m3 = max(m2, val(min(c + 2, last)));
        if (w.vtabs & 8) {
            long long r[6];
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    r[b * 3 + a] = val((int)min((unsigned)c + (unsigned)((b + 1) * n0 + a), (unsigned)last));
            tab[3][c] = max(m3, max(max(r[0], max(r[1], r[2])), max(r[3], max(r[4], r[5]))));
        }
        if (w.vtabs & 4) tab[2][c] = m3;
        if (w.vtabs & 2) tab[1][c] = m2;
    }
    if (w.vtabs & 1) tab[0][c] = v0;
}

// Recompute the value tables at cell c.
template <int K>
__device__ __forceinline__ void word_entry(const WordInst& w, int c) {
    if (K == kWordClass) {
        word_windows_at(w, w.tab, c, [&](int x) { return w.cls[x] ? kKeyMin : w.Vnew[x]; });
        word_windows_at(w, w.tabc, c, [&](int x) { return w.cls[x] ? w.Vnew[x] : kKeyMin; });
    } else {
        word_windows_at(w, w.tab, c, [&](int x) { return w.Vnew[x]; });
    }
}

// The tables phase after a pass of parity par (first: after the set-up, which
// counts as parity 1, every unit).  kWordMany: of the active instances, after
// the pass before sm.round.
template <int K>
__device__ __forceinline__ void word_tables(const WordInst& w0, const WordInst* insts, int n_insts, int par0, bool first0,
                                            WordSmem& sm) {
    constexpr bool M = K == kWordMany;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) sm.queued = 0u;
    __syncthreads();
    const int mine = M ? sm.before[n_insts] : sm.before[0];
    for (int i = wid; i < mine; i += kWordWarps) {
        const int inst = M ? word_find(sm, n_insts, i) : 0;
        const WordInst& w = M ? insts[inst] : w0;
        const int un = M ? word_first(inst) + (i - sm.before[inst]) * (int)gridDim.x : word_mine(w0, i);
        const int par = M ? (int)(sm.round[inst] + 1) & 1 : par0;
        const bool first = M ? sm.round[inst] == 0 : first0;
        const uint2* raw = w.raw[par];
        int p, k, n;
        word_unit(w, un, p, k, n);
        const bool in = lane < n;
        const int wd = p * w.plane_words + k + lane;
        const bool before = w.live[un] != 0u;                    // windows to clear
        // the unit's rows are read with its flags: most units that are looked at
        // late in a solve are touched, and the reads are in flight together
        WordRows rows;
        rows.load(w, raw + (long long)p * w.plane_words, k + lane, in, ((w.btabs | w.vtabs) & 0x8888) != 0, false);
        const unsigned own = rows.a[0].y;                        // the word itself: row 0 starts at its first bit
        if (first || word_touched(w, w.flags[par], p, k, n) || before) {
            unsigned any = 0u, tot;
            unsigned need = word_tables_at(w, raw, p, k + lane, in, rows, any);
            const unsigned live = __ballot_sync(0xFFFFFFFFu, any != 0u);
            if (lane == 0) w.live[un] = live;
            unsigned pos = word_scan((unsigned)__popc(need), tot);
            if (tot) {
                unsigned at = 0u;
                if (lane == 0) at = atomicAdd(&sm.queued, tot);
                at = __shfl_sync(0xFFFFFFFFu, at, 0);
                const int c0 = p * w.plane_cells + (k + lane) * 32;
                if (at + tot <= (unsigned)kWordEntries) {
                    for (pos += at; need; need &= need - 1u, ++pos) {
                        sm.t.cell[pos] = c0 + __ffs(need) - 1;
                        if (M) sm.t.inst[pos] = (unsigned char)inst;
                    }
                } else {
                    // the queue is full: its last places hold nothing, these
                    // entries are recomputed here
                    for (unsigned q = at + lane; q < (unsigned)kWordEntries; q += 32) sm.t.cell[q] = -1;
                    for (; need; need &= need - 1u) word_entry<K>(w, c0 + __ffs(need) - 1);
                }
            }
        }
        if (in) w.raw[par ^ 1][wd] = make_uint2(0u, own);
        if (lane == 0) w.flags[par ^ 1][un] = 0;
    }
    __syncthreads();
    const int n = (int)min(sm.queued, (unsigned)kWordEntries);
    for (int i = threadIdx.x; i < n; i += kWordThreads) {
        const int c = sm.t.cell[i];
        if (c >= 0) word_entry<K>(M ? insts[sm.t.inst[i]] : w0, c);
    }
}

// ---------------------------------------------------------------------------
// pass end and output
// ---------------------------------------------------------------------------

// After the relax phase of pass r (one thread of the grid): trace, counters,
// status.  `last`: the pass cap is reached and the frontier was only counted.
__device__ __forceinline__ void word_close(const WordInst& w, long long r, bool last) {
    WordCtr* k = w.ctr;
    const unsigned long long s = *(volatile unsigned long long*)&k->sums[r & 3];
    const unsigned long long f1 = s >> 32, nchg = s & 0xFFFFFFFFull;
    if (f1 == 0 || last) {
        k->done = 1;
        k->status = f1 == 0 ? BF_CONVERGED : (r >= w.g.C ? BF_NEG_CYCLE : BF_ITER_CAP);
        return;
    }
    if (w.trace && r < w.trace_cap) {
        long long* t = w.trace + r * 4;
        t[0] = (long long)f1;
        t[1] = (long long)nchg;
        t[2] = (long long)((f1 + 31) / 32);
        t[3] = -1;
    }
    k->total_relaxed += f1;
    k->total_changed += nchg;
    k->round = r + 1;
    k->sums[(r + 2) & 3] = 0ull;
    k->gate[(r + 2) & 3] = 0ull;
    if (nchg == 0) {
        k->done = 1;
        k->status = BF_CONVERGED;
    }
}

__device__ __forceinline__ void word_output(const WordInst& w) {
    for (long long c = blockIdx.x * (long long)kWordThreads + threadIdx.x; c < w.g.C;
         c += (long long)gridDim.x * kWordThreads)
        w.V[c] = val_of(w.Vnew[c]);
}

}  // namespace bfk
