// Internal types shared by the host driver and the kernels of the growth library.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace cg {

constexpr uint64_t kEmpty = ~0ull;   // empty hash slot: never a valid permutation key, n >= 2
constexpr int kMaxN = 16;            // permutations from the identity: 4 bits per element
constexpr int kMaxElems = 64;        // coset vectors: n elements of `width` bits, n * width <= 64
constexpr int kMaxTerms = 16;
constexpr int kMaxLayers = 16384;    // device layer-size array per job

// A generator acting on packed keys (element i in bits [w i, w i + w), w = 1, 2 or 4).
// kind 0, shift-and-mask form: the gather t[i] = s[g[i]] moves element g[i] to element i, a
// rotation of the key by w*(i - g[i]) bits; positions sharing one offset form one term:
// t = OR_t rotl(s, rot[t]) & mask[t].  Cyclic shifts need 2 terms, adjacent transpositions 3,
// any generator <= n, so every generator of n <= 16 elements.
// kind 1, the reversal of the element range [a, b], for long vectors where it would need more
// than kMaxTerms terms: the whole key is bit-reversed (elements land in reverse order, each
// with its bits reversed), the bits of every element put back in order, and the result shifted
// so that element e lands on a + b - e: t = (s & ~mask[0]) | (shift(rev(s), rev_shift) & mask[0]).
// Other generators of more than kMaxTerms offsets are not supported (CG_EINVAL at create).
//
// sel: permutations of n <= 16 elements (4 bits each) also as byte-permute selectors, for the
// kernels that hold a state as one byte per element (ByteState in cg_device.cuh): one prmt per
// output word for n <= 8, two for n <= 12, three for n <= 16, whatever the generator (the
// shift-and-mask form costs about ten instructions a term).  The inverse's tag sits in bits
// 28..31 of sel[0], above the selector bits prmt reads.  All zero for other vectors.
constexpr int kSelWords = 12;

struct GenSM {
    uint32_t nterms;
    uint32_t inv_tag;   // 1 + index of this generator's inverse in the set (< 15), or 0
    uint8_t kind;
    uint8_t width;      // bits per element
    int16_t rev_shift;  // kind 1: right shift (bits) of the reversed key; negative: left shift
    uint8_t rot[kMaxTerms];
    uint64_t mask[kMaxTerms];
    alignas(16) uint32_t sel[kSelWords];
    uint8_t map[16];    // the inverse, byte q = the i with g[i] = q: how a generator moves position q
};
static_assert(offsetof(GenSM, sel) % 16 == 0 && sizeof(GenSM) % 16 == 0, "GenSM: sel is read in 16-byte vectors");

// Where a state held as bytes keeps element p of n: word and byte (elements 0..7 alternate between
// words 0 and 1, which is how a packed key's nibbles fall apart under one mask; elements 8..11 are
// word 2, or, when n > 12, elements 8..15 alternate between words 2 and 3).
constexpr int byte_word(int n, int p) { return p < 8 ? (p & 1) : n <= 12 ? 2 : 2 + (p & 1); }
constexpr int byte_slot(int n, int p) { return p < 8 ? (p >> 1) : n <= 12 ? p - 8 : (p - 8) >> 1; }

// Byte-permute selectors of the gather t[i] = s[g[i]] on n <= 16 elements (GenSM::sel, without
// the tag).  Positions past n (zero bytes) stay where they are.
inline void make_selectors(const uint8_t* g, int n, uint32_t* sel) {
    for (int i = 0; i < kSelWords; ++i) sel[i] = 0;
    const int words = n <= 8 ? 2 : n <= 12 ? 3 : 4, elems = words * 4;
    for (int p = 0; p < elems; ++p) {
        const int q = p < n ? g[p] : p;
        const uint32_t o = (uint32_t)byte_word(n, p), b = (uint32_t)byte_slot(n, p);
        const uint32_t sw = (uint32_t)byte_word(n, q), sb = (uint32_t)byte_slot(n, q);
        if (words == 2) {
            sel[o] |= (sw * 4 + sb) << (4 * b);
        } else if (words == 3) {        // from words 0, 1; then from that and word 2
            sel[2 * o] |= (sw < 2 ? sw * 4 + sb : 0) << (4 * b);
            sel[2 * o + 1] |= (sw < 2 ? b : 4 + sb) << (4 * b);
        } else {                        // from words 0, 1; from words 2, 3; then from both
            sel[3 * o] |= (sw < 2 ? sw * 4 + sb : 0) << (4 * b);
            sel[3 * o + 1] |= (sw >= 2 ? (sw - 2) * 4 + sb : 0) << (4 * b);
            sel[3 * o + 2] |= (sw < 2 ? b : 4 + b) << (4 * b);
        }
    }
}

// Keys of more than 64 bits (two words): vectors of n elements of w bits with 64 < n w <= 128 --
// coset vectors of 4-bit values up to n = 32, 2-bit up to 64, 1-bit up to 128, and permutations
// of 17..25 elements from the identity with 5-bit elements.  Element i occupies bits
// [w i, w i + w) of the 128-bit number hi:lo.
struct alignas(16) Key128 {
    uint64_t lo, hi;
};

constexpr int kMaxWideElems = 128;
constexpr int kMaxWideTerms = 32;

// A generator acting on two-word keys: kind 0 is the shift-and-mask form over 128 bits (one term
// per distinct element offset, at most kMaxWideTerms); kind 1 the reversal of the element range
// covered by mask (bit-reverse the 128-bit key, put each element's bits back in order, shift by
// rev_shift bits: right if positive).
struct WideGen {
    uint32_t nterms;
    uint32_t inv_tag;   // 1 + index of the inverse (< 15), or 0
    uint8_t kind;
    uint8_t width;
    int16_t rev_shift;
    uint8_t rot[kMaxWideTerms];
    uint64_t mlo[kMaxWideTerms];
    uint64_t mhi[kMaxWideTerms];
};

// Ranking of a start vector's arrangements (wide_rank in wide_path.cu): `steps` steps of `bits` key
// bits, `states` rows of 1 << bits words a step.  table: 1 << bits count increments, then the rows.
// steps = 0: none.
constexpr int kWideRankWords = 12288;       // at most 48 KB
struct WideRank {
    const uint32_t* table;
    int steps, bits, states, words;
};

// One growth with two-word keys (hash strategy): every layer back to back in `keys`, the visited
// set an open-addressing table of 16-byte slots (empty = all ones).  A state found by generator g
// carries the tag (1 + index of g's inverse) in bits 124-127 when n w <= 124.
struct alignas(128) WideDev {
    Key128* keys;
    uint64_t keys_cap;
    Key128* table;
    uint64_t table_mask;
    const WideGen* gens;
    uint64_t* layer_sizes;
    uint64_t stop_above;
    Key128 start;
    int k;
    int n;
    int layers_cap;
    int max_radius;
    int tagged;
    int pad0;
    alignas(128) unsigned long long lo;     // frontier = keys[lo, hi)
    unsigned long long hi;
    unsigned long long tail;
    int radius;
    int status;
    int overflow;
    int pad1;
};

// States found by generator j are stored with tag (1 + index of j's inverse) in key bits 60-63
// when the key leaves them free (n * width <= 60): that inverse leads back to the state's
// parent, in the previous layer, so the expansion skips it.  The visited set always holds
// untagged keys.
constexpr uint64_t kKeyBits60 = (1ull << 60) - 1;

constexpr int kVisitHash = 0;
constexpr int kVisitBitmap = 2;
constexpr int kVisitComb = 3;           // bitmap over the C(n, m) binary vectors (comb_rank)
constexpr int kVariantBitmap = 17;      // kernel variants of the rank bitmap (one form, whatever CG_OPT_ILP says)
constexpr int kVariantComb = 21;        // and of the arrangement bitmap
constexpr int kCombMaxWords = 6144;     // ranking table: at most 96 rows of 64

// Generators beyond the parent edge from which a single rank-bitmap job's first round reads a visited
// word before its atomic (later rounds, and those of several jobs, go by the last round's yield: see
// bitmap_test_first and job_reads_first in hash_path.cu).
constexpr int kTestMinDegree = 4;

enum JobStatus : int {
    kRunning = 0,
    kDone = 1,          // empty next layer: growth complete
    kTruncRadius = 2,   // reached max_radius (or the layer array's capacity)
    kTruncAbove = 3,    // recorded the first layer larger than stop_above
    kNeedMem = 4,       // the layer being built did not fit; layers up to `radius` are exact
    kDeviceError = 5,
    kFresh = 6,         // admitted, not yet initialised (the next init launch sets it up)
    kEmptySlot = 7,     // no job in this slot
};

// One growth job of the hash strategy as the persistent kernel sees it.
// 256 bytes: the read-only fields fill the first 128-byte line, the fields updated during a
// run (read by every SM, bumped with atomics) live alone in the second.
struct alignas(128) JobDev {
    // static, written by the host
    uint64_t* keys;            // all layers back to back; layer r = keys[off_r, off_{r+1})
    uint64_t keys_cap;
    uint64_t* table;           // visited set, table_mask + 1 slots
    uint64_t table_mask;
    const GenSM* gens;         // k entries
    uint64_t* layer_sizes;     // device, layers_cap entries; [0] = 1
    uint64_t stop_above;       // 0: none
    int k;
    int n;
    int layers_cap;
    int max_radius;            // < 0: unlimited
    int mode;                  // visited set: 0 hash table, 2 rank bitmap (kVisitBitmap)
    int use_start;             // 1: grow from start_key (a central state), 0: from the identity
    uint64_t start_key;        // packed start vector when use_start
    int tagged;                // 1: keys leave bits 60-63 free for the parent-edge tag
    int closed;                // 1: every generator's inverse is in the set (every state but
                               //    the start carries a parent-edge tag)
    int test;                  // rank bitmap, one job: the launch's first round reads visited
                               //    words before its atomics (later rounds decide themselves)
    int ones;                  // kVisitComb: ones of a vector (< 0: zeros), ranking table and its words
    const uint32_t* comb;
    int comb_words;
    // dynamic, updated between rounds by block 0
    alignas(128) unsigned long long lo;     // frontier = keys[lo, hi)
    unsigned long long hi;
    unsigned long long tail;   // append cursor (atomic during a round)
    int radius;                // radius of the frontier layer
    int status;                // JobStatus
    int overflow;              // set during a round: keys or table ran out
    int reads_first;           // rank bitmap, one of several jobs: this round reads visited words
                               //    before its atomics
};
// The round close loads (lo, hi) and (tail, radius | status << 32) as two 16-byte vectors.
static_assert(offsetof(JobDev, lo) % 16 == 0 && offsetof(JobDev, hi) == offsetof(JobDev, lo) + 8,
              "JobDev: lo, hi must form one aligned 16-byte vector");
static_assert(offsetof(JobDev, tail) % 16 == 0 && offsetof(JobDev, radius) == offsetof(JobDev, tail) + 8 &&
                  offsetof(JobDev, status) == offsetof(JobDev, radius) + 4,
              "JobDev: tail, radius, status must form one aligned 16-byte vector");

// One growth of the sweep strategy: the visited set and two layers are bitmaps over the
// position-major Lehmer ranks 0..n!-1 (one bit per element of S_n each: 3 bits per element, as in
// the bitmask BFS of Section 3.1.3).  Layer r lives in F[r & 1]; its nonempty 1024-rank blocks
// (32 words of F) are listed, once each, in L[r & 1][0, lcount[r & 1]); S[r & 1] has one bit per
// block and is what makes a block's entry in the list unique.  Round r first clears layer r - 1
// (the other bitmap, its listed blocks) and then writes layer r + 1 there.
struct alignas(128) SweepDev {
    // static, written by the host
    unsigned* V;               // visited
    unsigned* F[2];            // layer r in F[r & 1]; the other holds layer r-1, then r+1
    unsigned* S[2];            // per-block bits of F (one bit per 32 words)
    unsigned* L[2];            // nonempty blocks of F (block index = rank >> 10)
    const GenSM* gens;         // k entries
    uint64_t* layer_sizes;     // layers_cap entries; [0] = 1
    uint64_t nblocks;          // 1024-rank blocks: every F has 32 * nblocks words
    uint64_t stop_above;       // 0: none
    uint64_t start_rank;       // rank of the start state
    int k;
    int n;
    int layers_cap;
    int max_radius;            // < 0: unlimited
    // dynamic, updated during a run
    alignas(128) unsigned long long grab;   // next work item of the round
    unsigned long long fresh;               // states found in the round
    unsigned long long lcount[2];           // entries of L[i]
    int radius;                // radius of the frontier layer
    int status;                // JobStatus
};

// One growth in blocks of 2^M states that the generators move together (block_path.cu): the visited
// set and three layers, one bit per element of S_n each, as one word per block; layer r lives in
// N[r % 3].  flag[i][g] is nonzero when one of the blocks 32 g .. 32 g + 31 may have bits in N[i].
constexpr int block_pairs(int n) { return n >= 12 ? 6 : n / 2; }
constexpr int kBlockMinN = 10, kBlockMaxN = 14;
constexpr int kBlockSmemGens = 128;
struct alignas(128) BlockDev {
    // static, written by the host
    void* V;                   // 64-bit words for M = 6, 32-bit words for M = 5
    void* N[3];
    unsigned char* flag[3];
    uint2* top;                // unranking tables (block_tables_kernel)
    unsigned* bottom;
    const uint4* maps;         // k generators: byte q = the position that position q's value goes to
    uint64_t* layer_sizes;     // layers_cap entries; [0] = 1
    uint64_t stop_above;       // 0: none
    uint64_t start;            // the start state's packed key
    uint64_t max_states;       // > 0: a layer that takes the states past this ends the growth (kNeedMem)
    unsigned nblocks, ngroups, ntop;
    int k, n;
    int layers_cap;
    int max_radius;            // < 0: unlimited
    // dynamic, updated during a run
    alignas(128) unsigned long long fresh;  // states found in the round
    unsigned long long states;              // states of the layers so far
    int radius;                // radius of the frontier layer
    int status;                // JobStatus
};

// Growths of S_n, n <= kClusterMaxN, one thread-block cluster each (block_path.cu).  Of a JobDev the
// kernel reads gens (GenSM::map), k, n, layer_sizes, layers_cap, max_radius, stop_above and keys_cap
// (the states the job may hold) and writes layer_sizes, radius and status.
struct Ctl;
constexpr int kClusterMaxN = 10;
constexpr int kClusterSmemN = 8;            // up to this n one block each, all in its shared memory
constexpr int kClusterGens = 64;            // generators kept in shared memory
struct ClusterArgs {
    JobDev* jobs;                           // in the order they are taken
    int first, njobs;                       // cluster_grow_kernel: [0, njobs); the small kernel: [first, njobs)
    unsigned* words;                        // per cluster `stride` words: visited and three layers
    uint64_t stride;
    const uint64_t* table[kClusterMaxN + 1];    // unranking tables (cluster_grow_kernel)
    uint64_t* last;                         // one job in shared memory: receives the last layer's keys (n! fit), or null
    uint64_t start;                         // the start state's packed key, for `last`
    Ctl* ctl;                               // zeroed: total_units and dyn_next, the two queues; err
};

// Admission of many jobs into one persistent launch (a batch): the jobs are grown in index
// order, at most max_active at a time and with the visited sets of the active jobs summing to at
// most `window` bytes, so that their random accesses stay in L2.  Whenever jobs end, the block
// that closes the round admits the next ones and sets them up; a job whose visited set alone
// exceeds the window is counted as 0 (it misses L2 wherever it runs).
struct AdmitDev {
    int* act[2];               // active job indices, double-buffered (Ctl::adm.act_sel selects)
    const uint64_t* vis;       // per job: visited-set bytes counted against `window`
    uint64_t window;
    int max_active;            // capacity of each act[]; the unit table holds max_active + 1
    int njobs;
    int unit_mult;             // frontier states per warp work unit: 32 * unit_mult
    int pad;
};

// Control block of the persistent kernel (device memory, zero-initialised by the host).
// The counter on which blocks arrive at the grid barrier and the generation word that waiting blocks
// poll sit in their own 128-byte lines, so arrivals and polling do not queue at one L2 slice.
constexpr int kGenBits = 20;
constexpr unsigned long long kGenMask = (1ull << kGenBits) - 1;

struct alignas(128) Ctl {
    unsigned int bar_count;
    unsigned int pad0[31];
    // Barrier word: the low kGenBits bits count the barriers completed in this launch; the rest
    // is a payload the releasing block hands to every block (for a single job: the size of the
    // next frontier, 0 when the growth stops).
    unsigned long long bar_word;
    unsigned int pad1[30];
    int err;                        // 0, or a CG_E* code set by a kernel
    int rounds;                     // rounds completed
    unsigned long long total_units; // warp work units of the current round
    unsigned int pad2[28];
    // A round's units split into a static part, in equal contiguous ranges per block, and the
    // second half, which blocks that finish their range draw from this counter.
    unsigned long long dyn_next;
    unsigned int pad3[30];
    // Admission of a batch into one launch (AdmitDev), updated by the block that closes a round.
    struct alignas(128) Admit {
        int act_sel;                    // AdmitDev::act[act_sel] lists the active jobs
        int nactive;
        unsigned long long next_admit;  // next job index to admit
        unsigned long long vis_used;    // counted visited-set bytes of the active jobs
    } adm;
};

}  // namespace cg
