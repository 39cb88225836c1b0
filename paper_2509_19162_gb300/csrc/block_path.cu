// Bitmask BFS in blocks of states that every generator moves together (the sweep strategy for
// whole growths of S_10 .. S_14).
//
// The graph has the symmetries s -> sigma s (relabelling the values): generators act on positions,
// (sigma s) g = sigma (s g).  Take for sigma the 2^M products of the swaps of the values (0 1),
// (2 3), .. (2M-2 2M-1): they cut S_n into blocks of 2^M states, and a generator sends block to
// block, state by state.  So one expansion serves all states of a block that lie in the layer.
//
// States are held as their inverses p = s^-1 (p_v = the position of value v), on which a generator
// acts element by element: p_v -> h[p_v], h = g^-1.  A block is p up to the order inside the pairs
// {p_0, p_1}, {p_2, p_3}, ..; its canonical member has every pair ascending, and bit e of the
// block's word is the member whose pair i is swapped where bit i of e is set.  The image of member e
// is member e ^ m of the image block, m_i = the generator swaps the order of the canonical pair i:
// a permutation of the word's bits by an exclusive or, log2 steps.
//
// Index of a block: mixed radix from the top value down, one digit per single value (its place among
// the positions not yet taken: v + 1 choices for value v >= 2M) and one per pair (C(2i+2, 2) choices
// for pair i).  Generators act on p elementwise, so the blocks that agree in their top digits go to
// blocks that agree in theirs: whatever the generators, the grid, working through the blocks in
// index order, writes into k stretches of the visited set that it also walks through in order.
// That is what keeps a visited set larger than L2 (n >= 13) out of DRAM's random-access rate.
//
// A growth from another state s0 is the identity's with s0's values in the export.  Which values are
// paired matters: members of a block are expanded together when they lie in the same layer, and under
// adjacent transpositions swapping two neighbouring values changes the distance from the identity by
// one (S_12: 5.9 ms; 13.0 ms with the pairs of a random relabelling).
//
// Data: visited words V, and words N[3] of the layers r, r + 1 and r - 1 (the last one cleared
// during round r, so that it can take layer r + 2), four bits per element of S_n, and one byte per
// 32 blocks and layer that says whether any of them is set.  One round of the persistent launch:
// every warp takes groups of 32 blocks, warp w groups w, w + W, ..; the nonempty blocks go through a
// queue in shared memory so that 32 of them are expanded at a time, one per lane.
//
// Measured against the state-by-state rank bitmap and sweep kernels it takes the place of: see
// block_preferred in host_api.cu.
#include <cooperative_groups.h>
#include <cstdio>
#include <type_traits>
#include <utility>

#include "cg_device.cuh"
#include "cg_kernels.h"

namespace cg {

namespace {

constexpr int kBlkThreads = 256;
constexpr int kBlkWarps = kBlkThreads / 32;
constexpr int kBlkQueue = 64;          // queued blocks per warp, and claims per warp
constexpr int kPairBlocks = 8;         // at most this many blocks are expanded a lane per pair
constexpr unsigned kBottom = 2520;     // arrangements of the pairs 0..3 among eight positions

constexpr unsigned block_count(int n) {
    unsigned long long f = 1;
    for (int i = 2; i <= n; ++i) f *= (unsigned long long)i;
    return (unsigned)(f >> block_pairs(n));
}

template <int N>
struct BlockShape {
    static constexpr int M = block_pairs(N);
    using Word = std::conditional_t<M == 6, unsigned long long, unsigned>;
    static constexpr int kWords = (N + 3) / 4;       // four elements of p per 32-bit word
};

// ---- the pieces of one expansion ---------------------------------------------------------------
// A block's canonical p, ready to be looked up: four elements per word as prmt selectors (their low
// three bits, one nibble each) and the bytes whose element is 8 or more.
template <int N>
struct BlockPerm {
    uint32_t sel[BlockShape<N>::kWords];
    uint32_t high[BlockShape<N>::kWords];
};

__device__ __forceinline__ void lookup_form(uint32_t nibbles, uint32_t& sel, uint32_t& high) {
    sel = nibbles & 0x7777u;
    // nibble j's bit 3 to the sign of byte j, then spread over the byte
    const uint32_t b = ((nibbles & 0x00FFu) | (nibbles & 0xFF00u) << 8);
    const uint32_t c = ((b & 0x000F000Fu) << 4) | ((b & 0x00F000F0u) << 8);
    // (prmt's sign mode: __byte_perm documents three selector bits only)
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(high) : "r"(c), "r"(0u), "r"(0xBA98u));
}

template <int N>
__device__ __forceinline__ BlockPerm<N> block_unrank(const uint2* __restrict__ tops, const unsigned* __restrict__ bottoms,
                                                     unsigned idx) {
    BlockPerm<N> P;
    const unsigned t = idx / kBottom;
    const uint2 top = __ldg(tops + t);                         // p_8.. as nibbles, the rest ascending
    const unsigned low = __ldg(bottoms + (idx - t * kBottom));     // p_0..p_7 as indices into the rest
    const unsigned r0 = top.y & 0x0F0F0F0Fu, r1 = (top.y >> 4) & 0x0F0F0F0Fu;
    // r0: elements 0 2 4 6 of the rest, r1: 1 3 5 7; the table's indices are in that byte order
    const unsigned a = __byte_perm(r0, r1, low), b = __byte_perm(r0, r1, low >> 16);
    const unsigned na = __byte_perm(a | (a >> 4), 0, 0x4420u), nb = __byte_perm(b | (b >> 4), 0, 0x4420u);
    lookup_form(na, P.sel[0], P.high[0]);
    lookup_form(nb, P.sel[1], P.high[1]);
    lookup_form(top.x & 0xFFFFu, P.sel[2], P.high[2]);
    if constexpr (N > 12) lookup_form(top.x >> 16, P.sel[3], P.high[3]);
    return P;
}

// h[p], four elements per word, one byte each.
template <int N>
__device__ __forceinline__ void block_map(const uint4& h, const BlockPerm<N>& P, uint32_t (&q)[BlockShape<N>::kWords]) {
#pragma unroll
    for (int i = 0; i < BlockShape<N>::kWords; ++i) {
        const uint32_t a = __byte_perm(h.x, h.y, P.sel[i]), b = __byte_perm(h.z, h.w, P.sel[i]);
        q[i] = (a & ~P.high[i]) | (b & P.high[i]);
    }
}

template <int N>
__device__ __forceinline__ unsigned element(const uint32_t (&q)[BlockShape<N>::kWords], int v) {
    return __byte_perm(q[v >> 2], 0, 0x4440u | (unsigned)(v & 3));
}

// Index of q's block and the pairs that q has in descending order.  As in rank_bytes: with the
// positions taken so far in bits 0..15 of `taken` and ones above them, the arithmetic shift
// taken >> x holds 16 + x + #{taken > x} ones, which is x's place among the free positions plus a
// constant.
template <int N>
__device__ __forceinline__ unsigned block_rank(const uint32_t (&q)[BlockShape<N>::kWords], unsigned& m) {
    constexpr int M = BlockShape<N>::M;
    int taken = (int)0xFFFF0000u;
    unsigned idx = 0;
    m = 0;
#pragma unroll
    for (int v = N - 1; v >= 2 * M; --v) {
        const unsigned x = element<N>(q, v);
        const unsigned c = 16u + (unsigned)(N - 1 - v);
        const unsigned d = v == N - 1 ? x : (unsigned)__popc((unsigned)(taken >> x)) - c;
        idx = idx * (unsigned)(v + 1) + d;
        taken |= 1 << x;
    }
#pragma unroll
    for (int i = M - 1; i >= 1; --i) {
        const unsigned x = element<N>(q, 2 * i), y = element<N>(q, 2 * i + 1);
        const bool first = N == 2 * M && i == M - 1;        // nothing taken yet
        const unsigned c = 16u + (unsigned)(N - 2 - 2 * i);
        const unsigned dx = first ? x : (unsigned)__popc((unsigned)(taken >> x)) - c;
        const unsigned dy = first ? y : (unsigned)__popc((unsigned)(taken >> y)) - c;
        const unsigned lo = min(dx, dy), hi = max(dx, dy);
        idx = idx * (unsigned)((2 * i + 2) * (2 * i + 1) / 2) + (hi * (hi - 1u)) / 2u + lo;
        m |= x > y ? 1u << i : 0u;
        taken |= (1 << x) | (1 << y);
    }
    m |= element<N>(q, 0) > element<N>(q, 1) ? 1u : 0u;
    return idx;
}

// Bit e of the result is bit e ^ m of f.
__device__ __forceinline__ unsigned xor_bits32(unsigned f, unsigned m) {
    const unsigned m1 = (m & 1u) ? 0x55555555u : 0u, m2 = (m & 2u) ? 0x33333333u : 0u, m4 = (m & 4u) ? 0x0F0F0F0Fu : 0u;
    unsigned t = (f ^ (f >> 1)) & m1;
    f ^= t ^ (t << 1);
    t = (f ^ (f >> 2)) & m2;
    f ^= t ^ (t << 2);
    t = (f ^ (f >> 4)) & m4;
    f ^= t ^ (t << 4);
    return __byte_perm(f, 0, 0x3210u ^ ((m >> 3) & 3u) * 0x1111u);
}
__device__ __forceinline__ unsigned xor_bits(unsigned f, unsigned m) { return xor_bits32(f, m); }
__device__ __forceinline__ unsigned long long xor_bits(unsigned long long f, unsigned m) {
    const unsigned lo = xor_bits32((unsigned)f, m), hi = xor_bits32((unsigned)(f >> 32), m);
    return (m & 32u) ? ((unsigned long long)lo << 32 | hi) : ((unsigned long long)hi << 32 | lo);
}

__device__ __forceinline__ int popc_word(unsigned w) { return __popc(w); }
__device__ __forceinline__ int popc_word(unsigned long long w) { return __popcll(w); }

// A visited word, possibly from this SM's L1: bits are only ever set during a launch, so a set bit
// is the truth and a stale clear one is caught by the atomicOr that follows.
__device__ __forceinline__ unsigned ld_visited(const unsigned* p) {
    unsigned v;
    asm volatile("ld.relaxed.cta.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned long long ld_visited(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.cta.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

// ---- tables, start ---------------------------------------------------------------------------------
// Canonical arrangement number `b` of the pairs 0..npairs-1 among 2 npairs places, as it is ranked:
// pair npairs-1 first.  place[v] receives value v's place (0..2 npairs - 1).
__device__ void arrange_pairs(unsigned b, int npairs, unsigned char* place) {
    unsigned char free_[16];
    for (int i = 0; i < 2 * npairs; ++i) free_[i] = (unsigned char)i;
    unsigned digit[8];
    for (int i = 0; i < npairs; ++i) {                 // radix of pair i: C(2i+2, 2)
        const unsigned radix = (unsigned)((2 * i + 2) * (2 * i + 1) / 2);
        digit[i] = b % radix;
        b /= radix;
    }
    for (int i = npairs - 1; i >= 0; --i) {
        unsigned hi = 1;
        while (hi * (hi + 1) / 2 <= digit[i]) ++hi;
        const unsigned lo = digit[i] - hi * (hi - 1) / 2;
        place[2 * i] = free_[lo];
        place[2 * i + 1] = free_[hi];
        int n = 0;
        for (int j = 0; j < 2 * i + 2; ++j)
            if (j != (int)lo && j != (int)hi) free_[n++] = free_[j];
    }
}

// Fills D.top (the values 8..n-1: nibbles of their positions, and the free positions ascending) and
// D.bottom (the values 0..7: nibbles of their index into the free positions, as prmt selectors for
// the free positions' even and odd halves).
__global__ void block_tables_kernel(BlockDev D) {
    const unsigned i0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
    const int n = D.n, M = block_pairs(n);
    for (unsigned b = i0; b < kBottom; b += step) {
        unsigned char place[16];
        arrange_pairs(b, 4, place);
        unsigned w = 0;
        for (int v = 0; v < 8; ++v) {
            const unsigned j = place[v];               // free position j sits in half j & 1, byte j >> 1
            w |= (((j & 1u) << 2) | (j >> 1)) << (4 * v);
        }
        D.bottom[b] = w;
    }
    for (unsigned t = i0; t < D.ntop; t += step) {
        unsigned digit[16];
        unsigned x = t;
        for (int i = 4; i < M; ++i) {                  // pairs above 3, then the singles
            const unsigned radix = (unsigned)((2 * i + 2) * (2 * i + 1) / 2);
            digit[i] = x % radix;
            x /= radix;
        }
        unsigned single[16];
        for (int v = 2 * M; v < n; ++v) {
            single[v] = x % (unsigned)(v + 1);
            x /= (unsigned)(v + 1);
        }
        unsigned char free_[16];
        for (int i = 0; i < n; ++i) free_[i] = (unsigned char)i;
        unsigned pos[16];
        int left = n;
        for (int v = n - 1; v >= 2 * M; --v) {
            const unsigned d = single[v];
            pos[v] = free_[d];
            for (int j = (int)d; j + 1 < left; ++j) free_[j] = free_[j + 1];
            --left;
        }
        for (int i = M - 1; i >= 4; --i) {
            unsigned hi = 1;
            while (hi * (hi + 1) / 2 <= digit[i]) ++hi;
            const unsigned lo = digit[i] - hi * (hi - 1) / 2;
            pos[2 * i] = free_[lo];
            pos[2 * i + 1] = free_[hi];
            int c = 0;
            for (int j = 0; j < left; ++j)
                if (j != (int)lo && j != (int)hi) free_[c++] = free_[j];
            left = c;
        }
        uint2 e = make_uint2(0u, 0u);
        for (int v = 8; v < n; ++v) e.x |= pos[v] << (4 * (v - 8));
        for (int j = 0; j < 8; ++j) e.y |= (unsigned)free_[j] << (4 * j);
        D.top[t] = e;
    }
}

template <int N>
__global__ void block_init_kernel(BlockDev* Dp) {
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    using Word = typename BlockShape<N>::Word;
    BlockDev& D = *Dp;
    uint32_t q[BlockShape<N>::kWords] = {};
    for (int v = 0; v < N; ++v) q[v >> 2] |= (uint32_t)v << (8 * (v & 3));      // the identity
    unsigned m = 0;
    const unsigned idx = block_rank<N>(q, m);
    if (idx >= D.nblocks) { D.status = kDeviceError; return; }
    static_cast<Word*>(D.V)[idx] = (Word)1 << m;
    static_cast<Word*>(D.N[0])[idx] = (Word)1 << m;
    D.flag[0][idx >> 5] = 1;
    D.layer_sizes[0] = 1;
    D.fresh = 0;
    D.states = 1;
    D.radius = 0;
    D.status = D.max_radius == 0 ? kTruncRadius : kRunning;
}

// The stored states of a key-list growth: keys[0, hi), of which keys[lo, hi) are layer D.radius, set in
// the (cleared) visited words and that layer's words.  A stored key s = s0 w gives w^-1: the place i
// of s0's value v in s is the place of v in w.
template <int N>
__global__ void block_import_kernel(BlockDev* Dp, const uint64_t* __restrict__ keys, unsigned long long lo,
                                    unsigned long long hi, int* err) {
    using Word = typename BlockShape<N>::Word;
    const BlockDev& D = *Dp;
    const int which = D.radius % 3;
    Word* V = static_cast<Word*>(D.V);
    Word* F = static_cast<Word*>(D.N[which]);
    unsigned char* flag = D.flag[which];
    uint64_t place = 0;                                // nibble x: the v with s0[v] = x
    for (int v = 0; v < N; ++v) place |= (uint64_t)v << (4 * ((D.start >> (4 * v)) & 15u));
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < hi; i += step) {
        const uint64_t s = __ldcg(keys + i);
        uint64_t inv = 0;                              // nibble v: position of v in w
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const unsigned v = (unsigned)(place >> (4 * ((unsigned)(s >> (4 * j)) & 15u))) & 15u;
            inv |= (uint64_t)j << (4 * v);
        }
        uint32_t q[BlockShape<N>::kWords] = {};
#pragma unroll
        for (int v = 0; v < N; ++v) q[v >> 2] |= (uint32_t)((inv >> (4 * v)) & 15u) << (8 * (v & 3));
        unsigned m;
        const unsigned idx = block_rank<N>(q, m);
        if (idx >= D.nblocks) {                        // not a permutation: never expected
            atomicExch(err, CG_EDEVICE);
            continue;
        }
        atomicOr(V + idx, (Word)1 << m);
        if (i >= lo) {
            atomicOr(F + idx, (Word)1 << m);
            flag[idx >> 5] = 1;
        }
    }
}

// ---- the persistent kernel ---------------------------------------------------------------------------
// Close a round (one thread of the last block to arrive).
__device__ void block_close(BlockDev& D, Ctl* ctl) {
    volatile BlockDev& W = D;
    const unsigned long long fresh = ld_relaxed_ull(&D.fresh);
    if (fresh == 0) {
        W.status = kDone;
    } else if (D.max_states > 0 && W.states + fresh > D.max_states) {
        W.status = kNeedMem;                // the layer is past the states the job may keep
    } else {
        const int r1 = W.radius + 1;
        W.states = W.states + fresh;
        D.layer_sizes[r1] = fresh;
        W.radius = r1;
        if (D.max_radius >= 0 && r1 >= D.max_radius) W.status = kTruncRadius;
        else if (D.stop_above > 0 && fresh > D.stop_above) W.status = kTruncAbove;
        else if (r1 + 1 >= D.layers_cap) W.status = kTruncRadius;
    }
    W.fresh = 0;
    *(volatile int*)&ctl->rounds += 1;
    __threadfence();
}

// Bound by issue and the latency of what is left between (S_12 pancake: 2.18 G warp instructions, issue
// slots 50 % busy, DRAM at 11 % of its rate, 64 % of L2 accesses hit): four blocks an SM at 64 registers
// are faster than three at 77 (S_12 pancake 3.27 / 3.52 ms, S_13 pancake 47.3 / 51.9 ms).
template <int N>
__global__ void __launch_bounds__(kBlkThreads, 4)
block_grow_kernel(BlockDev* Dp, Ctl* ctl, int max_rounds, uint64_t timeout_ns) {
    using Word = typename BlockShape<N>::Word;
    __shared__ uint4 s_map[kBlockSmemGens];
    __shared__ unsigned s_qidx[kBlkWarps][kBlkQueue];
    __shared__ Word s_qf[kBlkWarps][kBlkQueue];
    __shared__ unsigned s_cidx[kBlkWarps][kBlkQueue];
    __shared__ Word s_cf[kBlkWarps][kBlkQueue];
    __shared__ unsigned long long s_fresh;
    const BlockDev& D = *Dp;
    const int k = D.k;
    const unsigned nblocks = D.nblocks, ngroups = D.ngroups;
    const uint2* tops = D.top;
    const unsigned* bottoms = D.bottom;
    const uint4* maps = D.maps;
    if (k <= kBlockSmemGens) {
        for (int j = threadIdx.x; j < k; j += blockDim.x) s_map[j] = D.maps[j];
        maps = s_map;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned* qidx = s_qidx[wid];
    Word* qf = s_qf[wid];
    unsigned* cidx = s_cidx[wid];
    Word* cf = s_cf[wid];
    Word* V = static_cast<Word*>(D.V);
    const unsigned W = gridDim.x * kBlkWarps, w = blockIdx.x + gridDim.x * wid;

    unsigned nbar = 0;                      // grid barriers this block has passed
    for (int round = 0; round < max_rounds; ++round) {
        if (ld_relaxed_int(&Dp->status) != kRunning) break;
        const int r = ld_relaxed_int(&Dp->radius);
        const int cur = r % 3, nxt = (r + 1) % 3, old = (r + 2) % 3;
        const Word* F = static_cast<const Word*>(D.N[cur]);
        Word* X = static_cast<Word*>(D.N[nxt]);
        Word* O = static_cast<Word*>(D.N[old]);
        const unsigned char* fcur = D.flag[cur];
        unsigned char* fnxt = D.flag[nxt];
        unsigned char* fold = D.flag[old];
        if (threadIdx.x == 0) s_fresh = 0;
        __syncthreads();

        unsigned fresh = 0;                 // states this lane found (flushed before it can wrap)
        unsigned long long found = 0;
        int qn = 0, cn = 0;                 // queued blocks, pending claims
        unsigned pidx = 0;                  // the candidate whose visited word is on its way
        Word pf = 0, pv = 0;

        // Claim the last `take` pending candidates; the bits this claim sets are new.
        auto claim = [&](int take) {
            cn -= take;
            if (lane < take) {
                const unsigned i = cidx[cn + lane];
                const Word f = cf[cn + lane];
                const Word neu = f & ~(Word)atomicOr(V + i, f);
                if (neu) {
                    fresh += popc_word(neu);
                    if (atomicOr(X + i, neu) == 0) fnxt[i >> 5] = 1;
                }
            }
            __syncwarp();
        };
        auto settle = [&]() {
            const Word neu = pf & ~pv;
            const unsigned b = __ballot_sync(0xffffffffu, neu != 0);
            if (b == 0) return;
            if (neu) {
                const int at = cn + __popc(b & lanemask_lt());
                cidx[at] = pidx;
                cf[at] = neu;
            }
            cn += __popc(b);
            __syncwarp();
            if (cn >= 32) claim(32);
        };
        // Expand the last `take` queued blocks, one per lane.
        auto expand = [&](int take) {
            qn -= take;
            const bool active = lane < take;
            const unsigned idx = active ? qidx[qn + lane] : 0u;
            const Word f = active ? qf[qn + lane] : (Word)0;
            __syncwarp();
            const BlockPerm<N> P = block_unrank<N>(tops, bottoms, idx);
            for (int g = 0; g < k; ++g) {
                uint32_t q[BlockShape<N>::kWords];
                block_map<N>(maps[g], P, q);
                unsigned m;
                const unsigned i = block_rank<N>(q, m);
                const Word t = xor_bits(f, m);
                // (the index of a permutation is below nblocks; a violated invariant is reported and
                // touches nothing)
                const bool live = active && i < nblocks;
                if (active && !live) atomicCAS(&ctl->err, 0, CG_EDEVICE);
                Word v = 0;
                if (live) v = ld_visited(V + i);
                settle();
                pidx = i;
                pf = live ? t : (Word)0;
                pv = v;
            }
            if (fresh >> 30) { found += fresh; fresh = 0; }
        };

        // the warp's groups, 32 at a time: which hold blocks of this layer, which of the layer to clear
        for (unsigned base = w; base < ngroups; base += 32u * W) {
            const unsigned long long mine = (unsigned long long)base + (unsigned long long)lane * W;
            const bool in = mine < ngroups;
            unsigned dirty = __ballot_sync(0xffffffffu, in && __ldcg(fcur + mine) != 0);
            unsigned stale = __ballot_sync(0xffffffffu, in && __ldcg(fold + mine) != 0);
            while (stale) {
                const int l = __ffs(stale) - 1;
                stale &= stale - 1;
                const unsigned g = base + (unsigned)l * W;
                const unsigned b = g * 32u + lane;
                if (b < nblocks) O[b] = 0;
                if (lane == 0) fold[g] = 0;
            }
            while (dirty) {
                const int l = __ffs(dirty) - 1;
                dirty &= dirty - 1;
                const unsigned b = (base + (unsigned)l * W) * 32u + lane;
                const Word f = b < nblocks ? __ldcg(F + b) : (Word)0;
                const unsigned have = __ballot_sync(0xffffffffu, f != 0);
                if (f) {
                    const int at = qn + __popc(have & lanemask_lt());
                    qidx[at] = b;
                    qf[at] = f;
                }
                qn += __popc(have);
                __syncwarp();
                if (qn >= 32) expand(32);
            }
            if (32ull * W + base > 0xffffffffull) break;
        }
        if (qn > kPairBlocks) expand(qn);
        settle();
        pf = 0;
        // a short remainder, a lane per (block, generator) pair (as in cluster_grow)
        for (int first = 0; first < qn * k; first += 32) {
            const int pair = first + lane;
            const bool live = pair < qn * k;
            const int b = live ? pair / k : 0, g = live ? pair - b * k : 0;
            const BlockPerm<N> P = block_unrank<N>(tops, bottoms, live ? qidx[b] : 0u);
            uint32_t q[BlockShape<N>::kWords];
            block_map<N>(maps[g], P, q);
            unsigned m;
            const unsigned i = block_rank<N>(q, m);
            if (live && i < nblocks) {
                const Word f = xor_bits(qf[b], m);
                const Word neu = f & ~(Word)atomicOr(V + i, f);
                if (neu) {
                    fresh += popc_word(neu);
                    if (atomicOr(X + i, neu) == 0) fnxt[i >> 5] = 1;
                }
            } else if (live) {
                atomicCAS(&ctl->err, 0, CG_EDEVICE);
            }
        }
        qn = 0;
        if (cn > 0) claim(cn);
        found += fresh;
#pragma unroll
        for (int o = 16; o; o >>= 1) found += __shfl_xor_sync(0xffffffffu, found, o);
        if (lane == 0 && found) atomicAdd(&s_fresh, found);
        __syncthreads();
        if (threadIdx.x == 0 && s_fresh) atomicAdd(&Dp->fresh, s_fresh);

        unsigned long long word = 0;
        const int arrive = grid_arrive(ctl, timeout_ns, word, nbar++);
        if (arrive < 0) return;
        if (arrive == 1) {
            if (threadIdx.x == 0) block_close(*Dp, ctl);
            grid_release(ctl, word, 0);
        }
    }
}

// Packed keys of the states of one layer, in no particular order: a growth from the start state s0 is
// run from the identity (s = s0 w), so the value v of a state stands for s0's.
template <int N>
__global__ void block_export_kernel(BlockDev D, int which, uint64_t* out, unsigned long long cap,
                                    unsigned long long* count) {
    using Word = typename BlockShape<N>::Word;
    const Word* F = static_cast<const Word*>(D.N[which]);
    const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long g = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; g < D.ngroups; g += step) {
        if (!D.flag[which][g]) continue;
        for (unsigned b = (unsigned)g * 32u; b < (unsigned)g * 32u + 32u && b < D.nblocks; ++b) {
            Word f = F[b];
            if (!f) continue;
            const unsigned t = b / kBottom;
            const uint2 top = D.top[t];
            const unsigned low = D.bottom[b - t * kBottom];
            unsigned p[16];
            for (int v = 0; v < 8; ++v) {
                const unsigned c = (low >> (4 * v)) & 7u;
                p[v] = (top.y >> (4 * (((c & 3u) << 1) | (c >> 2)))) & 15u;
            }
            for (int v = 8; v < N; ++v) p[v] = (top.x >> (4 * (v - 8))) & 15u;
            const unsigned long long at = atomicAdd(count, (unsigned long long)popc_word(f));
            unsigned long long o = at;
            for (int e = 0; e < 1 << BlockShape<N>::M; ++e) {
                if (!(f >> e & 1)) continue;
                uint64_t key = 0;
                for (int v = 0; v < N; ++v) {
                    const int u = v < 2 * BlockShape<N>::M && (e >> (v >> 1) & 1) ? (v ^ 1) : v;
                    key |= ((D.start >> (4 * v)) & 15ull) << (4 * p[u]);
                }
                if (o < cap) out[o] = key;
                ++o;
            }
        }
    }
}

// ---- small groups: a thread-block cluster per growth ---------------------------------------------------
// Batches of growths of S_n for n <= 10, each in blocks of states by one cluster: a round ends with the
// cluster's hardware barrier instead of a grid barrier through L2, many growths run side by side
// without a common round, and a cluster that finishes one takes the next from the queue.  (1024
// random groups of n in 6..10: 36.2 ms as key lists in one launch with a grid barrier per round,
// 6.3 ms here.)  All words of a layer are looked at every round (113,400 for n = 10,
// 454 KB), no flags.  The words live in L2: 38 clusters of eight blocks hold 69 MB of them.
// Decisions are taken by every thread from the same counts, which the blocks write into each
// other's shared memory before the barrier.
namespace cgr = cooperative_groups;

constexpr int kClThreads = 512;
constexpr int kClMaxCluster = 16;

template <int T>
struct ClusterShared {
    static constexpr int kClWarps = T / 32;
    uint4 map[kClusterGens];
    unsigned qidx[kClWarps][kBlkQueue];
    unsigned qf[kClWarps][kBlkQueue];
    unsigned cidx[kClWarps][kBlkQueue];
    unsigned cf[kClWarps][kBlkQueue];
    unsigned acc[2];                       // states the block found, this round and (cleared) the next
    unsigned cnt[2][kClMaxCluster];        // states each block of the cluster found, by round parity
    int job;
};

template <int N>
__device__ __forceinline__ BlockPerm<N> cluster_unrank(const uint64_t* table, unsigned idx) {
    const uint64_t p = table[idx];
    BlockPerm<N> P;
    lookup_form((uint32_t)p & 0xFFFFu, P.sel[0], P.high[0]);
    if constexpr (N > 4) lookup_form((uint32_t)p >> 16, P.sel[1], P.high[1]);
    if constexpr (N > 8) lookup_form((uint32_t)(p >> 32), P.sel[2], P.high[2]);
    return P;
}

// Nibble v = position of value v in the canonical member of block b (the inverse of block_rank), in
// registers: the free positions are kept ascending in nibbles.
template <int N>
__device__ __forceinline__ uint64_t small_unrank(unsigned b) {
    constexpr int M = BlockShape<N>::M;
    using Nibbles = std::conditional_t<(N > 8), uint64_t, uint32_t>;
    Nibbles avail = (Nibbles)0x9876543210ull;
    Nibbles key = 0;
    auto take = [&](unsigned at) {
        const unsigned sh = 4u * at;
        const Nibbles v = (avail >> sh) & 15u;
        const Nibbles below = ((Nibbles)1 << sh) - 1u;
        avail = (avail & below) | ((avail >> 4) & ~below);
        return v;
    };
    constexpr unsigned pairs = N > 2 * M ? block_count(N) / N : block_count(N);
    if (N > 2 * M) {
        key |= take(b / pairs) << (4 * (N - 1));
        b %= pairs;
    }
    unsigned radix = pairs;
#pragma unroll
    for (int i = M - 1; i >= 1; --i) {
        radix /= (unsigned)((2 * i + 2) * (2 * i + 1) / 2);
        const unsigned d = b / radix;
        b -= d * radix;
        unsigned hi = 1;
#pragma unroll
        for (int h = 2; h < 2 * i + 2; ++h) hi += (unsigned)(h * (h - 1) / 2) <= d ? 1u : 0u;
        const unsigned lo = d - hi * (hi - 1u) / 2u;
        key |= take(hi) << (4 * (2 * i + 1));           // the larger place first: the smaller keeps its own
        key |= take(lo) << (4 * (2 * i));
    }
    return key | (avail & 0xFFu);                       // pair 0: the two free positions, ascending
}

// Where a growth's words live: in L2 (its blocks share them through a cluster), in the shared memory of
// the one block that grows it, or spread over the shared memory of its cluster (word i in block
// i mod size).
constexpr int kInL2 = 0, kInBlock = 1, kInCluster = 2;

// The barrier of a growth's blocks.
template <int kWhere>
__device__ __forceinline__ void growth_sync(const cgr::cluster_group& cl) {
    if (kWhere == kInBlock) __syncthreads();
    else cl.sync();
}

// A word of the growth that its blocks change: from shared memory, or through L2 (this SM's L1 may
// hold words of the growth before).
template <int kWhere>
__device__ __forceinline__ unsigned growth_word(const unsigned* p) {
    return kWhere == kInL2 ? __ldcg(p) : *(const volatile unsigned*)p;
}

// One growth by one cluster of blocks of T threads.  In shared memory (kInBlock, kInCluster) a block
// keeps the words of its share of the blocks of states, and their unranking table, and expands them.
template <int N, int kWhere, int T>
__device__ __forceinline__ void cluster_grow(ClusterShared<T>& S, const ClusterArgs& A, JobDev& J, unsigned* ws,
                                             std::conditional_t<kWhere != kInL2, uint64_t*, const uint64_t*> table, bool build,
                                             const cgr::cluster_group& cl) {
    constexpr unsigned kBlocks = block_count(N);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned size = kWhere == kInBlock ? 1u : cl.num_blocks();
    const unsigned rank = kWhere == kInBlock ? 0u : cl.block_rank();
    // the words one array of ws holds (kInCluster: this block's share; sizes are powers of two)
    const int sh = kWhere == kInCluster ? __ffs((int)size) - 1 : 0;
    const unsigned held = kWhere == kInCluster ? (kBlocks + size - 1u) >> sh : kBlocks;
    // word i of array `arr` (0: visited, 1..3: layers), wherever it is
    auto word = [&](unsigned arr, unsigned i) -> unsigned* {
        if constexpr (kWhere == kInCluster) return cl.map_shared_rank(ws + arr * held + (i >> sh), i & (size - 1u));
        else return ws + arr * kBlocks + i;
    };
    const int k = J.k;
    const GenSM* gens = J.gens;
    const bool smem = k <= kClusterGens;
    unsigned* qidx = S.qidx[wid];
    unsigned* qf = S.qf[wid];
    unsigned* cidx = S.cidx[wid];
    unsigned* cf = S.cf[wid];
    // the words of this growth, empty
    const unsigned all = size * T, me = rank * T + tid;
    if (kWhere == kInCluster) {
        for (unsigned i = tid; i < 4 * held; i += T) ws[i] = 0;
    } else {
        for (unsigned i = me; i < 4 * kBlocks; i += all) ws[i] = 0;
    }
    if constexpr (kWhere != kInL2) {
        if (build)
            for (unsigned i = tid; i < held; i += T)
                table[i] = (i << sh) + rank < kBlocks ? small_unrank<N>((i << sh) + rank) : 0;
    }
    if (smem)
        for (int j = tid; j < k; j += T) S.map[j] = *reinterpret_cast<const uint4*>(gens[j].map);
    if (tid < 2) S.acc[tid] = 0;
    growth_sync<kWhere>(cl);
    if (me == 0) {
        uint32_t q[BlockShape<N>::kWords] = {};
        for (int v = 0; v < N; ++v) q[v >> 2] |= (uint32_t)v << (8 * (v & 3));      // the identity
        unsigned m = 0;
        const unsigned idx = block_rank<N>(q, m);
        *word(0, idx) = 1u << m;
        *word(1, idx) = 1u << m;
        J.layer_sizes[0] = 1;
    }
    growth_sync<kWhere>(cl);
    int radius = 0, status = kRunning;
    unsigned long long states = 1;
    const int max_radius = J.max_radius, layers_cap = J.layers_cap;
    const unsigned long long max_states = J.keys_cap, stop_above = J.stop_above;
    while (status == kRunning) {
        const unsigned* F = ws + held * (1u + (unsigned)radius % 3u);
        unsigned* O = ws + held * (1u + (unsigned)(radius + 2) % 3u);
        const unsigned next = 1u + (unsigned)(radius + 1) % 3u;
        const int par = radius & 1;
        unsigned found = 0;
        int qn = 0, cn = 0;
        unsigned pidx = 0, pf = 0, pv = 0;
        auto claim = [&](int take) {
            cn -= take;
            if (lane < take) {
                const unsigned i = cidx[cn + lane], f = cf[cn + lane];
                const unsigned neu = f & ~atomicOr(word(0, i), f);
                if (neu) {
                    found += __popc(neu);
                    atomicOr(word(next, i), neu);
                }
            }
            __syncwarp();
        };
        auto settle = [&]() {
            const unsigned neu = pf & ~pv;
            const unsigned b = __ballot_sync(0xffffffffu, neu != 0);
            if (b == 0) return;
            if (neu) {
                const int at = cn + __popc(b & lanemask_lt());
                cidx[at] = pidx;
                cf[at] = neu;
            }
            cn += __popc(b);
            __syncwarp();
            if (cn >= 32) claim(32);
        };
        auto expand = [&](int take) {
            qn -= take;
            const bool active = lane < take;
            const unsigned idx = active ? qidx[qn + lane] : 0u;
            const unsigned f = active ? qf[qn + lane] : 0u;
            __syncwarp();
            const BlockPerm<N> P = cluster_unrank<N>(table, idx);
            for (int g = 0; g < k; ++g) {
                uint32_t q[BlockShape<N>::kWords];
                block_map<N>(smem ? S.map[g] : *reinterpret_cast<const uint4*>(gens[g].map), P, q);
                unsigned m;
                const unsigned i = block_rank<N>(q, m);
                // (as in block_grow_kernel: never past the words, whatever the tables hold)
                const bool live = active && i < kBlocks;
                if (active && !live) atomicCAS(&A.ctl->err, 0, CG_EDEVICE);
                const unsigned t = xor_bits32(f, m);
                unsigned v = 0;
                if (live) v = growth_word<kWhere>(word(0, i));
                settle();
                pidx = i;
                pf = live ? t : 0u;
                pv = v;
            }
        };
        const unsigned start = kWhere == kInCluster ? (unsigned)tid : me, step = kWhere == kInCluster ? (unsigned)T : all;
        for (unsigned base = start - lane; base < held; base += step) {
            const unsigned i = base + lane;
            unsigned f = 0;
            if (i < held) {
                f = growth_word<kWhere>(F + i);
                O[i] = 0;
            }
            const unsigned have = __ballot_sync(0xffffffffu, f != 0);
            if (have == 0) continue;
            if (f) {
                const int at = qn + __popc(have & lanemask_lt());
                qidx[at] = i;
                qf[at] = f;
            }
            qn += __popc(have);
            __syncwarp();
            if (qn >= 32) expand(32);
        }
        if (qn > kPairBlocks) expand(qn);
        settle();
        pf = 0;
        // A short remainder (in a small round all there is): a lane per (block, generator) pair instead
        // of per block, so that the lookups of a block are on their way together, and no look at the
        // visited word before the atomic.
        for (int first = 0; first < qn * k; first += 32) {
            const int pair = first + lane;
            const bool live = pair < qn * k;
            const int b = live ? pair / k : 0, g = live ? pair - b * k : 0;
            const BlockPerm<N> P = cluster_unrank<N>(table, live ? qidx[b] : 0u);
            uint32_t q[BlockShape<N>::kWords];
            block_map<N>(smem ? S.map[g] : *reinterpret_cast<const uint4*>(gens[g].map), P, q);
            unsigned m;
            const unsigned i = block_rank<N>(q, m);
            if (live && i < kBlocks) {
                const unsigned f = xor_bits32(qf[b], m);
                const unsigned neu = f & ~atomicOr(word(0, i), f);
                if (neu) {
                    found += __popc(neu);
                    atomicOr(word(next, i), neu);
                }
            } else if (live) {
                atomicCAS(&A.ctl->err, 0, CG_EDEVICE);
            }
        }
        qn = 0;
        if (cn > 0) claim(cn);
#pragma unroll
        for (int o = 16; o; o >>= 1) found += __shfl_xor_sync(0xffffffffu, found, o);
        if (lane == 0 && found) atomicAdd(&S.acc[par], found);
        __syncthreads();
        if (kWhere == kInBlock) {
            if (tid == 0) S.cnt[par][0] = S.acc[par];
        } else if (tid < (int)size) {
            *cl.map_shared_rank(&S.cnt[par][rank], tid) = S.acc[par];
        }
        if (tid == 0) S.acc[par ^ 1] = 0;
        growth_sync<kWhere>(cl);
        unsigned long long fresh = 0;
        for (unsigned q = 0; q < size; ++q) fresh += S.cnt[par][q];
        if (fresh == 0) {
            status = kDone;
        } else if (states + fresh > max_states) {
            status = kNeedMem;              // the layer is past the states the job may keep
        } else {
            states += fresh;
            ++radius;
            if (me == 0) J.layer_sizes[radius] = fresh;
            if (max_radius >= 0 && radius >= max_radius) status = kTruncRadius;
            else if (stop_above > 0 && fresh > stop_above) status = kTruncAbove;
            else if (radius + 1 >= layers_cap) status = kTruncRadius;
        }
    }
    if (me == 0) {
        J.radius = radius;
        J.status = status;
    }
    if constexpr (kWhere != kInL2) {
        // the last layer's packed keys, in no particular order: the value v of a state stands for the
        // start state's (see block_export_kernel)
        if (A.last == nullptr) return;
        constexpr int M = BlockShape<N>::M;
        const unsigned* F = ws + held * (1u + (unsigned)radius % 3u);
        for (unsigned i = tid; i < held; i += T) {
            unsigned f = F[i];
            if (!f) continue;
            const uint64_t p = table[i];
            unsigned at = (unsigned)atomicAdd(&A.ctl->adm.vis_used, (unsigned long long)__popc(f));
            for (; f; f &= f - 1u) {
                const int e = __ffs(f) - 1;
                uint64_t key = 0;
#pragma unroll
                for (int v = 0; v < N; ++v) {
                    const int swapped = v < 2 * M ? (e >> (v >> 1)) & 1 : 0;
                    key |= ((A.start >> (4 * v)) & 15ull) << (4u * ((unsigned)(p >> (4 * (v ^ swapped))) & 15u));
                }
                A.last[at++] = key;
            }
        }
    }
}

__global__ void __launch_bounds__(kClThreads, 2) cluster_grow_kernel(const ClusterArgs A) {
    __shared__ ClusterShared<kClThreads> S;
    const cgr::cluster_group cl = cgr::this_cluster();
    const unsigned size = cl.num_blocks();
    unsigned* ws = A.words + (uint64_t)(blockIdx.x / size) * A.stride;
    cl.sync();                              // every block runs: block 0 may write the others' S.job
    for (;;) {
        if (cl.block_rank() == 0 && threadIdx.x < size) {
            int j = 0;
            if (threadIdx.x == 0) j = (int)atomicAdd(&A.ctl->total_units, 1ull);
            j = __shfl_sync((1u << size) - 1u, j, 0);
            *cl.map_shared_rank(&S.job, threadIdx.x) = j;
        }
        cl.sync();
        const int job = S.job;
        if (job >= A.njobs) break;
        JobDev& J = A.jobs[job];
        switch (J.n) {
            case 9: cluster_grow<9, kInL2, kClThreads>(S, A, J, ws, A.table[9], false, cl); break;
            case 10: cluster_grow<10, kInL2, kClThreads>(S, A, J, ws, A.table[10], false, cl); break;
            default: break;                 // planned for n = 9, 10 only
        }
        cl.sync();                          // everyone is done with this job's shared state
    }
}

// Growths of n <= kClusterSmemN by one block each, words (40 KB for n = 8) and unranking table in its
// shared memory: a round costs shared-memory latencies and a block barrier, no trip to L2 (one growth
// of S_6 under adjacent transpositions 49 us on the grid, 29 us here; S_7 86 / 55, S_8 161 / 146, where
// one SM's issue rate takes over and more than ten generators are faster on the grid).  The jobs
// [A.first, A.njobs) of the queue (the first ones are the larger, for cluster_grow_kernel).
// 512 threads a block, two to an SM, for many jobs; 1024 for one, whose rounds they share.
template <int T>
__global__ void __launch_bounds__(T, 1024 / T) cluster_grow_small_kernel(const ClusterArgs A) {
    __shared__ ClusterShared<T> S;
    extern __shared__ uint64_t s_words[];
    const cgr::cluster_group cl = cgr::this_cluster();
    unsigned* ws = reinterpret_cast<unsigned*>(s_words);
    uint64_t* table = s_words + 2 * block_count(kClusterSmemN);
    int have = 0;                           // the n whose table is in shared memory
    for (;;) {
        if (threadIdx.x == 0) S.job = A.first + (int)atomicAdd(&A.ctl->dyn_next, 1ull);
        __syncthreads();
        const int job = S.job;
        if (job >= A.njobs) break;
        JobDev& J = A.jobs[job];
        const int n = J.n;
        const bool build = n != have;
        have = n;
        switch (n) {
#define CG_CLUSTER(n) case n: cluster_grow<n, kInBlock, T>(S, A, J, ws, table, build, cl); break;
            CG_CLUSTER(2) CG_CLUSTER(3) CG_CLUSTER(4) CG_CLUSTER(5) CG_CLUSTER(6) CG_CLUSTER(7) CG_CLUSTER(8)
#undef CG_CLUSTER
            default: break;                 // planned for n in 2..8 only
        }
        __syncthreads();                    // everyone is done with this job's shared state
    }
}

// One growth of S_8 or S_9 by one cluster with everything in its shared memory: the issue rate of as
// many SMs, and rounds without a trip to L2 (which blocks take part, and for which sizes: spread_blocks
// in host_api.cu).
constexpr int kSpreadThreads = 1024;
__global__ void __launch_bounds__(kSpreadThreads, 1) cluster_grow_spread_kernel(const ClusterArgs A) {
    __shared__ ClusterShared<kSpreadThreads> S;
    extern __shared__ uint64_t s_words[];
    const cgr::cluster_group cl = cgr::this_cluster();
    JobDev& J = A.jobs[0];
    const unsigned size = cl.num_blocks();
    const unsigned held = ((J.n == 8 ? block_count(8) : block_count(9)) + size - 1u) / size;
    unsigned* ws = reinterpret_cast<unsigned*>(s_words);
    uint64_t* table = s_words + 2 * held;
    switch (J.n) {
        case 8: cluster_grow<8, kInCluster, kSpreadThreads>(S, A, J, ws, table, true, cl); break;
        case 9: cluster_grow<9, kInCluster, kSpreadThreads>(S, A, J, ws, table, true, cl); break;
        default: break;                     // planned for n = 8, 9 only
    }
    cl.sync();                              // nobody leaves while its words are in use
}

// Unranking tables of cluster_grow_kernel, one for each n asked for: block idx -> nibble v = position
// of value v.
__global__ void cluster_prepare_kernel(const ClusterArgs A, unsigned want) {
    for (int n = kClusterSmemN + 1; n <= kClusterMaxN; ++n) {
        if (!(want >> n & 1u)) continue;
        uint64_t* out = const_cast<uint64_t*>(A.table[n]);
        const int M = block_pairs(n);
        const unsigned count = block_count(n);
        for (unsigned b = blockIdx.x * blockDim.x + threadIdx.x; b < count; b += gridDim.x * blockDim.x) {
            unsigned pairs = 1;
            for (int i = 0; i < M; ++i) pairs *= (unsigned)((2 * i + 2) * (2 * i + 1) / 2);
            unsigned char place[16];
            arrange_pairs(b % pairs, M, place);
            unsigned char free_[16];
            for (int i = 0; i < n; ++i) free_[i] = (unsigned char)i;
            uint64_t key = 0;
            if (n > 2 * M) {                // the single top value (n odd)
                const unsigned d = b / pairs;
                key |= (uint64_t)d << (4 * (n - 1));
                for (int j = (int)d; j + 1 < n; ++j) free_[j] = free_[j + 1];
            }
            for (int v = 0; v < 2 * M; ++v) key |= (uint64_t)free_[place[v]] << (4 * v);
            out[b] = key;
        }
    }
}

using block_fn = void (*)(BlockDev*, Ctl*, int, uint64_t);

block_fn block_kernel(int n) {
    switch (n) {
        case 10: return block_grow_kernel<10>;
        case 11: return block_grow_kernel<11>;
        case 12: return block_grow_kernel<12>;
        case 13: return block_grow_kernel<13>;
        default: return block_grow_kernel<14>;
    }
}

}  // namespace

uint64_t cluster_words(int n) { return 4ull * block_count(n); }
uint64_t cluster_table_entries(int n) { return block_count(n); }

cudaError_t launch_cluster_prepare(const ClusterArgs& A, unsigned want, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    cluster_prepare_kernel<<<152, 256, 0, st>>>(A, want);
    return cudaGetLastError();
}

int cluster_max_clusters(int size) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3(kClThreads);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)size, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, cluster_grow_kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_cluster_grow(const ClusterArgs& A, int clusters, int size, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * size));
    cfg.blockDim = dim3(kClThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {(unsigned)size, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cluster_grow_kernel, A);
}

namespace {
constexpr size_t small_smem() { return (size_t)block_count(kClusterSmemN) * (4 * 4 + 8); }
}

namespace {
size_t spread_smem(int n, int size) { return (size_t)((block_count(n) + size - 1) / size) * (4 * 4 + 8); }
cudaLaunchConfig_t spread_config(int n, int size, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size);
    cfg.blockDim = dim3(kSpreadThreads);
    cfg.dynamicSmemBytes = spread_smem(n, size);
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim = {(unsigned)size, 1, 1};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}
}

bool cluster_spread_ok(int n, int size) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = spread_config(n, size, &attr);
    int clusters = 0;
    if (cudaFuncSetAttribute(cluster_grow_spread_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)spread_smem(9, 4)) != cudaSuccess ||
        cudaFuncSetAttribute(cluster_grow_spread_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, cluster_grow_spread_kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return clusters > 0;
}

cudaError_t launch_cluster_spread(const ClusterArgs& A, int n, int size, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg = spread_config(n, size, &attr);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, cluster_grow_spread_kernel, A);
}

int cluster_small_blocks(int device) {
    int sms = 0, per_sm = 0;
    const cudaFuncAttribute at = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(cluster_grow_small_kernel<512>, at, (int)small_smem()) != cudaSuccess ||
        cudaFuncSetAttribute(cluster_grow_small_kernel<1024>, at, (int)small_smem()) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cluster_grow_small_kernel<512>, 512, small_smem()) !=
            cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return sms * per_sm;
}

cudaError_t launch_cluster_small(const ClusterArgs& A, int blocks, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    if (blocks == 1) cluster_grow_small_kernel<1024><<<1, 1024, small_smem(), st>>>(A);
    else cluster_grow_small_kernel<512><<<blocks, 512, small_smem(), st>>>(A);
    return cudaGetLastError();
}

int block_max_grid(int device, int n) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, block_kernel(n), kBlkThreads, 0) != cudaSuccess)
        return 0;
    return sms * per_sm;
}

cudaError_t launch_block_tables(const BlockDev& host, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    const unsigned work = host.ntop > kBottom ? host.ntop : kBottom;
    unsigned grid = (work + 127) / 128;
    if (grid > 152u * 16) grid = 152u * 16;
    block_tables_kernel<<<grid, 128, 0, st>>>(host);
    return cudaGetLastError();
}

cudaError_t launch_block_init(BlockDev* d, int n, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    switch (n) {
        case 10: block_init_kernel<10><<<1, 32, 0, st>>>(d); break;
        case 11: block_init_kernel<11><<<1, 32, 0, st>>>(d); break;
        case 12: block_init_kernel<12><<<1, 32, 0, st>>>(d); break;
        case 13: block_init_kernel<13><<<1, 32, 0, st>>>(d); break;
        default: block_init_kernel<14><<<1, 32, 0, st>>>(d); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_block_import(BlockDev* d, int n, const uint64_t* keys, unsigned long long lo,
                                unsigned long long hi, int* d_err, int grid, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    switch (n) {
        case 10: block_import_kernel<10><<<grid, 256, 0, st>>>(d, keys, lo, hi, d_err); break;
        case 11: block_import_kernel<11><<<grid, 256, 0, st>>>(d, keys, lo, hi, d_err); break;
        case 12: block_import_kernel<12><<<grid, 256, 0, st>>>(d, keys, lo, hi, d_err); break;
        case 13: block_import_kernel<13><<<grid, 256, 0, st>>>(d, keys, lo, hi, d_err); break;
        default: block_import_kernel<14><<<grid, 256, 0, st>>>(d, keys, lo, hi, d_err); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_block_grow(BlockDev* d, Ctl* ctl, int n, int grid, int max_rounds, uint64_t timeout_ns,
                              cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kBlkThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, block_kernel(n), d, ctl, max_rounds, timeout_ns);
}

cudaError_t launch_block_export(const BlockDev& host, int which, uint64_t* out, unsigned long long cap,
                                unsigned long long* count, int grid, cudaStream_t st) {
    (void)cudaGetLastError();   // clear a stale error: the check after the launch is about this one
    switch (host.n) {
        case 10: block_export_kernel<10><<<grid, 128, 0, st>>>(host, which, out, cap, count); break;
        case 11: block_export_kernel<11><<<grid, 128, 0, st>>>(host, which, out, cap, count); break;
        case 12: block_export_kernel<12><<<grid, 128, 0, st>>>(host, which, out, cap, count); break;
        case 13: block_export_kernel<13><<<grid, 128, 0, st>>>(host, which, out, cap, count); break;
        default: block_export_kernel<14><<<grid, 128, 0, st>>>(host, which, out, cap, count); break;
    }
    return cudaGetLastError();
}

}  // namespace cg
