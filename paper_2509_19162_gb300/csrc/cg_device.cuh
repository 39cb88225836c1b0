// Device-side building blocks of the growth kernels: the generator action on packed keys,
// the key hash, the open-addressing insert, and a bounded grid-wide barrier.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cg_internal.h"
#include "../../include/cg_growth.h"

namespace cg {

// Rotation of the 64-bit word hi:lo left by r (0..63), as two 32-bit funnel shifts: the halves
// trade places when r >= 32, then each result half is the top word of a 64-bit concatenation
// shifted left by r mod 32.  (A 64-bit rotate by a run-time amount costs several times this.)
__device__ __forceinline__ void rotl_halves(uint32_t lo, uint32_t hi, unsigned r, uint32_t& rlo,
                                            uint32_t& rhi) {
    const bool swap = (r & 32u) != 0;
    const uint32_t a = swap ? hi : lo, b = swap ? lo : hi;
    rhi = __funnelshift_l(a, b, r);
    rlo = __funnelshift_l(b, a, r);
}

// t[i] = s[g[i]] on packed keys (see GenSM): a range reversal by bit reversal, otherwise a union
// of rotated, masked copies of s, built on 32-bit halves.  kRev = false compiles the
// shift-and-mask form only: for kernels that run generators of at most 16 elements, where
// reversals are in that form.
template <bool kRev = true>
__device__ __forceinline__ uint64_t apply_gen(const GenSM& g, uint64_t s) {
    if (kRev && g.kind == 1) {
        uint64_t r = __brevll(s);
        if (g.width >= 2) r = ((r >> 1) & 0x5555555555555555ull) | ((r & 0x5555555555555555ull) << 1);
        if (g.width == 4) r = ((r >> 2) & 0x3333333333333333ull) | ((r & 0x3333333333333333ull) << 2);
        const int sh = g.rev_shift;
        r = sh >= 0 ? (r >> sh) : (r << -sh);
        return (s & ~g.mask[0]) | (r & g.mask[0]);
    }
    const uint32_t lo = (uint32_t)s, hi = (uint32_t)(s >> 32);
    uint32_t tlo = 0, thi = 0;
    const uint32_t nt = g.nterms;
#pragma unroll 2
    for (uint32_t i = 0; i < nt; ++i) {
        uint32_t rlo, rhi;
        rotl_halves(lo, hi, g.rot[i], rlo, rhi);
        const uint64_t m = g.mask[i];
        tlo |= rlo & (uint32_t)m;
        thi |= rhi & (uint32_t)(m >> 32);
    }
    return ((uint64_t)thi << 32) | tlo;
}

// 64-bit finaliser of MurmurHash3 (A. Appleby, public domain): a bijection of uint64.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t k) {
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k;
}

// Relaxed load served by L2 (never a stale L1 line): used for data other SMs write.
__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed_ull(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ int ld_relaxed_int(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Insert-if-absent with linear probing.  Returns 1 if this call inserted the key, 0 if it was
// present (or inserted concurrently by another thread), -1 if `max_probe` slots were visited
// without finding the key or an empty slot.
__device__ __forceinline__ int table_insert(uint64_t* table, uint64_t mask, uint64_t key,
                                            uint64_t max_probe) {
    uint64_t h = mix64(key) & mask;
    for (uint64_t p = 0; p < max_probe; ++p) {
        uint64_t cur = ld_relaxed(table + h);
        if (cur == key) return 0;
        if (cur == kEmpty) {
            unsigned long long prev = atomicCAS(reinterpret_cast<unsigned long long*>(table + h),
                                                (unsigned long long)kEmpty,
                                                (unsigned long long)key);
            if (prev == kEmpty) return 1;
            if (prev == key) return 0;
        }
        h = (h + 1) & mask;
    }
    return -1;
}

// Two 16-byte loads served by L2 (cache-global, never a stale L1 line) covering one aligned
// 32-byte sector = 4 table slots.  Weak loads are enough: a slot, once written, never changes,
// and a stale "empty" is caught by the CAS that follows.
__device__ __forceinline__ void ld_sector(const uint64_t* p, uint64_t (&v)[4]) {
    const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2*>(p));
    const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// G independent insert-if-absent sequences (linear probing) advanced together, so that one
// thread keeps G sector loads (and CASes) in flight.  Each step reads the aligned 4-slot
// sector holding the current slot and scans it from that slot on: a match ends the sequence
// (already present); the first empty slot gets a CAS; a full sector moves on to the next.
// res[i] as for table_insert; entries whose bit in vmask is clear are left at 0.
template <int G>
__device__ __forceinline__ void table_insert_multi_sector(uint64_t* table, uint64_t mask,
                                                          const uint64_t (&key)[G], int (&res)[G],
                                                          unsigned vmask, uint64_t max_steps) {
    uint64_t h[G];
    unsigned pend = vmask;   // bit i: sequence i still probing
#pragma unroll
    for (int i = 0; i < G; ++i) {
        res[i] = 0;
        h[i] = mix64(key[i]) & mask;
    }
    for (uint64_t step = 0; pend && step < max_steps; ++step) {
        uint64_t v[G][4];
#pragma unroll
        for (int i = 0; i < G; ++i)
            if (pend >> i & 1u) ld_sector(table + (h[i] & ~3ull), v[i]);
        unsigned cas = 0;
        uint64_t old[G];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (!(pend >> i & 1u)) continue;
            const unsigned off = (unsigned)(h[i] & 3u);
            int hit = -1, empty = -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if ((unsigned)q >= off && hit < 0 && empty < 0) {
                    if (v[i][q] == key[i]) hit = q;
                    else if (v[i][q] == kEmpty) empty = q;
                }
            }
            if (hit >= 0) {
                pend &= ~(1u << i);
            } else if (empty >= 0) {
                h[i] = (h[i] & ~3ull) | (unsigned)empty;
                cas |= 1u << i;
                old[i] = atomicCAS(reinterpret_cast<unsigned long long*>(table + h[i]),
                                   (unsigned long long)kEmpty, (unsigned long long)key[i]);
            } else {
                h[i] = ((h[i] | 3ull) + 1) & mask;   // next sector
            }
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (cas >> i & 1u) {
                if (old[i] == kEmpty) { res[i] = 1; pend &= ~(1u << i); }
                else if (old[i] == key[i]) { pend &= ~(1u << i); }
                else h[i] = (h[i] + 1) & mask;       // lost the slot: continue after it
            }
        }
    }
#pragma unroll
    for (int i = 0; i < G; ++i)
        if (pend >> i & 1u) res[i] = -1;
}

// As table_insert_multi_sector, but each step reads the single current slot (8 bytes).
template <int G>
__device__ __forceinline__ void table_insert_multi_slot(uint64_t* table, uint64_t mask,
                                                        const uint64_t (&key)[G], int (&res)[G],
                                                        unsigned vmask, uint64_t max_steps) {
    uint64_t h[G];
    unsigned pend = vmask;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        res[i] = 0;
        h[i] = mix64(key[i]) & mask;
    }
    for (uint64_t step = 0; pend && step < max_steps; ++step) {
        uint64_t v[G];
#pragma unroll
        for (int i = 0; i < G; ++i)
            if (pend >> i & 1u) v[i] = __ldcg(table + h[i]);
        unsigned cas = 0;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (pend >> i & 1u) {
                if (v[i] == key[i]) {
                    pend &= ~(1u << i);
                } else if (v[i] == kEmpty) {
                    cas |= 1u << i;
                    v[i] = atomicCAS(reinterpret_cast<unsigned long long*>(table + h[i]),
                                     (unsigned long long)kEmpty, (unsigned long long)key[i]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (cas >> i & 1u) {
                if (v[i] == kEmpty) { res[i] = 1; pend &= ~(1u << i); }
                else if (v[i] == key[i]) { pend &= ~(1u << i); }
            }
            if (pend >> i & 1u) h[i] = (h[i] + 1) & mask;
        }
    }
#pragma unroll
    for (int i = 0; i < G; ++i)
        if (pend >> i & 1u) res[i] = -1;
}

// Index of a permutation in a bitmap over S_n: the position-major Lehmer rank
//     rank(s) = sum_{i=1}^{n-1} d_i * i!,   d_i = #{ j < i : s_j < s_i },
// a bijection onto [0, n!) (identity -> n!-1, full reversal -> 0).  A generator that moves only
// positions below j changes only the digits below j, so the image of a state lies within j!
// ranks of it: the probes of prefix reversals and other short-support generators of one state
// share cache lines.  Digits are taken from the top position down, d_i = s_i - #{j > i : s_j <
// s_i}; the digits of positions 12.. and 1..11 form two 32-bit Horner sums, then joined.
template <int N>
__device__ __forceinline__ uint64_t perm_rank_n(uint64_t key) {
    unsigned right = 0, top = 0, low = 0;
#pragma unroll
    for (int i = N - 1; i >= 1; --i) {
        const unsigned v = (unsigned)(key >> (4 * i)) & 15u;
        const unsigned d = v - __popc(right & ((1u << v) - 1u));
        right |= 1u << v;
        if (i >= 12) top = top * (unsigned)(i + 1) + d;
        else low = low * (unsigned)(i + 1) + d;
    }
    if (N > 12) return (uint64_t)top * 479001600ull + low;   // 12!
    return low;
}

// The same rank with n known only at run time (n <= 16).
__device__ __forceinline__ uint64_t perm_rank(uint64_t key, int n) {
    unsigned right = 0, top = 0, low = 0;
#pragma unroll
    for (int i = 15; i >= 1; --i) {
        if (i < n) {
            const unsigned v = (unsigned)(key >> (4 * i)) & 15u;
            const unsigned d = v - __popc(right & ((1u << v) - 1u));
            right |= 1u << v;
            if (i >= 12) top = top * (unsigned)(i + 1) + d;
            else low = low * (unsigned)(i + 1) + d;
        }
    }
    return (uint64_t)top * 479001600ull + low;
}

// A permutation of N <= 16 elements held as one byte per element (byte_word, byte_slot): what the
// byte-permute generators (GenSM::sel) act on and what rank_bytes reads an element from in one
// instruction.
template <int N>
struct ByteState {
    static constexpr int kWords = N <= 8 ? 2 : N <= 12 ? 3 : 4;
    uint32_t w[kWords];
};

// The bytes of a packed key; a parent-edge tag in bits 60..63 (N <= 15) is dropped.
template <int N>
__device__ __forceinline__ ByteState<N> unpack_bytes(uint64_t key) {
    const uint32_t lo = (uint32_t)key, hi = (uint32_t)(key >> 32);
    ByteState<N> s;
    s.w[0] = lo & 0x0F0F0F0Fu;
    s.w[1] = (lo >> 4) & 0x0F0F0F0Fu;
    if constexpr (N > 8 && N <= 12) {
        const uint32_t x = __byte_perm(hi, 0, 0x1100);
        s.w[2] = (x & 0x000F000Fu) | ((x >> 4) & 0x0F000F00u);
    }
    if constexpr (N > 12) {
        s.w[2] = hi & 0x0F0F0F0Fu;
        s.w[3] = (hi >> 4) & (N <= 15 ? 0x000F0F0Fu : 0x0F0F0F0Fu);
    }
    return s;
}

// The packed key of a byte state, as its two halves.
template <int N>
__device__ __forceinline__ void pack_bytes(const ByteState<N>& s, uint32_t& lo, uint32_t& hi) {
    lo = s.w[0] | (s.w[1] << 4);
    hi = 0;
    if constexpr (N > 8 && N <= 12) {
        const uint32_t x = s.w[2] | (s.w[2] >> 4);
        hi = __byte_perm(x, 0, 0x4420);
    }
    if constexpr (N > 12) hi = s.w[2] | (s.w[3] << 4);
}

// t[i] = s[g[i]] with the generator's selectors (16-byte aligned); *head receives sel[0], whose
// top four bits are the inverse's tag.
template <int N>
__device__ __forceinline__ ByteState<N> apply_selectors(const uint32_t* sel, const ByteState<N>& s, uint32_t* head) {
    ByteState<N> t;
    if constexpr (N <= 8) {
        const uint2 a = *reinterpret_cast<const uint2*>(sel);
        *head = a.x;
        t.w[0] = __byte_perm(s.w[0], s.w[1], a.x);
        t.w[1] = __byte_perm(s.w[0], s.w[1], a.y);
    } else if constexpr (N <= 12) {
        const uint4 a = *reinterpret_cast<const uint4*>(sel);
        const uint2 b = *reinterpret_cast<const uint2*>(sel + 4);
        *head = a.x;
        t.w[0] = __byte_perm(__byte_perm(s.w[0], s.w[1], a.x), s.w[2], a.y);
        t.w[1] = __byte_perm(__byte_perm(s.w[0], s.w[1], a.z), s.w[2], a.w);
        t.w[2] = __byte_perm(__byte_perm(s.w[0], s.w[1], b.x), s.w[2], b.y);
    } else {
        const uint4 a = *reinterpret_cast<const uint4*>(sel);
        const uint4 b = *reinterpret_cast<const uint4*>(sel + 4);
        const uint4 c = *reinterpret_cast<const uint4*>(sel + 8);
        *head = a.x;
        t.w[0] = __byte_perm(__byte_perm(s.w[0], s.w[1], a.x), __byte_perm(s.w[2], s.w[3], a.y), a.z);
        t.w[1] = __byte_perm(__byte_perm(s.w[0], s.w[1], a.w), __byte_perm(s.w[2], s.w[3], b.x), b.y);
        t.w[2] = __byte_perm(__byte_perm(s.w[0], s.w[1], b.z), __byte_perm(s.w[2], s.w[3], b.w), c.x);
        t.w[3] = __byte_perm(__byte_perm(s.w[0], s.w[1], c.y), __byte_perm(s.w[2], s.w[3], c.z), c.w);
    }
    return t;
}

// perm_rank_n of a byte state.  A digit is d_i = v_i - (N-1-i) + #{j > i : s_j > v_i}; with the
// values to the right as bits 0..15 of `right` and ones above them, the arithmetic shift
// right >> v_i holds 16 + v_i + #{j > i : s_j > v_i} ones, so one popc gives d_i plus a constant
// and the constants of all positions come off at the end: six instructions a position.
template <int N>
__device__ __forceinline__ uint64_t rank_bytes(const ByteState<N>& s) {
    int right = (int)0xFFFF0000u;
    unsigned top = 0, low = 0, ctop = 0, clow = 0;
#pragma unroll
    for (int i = N - 1; i >= 1; --i) {
        const unsigned v = __byte_perm(s.w[byte_word(N, i)], 0, 0x4440u | (unsigned)byte_slot(N, i));
        // (the top position has nothing to its right: its digit is its value)
        const unsigned p = i == N - 1 ? v : (unsigned)__popc((unsigned)(right >> v));
        const unsigned c = i == N - 1 ? 0u : 16u + (unsigned)(N - 1 - i);
        if (i >= 12) {
            top = top * (unsigned)(i + 1) + p;
            ctop = ctop * (unsigned)(i + 1) + c;
        } else {
            low = low * (unsigned)(i + 1) + p;
            clow = clow * (unsigned)(i + 1) + c;
        }
        right |= 1 << v;
    }
    if (N > 12) return (uint64_t)(top - ctop) * 479001600ull + (low - clow);   // 12!
    return low - clow;
}

// Rank of a binary vector of n elements with m ones among all C(n, m): sum over its ones p_1 < p_2 < ..
// of C(p_t, t) (the combinatorial number system), six elements at a time: row c of group j holds, for
// every value of the elements 6j .. 6j+5, their part of the sum when c ones come before them
// (make_comb_table in host_api.cu lays the rows out, min(6j, m) + 1 of group j).  Moving elements below
// position j leaves the parts of the ones above it alone, as with perm_rank.  m < 0: the vector has -m
// zeros, and they are ranked.
__device__ __forceinline__ uint32_t comb_rank(const uint32_t* table, uint64_t v, int n, int m) {
    if (m < 0) {
        v ^= n >= 64 ? ~0ull : (1ull << n) - 1ull;
        m = -m;
    }
    uint32_t r = 0;
    unsigned c = 0, row = 0;
    for (int j = 0; j < n; j += 6) {
        const unsigned x = (unsigned)v & 63u;
        v >>= 6;
        r += table[(row + c) * 64u + x];
        c += __popc(x);
        row += (unsigned)min(j, m) + 1u;
    }
    return r;
}

__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

__device__ __forceinline__ unsigned long long ld_acquire_ull(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_ull(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.b64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
}

// Arrival half of a grid barrier whose last arriving block does some work before releasing
// the others (cooperative launch: all blocks co-resident).  `gen` is the number of barriers
// this block has passed in the launch (every block passes the same ones).  Returns 1 in every
// thread of the block that arrived last (it must call grid_release after its work), 0 in the
// other blocks once the last block has released them, -1 on error (timeout or an error word
// set by another block: the caller returns from the kernel).  `word` receives the barrier word:
// for the last block the one it arrived on (pass it to grid_release), for the others the one
// the release wrote, whose payload is word >> kGenBits.
// Ordering: every arrival is an acquire-release atomic (the block's writes before it, ordered
// by the block's own barrier, are visible to whoever observes it later, and the last arrival
// acquires everything released before), and the waiters' poll of the barrier word is an
// acquire of the closing block's work.
__device__ __forceinline__ int grid_arrive(Ctl* ctl, uint64_t timeout_ns, unsigned long long& word,
                                           unsigned gen) {
    __shared__ int s_state;
    __shared__ unsigned long long s_word;
    __syncthreads();
    if (threadIdx.x == 0) {
        gen &= (unsigned)kGenMask;
        int state = 0;
        unsigned long long w = gen;
        // The counter only grows (zeroed before each launch): barrier `gen` is complete when it reaches
        // gridDim.x * (gen + 1), so nothing is reset on the way.  One counter for every block: the last
        // arrival is one L2 round trip from the release, and 608 additions queue for less than the second
        // trip that a level of group counters costs (S_10 under L, X, 59 rounds: 0.401 ms with 32 groups,
        // 0.360 ms so; S_11 under L, R, X 1.016 / 0.981 ms).
        if (atom_add_acq_rel(&ctl->bar_count, 1u) == gridDim.x * (gen + 1) - 1) state = 1;
        if (state == 0) {
            const uint64_t t0 = globaltimer_ns();
            unsigned spins = 0;
            while (((w = ld_acquire_ull(&ctl->bar_word)) & kGenMask) == gen) {
                if ((++spins & 63u) == 0) {
                    if (*(volatile int*)&ctl->err != 0) { state = -1; break; }
                    if (globaltimer_ns() - t0 > timeout_ns) {
                        atomicCAS(&ctl->err, 0, CG_ETIMEOUT);
                        state = -1;
                        break;
                    }
                }
                __nanosleep(spins < 64 ? 32 : 256);
            }
        }
        s_state = state;
        s_word = w;
    }
    __syncthreads();
    word = s_word;
    return s_state;
}

// Release half: called by every thread of the last arriving block after its work, with the
// word grid_arrive gave it and the payload for every block (below 2^(64 - kGenBits)).
__device__ __forceinline__ void grid_release(Ctl* ctl, unsigned long long word, unsigned long long payload) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long gen = ((word & kGenMask) + 1) & kGenMask;
        st_release_ull(&ctl->bar_word, gen | (payload << kGenBits));
    }
}

}  // namespace cg
