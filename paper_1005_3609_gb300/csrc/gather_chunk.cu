// The per-site gather on rows of 16-byte chunks.
//
// Same operation as gather_kernel: out[dst] = sum_e coef_e w^{shift_e} in[src_e]
// (mod p), one per-site factor of Sec. 3.2-3.3, or two composed (multiplication
// by w a shift of the degree index), on the degree windows of cp_internal.h:
// only the degrees that can be non-zero are read, computed and written.
//
// A warp takes one unit of work (a few consecutive destination rows with up to 64
// edges together, or one heavier row or a part of it, cp_internal.h), all its degrees or a
// share of them, and works alone:
//   front end  32 edges at a time, one per lane: the edge's word and its source's
//              window, the window of its destination row, their intersection; the
//              edges that contribute are listed in shared memory;
//   copies     per listed edge, ahead of its use, the lanes copy the source words
//              into a slot of the warp's own (cp.async, 16 bytes a lane, a lane's
//              own chunks only, so no barrier is needed), zeros where the edge
//              does not reach: what follows needs no bounds;
//   sums       per destination row the warp holds the sums of the whole window in
//              registers, 32 chunks of 16 bytes (four primes of one degree) per
//              step, kSteps steps; a row with a longer window is walked in several
//              passes.  Per edge and step: one 16-byte shared load and two
//              multiply-adds per word.
//
// What bounds it: the shared-memory data path, each source word going through it twice
// (copy and load; 78% of its rate in the middle launches of the square width-16 row, where
// DRAM gives 3.8 TB/s and L2 is at 46%), with the issue slots next (66%).  Width 14, D = 63, 16 primes (57 346 rows, 365 000
// edges of a two-site table): 0.66 instructions per scheduler and cycle, 66% of the
// shared-memory data path, DRAM at a quarter of its rate, 0.107 ms; the
// producer/consumer kernel on whole rows that this one replaces took 0.155 ms.  One
// row of the width-16 strip 7.73 -> 3.94 ms, triangular (D = 32) 5.32 -> 1.42 ms; with
// the constants of a row's primes loaded once per row, the lane's prime group computed
// once and an edge's first word kept from its copy, 3.73 and 1.28 ms; with two-warp
// instead of four-warp blocks 3.67 and 1.25 ms (one-warp blocks 3.72, 1.30); units of 64
// edges instead of 32 took the square k = 33 sweep from 86.4 to 82.2 ms (cp_internal.h).
// 28 warps per SM (72 registers) beat 24 (4.31 before the last two changes) and 20, and
// 32, which spill (4.02 after them); two edges in flight beat four (4.22 at 24 warps) in launches that fill the chip;
// four steps beat six (4.26) and eight (4.87), which hold wider rows in one pass but
// leave fewer warps.  Bulk copies with an mbarrier per slot (5.1) and loads straight to
// registers (5.8) halve the shared-memory traffic but wait longer.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "cp_internal.h"
#include "modred.cuh"

namespace cp {

constexpr int kWarps = kChunkWarps;                      // warps per block
constexpr int kSteps = kChunkSteps;                      // 32-chunk steps of a row held in registers
constexpr uint32_t kSlotBytes = kSteps * 512u;         // one edge's source words

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Streaming 16-byte global store where pred != 0, without a branch.
__device__ __forceinline__ void stcs128_if(uint4 *ptr, uint4 v, uint32_t pred) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t"
        "@p st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(ptr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w),
        "r"(pred)
        : "memory");
}

// ---------------------------------------------------------------- sums and their reduction
// An input word x (a residue in [0, p) or a signed representative in [-p, p), as
// 32-bit two's complement) is x = xh 2^16 + xl with xl = x & 0xffff (unsigned)
// and xh = x >> 16 (signed).  The edge's coefficient c (|c| <= 127) sits in byte
// 3 of b, byte 2 is zero, so dp2a.hi (x's halves times b's bytes 2, 3) adds c xh.
struct Acc2 {
    uint32_t lo;
    int hi;
};

// Fast sums: lo = sum c x modulo 2^32 (one 32-bit multiply-add), hi = sum c xh - k0
// with k0 = fast_offset(S), S an upper bound of sum |c| over the row.
//
// Reduction (32-bit, two multiplies a word): u = sum c x = hi 2^16 + L with
// L = sum c xl + k0 2^16 in (S 2^15, 5 S 2^15 + 2^16] since |sum c xl| < S 2^16
// and 3 S / 2 <= k0 <= 3 S / 2 + 1.  With m = floor(2^48 / p) and q = floor(hi m / 2^32):
//   |hi m - hi 2^48 / p| <= |hi| <= S 2^15 + k0, so with e = (S 2^15 + k0) / 2^32
//   q <= hi 2^16 / p + e = u / p - L / p + e < u / p     (L / p > S 2^15 / 2^31 > e),
//   q > hi 2^16 / p - e - 1 = u / p - L / p - e - 1,
// hence 0 < r = u - q p < p + L + e p, and the word stored, r - p = lo - (q + 1) p
// (exact modulo 2^32), lies in [-p, L + e p).  It is a representative in
// [-p, p) when 5 S 2^15 + 2^16 + (S + 2) p / 2^17 + 1 < p: fast_ok.
__device__ __forceinline__ uint32_t fast_reduce(const Acc2 &a, uint32_t p, uint32_t m) {
    int q1;
    asm("mad.hi.s32 %0, %1, %2, 1;" : "=r"(q1) : "r"(a.hi), "r"(m));
    return a.lo - (uint32_t)q1 * p;
}

// The same for any prime, and sums of coefficients S < 2^15 (kChunkMaxSum): h = hi + k0 =
// sum c xh, l = lo - h 2^16 = sum c xl as a signed word (|l| < S 2^16 < 2^31), so
// v = sum c x = h 2^16 + l exactly and u = v + p 2^15 lies in (0, p 2^16).  With t =
// chunk_shift(p), m = floor(2^(32 + t) / p) and q = floor(floor(u / 2^t) m / 2^32),
//   u / p >= q > u / p - u / 2^(32 + t) - 2^t / p - 1 > u / p - 2:
// for p >= 2^17, t = 16, the terms are below p / 2^32 < 1/2 and 1/2, for smaller p of b
// bits, t = b - 2, below 2^-14 and 1/2.  So r = u - q p lies in [0, 2p), and the word
// stored, r - p, in [-p, p).  A few times the instructions of the 32-bit reduction, once a
// row and word: square 12 x 13 on 8 primes near 10^6 1.28 ms, near 2^31 with the 32-bit one
// 1.14; square width 16, D 63, 16 primes, eight rows 19.5 ms (on the register kernel 13.2
// and 64.7).
__device__ __forceinline__ uint32_t any_reduce(const Acc2 &a, uint32_t k0, uint32_t p, uint32_t m, uint32_t t) {
    const int h = a.hi + (int)k0;
    const int l = (int)(a.lo - ((uint32_t)h << 16));
    const unsigned long long u = (unsigned long long)((long long)h * 65536 + l + ((long long)p << 15));
    return (uint32_t)u - (__umulhi((uint32_t)(u >> t), m) + 1u) * p;
}

// Asynchronous 16-byte copy to shared memory where t < len (unsigned), zeros written elsewhere.
__device__ __forceinline__ void cp16_below(uint32_t dst, const uint4 *src, uint32_t t, uint32_t len) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ge.u32 p, %2, %3;\n\t"
        "cp.async.cg.shared.global [%0], [%1], 16, p;\n\t}" ::"r"(dst), "l"(src), "r"(t), "r"(len)
        : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void add_word(Acc2 &a, uint32_t x, int c, uint32_t b) {
    asm("mad.lo.u32 %0, %2, %3, %0;\n\tdp2a.hi.s32.s32 %1, %2, %4, %1;" : "+r"(a.lo), "+r"(a.hi) : "r"(x), "r"(c), "r"(b));
}

// ---------------------------------------------------------------- a warp's state
// One listed edge.  x: coefficient (byte 3), 0 (byte 2), first-edge-of-its-row flag
// (bit 15), row within the unit (bits 8..12), first chunk within the row's segment
// (bits 0..7); y: chunks (low 16 bits), steps of the row's segment (high 16 bits); z, w: address of the source chunk that would meet the
// segment's chunk 0.
constexpr uint32_t kFirstFlag = 1u << 15;

__device__ __forceinline__ uint32_t lo32(const void *p) { return (uint32_t)(uintptr_t)p; }
__device__ __forceinline__ uint32_t hi32(const void *p) { return (uint32_t)((uintptr_t)p >> 32); }
__device__ __forceinline__ const uint4 *ptr64(uint32_t lo, uint32_t hi) {
    return reinterpret_cast<const uint4 *>(((uint64_t)hi << 32) | lo);
}

// kDepth: edges whose copies are in flight (a power of two); kAny: any_reduce.
template <uint32_t kDepth, bool kAny>
struct Warp {
    const GatherTask &t;
    uint4 *list;
    uint32_t lane, slots;  // shared address of the lane's 16 bytes in the warp's first slot
    uint32_t n;            // listed edges
    uint32_t nch, nk;      // chunks and steps of the current row segment
    uint4 *out;
    uint32_t xa, xb;       // first words of the next two edges to add
    uint32_t g0;           // lane % cpd
    Acc2 acc[kSteps][4];

    __device__ __forceinline__ Warp(const GatherTask &t_, uint4 *list_) : t(t_), list(list_) {}

    // First edge of a row segment [a, b): its output and fresh sums.
    __device__ __forceinline__ void begin_row(uint32_t row, uint32_t a, uint32_t b) {
        nch = (b - a) * t.cpd;
        nk = (nch + 31) >> 5;
        out = reinterpret_cast<uint4 *>(t.out) + ((size_t)row * t.C + a * t.cpd + lane);
        const int h = -(int)t.fast_k0;
#pragma unroll
        for (int k = 0; k < kSteps; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[k][i] = Acc2{0u, h};
    }
    // Reduce and store the current row segment.
    __device__ __forceinline__ void flush() {
        const uint4 *consts = reinterpret_cast<const uint4 *>(t.primes);
        uint4 p = make_uint4(0, 0, 0, 0), m = p;
        uint32_t g = g0;  // the primes of the lane's chunk
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            if (k >= (int)nk) break;
            if (k == 0 || t.r32) {
                p = __ldg(consts + g);
                m = __ldg(consts + CP_MAX_PRIMES / 4 + g);
            }
            auto reduced = [&](const Acc2 &a, uint32_t pi, uint32_t mi) {
                return kAny ? any_reduce(a, t.fast_k0, pi, mi, chunk_shift(pi)) : fast_reduce(a, pi, mi);
            };
            const uint4 v = make_uint4(reduced(acc[k][0], p.x, m.x), reduced(acc[k][1], p.y, m.y),
                                       reduced(acc[k][2], p.z, m.z), reduced(acc[k][3], p.w, m.w));
            stcs128_if(out + 32 * k, v, lane + 32 * k < nch ? 1u : 0u);
            g += t.r32;
            g = g >= t.cpd ? g - t.cpd : g;
        }
    }
    // Start the copies of the `steps` steps of listed edge i (one commit group).
    __device__ __forceinline__ void copy_begin(uint32_t i, uint4 &d, uint32_t &dst) const {
        d = list[i];
        dst = slots + (i & (kDepth - 1)) * kSlotBytes;
    }
    __device__ __forceinline__ void copy_step(const uint4 &d, uint32_t dst, int k) const {
        cp16_below(dst + 512u * k, ptr64(d.z, d.w) + lane + 32 * k, lane - (d.x & 0xffu) + 32u * k, d.y & 0xffffu);
    }
    // Any listed edge (an empty group past the list's end).
    __device__ __forceinline__ void copy_any(uint32_t i) {
        xa = xb;
        if (i < n) {
            uint4 d;
            uint32_t dst;
            copy_begin(i, d, dst);
            xb = d.x;
            const uint32_t steps = d.y >> 16;
#pragma unroll
            for (int k = 0; k < kSteps; ++k) {
                if (k >= (int)steps) break;
                copy_step(d, dst, k);
            }
        }
        cp_commit();
    }
    // One of the current row, of NK steps.
    template <int NK>
    __device__ __forceinline__ void copy_row(uint32_t i) {
        uint4 d;
        uint32_t dst;
        copy_begin(i, d, dst);
        xa = xb;
        xb = d.x;
#pragma unroll
        for (int k = 0; k < NK; ++k) copy_step(d, dst, k);
        cp_commit();
    }
    // Add listed edge i to the current row's sums.
    template <int NK>
    __device__ __forceinline__ void add_edge(uint32_t i) {
        const uint32_t x = kDepth == 2 ? xa : list[i].x, slot = slots + (i & (kDepth - 1)) * kSlotBytes;
        const int c = (int)x >> 24;
        cp_wait<kDepth - 1>();
#pragma unroll
        for (int k = 0; k < NK; ++k) {
            const uint4 v = lds128(slot + 512u * k);
            add_word(acc[k][0], v.x, c, x);
            add_word(acc[k][1], v.y, c, x);
            add_word(acc[k][2], v.z, c, x);
            add_word(acc[k][3], v.w, c, x);
        }
    }
    // The current row's listed edges [i, last), NK steps each.
    template <int NK>
    __device__ __forceinline__ void run_edges(uint32_t i, uint32_t last) {
#pragma unroll 1
        for (; i + kDepth < last; ++i) {
            add_edge<NK>(i);
            copy_row<NK>(i + kDepth);
        }
#pragma unroll 1
        for (; i < last; ++i) {
            add_edge<NK>(i);
            copy_any(i + kDepth);
        }
    }
    // The listed edges; a, b: the segments of the unit's rows, one per lane; firsts: bit i = edge i is
    // its row's first.
    __device__ __forceinline__ void run_list(uint32_t firsts, uint32_t row0, uint32_t a, uint32_t b, bool &open_row) {
#pragma unroll 1
        for (uint32_t i = 0; i < kDepth; ++i) copy_any(i);
        uint32_t pos = 0;
#pragma unroll 1
        while (pos < n) {
            if ((firsts >> pos) & 1u) {
                if (open_row) flush();
                const uint32_t r = (list[pos].x >> 8) & 31u;
                begin_row(row0 + r, __shfl_sync(0xffffffffu, a, r), __shfl_sync(0xffffffffu, b, r));
                open_row = true;
            }
            const uint32_t rest = (firsts >> pos) & ~1u;  // row starts after pos
            const uint32_t last = rest ? min(pos + (uint32_t)__ffs(rest) - 1u, n) : n;
            switch (nk) {
                case 1: run_edges<1>(pos, last); break;
                case 2: run_edges<2>(pos, last); break;
                case 3: run_edges<3>(pos, last); break;
                default: run_edges<4>(pos, last); break;
            }
            pos = last;
        }
        __syncwarp();
    }

    // One unit of work: its part `part` of `parts` by degrees.
    __device__ __forceinline__ void unit(const uint4 &u, uint32_t part, uint32_t parts, int v_in, int v_out, int cap_in) {
        const uint32_t row0 = u.x, nrows = u.y & 63u, e_end = u.w;
        uint2 q = u.z + lane < e_end ? __ldg(t.edges + u.z + lane) : make_uint2(0, 0xff);
        uint32_t a = 0, hi = 0;
        if (lane < nrows) {
            const uint32_t w = __ldg(t.win_out + row0 + lane);
            a = w & 0xffu;
            const int e = min(t.cap, v_out - (int)(w >> 8)) + 1;
            hi = (a == 0xffu || e <= (int)a) ? a : (uint32_t)e;
            const bool heavy = (u.y >> 6) & 1u;
            if (parts > 1 || heavy) {
                // equal shares of the degrees for the launch's parts, one pass of them at least, and
                // for the parts of a heavy row, one step of them at least
                const uint32_t len = hi - a, least = heavy ? t.seg / kSteps : t.seg;
                uint32_t i = u.y >> 8, share = (len + kSplitParts - 1) / kSplitParts;
                if (parts > 1) {
                    const uint32_t all = heavy ? kSplitParts * parts : parts;
                    i = (heavy ? i * parts : 0) + part;
                    share = (len + all - 1) / all;
                }
                share = max(share, least);
                a = min(a + i * share, hi);
                hi = min(a + share, hi);
            }
        }
        const uint32_t smask = (1u << t.src_bits) - 1u;
        bool open_row = false;
        asm volatile("griddepcontrol.wait;" ::: "memory");  // the launch before this one has finished
#pragma unroll 1
        for (uint32_t cb = u.z;;) {  // passes over the unit, at most t.seg degrees of each row at a time
            const uint32_t b = min(a + t.seg, hi);
            if (__all_sync(0xffffffffu, a >= b)) break;
#pragma unroll 1
            for (;;) {
                const uint32_t r = (q.y >> 16) & 31u;  // the edge's row
                const bool is_first = (q.y >> 21) & 1u;
                const uint32_t ra = __shfl_sync(0xffffffffu, a, r), rb = __shfl_sync(0xffffffffu, b, r);
                const uint32_t sh = (q.x >> t.src_bits) & 3u, slo = q.y & 0xffu;
                const int send = min(cap_in, v_in - (int)((q.y >> 8) & 0xffu)) + 1;  // one past the source's highest degree
                const int l0 = max((int)(slo + sh), (int)ra), l1 = min(send + (int)sh, (int)rb);
                const uint32_t len = (slo == 0xffu || l1 <= l0) ? 0u : (uint32_t)(l1 - l0) * t.cpd;
                const bool valid = cb + lane < e_end && rb > ra && (len > 0 || is_first);
                const uint32_t mask = __ballot_sync(0xffffffffu, valid);
                const uint32_t steps = valid ? ((rb - ra) * t.cpd + 31) >> 5 : 0u;  // of the row's segment
                if (valid) {
                    const uint32_t c = (uint32_t)((int)q.x >> (t.src_bits + 2)) << 24;
                    const uint32_t off = len ? ((uint32_t)l0 - ra) * t.cpd : 0u;
                    const uint4 *src = reinterpret_cast<const uint4 *>(t.in) + (size_t)(q.x & smask) * t.C +
                                       (long long)((int)ra - (int)sh) * (int)t.cpd;
                    list[__popc(mask & ((1u << lane) - 1u))] = make_uint4(
                        c | (is_first ? kFirstFlag : 0u) | (r << 8) | off, len | (steps << 16), lo32(src), hi32(src));
                }
                n = __popc(mask);
                const uint32_t firsts =
                    __reduce_or_sync(0xffffffffu, valid && is_first ? 1u << __popc(mask & ((1u << lane) - 1u)) : 0u);
                __syncwarp();
                run_list(firsts, row0, a, b, open_row);
                cb += 32;
                if (cb >= e_end) break;
                q = cb + lane < e_end ? __ldg(t.edges + cb + lane) : make_uint2(0, 0xff);
            }
            if (open_row) flush();
            open_row = false;
            a = b;
            if (__all_sync(0xffffffffu, a >= hi)) break;
            cb = u.z;
            q = cb + lane < e_end ? __ldg(t.edges + cb + lane) : make_uint2(0, 0xff);
        }
    }
};

// dv is added to the tasks' vertex counts; first: as if every task's `first` were set;
// parts: warps per unit (degree_parts).
// Launches overlap: a launch's blocks may start while the one before it drains, load
// their unit's tables (which no launch writes) and only then wait for it.
template <int N, uint32_t kDepth, bool kAny>
__global__ void __launch_bounds__(32 * kWarps, kChunkBlocksPerSM)
    gather_chunk_kernel(const __grid_constant__ TaskPack<N> pack, int n_tasks, uint32_t n_units, uint32_t parts, int dv,
                        int first) {
    extern __shared__ __align__(128) uint8_t slots[];  // per warp: kDepth slots of kSlotBytes
    __shared__ uint4 lists[kWarps][32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t id = blockIdx.x * kWarps + warp, part = 0;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (id >= n_units * parts) return;
    if (parts > 1) {
        part = id / n_units;
        id -= part * n_units;
    }
    const GatherTask &t = pack.t[find_task(pack, n_tasks, id)];
    Warp<kDepth, kAny> w(t, lists[warp]);
    w.lane = lane;
    w.g0 = lane % t.cpd;
    w.slots = smem_addr(slots) + warp * kDepth * kSlotBytes + lane * 16u;
    w.unit(__ldg(t.units + (id - t.block_begin)), part, parts, t.v_in + dv, t.v_out + dv, first || t.first ? 0 : t.cap);
}

bool chunk_usable(const GatherTask &t) { return t.chunk != 0; }

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t a, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok != 0;
}
// Wait for the phase of parity `parity` to complete; false once the deadline passes.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, long long deadline) {
    while (!mbar_try_wait(a, parity))
        if (clock64() > deadline) return false;
    return true;
}

// Diagnostic: a wait that can never complete (an mbarrier nothing arrives on),
// bounded by `cycles`; on expiry it sets bit 16 of *err and returns.  (The gathers
// themselves wait for nothing but their own copies and the launch before.)
__global__ void wait_timeout_kernel(long long cycles, int *err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) mbar_init(smem_addr(&bar), 1);
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(smem_addr(&bar), 0, clock64() + cycles)) atomicOr_system(err, 1 << 16);
}

int debug_wait_timeout(long long cycles, cudaStream_t st) {
    wait_timeout_kernel<<<1, 32, 0, st>>>(cycles, device_error_flag());
    CP_CUDA_TRY(cudaGetLastError());
    return check_device_error(st);
}

// Launches of few units keep four edges in flight instead of two: there the chain of one
// warp's edges is what they last, not the SMs' throughput.  Four take 16 KB a block, 12
// blocks of two warps on each of the 152 SMs; up to two waves of those gain (k = 17 sweep
// 457 -> 420 us, triangular 12x12 on one prime 793 -> 714, square 12x13 on 8 primes 1227 ->
// 1180), a third, just begun, loses (Potts 10x10, 8 000 units: 1212 -> 1286).  Eight in
// flight gain no more (429 us).
constexpr uint32_t kFewUnits = 2 * 24 * 152;

// Parts that the degrees of a launch's rows are dealt out in, a warp for each part of a
// unit: as many as the longest row has passes, where that leaves the launch below
// kFewUnits.  A warp walks its passes one after another, so a strip of few states and
// long rows (square 4 x 200 on 32 primes as integers: up to 50 passes a row) took 20.2 ms on one
// part, 4.4 with a block for the columns of a row, and takes 1.4 on these.
static uint32_t degree_parts(const GatherTask *tasks, int n_tasks, uint32_t n_units, int dv) {
    uint32_t passes = 1;
    for (int k = 0; k < n_tasks; ++k) {
        const uint32_t degrees = (uint32_t)std::min(tasks[k].cap, std::max(tasks[k].v_out + dv, 0)) + 1;
        passes = std::max(passes, (degrees + tasks[k].seg - 1) / tasks[k].seg);
    }
    return std::min(passes, std::max(1u, kFewUnits / std::max(1u, n_units)));
}

int launch_gather_chunk(const GatherTask *tasks, int n_tasks, uint32_t n_units, cudaStream_t st, int dv, bool first) {
    return for_packs(tasks, n_tasks, n_units, [&](const auto &pack, int n, uint32_t units) -> int {
        constexpr int N = sizeof(pack.t) / sizeof(GatherTask);
        if (!units) return CP_OK;
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        const uint32_t parts = degree_parts(pack.t, n, units, dv);
        cfg.gridDim = dim3((units * parts + kWarps - 1) / kWarps);
        cfg.blockDim = dim3(32 * kWarps);
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        bool any = false;
        for (int k = 0; k < n; ++k) any = any || !pack.t[k].fast;
        auto go = [&](auto depth, auto any_prime) -> cudaError_t {
            cfg.dynamicSmemBytes = kWarps * decltype(depth)::value * kSlotBytes;
            return cudaLaunchKernelEx(&cfg, gather_chunk_kernel<N, decltype(depth)::value, decltype(any_prime)::value>, pack,
                                      n, units, parts, dv, first ? 1 : 0);
        };
        auto pick = [&](auto depth) { return any ? go(depth, std::true_type()) : go(depth, std::false_type()); };
        CP_CUDA_TRY(units * parts <= kFewUnits ? pick(std::integral_constant<uint32_t, 4>())
                                       : pick(std::integral_constant<uint32_t, 2>()));
        return CP_OK;
    });
}

}  // namespace cp

// Diagnostic: the kernel's sums and reductions on given values (one thread per value).
namespace cp {
__global__ void debug_chunk_sum_kernel(const int *coefs, const int *words, int n_edges, const uint32_t *s,
                                       const uint32_t *pr, int n, int any_prime, int *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint32_t p = pr[k], k0 = fast_offset(s[k]), t = chunk_shift(p);
    const uint32_t m = (uint32_t)((1ull << (32 + t)) / p);  // chunk_magic
    Acc2 a{0u, -(int)k0};
    for (int e = 0; e < n_edges; ++e) {
        const size_t i = (size_t)k * n_edges + e;
        add_word(a, (uint32_t)words[i], coefs[i], (uint32_t)coefs[i] << 24);
    }
    out[k] = (int)(any_prime ? any_reduce(a, k0, p, m, t) : fast_reduce(a, p, m));
}
}  // namespace cp

extern "C" int cp_debug_chunk_sum(const int32_t *coefs_host, const int32_t *words_host, int n_edges,
                                  const uint32_t *s_host, const uint32_t *p_host, int n, int any_prime,
                                  int32_t *out_host) {
    using namespace cp;
    if (n < 0 || n_edges < 0 || (n > 0 && (!coefs_host || !words_host || !s_host || !p_host || !out_host)))
        return fail(CP_EINVAL, "bad arguments");
    for (int k = 0; k < n; ++k) {
        const uint32_t p = p_host[k];
        if (p < 2 || p >= (1u << 31)) return fail(CP_EINVAL, "p must be in [2, 2^31)");
        if (s_host[k] >= kChunkMaxSum || (!any_prime && !fast_ok(s_host[k], p)))
            return fail(CP_EINVAL, "the coefficient sum's bound does not suit the reduction");
        uint64_t sum = 0;
        for (int e = 0; e < n_edges; ++e) {
            const long long c = coefs_host[(size_t)k * n_edges + e], x = words_host[(size_t)k * n_edges + e];
            if (c < -(int)kChunkMaxCoef || c > (int)kChunkMaxCoef) return fail(CP_EINVAL, "|coefficient| must be at most 127");
            if (x < -(long long)p || x > (long long)p) return fail(CP_EINVAL, "|word| must be at most p");
            sum += (uint64_t)(c < 0 ? -c : c);
        }
        if (sum > s_host[k]) return fail(CP_EINVAL, "sum of |coefficient| exceeds its bound");
    }
    if (n == 0) return CP_OK;
    const size_t words = (size_t)n * n_edges;
    uint32_t *d = nullptr;  // coefficients, words, bounds, primes, results
    int rc = dev_alloc((void **)&d, 4 * (2 * words + 3 * (size_t)n));
    if (rc) return rc;
    int *c_d = (int *)d, *x_d = c_d + words, *o_d = x_d + words;
    uint32_t *s_d = (uint32_t *)(o_d + n), *p_d = s_d + n;
    cudaError_t e = cudaMemcpy(c_d, coefs_host, 4 * words, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(x_d, words_host, 4 * words, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(s_d, s_host, 4ull * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(p_d, p_host, 4ull * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        debug_chunk_sum_kernel<<<(n + 255) / 256, 256>>>(c_d, x_d, n_edges, s_d, p_d, n, any_prime, o_d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out_host, o_d, 4ull * n, cudaMemcpyDeviceToHost);
    dev_free(d);
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("cp_debug_chunk_sum: ") + cudaGetErrorString(e));
    return CP_OK;
}

// Diagnostic: a 32-bit reduction of two-halves sums on given values (one thread per
// value), for an entry point alone: no gather uses it.
namespace cp {
// For primes p >= 2^17 the sums start at B = p 2^15 (a multiple of p above
// |sum c x| <= S p), so u = hi 2^16 + lo lies in (0, p 2^16), and the quotient
// estimate of modred.cuh with s = b - 2 >= 16 takes h = floor(u / 2^s) =
// floor((hi + floor(lo / 2^16)) / 2^(s-16)) (c = s - 16); as u < 2^(b+16) the
// error terms stay below 2^-14 + 1/2, so r = u - q p (taken modulo 2^32, with u's
// low word hi 2^16 + lo) lies in [0, 2p).  Returns r reduced (full) or r - p.
__device__ __forceinline__ uint32_t reduce_halves(const Acc2 &a, uint32_t p, uint32_t m, uint32_t c, bool full) {
    const uint32_t h = (uint32_t)(a.hi + ((int)a.lo >> 16)) >> c;
    const uint32_t q = __umulhi(h, m);
    const uint32_t r = ((uint32_t)a.hi << 16) + a.lo - q * p;
    return full ? min(r, r - p) : r - p;
}

__global__ void debug_halves_kernel(const int *lo, const int *hi, const uint32_t *pr, int n, int full, uint32_t *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const ModRed mr = modred_make(pr[k]);
    out[k] = reduce_halves(Acc2{(uint32_t)lo[k], hi[k]}, mr.p, mr.m, mr.s - 16, full != 0);
}
}  // namespace cp

extern "C" int cp_debug_reduce_halves(const int32_t *lo_host, const int32_t *hi_host, const uint32_t *p_host, int n,
                                      int full, uint32_t *out_host) {
    using namespace cp;
    if (n < 0 || (n > 0 && (!lo_host || !hi_host || !p_host || !out_host))) return fail(CP_EINVAL, "bad arguments");
    for (int k = 0; k < n; ++k) {
        const uint32_t p = p_host[k];
        if (p < (1u << 17) || p >= (1u << 31)) return fail(CP_EINVAL, "p must be in [2^17, 2^31)");
        const long long u = (long long)hi_host[k] * 65536 + lo_host[k];
        if (u <= 0 || u >= (long long)p * 65536) return fail(CP_EINVAL, "hi 2^16 + lo must lie in (0, p 2^16)");
    }
    if (n == 0) return CP_OK;
    int *lo_d = nullptr, *hi_d = nullptr;
    uint32_t *p_d = nullptr, *o_d = nullptr;
    int rc = dev_alloc((void **)&lo_d, 4ull * n);
    if (!rc) rc = dev_alloc((void **)&hi_d, 4ull * n);
    if (!rc) rc = dev_alloc((void **)&p_d, 4ull * n);
    if (!rc) rc = dev_alloc((void **)&o_d, 4ull * n);
    cudaError_t e = cudaSuccess;
    if (!rc) {
        e = cudaMemcpy(lo_d, lo_host, 4ull * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(hi_d, hi_host, 4ull * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(p_d, p_host, 4ull * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            debug_halves_kernel<<<(n + 255) / 256, 256>>>(lo_d, hi_d, p_d, n, full, o_d);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpy(out_host, o_d, 4ull * n, cudaMemcpyDeviceToHost);
    }
    dev_free(lo_d);
    dev_free(hi_d);
    dev_free(p_d);
    dev_free(o_d);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("cp_debug_reduce_halves: ") + cudaGetErrorString(e));
    return CP_OK;
}
