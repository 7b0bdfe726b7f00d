// lookahead.cu -- the default search form's production kernel (layout REGP):
// Algorithm 2 with a one-row look-ahead.
//
// A child is entered only if its own row has a free column AND the row after
// that would still have one under the child's state. Both tests are NORs of
// the same masks, and the second one's shifted masks are the ones that the
// child's frame needs anyway, so the look-ahead costs one logic instruction
// and no state. It removes a fifth of the steps and a quarter of the stack
// traffic at N = 18 (counted on a sampled tree: 14.8 M steps, 9.4 M entered
// frames -> 11.9 M, 7.3 M).
//
// What bounds it (N = 18, d = 7, 7.4 M subproblems in one launch, 20.0 ms
// against 26.2 ms for the same search without look-ahead): issue slots 85 %, the ALU pipe 84 % and the shared
// memory data path 86 % at once, so a step has to lose instructions, ALU work
// and stack traffic together to get faster. Tried and slower, all on that
// workload: high-half multiplies in place of the right shifts (22.6 ms), a
// compare for the last column in place of the population count (22.4 ms),
// dropping the candidates that a forced next row rules out (25.7 ms: five more
// instructions for 16 % fewer steps).
//
// Records that are few or heavy are split into units (look_kernel_split) by the
// digits of the unit's index, so that splitting needs no memory and no launch of
// its own; the lanes of a warp that has nothing left to take share its last
// subtrees. Before, one lane searched each record: 2048 records of N = 22, d = 7
// took 509 ms of which 3.5 ms were work, now 4.3 ms; N = 14 from d = 3 1.97 ms,
// now 0.07 ms; N = 18 from d = 5 53.6 ms, now 18.5 ms.
#include "nq_internal.h"

namespace nqi {
namespace {

constexpr int kLookSteps = 31;  // steps between bookkeeping points

// The sentinel frame, in slot 0 of every stack: whatever candidate bit p is
// taken, cols + p, L + 2p and R + p/2 together cover all 32 bits (each of the
// three patterns keeps one bit of every pair of columns, also where p's carry
// moves it), so a child is never live. All 32 bits are candidates, which holds
// 32 idle steps: one frame lasts a whole round.
constexpr uint32_t kSentC = 0x55555555u, kSentL = 0xAAAAAAAAu, kSentR = 0x55555555u;
constexpr uint32_t kSentAv = 0xFFFFFFFFu;
// Under masks: the frame above row 31, whose masks are 0, with no diagonals.
constexpr uint32_t kSentMaskedC = 31u << kRowShift;
static_assert(kLookSteps < 32, "an idle lane must not use up the sentinel's candidates");

extern __shared__ __align__(16) unsigned char look_smem[];

__device__ __forceinline__ void look_error(int *status, int code) {
    if (status) atomicCAS(status, 0, code);
}

// One step. The top frame is in registers: c = columns taken (columns >= N
// pre-set), L and R = the diagonals as they reach the NEXT row before this
// row's queen is placed (kept shifted, so that placing p adds 2p and p/2 to
// them and nothing else), av = candidates left. (c, L, R, av) of a frame with
// candidates left is saved in 16 bytes of the lane's stack.
//   p          the lowest candidate, ar the others
//   c2 l2 r2   the child's masks, a2 its free columns
//   L2 R2      the same masks one row on, b2 that row's free columns
// Every sum is of disjoint bits, so the integer multiply-adds by the run-time
// multipliers m1 = 1, m2 = 2, mneg = 2^32 - 1 are exact; they issue on the FMA
// pipe, which this integer loop would otherwise leave idle.
// A solution is counted when the child has one free column left (rows 0..N-2
// hold queens) and its row has it free; such a child may be entered too (its
// look-ahead row does not exist), which costs a step and finds nothing.
__device__ __forceinline__ void look_step(uint32_t &c, uint32_t &L, uint32_t &R, uint32_t &av,
                                          uint32_t &top, const uint32_t stride, uint32_t &s32,
                                          const uint32_t m1, const uint32_t m2,
                                          const uint32_t mneg) {
    const uint32_t p = av & (av * mneg);
    const uint32_t ar = p * mneg + av;
    const uint32_t c2 = p * m1 + c;
    const uint32_t l2 = L + 2u * p;
    const uint32_t r2 = (p >> 1) + R;
    const uint32_t L2 = l2 * m2;
    const uint32_t R2 = r2 >> 1;
    const uint32_t pc = (uint32_t)__popc(c2);
    // %0..%5 c, L, R, av, top, s32; %6 l2, %7 pc, %8 ar, %9 c2, %10 r2,
    // %11 stride, %12 L2, %13 R2. lop3 table 0x01: NOR of its three inputs;
    // the predicate beside the result says that it is not zero (and-ed with
    // the last operand).
    asm volatile(
        "{\n\t"
        ".reg .pred ptrue, plive, ppush, pcnt, psave, ppop;\n\t"
        ".reg .b32 a2, b2;\n\t"
        "setp.eq.u32 ptrue, 0, 0;\n\t"
        "lop3.and.b32 a2|plive, %9, %6, %10, 0x01, ptrue;\n\t"    // the child's row has a column
        "lop3.and.b32 b2|ppush, %9, %12, %13, 0x01, plive;\n\t"   // ... and so has the row after
        "setp.eq.and.u32 pcnt, %7, 31, plive;\n\t"                // one column left, and free: a solution
        "@pcnt add.u32 %5, %5, 1;\n\t"
        "setp.ne.and.u32 psave, %8, 0, ppush;\n\t"                // entered with candidates left: save
        "setp.eq.and.u32 ppop, %8, 0, !ppush;\n\t"                // nothing left, nothing entered: pop
        "@psave st.shared.v4.u32 [%4], {%0, %1, %2, %8};\n\t"
        "@psave add.u32 %4, %4, %11;\n\t"
        "@ppop sub.u32 %4, %4, %11;\n\t"
        "selp.b32 %3, a2, %8, ppush;\n\t"
        "@ppush mov.b32 %0, %9;\n\t"
        "@ppush mov.b32 %1, %12;\n\t"
        "@ppush mov.b32 %2, %13;\n\t"
        "@ppop ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n\t"
        "}"
        : "+r"(c), "+r"(L), "+r"(R), "+r"(av), "+r"(top), "+r"(s32)
        : "r"(l2), "r"(pc), "r"(ar), "r"(c2), "r"(r2), "r"(stride), "r"(L2), "r"(R2)
        : "memory");
}

// The same step under per-row masks (partial-board queries): the row rides in
// bits 27..31 of c, already counted up for the child (c = columns | (row + 1)
// << 27), so entering a child adds the next row where look_step moves a
// register. The masks of the child's row and of the row after it come as one
// 8-byte load whose address depends on the frame alone; rows at or below the
// last have mask 0 after them, so a last-row child is counted and not entered.
// The last row is a compare of the row field, no population count.
// Six queries of two queens at N = 16: 98 ms with the host enumerating the
// subproblems on one core, 1.8 ms as one split record (of which 1.2 ms are the
// six calls' own cost).
__device__ __forceinline__ void look_step_masked(uint32_t &c, uint32_t &L, uint32_t &R,
                                                 uint32_t &av, uint32_t &top,
                                                 const uint32_t stride, const uint32_t table,
                                                 const uint32_t thr, uint32_t &s32,
                                                 const uint32_t m1, const uint32_t m2,
                                                 const uint32_t mneg) {
    uint32_t A1, A2;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];"
                 : "=r"(A1), "=r"(A2)
                 : "r"(((c >> kRowShift) << 3) + table)
                 : "memory");
    const uint32_t p = av & (av * mneg);
    const uint32_t ar = p * mneg + av;
    const uint32_t c2 = p * m1 + c;
    const uint32_t l2 = L + 2u * p;
    const uint32_t r2 = (p >> 1) + R;
    const uint32_t L2 = l2 * m2;
    const uint32_t R2 = r2 >> 1;
    const uint32_t t1 = c2 | l2 | r2, t2 = c2 | L2 | R2;
    // operands as in look_step, but %6 t1, %7 thr, %10 t2, %14 A1, %15 A2;
    // lop3 table 0x30: the first input without the second
    asm volatile(
        "{\n\t"
        ".reg .pred ptrue, plive, ppush, pcnt, psave, ppop;\n\t"
        ".reg .b32 a2, b2;\n\t"
        "setp.eq.u32 ptrue, 0, 0;\n\t"
        "lop3.and.b32 a2|plive, %14, %6, 0, 0x30, ptrue;\n\t"    // the child's row has a column
        "lop3.and.b32 b2|ppush, %15, %10, 0, 0x30, plive;\n\t"   // ... and so has the row after
        "setp.ge.and.u32 pcnt, %9, %7, plive;\n\t"               // the last row has one: a solution
        "@pcnt add.u32 %5, %5, 1;\n\t"
        "setp.ne.and.u32 psave, %8, 0, ppush;\n\t"
        "setp.eq.and.u32 ppop, %8, 0, !ppush;\n\t"
        "@psave st.shared.v4.u32 [%4], {%0, %1, %2, %8};\n\t"
        "@psave add.u32 %4, %4, %11;\n\t"
        "@ppop sub.u32 %4, %4, %11;\n\t"
        "selp.b32 %3, a2, %8, ppush;\n\t"
        "@ppush add.u32 %0, %9, %16;\n\t"
        "@ppush mov.b32 %1, %12;\n\t"
        "@ppush mov.b32 %2, %13;\n\t"
        "@ppop ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n\t"
        "}"
        : "+r"(c), "+r"(L), "+r"(R), "+r"(av), "+r"(top), "+r"(s32)
        : "r"(t1), "r"(thr), "r"(ar), "r"(c2), "r"(t2), "r"(stride), "r"(L2), "r"(R2), "r"(A1),
          "r"(A2), "n"(1u << kRowShift)
        : "memory");
}

// One unit of split work: the part of a record's subtree that the digits of s
// name. Level j (row d + j) has a digit of several bits, the most significant
// level first. Every level but the last: the t-th free column, or nothing
// when there are fewer (the digit covers every column the row could have
// free). The last level: the free columns t, t + R, t + 2R, ... of R = 2^bits,
// so nothing is left out there with a small digit. The units of a record
// partition its solutions.
//   returns  0: nothing here, 1: search from (c, l, r) with candidates av
//            (l, r as they reach this row), 2: *found solutions and no search
//   skip     units to the next one that may hold something
// MASKED: row `row` takes only the columns of its mask (table: 8 bytes a row),
// and the board ends after `rows` rows; c holds no pre-set columns.
template <bool MASKED>
__device__ __forceinline__ int split_unit(uint32_t s, const int levels, uint32_t digits,
                                          int shift, uint32_t &c, uint32_t &l, uint32_t &r,
                                          uint32_t &av, uint32_t &found, uint32_t &skip,
                                          const uint32_t table, uint32_t row, uint32_t rows) {
    skip = 1u;
    for (int j = 0; j < levels; ++j, digits >>= 4, ++row) {
        const uint32_t bits = digits & 15u;
        const uint32_t here = s & ((1u << shift) - 1u);  // this level's digit and those below
        shift -= (int)bits;
        if (MASKED ? row == rows : c == ~0u) {  // every row is placed: the solution belongs to the unit of zeros
            skip = (1u << (shift + (int)bits)) - here;
            found = here == 0u ? 1u : 0u;
            return 2;
        }
        uint32_t x = ~(c | l | r);
        if (MASKED) {
            uint32_t mask;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(mask) : "r"(table + 8u * row) : "memory");
            x &= mask;
        }
        for (uint32_t t = here >> shift; t && x; --t) x &= x - 1u;
        if (x == 0u) {  // and nothing at any higher value of this digit
            skip = (1u << (shift + (int)bits)) - here;
            return 0;
        }
        const uint32_t p = x & (0u - x);
        if (j + 1 < levels) {
            c |= p;
            l = (l | p) << 1;
            r = (r | p) >> 1;
        } else {
            av = p;
            for (x ^= p; x;) {
                for (uint32_t t = (1u << bits) - 1u; t && x; --t) x &= x - 1u;
                const uint32_t q = x & (0u - x);
                av |= q;
                x ^= q;
            }
        }
    }
    // the last row (the last level's row is row - 1 now): each candidate is a solution
    if (MASKED ? row == rows : __popc(c) == 31) {
        found = (uint32_t)__popc(av);
        return 2;
    }
    return 1;
}

// The persistent search: every warp takes ranges of record indices (the first
// one by its number, the others from the work cursor) and hands them to its
// lanes as they become idle. One atomic serves a whole range, and a launch
// whose records fit the first ranges needs no cursor. Consecutive ranges go to
// different blocks first, so that few records spread over the SMs.
// SPLIT: the indices are units (split_unit), 2^split_shift to a record, and a
// unit's count is added into its record's entry (zeroed before the launch).
// Units that cannot hold anything are passed over in one go: the warp's
// position moves on by the last asking lane's skip.
// MASKED (split only): one table of row masks for the launch, above the stacks.
template <bool SPLIT, bool MASKED>
__device__ __forceinline__ void look_body(const SearchArgs &a) {
    static_assert(SPLIT || !MASKED, "masked searches are split");
    constexpr uint32_t kSC = MASKED ? kSentMaskedC : kSentC, kSL = MASKED ? 0u : kSentL,
                       kSR = MASKED ? 0u : kSentR;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(look_smem);
    const uint32_t stride = stack_slot_offset(blockDim.x, 0u, 1u, 16u);
    const uint32_t base = sbase + stack_slot_offset(blockDim.x, threadIdx.x, 0u, 16u);
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t m1 = a.mul[0], m2 = a.mul[1], mneg = a.mul[2];
    const uint32_t range = a.range;
    const uint64_t total = SPLIT ? a.n << a.split_shift : a.n;
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);

    const uint32_t table = sbase + (uint32_t)a.slots * stride;
    const uint32_t thr = MASKED ? (uint32_t)(a.expect_n - 1) << kRowShift : 0u;
    if (MASKED) {
        if (threadIdx.x < 32u)
            asm volatile("st.shared.v2.u32 [%0], {%1, %2};"
                         :
                         : "r"(table + 8u * threadIdx.x), "r"(a.allowed[threadIdx.x]),
                           "r"(threadIdx.x < 31u ? a.allowed[threadIdx.x + 1u] : 0u)
                         : "memory");
        __syncthreads();
    }

    uint32_t c = kSC, L = kSL, R = kSR, av = kSentAv, top = base;
    uint32_t bot = base;        // SPLIT: the lane's sentinel slot (frames below were given away)
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};"
                 :
                 : "r"(base), "r"(c), "r"(L), "r"(R), "r"(av)
                 : "memory");

    bool busy = false;          // a subproblem is being searched
    uint64_t idx = 0;           // its record
    uint32_t wn = 0;            // its weight | N << 2
    uint64_t sol = 0;
    uint64_t wsum = 0;          // weighted solutions not yet in totals[wsum_n]
    uint32_t wsum_n = 0;
    // the warp's range (the same in every lane)
    uint64_t next = ((uint64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * range;
    uint32_t rem = next < total ? (uint32_t)(total - next < range ? total - next : range) : 0u;
    bool exhausted = a.cursor == nullptr;

    auto finish = [&](uint64_t i, uint64_t s, uint32_t w_n) {
        if (SPLIT) {
            if (a.counts && s)
                atomicAdd(reinterpret_cast<unsigned long long *>(&a.counts[i]),
                          (unsigned long long)s);
        } else if (a.counts) {
            a.counts[i] = s;
        }
        if (a.totals && s) {
            const uint32_t n = w_n >> 2;
            if (n != wsum_n && wsum != 0) {
                atomicAdd(reinterpret_cast<unsigned long long *>(&a.totals[wsum_n]),
                          (unsigned long long)wsum);
                wsum = 0;
            }
            wsum_n = n;
            wsum += (uint64_t)(w_n & 3u) * s;
        }
    };

    for (;;) {
        const bool idle = top == (SPLIT ? bot : base);  // on the sentinel
        if (idle) {
            if (busy) finish(idx, sol, wn);
            busy = false;
            if (SPLIT) bot = top = base;
            c = kSC;
            L = kSL;
            R = kSR;
            av = kSentAv;
        }
        bool need = idle;
        unsigned need_mask = __ballot_sync(~0u, need);
        while (need_mask) {
            if (rem == 0u) {
                if (exhausted || (SPLIT && __popc(need_mask) < a.refill)) break;
                unsigned long long f = 0;
                if (lane == 0) f = atomicAdd(a.cursor, (unsigned long long)range);
                next = __shfl_sync(~0u, f, 0) + warps * range;
                if (next >= total) {
                    exhausted = true;
                    break;
                }
                rem = total - next < range ? (uint32_t)(total - next) : range;
            }
            const uint32_t ready = rem;
            const uint32_t rank = __popc(need_mask & lt_mask);
            uint32_t skip = 1u;
            if (need && rank < ready) {
                uint64_t at = next + rank;
                uint32_t s = 0u;  // the unit's digits
                if (SPLIT) {
                    s = (uint32_t)at & ((1u << a.split_shift) - 1u);
                    at >>= a.split_shift;
                }
                const uint64_t pi = a.order ? a.n - 1 - at : at;
                const uint4 P = __ldg(reinterpret_cast<const uint4 *>(a.pre) + pi);
                const uint32_t n = (P.w >> 2) & 31u, d = (P.w >> 7) & 31u, w = P.w & 3u;
                const uint32_t last = (n >= 1u) ? (0xFFFFFFFFu >> (32u - n)) : 0u;
                const bool ok = n >= 1u && (a.expect_n == 0 || (int)n == a.expect_n) &&
                                (w == 1u || w == 2u) && d <= n && (P.x & ~last) == 0u &&
                                (uint32_t)__popc(P.x) == d;
                // (the stack holds the sentinel and the ancestors down to row N-2
                // of a record with a.rows rows left)
                if (!ok || (d + 1u < n && (int)(n - d) > a.rows)) {
                    look_error(a.status, ok ? NQ_ESTACK : NQ_EINVAL);
                    finish(pi, 0, 0);
                    if (SPLIT) skip = (1u << a.split_shift) - s;
                } else if (SPLIT) {
                    uint32_t cc = MASKED ? P.x : P.x | ~last;
                    uint32_t ll = P.y, rr = P.z & last, a0 = 0, found = 0;
                    const int got = split_unit<MASKED>(s, a.levels, a.digits, a.split_shift, cc,
                                                       ll, rr, a0, found, skip, table, d, n);
                    if (got == 2) finish(pi, found, w | (n << 2));
                    if (got == 1) {
                        idx = pi;
                        wn = w | (n << 2);
                        sol = 0;
                        busy = true;
                        c = MASKED ? cc | ((d + (uint32_t)a.levels) << kRowShift) : cc;
                        L = ll << 1;
                        R = rr >> 1;
                        av = a0;
                        top = base + stride;
                        need = false;
                    }
                } else {
                    const uint32_t c0 = P.x | ~last;
                    const uint32_t l0 = P.y, r0 = P.z & last;
                    const uint32_t a0 = ~(c0 | l0 | r0);
                    if (d == n) {
                        finish(pi, 1, w | (n << 2));  // the prefix is a solution
                    } else if (d + 1u == n || a0 == 0u) {
                        finish(pi, (uint64_t)__popc(a0), w | (n << 2));  // last row or dead end
                    } else {
                        idx = pi;
                        wn = w | (n << 2);
                        sol = 0;
                        busy = true;
                        c = c0;
                        L = l0 << 1;
                        R = r0 >> 1;
                        av = a0;
                        top = base + stride;
                        need = false;
                    }
                }
            }
            const uint32_t asked = __popc(need_mask);
            uint32_t taken = asked < ready ? asked : ready;
            if (SPLIT && asked <= ready) {  // every asker had a unit: pass over empty ones
                taken += __shfl_sync(~0u, skip, 31 - __clz((int)need_mask)) - 1u;
                taken = taken < rem ? taken : rem;
            }
            next += taken;
            rem -= taken;
            need_mask = __ballot_sync(~0u, need);
        }
        if (need_mask == ~0u) break;  // the whole warp is idle, and nothing is left

        if (SPLIT && need_mask && rem == 0u) {
            // Each idle lane takes the shallowest saved frame of a busy lane of
            // its warp, and leaves a sentinel in its place.
            const bool giver = !need && top > bot + stride;
            const unsigned givers = __ballot_sync(~0u, giver);
            if (givers) {
                const uint32_t pairs = min(__popc(need_mask), __popc(givers));
                const uint32_t rank = __popc((need ? need_mask : givers) & lt_mask);
                const bool taker = need && rank < pairs;
                const int from = taker ? (int)__fns(givers, 0, (int)rank + 1) : (int)lane;
                const uint32_t slot = __shfl_sync(~0u, bot + stride, from);
                const uint64_t i = __shfl_sync(~0u, idx, from);
                const uint32_t w_n = __shfl_sync(~0u, wn, from);
                if (taker) {
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(c), "=r"(L), "=r"(R), "=r"(av)
                                 : "r"(slot)
                                 : "memory");
                    idx = i;
                    wn = w_n;
                    sol = 0;
                    busy = true;
                    top = base + stride;
                }
                __syncwarp();
                if (giver && rank < pairs) {
                    bot += stride;
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};"
                                 :
                                 : "r"(bot), "r"(kSC), "r"(kSL), "r"(kSR), "r"(kSentAv)
                                 : "memory");
                }
                __syncwarp();
            }
        }

        uint32_t s32 = 0;
#pragma unroll
        for (int j = 0; j < kLookSteps; ++j) {
            if constexpr (MASKED)
                look_step_masked(c, L, R, av, top, stride, table, thr, s32, m1, m2, mneg);
            else
                look_step(c, L, R, av, top, stride, s32, m1, m2, mneg);
        }
        sol += s32;
    }

    if (a.totals) {
        const unsigned has = __ballot_sync(~0u, wsum != 0);
        if (has) {
            const uint32_t n0 = __shfl_sync(~0u, wsum_n, __ffs(has) - 1);
            if (__all_sync(~0u, wsum == 0 || wsum_n == n0)) {
                uint64_t v = wsum;
                for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(~0u, v, o);
                if (lane == 0)
                    atomicAdd(reinterpret_cast<unsigned long long *>(&a.totals[n0]),
                              (unsigned long long)v);
            } else if (wsum) {
                atomicAdd(reinterpret_cast<unsigned long long *>(&a.totals[wsum_n]),
                          (unsigned long long)wsum);
            }
        }
    }
}

__global__ void __maxnreg__(48) look_kernel(const SearchArgs a) { look_body<false, false>(a); }
__global__ void __maxnreg__(48) look_kernel_split(const SearchArgs a) {
    look_body<true, false>(a);
}
__global__ void __maxnreg__(48) look_kernel_masked(const SearchArgs a) {
    look_body<true, true>(a);
}

}  // namespace

void *look_kernel_ptr(bool split, bool masked) {
    return masked  ? reinterpret_cast<void *>(&look_kernel_masked)
           : split ? reinterpret_cast<void *>(&look_kernel_split)
                   : reinterpret_cast<void *>(&look_kernel);
}

}  // namespace nqi
