// lookahead.cu -- the default search form's production kernels (layout REGP):
// Algorithm 2 with a one-row look-ahead, on whole records, on records split into
// units, under row masks (nq_count_constrained), and fed by a ring (the server).
//
// A child is entered only if its own row has a free column AND the row after
// that would still have one under the child's state. Both tests are NORs of
// the same masks, and the second one's shifted masks are the ones that the
// child's frame needs anyway, so the look-ahead costs one logic instruction
// and no state. It removes a fifth of the steps and a quarter of the stack
// traffic at N = 18 (counted on a sampled tree: 14.8 M steps, 9.4 M entered
// frames -> 11.9 M, 7.3 M).
//
// What bounds it (N = 18, d = 7, 7.4 M subproblems in one launch, 19.4 ms
// against 26.2 ms for the same search without look-ahead): issue slots 85 %, the
// ALU pipe 84 % and the shared memory data path 86 % at once, so a step has to
// lose instructions, ALU work and stack traffic together to get faster. Tried
// and slower, all on that workload, against 20.0 ms for the step as it is in a
// bare kernel: high-half multiplies in place of the right shifts (22.6 ms), a
// compare for the last column in place of the population count (22.4 ms),
// dropping the candidates that a forced next row rules out (25.7 ms: five more
// instructions for 16 % fewer steps).
//
// Records that are few or heavy are split (look_kernel_split) by the digits of an
// index, so that splitting needs no memory and no launch of its own; a warp's
// idle lanes take frames of its busy ones when its range is used up. Before, one
// lane searched each record: 2048 records of N = 22, d = 7 took 509 ms of which
// 3.5 ms were work, now 4.1 ms; N = 14 from d = 3 1.97 ms, now 0.057 ms (about 8
// us of work: searches of about 100 steps are as small as pays); N = 18 from d =
// 5 53.6 ms, now 17.8 ms.
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
// Under masks: the frame above a row that no board has, whose mask is 0, with no
// diagonals.
constexpr uint32_t kSentMaskedC = (uint32_t)kSentinelRow << kRowShift;
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
// register. The masks of the child's row and of the row after it are loaded from
// a table whose address depends on the frame alone: 8 bytes a row holding both
// (ROW = 8, one load), or a word a row (ROW = 4, two loads, half the table: the
// server keeps one for each request). Rows at or below the last have mask 0
// after them, so a last-row child is counted and not entered.
// The last row is a compare of the row field, no population count.
// Six queries of two queens at N = 16: 98 ms with the host enumerating the
// subproblems on one core, 0.50 ms as one split record (of which 0.2 ms are the
// six calls' own cost).
template <uint32_t ROW>
__device__ __forceinline__ void look_step_masked(uint32_t &c, uint32_t &L, uint32_t &R,
                                                 uint32_t &av, uint32_t &top,
                                                 const uint32_t stride, const uint32_t table,
                                                 const uint32_t thr, uint32_t &s32,
                                                 const uint32_t m1, const uint32_t m2,
                                                 const uint32_t mneg) {
    uint32_t A1, A2;
    const uint32_t at = (c >> kRowShift) * ROW + table;
    if constexpr (ROW == 8u)
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(A1), "=r"(A2) : "r"(at) : "memory");
    else
        asm volatile("ld.shared.u32 %0, [%2];\n\tld.shared.u32 %1, [%2+4];"
                     : "=&r"(A1), "=r"(A2)
                     : "r"(at)
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

// Split work: the part of a record's subtree that the digits of s name. Level j
// (row d + j) has a digit of several bits, the most significant level first,
// which names the t-th free column of its row, or nothing when there are fewer
// (the digit covers every column the row could have free). The parts of a record
// partition its solutions.
//
// Place the first `levels` rows' queens:
//   returns  0: nothing here, 1: (c, l, r) reach row + levels, with `shift` bits
//            of s left, 2: the board is complete and *found solutions
//   skip     values of s to the next one that may hold something
// ROW > 0: row `row` takes only the columns of its mask (a table of ROW bytes a
// row), and the board ends after `rows` rows; c holds no pre-set columns.
template <uint32_t ROW>
__device__ __forceinline__ uint32_t free_columns(uint32_t c, uint32_t l, uint32_t r,
                                                 const uint32_t table, uint32_t row) {
    uint32_t x = ~(c | l | r);
    if (ROW > 0u) {
        uint32_t mask;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(mask) : "r"(table + ROW * row) : "memory");
        x &= mask;
    }
    return x;
}
template <uint32_t ROW>
__device__ __forceinline__ int descend(uint32_t s, const int levels, uint64_t &digits, int &shift,
                                       uint32_t &c, uint32_t &l, uint32_t &r, uint32_t &found,
                                       uint32_t &skip, const uint32_t table, uint32_t row,
                                       const uint32_t rows) {
    skip = 1u;
    for (int j = 0; j <= levels; ++j, ++row) {
        const uint32_t here = s & ((1u << shift) - 1u);  // this level's digit and those below
        if (ROW > 0u ? row == rows : c == ~0u) {  // the solution belongs to the digits of zeros
            skip = (1u << shift) - here;
            found = here == 0u ? 1u : 0u;
            return 2;
        }
        if (j == levels) return 1;
        const uint32_t bits = (uint32_t)digits & 15u;
        digits >>= 4;
        shift -= (int)bits;
        uint32_t x = free_columns<ROW>(c, l, r, table, row);
        for (uint32_t t = here >> shift; t && x; --t) x &= x - 1u;
        if (x == 0u) {  // and nothing at any higher value of this digit
            skip = (1u << (shift + (int)bits)) - here;
            return 0;
        }
        const uint32_t p = x & (0u - x);
        c |= p;
        l = (l | p) << 1;
        r = (r | p) >> 1;
    }
    return 1;
}

// A parent: the frame that the digits lead to, in row + levels - 1, whose
// candidates x are handed out one by one. Returns as descend.
template <uint32_t ROW>
__device__ __forceinline__ int split_parent(uint32_t s, const int levels, uint64_t digits,
                                            int shift, uint32_t &c, uint32_t &l, uint32_t &r,
                                            uint32_t &x, uint32_t &found, uint32_t &skip,
                                            const uint32_t table, uint32_t row, uint32_t rows) {
    const int got = descend<ROW>(s, levels - 1, digits, shift, c, l, r, found, skip, table, row,
                                 rows);
    if (got != 1) return got;
    row += (uint32_t)levels - 1u;
    x = free_columns<ROW>(c, l, r, table, row);
    if (x == 0u) return 0;
    if (ROW > 0u ? row + 1u == rows : __popc(c) == 31) {  // the last row
        found = (uint32_t)__popc(x);
        return 2;
    }
    return 1;
}

// A unit (the server's kernel): as a parent, with one more digit of the last
// row's free columns t, t + R, t + 2R, ... of R = 2^bits, so that a small digit
// leaves nothing out: search from (c, l, r) with candidates av.
template <uint32_t ROW>
__device__ __forceinline__ int split_unit(uint32_t s, const int levels, uint64_t digits,
                                          int shift, uint32_t &c, uint32_t &l, uint32_t &r,
                                          uint32_t &av, uint32_t &found, uint32_t &skip,
                                          const uint32_t table, uint32_t row, uint32_t rows) {
    const int got = descend<ROW>(s, levels - 1, digits, shift, c, l, r, found, skip, table, row,
                                 rows);
    if (got != 1) return got;
    row += (uint32_t)levels - 1u;
    const uint32_t here = s & ((1u << shift) - 1u);
    uint32_t x = free_columns<ROW>(c, l, r, table, row);
    for (uint32_t t = here; t && x; --t) x &= x - 1u;
    if (x == 0u) {
        skip = (1u << shift) - here;
        return 0;
    }
    av = x & (0u - x);
    for (x ^= av; x;) {
        for (uint32_t t = (1u << shift) - 1u; t && x; --t) x &= x - 1u;
        const uint32_t q = x & (0u - x);
        av |= q;
        x ^= q;
    }
    if (ROW > 0u ? row + 1u == rows : __popc(c) == 31) {  // the last row
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
// SPLIT: the indices are parents (split_parent), 2^split_shift to a record, and
// what is found below one is added into its record's entry (zeroed before the
// launch). The warp opens 32 parents at once, every lane one, busy or not, and
// queues those that hold something in shared memory; idle lanes take the queued
// parents' candidates one by one. (Each idle lane decoding its own unit, as it
// became idle, cost some 350 instructions a unit for mostly one lane at a time:
// 2048 records of N = 22 4.36 ms, 4.12 ms so; 10^5 records of N = 12..17 0.97 and
// 0.85 ms.) Parents that cannot hold anything are passed over in one go: the
// warp's position moves on by the last lane's skip.
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

    // above the stacks, the warp's queue of 32 opened parents: {c, l, r, candidates},
    // and {record, weight | N << 2 above its 48 bits}
    unsigned char *const above = look_smem + (uint32_t)a.slots * stride;
    uint4 *const q_frame = reinterpret_cast<uint4 *>(above) + (threadIdx.x & ~31u);
    uint2 *const q_from =
        reinterpret_cast<uint2 *>(above + 16u * blockDim.x) + (threadIdx.x & ~31u);
    uint32_t q_at = 0, q_end = 0, q_x = 0;  // entries left, candidates left of entry q_at
    const uint32_t table = sbase + (uint32_t)a.slots * stride + kSplitQueueBytes * blockDim.x;
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
            if (SPLIT && q_at < q_end) {  // hand out the candidates of one parent
                const uint32_t rank = __popc(need_mask & lt_mask);
                const uint32_t asked = __popc(need_mask), open = __popc(q_x);
                if (need && rank < open) {
                    const uint4 f = q_frame[q_at];
                    const uint2 from = q_from[q_at];
                    uint32_t x = q_x;
                    for (uint32_t t = rank; t; --t) x &= x - 1u;
                    idx = (uint64_t)from.x | (uint64_t)(from.y & 0xFFFFu) << 32;
                    wn = from.y >> 16;
                    sol = 0;
                    busy = true;
                    c = f.x;
                    L = f.y << 1;
                    R = f.z >> 1;
                    av = x & (0u - x);
                    top = base + stride;
                    need = false;
                }
                if (asked >= open) {
                    ++q_at;
                    if (q_at < q_end) q_x = q_frame[q_at].w;
                } else {
                    for (uint32_t t = asked; t; --t) q_x &= q_x - 1u;
                }
                need_mask = __ballot_sync(~0u, need);
                continue;
            }
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
            // each idle lane takes a record, or (SPLIT) every lane opens a parent
            const uint32_t rank = SPLIT ? lane : (uint32_t)__popc(need_mask & lt_mask);
            uint32_t skip = 1u;
            bool open = false;
            uint4 frame = make_uint4(0u, 0u, 0u, 0u);
            uint2 from = make_uint2(0u, 0u);
            if ((SPLIT || need) && rank < rem) {
                uint64_t at = next + rank;
                uint32_t s = 0u;  // the parent's digits
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
                    uint32_t ll = P.y, rr = P.z & last, x = 0, found = 0;
                    const int got =
                        split_parent<MASKED ? 8u : 0u>(s, a.levels, a.digits, a.split_shift, cc, ll,
                                                       rr, x, found, skip, table, d, n);
                    if (got == 2) finish(pi, found, w | (n << 2));
                    open = got == 1;
                    frame = make_uint4(MASKED ? cc | ((d + (uint32_t)a.levels) << kRowShift) : cc,
                                       ll, rr, x);
                    from = make_uint2((uint32_t)pi, (uint32_t)(pi >> 32) | (w | (n << 2)) << 16);
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
            const uint32_t asked = SPLIT ? 32u : (uint32_t)__popc(need_mask);
            uint32_t taken = asked < rem ? asked : rem;
            if (SPLIT) {
                const unsigned opened = __ballot_sync(~0u, open);
                __syncwarp();
                if (open) {
                    const uint32_t e = (uint32_t)__popc(opened & lt_mask);
                    q_frame[e] = frame;
                    q_from[e] = from;
                }
                __syncwarp();
                q_at = 0u;
                q_end = (uint32_t)__popc(opened);
                if (q_end) q_x = q_frame[0].w;
                __syncwarp();
                // pass over parents that hold nothing
                taken += __shfl_sync(~0u, skip, (int)taken - 1) - 1u;
                taken = taken < rem ? taken : rem;
            }
            next += taken;
            rem -= taken;
            need_mask = __ballot_sync(~0u, need);
        }
        if (need_mask == ~0u) break;  // the whole warp is idle, and nothing is left

        if (SPLIT && need_mask && rem == 0u && q_at == q_end) {
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
                look_step_masked<8u>(c, L, R, av, top, stride, table, thr, s32, m1, m2, mneg);
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

// ---------------------------------------------------------------------------
// Served mode: one persistent launch that keeps taking work of newly admitted
// requests from a device ring while earlier ones are still being searched
// (continuous batching). A ring record is a prefix of a request; its tag names
// the request's slot, which holds the row masks and how the record's subtree is
// cut into units. A warp takes one record at a time and hands its units to its
// lanes, whose idle ones first take frames of the warp's busy ones; the masks
// are cached per block in shared memory and refreshed by generation number.
// Records come from the ring to a block in batches, by compare-and-swap on the
// cursor (which must not pass the published head); one by one for each warp, the
// 3,648 warps of the grid got a record every 0.7 us between them.
//
// A slot's `remaining` counts what is still held of the request: its records not
// yet searched (a warp gives its own back together), and lanes that hold it by
// themselves. Whoever gives back the last publishes the slot's total to mapped
// host memory.
//
// Every wait is bounded: the claim retries a fixed number of times; a warp with
// nothing to do polls the ring with back-off, counts itself idle after
// idle_polls rounds, and the grid leaves together once every started warp is
// idle (or after 64x that many rounds in any case), so the kernel always ends
// by itself once the host stops feeding it.
//
// A burst of 32 requests of N = 10..15 takes 1.7 ms (0.9 ms of it the 32
// submissions); with the host enumerating subproblems down to four per lane on
// one core it took 123-190 ms.
// ---------------------------------------------------------------------------
constexpr int kServeRefill = 8;  // idle lanes for which a warp takes a new record

__device__ __forceinline__ uint4 ld_cg4(const void *p) {
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_cg1(const void *p) {
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void sts1(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" : : "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds1(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

__global__ void __maxnreg__(64) serve_kernel(const ServeArgs a) {
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(look_smem);
    const uint32_t stride = stack_slot_offset(blockDim.x, 0u, 1u, 16u);
    const uint32_t base = sbase + stack_slot_offset(blockDim.x, threadIdx.x, 0u, 16u);
    const uint32_t tables = sbase + (uint32_t)a.slots * stride;  // nslots x kServeTable
    // the block's batch of ring records: [first, end), taken under `lock`
    __shared__ unsigned long long batch_first, batch_end;
    __shared__ int batch_lock;
    if (threadIdx.x == 0) {
        batch_first = batch_end = 0ull;
        batch_lock = 0;
    }
    for (int i = threadIdx.x; i < a.nslots * (int)(kServeTable / 4u); i += blockDim.x)
        sts1(tables + 4u * i, i % (int)(kServeTable / 4u) == (int)(kServeGen / 4u) ? 0xFFFFFFFFu : 0u);
    __syncthreads();
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt_mask = (1u << lane) - 1u;
    const uint32_t m1 = a.mul[0], m2 = a.mul[1], mneg = a.mul[2];

    uint32_t c = kSentMaskedC, L = 0u, R = 0u, av = kSentAv, top = base, bot = base;
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};"
                 :
                 : "r"(base), "r"(c), "r"(L), "r"(R), "r"(av)
                 : "memory");
    int cur_slot = -1;         // the request this lane searches a part of
    uint32_t cur_w = 1;        // symmetry weight of its record
    uint32_t table = tables, thr = 0;
    uint64_t sol = 0;
    // the record the warp hands out (the same in every lane)
    uint32_t next = 0, rem = 0, rec_tab = tables;
    uint4 P = make_uint4(0u, 0u, 0u, 0u);
    int rec_slot = 0, levels = 0, shift = 0;
    uint64_t digits = 0;
    unsigned int idle_polls = 0;
    bool counted = false;  // warp-uniform: this warp is in *idle_warps
    if (lane == 0) atomicAdd(a.started_warps, 1u);
    // Claim back-off (warp-uniform): after a claim that found the ring empty
    // the warp skips its next `skip` claim rounds, doubling up to 64, so that
    // lanes still searching are not held up by lookups that find nothing.
    uint32_t backoff = 0, skip = 0;

    // The warp holds the records that it took of one request (`held` of them, of
    // held_slot) until none of its lanes works on them, and adds their solutions
    // up in its lanes (acc). Only when it turns to another request while lanes
    // still search the old one do those lanes hold the request each for itself
    // (own). One atomic per record and lane instead put all of a large request's
    // traffic on one address: N = 17 alone 13.9 ms, 5.2 ms so.
    int held_slot = 0;
    uint32_t held = 0;
    bool own = false;
    uint64_t acc = 0;

    auto give_back = [&](int slot, uint64_t s, uint32_t tokens) {
        ServeSlot &q = a.slot_info[slot];
        if (s) atomicAdd(&q.total, (unsigned long long)s);
        __threadfence();
        if (atomicSub(&q.remaining, tokens) == tokens) {
            __threadfence();
            const unsigned long long tot = atomicAdd(&q.total, 0ull);
            const unsigned long long seq =
                *reinterpret_cast<const volatile unsigned long long *>(&q.seq);
            a.done[slot].total = tot;
            a.done[slot].refused = *reinterpret_cast<const volatile uint32_t *>(&q.refused);
            __threadfence_system();
            a.done[slot].seq = seq;
            __threadfence_system();
        }
    };
    // Give the held records back; lanes still at work on them hold the request.
    auto let_go = [&]() {
        const bool works = cur_slot >= 0 && !own;
        const unsigned at_work = __ballot_sync(~0u, works);
        uint64_t sum = acc;
        for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(~0u, sum, o);
        if (lane == 0) {
            if (at_work)
                atomicAdd(&a.slot_info[held_slot].remaining, (unsigned)__popc(at_work));
            give_back(held_slot, sum, held);
        }
        own = own || works;
        acc = 0;
        held = 0;
        __syncwarp();
    };

    for (;;) {
        const bool idle = top == bot;
        if (idle) {
            if (cur_slot >= 0) {
                if (own) give_back(cur_slot, sol * cur_w, 1u);
                else acc += sol * cur_w;
                cur_slot = -1;
                own = false;
            }
            bot = top = base;
            c = kSentMaskedC;
            L = R = 0u;
            av = kSentAv;
        }
        bool need = idle;
        unsigned need_mask = __ballot_sync(~0u, need);
        bool stopping = false, may_claim = true;
        if (need_mask == ~0u) {
            // the mapped stop flag: read by an all-idle warp, and by each one only
            // every 64th poll (3,648 warps reading host memory at every poll made
            // the polls themselves take 100 us)
            if (((idle_polls + blockIdx.x) & 63u) == 0u) {
                int st = 0;
                if (lane == 0) st = a.ctl->stop;
                stopping = __shfl_sync(~0u, st, 0) != 0;
            }
        } else if (skip) {
            --skip;
            may_claim = false;
        }
        while (need_mask && !stopping) {
            if (rem == 0u) {
                if (!may_claim || __popc(need_mask) < kServeRefill) break;
                unsigned long long at = 0;
                // 1: record `at`, 0: there is none, -1: another warp is looking
                int got = 0, closing = 0;
                if (lane == 0) {
                    got = -1;
                    if (atomicCAS(&batch_lock, 0, 1) == 0) {
                        got = 0;
                        __threadfence_block();
                        volatile unsigned long long *first = &batch_first, *end = &batch_end;
                        unsigned long long f = *first, e = *end;
                        if (f == e)  // (1: the grid is leaving, nothing more from the ring)
                            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(closing)
                                         : "l"(a.closing) : "memory");
                        if (f == e && !closing) {
                            unsigned long long h, cur;
                            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(h)
                                         : "l"(a.head) : "memory");
                            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(cur)
                                         : "l"(a.cursor) : "memory");
                            for (int t = 0; t < 32 && cur < h; ++t) {
                                unsigned long long g = (h - cur) / (2ull * gridDim.x);
                                g = g < 1ull ? 1ull : g > 64ull ? 64ull : g;
                                const unsigned long long old = atomicCAS(a.cursor, cur, cur + g);
                                if (old == cur) {
                                    f = cur;
                                    e = cur + g;
                                    break;
                                }
                                cur = old;
                            }
                            __threadfence();  // records published before head are visible
                        }
                        if (f != e) {
                            at = f++;
                            got = 1;
                        }
                        *first = f;
                        *end = e;
                        __threadfence_block();
                        atomicExch(&batch_lock, 0);
                    }
                }
                at = __shfl_sync(~0u, at, 0);
                got = __shfl_sync(~0u, got, 0);
                closing = __shfl_sync(~0u, closing, 0);
                if (got <= 0) {
                    if (got == 0) {
                        backoff = backoff ? (backoff < 64u ? 2u * backoff : 64u) : 1u;
                        skip = backoff;
                        stopping = closing != 0;  // (the block's batch is used up as well)
                    }
                    break;
                }
                backoff = 0;
                if (counted) {  // back to work: out of the idle count
                    if (lane == 0) atomicSub(a.idle_warps, 1u);
                    counted = false;
                    idle_polls = 0;
                }
                P = ld_cg4(a.ring + (at & a.ring_mask));
                const uint32_t n = (P.w >> 2) & 31u, d = (P.w >> 7) & 31u, w = P.w & 3u;
                rec_slot = (int)(P.w >> 12);
                if (held && rec_slot != held_slot) let_go();
                const uint32_t last = (n >= 1u) ? (0xFFFFFFFFu >> (32u - n)) : 0u;
                bool ok = rec_slot < a.nslots && n >= 1u && n <= (uint32_t)kMaxConstrainedN &&
                          (w == 1u || w == 2u) && d <= n && (P.x & ~last) == 0u &&
                          (uint32_t)__popc(P.x) == d;
                if (ok) {
                    const ServeSlot *q = a.slot_info + rec_slot;
                    levels = (int)ld_cg1(&q->levels);
                    shift = (int)ld_cg1(&q->split_shift);
                    digits = (uint64_t)ld_cg1(&q->digits) |
                             (uint64_t)ld_cg1(reinterpret_cast<const uint32_t *>(&q->digits) + 1) << 32;
                    ok = serve_accepts((int)n, (int)d, levels, shift, a.slots);
                }
                if (!ok) {
                    if (lane == 0) {
                        look_error(a.status, NQ_EINVAL);
                        a.ctl->error = NQ_EINVAL;  // mapped: the next poll reports it
                        if (rec_slot < a.nslots) {
                            atomicExch(&a.slot_info[rec_slot].refused, 1u);
                            give_back(rec_slot, 0, 1u);
                        }
                    }
                    __syncwarp();
                    continue;
                }
                // the slot's masks, cached in this block's shared memory
                rec_tab = tables + kServeTable * (uint32_t)rec_slot;
                const uint32_t gen = ld_cg1(&a.slot_info[rec_slot].gen);
                __threadfence_block();
                if (__any_sync(~0u, lds1(rec_tab + kServeGen) != gen)) {
                    if (lane <= (unsigned)kSentinelRow)
                        sts1(rec_tab + 4u * lane, ld_cg1(&a.slot_info[rec_slot].allowed[lane]));
                    __threadfence_block();
                    __syncwarp();
                    if (lane == 0) sts1(rec_tab + kServeGen, gen);
                }
                __syncwarp();
                held_slot = rec_slot;
                ++held;
                next = 0u;
                rem = 1u << shift;
            }
            const uint32_t n = (P.w >> 2) & 31u, d = (P.w >> 7) & 31u, w = P.w & 3u;
            const uint32_t last = 0xFFFFFFFFu >> (32u - n);
            const uint32_t rank = __popc(need_mask & lt_mask);
            uint32_t past = 1u;
            if (need && rank < rem) {
                uint32_t cc = P.x, ll = P.y, rr = P.z & last, a0 = 0, found = 0;
                const int got = split_unit<4u>(next + rank, levels, digits, shift, cc, ll, rr, a0,
                                               found, past, rec_tab, d, n);
                if (got == 2) acc += (uint64_t)found * w;
                if (got == 1) {
                    cur_slot = rec_slot;
                    cur_w = w;
                    sol = 0;
                    table = rec_tab;
                    thr = (n - 1u) << kRowShift;
                    c = cc | ((d + (uint32_t)levels) << kRowShift);
                    L = ll << 1;
                    R = rr >> 1;
                    av = a0;
                    top = base + stride;
                    need = false;
                }
            }
            const uint32_t asked = __popc(need_mask);
            uint32_t taken = asked < rem ? asked : rem;
            if (asked <= rem) {  // every asker had a unit: pass over empty ones
                taken += __shfl_sync(~0u, past, 31 - __clz((int)need_mask)) - 1u;
                taken = taken < rem ? taken : rem;
            }
            next += taken;
            rem -= taken;
            need_mask = __ballot_sync(~0u, need);
        }
        if (need_mask && need_mask != ~0u && rem == 0u) {
            // idle lanes take the shallowest saved frames of busy ones (look_body)
            const bool giver = !need && top > bot + stride;
            const unsigned givers = __ballot_sync(~0u, giver);
            if (givers) {
                const uint32_t pairs = min(__popc(need_mask), __popc(givers));
                const uint32_t rank = __popc((need ? need_mask : givers) & lt_mask);
                const bool taker = need && rank < pairs;
                const int from = taker ? (int)__fns(givers, 0, (int)rank + 1) : (int)lane;
                const uint32_t at = __shfl_sync(~0u, bot + stride, from);
                const int slot = __shfl_sync(~0u, cur_slot, from);
                const uint32_t w = __shfl_sync(~0u, cur_w, from);
                const uint32_t tab = __shfl_sync(~0u, table, from);
                const uint32_t th = __shfl_sync(~0u, thr, from);
                const bool hold = __shfl_sync(~0u, (int)own, from) != 0;
                if (taker) {
                    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                                 : "=r"(c), "=r"(L), "=r"(R), "=r"(av)
                                 : "r"(at)
                                 : "memory");
                    cur_slot = slot;
                    cur_w = w;
                    table = tab;
                    thr = th;
                    sol = 0;
                    own = hold;
                    top = base + stride;
                    if (hold) atomicAdd(&a.slot_info[slot].remaining, 1u);
                }
                __threadfence();
                __syncwarp();
                if (giver && rank < pairs) {
                    bot += stride;
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};"
                                 :
                                 : "r"(bot), "r"(kSentMaskedC), "r"(0u), "r"(0u), "r"(kSentAv)
                                 : "memory");
                }
                __syncwarp();
            }
        }
        if (held && rem == 0u && !__any_sync(~0u, cur_slot >= 0 && !own)) let_go();
        if (need_mask == ~0u) {
            if (stopping) break;
            ++idle_polls;
            if (idle_polls > a.idle_polls && !counted) {
                if (lane == 0) atomicAdd(a.idle_warps, 1u);
                counted = true;
            }
            if (counted && (idle_polls & 15u) == 0u) {
                int leave = 0;
                if (lane == 0) {
                    unsigned int iw, sw;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(iw)
                                 : "l"(a.idle_warps) : "memory");
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(sw)
                                 : "l"(a.started_warps) : "memory");
                    leave = iw >= sw || (unsigned long long)idle_polls > 64ull * a.idle_polls;
                    if (leave) atomicExch(a.closing, 1u);
                }
                if (__shfl_sync(~0u, leave, 0)) break;
            }
            __nanosleep(idle_polls < 64 ? 256u : 4096u);
            continue;
        }
        idle_polls = 0;
        uint32_t s32 = 0;
#pragma unroll
        for (int j = 0; j < kLookSteps; ++j)
            look_step_masked<4u>(c, L, R, av, top, stride, table, thr, s32, m1, m2, mneg);
        sol += s32;
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

void *serve_kernel_ptr() { return reinterpret_cast<void *>(&serve_kernel); }

}  // namespace nqi
