// The host side of libnq's calls without a GPU, on a device that is faked here (the
// executable's definitions of the runtime's functions stand before libcudart's).
// Its server's kernel takes the published records one by one, asks the function that
// the real kernel asks whether it searches such a record, and answers a request with
// the number of its records. Its search kernels answer with the number of theirs.
//
//   cuts    the cuts that serve_cut makes, over boards, depths, stacks, record
//           counts and seeded queens, that the kernel would not take or whose digits
//           do not cover their rows
//   shapes  launch shapes that fit an SM with 33 words a request slot beside the stacks
//           and that serve_plan refuses
//   total N d    nq_total_ex in the default form (d = 0: no depth given): records
//           launched and the rows placed in them, records and rows in the timing
//   nomem   nq_total(5) with room for no host allocation, for one, for two, ...: the
//           number of calls until one had enough; nq_count_ex of new shapes with none
//   burst max_n stack_slots N [row col]...    one request: records, answer, errors
//   refuse max_n stack_slots N [row col]...   the same, its last record not searched
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include <cuda.h>

#include "nq_internal.h"

using namespace nqi;

// Host allocations left before all fail; -1: none does.
long allocations_left = -1;
bool out_of_memory = false;

void *operator new(size_t n) {
    if (allocations_left == 0) out_of_memory = true;
    if (allocations_left == 0) throw std::bad_alloc();
    if (allocations_left > 0) --allocations_left;
    if (void *p = std::malloc(n)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, size_t) noexcept { std::free(p); }

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *fa, const void *) {
    std::memset(fa, 0, sizeof(*fa));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *nb, const void *, int block,
                                                                   size_t smem, unsigned) {
    // (of shared memory, 1 KB a block and the kernel's own 32 bytes are taken)
    const int by_regs = 65536 / (64 * block), by_smem = (int)(233472 / (smem + 1024 + 32));
    *nb = by_regs < by_smem ? by_regs : by_smem;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(16);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c) {
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    *p = nullptr;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) {
    return cudaMalloc(p, n);
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) { return cudaMalloc(p, 1 << 20); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
CUresult get_current(CUcontext *c) { *c = reinterpret_cast<CUcontext>(8); return CUDA_SUCCESS; }
CUresult get_id(CUcontext, unsigned long long *id) { *id = 8; return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    *f = !std::strcmp(name, "cuCtxGetCurrent") ? reinterpret_cast<void *>(&get_current)
                                                : reinterpret_cast<void *>(&get_id);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }

bool refuse_last = false;

// serve_kernel: every published record, in order; the others: what they are given.
cudaError_t cudaLaunchKernel(const void *k, dim3, dim3, void **params, size_t, cudaStream_t) {
    if (k != serve_kernel_ptr()) {
        const SearchArgs &a = *static_cast<const SearchArgs *>(params[0]);
        std::printf("search %llu records of %u rows, ", (unsigned long long)a.n,
                    NQ_META_D(a.pre[0].meta));
        a.totals[a.expect_n] = a.n;
        return cudaSuccess;
    }
    const ServeArgs &a = *static_cast<const ServeArgs *>(params[0]);
    for (; *a.cursor < *a.head; ++*a.cursor) {
        const nq_prefix &P = a.ring[*a.cursor & a.ring_mask];
        ServeSlot &q = a.slot_info[NQ_META_TAG(P.meta)];
        if (!(refuse_last && q.remaining == 1) &&
            serve_accepts((int)NQ_META_N(P.meta), (int)NQ_META_D(P.meta), q.levels, q.split_shift,
                          a.slots)) {
            ++q.total;
        } else {
            q.refused = 1;
            a.ctl->error = NQ_EINVAL;
        }
        if (--q.remaining == 0) {
            ServeDone &done = a.done[NQ_META_TAG(P.meta)];
            done.total = q.total;
            done.refused = q.refused;
            done.seq = q.seq;
        }
    }
    return cudaSuccess;
}
}

namespace {

// Seeded queens, no two attacking each other: the row masks of a partial board.
bool draw_masks(uint64_t &seed, int n, int k, uint32_t *allowed) {
    auto next = [&]() {
        seed = seed * 6364136223846793005ull + 1442695040888963407ull;
        return (uint32_t)(seed >> 33);
    };
    nq_queen q[4];
    for (int i = 0; i < k; ++i) q[i] = {(int8_t)(next() % n), (int8_t)(next() % n)};
    bool conflict = false;
    return constraint_masks(n, q, k, allowed, &conflict) == NQ_OK && !conflict;
}

int cuts() {
    long made = 0, wide = 0, refused = 0, short_digit = 0;
    uint64_t seed = 11;
    for (int n = 1; n <= kMaxConstrainedN; ++n)
        for (int k = 0; k <= 4; ++k) {
            uint32_t allowed[32];
            if (!draw_masks(seed, n, k, allowed)) continue;
            for (int d = 0; d <= n; ++d)
                for (int slots = 2; slots <= 27; ++slots)
                    for (uint64_t records : {1ull, 700ull, 30000ull, 4000000ull})
                        for (double lanes : {19456.0, 155648.0}) {
                            ServeSlot s{};
                            if (serve_cut(n, d, allowed, records, lanes, slots, &s)) continue;
                            ++made;
                            wide += s.split_shift == 31;
                            refused += !serve_accepts(n, d, s.levels, s.split_shift, slots);
                            int bits = 0;
                            for (int j = 0; j < s.levels; ++j) {
                                const int b = (int)(s.digits >> (4 * j) & 15u);
                                bits += b;
                                // (a row's free columns: those of its mask, less the rows above)
                                if (j + 1 < s.levels && d + j < n) {
                                    const int m = __builtin_popcount(allowed[d + j]);
                                    short_digit += (1 << b) < (m < n - d - j ? m : n - d - j);
                                }
                            }
                            short_digit += bits != s.split_shift;
                        }
        }
    std::printf("%ld cuts, %ld of 31 bits, %ld refused, %ld short digits\n", made, wide, refused,
                short_digit);
    return 0;
}

int shapes() {
    long fit = 0, refused = 0;
    for (int block = 32; block <= 1024; block += 32)
        for (int max_n = 1; max_n <= kMaxConstrainedN; ++max_n)
            for (int nslots = 1; nslots <= kServeMaxSlots; ++nslots) {
                const size_t stacks = (size_t)(max_n > 2 ? max_n : 2) * 16 * block;
                if (stacks + nslots * 132 > 232448) continue;
                int grid = 0, slots = 0;
                size_t smem = 0;
                ++fit;
                refused += serve_plan(max_n, 0, nslots, block, &grid, &smem, &slots) != NQ_OK;
            }
    std::printf("%ld shapes, %ld refused\n", fit, refused);
    return 0;
}

int total(int n, int d) {
    nq_config cfg{};
    cfg.d = d;
    nq_timing t{};
    uint64_t q = 0;
    const int rc = nq_total_ex(n, d ? &cfg : nullptr, &q, nullptr, &t);
    std::printf("rc %d, total %llu, timing %llu of %d\n", rc, (unsigned long long)q,
                (unsigned long long)t.prefixes, t.d);
    return 0;
}

int nomem() {
    int calls = 0;
    do {
        uint64_t q = 0;
        out_of_memory = false;
        allocations_left = calls++;
        try {
            nq_total(5, &q);
        } catch (const std::bad_alloc &) {
        }
        allocations_left = -1;
    } while (out_of_memory);
    // an asynchronous call's stream is known from its first; then no memory, and shapes
    // that no call has planned yet
    const nq_prefix root{0, 0, 0, NQ_META(1, 9, 0, 0)};
    uint64_t counts[1], totals[32] = {};
    nq_config cfg{};
    int rc[3] = {1, 1, 1};  // (1: it threw)
    for (int i = 0; i < 3; ++i) {
        cfg.block = 32 + 32 * i;
        if (i) allocations_left = 0;
        try {
            rc[i] = nq_count_ex(&root, 1, 0, 9, counts, nullptr, totals, &cfg, nullptr);
        } catch (const std::bad_alloc &) {
        }
        allocations_left = -1;
    }
    std::printf("%d calls, count %d %d %d\n", calls, rc[0], rc[1], rc[2]);
    return 0;
}

int burst(int max_n, int stack_slots, int n, const std::vector<nq_queen> &q) {
    nq_server_config cfg{};
    cfg.max_n = max_n;
    cfg.stack_slots = stack_slots;
    nq_server *s = nullptr;
    uint64_t ticket = 0, published = 0, tickets[4], counts[4];
    int rc = nq_server_create(&cfg, &s), got = 0;
    if (!rc) rc = nq_server_submit(s, n, q.data(), (int)q.size(), &ticket);
    if (rc) {
        std::printf("refused %d\n", rc);
        return 0;
    }
    nq_server_stats(s, nullptr, nullptr, nullptr, &published);
    std::printf("%llu records", (unsigned long long)published);
    for (int i = 0; i < 2; ++i) {
        rc = nq_server_poll(s, tickets, counts, 4, &got);
        std::printf(", poll %d:", rc);
        for (int j = 0; j < got; ++j)
            std::printf(" %s %llu", tickets[j] == ticket ? "answer" : "stranger",
                        (unsigned long long)counts[j]);
    }
    std::printf("\n");
    return nq_server_destroy(s);
}

}  // namespace

int main(int argc, char **argv) {
    if (argc == 2 && !std::strcmp(argv[1], "cuts")) return cuts();
    if (argc == 2 && !std::strcmp(argv[1], "shapes")) return shapes();
    if (argc == 2 && !std::strcmp(argv[1], "nomem")) return nomem();
    if (argc == 4 && !std::strcmp(argv[1], "total"))
        return total(std::atoi(argv[2]), std::atoi(argv[3]));
    refuse_last = argc > 1 && !std::strcmp(argv[1], "refuse");
    if (argc < 5 || (!refuse_last && std::strcmp(argv[1], "burst"))) return 2;
    std::vector<nq_queen> q;
    for (int i = 5; i + 1 < argc; i += 2)
        q.push_back({(int8_t)std::atoi(argv[i]), (int8_t)std::atoi(argv[i + 1])});
    return burst(std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]), q);
}
