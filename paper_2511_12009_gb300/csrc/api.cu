// api.cu -- the extern "C" entry points of libnq (declared in include/nq.h).
#include <algorithm>
#include <chrono>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <unordered_map>
#include <vector>

#include "nq_internal.h"
#include "prefix.h"

#include <nvtx3/nvToolsExt.h>

using namespace nqi;

namespace {

using Clock = std::chrono::steady_clock;

double ms_since(Clock::time_point t0) {
    return std::chrono::duration<double, std::milli>(Clock::now() - t0).count();
}

bool aligned(const void *p, size_t a) { return ((uintptr_t)p % a) == 0; }

int cuda_rc(cudaError_t e) { return e == cudaSuccess ? NQ_OK : NQ_ECUDA; }

// Host phases show up as named ranges in a timeline profiler (no-ops without one).
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
};

int env_int(const char *name) {
    const char *v = std::getenv(name);
    if (!v || !*v) return 0;
    char *end = nullptr;
    const long x = std::strtol(v, &end, 10);
    return (end && *end == '\0' && x > 0 && x < (1L << 30)) ? (int)x : 0;
}

int env_layout() {
    const char *v = std::getenv("NQ_LAYOUT");
    if (!v || !*v) return 0;
    static const char *names[] = {"default", "paper", "reg",  "wt",   "wt32",  "wt32a",
                                  "wtm",     "regm",  "regp", "regz", "regpz", "avail"};
    static_assert(sizeof(names) / sizeof(names[0]) == NQ_LAYOUT_LAST + 1, "one name per layout");
    for (int i = 0; i <= NQ_LAYOUT_LAST; ++i)
        if (std::strcmp(v, names[i]) == 0) return i;
    const int x = env_int("NQ_LAYOUT");
    return x <= NQ_LAYOUT_LAST ? x : 0;
}

// The configuration a call runs with: the caller's fields, and for the ones it
// leaves at 0 the environment's NQ_LAYOUT (number or name), NQ_BLOCK, NQ_CLAIM
// and NQ_D, else the library defaults.
nq_config with_env(const nq_config *cfg) {
    nq_config c = cfg ? *cfg : nq_config{};
    if (!c.layout) c.layout = env_layout();
    if (!c.block) c.block = env_int("NQ_BLOCK");
    if (!c.claim) c.claim = env_int("NQ_CLAIM");
    if (!c.d) c.d = env_int("NQ_D");
    return c;
}

// Pinned host staging buffer, one per host thread (grown on demand).
struct PinnedBuf {
    void *p = nullptr;
    size_t cap = 0;
    ~PinnedBuf() {
        if (p) cudaFreeHost(p);
    }
    void *get(size_t bytes) {
        if (bytes <= cap) return p;
        if (p) cudaFreeHost(p);
        p = nullptr;
        cap = 0;
        if (cudaMallocHost(&p, bytes) != cudaSuccess) {
            p = nullptr;
            return nullptr;
        }
        cap = bytes;
        return p;
    }
};
thread_local PinnedBuf t_stage;

// What synchronous calls keep between them, per device context: a memory pool
// of the library's own that holds on to kPoolKeep bytes when a stream
// synchronises (the device's default pool gives everything back to the driver
// then, so that each call mapped its few kilobytes anew: most of the 290 us
// that nq_total(8) took), and up to kStreamsKept idle streams. A stream is
// kept only once its work is done, and by one call at a time.
constexpr uint64_t kPoolKeep = 64ull << 20;  // (a pool grows by 32 MB at a time)
constexpr size_t kStreamsKept = 8;

struct Kept {
    cudaMemPool_t pool = nullptr;
    cudaStream_t streams[kStreamsKept] = {};
    size_t n_streams = 0;
};
std::mutex g_kept_mu;

// The current context's entry (NULL if there is no context, or no host memory for
// one). Caller holds the lock.
Kept *kept_locked() {
    unsigned long long ctx = 0;
    if (current_context_id(&ctx) != NQ_OK) return nullptr;
    try {
        static std::unordered_map<unsigned long long, Kept> *kept =
            new std::unordered_map<unsigned long long, Kept>();  // (may outlive static teardown)
        return &(*kept)[ctx];
    } catch (const std::bad_alloc &) {
        return nullptr;
    }
}

// The library's memory pool on the current device.
int memory_pool(cudaMemPool_t *out) {
    std::lock_guard<std::mutex> g(g_kept_mu);
    Kept *k = kept_locked();
    unsigned long long ctx = 0;
    if (!k) return current_context_id(&ctx) == NQ_OK ? NQ_ENOMEM : NQ_ECUDA;
    if (!k->pool) {
        int dev = 0;
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        if (cudaGetDevice(&dev) != cudaSuccess) return NQ_ECUDA;
        props.location.id = dev;
        if (cudaMemPoolCreate(&k->pool, &props) != cudaSuccess) {
            k->pool = nullptr;
            return NQ_ENOMEM;
        }
        uint64_t keep = kPoolKeep;
        cudaMemPoolSetAttribute(k->pool, cudaMemPoolAttrReleaseThreshold, &keep);
    }
    *out = k->pool;
    return NQ_OK;
}

int pool_alloc(void **out, size_t bytes, cudaStream_t s) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess ||
        capture != cudaStreamCaptureStatusNone)  // (the graph owns its allocation)
        return cudaMallocAsync(out, bytes, s) == cudaSuccess ? NQ_OK : NQ_ENOMEM;
    cudaMemPool_t pool = nullptr;
    const int rc = memory_pool(&pool);
    if (rc) return rc;
    return cudaMallocFromPoolAsync(out, bytes, pool, s) == cudaSuccess ? NQ_OK : NQ_ENOMEM;
}

// Owns a non-blocking stream and the stream-ordered device allocations of one
// synchronous call.
struct CallCtx {
    cudaStream_t s = nullptr;
    std::vector<void *> bufs;
    ~CallCtx() {
        if (!s) return;
        for (void *b : bufs) cudaFreeAsync(b, s);
        if (cudaStreamSynchronize(s) == cudaSuccess) {
            std::lock_guard<std::mutex> g(g_kept_mu);
            Kept *k = kept_locked();
            if (k && k->n_streams < kStreamsKept) {
                k->streams[k->n_streams++] = s;
                return;
            }
        }
        cudaStreamDestroy(s);
    }
    int init() {
        {
            std::lock_guard<std::mutex> g(g_kept_mu);
            Kept *k = kept_locked();
            if (k && k->n_streams) {
                s = k->streams[--k->n_streams];
                return NQ_OK;
            }
        }
        return cuda_rc(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    }
    template <typename T>
    int alloc(T **out, size_t bytes) {
        void *p = nullptr;
        if (const int rc = pool_alloc(&p, bytes ? bytes : 16, s)) return rc;
        bufs.push_back(p);
        *out = static_cast<T *>(p);
        return NQ_OK;
    }
};

// The three timing events of a synchronous call.
struct CallEvents {
    cudaEvent_t e[3] = {};
    int init() {
        for (auto &x : e)
            if (cudaEventCreate(&x) != cudaSuccess) {
                x = nullptr;
                return NQ_ECUDA;
            }
        return NQ_OK;
    }
    ~CallEvents() {
        for (auto &x : e)
            if (x) cudaEventDestroy(x);
    }
};

// Enqueue one search over device-resident prefixes (shared by nq_count*,
// nq_total_ex, nq_count_constrained and nq_count_split). n_tags > 0: the
// records are split subproblems whose counts and nodes are added into entry
// tag of d_counts / d_nodes (zeroed here, n_tags entries). cursor_ext: a work
// cursor the caller allocated and zeroed in stream order (used unless the
// launch donates subtrees); NULL: the call allocates its own on `s`.
// published: streamed input (SearchArgs::published); no donation then.
// status: the device word the launch records its first error in.
int enqueue_search(const nq_prefix *d_prefixes, uint64_t n, int expect_n, int min_d, int max_n,
                   uint64_t *d_counts, uint64_t *d_nodes, uint64_t *d_totals,
                   const nq_config *cfg_in, const uint32_t *allowed, cudaStream_t s, Plan *used,
                   int *status, uint64_t n_tags = 0, unsigned long long *cursor_ext = nullptr,
                   const unsigned long long *published = nullptr) {
    const nq_config cfg_eff = with_env(cfg_in);
    const nq_config *cfg = &cfg_eff;
    if (n_tags && !d_counts) return NQ_EINVAL;
    if (n_tags) {
        if (cudaMemsetAsync(d_counts, 0, n_tags * sizeof(uint64_t), s) != cudaSuccess ||
            (d_nodes && cudaMemsetAsync(d_nodes, 0, n_tags * sizeof(uint64_t), s) != cudaSuccess))
            return NQ_ECUDA;
    }
    if (n == 0) return NQ_OK;
    if (!d_prefixes || !aligned(d_prefixes, 16) || (d_counts && !aligned(d_counts, 8)) ||
        (d_nodes && !aligned(d_nodes, 8)) || (d_totals && !aligned(d_totals, 8)))
        return NQ_EINVAL;
    const bool diag = d_nodes != nullptr;
    const bool constrained = allowed != nullptr;
    Plan p;
    int rc = make_plan(max_n, min_d, diag, constrained, cfg, &p, false, published != nullptr);
    if (rc) return rc;
    // Scratch: the work cursor, and with donation its counters and item ring.
    const bool reg = p.layout == NQ_LAYOUT_REG || p.layout == NQ_LAYOUT_REGM;  // donation forms
    // Donation (its own kernel variant, planned again: its occupancy differs)
    // only when asked for: measured on GB300 it has not paid for its queue
    // traffic yet, so batches short of work are better split (on the device in
    // the default form, by nq_count_split in the others).
    const bool donate = reg && !constrained && !n_tags && !published && cfg && cfg->donate == 2;
    if (donate && (rc = make_plan(max_n, min_d, diag, constrained, cfg, &p, true))) return rc;
    if ((rc = plan_records(max_n, min_d, diag, cfg, n, !n_tags, &p, allowed))) return rc;
    if (p.levels && d_counts &&
        cudaMemsetAsync(d_counts, 0, n * sizeof(uint64_t), s) != cudaSuccess)
        return NQ_ECUDA;
    const size_t head_bytes = 128 + sizeof(DonateCtl);  // cursor line, counters
    const size_t bytes = donate ? head_bytes + kDonateCap * sizeof(DonateItem) : 64;
    const bool own = donate || (!cursor_ext && (!p.look || p.cursor));
    unsigned char *scratch = nullptr;
    if (own && (rc = pool_alloc(reinterpret_cast<void **>(&scratch), bytes, s))) return rc;
    unsigned long long *cursor =  // (NULL: the launch needs none)
        own ? reinterpret_cast<unsigned long long *>(scratch) : cursor_ext;
    if (own) rc = cuda_rc(cudaMemsetAsync(scratch, 0, donate ? bytes : 64, s));
    if (!rc && donate && d_counts)
        rc = cuda_rc(cudaMemsetAsync(d_counts, 0, n * sizeof(uint64_t), s));
    if (!rc && donate && d_nodes)
        rc = cuda_rc(cudaMemsetAsync(d_nodes, 0, n * sizeof(uint64_t), s));
    if (!rc) {
        SearchArgs a{};
        a.pre = d_prefixes;
        a.n = n;
        a.counts = d_counts;
        a.nodes = d_nodes;
        a.totals = d_totals;
        a.cursor = cursor;
        a.expect_n = expect_n;
        a.min_d = min_d;
        a.slots = p.slots;
        // claim order: last index first unless index order is asked for
        a.order = (cfg && cfg->order == 1) ? 0 : 1;
        a.claim = (cfg && cfg->claim > 0) ? cfg->claim : 1;
        a.by_tag = n_tags ? 1 : 0;
        a.n_tags = n_tags;
        if (donate) {
            a.dq = reinterpret_cast<DonateCtl *>(scratch + 128);
            a.items = reinterpret_cast<DonateItem *>(scratch + head_bytes);
        }
        if (allowed) std::memcpy(a.allowed, allowed, sizeof(a.allowed));
        a.mul[0] = 1u;
        a.mul[1] = 2u;
        a.mul[2] = 0xFFFFFFFFu;
        a.mul[3] = 0x80000000u;
        a.published = published;
        a.status = status;
        rc = launch_search(a, p, diag, constrained, s);
    }
    if (own) cudaFreeAsync(scratch, s);
    if (used) *used = p;
    return rc;
}

}  // namespace

extern "C" const char *nq_strerror(int code) {
    switch (code) {
        case NQ_OK: return "ok";
        case NQ_EINVAL: return "invalid argument or malformed prefix record";
        case NQ_ENOMEM: return "out of memory";
        case NQ_ECUDA: return "CUDA runtime error";
        case NQ_EOVERFLOW: return "result or buffer overflow";
        case NQ_ETIMEOUT: return "bounded device wait timed out";
        case NQ_ESTACK: return "prefix needs more stack levels than the launch provides";
        case NQ_EBUSY: return "busy";
        default: return "unknown status code";
    }
}

extern "C" int nq_count_ex(const nq_prefix *d_prefixes, uint64_t n, int min_d, int max_n,
                           uint64_t *d_counts, uint64_t *d_nodes, uint64_t *d_totals,
                           const nq_config *cfg, void *stream) {
    if (max_n < 1 || max_n > NQ_MAX_N || min_d < 0 || min_d > max_n) return NQ_EINVAL;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    int *status = nullptr;
    const int rc = stream_status(s, &status);
    if (rc) return rc;
    return enqueue_search(d_prefixes, n, 0, min_d, max_n, d_counts, d_nodes, d_totals, cfg,
                          nullptr, s, nullptr, status);
}

extern "C" int nq_count(int N, int d, const nq_prefix *d_prefixes, uint64_t n,
                        uint64_t *d_counts, void *stream) {
    if (N < 1 || N > NQ_MAX_N || d < 0 || d > N || !d_counts) return NQ_EINVAL;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    int *status = nullptr;
    const int rc = stream_status(s, &status);
    if (rc) return rc;
    return enqueue_search(d_prefixes, n, N, d, N, d_counts, nullptr, nullptr, nullptr, nullptr, s,
                          nullptr, status);
}

extern "C" int nq_sync(void *stream) {
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(s) != cudaSuccess) return NQ_ECUDA;
    int *status = nullptr;
    const int rc = stream_status(s, &status);
    if (rc) return rc;
    return take_status(status, s);
}

namespace {

// nq_total_ex in the default form: the launch splits subtrees by itself
// (plan_records), so with no depth given only the prefixes of the first kTotalRows
// rows are made and copied (2.5 MB at N = 28, the largest), and the default depth's
// set is only counted, beside the search, for the caller who asks. Before, the host
// wrote all of it (N = 18: 7.4 M records, 2.8 ms of host work and 118 MB beside the
// search). A depth that the caller gives is the depth that is searched: N = 18 at
// d = 7 22.7 ms (20.1 ms with none given), N = 20 at d = 7 1.16 s (1.20 s).
// kTotalRows: rows 0 and 1 hold the symmetry rules; two more leave the launch two
// levels less to split at next to no host work (N = 14: search of 0.081, 0.082,
// 0.064, 0.091 ms from 2, 3, 4, 5 rows; N = 17: 3.45, 3.58, 3.26, 3.15 ms).
constexpr int kTotalRows = 4;

// The records behind a block's head, and the head itself: [0] work cursor, [1]
// status, [2..33] totals. One copy takes both to the device and one brings the
// head back.
constexpr size_t kHead = 34 * sizeof(uint64_t);
static_assert(kHead % sizeof(nq_prefix) == 0, "the records are 16-byte aligned");
nq_prefix *staged_records(unsigned char *stage) {
    return reinterpret_cast<nq_prefix *>(stage + kHead);
}

// Count the n records staged behind `stage` (pinned), every one an N x N board
// with at least d rows placed (allowed: under row masks), and their weighted
// total. beside(): host work done while the search runs.
template <typename F>
int search_staged(int N, int d, unsigned char *stage, uint64_t n, const nq_config *cfg,
                  const uint32_t *allowed, uint64_t *total_out, nq_timing *timing, F beside) {
    const size_t bytes = kHead + n * sizeof(nq_prefix);
    std::memset(stage, 0, kHead);
    int rc;
    CallCtx ctx;
    if ((rc = ctx.init())) return rc;
    unsigned char *dev = nullptr;
    if ((rc = ctx.alloc(&dev, bytes))) return rc;
    auto *d_head = reinterpret_cast<uint64_t *>(dev);
    CallEvents ev;
    if (timing && (rc = ev.init())) return rc;
    if (timing) cudaEventRecord(ev.e[0], ctx.s);
    {
        Range r("nq.upload");
        rc = cuda_rc(cudaMemcpyAsync(dev, stage, bytes, cudaMemcpyHostToDevice, ctx.s));
    }
    if (timing) cudaEventRecord(ev.e[1], ctx.s);
    Plan p{};
    if (!rc)
        rc = enqueue_search(staged_records(dev), n, N, d, N, nullptr, nullptr, d_head + 2, cfg,
                            allowed, ctx.s, &p, reinterpret_cast<int *>(d_head + 1), 0,
                            reinterpret_cast<unsigned long long *>(d_head));
    if (timing) cudaEventRecord(ev.e[2], ctx.s);
    if (!rc) rc = cuda_rc(cudaMemcpyAsync(stage, dev, kHead, cudaMemcpyDeviceToHost, ctx.s));
    const int brc = rc ? NQ_OK : beside();
    if (cudaStreamSynchronize(ctx.s) != cudaSuccess) return NQ_ECUDA;
    if (rc || brc) return rc ? rc : brc;
    const auto *head = reinterpret_cast<const uint64_t *>(stage);
    if (const int st = *reinterpret_cast<const int *>(head + 1)) return st;
    *total_out = head[2 + N];
    if (timing) {
        float up = 0, kern = 0;
        cudaEventElapsedTime(&up, ev.e[0], ev.e[1]);
        cudaEventElapsedTime(&kern, ev.e[1], ev.e[2]);
        timing->upload_ms = up;
        timing->kernel_ms = kern;
        timing->layout = p.layout;
        timing->block = p.block;
        timing->grid = p.grid;
    }
    return NQ_OK;
}

// Search the set of depth b, report the one of depth d.
int total_split(int N, int b, int d, const nq_config *cfg, uint64_t *total_out,
                nq_timing *timing) {
    const auto t_start = Clock::now();
    PrefixCut cut;
    int rc;
    {
        Range r("nq.enumerate.count");
        rc = cut_prefixes(N, b, &cut);
    }
    if (rc) return rc;
    const uint64_t n = cut.first.back();
    unsigned char *stage =
        static_cast<unsigned char *>(t_stage.get(kHead + n * sizeof(nq_prefix)));
    if (!stage) return NQ_ENOMEM;
    {
        Range r("nq.enumerate.write");
        write_prefix_nodes(cut, 0, cut.nodes.size(), staged_records(stage), n);
    }
    const double enum_ms = ms_since(t_start);
    uint64_t prefixes = n;
    rc = search_staged(N, b, stage, n, cfg, nullptr, total_out, timing, [&]() -> int {
        if (!timing || d == b) return NQ_OK;
        Range r("nq.enumerate.count");
        return nq_enumerate_prefixes(N, d, nullptr, 0, &prefixes);
    });
    if (rc) return rc;
    if (timing) {
        timing->enumerate_ms = enum_ms;
        timing->prefixes = prefixes;
        timing->d = d;
        timing->total_ms = ms_since(t_start);
    }
    return NQ_OK;
}

}  // namespace

// The other forms stream large prefix sets: below this many subproblems the set
// is written, copied and searched in one go.
constexpr uint64_t kStreamMin = 1ull << 20;
constexpr int kStreamPieces = 8;

extern "C" int nq_total_ex(int N, const nq_config *cfg, uint64_t *total_out, uint64_t *nodes_out,
                           nq_timing *timing) {
    const auto t_start = Clock::now();
    if (N < 1 || N > NQ_MAX_N || !total_out) return NQ_EINVAL;
    if (N >= 29) return NQ_EOVERFLOW;  // Q(29) > 2^64 (Section 4.5: int64 ends at N = 28)
    const nq_config cfg_eff = with_env(cfg);
    cfg = &cfg_eff;
    const int d = cfg->d > 0 ? cfg->d : nq_default_depth(N);
    if (d < 0 || d > N) return NQ_EINVAL;

    const int lay = cfg->layout ? cfg->layout : NQ_LAYOUT_DEFAULT_SEARCH;
    if (lay == NQ_LAYOUT_REGP && !nodes_out)
        return total_split(N, cfg->d > 0 ? d : std::min(d, kTotalRows), d, cfg, total_out, timing);

    // a1 (counting pass): the set cut at its depth-3 nodes, the size of each part
    const auto t_enum = Clock::now();
    PrefixCut cut;
    int rc;
    {
        Range r("nq.enumerate.count");
        rc = cut_prefixes(N, d, &cut);
    }
    if (rc) return rc;
    const uint64_t np = cut.first.back();
    double enum_ms = ms_since(t_enum);

    // Pieces of whole depth-3 nodes in the kernel's claim order: from the end
    // of the canonical order (the heavier subtrees) unless index order is
    // configured. After piece j is copied in, the first pub[j] indices in
    // claim order may be searched.
    const bool from_end = cfg->order != 1;
    const size_t nn = cut.nodes.size();
    std::vector<std::pair<size_t, size_t>> pieces;  // node ranges, claim order
    {
        const int k = np >= kStreamMin ? kStreamPieces : 1;
        size_t done = 0;  // nodes taken so far (from the chosen end)
        for (int j = 1; j <= k && done < nn; ++j) {
            const uint64_t want = (np * (uint64_t)j) / (uint64_t)k;  // records covered after j
            size_t take = done;
            auto covered = [&](size_t t) {
                return from_end ? np - cut.first[nn - t] : cut.first[t];
            };
            while (take < nn && (j == k || covered(take) < want)) ++take;
            if (take == done) continue;
            pieces.emplace_back(from_end ? nn - take : done, from_end ? nn - done : take);
            done = take;
        }
        if (pieces.empty()) pieces.emplace_back(0, 0);
    }
    const size_t npieces = pieces.size();
    // pinned staging: the records, then the published counts
    const size_t rec_bytes = ((np ? np : 1) * sizeof(nq_prefix) + 15) / 16 * 16;
    unsigned char *stage =
        static_cast<unsigned char *>(t_stage.get(rec_bytes + (npieces + 1) * sizeof(uint64_t)));
    if (!stage) return NQ_ENOMEM;
    nq_prefix *h_pre = reinterpret_cast<nq_prefix *>(stage);
    unsigned long long *h_pub = reinterpret_cast<unsigned long long *>(stage + rec_bytes);

    CallCtx ctx;
    if ((rc = ctx.init())) return rc;
    nq_prefix *d_pre = nullptr;
    uint64_t *d_tot = nullptr, *d_nodes = nullptr;
    unsigned long long *d_ctl = nullptr;  // [0] work cursor, [16] published count, [24] status
    if ((rc = ctx.alloc(&d_pre, np * sizeof(nq_prefix)))) return rc;
    if ((rc = ctx.alloc(&d_tot, 32 * sizeof(uint64_t)))) return rc;
    if ((rc = ctx.alloc(&d_ctl, 256))) return rc;
    if (nodes_out && (rc = ctx.alloc(&d_nodes, np * sizeof(uint64_t)))) return rc;
    cudaStream_t cs = nullptr;  // copies and publication
    cudaEvent_t ev[5] = {};
    struct Guard {
        cudaStream_t &cs;
        cudaEvent_t *e;
        ~Guard() {  // runs before ctx frees the buffers the copies may still use
            if (cs) {
                cudaStreamSynchronize(cs);
                cudaStreamDestroy(cs);
            }
            for (int i = 0; i < 5; ++i)
                if (e[i]) cudaEventDestroy(e[i]);
        }
    } guard{cs, ev};
    for (auto &e : ev)
        if (cudaEventCreate(&e) != cudaSuccess) {
            e = nullptr;
            return NQ_ECUDA;
        }
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
        cs = nullptr;
        return NQ_ECUDA;
    }
    // streamed input needs a register-stack layout; any other layout searches
    // once every piece is in
    const bool stream_in = npieces > 1 && layout_register_top(lay);
    cudaEventRecord(ev[0], ctx.s);
    rc = cuda_rc(cudaMemsetAsync(d_tot, 0, 32 * sizeof(uint64_t), ctx.s));
    if (!rc) rc = cuda_rc(cudaMemsetAsync(d_ctl, 0, 256, ctx.s));
    if (!rc) rc = cuda_rc(cudaEventRecord(ev[1], ctx.s));
    if (!rc) rc = cuda_rc(cudaStreamWaitEvent(cs, ev[1], 0));
    Plan p{};
    // a3-a4: one persistent search over the whole set; with streamed input it
    // starts now and takes pieces as they are published
    int *d_status = reinterpret_cast<int *>(d_ctl + 24);
    if (!rc && stream_in)
        rc = enqueue_search(d_pre, np, N, d, N, nullptr, d_nodes, d_tot, cfg, nullptr, ctx.s, &p,
                            d_status, 0, d_ctl, d_ctl + 16);
    // a1 (writing) + a2 upload, piece by piece
    uint64_t published = 0;
    if (!rc) rc = cuda_rc(cudaEventRecord(ev[3], cs));
    for (size_t j = 0; j < npieces && !rc; ++j) {
        const auto [lo, hi] = pieces[j];
        const uint64_t r0 = cut.first[lo], r1 = cut.first[hi];
        const auto tw = Clock::now();
        {
            Range r("nq.enumerate.write");
            write_prefix_nodes(cut, lo, hi, h_pre, np);
        }
        enum_ms += ms_since(tw);
        Range r("nq.upload");
        if (r1 > r0)
            rc = cuda_rc(cudaMemcpyAsync(d_pre + r0, h_pre + r0, (r1 - r0) * sizeof(nq_prefix),
                                         cudaMemcpyHostToDevice, cs));
        published += r1 - r0;
        h_pub[j] = published;
        if (!rc && stream_in)
            rc = cuda_rc(cudaMemcpyAsync(d_ctl + 16, h_pub + j, sizeof(uint64_t),
                                         cudaMemcpyHostToDevice, cs));
    }
    if (!rc) rc = cuda_rc(cudaEventRecord(ev[4], cs));
    if (!rc && !stream_in) {
        rc = cuda_rc(cudaStreamWaitEvent(ctx.s, ev[4], 0));
        if (!rc)
            rc = enqueue_search(d_pre, np, N, d, N, nullptr, d_nodes, d_tot, cfg, nullptr, ctx.s,
                                &p, d_status, 0, d_ctl);
    }
    if (rc && stream_in) {
        // the search is waiting for records that will not come: publish the
        // whole (zeroed, hence rejected) set so that it ends at once
        h_pub[npieces] = np;
        cudaMemsetAsync(d_pre, 0, np * sizeof(nq_prefix), cs);
        cudaMemcpyAsync(d_ctl + 16, h_pub + npieces, sizeof(uint64_t), cudaMemcpyHostToDevice, cs);
    }
    cudaEventRecord(ev[2], ctx.s);
    // a5: the weighted total
    uint64_t tot = 0;
    if (!rc)
        rc = cuda_rc(cudaMemcpyAsync(&tot, d_tot + N, sizeof(uint64_t), cudaMemcpyDeviceToHost,
                                     ctx.s));
    if (cudaStreamSynchronize(ctx.s) != cudaSuccess || cudaStreamSynchronize(cs) != cudaSuccess)
        return NQ_ECUDA;
    const int st = take_status(d_status, ctx.s);
    if (rc) return rc;
    if (st) return st;
    *total_out = tot;
    if (nodes_out) {
        std::vector<uint64_t> nodes(np);
        if (np && cudaMemcpy(nodes.data(), d_nodes, np * sizeof(uint64_t),
                             cudaMemcpyDeviceToHost) != cudaSuccess)
            return NQ_ECUDA;
        uint64_t sum = 0;
        for (uint64_t v : nodes) sum += v;
        *nodes_out = sum;
    }
    if (timing) {
        // upload: first to last copy (overlapping the search when streamed);
        // kernel: from the search's launch point to its end
        float up = 0, kern = 0;
        cudaEventElapsedTime(&up, ev[3], ev[4]);
        cudaEventElapsedTime(&kern, ev[1], ev[2]);
        timing->enumerate_ms = enum_ms;
        timing->upload_ms = up;
        timing->kernel_ms = kern;
        timing->prefixes = np;
        timing->d = d;
        timing->layout = p.layout;
        timing->block = p.block;
        timing->grid = p.grid;
        timing->total_ms = ms_since(t_start);
    }
    return NQ_OK;
}

extern "C" int nq_total(int N, uint64_t *total_out) {
    return nq_total_ex(N, nullptr, total_out, nullptr, nullptr);
}

// ---------------------------------------------------------------------------
// Host-side split: few heavy subproblems (fewer than the grid has lanes) are
// extended a few rows deeper on the host, every child carrying its parent's
// index in the tag field, and the kernel adds each child's count into its
// parent's entry. The subtree of a prefix is the disjoint union of its
// children's subtrees (Section 1), so the per-parent sums are exact. (The
// default form's production build splits on the device instead.)
// ---------------------------------------------------------------------------
extern "C" int nq_count_split(const nq_prefix *h_prefixes, uint64_t n, int rows,
                              const nq_config *cfg, uint64_t *h_counts, uint64_t *h_nodes,
                              uint64_t *h_totals, int *rows_used, nq_timing *timing) {
    const auto t_start = Clock::now();
    if (!h_counts || (n && !h_prefixes) || rows < -1 || rows > NQ_MAX_N || n > kMaxSplitParents)
        return NQ_EINVAL;
    const nq_config cfg_eff = with_env(cfg);
    cfg = &cfg_eff;
    if (h_totals) std::memset(h_totals, 0, 32 * sizeof(uint64_t));
    if (n == 0) {
        if (rows_used) *rows_used = 0;
        return NQ_OK;
    }
    int min_d = NQ_MAX_N, max_n = 0;
    for (uint64_t i = 0; i < n; ++i) {
        min_d = std::min(min_d, (int)NQ_META_D(h_prefixes[i].meta));
        max_n = std::max(max_n, (int)NQ_META_N(h_prefixes[i].meta));
    }
    if (max_n < 1 || max_n > NQ_MAX_N) return NQ_EINVAL;
    const bool diag = h_nodes != nullptr;
    int r = rows, rc;
    if ((rc = check_parents(h_prefixes, n))) return rc;
    uint64_t m = 0;
    Plan shape{};
    const int lay = cfg->layout ? cfg->layout : NQ_LAYOUT_DEFAULT_SEARCH;
    if ((rows < 0 || (lay == NQ_LAYOUT_REGP && !diag)) &&
        (rc = make_plan(max_n, min_d, diag, false, cfg, &shape)))
        return rc;
    // -1: the fewest rows giving at least 32 children per resident lane
    const uint64_t want = 32ull * (uint64_t)shape.grid * (uint64_t)shape.block;
    auto count_rows = [&]() -> int {
        if (r < 0) {
            for (r = 0; r < max_n - min_d; ++r) {
                if (const int e = split_prefixes(h_prefixes, n, r, nullptr, nullptr, &m)) return e;
                if (m >= want) return m > kMaxSplitChildren ? NQ_EOVERFLOW : NQ_OK;
            }
        }
        if (const int e = split_prefixes(h_prefixes, n, r, nullptr, nullptr, &m)) return e;
        return m > kMaxSplitChildren ? NQ_EOVERFLOW : NQ_OK;
    };
    auto kid_depth = [&]() {
        int k = NQ_MAX_N;
        for (uint64_t i = 0; i < n; ++i)
            k = std::min(k, std::min((int)NQ_META_N(h_prefixes[i].meta),
                                     (int)NQ_META_D(h_prefixes[i].meta) + r));
        return k;
    };
    if (shape.look) {
        // The default form splits subtrees by itself (plan_records): the parents
        // are searched as they are, and the host only counts the children, while
        // the search runs unless there might be too many of them to accept.
        int left = 0;  // rows below the shallowest record
        for (uint64_t i = 0; i < n; ++i)
            left = std::max(left, (int)NQ_META_N(h_prefixes[i].meta) -
                                      (int)NQ_META_D(h_prefixes[i].meta));
        double most = r < 0 ? (double)want * std::max(left, 1) : (double)n;
        for (int j = 0; j < r && j < left; ++j) most *= left - j;
        const bool count_first = std::max(most, (double)n) > (double)kMaxSplitChildren;
        if (count_first && (rc = count_rows())) return rc;
        CallCtx ctx;
        if ((rc = ctx.init())) return rc;
        nq_prefix *d_pre = nullptr;
        uint64_t *d_out = nullptr;  // [0..31] totals, [32] status, then the counts
        if ((rc = ctx.alloc(&d_pre, n * sizeof(nq_prefix)))) return rc;
        if ((rc = ctx.alloc(&d_out, (34 + n) * sizeof(uint64_t)))) return rc;
        CallEvents ev;
        if ((rc = ev.init())) return rc;
        cudaEventRecord(ev.e[0], ctx.s);
        rc = cuda_rc(cudaMemcpyAsync(d_pre, h_prefixes, n * sizeof(nq_prefix),
                                     cudaMemcpyHostToDevice, ctx.s));
        if (!rc) rc = cuda_rc(cudaMemsetAsync(d_out, 0, 34 * sizeof(uint64_t), ctx.s));
        cudaEventRecord(ev.e[1], ctx.s);
        Plan p{};
        int *d_status = reinterpret_cast<int *>(d_out + 32);
        if (!rc)
            rc = enqueue_search(d_pre, n, 0, max_n - left, max_n, d_out + 34, nullptr, d_out, cfg,
                                nullptr, ctx.s, &p, d_status);
        cudaEventRecord(ev.e[2], ctx.s);
        const auto t_count = Clock::now();
        const int crc = count_first ? NQ_OK : count_rows();
        const double count_ms = ms_since(t_count);
        if (!rc)
            rc = cuda_rc(cudaMemcpyAsync(h_counts, d_out + 34, n * sizeof(uint64_t),
                                         cudaMemcpyDeviceToHost, ctx.s));
        if (!rc && h_totals)
            rc = cuda_rc(cudaMemcpyAsync(h_totals, d_out, 32 * sizeof(uint64_t),
                                         cudaMemcpyDeviceToHost, ctx.s));
        if (cudaStreamSynchronize(ctx.s) != cudaSuccess) return NQ_ECUDA;
        if (rc || crc) return rc ? rc : crc;
        const int st = take_status(d_status, ctx.s);
        if (st) return st;
        if (rows_used) *rows_used = r;
        if (timing) {
            float up = 0, kern = 0;
            cudaEventElapsedTime(&up, ev.e[0], ev.e[1]);
            cudaEventElapsedTime(&kern, ev.e[1], ev.e[2]);
            timing->enumerate_ms = count_ms;
            timing->upload_ms = up;
            timing->kernel_ms = kern;
            timing->prefixes = m;
            timing->d = kid_depth();
            timing->layout = p.layout;
            timing->block = p.block;
            timing->grid = p.grid;
            timing->total_ms = ms_since(t_start);
        }
        return NQ_OK;
    }
    if (r < 0 && (rc = count_rows())) return rc;
    std::vector<nq_prefix> kids;
    std::vector<uint64_t> extra;
    if ((rc = split_prefixes(h_prefixes, n, r, &kids, &extra, &m))) return rc;
    const double split_ms = ms_since(t_start);
    const int kid_min_d = kid_depth();

    CallCtx ctx;
    if ((rc = ctx.init())) return rc;
    nq_prefix *d_kids = nullptr;
    uint64_t *d_counts = nullptr, *d_nodes = nullptr, *d_tot = nullptr;
    if ((rc = ctx.alloc(&d_kids, m * sizeof(nq_prefix)))) return rc;
    if ((rc = ctx.alloc(&d_counts, n * sizeof(uint64_t)))) return rc;
    if (diag && (rc = ctx.alloc(&d_nodes, n * sizeof(uint64_t)))) return rc;
    if ((rc = ctx.alloc(&d_tot, 32 * sizeof(uint64_t) + 16))) return rc;
    int *d_status = reinterpret_cast<int *>(d_tot + 32);
    CallEvents evs;
    if ((rc = evs.init())) return rc;
    cudaEvent_t *ev = evs.e;
    cudaEventRecord(ev[0], ctx.s);
    rc = m ? cuda_rc(cudaMemcpyAsync(d_kids, kids.data(), m * sizeof(nq_prefix),
                                     cudaMemcpyHostToDevice, ctx.s))
           : NQ_OK;
    if (!rc) rc = cuda_rc(cudaMemsetAsync(d_tot, 0, 32 * sizeof(uint64_t) + 16, ctx.s));
    cudaEventRecord(ev[1], ctx.s);
    Plan p{};
    if (!rc)
        rc = enqueue_search(d_kids, m, 0, kid_min_d, max_n, d_counts, d_nodes, d_tot, cfg,
                            nullptr, ctx.s, &p, d_status, n);
    cudaEventRecord(ev[2], ctx.s);
    if (!rc)
        rc = cuda_rc(cudaMemcpyAsync(h_counts, d_counts, n * sizeof(uint64_t),
                                     cudaMemcpyDeviceToHost, ctx.s));
    if (!rc && diag)
        rc = cuda_rc(cudaMemcpyAsync(h_nodes, d_nodes, n * sizeof(uint64_t),
                                     cudaMemcpyDeviceToHost, ctx.s));
    if (!rc && h_totals)
        rc = cuda_rc(cudaMemcpyAsync(h_totals, d_tot, 32 * sizeof(uint64_t),
                                     cudaMemcpyDeviceToHost, ctx.s));
    if (cudaStreamSynchronize(ctx.s) != cudaSuccess) return NQ_ECUDA;
    if (rc) return rc;
    const int st = take_status(d_status, ctx.s);
    if (st) return st;
    if (diag)
        for (uint64_t i = 0; i < n; ++i) h_nodes[i] += extra[i];
    if (rows_used) *rows_used = r;
    if (timing) {
        float up = 0, kern = 0;
        cudaEventElapsedTime(&up, ev[0], ev[1]);
        cudaEventElapsedTime(&kern, ev[1], ev[2]);
        timing->enumerate_ms = split_ms;
        timing->upload_ms = up;
        timing->kernel_ms = kern;
        timing->prefixes = m;
        timing->d = kid_min_d;
        timing->layout = p.layout;
        timing->block = p.block;
        timing->grid = p.grid;
        timing->total_ms = ms_since(t_start);
    }
    return NQ_OK;
}

// ---------------------------------------------------------------------------
// Partial-board constraints: every listed queen's row may take only its
// column, every other row loses the cells the listed queens attack.
// ---------------------------------------------------------------------------
extern "C" int nq_count_constrained(int N, const nq_queen *q, int k, uint64_t *count_out) {
    if (!count_out) return NQ_EINVAL;
    uint32_t allowed[32];
    bool conflict = false;
    const int rc0 = constraint_masks(N, q, k, allowed, &conflict);
    if (rc0) return rc0;
    if (conflict) {
        *count_out = 0;
        return NQ_OK;
    }
    if (k == 0) {  // nothing given: the board's symmetries hold
        nq_config cfg{};  // (of nq_total's, NQ_LAYOUT and NQ_D do not reach this call)
        cfg.layout = NQ_LAYOUT_REGP;
        const int b = std::min(N, kTotalRows);
        return total_split(N, b, b, &cfg, count_out, nullptr);
    }
    for (int r = 0; r < N; ++r)
        if (!allowed[r]) {  // a row that the given queens leave no column
            *count_out = 0;
            return NQ_OK;
        }
    // The whole board as one record; the launch splits it (plan_records).
    const nq_prefix root{0, 0, 0, NQ_META(1, N, 0, 0)};
    unsigned char *stage = static_cast<unsigned char *>(t_stage.get(kHead + sizeof(root)));
    if (!stage) return NQ_ENOMEM;
    *staged_records(stage) = root;
    return search_staged(N, 0, stage, 1, nullptr, allowed, count_out, nullptr, [] { return NQ_OK; });
}
