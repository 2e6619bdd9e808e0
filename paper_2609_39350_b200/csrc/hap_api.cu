// Host side of libhap: descriptor validation and copies, enumeration of the 6-D space,
// work partitioning, kernel launches.  Every step of the hot path runs in the kernels of
// hap_device.cuh; nothing here evaluates a cost.
#include "hap_device.cuh"
#include "hap_tree.cuh"
#include "hap_tree_host.h"
#include "hap_joint.cuh"

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cmath>
#include <cstring>
#include <array>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <unordered_map>
#include <vector>
#if defined(__SSE2__)
#include <emmintrin.h>
#endif

using namespace hap;

// read-only view of a vector that someone else keeps alive
template <typename E> struct View {
    const E *ptr = nullptr;
    size_t n = 0;
    size_t size() const { return n; }
    bool empty() const { return n == 0; }
    const E *data() const { return ptr; }
    const E &operator[](size_t i) const { return ptr[i]; }
    const E *begin() const { return ptr; }
    const E *end() const { return ptr + n; }
};

// Configuration table and prefix trees on a device, laid out once and shared by the problems of the process whose model
// dimensions, cluster and search options are the same (they do not depend on the profiled tables).
struct DeviceImage {
    int device = 0;
    unsigned char *base = nullptr;
    hap_pconf *d_pconf = nullptr;
    TreeClass *d_cls = nullptr;
    std::vector<TreeClass> cls;            // the classes that walk a tree, deepest pipeline first (device pointers inside)
    std::vector<int> tree_of;              // per PP class: its entry in cls, -1 for none
    std::vector<unsigned> masks_used;      // per PP class: type masks that occur
    size_t rec_total = 0, prep_smem = 0;
    DeviceImage() = default;
    DeviceImage(const DeviceImage &) = delete;
    DeviceImage &operator=(const DeviceImage &) = delete;
    ~DeviceImage();
};

struct hap_problem {
    int device = 0;
    // host copies
    hap_model model{};
    std::vector<uint8_t> kind;
    int T = 0;
    std::vector<int64_t> P, C, cap_eff;
    std::vector<int32_t> node_size, node_type, tp_list, cp_list, mb_list, ep_list, pp_list, tpe_list, xi_q, tau_q;
    std::vector<double> bw_intra, node_bw_inter, eta, croute, alpha, rho, act_coef, copt;
    std::vector<uint32_t> rc_masks;
    hap_profile prof{};
    hap_search_opts opts{};
    int64_t m[HAP_MAX_TYPES] = {0, 0, 0, 0};
    int64_t W = 0;
    // enumeration: the configuration table and the work items belong to the per-process enumeration result that
    // `enum_ref` keeps alive (problems with the same lists share one)
    bool enumerated = false;
    View<hap_pconf> pconfs;
    uint64_t n_cand = 0;
    View<WorkItem> items;                  // grouped by PP class, heaviest class first
    std::shared_ptr<const void> enum_ref;
    std::shared_ptr<const DeviceImage> image;
    struct PpClass { int PP; int warps; size_t smem; size_t item_lo, item_hi; u64 map_base; bool has_tab; bool multiset; unsigned masks_used;
                     int tree = -1;                          // entry in image->cls; -1: the class runs in pipeline_dp_kernel only
                     cudaStream_t stream = nullptr; cudaEvent_t done = nullptr;
                     mutable bool tab_valid = false; };      // the device table of decoded mappings of this class has been filled
    std::vector<PpClass> classes;
    bool all_trees = false;
    u64 tab_bytes = 0;
    // device
    DevConst dc{};
    TreeArgs targs{};
    LiveArgs largs{};
    bool state_dirty = false;              // a pass was cut short between its kernels: its counters have to be cleared
    double *d_tables = nullptr;            // all six tables in one allocation (behind the range flag's slot)
    u64 *d_range = nullptr;                // sticky flag: a cost left the supported value range
    unsigned char *d_arena = nullptr;      // what every pass needs, in one allocation
    i64 *d_coef = nullptr;
    TypeConst *d_tc = nullptr;             // scratch: per (configuration, type) constants of the layer costs
    i64 *d_lb = nullptr;                   // scratch: per-configuration lower bound on the summed stage time
    i64 *d_pcost = nullptr;                // per-block partial minima
    u64 *d_pindex = nullptr;
    PlanSlot *d_plans = nullptr;           // per block of a tree search the plan of its best candidate
    u64 *d_counters = nullptr;             // general kernel: [0] evaluated [1] feasible [2] pruned [3] incumbent
    i64 *d_best = nullptr;                 // (cost, index) of the search
    void *d_single = nullptr;              // outputs of the one-candidate re-evaluation
    size_t n_partial = 0;                  // allocated slots of the partial minima
    // general kernel, layer-cost array (first use)
    unsigned char *d_gen_arena = nullptr;
    bool gen_ready = false;
    WorkItem *d_items = nullptr;
    i64 *d_c2 = nullptr;
    uint8_t *d_maptab = nullptr;           // decoded mappings of every class that is small enough
    double *d_c2f = nullptr, *d_coeff = nullptr;   // fp64-mode layer costs and coefficients (first use)
    i64 *d_fcost = nullptr;                // fp64-mode search through the general kernel: per-candidate costs (bit patterns), first use
    i64 *d_cand_lb = nullptr;              // scratch of the refinement searches: per-candidate bottleneck, then lower bound (first use)
    // joint device-state recurrence (built on first use)
    struct JointHost { JointClass jc; std::vector<unsigned> ids; unsigned *d_ids = nullptr; int *d_arrays = nullptr; size_t smem = 0; };
    std::vector<JointHost> joint;
    i64 *d_joint_scratch = nullptr;
    int joint_grid = 0;
    // ... in the form of a search over reachable end layers: by 64-bit words per state
    struct ReachHost { std::vector<JointReach> classes; std::vector<unsigned> ids; unsigned char *d = nullptr; size_t o_ids = 0, smem = 0; };
    ReachHost reach[kReachWords];
    bool joint_ready = false;
    TreeResult *host_result = nullptr;     // page-locked, mapped: the last block of a search writes the plan here
    int timed = 0;                         // 1: events around the last pass, 2: the tree kernels' own time stamps
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    cudaEvent_t ev_upload = nullptr;       // the upload of the tables
    bool upload_pending = false;           // no completed call has waited for that upload yet
    cudaEvent_t ev_fork = nullptr;         // general kernel: classes run on their own streams between this event and their `done` events
    bool in_flight = false;                // an asynchronous call has not been waited for
    unsigned long long last_id = 0;        // the stream it went to (its id: handles are used again)
    bool last_default = false;             // that was the default stream; else ev_order stands behind the call
    cudaEvent_t ev_order = nullptr;
    bool captured = false;                 // a graph that the caller holds may run calls of this problem
    bool upload_waited = false;            // a call on stream upload_id has waited for the upload: later ones on it are behind it
    unsigned long long upload_id = 0;
    std::string err;
};

// device-side landing area of the one-candidate re-evaluation that fills the plan
struct SingleOut {
    i64 cost, bott, detail[3];
    uint8_t part[HAP_MAX_PP], rec[HAP_MAX_PP];
    hap_candidate cand;
};

// The side streams the PP classes run on are shared by all problems of a device and live until the process ends:
// creating half a dozen streams costs more than a whole search.  Index = position of the class in the problem,
// classes ordered from the deepest pipeline down.  A block of a deep class is a long chain of short steps (one
// barrier-separated depth of its tree per stage and policy) that leaves most issue slots idle, a block of the class
// with the most mappings keeps them busy but fills an SM's registers: the deep classes' blocks should be resident
// first and the busy class should fill in behind them, so the streams get priorities in class order: the phase is
// shorter and takes the same time in every pass.
static cudaStream_t pooled_stream(int device, size_t index)
{
    static std::mutex mu;
    static cudaStream_t pool[64][HAP_MAX_PP + 1];
    std::lock_guard<std::mutex> lock(mu);
    cudaStream_t &s = pool[device & 63][index % (HAP_MAX_PP + 1)];
    if (!s) {
        int least = 0, greatest = 0;                    // numerically: greatest priority <= least priority
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) { least = greatest = 0; cudaGetLastError(); }
        const int pr = std::min(least, greatest + (int)(index % (HAP_MAX_PP + 1)));
        if (cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, pr) != cudaSuccess) s = nullptr;
    }
    return s;
}

// Uploads (profiled tables, configuration table, prefix trees) go through page-locked staging buffers and an
// upload stream of their own, asynchronously: the host builds the next thing while the copy runs, and the first call
// that uses the data waits for the upload's event.  The staging buffers are kept per process (a page-locked
// allocation costs more than a search); a buffer is reused once the copy that last read it has completed.
namespace {
struct PinnedBuf { void *ptr = nullptr; size_t cap = 0; cudaEvent_t done = nullptr; int device = -1; bool busy = false; };   // busy: being filled
struct UploadState {
    std::mutex mu;
    std::vector<PinnedBuf> bufs;
    cudaStream_t stream[64] = {};
};
UploadState &upload_state() { static UploadState *u = new UploadState(); return *u; }      // never destroyed
constexpr size_t kPinnedBufs = 8;
constexpr size_t kRangeSlot = 512;          // bytes in front of a problem's tables that hold its range flag and a pass's counters
static_assert(16 + sizeof(TreeState) <= kRangeSlot, "flag, then counters");
constexpr unsigned kTreeSlots = 4096;       // per-block minima of the tree kernel
}  // namespace

static cudaStream_t upload_stream(int device)
{
    UploadState &u = upload_state();
    std::lock_guard<std::mutex> lock(u.mu);
    cudaStream_t &s = u.stream[device & 63];
    if (!s && cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) s = nullptr;
    return s;
}

// a page-locked buffer of at least `bytes` whose previous copy (if any) has completed, marked busy until pinned_put;
// nullptr: use pageable memory
static PinnedBuf *pinned_get(int device, size_t bytes)
{
    UploadState &u = upload_state();
    std::lock_guard<std::mutex> lock(u.mu);
    PinnedBuf *small = nullptr;                             // an idle buffer of the device that is too small
    for (auto &b : u.bufs) {
        if (b.device != device || b.busy || cudaEventQuery(b.done) != cudaSuccess) continue;
        if (b.cap >= bytes) { b.busy = true; return &b; }
        small = &b;
    }
    cudaGetLastError();                                  // cudaErrorNotReady of a buffer in flight is not an error
    if (u.bufs.size() >= kPinnedBufs) {                  // regrow an idle one
        if (!small) return nullptr;
        cudaFreeHost(small->ptr); small->ptr = nullptr; small->cap = 0;
        if (cudaHostAlloc(&small->ptr, bytes, cudaHostAllocDefault) != cudaSuccess) { cudaGetLastError(); small->ptr = nullptr; return nullptr; }
        small->cap = bytes;
        small->busy = true;
        return small;
    }
    u.bufs.reserve(kPinnedBufs);                          // pointers into the vector stay valid
    PinnedBuf b;
    b.device = device;
    b.cap = std::max<size_t>(bytes, 1 << 20);
    if (cudaHostAlloc(&b.ptr, b.cap, cudaHostAllocDefault) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    if (cudaEventCreateWithFlags(&b.done, cudaEventDisableTiming) != cudaSuccess) { cudaFreeHost(b.ptr); cudaGetLastError(); return nullptr; }
    b.busy = true;
    u.bufs.push_back(b);
    return &u.bufs.back();
}

static void pinned_put(PinnedBuf *b)
{
    std::lock_guard<std::mutex> lock(upload_state().mu);
    b->busy = false;
}

// host -> device copy of `bytes` that `fill` writes into a staging buffer; asynchronous when a page-locked buffer
// and the upload stream are available (the problem's upload event then marks its completion), synchronous otherwise
// Events without timing are pooled per process: creating and destroying a handful per problem costs as much as a launch.
namespace {
struct EventPool { std::mutex mu; std::vector<cudaEvent_t> idle[64]; };
EventPool &event_pool() { static EventPool *e = new EventPool(); return *e; }           // never destroyed
constexpr size_t kPooledEvents = 64;
}  // namespace

static cudaEvent_t pooled_event(int device)
{
    EventPool &ep = event_pool();
    {
        std::lock_guard<std::mutex> lock(ep.mu);
        auto &v = ep.idle[device & 63];
        if (!v.empty()) { cudaEvent_t e = v.back(); v.pop_back(); return e; }
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return e;
}

static void pooled_event_put(int device, cudaEvent_t e)
{
    if (!e) return;
    EventPool &ep = event_pool();
    {
        std::lock_guard<std::mutex> lock(ep.mu);
        auto &v = ep.idle[device & 63];
        if (v.size() < kPooledEvents) { v.push_back(e); return; }
    }
    cudaEventDestroy(e);
}

// Page-locked, mapped result slots of searches: one page per process, a slot per problem that has searched.
namespace {
constexpr int kResultSlots = 128;
struct ResultPool { std::mutex mu; unsigned char *base = nullptr; bool failed = false; std::vector<int> idle; };
ResultPool &result_pool() { static ResultPool *r = new ResultPool(); return *r; }       // never destroyed
constexpr size_t kResultStride = (sizeof(TreeResult) + 255) / 256 * 256;
}  // namespace

static TreeResult *result_slot_get()
{
    ResultPool &rp = result_pool();
    std::lock_guard<std::mutex> lock(rp.mu);
    if (!rp.base && !rp.failed) {
        void *ptr = nullptr;
        if (cudaHostAlloc(&ptr, kResultSlots * kResultStride, cudaHostAllocMapped | cudaHostAllocPortable) != cudaSuccess) { cudaGetLastError(); rp.failed = true; }
        else { rp.base = static_cast<unsigned char *>(ptr); for (int i = kResultSlots; i-- > 0;) rp.idle.push_back(i); }
    }
    if (rp.idle.empty()) return nullptr;                     // the caller copies from the device instead
    const int i = rp.idle.back();
    rp.idle.pop_back();
    return reinterpret_cast<TreeResult *>(rp.base + (size_t)i * kResultStride);
}

static void result_slot_put(TreeResult *r)
{
    if (!r) return;
    ResultPool &rp = result_pool();
    std::lock_guard<std::mutex> lock(rp.mu);
    rp.idle.push_back((int)((reinterpret_cast<unsigned char *>(r) - rp.base) / (ptrdiff_t)kResultStride));
}

template <class Fill>
static cudaError_t upload(hap_problem *p, void *dst, size_t bytes, Fill fill)
{
    cudaStream_t us = upload_stream(p->device);
    PinnedBuf *pb = us ? pinned_get(p->device, bytes) : nullptr;
    if (!pb) {
        std::vector<unsigned char> stage(bytes, 0);
        if (!fill(stage.data())) return cudaErrorInvalidValue;
        return cudaMemcpy(dst, stage.data(), bytes, cudaMemcpyHostToDevice);
    }
    struct Put { PinnedBuf *b; ~Put() { pinned_put(b); } } put{pb};
    if (!fill(static_cast<unsigned char *>(pb->ptr))) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemcpyAsync(dst, pb->ptr, bytes, cudaMemcpyHostToDevice, us);
    if (e != cudaSuccess) return e;
    if ((e = cudaEventRecord(pb->done, us)) != cudaSuccess) return e;
    if (!p->ev_upload && !(p->ev_upload = pooled_event(p->device))) return cudaErrorUnknown;
    if ((e = cudaEventRecord(p->ev_upload, us)) != cudaSuccess) return e;
    p->upload_pending = true;
    return cudaSuccess;
}

// a call that hands data to the host waits for the upload itself; every other one lets its stream wait
static cudaError_t uploads_done(hap_problem *p)
{
    if (!p->upload_pending) return cudaSuccess;
    p->upload_pending = false;
    return cudaEventSynchronize(p->ev_upload);
}


// Device memory of destroyed problems is kept for the next problem of the process: allocating and freeing the
// three arenas of a problem costs about as much as the search itself.  A freed block serves a later request
// of its device that it fits with at most a quarter (plus 1 MiB) to spare.  At most kCacheBlocks blocks and kCacheBytes
// bytes are held; hap_release_cached_memory() returns everything to the driver.
namespace {
struct CachedBlock { int device; size_t bytes; void *ptr; };
struct MemCache {
    std::mutex mu;
    std::vector<CachedBlock> idle;
    std::unordered_map<void *, CachedBlock> live;
    size_t idle_bytes = 0;
};
constexpr size_t kCacheBlocks = 24;
constexpr size_t kCacheBytes = 4ull << 30;
MemCache &mem_cache() { static MemCache *c = new MemCache(); return *c; }     // never destroyed: outlives static teardown
}  // namespace

static cudaError_t cached_malloc(int device, void **out, size_t bytes)
{
    MemCache &mc = mem_cache();
    bytes = (std::max<size_t>(bytes, 1) + 0xffff) & ~(size_t)0xffff;
    std::lock_guard<std::mutex> lock(mc.mu);
    size_t best = mc.idle.size();
    for (size_t i = 0; i < mc.idle.size(); ++i) {
        const CachedBlock &b = mc.idle[i];
        if (b.device != device || b.bytes < bytes || b.bytes > bytes + bytes / 4 + (1u << 20)) continue;
        if (best == mc.idle.size() || b.bytes < mc.idle[best].bytes) best = i;
    }
    if (best != mc.idle.size()) {
        const CachedBlock b = mc.idle[best];
        mc.idle.erase(mc.idle.begin() + (long)best);
        mc.idle_bytes -= b.bytes;
        mc.live[b.ptr] = b;
        *out = b.ptr;
        return cudaSuccess;
    }
    void *ptr = nullptr;
    cudaError_t e = cudaMalloc(&ptr, bytes);
    if (e == cudaErrorMemoryAllocation) {           // give the idle blocks of this device back and try once more
        cudaGetLastError();
        for (size_t i = mc.idle.size(); i-- > 0;)
            if (mc.idle[i].device == device) { cudaFree(mc.idle[i].ptr); mc.idle_bytes -= mc.idle[i].bytes; mc.idle.erase(mc.idle.begin() + (long)i); }
        e = cudaMalloc(&ptr, bytes);
    }
    if (e != cudaSuccess) { *out = nullptr; return e; }
    mc.live[ptr] = CachedBlock{device, bytes, ptr};
    *out = ptr;
    return cudaSuccess;
}

// The caller has made sure that no work that touches the block is still in flight.
static void cached_free(void *ptr)
{
    if (!ptr) return;
    MemCache &mc = mem_cache();
    std::lock_guard<std::mutex> lock(mc.mu);
    auto it = mc.live.find(ptr);
    if (it == mc.live.end()) { cudaFree(ptr); return; }
    const CachedBlock b = it->second;
    mc.live.erase(it);
    if (b.bytes > kCacheBytes) { cudaFree(ptr); return; }
    // full: the block that has been idle longest goes (sizes that are no longer asked for would otherwise keep every new size
    // out, and each problem of that size would pay for an allocation and a release: 0.8 ms instead of 0.2)
    while (mc.idle.size() >= kCacheBlocks || mc.idle_bytes + b.bytes > kCacheBytes) {
        cudaFree(mc.idle.front().ptr);
        mc.idle_bytes -= mc.idle.front().bytes;
        mc.idle.erase(mc.idle.begin());
    }
    mc.idle.push_back(b);
    mc.idle_bytes += b.bytes;
}


DeviceImage::~DeviceImage() { cached_free(base); }

// device images kept per process, by device and everything they are derived from
namespace {
struct ImageCache { std::mutex mu; std::map<std::string, std::shared_ptr<const DeviceImage>> map; };
ImageCache &image_cache() { static ImageCache *c = new ImageCache(); return *c; }       // never destroyed
constexpr size_t kImages = 16;
}  // namespace

extern "C" hap_status hap_release_cached_memory(void)
{
    {   // images that no problem holds go back to the cache of device memory first
        ImageCache &ic = image_cache();
        std::map<std::string, std::shared_ptr<const DeviceImage>> drop;
        std::lock_guard<std::mutex> lock(ic.mu);
        drop.swap(ic.map);
    }
    MemCache &mc = mem_cache();
    std::lock_guard<std::mutex> lock(mc.mu);
    int prev = 0;
    const bool have_prev = cudaGetDevice(&prev) == cudaSuccess;
    hap_status st = HAP_OK;
    for (const CachedBlock &b : mc.idle)
        if (cudaSetDevice(b.device) != cudaSuccess || cudaFree(b.ptr) != cudaSuccess) st = HAP_E_CUDA;
    mc.idle.clear();
    mc.idle_bytes = 0;
    if (have_prev) cudaSetDevice(prev);
    if (st != HAP_OK) cudaGetLastError();
    return st;
}

static hap_status fail(hap_problem *p, hap_status s, const char *fmt, ...)
{
    if (p) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof(buf), fmt, ap);
        va_end(ap);
        p->err = buf;
    }
    return s;
}

static hap_status argmin_launch(hap_problem *p, const hap::i64 *dev_cost, uint64_t count, hap::i64 *dev_out, cudaStream_t st, hap::i64 init);

#define CUDA_TRY(p, call)                                                                          \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return fail(p, e_ == cudaErrorMemoryAllocation ? HAP_E_NOMEM : HAP_E_CUDA, "%s: %s", #call, \
                        cudaGetErrorString(e_));                                                   \
    } while (0)

extern "C" const char *hap_status_str(hap_status s)
{
    switch (s) {
    case HAP_OK: return "HAP_OK";
    case HAP_E_INVALID: return "HAP_E_INVALID";
    case HAP_E_NOMEM: return "HAP_E_NOMEM";
    case HAP_E_CUDA: return "HAP_E_CUDA";
    case HAP_E_RANGE: return "HAP_E_RANGE";
    case HAP_E_STATE: return "HAP_E_STATE";
    case HAP_E_INFEASIBLE: return "HAP_E_INFEASIBLE";
    }
    return "HAP_E_?";
}

extern "C" const char *hap_last_error(const hap_problem *p) { return p ? p->err.c_str() : "null problem"; }

static void release_device(hap_problem *p)
{
    // nothing of this problem may still be running when its memory goes back to the cache
    if (p->upload_pending) { cudaEventSynchronize(p->ev_upload); p->upload_pending = false; }
    if (p->captured) cudaDeviceSynchronize();
    else if (p->in_flight) p->last_default ? cudaStreamSynchronize(cudaStreamLegacy) : cudaEventSynchronize(p->ev_order);
    cached_free(p->d_tables); cached_free(p->d_arena); cached_free(p->d_gen_arena);
    cached_free(p->d_joint_scratch);
    for (auto &r : p->reach) cached_free(r.d);
    for (auto &j : p->joint) { cached_free(j.d_ids); cached_free(j.d_arrays); }
    cached_free(p->d_c2f); cached_free(p->d_coeff); cached_free(p->d_fcost); cached_free(p->d_cand_lb);
    for (auto &e : p->ev) if (e) cudaEventDestroy(e);
    pooled_event_put(p->device, p->ev_fork); pooled_event_put(p->device, p->ev_upload); pooled_event_put(p->device, p->ev_order);
    for (auto &cl : p->classes) pooled_event_put(p->device, cl.done);              // the class streams belong to the pool
    result_slot_put(p->host_result);
}

extern "C" void hap_problem_destroy(hap_problem *p)
{
    if (!p) return;
    cudaSetDevice(p->device);
    release_device(p);
    delete p;
}

template <class T>
static bool copy_list(std::vector<T> &dst, const T *src, int n)
{
    if (n < 0 || (n > 0 && !src)) return false;
    dst.assign(src, src + n);
    return true;
}

static bool finite_nonneg(const std::vector<double> &v)
{
    for (double x : v) if (!(x >= 0.0) || x > 1e300) return false;
    return true;
}

extern "C" hap_status hap_problem_create(const hap_model *mo, const hap_cluster *cl, const hap_profile *pf,
                                         const hap_search_opts *so, hap_problem **out)
{
    if (!out) return HAP_E_INVALID;
    *out = nullptr;
    if (!mo || !cl || !pf || !so) return HAP_E_INVALID;
    hap_problem *p = new (std::nothrow) hap_problem();
    if (!p) return HAP_E_NOMEM;
    // the problem is handed back even on failure paths below only through *out on success
    struct Guard { hap_problem *p; bool keep = false; ~Guard() { if (!keep) { release_device(p); delete p; } } } guard{p};

    // ---- validate and copy ------------------------------------------------------------------
    const int N = mo->N, T = cl->n_types;
    if (N < 1 || N > HAP_MAX_LAYERS || !mo->kind) return HAP_E_INVALID;
    if (T < 1 || T > HAP_MAX_TYPES || cl->n_nodes < 1) return HAP_E_INVALID;
    if ((int64_t)mo->GB * mo->N > (1ll << 22)) return HAP_E_RANGE;     // keeps M * sum of layer times below 2^62
    if (mo->S < 1 || mo->H < 1 || mo->E < 1 || mo->k < 1 || mo->nq < 1 || mo->nkv < 1 || mo->GB < 1 || mo->V < 0 ||
        mo->n_shared < 0 || mo->F_dense < 0 || mo->F_exp < 0 || !(mo->beta > 0.0) || mo->nq % mo->nkv != 0)
        return HAP_E_INVALID;
    if (pf->ntp < 1 || pf->ncp < 1 || pf->nmb < 1 || pf->nep < 1 || pf->ntp > HAP_MAX_LIST || pf->ncp > HAP_MAX_LIST ||
        pf->nmb > HAP_MAX_LIST || pf->nep > HAP_MAX_LIST || pf->R < 1 || pf->R > HAP_MAX_RC)
        return HAP_E_INVALID;
    if (so->npp < 1 || so->npp > HAP_MAX_LIST || so->ntpe < 1 || so->ntpe > HAP_MAX_LIST || so->n_rc < 1 ||
        so->n_rc > HAP_MAX_RC_MASKS || so->map_cap < 1 || so->map_cap > (1ull << 56) || so->delta_q >= 1024)
        return HAP_E_INVALID;
    p->model = *mo;
    p->kind.assign(mo->kind, mo->kind + N);
    p->model.kind = nullptr;
    for (uint8_t kd : p->kind) if (kd > 1) return HAP_E_INVALID;
    p->T = T;
    bool ok = copy_list(p->P, cl->P, T) && copy_list(p->C, cl->C, T) && copy_list(p->node_size, cl->node_size, T) &&
              copy_list(p->bw_intra, cl->bw_intra, T) && copy_list(p->node_type, cl->node_type, cl->n_nodes) &&
              copy_list(p->node_bw_inter, cl->node_bw_inter, cl->n_nodes) &&
              copy_list(p->tp_list, pf->tp_list, pf->ntp) && copy_list(p->cp_list, pf->cp_list, pf->ncp) &&
              copy_list(p->mb_list, pf->mb_list, pf->nmb) && copy_list(p->ep_list, pf->ep_list, pf->nep) &&
              copy_list(p->eta, pf->eta, T) && copy_list(p->croute, pf->croute, T) && copy_list(p->alpha, pf->alpha, 3) &&
              copy_list(p->rho, pf->rho, pf->nep) && copy_list(p->act_coef, pf->act_coef, 2) &&
              copy_list(p->copt, pf->copt, T) && copy_list(p->cap_eff, pf->cap_eff, T) &&
              copy_list(p->xi_q, pf->xi_q, pf->R) && copy_list(p->tau_q, pf->tau_q, pf->R) &&
              copy_list(p->pp_list, so->pp_list, so->npp) && copy_list(p->tpe_list, so->tpe_list, so->ntpe) &&
              copy_list(p->rc_masks, so->rc_masks, so->n_rc);
    if (!ok || !pf->tdf || !pf->tdb || !pf->tff || !pf->tfb || !pf->tpre || !pf->tpost) return HAP_E_INVALID;
    p->prof = *pf;
    p->opts = *so;
    for (int h = 0; h < T; ++h) {
        if (p->P[h] < 1 || p->P[h] > (1ll << 40) || p->node_size[h] < 1 || !(p->bw_intra[h] > 0.0) || p->cap_eff[h] < 0 ||
            !(p->eta[h] > 0.0))
            return HAP_E_INVALID;
    }
    double bw_inter[HAP_MAX_TYPES];
    bool has[HAP_MAX_TYPES] = {false, false, false, false};
    for (int n = 0; n < cl->n_nodes; ++n) {
        const int t = p->node_type[n];
        if (t < 0 || t >= T || !(p->node_bw_inter[n] > 0.0)) return HAP_E_INVALID;
        p->m[t] += p->node_size[t];
        bw_inter[t] = has[t] ? std::min(bw_inter[t], p->node_bw_inter[n]) : p->node_bw_inter[n];
        has[t] = true;
    }
    for (int h = 0; h < T; ++h) { if (!has[h]) return HAP_E_INVALID; p->W += p->m[h]; }
    auto positive = [](const std::vector<int32_t> &v) { for (int x : v) if (x < 1) return false; return true; };
    for (size_t i = 0; i < p->pp_list.size(); ++i)                   // a repeated PP would enumerate its configurations twice
        for (size_t j = 0; j < i; ++j) if (p->pp_list[i] == p->pp_list[j]) return HAP_E_INVALID;
    if (!positive(p->tp_list) || !positive(p->cp_list) || !positive(p->mb_list) || !positive(p->ep_list) ||
        !positive(p->pp_list) || !positive(p->tpe_list))
        return HAP_E_INVALID;
    for (int r = 0; r < pf->R; ++r) if (p->xi_q[r] < 0 || p->tau_q[r] < 0 || p->xi_q[r] > (1 << 20) || p->tau_q[r] > (1 << 20)) return HAP_E_INVALID;
    for (uint32_t mk : p->rc_masks) if (mk == 0 || mk >= (1u << pf->R)) return HAP_E_INVALID;
    if (!finite_nonneg(p->croute) || !finite_nonneg(p->alpha) || !finite_nonneg(p->act_coef) || !finite_nonneg(p->copt) ||
        !(pf->kappa >= 0.0) || !(pf->chi > 0.0) || !(pf->gamma >= 0.0) || !(pf->ovl_tp >= 0.0) || !(pf->ovl_cp >= 0.0) ||
        !(pf->ovl_dp >= 0.0) || !(pf->capf >= 0.0))
        return HAP_E_INVALID;
    for (double r : p->rho) if (!(r >= 1.0)) return HAP_E_INVALID;
    if (pf->n_fsize < 0 || pf->n_fsize > HAP_MAX_LIST || (pf->n_fsize > 0 && (!pf->fsize || !pf->feff))) return HAP_E_INVALID;
    for (int i = 0; i < pf->n_fsize; ++i) {
        if (!(pf->fsize[i] > 0.0) || !std::isfinite(pf->fsize[i]) || (i > 0 && !(pf->fsize[i] > pf->fsize[i - 1]))) return HAP_E_INVALID;
        for (int c = 0; c < 3; ++c) { const double e = pf->feff[c * pf->n_fsize + i]; if (!(e > 0.0 && e <= 1.0)) return HAP_E_INVALID; }
    }

    const size_t n4 = (size_t)T * pf->ntp * pf->ncp * pf->nmb, n5 = n4 * N;
    // device layout: the four per-layer tables interleaved entry by entry (one 32-byte record per (type, row, layer):
    // the layer-cost kernel reads a record with two 16-byte loads), then tpre, then tpost
    const size_t n_tab = 4 * n5 + 2 * n4;
    auto fill_tables = [&](unsigned char *dst) -> bool {
        double *__restrict__ tables = reinterpret_cast<double *>(dst);
        const double *__restrict__ A = pf->tdf, *__restrict__ B = pf->tdb, *__restrict__ F = pf->tff, *__restrict__ G = pf->tfb;
        bool ok = true;
        size_t i = 0;
        // t_dense includes its FFN; every entry finite, non-negative, < 2^50 ns (NaN fails every comparison)
#if defined(__SSE2__)
        {   // two entries per step: the records are the 2 x 2 transposes of the four streams
            const __m128d zero = _mm_setzero_pd(), big = _mm_set1_pd(1e15);
            __m128d okv = _mm_castsi128_pd(_mm_set1_epi32(-1));
            for (; i + 2 <= n5; i += 2) {
                const __m128d a = _mm_loadu_pd(A + i), b = _mm_loadu_pd(B + i), c = _mm_loadu_pd(F + i), d = _mm_loadu_pd(G + i);
                double *rec = tables + 4 * i;
                _mm_storeu_pd(rec, _mm_unpacklo_pd(a, b)); _mm_storeu_pd(rec + 2, _mm_unpacklo_pd(c, d));
                _mm_storeu_pd(rec + 4, _mm_unpackhi_pd(a, b)); _mm_storeu_pd(rec + 6, _mm_unpackhi_pd(c, d));
                __m128d v = _mm_and_pd(_mm_cmpge_pd(a, c), _mm_cmpge_pd(b, d));
                v = _mm_and_pd(v, _mm_and_pd(_mm_cmpge_pd(c, zero), _mm_cmpge_pd(d, zero)));
                v = _mm_and_pd(v, _mm_and_pd(_mm_cmple_pd(a, big), _mm_cmple_pd(b, big)));
                okv = _mm_and_pd(okv, v);
            }
            ok = _mm_movemask_pd(okv) == 3;
        }
#endif
        for (; i < n5; ++i) {
            const double a = A[i], b = B[i], c = F[i], d = G[i];
            double *rec = tables + 4 * i;
            rec[0] = a; rec[1] = b; rec[2] = c; rec[3] = d;
            ok &= (a >= c) & (b >= d) & (c >= 0.0) & (d >= 0.0) & (a <= 1e15) & (b <= 1e15);
        }
        for (size_t i = 0; i < n4; ++i) {
            const double a = pf->tpre[i], b = pf->tpost[i];
            tables[4 * n5 + i] = a; tables[4 * n5 + n4 + i] = b;
            ok &= (a >= 0.0) & (b >= 0.0) & (a <= 1e15) & (b <= 1e15);
        }
        return ok;
    };

    // ---- device ------------------------------------------------------------------------------
    if (cudaGetDevice(&p->device) != cudaSuccess) return HAP_E_CUDA;
    // the range flag and the counters travel in front of the tables, cleared
    if (cached_malloc(p->device, (void **)&p->d_range, kRangeSlot + n_tab * sizeof(double)) != cudaSuccess) return HAP_E_NOMEM;
    p->d_tables = reinterpret_cast<double *>(p->d_range);                   // (the allocation, until release)
    {
        const cudaError_t e = upload(p, p->d_range, kRangeSlot + n_tab * sizeof(double), [&](unsigned char *dst) {
            std::memset(dst, 0, kRangeSlot);
            return fill_tables(dst + kRangeSlot); });
        if (e == cudaErrorInvalidValue) { cudaGetLastError(); return HAP_E_INVALID; }
        if (e != cudaSuccess) return HAP_E_CUDA;
    }

    DevConst &dc = p->dc;
    std::memset(&dc, 0, sizeof(dc));
    dc.N = N; dc.T = T; dc.R = pf->R; dc.n_rc = so->n_rc; dc.ntp = pf->ntp; dc.ncp = pf->ncp; dc.nmb = pf->nmb; dc.nep = pf->nep;
    dc.S = mo->S; dc.H = mo->H; dc.E = mo->E; dc.k = mo->k; dc.n_shared = mo->n_shared; dc.F_dense = mo->F_dense;
    dc.F_exp = mo->F_exp; dc.nq = mo->nq; dc.nkv = mo->nkv; dc.V = mo->V; dc.GB = mo->GB; dc.delta_q = so->delta_q; dc.eta_q = so->eta_q; dc.uniform = (so->flags & HAP_OPT_UNIFORM) != 0;
    dc.het_dispatch = (so->flags & HAP_OPT_HETERO_DISPATCH) != 0;
    dc.beta = mo->beta; dc.kappa = pf->kappa; dc.chi = pf->chi; dc.gamma = pf->gamma; dc.ovl_tp = pf->ovl_tp;
    dc.ovl_cp = pf->ovl_cp; dc.ovl_dp = pf->ovl_dp; dc.capf = pf->capf;
    for (int i = 0; i < 3; ++i) dc.alpha[i] = p->alpha[i];
    for (int h = 0; h < T; ++h) {
        dc.eta[h] = p->eta[h]; dc.croute[h] = p->croute[h]; dc.copt[h] = p->copt[h]; dc.bw_intra[h] = p->bw_intra[h];
        dc.bw_inter[h] = bw_inter[h]; dc.P[h] = p->P[h]; dc.cap_eff[h] = p->cap_eff[h]; dc.m[h] = p->m[h];
        dc.node_size[h] = p->node_size[h];
    }
    dc.act_coef[0] = p->act_coef[0]; dc.act_coef[1] = p->act_coef[1];
    for (int i = 0; i < pf->nep; ++i) dc.rho[i] = p->rho[i];
    for (int i = 0; i < so->n_rc; ++i) dc.rc_masks[i] = p->rc_masks[i];
    {   // evaluation order of the policies: more allowed levels first (stable), and who contains whom
        std::vector<int> order(so->n_rc);
        for (int i = 0; i < so->n_rc; ++i) order[i] = i;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
            return __builtin_popcount(p->rc_masks[a]) > __builtin_popcount(p->rc_masks[b]);
        });
        for (int j = 0; j < so->n_rc; ++j) {
            dc.rc_order[j] = order[j];
            dc.rc_sup[j] = 0;
            for (int q = 0; q < j; ++q)
                if ((p->rc_masks[order[q]] & p->rc_masks[order[j]]) == p->rc_masks[order[j]]) dc.rc_sup[j] |= 1u << q;
        }
    }
    dc.n_fsize = pf->n_fsize;
    for (int i = 0; i < pf->n_fsize; ++i) {
        dc.fsize[i] = pf->fsize[i];
        for (int c = 0; c < 3; ++c) dc.feff[c][i] = pf->feff[c * pf->n_fsize + i];
    }
    dc.tau_linear = 1;
    for (int r = 0; r < pf->R; ++r) { dc.xi_q[r] = p->xi_q[r]; dc.tau_q[r] = p->tau_q[r]; if (p->tau_q[r] % 1024) dc.tau_linear = 0; }
    for (int l = 0; l < N; ++l) if (p->kind[l] == HAP_MOE) dc.kindbits[l >> 6] |= 1ull << (l & 63);
    dc.kind_uniform_from = N - 1;
    while (dc.kind_uniform_from > 0 && p->kind[dc.kind_uniform_from - 1] == p->kind[N - 1]) --dc.kind_uniform_from;
    dc.tab4 = p->d_tables + kRangeSlot / sizeof(double);
    dc.tpre = dc.tab4 + 4 * n5; dc.tpost = dc.tpre + n4;

    guard.keep = true;
    *out = p;
    return HAP_OK;
}

// ------------------------------------------------------------------------------------------
// enumeration (host; at most a few thousand rows)
// ------------------------------------------------------------------------------------------
static uint64_t binom_sat(int n, int k, uint64_t sat)
{
    if (k < 0 || k > n) return 0;
    if (k > n - k) k = n - k;
    unsigned __int128 r = 1;
    for (int i = 1; i <= k; ++i) {
        r = r * (unsigned)(n - k + i) / (unsigned)i;
        if (r > sat) return sat;
    }
    return (uint64_t)r;
}

// distinct sequences with cnt[h] stages of type h: product of binomials, saturating
static uint64_t sequences_sat(const int *cnt, int T, uint64_t sat)
{
    int rem = 0;
    for (int h = 0; h < T; ++h) rem += cnt[h];
    unsigned __int128 r = 1;
    for (int h = 0; h < T; ++h) {
        r *= binom_sat(rem, cnt[h], sat);
        if (r > sat) return sat;
        rem -= cnt[h];
    }
    return (uint64_t)r;
}

template <class V> static void key_put(std::string &k, const V &v) { k.append(reinterpret_cast<const char *>(&v), sizeof(v)); }

static int sm_count(int device)
{
    static int n[64];                                       // (the same value whoever writes it)
    int &v = n[device & 63];
    if (!v && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) { cudaGetLastError(); v = 148; }
    return v;
}

// ---- per-process cache of the classes' prefix trees (host side) ------------------------------------------
namespace {
struct TreeCache { std::mutex mu; std::map<std::string, std::shared_ptr<const TreeClassHost>> map; };
TreeCache &tree_cache() { static TreeCache *c = new TreeCache(); return *c; }
constexpr size_t kTreeCacheEntries = 256;
}

// everything the mappings, the windows, the bands, the task lists and the split into parts depend on
static std::string tree_cache_key(const hap_problem *p, const hap_problem::PpClass &cl, bool want_tree)
{
    std::string k("hap-tree-3");
    const hap_pconf &rep = p->pconfs[p->items[cl.item_lo].p];
    const size_t n_conf = p->items[cl.item_hi - 1].p - p->items[cl.item_lo].p + 1;
    const int32_t head[] = {p->model.N, p->T, p->prof.R, cl.PP, rep.G, rep.mode, p->opts.delta_q, (int32_t)(p->opts.flags & HAP_OPT_UNIFORM),
                            p->dc.kind_uniform_from, (int32_t)n_conf, p->dc.tau_linear, (int32_t)want_tree, sm_count(p->device)};
    key_put(k, head);
    key_put(k, rep.nmap);
    for (int h = 0; h < p->T; ++h) { key_put(k, p->P[h]); key_put(k, p->cap_eff[h]); key_put(k, p->dc.m[h]); key_put(k, p->dc.node_size[h]); }
    return k;
}

static std::shared_ptr<const TreeClassHost> tree_of_class(const hap_problem *p, const hap_problem::PpClass &cl, bool want_tree)
{
    const std::string key = tree_cache_key(p, cl, want_tree);
    TreeCache &tc = tree_cache();
    {
        std::lock_guard<std::mutex> lock(tc.mu);
        auto it = tc.map.find(key);
        if (it != tc.map.end()) return it->second;
    }
    auto th = std::make_shared<TreeClassHost>();
    TreeInputs in{};
    in.dc = &p->dc; in.rep = p->pconfs[p->items[cl.item_lo].p];
    in.n_conf = p->items[cl.item_hi - 1].p - p->items[cl.item_lo].p + 1;
    in.n_sm = sm_count(p->device);
    in.want_tree = want_tree;
    TreeBuilder(in).build(*th);
    if (th->ok) {
        th->cls.n_conf = (u32)in.n_conf;
        // (a record or a part that does not leave room for one block on an SM: the class runs one warp per candidate)
        th->ok = tree_smem_bytes(th->cls) <= kTreeSmemMost && tree_prep_smem_bytes(th->cls, p->model.N, p->T) <= kTreeSmemMost;
    }
    std::lock_guard<std::mutex> lock(tc.mu);
    if (tc.map.size() >= kTreeCacheEntries) tc.map.clear();
    tc.map[key] = th;
    return th;
}

// ---- per-process cache of enumerations -----------------------------------------------------------------------
struct EnumResult {
    std::vector<hap_pconf> rows;
    std::vector<WorkItem> items;
    std::vector<hap_problem::PpClass> classes;       // streams and events are per problem: empty here
    uint64_t n_cand = 0;
    u64 tab_bytes = 0;
};
namespace {
struct EnumCache { std::mutex mu; std::map<std::string, std::shared_ptr<const EnumResult>> map; };
EnumCache &enum_cache() { static EnumCache *c = new EnumCache(); return *c; }
constexpr size_t kEnumCacheEntries = 64;
}

// every input of the enumeration loop nest and of the block shapes of the classes
static std::string enum_cache_key(const hap_problem *p)
{
    std::string k("hap-enum-1");
    const hap_model &mo = p->model;
    const int64_t head[] = {mo.N, mo.S, mo.E, mo.GB, mo.nq, mo.nkv, p->T, p->W, p->prof.R, p->dc.tau_linear, p->opts.tp_max,
                            p->opts.n_rc, (int64_t)p->opts.map_cap, (int64_t)(p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT | HAP_OPT_NO_MAPTAB))};
    key_put(k, head);
    for (int h = 0; h < p->T; ++h) key_put(k, p->m[h]);
    auto put_list = [&](const std::vector<int> &v) { const int64_t n = (int64_t)v.size(); key_put(k, n); for (int x : v) key_put(k, x); };
    put_list(p->pp_list); put_list(p->tp_list); put_list(p->cp_list); put_list(p->ep_list); put_list(p->tpe_list); put_list(p->mb_list);
    return k;
}

static std::shared_ptr<const EnumResult> enum_cache_find(const std::string &key)
{
    EnumCache &ec = enum_cache();
    std::lock_guard<std::mutex> lock(ec.mu);
    auto it = ec.map.find(key);
    return it == ec.map.end() ? nullptr : it->second;
}

static void enum_cache_insert(const std::string &key, std::shared_ptr<const EnumResult> r)
{
    EnumCache &ec = enum_cache();
    std::lock_guard<std::mutex> lock(ec.mu);
    if (ec.map.size() >= kEnumCacheEntries) ec.map.clear();
    ec.map[key] = std::move(r);
}

// Configuration table and trees on the problem's device: from the process's images when one of the same key exists, else
// laid out and copied now (once per cluster, model dimensions and search options).
static hap_status image_for(hap_problem *p, const std::string &ekey, bool allow_trees)
{
    // the tree kernel holds times as doubles: exact while every prefix row stays below 2^52, which the per-layer limit of
    // 2^36 ns guarantees when N (2 + max tau) <= 2^16; rows that are not combined by level also form tau x forward time
    int tau_max = 0;
    for (int r = 0; r < p->prof.R; ++r) tau_max = std::max(tau_max, p->tau_q[r]);
    const int64_t N = p->model.N;
    const bool exact = N * (2 + (tau_max >> 10)) <= 65536 && (p->dc.tau_linear || N * tau_max < (1 << 17));
    // and the split pointer of the scan needs levels that repeat no less forward work the higher they are
    bool ordered = true;
    for (uint32_t mk : p->rc_masks) {
        int last = -1;
        for (int r = 0; r < p->prof.R; ++r)
            if ((mk >> r) & 1u) { ordered = ordered && p->tau_q[r] >= last; last = p->tau_q[r]; }
    }
    const bool want_tree = allow_trees && !(p->opts.flags & (HAP_OPT_NO_TRIE | HAP_OPT_NO_MAPTAB)) && exact && ordered;
    std::string key = ekey;
    const int32_t head[] = {p->device, want_tree, p->prof.R, p->opts.delta_q, (int32_t)(p->opts.flags & HAP_OPT_UNIFORM), p->dc.kind_uniform_from,
                            p->dc.tau_linear};
    key_put(key, head);
    for (int h = 0; h < p->T; ++h) { key_put(key, p->P[h]); key_put(key, p->cap_eff[h]); key_put(key, p->dc.node_size[h]); }
    ImageCache &ic = image_cache();
    {
        std::lock_guard<std::mutex> lock(ic.mu);
        auto it = ic.map.find(key);
        if (it != ic.map.end()) { p->image = it->second; return HAP_OK; }
    }
    auto im = std::make_shared<DeviceImage>();
    im->device = p->device;
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    std::vector<std::shared_ptr<const TreeClassHost>> trees;
    size_t o = up(p->pconfs.size() * sizeof(hap_pconf));
    for (const auto &cl : p->classes) {
        std::shared_ptr<const TreeClassHost> th = tree_of_class(p, cl, want_tree);
        im->masks_used.push_back(th->masks_used);
        im->tree_of.push_back(th->ok ? (int)trees.size() : -1);
        if (!th->ok) continue;
        TreeClass c = th->cls;
        c.p_lo = p->items[cl.item_lo].p;
        c.rec_off = im->rec_total;
        im->rec_total += up((size_t)c.n_conf * c.rec_bytes);
        im->prep_smem = std::max(im->prep_smem, tree_prep_smem_bytes(c, p->model.N, p->T));
        im->cls.push_back(c);
        trees.push_back(th);
    }
    tree_policy_items(im->cls, trees, sm_count(p->device), p->opts.n_rc);
    const size_t o_cls = o;
    o = up(o + trees.size() * sizeof(TreeClass));
    std::vector<size_t> o_parts;
    for (const auto &th : trees) {
        o_parts.push_back(o);
        o = up(o + th->parts.size() * sizeof(TreePart));
        for (const auto &pt : th->parts) o = up(up(up(o + pt.tasks.size() * sizeof(TreeTask)) + pt.path.size() * 4) + pt.leaf.size() * 4);
    }
    CUDA_TRY(p, cached_malloc(p->device, (void **)&im->base, o));
    std::vector<unsigned char> stage(o, 0);
    std::memcpy(stage.data(), p->pconfs.data(), p->pconfs.size() * sizeof(hap_pconf));
    for (size_t t = 0; t < trees.size(); ++t) {
        size_t at = up(o_parts[t] + trees[t]->parts.size() * sizeof(TreePart));
        TreePart *parts = reinterpret_cast<TreePart *>(stage.data() + o_parts[t]);
        for (size_t q = 0; q < trees[t]->parts.size(); ++q) {
            const TreePartHost &ph = trees[t]->parts[q];
            parts[q] = ph.meta;
            parts[q].tasks = reinterpret_cast<const TreeTask *>(im->base + at);
            if (!ph.tasks.empty()) std::memcpy(stage.data() + at, ph.tasks.data(), ph.tasks.size() * sizeof(TreeTask));
            at = up(at + ph.tasks.size() * sizeof(TreeTask));
            parts[q].path = reinterpret_cast<const u32 *>(im->base + at);
            std::memcpy(stage.data() + at, ph.path.data(), ph.path.size() * 4);
            at = up(at + ph.path.size() * 4);
            parts[q].leaf = reinterpret_cast<const u32 *>(im->base + at);
            std::memcpy(stage.data() + at, ph.leaf.data(), ph.leaf.size() * 4);
            at = up(at + ph.leaf.size() * 4);
        }
        im->cls[t].parts = reinterpret_cast<const TreePart *>(im->base + o_parts[t]);
    }
    if (!im->cls.empty()) std::memcpy(stage.data() + o_cls, im->cls.data(), im->cls.size() * sizeof(TreeClass));
    CUDA_TRY(p, cudaMemcpy(im->base, stage.data(), o, cudaMemcpyHostToDevice));
    im->d_pconf = reinterpret_cast<hap_pconf *>(im->base);
    im->d_cls = reinterpret_cast<TreeClass *>(im->base + o_cls);
    p->image = im;
    std::lock_guard<std::mutex> lock(ic.mu);
    if (ic.map.size() >= kImages) ic.map.clear();
    ic.map[key] = im;
    return HAP_OK;
}

extern "C" hap_status hap_enumerate(hap_problem *p, uint64_t *n_pconf, uint64_t *n_candidates)
{
    if (!p) return HAP_E_INVALID;
    if (cudaSetDevice(p->device) != cudaSuccess) return fail(p, HAP_E_CUDA, "cudaSetDevice");
    if (!p->enumerated) {
        const hap_model &mo = p->model;
        const int N = mo.N, T = p->T;
        // The configuration table, the work items and the PP classes are a function of the model's dimensions, the
        // cluster inventory and the search options -- not of the profiled tables: they are kept per process, so that
        // planning again for the same cluster and lists copies them instead of running the loop nest.
        const std::string ekey = enum_cache_key(p);
        std::shared_ptr<const EnumResult> er = enum_cache_find(ekey);
        if (!er) {
            auto fresh = std::make_shared<EnumResult>();
            hap_status es = [&]() -> hap_status {
        std::vector<hap_pconf> rows;
            rows.reserve(p->pp_list.size() * p->tp_list.size() * p->cp_list.size() * p->ep_list.size() * p->tpe_list.size() * p->mb_list.size() / 4 + 16);
            uint64_t off = 0;
            const uint64_t SAT = 1ull << 62;
            for (int PP : p->pp_list) {
                if (PP > N || PP > HAP_MAX_PP || p->W % PP) continue;
                const int64_t G = p->W / PP;
                if (G > 0x7fffffffll) continue;
                bool homog = true;
                int cnt[HAP_MAX_TYPES] = {0, 0, 0, 0};
                for (int h = 0; h < T; ++h) { if (p->m[h] % G) homog = false; cnt[h] = (int)(p->m[h] / G); }
                const uint64_t nms = homog ? sequences_sat(cnt, T, SAT) : 0;
                const int mode = (homog && nms <= p->opts.map_cap) ? HAP_MAP_MULTISET : HAP_MAP_BLOCK;
                uint64_t nmap = nms;
                if (mode == HAP_MAP_BLOCK) { nmap = 1; for (int i = 2; i <= T; ++i) nmap *= (uint64_t)i; }
                for (int itp = 0; itp < (int)p->tp_list.size(); ++itp) {
                    const int TP = p->tp_list[itp];
                    if (G % TP || TP > p->opts.tp_max || mo.nq % TP || mo.nkv % TP) continue;
                    for (int icp = 0; icp < (int)p->cp_list.size(); ++icp) {
                        const int CP = p->cp_list[icp];
                        if (G % ((int64_t)TP * CP) || mo.S % (2 * CP)) continue;
                        const int64_t DP = G / ((int64_t)TP * CP);
                        for (int iep = 0; iep < (int)p->ep_list.size(); ++iep) {
                            const int EP = p->ep_list[iep];
                            if (mo.E % EP || G % EP) continue;
                            for (int TPE : p->tpe_list) {
                                if (G % ((int64_t)EP * TPE) || TPE > p->opts.tp_max) continue;
                                const int64_t EDP = G / ((int64_t)EP * TPE);
                                for (int ib = 0; ib < (int)p->mb_list.size(); ++ib) {
                                    const int b = p->mb_list[ib];
                                    if (mo.GB % (DP * b)) continue;
                                    hap_pconf q{};
                                    q.PP = PP; q.TP = TP; q.CP = CP; q.DP = (int)DP; q.EP = EP; q.TPE = TPE; q.b = b;
                                    q.M = (int)(mo.GB / (DP * b)); q.EDP = (int)EDP; q.G = (int)G;
                                    q.itp = itp; q.icp = icp; q.ib = ib; q.iep = iep; q.mode = mode; q.reserved = 0;
                                    q.nmap = nmap; q.offset = off;
                                    if (nmap > (SAT - off) / (uint64_t)p->opts.n_rc) return fail(p, HAP_E_RANGE, "candidate space overflows 2^62");
                                    off += nmap * (uint64_t)p->opts.n_rc;
                                    rows.push_back(q);
                                }
                            }
                        }
                    }
                }
            }
            if (rows.empty()) return fail(p, HAP_E_INFEASIBLE, "no parallel configuration divides the cluster");
            if (rows.size() > 0xffffffffull) return fail(p, HAP_E_RANGE, "too many configurations");

            // PP classes (heaviest first).  Each class is one launch with its own block shape; a class keeps a
            // table of its decoded mappings when that table is small.
            std::vector<int> pps;
            for (const auto &r : rows) if (std::find(pps.begin(), pps.end(), r.PP) == pps.end()) pps.push_back(r.PP);
            std::sort(pps.begin(), pps.end(), [](int a, int b) { return a > b; });
            std::vector<WorkItem> items;
            items.reserve(rows.size() * 2);
            std::vector<hap_problem::PpClass> classes;
            u64 tab_bytes = 0;
            for (int PP : pps) {
                hap_problem::PpClass cl{};
                cl.PP = PP;
                cl.masks_used = 0xffffffffu;
                cl.stream = nullptr; cl.done = nullptr;
                cl.warps = 0;
                // the rows of a PP value are contiguous (PP is the outermost loop of the enumeration)
                size_t row_lo = 0;
                while (row_lo < rows.size() && rows[row_lo].PP != PP) ++row_lo;
                size_t row_hi = row_lo;
                while (row_hi < rows.size() && rows[row_hi].PP == PP) ++row_hi;
                cl.multiset = rows[row_lo].mode == HAP_MAP_MULTISET;
                // most warps per SM: try block shapes from large to small, keep the one with the most resident warps
                int best_resident = 0;
                const uint64_t class_nmap = rows[row_lo].nmap;
                const uint64_t per_pconf = class_nmap * (uint64_t)p->opts.n_rc;     // candidates a block can have at most
                for (int w : {12, 8, 6, 4, 2, 1}) {
                    if ((uint64_t)w * 8 > per_pconf && w > 2) continue;             // keep about 8 candidates per warp
                    const size_t sm = dp_smem_bytes(N, PP, T, p->prof.R, w, cl.multiset, p->dc.tau_linear != 0,
                                                    (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) != 0);
                    if (sm > 227 * 1024) continue;
                    const int per_sm = std::min<int>((int)((227 * 1024) / (sm + 1024)), std::min(32, 64 / w));
                    const int resident = std::min(per_sm * w, 24);           // registers allow about 24 warps per SM
                    if (resident > best_resident) { best_resident = resident; cl.warps = w; cl.smem = sm; }
                }
                if (!cl.warps) return fail(p, HAP_E_RANGE, "shared memory need of a PP=%d block exceeds the SM", PP);
                // a warp takes a slice of at most 64 consecutive mappings (one bit each in its infeasibility masks)
                const uint64_t chunk_cap = 32ull * cl.warps;
                cl.item_lo = items.size();
                uint64_t nmap = 0;
                for (size_t pi = row_lo; pi < row_hi; ++pi) {
                    nmap = rows[pi].nmap;
                    const uint64_t n_chunks = (nmap + chunk_cap - 1) / chunk_cap;
                    const uint64_t chunk = (nmap + n_chunks - 1) / n_chunks;          // balanced chunks
                    for (uint64_t lo = 0; lo < nmap; lo += chunk) {
                        WorkItem it; it.p = (uint32_t)pi; it.lo = lo; it.count = (uint32_t)std::min<uint64_t>(chunk, nmap - lo);
                        items.push_back(it);
                    }
                }
                cl.item_hi = items.size();
                cl.has_tab = !(p->opts.flags & HAP_OPT_NO_MAPTAB) && nmap * (uint64_t)PP * 2 <= (64ull << 20) &&
                             tab_bytes + nmap * PP * 2 <= (256ull << 20);
                cl.map_base = tab_bytes;
                if (cl.has_tab) tab_bytes += (nmap * (uint64_t)PP * 2 + 255) / 256 * 256;
                classes.push_back(cl);
            }
            if (items.size() > 0x7fffffffull) return fail(p, HAP_E_RANGE, "too many work items");

            fresh->rows.swap(rows); fresh->items.swap(items); fresh->classes.swap(classes);
            fresh->n_cand = off; fresh->tab_bytes = tab_bytes;
            return HAP_OK;
            }();
            if (es != HAP_OK) return es;
            enum_cache_insert(ekey, fresh);
            er = fresh;
        }
        p->enum_ref = er;
        p->pconfs.ptr = er->rows.data(); p->pconfs.n = er->rows.size();
        p->items.ptr = er->items.data(); p->items.n = er->items.size();
        p->classes = er->classes;
        p->tab_bytes = er->tab_bytes;
        p->n_cand = er->n_cand;
        const size_t np = p->pconfs.size();
        // (a device without room for the records of the trees runs one warp per candidate)
        for (bool trees : {true, false}) {
        const hap_status is = image_for(p, ekey, trees);
        if (is != HAP_OK) return is;
        const DeviceImage &im = *p->image;
        p->all_trees = true;
        for (size_t ci = 0; ci < p->classes.size(); ++ci) {
            p->classes[ci].tree = im.tree_of[ci];
            p->classes[ci].masks_used = im.masks_used[ci];
            p->all_trees = p->all_trees && im.tree_of[ci] >= 0;
        }
        // one allocation for everything a pass needs (an allocation costs far more than the microseconds a pass takes):
        // coefficients | per-type constants | lower bounds | partial minima | plans | records | small scalars; partial
        // minima: one slot per block of the tree kernel, then one per block of the general one
        p->n_partial = std::max<size_t>(1024, kTreeSlots + p->items.size());
        {
            auto up = [](size_t v) { return (v + 255) / 256 * 256; };
            size_t o = 0;
            const bool refining = (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) != 0 && !im.cls.empty(), ordering = p->opts.prune || refining;
            const size_t o_coef = o; o = up(o + np * T * HAP_NCOEF * sizeof(i64));
            const size_t o_tc = o; o = up(o + np * T * sizeof(TypeConst));
            const size_t o_lb = o; o = up(o + np * sizeof(i64));
            const size_t o_pcost = o; o = up(o + p->n_partial * sizeof(i64));
            const size_t o_pindex = o; o = up(o + p->n_partial * sizeof(u64));
            const size_t o_plans = o; o = up(o + (im.cls.empty() ? 0 : kTreeSlots) * sizeof(PlanSlot));
            const size_t o_rec = o; o = up(o + im.rec_total);
            const size_t o_counters = o; o = up(o + 8 * sizeof(u64));
            const size_t o_best = o; o = up(o + 2 * sizeof(i64));
            const size_t o_single = o; o = up(o + sizeof(SingleOut));
            const size_t o_report = o; o = up(o + sizeof(TreeReport));
            const size_t o_live = o; o = up(o + np * sizeof(u32));
            const size_t o_dead = o; o = up(o + np * sizeof(u32));
            const u64 n_surv = std::min<u64>(kMaxSurvivors, p->n_cand);
            const size_t o_hist = o; o = up(o + (ordering ? kOrderBuckets * sizeof(u64) : 0));
            const size_t o_key = o; o = up(o + (ordering ? np * sizeof(uint4) : 0));
            const size_t o_order = o; o = up(o + (ordering ? (np + 1) * sizeof(uint4) : 0));
            const size_t o_surv = o; o = up(o + (refining ? n_surv * sizeof(Survivor) : 0));
            const size_t o_res = o; o = up(o + sizeof(TreeResult));
            const cudaError_t e = cached_malloc(p->device, (void **)&p->d_arena, o);
            if (e == cudaErrorMemoryAllocation && trees && im.rec_total) { cudaGetLastError(); continue; }
            CUDA_TRY(p, e);
            unsigned char *base = p->d_arena;
            p->d_coef = reinterpret_cast<i64 *>(base + o_coef);
            p->d_tc = reinterpret_cast<TypeConst *>(base + o_tc); p->d_lb = reinterpret_cast<i64 *>(base + o_lb);
            p->d_pcost = reinterpret_cast<i64 *>(base + o_pcost); p->d_pindex = reinterpret_cast<u64 *>(base + o_pindex);
            p->d_plans = reinterpret_cast<PlanSlot *>(base + o_plans);
            p->d_counters = reinterpret_cast<u64 *>(base + o_counters);
            p->d_best = reinterpret_cast<i64 *>(base + o_best); p->d_single = base + o_single;
            TreeArgs &ta = p->targs;
            ta.rec = base + o_rec;
            ta.state = reinterpret_cast<TreeState *>(reinterpret_cast<unsigned char *>(p->d_range) + 16);
            ta.report = reinterpret_cast<TreeReport *>(base + o_report);
            ta.live_list = reinterpret_cast<const u32 *>(base + o_live); ta.dead_list = reinterpret_cast<const u32 *>(base + o_dead);
            ta.hist = reinterpret_cast<u64 *>(base + o_hist);
            ta.order_key = reinterpret_cast<uint4 *>(base + o_key); ta.order = reinterpret_cast<uint4 *>(base + o_order);
            ta.surv = reinterpret_cast<Survivor *>(base + o_surv); ta.max_surv = n_surv;
            LiveArgs &la = p->largs;
            la.hist = ta.hist; la.n_hist = 0;
            la.state = ta.state; la.report = ta.report;
            la.live_list = reinterpret_cast<u32 *>(base + o_live); la.dead_list = reinterpret_cast<u32 *>(base + o_dead);
            la.n_cls = ta.n_cls = (int)im.cls.size();
            for (size_t c = 0; c < im.cls.size(); ++c) {
                la.p_lo[c] = ta.p_lo[c] = im.cls[c].p_lo; la.p_hi[c] = im.cls[c].p_lo + im.cls[c].n_conf;
                ta.nmap[c] = (u32)p->pconfs[im.cls[c].p_lo].nmap;
                la.first_min[c] = 0;
                for (int h = 0; h < HAP_MAX_TYPES; ++h) la.first_min[c] |= (u32)im.cls[c].first_min[h] << (8 * h);
            }
            ta.res_dev = reinterpret_cast<TreeResult *>(base + o_res);
            ta.N = N; ta.T = T; ta.R = p->prof.R; ta.n_rc = p->opts.n_rc; ta.RW = p->dc.tau_linear ? p->prof.R : 2;
            ta.eta_q = p->dc.eta_q;
            for (int i = 0; i < p->opts.n_rc; ++i) { ta.rc_masks[i] = p->dc.rc_masks[i]; ta.rc_sup[i] = p->dc.rc_sup[i]; ta.rc_order[i] = p->dc.rc_order[i]; }
            for (int r = 0; r < p->prof.R; ++r) ta.tau[r] = p->tau_q[r] / 1024.0;
            ta.cls = im.d_cls;
            ta.range_flag = p->d_range;
            ta.slots = p->d_plans; ta.slot_cost = p->d_pcost; ta.slot_index = p->d_pindex;
        }
        p->dc.pconf = im.d_pconf;
        p->dc.n_pconf = np;
        p->enumerated = true;
        break;
        }
    }
    if (n_pconf) *n_pconf = p->pconfs.size();
    if (n_candidates) *n_candidates = p->n_cand;
    return HAP_OK;
}

extern "C" hap_status hap_get_pconfs(const hap_problem *p, hap_pconf *host_out, uint64_t cap)
{
    if (!p || !host_out) return HAP_E_INVALID;
    if (!p->enumerated) return HAP_E_STATE;
    if (cap < p->pconfs.size()) return HAP_E_RANGE;
    std::memcpy(host_out, p->pconfs.data(), p->pconfs.size() * sizeof(hap_pconf));
    return HAP_OK;
}

// Calls that could be unsafe while some stream of the process is captured are allowed to a thread in this mode.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

static bool is_default(cudaStream_t st) { return st == nullptr || st == cudaStreamLegacy; }

// what a stream is told apart by (not its handle, which is used again); not for a stream that is being captured
static cudaError_t stream_id(cudaStream_t st, unsigned long long *id)
{
    if (is_default(st)) { *id = ~0ull; return cudaSuccess; }
    RelaxedCapture relaxed;
    return cudaStreamGetId(st, id);
}

// Every call that launches work starts here.  Its stream waits for the upload of the tables and, where the last call went to
// another stream, for that one's work, because a problem's passes share its scratch memory; the host waits for neither.
// While the stream is being captured it cannot wait for an event from outside of the capture: then the host does.
static hap_status enter(hap_problem *p, cudaStream_t st)
{
    if (!p) return HAP_E_INVALID;
    if (!p->enumerated) return fail(p, HAP_E_STATE, "hap_enumerate has not run");
    if (cudaSetDevice(p->device) != cudaSuccess) return fail(p, HAP_E_CUDA, "cudaSetDevice");
    if (!p->upload_pending && !p->in_flight) return HAP_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!is_default(st)) CUDA_TRY(p, cudaStreamIsCapturing(st, &cap));
    if (cap != cudaStreamCaptureStatusNone) {
        RelaxedCapture relaxed;
        if (p->upload_pending) { CUDA_TRY(p, cudaEventSynchronize(p->ev_upload)); p->upload_pending = false; }
        // (a call on the default stream has no event yet, and none may be recorded on it now: the caller orders the graph behind it)
        if (p->in_flight && !p->last_default) { CUDA_TRY(p, cudaEventSynchronize(p->ev_order)); p->in_flight = false; }
        return HAP_OK;
    }
    unsigned long long id = 0;
    CUDA_TRY(p, stream_id(st, &id));
    if (p->upload_pending && !(p->upload_waited && id == p->upload_id)) {
        CUDA_TRY(p, cudaStreamWaitEvent(st, p->ev_upload, 0));
        p->upload_waited = true; p->upload_id = id;
    }
    if (p->in_flight && id != p->last_id) {
        if (p->last_default) {
            if (!p->ev_order && !(p->ev_order = pooled_event(p->device))) return fail(p, HAP_E_CUDA, "cudaEventCreate");
            CUDA_TRY(p, cudaEventRecord(p->ev_order, cudaStreamLegacy));
        }
        CUDA_TRY(p, cudaStreamWaitEvent(st, p->ev_order, 0));
    }
    return HAP_OK;
}

// ... and ends here: the work it queued on `st` is in flight.  An event behind it is what a later call on another stream waits
// for; the default stream, which outlives every call, gets one only then (an event a call costs its stream 1 us: 36.6 instead
// of 35.5 us for an evaluation of two calls).  A captured call runs when its graph does: the caller orders that.
static hap_status leave_async(hap_problem *p, cudaStream_t st)
{
    if (!is_default(st)) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        CUDA_TRY(p, cudaStreamIsCapturing(st, &cap));
        if (cap != cudaStreamCaptureStatusNone) { p->captured = true; return HAP_OK; }
        if (!p->ev_order && !(p->ev_order = pooled_event(p->device))) return fail(p, HAP_E_CUDA, "cudaEventCreate");
        CUDA_TRY(p, cudaEventRecord(p->ev_order, st));
    }
    CUDA_TRY(p, stream_id(st, &p->last_id));
    p->in_flight = true;
    p->last_default = is_default(st);
    return HAP_OK;
}

// the host waits for the last asynchronous call
static hap_status wait_last(hap_problem *p)
{
    if (p->in_flight) CUDA_TRY(p, p->last_default ? cudaStreamSynchronize(cudaStreamLegacy) : cudaEventSynchronize(p->ev_order));
    p->in_flight = false;
    if (p->captured) CUDA_TRY(p, cudaDeviceSynchronize());
    return HAP_OK;
}

// ... or here, with everything it queued done
static hap_status leave_synced(hap_problem *p, cudaStream_t st)
{
    CUDA_TRY(p, cudaStreamSynchronize(st));
    p->in_flight = false;
    p->upload_pending = false;
    return HAP_OK;
}

static hap_status check_values(hap_problem *p)
{
    u64 flag = 0;
    CUDA_TRY(p, cudaMemcpy(&flag, p->d_range, sizeof(flag), cudaMemcpyDeviceToHost));
    if (flag) return fail(p, HAP_E_RANGE, "a layer time or stage coefficient exceeds the supported range (see hap.h)");
    return HAP_OK;
}

static hap_status check_range(hap_problem *p, uint64_t first, uint64_t count)
{
    if (first > p->n_cand || count > p->n_cand - first) return fail(p, HAP_E_RANGE, "candidate range outside [0, %llu)", (unsigned long long)p->n_cand);
    return HAP_OK;
}

extern "C" hap_status hap_decode(hap_problem *p, uint64_t first, uint64_t count, hap_candidate *dev_out, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return HAP_OK;
    if (!dev_out) return HAP_E_INVALID;
    const uint64_t blocks = (count + 3) / 4;
    if (blocks > 0x7fffffffull) return fail(p, HAP_E_RANGE, "count too large for one launch");
    decode_kernel<<<(unsigned)blocks, 128, 0, (cudaStream_t)stream>>>(p->dc, first, count, dev_out, nullptr);
    CUDA_TRY(p, cudaGetLastError());
    return leave_async(p, (cudaStream_t)stream);
}


// work items, layer-cost array and mapping table of the general kernel, with its streams and events (first use)
static hap_status ensure_general(hap_problem *p)
{
    if (p->gen_ready) return HAP_OK;
    const size_t np = p->pconfs.size();
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    size_t o = 0;
    const size_t o_items = o; o = up(o + p->items.size() * sizeof(WorkItem));
    const size_t o_c2 = o; o = up(o + np * p->T * p->model.N * 2 * sizeof(i64));
    const size_t o_maptab = o; o = up(o + p->tab_bytes);
    CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_gen_arena, o));
    p->d_items = reinterpret_cast<WorkItem *>(p->d_gen_arena + o_items);
    p->d_c2 = reinterpret_cast<i64 *>(p->d_gen_arena + o_c2);
    p->d_maptab = p->tab_bytes ? p->d_gen_arena + o_maptab : nullptr;
    CUDA_TRY(p, cudaMemcpy(p->d_items, p->items.data(), p->items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice));
    if (!(p->ev_fork = pooled_event(p->device))) return fail(p, HAP_E_CUDA, "cudaEventCreate");
    for (auto &e : p->ev) CUDA_TRY(p, cudaEventCreate(&e));
    for (size_t ci = 0; ci < p->classes.size(); ++ci) {
        auto &cl = p->classes[ci];
        if (!(cl.stream = pooled_stream(p->device, ci))) return fail(p, HAP_E_CUDA, "cudaStreamCreateWithFlags");
        if (!(cl.done = pooled_event(p->device))) return fail(p, HAP_E_CUDA, "cudaEventCreate");
    }
    p->gen_ready = true;
    return HAP_OK;
}

// per (configuration, type) constants and stage coefficients, then the layer costs of `n_conf` configurations from
// `p_first` on (all by default)
static hap_status launch_layer_kernel(hap_problem *p, i64 *c2, double *c2f, bool quant, cudaStream_t st, i64 *lb_sum,
                                      unsigned p_first, unsigned n_conf, bool dependent)
{
    const unsigned thr = (unsigned)((p->model.N + 31) / 32 * 32);
    // programmatic dependent launch: the blocks start while type_const_kernel drains and wait inside the kernel
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_conf); cfg.blockDim = dim3(thr); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dependent ? 1 : 0;
    const TypeConst *tcg = p->d_tc;
    i64 *no_i = nullptr; double *no_d = nullptr;
    // layer kinds: 0 all dense, 1 all MoE (uniform branch compiled away), 2 mixed
    const int kind = p->dc.kind_uniform_from > 0 ? 2 : (p->kind[0] == HAP_MOE ? 1 : 0);
    using Fn = void (*)(const DevConst, const TypeConst *, i64 *, double *, i64 *, u64 *, unsigned);
    if (quant) {
        static const Fn fns[3][2] = {{layer_cost_kernel<true, 0, false>, layer_cost_kernel<true, 0, true>},
                                     {layer_cost_kernel<true, 1, false>, layer_cost_kernel<true, 1, true>},
                                     {layer_cost_kernel<true, 2, false>, layer_cost_kernel<true, 2, true>}};
        CUDA_TRY(p, cudaLaunchKernelEx(&cfg, fns[kind][lb_sum ? 1 : 0], p->dc, tcg, c2, no_d, lb_sum, p->d_range, p_first));
    } else {
        static const Fn fns[3] = {layer_cost_kernel<false, 0, false>, layer_cost_kernel<false, 1, false>, layer_cost_kernel<false, 2, false>};
        CUDA_TRY(p, cudaLaunchKernelEx(&cfg, fns[kind], p->dc, tcg, no_i, c2f, no_i, p->d_range, p_first));
    }
    return HAP_OK;
}

// configurations that own candidates of [first, first + count): a contiguous range [lo, hi)
static void configs_of_range(const hap_problem *p, u64 first, u64 count, unsigned &lo, unsigned &hi)
{
    auto owner = [&](u64 c) {
        size_t a = 0, b = p->pconfs.size();
        while (b - a > 1) { const size_t mid = (a + b) / 2; if (p->pconfs[mid].offset <= c) a = mid; else b = mid; }
        return (unsigned)a;
    };
    if (count == 0 || p->pconfs.empty()) { lo = hi = 0; return; }
    lo = owner(first); hi = owner(first + count - 1) + 1;
}

// Per-type constants and stage coefficients of the configurations [p_lo, p_hi) in integer (coef) and / or fp64 form (coeff);
// `live`: also the classes' lists of configurations (a pass over the trees)
static hap_status launch_type_consts(hap_problem *p, i64 *coef, double *coeff, cudaStream_t st, unsigned p_lo, unsigned p_hi, const LiveArgs *live = nullptr)
{
    const unsigned n_conf = p_hi - p_lo;
    if (live) {
        const unsigned per = 32 / (unsigned)p->T;             // configurations of a block
        type_const_kernel<<<(n_conf + per - 1) / per, kTcThreads, 0, st>>>(p->dc, p->d_tc, coef, coeff, p->d_range, p_lo, n_conf, *live);
    } else {
        const unsigned blocks = (unsigned)(((u64)n_conf * HAP_MAX_TYPES + kTcPlainThreads - 1) / kTcPlainThreads);
        if (coeff) type_const_plain_kernel<false><<<dim3(blocks, 3), kTcPlainThreads, 0, st>>>(p->dc, p->d_tc, coef, coeff, p->d_range, p_lo, n_conf);
        else type_const_plain_kernel<true><<<dim3(blocks, 3), kTcPlainThreads, 0, st>>>(p->dc, p->d_tc, coef, nullptr, p->d_range, p_lo, n_conf);
    }
    CUDA_TRY(p, cudaGetLastError());
    return HAP_OK;
}

// ... and then (where an output array is given) the layer costs: a pass over a candidate range touches only the
// configurations that own its candidates.
static hap_status launch_layer_costs(hap_problem *p, i64 *c2, i64 *coef, double *c2f, double *coeff, bool quant, cudaStream_t st,
                                     i64 *lb_sum = nullptr, unsigned p_lo = 0, unsigned p_hi = ~0u)
{
    if (p_hi > p->pconfs.size()) p_hi = (unsigned)p->pconfs.size();
    if (p_lo >= p_hi) return HAP_OK;
    if (!(quant ? c2 != nullptr : c2f != nullptr)) return launch_type_consts(p, quant ? coef : nullptr, quant ? nullptr : coeff, st, p_lo, p_hi);
    const unsigned n_conf = p_hi - p_lo, per = 32 / (unsigned)p->T;
    // one launch up to three blocks an SM, all of them running at once: the chain of constants is then followed by the writes
    // without a second launch (12.3 -> 10.2 us at 2,392 configurations of three types); beyond, the constants of later blocks
    // delay the writes (1,024 devices, 7,783 configurations: 20.5 us in two launches, 26.8 us in one)
    if ((n_conf + per - 1) / per > 3 * (unsigned)sm_count(p->device)) {
        hap_status s = launch_type_consts(p, quant ? coef : nullptr, quant ? nullptr : coeff, st, p_lo, p_hi);
        if (s != HAP_OK) return s;
        return launch_layer_kernel(p, c2, c2f, quant, st, lb_sum, p_lo, n_conf, true);
    }
    const int kind = p->dc.kind_uniform_from > 0 ? 2 : (p->kind[0] == HAP_MOE ? 1 : 0);      // layer kinds: all dense, all MoE, mixed
    using Fn = void (*)(const DevConst, i64 *, double *, i64 *, double *, i64 *, u64 *, unsigned, unsigned);
    static const Fn fns[3][3] = {{cost_kernel<false, 0, false>, cost_kernel<true, 0, false>, cost_kernel<true, 0, true>},
                                 {cost_kernel<false, 1, false>, cost_kernel<true, 1, false>, cost_kernel<true, 1, true>},
                                 {cost_kernel<false, 2, false>, cost_kernel<true, 2, false>, cost_kernel<true, 2, true>}};
    fns[kind][!quant ? 0 : lb_sum ? 2 : 1]<<<(n_conf + per - 1) / per, kCostThreads, 0, st>>>(
        p->dc, c2, c2f, quant ? coef : nullptr, quant ? nullptr : coeff, lb_sum, p->d_range, p_lo, n_conf);
    CUDA_TRY(p, cudaGetLastError());
    return HAP_OK;
}

extern "C" hap_status hap_eval_layer_costs(hap_problem *p, int64_t *dev_c2, int64_t *dev_coef, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if (!dev_c2 && !dev_coef) return HAP_OK;
    if ((s = launch_layer_costs(p, (i64 *)dev_c2, (i64 *)dev_coef, nullptr, nullptr, true, (cudaStream_t)stream)) != HAP_OK) return s;
    return leave_async(p, (cudaStream_t)stream);
}

extern "C" hap_status hap_eval_layer_costs_f64(hap_problem *p, double *dev_c2, double *dev_coef, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if (!dev_c2 && !dev_coef) return HAP_OK;
    if ((s = launch_layer_costs(p, nullptr, nullptr, dev_c2, dev_coef, false, (cudaStream_t)stream)) != HAP_OK) return s;
    return leave_async(p, (cudaStream_t)stream);
}

// whether all candidates of the class lie outside the range the pass writes
static bool class_outside(const hap_problem *p, const hap_problem::PpClass &cl, const DpOut &out)
{
    const WorkItem &a = p->items[cl.item_lo], &b = p->items[cl.item_hi - 1];
    const u64 c0 = p->pconfs[a.p].offset, c1 = p->pconfs[b.p].offset + p->pconfs[b.p].nmap * (u64)p->opts.n_rc;
    return c1 <= out.first || c0 >= out.first + out.count;
}

// Plain passes walk the prefix trees of the classes that have one; tables, refinement, cell counting and the
// one-candidate re-evaluation stay in pipeline_dp_kernel.  (The tree kernel writes partitions in 16-byte pieces.)
static bool pass_uses_trees(const hap_problem *p, const DpOut &out)
{
    const bool refine = (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) != 0 && !out.force_plain;
    const bool aligned = ((reinterpret_cast<uintptr_t>(out.partition) | reinterpret_cast<uintptr_t>(out.recompute)) & 15) == 0;
    return !p->image->cls.empty() && !out.count_only && !refine && !out.dp_table && !out.choice && !out.detail && !out.first_dev && aligned;
}

// The dynamic shared memory limit is a per-kernel, per-device attribute shared by every problem of the process: raised
// (never lowered) before a launch that needs more.
static cudaError_t raise_smem_limit(int device, const void *fn, size_t bytes)
{
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, size_t> limit;
    std::lock_guard<std::mutex> lock(mu);
    size_t &l = limit[{device, fn}];
    if (bytes <= l) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) l = bytes;
    return e;
}


// launch behind the kernel before it in the stream, as its programmatic dependent
static cudaError_t launch_dependent(const void *fn, unsigned grid, unsigned threads, size_t smem, cudaStream_t st, void **args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

// One launch of the tree kernel: classes [c_lo, c_hi) of the image.
struct TreeLaunch { int c_lo, c_hi; size_t smem; unsigned grid; u64 items; int blocks; };

// A pass runs the deep pipelines (long chains of small depths) and the others in launches of their own, deep ones first:
// the blocks of each take the shared memory their own classes need.  From 16 stages on, measured against one launch and a line at
// 8 stages: 1,024 devices, classes of 24 mappings, two policies 244 us (251, 246), 60 layers 247 (275, 261), one policy 206
// (194, 200); a class of 840 mappings 390 (389, 394); 256 devices with partitions 474 (464, 466).  A search is one launch where it
// may prune (its items go in order of their bounds) or where everything starts at once.
static std::vector<TreeLaunch> tree_launches(const hap_problem *p, bool search, bool prune, bool grouped, unsigned p_lo, unsigned p_hi)
{
    const auto &cls = p->image->cls;
    std::vector<TreeLaunch> ls;
    auto group = [&](int c_lo, int c_hi) {
        TreeLaunch l{c_lo, c_hi, 0, 0, 0, kTreeBlocksPerSm};
        for (int c = c_lo; c < c_hi; ++c) {
            const TreeClass &cl = cls[(size_t)c];
            const unsigned a = std::max(p_lo, cl.p_lo), b = std::min(p_hi, cl.p_lo + cl.n_conf);
            if (a >= b) continue;
            l.items += (u64)(grouped ? (b - a + cl.group - 1) / cl.group : b - a) * cl.items_per_conf * (prune ? 1 : cl.policy_items);
            l.smem = std::max(l.smem, tree_smem_bytes(cl, grouped));
        }
        if (!l.items) return;
        if (search && !grouped && p->dc.tau_linear && kTreeLive * (double)l.items > 2.0 * kTreeBlocksPerSm * sm_count(p->device)) l.blocks = kTreeSearchBlocksPerSm;
        const unsigned per_sm = (unsigned)std::max<size_t>(1, std::min<size_t>((size_t)l.blocks, kSmemPerSm / (l.smem + kTreeSmemStatic)));
        l.grid = (unsigned)std::min<u64>(l.items, std::min<u64>((u64)sm_count(p->device) * per_sm, kTreeSlots / 2));
        ls.push_back(l);
    };
    if (search) {
        group(0, (int)cls.size());
        if (prune || ls.empty() || ls[0].items <= ls[0].grid) return ls;
        ls.clear();
    }
    int split = 0;
    while (split < (int)cls.size() && cls[(size_t)split].PP >= 16) ++split;
    if (split > 0) group(0, split);
    if (split < (int)cls.size()) group(split, (int)cls.size());
    return ls;
}

// A pass or a search over the prefix trees: per-type constants, (the layer-cost array where it is asked for,) records,
// recurrence -- each the programmatic dependent of the one before.  Classes without a tree are left to launch_dp; c2 / c2f
// then hold their layer costs.
static hap_status launch_trees(hap_problem *p, const DpOut &out_in, bool search, bool f64, cudaStream_t st, bool final_reduce, bool refine = false)
{
    DpOut out = out_in;
    out.range_flag = p->d_range;
    unsigned p_lo, p_hi;
    configs_of_range(p, out.first, out.count, p_lo, p_hi);
    const bool separate = (p->opts.flags & HAP_OPT_NO_FUSE) != 0;
    hap_status s;
    if (p->state_dirty) CUDA_TRY(p, cudaMemsetAsync(p->targs.state, 0, sizeof(TreeState), st));
    p->state_dirty = true;
    if (refine) out.prune = 1;
    const bool prune = search && !f64 && out.prune;
    const bool counting = (p->opts.flags & HAP_OPT_COUNT_SPLITS) && !f64 && !search;
    const bool grouped = !prune && !counting && tree_grouped(p->image->cls, p_lo, p_hi, sm_count(p->device), search);
    const std::vector<TreeLaunch> ls = tree_launches(p, search, prune, grouped, p_lo, p_hi);
    const bool ordered = prune && ls.size() == 1 && ls[0].items > ls[0].grid;      // (in one wave everything starts at once)
    p->largs.n_hist = ordered ? kOrderBuckets : 0;
    if ((s = launch_type_consts(p, p->d_coef, f64 ? p->d_coeff : nullptr, st, p_lo, p_hi, &p->largs)) != HAP_OK) return s;
    const void *c2v = nullptr;
    if (separate || !p->all_trees) {
        if (f64) { if ((s = launch_layer_kernel(p, nullptr, p->d_c2f, false, st, nullptr, p_lo, p_hi - p_lo, true)) != HAP_OK) return s; }
        else if ((s = launch_layer_kernel(p, p->d_c2, nullptr, true, st, p->d_lb, p_lo, p_hi - p_lo, true)) != HAP_OK) return s;
        if (separate) c2v = f64 ? (const void *)p->d_c2f : (const void *)p->d_c2;
    }
    const bool nl = !p->dc.tau_linear;
    const DeviceImage &im = *p->image;
    TreeArgs ta = p->targs;
    if (!ordered) ta.order = nullptr;
    ta.by_policy = !prune;
    int is_search = search ? 1 : 0;
    TreeInput in{p->d_tc, p->d_coef, p->d_coeff, c2v, {}};
    for (int r = 0; r < p->prof.R; ++r) in.tau[r] = (double)(p->tau_q[r] >> 10);
    {
        const void *fn = f64 ? (nl ? (const void *)tree_prep_kernel<true, true> : (const void *)tree_prep_kernel<true, false>)
                             : (nl ? (const void *)tree_prep_kernel<false, true> : (const void *)tree_prep_kernel<false, false>);
        CUDA_TRY(p, raise_smem_limit(p->device, fn, im.prep_smem));
        void *args[] = {(void *)&p->dc, (void *)&ta, (void *)&in, (void *)&out, (void *)&is_search};
        const unsigned per_sm = (unsigned)std::max<size_t>(1, std::min<size_t>(kTreePrepBlocksPerSm, (227 * 1024) / (im.prep_smem + 2048)));
        CUDA_TRY(p, launch_dependent(fn, std::min<unsigned>(p_hi - p_lo, (unsigned)sm_count(p->device) * per_sm), kTreePrepThreads, im.prep_smem, st, args));
    }
    ta.blocks_total = 0;
    for (const auto &l : ls) ta.blocks_total += l.grid;
    if (!final_reduce) ta.res_dev = nullptr;
    ta.res_host = final_reduce ? p->host_result : nullptr;
    // two row entries are held where there are at most two levels, else they are read by level
    const int form = nl ? 2 : p->prof.R > 2 ? 1 : 0;
    using Fn = void (*)(const TreeArgs, const DevConst, DpOut);
    constexpr int kP = kTreePass, kS = kTreeSearch, kL = kTreeList;
    constexpr int kB = kTreeSearchBlocksPerSm, kG = kTreeBlocksPerSm;
    static const Fn fns[13][3] = {
        {tree_dp_kernel<kP, false, 2, false, false>, tree_dp_kernel<kP, false, 4, false, false>, tree_dp_kernel<kP, false, 4, true, false>},
        {tree_dp_kernel<kS, false, 2, false, false>, tree_dp_kernel<kS, false, 4, false, false>, tree_dp_kernel<kS, false, 4, true, false>},
        {tree_dp_kernel<kP, true, 2, false, false>, tree_dp_kernel<kP, true, 4, false, false>, tree_dp_kernel<kP, true, 4, true, false>},
        {tree_dp_kernel<kS, true, 2, false, false>, tree_dp_kernel<kS, true, 4, false, false>, tree_dp_kernel<kS, true, 4, true, false>},
        {tree_dp_kernel<kP, false, 2, false, true>, tree_dp_kernel<kP, false, 4, false, true>, tree_dp_kernel<kP, false, 4, true, true>},
        {tree_dp_kernel<kL, false, 2, false, false>, tree_dp_kernel<kL, false, 4, false, false>, tree_dp_kernel<kL, false, 4, true, false>},
        // four blocks an SM: search, fp64 search, listing
        {tree_dp_kernel<kS, false, 2, false, false, kB>, tree_dp_kernel<kS, false, 4, false, false, kB>, nullptr},
        {tree_dp_kernel<kS, true, 2, false, false, kB>, tree_dp_kernel<kS, true, 4, false, false, kB>, nullptr},
        {tree_dp_kernel<kL, false, 2, false, false, kB>, tree_dp_kernel<kL, false, 4, false, false, kB>, nullptr},
        // grouped: pass, search, and both in fp64
        {tree_dp_kernel<kP, false, 2, false, false, kG, true>, tree_dp_kernel<kP, false, 4, false, false, kG, true>, tree_dp_kernel<kP, false, 4, true, false, kG, true>},
        {tree_dp_kernel<kS, false, 2, false, false, kG, true>, tree_dp_kernel<kS, false, 4, false, false, kG, true>, tree_dp_kernel<kS, false, 4, true, false, kG, true>},
        {tree_dp_kernel<kP, true, 2, false, false, kG, true>, tree_dp_kernel<kP, true, 4, false, false, kG, true>, tree_dp_kernel<kP, true, 4, true, false, kG, true>},
        {tree_dp_kernel<kS, true, 2, false, false, kG, true>, tree_dp_kernel<kS, true, 4, false, false, kG, true>, tree_dp_kernel<kS, true, 4, true, false, kG, true>}};
    const int mode = refine ? 5 : counting ? 4 : (f64 ? 2 : 0) + (search ? 1 : 0);
    int n = 0;
    for (const auto &l : ls) {
        ta.c_lo = l.c_lo; ta.c_hi = l.c_hi; ta.launch = n;
        ta.slot_lo = n == 0 ? 0 : ls[0].grid;
        const void *fn = (const void *)fns[grouped ? 9 + mode : l.blocks == kTreeBlocksPerSm ? mode : refine ? 8 : f64 ? 7 : 6][form];
        if (!fn) return fail(p, HAP_E_STATE, "no tree kernel of this form");
        CUDA_TRY(p, raise_smem_limit(p->device, fn, l.smem));
        void *args[] = {(void *)&ta, (void *)&p->dc, (void *)&out};
        CUDA_TRY(p, launch_dependent(fn, l.grid, kTreeThreads, l.smem, st, args));
        ++n;
    }
    if (refine) {
        // two blocks an SM: the candidates left are few
        int exact = (p->opts.flags & HAP_OPT_EXACT) != 0, max_pp = 1;
        for (const auto &cl : im.cls) max_pp = std::max(max_pp, cl.PP);
        const size_t smem = refine_smem_bytes(p->model.N, max_pp);
        ta.blocks_total = 2u * (unsigned)sm_count(p->device);
        const void *rf = nl ? (const void *)tree_refine_kernel<true> : (const void *)tree_refine_kernel<false>;
        CUDA_TRY(p, raise_smem_limit(p->device, rf, smem));
        void *args[] = {(void *)&ta, (void *)&p->dc, (void *)&exact, (void *)&max_pp};
        CUDA_TRY(p, launch_dependent(rf, ta.blocks_total, kRefineWarps * 32, smem, st, args));
    }
    p->state_dirty = ls.empty();                             // the last block of the recurrence clears the counters
    return HAP_OK;
}

// One launch of the general kernel per PP class (each has its own block shape); every block clips to the candidate range.
// skip_trees: only the classes without a tree.
static hap_status launch_dp(hap_problem *p, const DpOut &out, bool search, cudaStream_t st, bool f64 = false, bool skip_trees = false)
{
    // fork: every PP class runs on its own stream so that the tail of one class overlaps the next
    CUDA_TRY(p, cudaEventRecord(p->ev_fork, st));
    // the class with the most work goes first; the others fill the SMs it leaves free and its tail
    std::vector<const hap_problem::PpClass *> order;
    for (const auto &cl : p->classes) if (!(skip_trees && cl.tree >= 0)) order.push_back(&cl);
    std::stable_sort(order.begin(), order.end(), [](const hap_problem::PpClass *a, const hap_problem::PpClass *b) {
        return (a->item_hi - a->item_lo) * (size_t)a->PP > (b->item_hi - b->item_lo) * (size_t)b->PP;
    });
    // a pruning search wants a good incumbent early: the lower bound S + (M-1) ceil(S / PP) falls with PP, so the
    // deepest pipelines are the likeliest to hold the best plan and go first
    if (search && out.prune)
        std::stable_sort(order.begin(), order.end(), [](const hap_problem::PpClass *a, const hap_problem::PpClass *b) { return a->PP > b->PP; });
    for (const hap_problem::PpClass *clp : order) {
        const hap_problem::PpClass &cl = *clp;
        // skip classes whose candidates all lie outside the range
        if (!search && !out.first_dev && class_outside(p, cl, out)) continue;     // (a range that starts at a device-side index: every class looks)
        const bool lin = p->dc.tau_linear != 0;
        const bool refine = (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) != 0 && !out.count_only && !out.force_plain;
        const void *fn;
        if (f64) fn = lin ? (const void *)pipeline_dp_kernel<false, true, false, double> : (const void *)pipeline_dp_kernel<false, false, false, double>;
        else if (out.count_only) fn = lin ? (const void *)pipeline_dp_kernel<false, true, true> : (const void *)pipeline_dp_kernel<false, false, true>;
        else if (refine) fn = search ? (lin ? (const void *)pipeline_dp_kernel<true, true, false, i64, true> : (const void *)pipeline_dp_kernel<true, false, false, i64, true>)
                                     : (lin ? (const void *)pipeline_dp_kernel<false, true, false, i64, true> : (const void *)pipeline_dp_kernel<false, false, false, i64, true>);
        else fn = search ? (lin ? (const void *)pipeline_dp_kernel<true, true> : (const void *)pipeline_dp_kernel<true, false>)
                         : (lin ? (const void *)pipeline_dp_kernel<false, true> : (const void *)pipeline_dp_kernel<false, false>);
        CUDA_TRY(p, raise_smem_limit(p->device, fn, cl.smem));
        const unsigned blocks = (unsigned)(cl.item_hi - cl.item_lo);
        const uint8_t *tab = cl.has_tab ? p->d_maptab + cl.map_base : nullptr;
        DpOut o = out;
        o.exact = (p->opts.flags & HAP_OPT_EXACT) != 0 && !out.force_plain;
        if (search) { o.partial_cost += kTreeSlots + cl.item_lo; o.partial_index += kTreeSlots + cl.item_lo; }
        const WorkItem *its = p->d_items + cl.item_lo;
        int nw = cl.warps;
        unsigned used = cl.masks_used;
        void *c2arg = f64 ? (void *)p->d_c2f : (void *)p->d_c2;
        void *cvarg = f64 ? (void *)p->d_coeff : (void *)p->d_coef;
        void *args[] = {(void *)&p->dc, (void *)&its, (void *)&c2arg, (void *)&p->d_coef, (void *)&cvarg, (void *)&tab, (void *)&o, (void *)&nw, (void *)&used};
        CUDA_TRY(p, cudaStreamWaitEvent(cl.stream, p->ev_fork, 0));
        if (cl.has_tab && !cl.tab_valid) {        // stage masks and link classes of every mapping of the class
            const WorkItem &rep = p->items[cl.item_lo];
            const u64 nmap = p->pconfs[rep.p].nmap;
            maptab_kernel<<<(unsigned)((nmap + 3) / 4), 128, 0, cl.stream>>>(p->dc, rep.p, nmap, p->d_maptab + cl.map_base);
            CUDA_TRY(p, cudaGetLastError());
            cl.tab_valid = true;
        }
        CUDA_TRY(p, cudaLaunchKernel(fn, dim3(blocks), dim3(cl.warps * 32), args, cl.smem, cl.stream));
        CUDA_TRY(p, cudaEventRecord(cl.done, cl.stream));
        CUDA_TRY(p, cudaStreamWaitEvent(st, cl.done, 0));      // join
    }
    return HAP_OK;
}

static hap_status ensure_f64_buffers(hap_problem *p, bool layer_costs)
{
    const size_t np = p->pconfs.size();
    if (layer_costs && !p->d_c2f) CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_c2f, np * p->T * p->model.N * 2 * sizeof(double)));
    if (!p->d_coeff) CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_coeff, np * p->T * HAP_NCOEF * sizeof(double)));
    return HAP_OK;
}

// The recurrence of a pass: trees, the general kernel, or both.
static hap_status run_pass(hap_problem *p, DpOut &out, bool f64, cudaStream_t st)
{
    hap_status s;
    const bool trees = pass_uses_trees(p, out), general = !trees || !p->all_trees;
    if (general && (s = ensure_general(p)) != HAP_OK) return s;
    if (f64 && (s = ensure_f64_buffers(p, general || (p->opts.flags & HAP_OPT_NO_FUSE))) != HAP_OK) return s;
    if (trees && (p->opts.flags & HAP_OPT_NO_FUSE) && !f64 && (s = ensure_general(p)) != HAP_OK) return s;
    out.range_flag = p->d_range;
    if (trees && !general) {
        if ((s = launch_trees(p, out, false, f64, st, false)) != HAP_OK) return s;
        p->timed = 2;
        return HAP_OK;
    }
    out.counters = p->d_counters;
    CUDA_TRY(p, cudaMemsetAsync(p->d_counters, 0, 8 * sizeof(u64), st));
    CUDA_TRY(p, cudaEventRecord(p->ev[0], st));
    if (!trees) {
        unsigned p_lo, p_hi;
        configs_of_range(p, out.first, out.count, p_lo, p_hi);
        // the memory model stays on the integer byte coefficients in fp64 mode; times stay unrounded
        if (f64) {
            if ((s = launch_type_consts(p, p->d_coef, p->d_coeff, st, p_lo, p_hi)) != HAP_OK) return s;
            if ((s = launch_layer_kernel(p, nullptr, p->d_c2f, false, st, nullptr, p_lo, p_hi - p_lo, true)) != HAP_OK) return s;
        } else if ((s = launch_layer_costs(p, p->d_c2, p->d_coef, nullptr, nullptr, true, st, nullptr, p_lo, p_hi)) != HAP_OK) return s;
    }
    CUDA_TRY(p, cudaEventRecord(p->ev[1], st));
    if (trees && (s = launch_trees(p, out, false, f64, st, false)) != HAP_OK) return s;
    if ((s = launch_dp(p, out, false, st, f64, trees)) != HAP_OK) return s;
    CUDA_TRY(p, cudaEventRecord(p->ev[2], st));
    p->timed = 1;
    return HAP_OK;
}

extern "C" hap_status hap_pipeline_dp(hap_problem *p, uint64_t first, uint64_t count, int64_t *dev_cost,
                                      int64_t *dev_bottleneck, uint8_t *dev_partition, uint8_t *dev_recompute,
                                      int64_t *dev_dp_table, uint8_t *dev_choice, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    hap_status s = enter(p, st);
    if (s != HAP_OK) return s;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return HAP_OK;
    DpOut out{};
    out.cost = (i64 *)dev_cost; out.bottleneck = (i64 *)dev_bottleneck; out.partition = dev_partition;
    out.recompute = dev_recompute; out.dp_table = (i64 *)dev_dp_table; out.choice = dev_choice;
    out.first = first; out.count = count;
    if ((s = run_pass(p, out, false, st)) != HAP_OK) return s;
    return leave_async(p, st);
}

extern "C" hap_status hap_pipeline_dp_f64(hap_problem *p, uint64_t first, uint64_t count, double *dev_cost,
                                          double *dev_bottleneck, uint8_t *dev_partition, uint8_t *dev_recompute,
                                          void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    hap_status s = enter(p, st);
    if (s != HAP_OK) return s;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return HAP_OK;
    if (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) return fail(p, HAP_E_INVALID, "the refinement passes exist in integer mode only");
    DpOut out{};
    out.cost = (i64 *)dev_cost; out.bottleneck = (i64 *)dev_bottleneck; out.partition = dev_partition;
    out.recompute = dev_recompute; out.first = first; out.count = count;
    if ((s = run_pass(p, out, true, st)) != HAP_OK) return s;
    return leave_async(p, st);
}

// The plan a tree search's last block left, with the configuration's degrees
static void plan_of_result(const hap_problem *p, const TreeResult &r, hap_plan *host_out)
{
    const hap_pconf &pc = p->pconfs[r.pconf];
    host_out->index = r.index;
    host_out->PP = pc.PP; host_out->TP = pc.TP; host_out->CP = pc.CP; host_out->DP = pc.DP; host_out->EP = pc.EP;
    host_out->TPE = pc.TPE; host_out->b = pc.b; host_out->M = pc.M; host_out->rc_mask = r.rc_mask;
    std::memcpy(host_out->n, r.n, HAP_MAX_PP);
    std::memcpy(host_out->r, r.r, HAP_MAX_PP);
    std::memcpy(host_out->mask, r.mask, HAP_MAX_PP);
}

// Runs a search over the trees (every class has one) and waits for its result.
static hap_status tree_search(hap_problem *p, uint64_t first, uint64_t count, bool f64, cudaStream_t st, TreeResult &res, bool refine = false)
{
    hap_status s;
    if (f64 && (s = ensure_f64_buffers(p, (p->opts.flags & HAP_OPT_NO_FUSE) != 0)) != HAP_OK) return s;
    if ((p->opts.flags & HAP_OPT_NO_FUSE) && !f64 && (s = ensure_general(p)) != HAP_OK) return s;
    if (!p->host_result) p->host_result = result_slot_get();
    DpOut out{};
    out.first = first; out.count = count; out.prune = f64 ? 0 : p->opts.prune;
    if ((s = launch_trees(p, out, true, f64, st, true, refine)) != HAP_OK) return s;
    p->timed = 2;
    if (!p->host_result) CUDA_TRY(p, cudaMemcpyAsync(&res, p->targs.res_dev, sizeof(res), cudaMemcpyDeviceToHost, st));
    if ((s = leave_synced(p, st)) != HAP_OK) return s;
    if (p->host_result) std::memcpy(&res, p->host_result, sizeof(res));
    return HAP_OK;
}

extern "C" hap_status hap_search_range_f64(hap_problem *p, uint64_t first, uint64_t count, hap_plan *host_out,
                                           double *host_T_iter, double *host_bottleneck, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    hap_status s = enter(p, st);
    if (s != HAP_OK) return s;
    if (!host_out) return HAP_E_INVALID;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return fail(p, HAP_E_RANGE, "empty candidate range");
    if (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) return fail(p, HAP_E_INVALID, "the refinement passes exist in integer mode only");
    if (p->all_trees) {
        TreeResult r;
        if ((s = tree_search(p, first, count, true, st, r)) != HAP_OK) return s;
        std::memset(host_out, 0, sizeof(*host_out));
        double v[5];
        std::memcpy(&v[0], &r.cost, 8);
        if (!(v[0] < 1.0e300)) return fail(p, HAP_E_INFEASIBLE, "no candidate satisfies the memory constraint");
        std::memcpy(&v[1], &r.bott, 8); std::memcpy(&v[2], &r.T_pipe, 8); std::memcpy(&v[3], &r.T_sync, 8); std::memcpy(&v[4], &r.T_opt, 8);
        plan_of_result(p, r, host_out);
        host_out->T_iter = (int64_t)llrint(v[0]); host_out->bottleneck = (int64_t)llrint(v[1]);
        host_out->T_pipe = (int64_t)llrint(v[2]); host_out->T_sync = (int64_t)llrint(v[3]); host_out->T_opt = (int64_t)llrint(v[4]);
        if (host_T_iter) *host_T_iter = v[0];
        if (host_bottleneck) *host_bottleneck = v[1];
        return HAP_OK;
    }
    if ((s = ensure_general(p)) != HAP_OK || (s = ensure_f64_buffers(p, true)) != HAP_OK) return s;
    if (!p->d_fcost) CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_fcost, (size_t)p->n_cand * sizeof(i64)));
    if ((s = hap_pipeline_dp_f64(p, first, count, (double *)p->d_fcost, nullptr, nullptr, nullptr, stream)) != HAP_OK) return s;
    // non-negative doubles order like their bit patterns read as int64 (+inf is the largest), so the integer
    // (cost, index) argmin serves the fp64 costs unchanged
    if ((s = argmin_launch(p, p->d_fcost, count, p->d_best, st, 0x7fffffffffffffffll)) != HAP_OK) return s;
    i64 best[2];
    CUDA_TRY(p, cudaMemcpyAsync(best, p->d_best, sizeof(best), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(p, cudaStreamSynchronize(st));
    double bc;
    std::memcpy(&bc, &best[0], sizeof(bc));
    std::memset(host_out, 0, sizeof(*host_out));
    if (!(bc < 1.0e300)) return fail(p, HAP_E_INFEASIBLE, "no candidate satisfies the memory constraint");
    const u64 win = first + (u64)best[1];
    SingleOut *d1 = (SingleOut *)p->d_single;
    DpOut one{};
    one.cost = &d1->cost; one.bottleneck = &d1->bott; one.detail = d1->detail; one.partition = d1->part;
    one.recompute = d1->rec; one.first = win; one.count = 1;
    {   // the pass may have left the layer-cost array untouched: the winner's configuration is evaluated here
        size_t lo = 0, hi = p->pconfs.size();
        while (hi - lo > 1) { const size_t mid = (lo + hi) / 2; if (p->pconfs[mid].offset <= win) lo = mid; else hi = mid; }
        if ((s = launch_layer_kernel(p, nullptr, p->d_c2f, false, st, nullptr, (unsigned)lo, 1, false)) != HAP_OK) return s;
    }
    if ((s = launch_dp(p, one, false, st, true)) != HAP_OK) return s;
    decode_kernel<<<1, 32, 0, st>>>(p->dc, win, 1, &d1->cand, nullptr);
    CUDA_TRY(p, cudaGetLastError());
    SingleOut h1;
    CUDA_TRY(p, cudaMemcpyAsync(&h1, d1, sizeof(h1), cudaMemcpyDeviceToHost, st));
    if ((s = leave_synced(p, st)) != HAP_OK) return s;
    const hap_candidate &hc = h1.cand;
    const hap_pconf &pc = p->pconfs[hc.pconf];
    host_out->index = win;
    host_out->PP = pc.PP; host_out->TP = pc.TP; host_out->CP = pc.CP; host_out->DP = pc.DP; host_out->EP = pc.EP;
    host_out->TPE = pc.TPE; host_out->b = pc.b; host_out->M = pc.M; host_out->rc_mask = hc.rc_mask;
    std::memcpy(host_out->n, h1.part, HAP_MAX_PP);
    std::memcpy(host_out->r, h1.rec, HAP_MAX_PP);
    std::memcpy(host_out->mask, hc.mask, HAP_MAX_PP);
    double v[5];
    std::memcpy(&v[0], &h1.cost, 8); std::memcpy(&v[1], &h1.bott, 8); std::memcpy(&v[2], h1.detail, 24);
    host_out->T_iter = (int64_t)llrint(v[0]); host_out->bottleneck = (int64_t)llrint(v[1]);
    host_out->T_pipe = (int64_t)llrint(v[2]); host_out->T_sync = (int64_t)llrint(v[3]); host_out->T_opt = (int64_t)llrint(v[4]);
    if (host_T_iter) *host_T_iter = v[0];
    if (host_bottleneck) *host_bottleneck = v[1];
    return HAP_OK;
}

// The class's states as entries of joint_reach_kernel; false: its bits, masks or layer kinds do not fit that form.
static bool joint_reach_class(const hap_problem *p, int PP, int64_t G, const JointClass &jc, const std::vector<int> &lvl_off,
                              const std::vector<int> &st_idx, const std::vector<int> &slot, JointReach &jr, std::vector<unsigned> &ent)
{
    const int T = p->T, N = p->model.N;
    jr = JointReach{};
    jr.PP = PP; jr.lmax = jc.lmax; jr.nwin = 1;
    if (jc.lmax > 0xffff) return false;
    i64 Ps = 0;
    for (int h = 0; h < T; ++h) Ps += (p->m[h] / G) * p->dc.P[h];
    for (int h = 0; h < T; ++h) {
        // the window of dp_prologue_thr
        int lo = 1, hi = N - PP + 1;
        if (p->dc.delta_q >= 0) {
            const i64 den = 1024 * Ps, Ph = p->dc.P[h];
            const i64 a = ((i64)(1024 - p->dc.delta_q) * Ph * N) / den, b = ((i64)(1024 + p->dc.delta_q) * Ph * N + den - 1) / den;
            lo = a < 1 ? 1 : (int)a; hi = b > N - PP + 1 ? N - PP + 1 : (int)b;
        }
        if (p->dc.uniform) { lo = N / PP; hi = (N + PP - 1) / PP; }
        jr.nmin[h] = lo; jr.nmax[h] = hi; jr.cnt[h] = jc.cnt[h];
        if (lo < 1) return false;
        if (jc.cnt[h] == 0) continue;
        jr.nwin = std::max(jr.nwin, hi - lo + 1);
        // behind the first stage every span is of one layer kind
        if (PP > 1 && lo < p->dc.kind_uniform_from) return false;
    }
    int words = 1;
    for (int i = 0; i <= PP; ++i) {
        const int l0 = lvl_off[i], l1 = lvl_off[i + 1];
        jr.n_states[i] = (unsigned)(l1 - l0);
        int base = 1 << 20, top = -1;
        std::vector<uint8_t> out((size_t)(l1 - l0), 0);
        std::vector<int> u((size_t)(l1 - l0) * HAP_MAX_TYPES, 0);
        for (int q = l0; q < l1; ++q) {
            int smin = 0, smax = 0, rmin = 0, rmax = 0;
            for (int h = 0; h < T; ++h) {
                const int n = (st_idx[q] / jc.stride[h]) % (jc.cnt[h] + 1), left = jc.cnt[h] - n;
                u[(size_t)(q - l0) * HAP_MAX_TYPES + h] = n;
                smin += n * jr.nmin[h]; smax += n * jr.nmax[h]; rmin += left * jr.nmin[h]; rmax += left * jr.nmax[h];
            }
            const int bl = std::max(smin, N - rmax), bh = std::min(smax, N - rmin);
            if (bl > bh) { out[(size_t)(q - l0)] = 1; continue; }
            base = std::min(base, bl); top = std::max(top, bh);
        }
        jr.base[i] = top < 0 ? (i ? jr.base[i - 1] : 0) : base;
        jr.width[i] = top < 0 ? 0 : top - base + 1;
        if (i >= 1 && i < PP && top >= 0) {
            if (top - base + 1 > 128) return false;
            // a level's lengths are summed up from the shortest one's place and moved down from there where the level begins higher
            int down = 0;
            for (int h = 0; h < T && i >= 2; ++h) if (jc.cnt[h] > 0) down = std::max(down, jr.base[i] - jr.base[i - 1] - jr.nmin[h]);
            words = std::max(words, (jr.width[i] + down + 63) / 64);
        }
        jr.ent_off[i] = (unsigned)ent.size();
        if (i == 1)
            for (int h = 0; h < T; ++h) jr.first[h] = jc.cnt[h] > 0 ? (unsigned)slot[jc.stride[h]] : 0u;
        if (i == PP - 1)
            for (int h = 0; h < T; ++h) jr.fin[h] = jc.cnt[h] > 0 ? slot[jc.S - 1 - jc.stride[h]] : 0;
        if (i < 2 || i >= PP) continue;
        for (int t = 0; t < T; ++t)
            for (int q = l0; q < l1; ++q) {
                const int ut = u[(size_t)(q - l0) * HAP_MAX_TYPES + t];
                unsigned e = (unsigned)t << 16;
                if (ut > 0 && !out[(size_t)(q - l0)]) {
                    const i64 first = (i64)(ut - 1) * G;
                    const int same = (first - 1) / p->dc.node_size[t] == first / p->dc.node_size[t] ? 0 : 1;
                    e |= (unsigned)slot[st_idx[q] - jc.stride[t]] | (unsigned)same << 18 | 1u << 19;
                }
                ent.push_back(e);
            }
    }
    if (words > kReachWords) return false;
    jr.words = words;
    return reach_smem(N, T, p->prof.R, p->dc.tau_linear ? p->prof.R : 2, PP, jc.lmax, jr.nwin, words).total <= (words > 2 ? 140 : 110) * 1024;
}

static hap_status joint_setup(hap_problem *p)
{
    if (p->joint_ready) return HAP_OK;
    const int T = p->T, N = p->model.N;
    size_t lmax_all = 0;
    std::vector<int> pps;
    for (const auto &r : p->pconfs) if (std::find(pps.begin(), pps.end(), r.PP) == pps.end()) pps.push_back(r.PP);
    std::sort(pps.begin(), pps.end(), std::greater<int>());      // the longest configurations start first
    std::vector<unsigned> ent[kReachWords];
    // Where every class has few cells (states x types x layers) the value form is faster, whose chain is a level each where a
    // search is a dozen tests of it (64 devices, 32 layers, at most 18,496 cells: 297 us against 488; 32 devices, 24 layers, 16,200:
    // 208 against 340).  One class of many makes the search worth it (16 stages at 1,024 devices, 32,400 cells: 666 us against
    // 990; 32 stages at 32 devices, 132,192: 471 against 531, two policies 480 against 981), and then the others do better beside it in the
    // same launch than in launches of their own (32 devices, 32 layers: 492 us, 554 with the classes below 16,384 cells apart, 758
    // without a search).  A class in three words is a launch of its own, which its own cells have to make worth it: 32 devices, 255 layers, 400
    // configurations of four stages (9,180 cells) beside larger classes, 582 us in three words, 200 in the value form; 1,024 devices, 255
    // layers, 32 stages (3.9 million cells), 1.5 ms against 44.
    constexpr double kSearchCells = 20480.0;
    bool search = false;
    for (int PP : pps) {
        const int64_t G = p->W / PP;
        double cells = (double)T * N;
        for (int h = 0; h < T; ++h) cells = p->m[h] % G ? 0.0 : cells * (double)(p->m[h] / G + 1);
        search = search || cells >= kSearchCells;
    }
    for (int PP : pps) {
        const int64_t G = p->W / PP;
        bool homog = true;
        for (int h = 0; h < T; ++h) if (p->m[h] % G) homog = false;
        if (!homog) continue;
        hap_problem::JointHost jh;
        JointClass &jc = jh.jc;
        jc.PP = PP;
        int S = 1;
        for (int h = 0; h < HAP_MAX_TYPES; ++h) {
            jc.cnt[h] = h < T ? (int)(p->m[h] / G) : 0;
            jc.stride[h] = S;
            S *= jc.cnt[h] + 1;
            if (S > (1 << 22)) return fail(p, HAP_E_RANGE, "too many device states for the joint recurrence");
        }
        jc.S = S;
        std::vector<int> lvl_off(PP + 2, 0), st_idx(S), slot(S), level(S);
        for (int ui = 0; ui < S; ++ui) {
            int tot = 0;
            for (int h = 0; h < HAP_MAX_TYPES; ++h) tot += (ui / jc.stride[h]) % (jc.cnt[h] + 1);
            level[ui] = tot;
            lvl_off[tot + 1]++;
        }
        int lmax = 1;
        for (int l = 0; l <= PP; ++l) { lmax = std::max(lmax, lvl_off[l + 1]); lvl_off[l + 1] += lvl_off[l]; }
        std::vector<int> fill(lvl_off.begin(), lvl_off.end() - 1);
        for (int ui = 0; ui < S; ++ui) { slot[ui] = fill[level[ui]] - lvl_off[level[ui]]; st_idx[fill[level[ui]]++] = ui; }
        jc.lmax = lmax;
        JointReach jr;
        std::vector<unsigned> en;
        if (search && joint_reach_class(p, PP, G, jc, lvl_off, st_idx, slot, jr, en) && (jr.words <= 2 || (double)S * T * N >= kSearchCells)) {
            const int w = jr.words - 1;
            hap_problem::ReachHost &rh = p->reach[w];
            for (int i = 0; i <= HAP_MAX_PP; ++i) jr.ent_off[i] += (unsigned)ent[w].size();
            jr.id_lo = (unsigned)rh.ids.size();
            for (size_t pi = 0; pi < p->pconfs.size(); ++pi) if (p->pconfs[pi].PP == PP) rh.ids.push_back((unsigned)pi);
            jr.n_ids = (unsigned)rh.ids.size() - jr.id_lo;
            rh.smem = std::max<size_t>(rh.smem, reach_smem(N, T, p->prof.R, p->dc.tau_linear ? p->prof.R : 2, PP, lmax, jr.nwin, jr.words).total);
            rh.classes.push_back(jr);
            ent[w].insert(ent[w].end(), en.begin(), en.end());
            continue;
        }
        lmax_all = std::max(lmax_all, (size_t)lmax);
        std::vector<int> arrays;
        arrays.insert(arrays.end(), lvl_off.begin(), lvl_off.end());
        arrays.insert(arrays.end(), st_idx.begin(), st_idx.end());
        arrays.insert(arrays.end(), slot.begin(), slot.end());
        for (int pos = 0; pos < S; ++pos) {                      // stage counts per type of the states, in level order
            int dg = 0;
            for (int h = 0; h < HAP_MAX_TYPES; ++h) dg |= ((st_idx[pos] / jc.stride[h]) % (jc.cnt[h] + 1)) << (8 * h);
            arrays.push_back(dg);
        }
        arrays.insert(arrays.end(), (size_t)S, 0);               // band table, filled by the kernel
        CUDA_TRY(p, cached_malloc(p->device, (void **)&jh.d_arrays, arrays.size() * sizeof(int)));
        CUDA_TRY(p, cudaMemcpy(jh.d_arrays, arrays.data(), arrays.size() * sizeof(int), cudaMemcpyHostToDevice));
        jc.lvl_off = jh.d_arrays; jc.st_idx = jh.d_arrays + (PP + 2); jc.slot = jc.st_idx + S;
        jc.dig = jc.slot + S; jc.band = jh.d_arrays + (PP + 2) + 3 * (size_t)S;
        for (size_t pi = 0; pi < p->pconfs.size(); ++pi) if (p->pconfs[pi].PP == PP) jh.ids.push_back((unsigned)pi);
        CUDA_TRY(p, cached_malloc(p->device, (void **)&jh.d_ids, jh.ids.size() * sizeof(unsigned)));
        CUDA_TRY(p, cudaMemcpy(jh.d_ids, jh.ids.data(), jh.ids.size() * sizeof(unsigned), cudaMemcpyHostToDevice));
        jh.smem = joint_smem_bytes(N, PP, T, p->prof.R, p->dc.tau_linear != 0);
        if (jh.smem > 227 * 1024) return fail(p, HAP_E_RANGE, "shared memory need of the joint recurrence exceeds the SM");
        p->joint.push_back(jh);
    }
    for (int w = 0; w < kReachWords; ++w) {
        // classes | ids | entries
        hap_problem::ReachHost &rh = p->reach[w];
        if (rh.classes.empty()) continue;
        auto up = [](size_t v) { return (v + 255) / 256 * 256; };
        rh.o_ids = up(rh.classes.size() * sizeof(JointReach));
        const size_t o_ent = rh.o_ids + up(rh.ids.size() * sizeof(unsigned)), total = o_ent + up(ent[w].size() * sizeof(unsigned));
        CUDA_TRY(p, cached_malloc(p->device, (void **)&rh.d, total));
        for (auto &c : rh.classes) c.ent = reinterpret_cast<const unsigned *>(rh.d + o_ent);
        std::vector<unsigned char> img(total, 0);
        std::memcpy(img.data(), rh.classes.data(), rh.classes.size() * sizeof(JointReach));
        std::memcpy(img.data() + rh.o_ids, rh.ids.data(), rh.ids.size() * sizeof(unsigned));
        if (!ent[w].empty()) std::memcpy(img.data() + o_ent, ent[w].data(), ent[w].size() * sizeof(unsigned));
        CUDA_TRY(p, cudaMemcpy(rh.d, img.data(), total, cudaMemcpyHostToDevice));
    }
    p->joint_grid = 2 * sm_count(p->device);
    if (lmax_all) {
        const size_t bytes = (size_t)p->joint_grid * 2 * lmax_all * T * (N + 1) * sizeof(i64);
        CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_joint_scratch, bytes));
    }
    p->joint_ready = true;
    return HAP_OK;
}

extern "C" hap_status hap_joint_bottleneck(hap_problem *p, int64_t *dev_out, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if (!dev_out) return HAP_E_INVALID;
    if ((s = joint_setup(p)) != HAP_OK || (s = ensure_general(p)) != HAP_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t np = p->pconfs.size();
    CUDA_TRY(p, cudaMemsetAsync(dev_out, 0xff, np * p->opts.n_rc * sizeof(int64_t), st));     // -1: stages not homogeneous
    if ((s = launch_layer_costs(p, p->d_c2, p->d_coef, nullptr, nullptr, true, st)) != HAP_OK) return s;
    const bool lin = p->dc.tau_linear != 0;
    for (int w = 0; w < kReachWords; ++w) {
        const hap_problem::ReachHost &rh = p->reach[w];
        if (rh.classes.empty()) continue;
        using Fn = void (*)(const DevConst, const JointReach *, int, const unsigned *, const i64 *, const i64 *, i64 *);
        static const Fn fns[2][kReachWords] = {{joint_reach_kernel<false, 1>, joint_reach_kernel<false, 2>, joint_reach_kernel<false, 3>},
                                               {joint_reach_kernel<true, 1>, joint_reach_kernel<true, 2>, joint_reach_kernel<true, 3>}};
        const Fn fn = fns[lin][w];
        CUDA_TRY(p, raise_smem_limit(p->device, (const void *)fn, rh.smem));
        fn<<<(unsigned)rh.ids.size(), kReachThreads, rh.smem, st>>>(p->dc, reinterpret_cast<const JointReach *>(rh.d), (int)rh.classes.size(),
                                                                    reinterpret_cast<const unsigned *>(rh.d + rh.o_ids), p->d_c2, p->d_coef, (i64 *)dev_out);
        CUDA_TRY(p, cudaGetLastError());
    }
    for (const auto &jh : p->joint) {
        const void *fn = lin ? (const void *)joint_dp_kernel<true> : (const void *)joint_dp_kernel<false>;
        CUDA_TRY(p, raise_smem_limit(p->device, fn, jh.smem));
        const unsigned n_ids = (unsigned)jh.ids.size();
        const unsigned grid = std::min<unsigned>(n_ids, (unsigned)p->joint_grid);
        // scratch slices are sized for the widest class
        if (lin) joint_dp_kernel<true><<<grid, 256, jh.smem, st>>>(p->dc, jh.d_ids, n_ids, p->d_c2, p->d_coef, jh.jc, p->d_joint_scratch, (i64 *)dev_out);
        else joint_dp_kernel<false><<<grid, 256, jh.smem, st>>>(p->dc, jh.d_ids, n_ids, p->d_c2, p->d_coef, jh.jc, p->d_joint_scratch, (i64 *)dev_out);
        CUDA_TRY(p, cudaGetLastError());
    }
    return leave_async(p, st);
}

extern "C" hap_status hap_count_cells(hap_problem *p, uint64_t first, uint64_t count, uint64_t *host_cells, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if (!host_cells) return HAP_E_INVALID;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    *host_cells = 0;
    if (count == 0) return HAP_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if ((s = ensure_general(p)) != HAP_OK) return s;
    CUDA_TRY(p, cudaMemsetAsync(p->d_counters, 0, 8 * sizeof(u64), st));
    if ((s = launch_layer_costs(p, p->d_c2, p->d_coef, nullptr, nullptr, true, st)) != HAP_OK) return s;
    DpOut out{};
    out.counters = p->d_counters; out.first = first; out.count = count; out.count_only = 1;
    if ((s = launch_dp(p, out, false, st)) != HAP_OK) return s;
    CUDA_TRY(p, cudaMemcpyAsync(host_cells, p->d_counters + 4, sizeof(u64), cudaMemcpyDeviceToHost, st));
    if ((s = leave_synced(p, st)) != HAP_OK) return s;
    return check_values(p);
}

extern "C" hap_status hap_get_timings(hap_problem *p, float *ms_layer_cost, float *ms_dp, uint64_t *cells)
{
    if (!p) return HAP_E_INVALID;
    if (!p->enumerated || !p->timed) return fail(p, HAP_E_STATE, "no hap_pipeline_dp or hap_search_* call to report on");
    if (cudaSetDevice(p->device) != cudaSuccess) return fail(p, HAP_E_CUDA, "cudaSetDevice");
    { const hap_status w = wait_last(p); if (w != HAP_OK) return w; }
    if (p->timed == 2) {
        TreeReport ts;
        CUDA_TRY(p, cudaMemcpy(&ts, p->targs.report, sizeof(ts), cudaMemcpyDeviceToHost));
        if (ms_layer_cost) *ms_layer_cost = (float)((double)(ts.stamp[1] - ts.stamp[0]) * 1e-6);
        if (ms_dp) *ms_dp = (float)((double)(ts.stamp[2] - ts.stamp[1]) * 1e-6);
        if (cells) *cells = ts.splits;
        return check_values(p);
    }
    if (ms_layer_cost) CUDA_TRY(p, cudaEventElapsedTime(ms_layer_cost, p->ev[0], p->ev[1]));
    if (ms_dp) CUDA_TRY(p, cudaEventElapsedTime(ms_dp, p->ev[1], p->ev[2]));
    if (cells) CUDA_TRY(p, cudaMemcpy(cells, p->d_counters + 4, sizeof(u64), cudaMemcpyDeviceToHost));
    return check_values(p);
}

// The layer costs of the configurations that own the given plans, then the kernel that evaluates them as their programmatic
// dependent.
static hap_status launch_plan_eval(hap_problem *p, const void *fn, unsigned blocks, unsigned threads, u64 first, u64 count, const uint8_t *part,
                                   const uint8_t *rec, int64_t *t_iter, int64_t *detail, cudaStream_t st)
{
    unsigned p_lo, p_hi;
    configs_of_range(p, first, count, p_lo, p_hi);
    hap_status s;
    if ((s = launch_layer_costs(p, p->d_c2, p->d_coef, nullptr, nullptr, true, st, nullptr, p_lo, p_hi)) != HAP_OK) return s;
    const i64 *c2 = p->d_c2, *coef = p->d_coef;
    void *args[] = {(void *)&p->dc, (void *)&first, (void *)&count, (void *)&c2, (void *)&coef, (void *)&part, (void *)&rec, (void *)&t_iter, (void *)&detail,
                    (void *)&p_lo, (void *)&p_hi};
    CUDA_TRY(p, launch_dependent(fn, blocks, threads, 0, st, args));
    return HAP_OK;
}

extern "C" hap_status hap_eval_appendix_b(hap_problem *p, uint64_t first, uint64_t count, const uint8_t *dev_partition,
                                          const uint8_t *dev_recompute, int64_t *dev_t_iter, int64_t *dev_detail, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return HAP_OK;
    if (!dev_partition || !dev_recompute || !dev_t_iter) return HAP_E_INVALID;
    const uint64_t blocks = (count + 3) / 4;
    if (blocks > 0x7fffffffull) return fail(p, HAP_E_RANGE, "count too large for one launch");
    cudaStream_t st = (cudaStream_t)stream;
    if ((s = ensure_general(p)) != HAP_OK) return s;
    if ((s = launch_plan_eval(p, (const void *)appendix_b_kernel, (unsigned)blocks, 128, first, count, dev_partition, dev_recompute, dev_t_iter, dev_detail, st)) != HAP_OK) return s;
    return leave_async(p, st);
}

extern "C" hap_status hap_simulate_1f1b(hap_problem *p, uint64_t first, uint64_t count, const uint8_t *dev_partition,
                                        const uint8_t *dev_recompute, int64_t *dev_t_iter, int64_t *dev_detail, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return HAP_OK;
    if (!dev_partition || !dev_recompute || !dev_t_iter) return HAP_E_INVALID;
    if (count > 0x7fffffffull) return fail(p, HAP_E_RANGE, "count too large for one launch");
    cudaStream_t st = (cudaStream_t)stream;
    if ((s = ensure_general(p)) != HAP_OK) return s;
    if ((s = launch_plan_eval(p, (const void *)simulate_1f1b_kernel, (unsigned)count, 32, first, count, dev_partition, dev_recompute, dev_t_iter, dev_detail, st)) != HAP_OK) return s;
    return leave_async(p, st);
}

// ------------------------------------------------------------------------------------------
// hap_problem_save / hap_problem_load: the planner's inputs as one flat blob (the profiled tables are the
// expensive part of a planning problem: Sec. 4 caches them between runs)
// ------------------------------------------------------------------------------------------
namespace {
constexpr uint64_t kBlobMagic = 0x31424f4c42504148ull;        // "HAPBLOB1"
struct BlobWriter {
    unsigned char *buf; uint64_t cap, at = 0;
    void bytes(const void *src, uint64_t n) { if (buf && at + n <= cap) std::memcpy(buf + at, src, n); at += n; }
    template <class T> void pod(const T &v) { bytes(&v, sizeof(T)); }
    template <class T> void vec(const std::vector<T> &v) { pod<uint64_t>(v.size()); if (!v.empty()) bytes(v.data(), v.size() * sizeof(T)); }
};
struct BlobReader {
    const unsigned char *buf; uint64_t len, at = 0; bool ok = true;
    void bytes(void *dst, uint64_t n) { if (!ok || n > len - at) { ok = false; return; } std::memcpy(dst, buf + at, n); at += n; }
    template <class T> void pod(T &v) { bytes(&v, sizeof(T)); }
    template <class T> void vec(std::vector<T> &v, uint64_t max_n)
    {
        uint64_t n = 0; pod(n);
        if (!ok || n > max_n || n * sizeof(T) > len - at) { ok = false; return; }
        v.resize(n);
        if (n) bytes(v.data(), n * sizeof(T));
    }
};
}  // namespace

extern "C" hap_status hap_problem_save(hap_problem *p, void *host_buf, uint64_t cap, uint64_t *host_need)
{
    if (!p || !host_need) return HAP_E_INVALID;
    if (cudaSetDevice(p->device) != cudaSuccess) return fail(p, HAP_E_CUDA, "cudaSetDevice");
    const int N = p->model.N, T = p->T;
    const hap_profile &pf = p->prof;
    const size_t n4 = (size_t)T * pf.ntp * pf.ncp * pf.nmb, n5 = n4 * N;
    // the tables live on the device only (per-layer ones interleaved entry by entry): read them back in the caller's layout
    std::vector<double> dev(4 * n5 + 2 * n4), tab[4];
    CUDA_TRY(p, uploads_done(p));
    CUDA_TRY(p, cudaMemcpy(dev.data(), p->dc.tab4, dev.size() * sizeof(double), cudaMemcpyDeviceToHost));
    for (int t = 0; t < 4; ++t) { tab[t].resize(n5); for (size_t i = 0; i < n5; ++i) tab[t][i] = dev[4 * i + t]; }
    std::vector<double> tpre(dev.begin() + 4 * n5, dev.begin() + 4 * n5 + n4), tpost(dev.begin() + 4 * n5 + n4, dev.end());
    std::vector<double> fsize(p->dc.fsize, p->dc.fsize + pf.n_fsize), feff;
    for (int c = 0; c < 3; ++c) feff.insert(feff.end(), p->dc.feff[c], p->dc.feff[c] + pf.n_fsize);
    BlobWriter w{static_cast<unsigned char *>(host_buf), host_buf ? cap : 0};
    w.pod(kBlobMagic); w.pod<uint64_t>(0);                         // total size, patched below
    hap_model mo = p->model; mo.kind = nullptr;
    w.pod(mo); w.vec(p->kind);
    w.pod<int32_t>(T);
    w.vec(p->P); w.vec(p->C); w.vec(p->node_size); w.vec(p->bw_intra); w.vec(p->node_type); w.vec(p->node_bw_inter);
    w.vec(p->tp_list); w.vec(p->cp_list); w.vec(p->mb_list); w.vec(p->ep_list);
    for (int t = 0; t < 4; ++t) w.vec(tab[t]);
    w.vec(tpre); w.vec(tpost);
    w.vec(p->eta); w.vec(p->croute); w.vec(p->alpha); w.vec(p->rho); w.vec(p->act_coef); w.vec(p->copt); w.vec(p->cap_eff);
    w.vec(p->xi_q); w.vec(p->tau_q); w.vec(fsize); w.vec(feff);
    const double scal[7] = {pf.kappa, pf.chi, pf.gamma, pf.ovl_tp, pf.ovl_cp, pf.ovl_dp, pf.capf};
    w.bytes(scal, sizeof(scal));
    w.vec(p->pp_list); w.vec(p->tpe_list); w.vec(p->rc_masks);
    const hap_search_opts &so = p->opts;
    const int64_t oi[6] = {so.tp_max, so.delta_q, (int64_t)so.map_cap, so.prune, so.flags, so.eta_q};
    w.bytes(oi, sizeof(oi));
    *host_need = w.at;
    if (!host_buf || cap < w.at) return host_buf ? fail(p, HAP_E_RANGE, "the blob needs %llu bytes", (unsigned long long)w.at) : HAP_OK;
    std::memcpy(static_cast<unsigned char *>(host_buf) + 8, &w.at, 8);
    return HAP_OK;
}

extern "C" hap_status hap_problem_load(const void *host_buf, uint64_t len, hap_problem **out)
{
    if (!out) return HAP_E_INVALID;
    *out = nullptr;
    if (!host_buf || len < 16) return HAP_E_INVALID;
    BlobReader r{static_cast<const unsigned char *>(host_buf), len};
    uint64_t magic = 0, total = 0;
    r.pod(magic); r.pod(total);
    if (!r.ok || magic != kBlobMagic || total != len) return HAP_E_INVALID;
    constexpr uint64_t kMaxTab = 1ull << 28;
    hap_model mo{}; std::vector<uint8_t> kind;
    int32_t T = 0;
    std::vector<int64_t> P, C, cap_eff;
    std::vector<int32_t> node_size, node_type, tp, cp, mb, ep, xi, tau, pp, tpe;
    std::vector<double> bw_intra, node_bw, tab[4], tpre, tpost, eta, croute, alpha, rho, act, copt, fsize, feff;
    std::vector<uint32_t> rc;
    r.pod(mo); r.vec(kind, HAP_MAX_LAYERS);
    r.pod(T);
    r.vec(P, HAP_MAX_TYPES); r.vec(C, HAP_MAX_TYPES); r.vec(node_size, HAP_MAX_TYPES); r.vec(bw_intra, HAP_MAX_TYPES);
    r.vec(node_type, 1u << 20); r.vec(node_bw, 1u << 20);
    r.vec(tp, HAP_MAX_LIST); r.vec(cp, HAP_MAX_LIST); r.vec(mb, HAP_MAX_LIST); r.vec(ep, HAP_MAX_LIST);
    for (int t = 0; t < 4; ++t) r.vec(tab[t], kMaxTab);
    r.vec(tpre, kMaxTab); r.vec(tpost, kMaxTab);
    r.vec(eta, HAP_MAX_TYPES); r.vec(croute, HAP_MAX_TYPES); r.vec(alpha, 3); r.vec(rho, HAP_MAX_LIST); r.vec(act, 2);
    r.vec(copt, HAP_MAX_TYPES); r.vec(cap_eff, HAP_MAX_TYPES);
    r.vec(xi, HAP_MAX_RC); r.vec(tau, HAP_MAX_RC); r.vec(fsize, HAP_MAX_LIST); r.vec(feff, 3 * HAP_MAX_LIST);
    double scal[7] = {0}; r.bytes(scal, sizeof(scal));
    r.vec(pp, HAP_MAX_LIST); r.vec(tpe, HAP_MAX_LIST); r.vec(rc, HAP_MAX_RC_MASKS);
    int64_t oi[6] = {0}; r.bytes(oi, sizeof(oi));
    if (!r.ok || r.at != len) return HAP_E_INVALID;
    // sizes that hap_problem_create takes on trust from the pointers it is given
    if (T < 1 || T > HAP_MAX_TYPES || mo.N < 1 || (int64_t)kind.size() != mo.N || (int)P.size() != T || (int)C.size() != T ||
        (int)node_size.size() != T || (int)bw_intra.size() != T || node_type.size() != node_bw.size() || (int)eta.size() != T ||
        (int)croute.size() != T || alpha.size() != 3 || rho.size() != ep.size() || act.size() != 2 || (int)copt.size() != T ||
        (int)cap_eff.size() != T || xi.size() != tau.size() || xi.empty() || feff.size() != 3 * fsize.size())
        return HAP_E_INVALID;
    const size_t n4 = (size_t)T * tp.size() * cp.size() * mb.size(), n5 = n4 * (size_t)mo.N;
    for (int t = 0; t < 4; ++t) if (tab[t].size() != n5) return HAP_E_INVALID;
    if (tpre.size() != n4 || tpost.size() != n4) return HAP_E_INVALID;
    mo.kind = kind.data();
    hap_cluster cl{};
    cl.n_types = T; cl.P = P.data(); cl.C = C.data(); cl.node_size = node_size.data(); cl.bw_intra = bw_intra.data();
    cl.n_nodes = (int32_t)node_type.size(); cl.node_type = node_type.data(); cl.node_bw_inter = node_bw.data();
    hap_profile pf{};
    pf.ntp = (int32_t)tp.size(); pf.ncp = (int32_t)cp.size(); pf.nmb = (int32_t)mb.size(); pf.nep = (int32_t)ep.size();
    pf.tp_list = tp.data(); pf.cp_list = cp.data(); pf.mb_list = mb.data(); pf.ep_list = ep.data();
    pf.tdf = tab[0].data(); pf.tdb = tab[1].data(); pf.tff = tab[2].data(); pf.tfb = tab[3].data();
    pf.tpre = tpre.data(); pf.tpost = tpost.data();
    pf.eta = eta.data(); pf.croute = croute.data(); pf.kappa = scal[0]; pf.alpha = alpha.data(); pf.chi = scal[1];
    pf.rho = rho.data(); pf.gamma = scal[2]; pf.ovl_tp = scal[3]; pf.ovl_cp = scal[4]; pf.ovl_dp = scal[5];
    pf.act_coef = act.data(); pf.capf = scal[6]; pf.copt = copt.data(); pf.cap_eff = cap_eff.data();
    pf.R = (int32_t)xi.size(); pf.xi_q = xi.data(); pf.tau_q = tau.data();
    pf.n_fsize = (int32_t)fsize.size(); pf.fsize = fsize.empty() ? nullptr : fsize.data(); pf.feff = feff.empty() ? nullptr : feff.data();
    hap_search_opts so{};
    so.npp = (int32_t)pp.size(); so.ntpe = (int32_t)tpe.size(); so.pp_list = pp.data(); so.tpe_list = tpe.data();
    so.tp_max = (int32_t)oi[0]; so.delta_q = (int32_t)oi[1]; so.map_cap = (uint64_t)oi[2]; so.n_rc = (int32_t)rc.size();
    so.rc_masks = rc.data(); so.prune = (int32_t)oi[3]; so.flags = (int32_t)oi[4]; so.eta_q = (int32_t)oi[5];
    return hap_problem_create(&mo, &cl, &pf, &so, out);
}

extern "C" hap_status hap_problem_dims(const hap_problem *p, int32_t *host_N, int32_t *host_T, int32_t *host_n_rc)
{
    if (!p) return HAP_E_INVALID;
    if (host_N) *host_N = p->model.N;
    if (host_T) *host_T = p->T;
    if (host_n_rc) *host_n_rc = p->opts.n_rc;
    return HAP_OK;
}

extern "C" hap_status hap_self_check(uint64_t *host_sites)
{
    if (!host_sites) return HAP_E_INVALID;
    *host_sites = 0;
#ifdef HAP_CHECKED
    if (cudaDeviceSynchronize() != cudaSuccess) return HAP_E_CUDA;
    unsigned long long sites = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&sites, hap::g_hap_check_sites, sizeof(sites)) != cudaSuccess) return HAP_E_CUDA;
    if (cudaMemcpyToSymbol(hap::g_hap_check_sites, &zero, sizeof(zero)) != cudaSuccess) return HAP_E_CUDA;
    *host_sites = sites;
    return HAP_OK;
#else
    return HAP_E_STATE;                     // the checks are compiled away in this build
#endif
}

extern "C" hap_status hap_launches_per_pass(hap_problem *p, uint32_t *host_count)
{
    if (!p || !host_count) return HAP_E_INVALID;
    if (!p->enumerated) return fail(p, HAP_E_STATE, "hap_enumerate has not run");
    DpOut out{};
    const bool trees = pass_uses_trees(p, out);
    uint32_t n = 1 + 2;                                     // type constants; argmin partial and final
    if (!trees || !p->all_trees || (p->opts.flags & HAP_OPT_NO_FUSE)) n += 1;              // layer-cost array
    if (trees) n += 1 + (uint32_t)tree_launches(p, false, false, false, 0, (unsigned)p->pconfs.size()).size();     // records, recurrence
    for (const auto &cl : p->classes) if (!trees || cl.tree < 0) n += 1;                    // one warp per candidate
    *host_count = n;
    return HAP_OK;
}

static hap_status argmin_launch(hap_problem *p, const i64 *dev_cost, uint64_t count, i64 *dev_out, cudaStream_t st, i64 init)
{
    const unsigned blocks = (unsigned)std::min<uint64_t>((count + 255) / 256, 1024);
    argmin_partial_kernel<<<blocks, 256, 0, st>>>(dev_cost, count, p->d_pcost, p->d_pindex, init);
    CUDA_TRY(p, cudaGetLastError());
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    const i64 *pc = p->d_pcost; const u64 *pi = p->d_pindex; const u64 nb = blocks;
    CUDA_TRY(p, cudaLaunchKernelEx(&cfg, argmin_final_kernel, pc, pi, nb, dev_out, init));
    return HAP_OK;
}

extern "C" hap_status hap_argmin(hap_problem *p, const int64_t *dev_cost, uint64_t count, int64_t *dev_out, void *stream)
{
    hap_status s = enter(p, (cudaStream_t)stream);
    if (s != HAP_OK) return s;
    if (!dev_cost || !dev_out || count == 0) return HAP_E_INVALID;
    if ((s = argmin_launch(p, (const i64 *)dev_cost, count, (i64 *)dev_out, (cudaStream_t)stream, kInf)) != HAP_OK) return s;
    return leave_async(p, (cudaStream_t)stream);
}

static void search_stats(const hap_problem *p, hap_search_stats *st, u64 evaluated, u64 feasible, u64 pruned, float ms_lc, float ms_dp)
{
    if (!st) return;
    std::memset(st, 0, sizeof(*st));
    st->n_pconf = p->pconfs.size(); st->n_candidates = p->n_cand;
    st->n_evaluated = evaluated; st->n_feasible = feasible; st->n_pruned = pruned;
    st->ms_layer_cost = ms_lc; st->ms_dp = ms_dp; st->ms_total = ms_lc + ms_dp;
}

extern "C" hap_status hap_search_range(hap_problem *p, uint64_t first, uint64_t count, hap_plan *host_out,
                                       hap_search_stats *host_stats, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    hap_status s = enter(p, st);
    if (s != HAP_OK) return s;
    if (!host_out) return HAP_E_INVALID;
    if ((s = check_range(p, first, count)) != HAP_OK) return s;
    if (count == 0) return fail(p, HAP_E_RANGE, "empty candidate range");
    std::memset(host_out, 0, sizeof(*host_out));
    const bool refine_mode = (p->opts.flags & (HAP_OPT_REFINE | HAP_OPT_EXACT)) != 0;
    DpOut out{};
    out.first = first; out.count = count; out.prune = p->opts.prune;
    // A refinement objective costs a warp per candidate and up to dozens of recurrences each: the trees list the candidates
    // whose lower bound does not exceed the smallest plain T_iter, and those are refined.  (Where that does not decide the
    // search -- every refined T_iter above the plain one, or too long a list -- the general form below does.)
    DpOut as_plain = out;
    as_plain.force_plain = 1;
    TreeResult r;
    r.again = 1;
    if (p->all_trees && pass_uses_trees(p, as_plain)) {
        // the last block writes the plan of the winner to the host
        if ((s = tree_search(p, first, count, false, st, r, refine_mode)) != HAP_OK) return s;
    }
    if (!r.again) {
        search_stats(p, host_stats, count - r.n_pruned, r.n_feasible, r.n_pruned, (float)((double)(r.stamp[1] - r.stamp[0]) * 1e-6),
                     (float)((double)(r.stamp[2] - r.stamp[1]) * 1e-6));
        if (r.range_flag) return fail(p, HAP_E_RANGE, "a layer time or stage coefficient exceeds the supported range (see hap.h)");
        if (r.cost >= kInf) return fail(p, HAP_E_INFEASIBLE, "no candidate satisfies the memory constraint");
        plan_of_result(p, r, host_out);
        host_out->T_iter = r.cost; host_out->bottleneck = r.bott; host_out->T_pipe = r.T_pipe; host_out->T_sync = r.T_sync; host_out->T_opt = r.T_opt;
        return HAP_OK;
    }
    if ((s = ensure_general(p)) != HAP_OK) return s;
    const u64 init_counters[8] = {0, 0, 0, (u64)kInf, 0, 0, 0, 0};           // [3] = incumbent starts at +INF
    CUDA_TRY(p, cudaMemcpyAsync(p->d_counters, init_counters, sizeof(init_counters), cudaMemcpyHostToDevice, st));
    CUDA_TRY(p, cudaEventRecord(p->ev[0], st));
    out.lb_sum = p->d_lb;
    out.partial_cost = p->d_pcost; out.partial_index = p->d_pindex; out.counters = p->d_counters;
    out.incumbent = p->d_counters + 3; out.range_flag = p->d_range;
    const bool trees = pass_uses_trees(p, out);               // (some classes have a tree, some do not)
    unsigned p_lo, p_hi;
    configs_of_range(p, first, count, p_lo, p_hi);
    if (refine_mode && count > 1) { p_lo = 0; p_hi = ~0u; }          // (the bounds kernel below reads every configuration's S)
    if (!trees && (s = launch_layer_costs(p, p->d_c2, p->d_coef, nullptr, nullptr, true, st, p->d_lb, p_lo, p_hi)) != HAP_OK) return s;
    CUDA_TRY(p, cudaEventRecord(p->ev[1], st));
    if (refine_mode && count > 1) {
        // The refinement and the exact sweep cost one warp per candidate and up to dozens of passes each, so they run
        // only where they can matter.  A plain pass over the prefix trees leaves every candidate's bottleneck B*; with
        // S the configuration's lower bound on the stage-cost sum, no partition of the candidate gets below
        // S + (M-1) B* (sync and optimizer terms only add).  The candidate with the smallest bound is evaluated first
        // and its cost starts the incumbent; the refinement kernels then skip every candidate whose bound exceeds the
        // incumbent (strict, so the (cost, index) minimum is unchanged).
        if (!p->d_cand_lb) CUDA_TRY(p, cached_malloc(p->device, (void **)&p->d_cand_lb, (size_t)p->n_cand * sizeof(i64)));
        DpOut plain{};
        plain.bottleneck = p->d_cand_lb + first;         // the kernels index outputs by candidate - first: entry c of the array
        plain.first = first; plain.count = count; plain.force_plain = 1; plain.range_flag = p->d_range;
        const bool plain_trees = pass_uses_trees(p, plain);
        if (plain_trees && (s = launch_trees(p, plain, false, false, st, false)) != HAP_OK) return s;
        if ((!plain_trees || !p->all_trees) && (s = launch_dp(p, plain, false, st, false, plain_trees)) != HAP_OK) return s;
        cand_bound_kernel<<<(unsigned)p->pconfs.size(), 128, 0, st>>>(p->dc, p->d_lb, p->d_cand_lb, first, count);
        CUDA_TRY(p, cudaGetLastError());
        if ((s = argmin_launch(p, p->d_cand_lb + first, count, p->d_best, st, kInf)) != HAP_OK) return s;
        offset_index_kernel<<<1, 32, 0, st>>>(p->d_best + 1, (i64)first);
        SingleOut *d0 = (SingleOut *)p->d_single;
        DpOut seed{};
        seed.cost = &d0->cost; seed.first = 0; seed.count = 1; seed.first_dev = p->d_best + 1;
        if ((s = launch_dp(p, seed, false, st)) != HAP_OK) return s;
        set_incumbent_kernel<<<1, 32, 0, st>>>(p->d_counters + 3, &d0->cost, p->d_best + 1);
        CUDA_TRY(p, cudaGetLastError());
        out.cand_lb = p->d_cand_lb;
    }
    if (trees) {
        const unsigned slots = kTreeSlots + (unsigned)p->items.size();      // (the tree kernel's idle slots and the items it takes over)
        fill_partials_kernel<<<(slots + 255) / 256, 256, 0, st>>>(p->d_pcost, p->d_pindex, slots);
        CUDA_TRY(p, cudaGetLastError());
        if ((s = launch_trees(p, out, true, false, st, false)) != HAP_OK) return s;
    }
    if ((s = launch_dp(p, out, true, st, false, trees)) != HAP_OK) return s;
    const size_t slot0 = trees ? 0 : kTreeSlots;
    argmin_final_kernel<<<1, 256, 0, st>>>(p->d_pcost + slot0, p->d_pindex + slot0, kTreeSlots + p->items.size() - slot0, p->d_best, kInf);
    CUDA_TRY(p, cudaGetLastError());
    CUDA_TRY(p, cudaEventRecord(p->ev[2], st));
    p->timed = 1;
    // the winner is evaluated once more alone, for its partition and recomputation levels; its index stays on the device
    // (every class's kernel looks whether the index is its own), so the host waits only once
    SingleOut *d1 = (SingleOut *)p->d_single;
    DpOut one{};
    one.cost = &d1->cost; one.bottleneck = &d1->bott; one.detail = d1->detail; one.partition = d1->part;
    one.recompute = d1->rec; one.first = 0; one.count = 1; one.first_dev = p->d_best + 1;
    if ((s = launch_dp(p, one, false, st)) != HAP_OK) return s;
    decode_kernel<<<1, 32, 0, st>>>(p->dc, 0, 1, &d1->cand, p->d_best + 1);
    CUDA_TRY(p, cudaGetLastError());
    i64 best[2];
    u64 counters[4], flag = 0;
    SingleOut h1;
    TreeReport ts{};
    CUDA_TRY(p, cudaMemcpyAsync(&flag, p->d_range, sizeof(flag), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(p, cudaMemcpyAsync(counters, p->d_counters, sizeof(counters), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(p, cudaMemcpyAsync(best, p->d_best, sizeof(best), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(p, cudaMemcpyAsync(&h1, d1, sizeof(h1), cudaMemcpyDeviceToHost, st));
    if (trees) CUDA_TRY(p, cudaMemcpyAsync(&ts, p->targs.report, sizeof(ts), cudaMemcpyDeviceToHost, st));
    if ((s = leave_synced(p, st)) != HAP_OK) return s;
    float ms_lc = 0.0f, ms_dp = 0.0f;
    cudaEventElapsedTime(&ms_lc, p->ev[0], p->ev[1]);
    cudaEventElapsedTime(&ms_dp, p->ev[1], p->ev[2]);
    const u64 pruned = counters[2] + ts.n_pruned;
    search_stats(p, host_stats, count - pruned, counters[1] + ts.n_feasible, pruned, ms_lc, ms_dp);
    if (flag) return fail(p, HAP_E_RANGE, "a layer time or stage coefficient exceeds the supported range (see hap.h)");
    if (best[0] >= kInf) return fail(p, HAP_E_INFEASIBLE, "no candidate satisfies the memory constraint");
    const u64 win = (u64)best[1];
    const hap_candidate &hc = h1.cand;
    if (h1.cost != best[0] || hc.index != win) return fail(p, HAP_E_CUDA, "winner re-evaluation disagrees with the search");
    const hap_pconf &pc = p->pconfs[hc.pconf];
    host_out->index = win;
    host_out->PP = pc.PP; host_out->TP = pc.TP; host_out->CP = pc.CP; host_out->DP = pc.DP; host_out->EP = pc.EP;
    host_out->TPE = pc.TPE; host_out->b = pc.b; host_out->M = pc.M; host_out->rc_mask = hc.rc_mask;
    std::memcpy(host_out->n, h1.part, HAP_MAX_PP);
    std::memcpy(host_out->r, h1.rec, HAP_MAX_PP);
    std::memcpy(host_out->mask, hc.mask, HAP_MAX_PP);
    host_out->T_iter = h1.cost; host_out->bottleneck = h1.bott;
    host_out->T_pipe = h1.detail[0]; host_out->T_sync = h1.detail[1]; host_out->T_opt = h1.detail[2];
    return HAP_OK;
}

extern "C" hap_status hap_search_best(hap_problem *p, hap_plan *host_out, hap_search_stats *host_stats, void *stream)
{
    if (!p) return HAP_E_INVALID;
    if (!p->enumerated) return fail(p, HAP_E_STATE, "hap_enumerate has not run");
    return hap_search_range(p, 0, p->n_cand, host_out, host_stats, stream);
}

// ------------------------------------------------------------------------------------------
// hap_argmin_static: the (cost, index) minimum without any allocation
// ------------------------------------------------------------------------------------------
// Scratch for the per-block partial minima lives in the library image itself.  Every device that
// loads the library carries these 64 KiB until the process exits.
constexpr unsigned kStaticArgminTile = 16384;                                   // costs per block
constexpr unsigned kStaticArgminBlocks = (unsigned)(HAP_ARGMIN_STATIC_MAX_COUNT / kStaticArgminTile);
static __device__ __align__(256) unsigned char g_argmin_static_scratch[kStaticArgminBlocks * 16];

// In host code the name above is only a handle for the runtime, not an address a kernel can use.
// The device address is looked up once per device (with that device current) and cached here.
// The entry point has no handle, so it is the one most likely to be called from several host threads: the lookup
// is serialised (a lock per call costs nothing beside two kernel launches).
static void *g_argmin_static_ptr[64];
static bool g_argmin_static_ready[64];
static std::mutex g_argmin_static_mu;

extern "C" hap_status hap_argmin_static(const int64_t *dev_cost, uint64_t count, int64_t *dev_out, void *stream)
{
    if (!dev_cost || !dev_out) return HAP_E_INVALID;
    if (count == 0 || count > HAP_ARGMIN_STATIC_MAX_COUNT) return HAP_E_RANGE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HAP_E_CUDA;
    if (dev < 0 || dev >= 64) return HAP_E_RANGE;
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_argmin_static_mu);
        if (!g_argmin_static_ready[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_argmin_static_scratch) != cudaSuccess || !ptr) return HAP_E_CUDA;
            g_argmin_static_ptr[dev] = ptr;
            g_argmin_static_ready[dev] = true;
        }
        scratch = g_argmin_static_ptr[dev];
    }
    {   // the cost array must live on the current device (the scratch and the launches do)
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, dev_cost) != cudaSuccess) { cudaGetLastError(); return HAP_E_INVALID; }
        if (at.type == cudaMemoryTypeDevice && at.device != dev) return HAP_E_INVALID;
    }
    i64 *pcost = reinterpret_cast<i64 *>(scratch);
    u64 *pindex = reinterpret_cast<u64 *>(pcost + kStaticArgminBlocks);
    cudaStream_t st = (cudaStream_t)stream;
    const unsigned blocks = (unsigned)((count + kStaticArgminTile - 1) / kStaticArgminTile);
    // every partial that the second kernel reads is written by the first one in this same call, so
    // nothing left in the scratch by an earlier call is ever read and nothing has to be cleared
    argmin_partial_kernel<<<blocks, 256, 0, st>>>((const i64 *)dev_cost, count, pcost, pindex, kInf);
    if (cudaGetLastError() != cudaSuccess) return HAP_E_CUDA;
    argmin_final_kernel<<<1, 256, 0, st>>>(pcost, pindex, blocks, (i64 *)dev_out, kInf);
    if (cudaGetLastError() != cudaSuccess) return HAP_E_CUDA;
    return HAP_OK;
}
