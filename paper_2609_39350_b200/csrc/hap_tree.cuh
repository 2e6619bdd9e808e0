// Prefix-tree form of the min-max pipeline recurrence (sm_100a).
//
// The DP row of stage d of a candidate depends only on the candidate's stages 1..d (their device
// types, boundary links and load-balance windows), the configuration and the recomputation policy.
// All mappings of a PP class therefore form a prefix tree whose nodes are distinct stage prefixes;
// the tree, the band of reachable end layers of every node and the task list below depend on the
// class alone and are laid out once on the host.
//
//   type_const_kernel  (hap_device.cuh) constants of Eq. 2 / Eq. 3, and which configurations can place a first stage.
//   tree_prep_kernel   a block per such configuration at a time: Eq. 2 for every (device type, layer), the prefix rows of the
//                      stage time per type mask and level, the memory thresholds and the stage constants, written
//                      as one record for the DP kernel.  The other configurations' candidates are infeasible: a
//                      warp each writes their results.
//   tree_dp_kernel     persistent blocks of four warps that take (configuration, up to four of its tree's parts) items
//                      from a counter; in a pass an item of a class with long chains is one policy's.  A warp owns a
//                      part of the tree -- a few to some tens of mappings -- and walks it depth by depth on its own
//                      (parts of one configuration, or of a few where they have one or two):
//                      no block barrier inside an item.  A task is one, two or four consecutive end layers of a node (four
//                      where the lanes are full, fewer where lanes would idle); a lane keeps
//                      their running minima and slides one window of the parent's row over the stage lengths
//                      (tree_scan).  Then one lane per mapping evaluates the last stage, walks the choices back and
//                      assembles Eq. 4.  A search leaves the plan of the best candidate; the last block to finish
//                      reduces the blocks' minima and decodes the winner.
//
// Bounds and figures (B200).  1,024 devices, 96 layers, 2.4 million candidates: a pass takes 358 us (435 with a block per
// configuration and a barrier per depth); 256 devices with partitions 410 us (985); 64 devices with three levels 109 us.  The same
// 1,024 devices where no stage size is homogeneous, 374 thousand candidates in classes of 24 mappings: 244 us when a pass took 390
// (274 with that barrier, 371 while one to three of a block's warps had a part).  The recurrence is bound by instruction issue and by
// the chain of a part: a warp issues an instruction every seven to eight cycles, 20 to 25 of 32 lanes active; half of them are the
// scans', a fifth the ways' back; its row entries never leave shared memory.  A deeper
// split into blocks that share a tree needs a barrier per depth (31 of them at 32 stages); a warp of its own per part needs
// none.  Measured while a pass took 400 us: two end layers per task and eight blocks an SM 475 us, one end layer 536, eight parts an
// item instead of four 405 (373 against 359 now).
// Records computed by the items themselves instead of tree_prep_kernel: 270 us instead of 284 in classes of few mappings,
// but 513 instead of 475 at 256 devices, because the recurrence then has fewer registers; not kept.
//
// Integer mode holds times (integer ns below 2^52) as doubles: every sum, difference and comparison is exact.
#pragma once
#include "hap_device.cuh"

namespace hap {

constexpr int kTreeWarps = 4;             // warps of a DP block
constexpr int kTreeThreads = kTreeWarps * 32;
// Blocks an SM: five (96 registers a thread), or four (128) for searches of several waves of items, whose last chains run faster beside
// fewer warps and with what a plan takes in registers: pruned search at 1,024 devices 195 us with four, 214 with five, an unpruned plan from
// host tables 440 and 455, exact search at 256 devices 250 and 271.  Where the feasible items are two waves at most, every chain begins at
// once or nearly so: 64 devices 135 us with four, 130 with five.  Passes take five: 256 devices with partitions 420 us with four, 410 with
// five, against 355 and 358 at 1,024 devices.  Rows that are not combined by level need no more than 96 registers: 139 and 126.  (The number of
// parts is planned for five blocks, whichever kernel runs.)
constexpr int kTreeBlocksPerSm = 5, kTreeSearchBlocksPerSm = 4;
constexpr int kTreeJ = 4;                 // end layers of a task at most
template <int J> struct TreeWidth { static constexpr int value = J; };
constexpr int kTreePad = kTreeJ - 1;      // infinite entries in front of every row and behind the last one
constexpr int kTreeAhead = 2;             // and entries in front of them all: a scan asks for the next two before it knows that it is done
constexpr int kTreeKtab = 16 + HAP_MAX_TYPES * 6;    // stage constants: [0,16) pre-work by row group, then p2p [type][6]
constexpr int kTreeMinfo = 8;             // doubles per row group: sync latency, sync bandwidth x 2, optimizer x 2, cross dispatch, post-work, pad

// A task: one, two or up to four consecutive end layers j0..j0+cnt-1 of one node (a stage prefix of depth d < PP) and the stage lengths
// a..b that reach the parent's row from any of them.
//   x = slot of prev[j0 - a] in the previous depth's buffer | slot of j0's value in this depth's << 16
//   y = j0 | a << 8 | b << 16 | cnt << 24 | first of its row << 27 | last of the depth << 28
//   z = stage constant index | row group of the stage's types << 8 | threshold word (4 (d - 1) + capacity type) << 16
//   w = slot of j0's choice | end layers of the tasks in this iteration at most (1, 2, 4) << 16 | ends its depth << 19 |
//       thresholds by end layer << 20: all but the slot the same for the 32 tasks that a warp takes together
// A depth's last iteration is filled up with tasks of no end layer (cnt = 0, a > b), and one iteration of them follows the last depth,
// so that the next tasks are asked for without a look at how many there are.  With a list per depth, whose ends and first choice were
// looked up as it began, a third of the recurrence's instructions lay outside the scans: pass at 1,024 devices 379 us against 359, 256
// devices with partitions 439 against 419, pruned search 222 against 215.
typedef uint4 TreeTask;
constexpr u32 kTaskEnds = 1u << 19, kTaskByLayer = 1u << 20;

// A contiguous range of a class's mappings with the tree of their prefixes.
struct TreePart {
    const TreeTask *tasks;                  // grouped by depth
    const u32 *path;                        // [PP][nmap] stage d of mapping m: origin of its node among the choices (choice of
                                            // end layer 0, + 256), 20 bits; d = PP: slot of prev[N - a] of the last stage;
                                            // | stage constant index << 20 | row group << 26 | capacity type << 30
    const u32 *leaf;                        // [nmap] lengths of the last stage that reach the parent's row: a | b << 8;
                                            // a > b: the windows cannot add up to N
    u32 nmap, m_lo;                         // mappings [m_lo, m_lo + nmap) of the class
    u32 n_iter;                             // iterations of 32 tasks, depth by depth
};

// A PP class that walks its tree.
struct TreeClass {
    const TreePart *parts;
    u64 rec_off;                            // byte offset of the class's records
    u32 p_lo, n_conf;                       // its configurations are contiguous
    u32 rec_bytes;                          // one configuration's record
    u32 o_rows, o_thr_nf;                   // offsets in a record
    u32 buf_cells[2], ch_bytes;             // a warp's row buffers (even / odd depths, in values) and choices
    int PP, n_parts, n_mrows;
    u32 ipc_inverse;                        // 2^32 / items_per_conf, rounded up (0: one item)
    int items_per_conf;                     // an item is a group of the configuration's parts (at most a part a warp) ...
    int policy_items;                       // ... under all policies (1) or, in passes, under one (then: the number of policies)
    int group;                              // ... or, in the kernel's grouped form, of this many configurations whose parts all fit a block's warps
    uint8_t mrow_of[16], mask_of_row[16];   // type mask <-> row group
    uint8_t first_min[HAP_MAX_TYPES];       // per capacity type: shortest first stage (255: no first stage on it)
    uint8_t wmax[HAP_MAX_PP + 1];           // longest stage of depth d
    uint8_t tmask[HAP_MAX_PP + 1];          // capacity types that occur at depth d
    uint8_t jlo[HAP_MAX_PP + 1], jhi[HAP_MAX_PP + 1], kmin[HAP_MAX_PP + 1], kmax[HAP_MAX_PP + 1];
    uint8_t flat[HAP_MAX_PP + 1];           // depth d sees spans of one layer kind only: its thresholds are lengths (one word
                                            // per type, a byte per level); else a byte per (type, level, end layer) at nf_off[d]
    uint8_t all_flat;
    u32 nf_off[HAP_MAX_PP + 1], nf_w[HAP_MAX_PP + 1];
};

// Head of a configuration's record.
struct __align__(16) TreeHead {
    u64 offset;                             // first candidate of the configuration
    i64 m1;                                 // micro-batches - 1
    i64 lb;                                 // lower bound on T_iter of its candidates (searches)
    u32 p;
    u32 dead_policies;                      // by position in rc_order: no mapping can be feasible
    i64 S;                                  // lower bound on the summed stage time (searches)
    u64 pad[3];
};
static_assert(sizeof(TreeHead) == 64, "the stage constants start behind it");
constexpr u32 kTreeOffKtab = sizeof(TreeHead);
constexpr u32 kTreeOffThr = kTreeOffKtab + kTreeKtab * 8;                  // [depth - 1][HAP_MAX_TYPES] words
constexpr u32 kTreeOffMinfo = kTreeOffThr + HAP_MAX_PP * HAP_MAX_TYPES * 4;

// What a search brings back, written by the last block: to the host's mapped copy where there is one, else to device memory.
struct TreeResult {
    u64 range_flag, n_feasible, n_pruned, again;      // again: the listed candidates do not decide the search
    i64 cost; u64 index;
    i64 bott, T_pipe, T_sync, T_opt;
    u32 pconf, rc_mask;
    u64 stamp[3];                           // global timer: pass begins, recurrence begins, all done
    uint8_t n[HAP_MAX_PP], r[HAP_MAX_PP], mask[HAP_MAX_PP];
};

// Device words a pass counts in.  All zero between passes: the last block of a pass leaves them so.
struct TreeState {
    u32 live[HAP_MAX_PP + 2];               // configurations on each class's list; behind the last class, on the dead list
    u32 ticket[2];                          // next item of each DP launch
    u32 blocks_done, prep_done;
    u64 n_feasible, n_pruned, splits;
    u64 incumbent;                          // of a pruning search: ~(smallest T_iter so far)
    // searches with a refinement objective: entries of the survivor list, candidates with a feasible partition, refined
    // ones, feasible ones of those, ~(smallest refined T_iter so far)
    u64 n_surv, n_finite, n_refined, n_refined_ok, refined;
};

// A candidate whose lower bound on T_iter did not exceed the smallest plain T_iter when its part was evaluated.
struct __align__(16) Survivor { u64 c; i64 lb, bott; u32 ci, slot; };
constexpr u64 kMaxSurvivors = 1u << 17;

// A pruning search hands its configurations out by their lower bounds, smallest first: buckets of 1/64 octave between 2^20
// and 2^40 ns.
constexpr int kOrderSub = 6, kOrderLow = 20, kOrderBuckets = 20 << kOrderSub;
__device__ __forceinline__ int order_bucket(i64 lb)
{
    if (lb < (1ll << kOrderLow)) return 0;
    const int e = 63 - __clzll(lb);
    const int b = ((e - kOrderLow) << kOrderSub) + (int)((lb >> (e - kOrderSub)) & ((1 << kOrderSub) - 1));
    return b < kOrderBuckets ? b : kOrderBuckets - 1;
}
// smallest bound of bucket b
__device__ __forceinline__ i64 order_edge(int b)
{
    return b == 0 ? 0 : (i64)((1 << kOrderSub) + (b & ((1 << kOrderSub) - 1))) << ((b >> kOrderSub) + kOrderLow - kOrderSub);
}

// What the last block keeps of a pass.
struct TreeReport {
    u64 n_feasible, n_pruned, splits;
    u64 stamp[3];                           // global timer: pass begins, recurrence begins, all done
};

__device__ __forceinline__ u64 global_timer()
{
    u64 t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// items of a class's listed configurations, a part each
__device__ __forceinline__ u32 tree_groups(u32 live, int group) { return group == 1 ? live : (live + (u32)group - 1u) / (u32)group; }

__device__ u32 *tree_state_live(TreeState *state) { return state->live; }
__device__ void tree_stamp_begin(TreeReport *report) { report->stamp[0] = global_timer(); }

struct TreeArgs {
    int N, T, R, n_rc, RW;
    int eta_q;
    unsigned rc_masks[HAP_MAX_RC_MASKS], rc_sup[HAP_MAX_RC_MASKS];
    int rc_order[HAP_MAX_RC_MASKS];
    double tau[HAP_MAX_RC];                 // repeated forward fraction per level (rows that are not combined by level)
    u64 kindbits[4];
    const TreeClass *cls;
    int n_cls;
    u32 p_lo[HAP_MAX_PP + 1];               // first configuration of each class (its list starts there)
    u32 nmap[HAP_MAX_PP + 1];               // mappings of its configurations
    const u32 *live_list, *dead_list;
    int c_lo, c_hi;                         // classes of this launch
    int by_policy;                          // classes may have items of one policy (not where candidates are counted as pruned)
    int launch;                             // which ticket counter; blocks that must be done before the last one reduces
    u32 blocks_total;
    u32 slot_lo;                            // first per-block slot of this launch
    u64 *hist;                              // pruning searches of more than one wave of items: configurations | items << 32 per bucket
    uint4 *order_key, *order;               // by list position: class | bucket << 8, list entry, place in the bucket, items before it
                                            // by order: first item, class | bucket << 8, list entry, -
    unsigned char *rec;
    TreeState *state;
    TreeReport *report;
    TreeResult *res_dev, *res_host;
    const u64 *range_flag;
    PlanSlot *slots;                        // [blocks_total] per-block plan
    i64 *slot_cost; u64 *slot_index;        // [blocks_total]
    Survivor *surv;                         // [max_surv]
    u64 max_surv;
};

// shared-memory accesses by 32-bit address (the scans walk rows with plain address decrements)
__device__ __forceinline__ u32 smem_u32(const void *p) { return (u32)__cvta_generic_to_shared(p); }
#ifdef HAP_CHECKED
__device__ __forceinline__ bool smem_addr_ok(u32 a, u32 bytes)
{
    // the dynamic part lies behind the static variables of the kernel: nothing is addressable past its end
    extern __shared__ __align__(16) unsigned char dyn_smem_base[];
    u32 dyn;
    asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    return HAP_CHECK_OK(0, a % bytes == 0 && a + bytes <= smem_u32(dyn_smem_base) + dyn);
}
#else
__device__ __forceinline__ bool smem_addr_ok(u32, u32) { return true; }
#endif
__device__ __forceinline__ double lds_f64(u32 a)
{
    if (!smem_addr_ok(a, 8)) return 0.0;
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ u32 lds_u32(u32 a)
{
    if (!smem_addr_ok(a, 4)) return 0;
    u32 v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ int lds_u8(u32 a)
{
    if (!smem_addr_ok(a, 1)) return 0;
    u32 v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return (int)v;
}
__device__ __forceinline__ void sts_f64(u32 a, double v)
{
    if (!smem_addr_ok(a, 8)) return;
    asm volatile("st.shared.f64 [%0], %1;" :: "r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void sts_u8(u32 a, u32 v)
{
    if (!smem_addr_ok(a, 1)) return;
    asm volatile("st.shared.u8 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}

constexpr double kTreeInf = 4611686018427387904.0;        // 2^62, the integer INF: above every finite value
constexpr double kTreeBound = 2305843009213693952.0;      // 2^61: every finite value is below

// ------------------------------------------------------------------------------------------------------------------
// per-configuration records
// ------------------------------------------------------------------------------------------------------------------

// the candidates of a configuration none of whose first stages fits any device, results of a pass: by one warp
template <bool F64>
__device__ __forceinline__ void tree_fill_dead(const DpOut &out, u64 c0, u64 c1, int lane)
{
    const u64 a = c0 > out.first ? c0 : out.first, b = c1 < out.first + out.count ? c1 : out.first + out.count;
    if (a >= b) return;
    const i64 inf = F64 ? 0x7ff0000000000000ll : kInf;
    const u64 n = b - a, o = a - out.first;
    for (u64 q = lane; q < n; q += 32) {
        if (out.cost) out.cost[o + q] = inf;
        if (out.bottleneck) out.bottleneck[o + q] = inf;
    }
    const uint4 z = make_uint4(0, 0, 0, 0);
    static_assert(HAP_MAX_PP == 32, "two 16-byte pieces per candidate");
    if (out.partition) for (u64 q = lane; q < 2 * n; q += 32) reinterpret_cast<uint4 *>(out.partition + o * HAP_MAX_PP)[q] = z;
    if (out.recompute) for (u64 q = lane; q < 2 * n; q += 32) reinterpret_cast<uint4 *>(out.recompute + o * HAP_MAX_PP)[q] = z;
}

// What a record is computed from: constants of Eq. 2 and stage coefficients per (configuration, type), or the layer costs
// themselves where a launch before left them (c2v).
struct TreeInput {
    const TypeConst *tcg;
    const i64 *coef;
    const double *coeff;
    const void *c2v;
    double tau[HAP_MAX_RC];                 // whole repeated forward passes per level (rows that are combined by level)
};
constexpr int kTreePrepThreads = 128;
static_assert(kTreePrepThreads == kTreeThreads, "a block of either kernel computes a record");

// One configuration's record in shared memory, by a whole block of kTreePrepThreads threads; `scratch`: shared memory behind it.
// lb_sum (searches that prune; shared memory): the summed layer times at the cheapest type, 0 on entry.
// A chain of dependent steps bounds it, so what needs no layer costs (thresholds, stage constants) stands in front of the first
// barrier beside Eq. 2, and the blocks of 32 layers of a row are scanned side by side.
template <bool F64, bool NL>
__device__ __forceinline__ void tree_record(const DevConst &dc, const TreeClass &cl, u32 p, const hap_pconf &pc, const TreeInput &in,
                                            u64 *range_flag, unsigned char *rec, unsigned char *scratch, i64 *lb_sum)
{
    constexpr int nthreads = kTreePrepThreads, nwarps = kTreePrepThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int N = dc.N, T = dc.T, R = dc.R, n1 = N + 1, PP = pc.PP;
    unsigned all_levels = 0;
    for (int q = 0; q < dc.n_rc; ++q) all_levels |= dc.rc_masks[q];
    const i64 *cfp = in.coef + (size_t)p * T * HAP_NCOEF;                                     // integer coefficients (bytes)
    auto cv = [&](int h, int q) -> double {                                                  // time coefficients
        const size_t at = ((size_t)p * T + h) * HAP_NCOEF + q;
        return F64 ? in.coeff[at] : (double)in.coef[at];
    };

    double2 *sC = reinterpret_cast<double2 *>(scratch);                                       // [T][N] forward, backward
    u32 *w4 = reinterpret_cast<u32 *>(rec + kTreeOffThr);
    i64 *sW = reinterpret_cast<i64 *>(sC + (size_t)T * N);
    i64 *sA = sW + n1;                                                                        // byte prefixes (mixed kinds only)
    uint8_t *sK = reinterpret_cast<uint8_t *>(sA + n1);
    const i64 mx = cfp[HAP_MX], mpre = cfp[HAP_MPRE], mpost = cfp[HAP_MPOST];

    // ---- Eq. 2 for every (device type, layer), with the arithmetic of layer_cost_kernel -------------------------
    if (in.c2v) {                                                                             // a preceding launch left them
        for (int q = tid; q < T * N; q += nthreads) {
            if (F64) sC[q] = reinterpret_cast<const double2 *>(in.c2v)[(size_t)p * T * N + q];
            else { const longlong2 v = reinterpret_cast<const longlong2 *>(in.c2v)[(size_t)p * T * N + q]; sC[q] = make_double2((double)v.x, (double)v.y); }
        }
    } else {
        const size_t row = ((size_t)pc.itp * dc.ncp + pc.icp) * dc.nmb + pc.ib;              // the same table row for every type
        const size_t stride_h = (size_t)dc.ntp * dc.ncp * dc.nmb * N * 2;                     // 16-byte pairs between device types
        const double2 *tab = reinterpret_cast<const double2 *>(dc.tab4) + row * N * 2;
        const TypeConst *tcp = in.tcg + (size_t)p * T;
        bool bad = false;
        int h = tid / N, l = tid - h * N;
        for (int q = tid; q < T * N; q += nthreads) {
            const bool dense = layer_kind(dc, l) == HAP_DENSE;
            const double2 *tp = tab + (size_t)h * stride_h + (size_t)l * 2;
            const double2 tb = __ldg(tp);
            const double2 tf = dense ? make_double2(0.0, 0.0) : __ldg(tp + 1);
            double cf, cb;
            layer_cost_pair(reinterpret_cast<const double2 *>(tcp + h), tb, tf, dense, dc.kappa, cf, cb);
            bad |= !(cf < 6.8719e10) | !(cb < 6.8719e10);                                     // 2^36 ns per layer
            sC[q] = F64 ? make_double2(cf, cb) : make_double2(rint(cf), rint(cb));
            for (l += nthreads; l >= N && h < T; l -= N) ++h;
        }
        if (bad) atomicOr(range_flag, 1ull);
    }
    if (!cl.all_flat) {
        for (int l = tid; l <= N; l += nthreads) sK[l] = (uint8_t)moe_before(dc, l);
        for (int l = tid; l <= N; l += nthreads) {                                            // byte prefixes from the counts of layers per kind
            const i64 nm = moe_before(dc, l), nd = (i64)l - nm;
            sW[l] = nd * cfp[HAP_MW] + nm * cfp[HAP_MW + 1];
            sA[l] = nd * cfp[HAP_MA] + nm * cfp[HAP_MA + 1];
        }
    }
    // ---- stage constants ---------------------------------------------------------------------------------------------
    {
        double *ktab = reinterpret_cast<double *>(rec + kTreeOffKtab), *mi = reinterpret_cast<double *>(rec + kTreeOffMinfo);
        for (int q = tid; q < cl.n_mrows * kTreeMinfo; q += nthreads) {
            const int mr = q / kTreeMinfo, e = q % kTreeMinfo, mk = cl.mask_of_row[mr];
            // the slowest member of a stage of several types (column 7: pre-work, a stage constant)
            const int col = e == 0 ? HAP_SLAT : e <= 2 ? HAP_SBW + e - 1 : e <= 4 ? HAP_OPT + e - 3 : e == 5 ? HAP_KXD : e == 6 ? HAP_KPOST : HAP_KPRE;
            double v = 0.0;
#pragma unroll
            for (int h = 0; h < HAP_MAX_TYPES; ++h)
                if (mk >> h & 1) { const double x = cv(h, col); v = x > v ? x : v; }
            if (e == 5 && !(dc.het_dispatch && (mk & (mk - 1)) != 0)) v = 0.0;
            if (e == 7) ktab[mr] = v;
            else mi[q] = v;
        }
        for (int q = tid; q < T * 6; q += nthreads) ktab[16 + q] = cv(q / 6, HAP_KP2P_INTRA + q % 6);   // intra, inter, cross[0..3]
    }
    // ---- memory thresholds of the depths whose spans are of one kind: the longest length that fits, a byte per level in one word
    // per (depth, type) -------------------------------------------------------------------------------------------------
    {
        const int last = layer_kind(dc, N - 1), len_cap = N - dc.kind_uniform_from;
        const i64 mwk = cfp[HAP_MW + last], mak = cfp[HAP_MA + last], mxk = last == HAP_MOE ? mx : 0;
        for (int q = tid; q < PP * HAP_MAX_TYPES; q += nthreads) {
            const int t = q % HAP_MAX_TYPES, d = q / HAP_MAX_TYPES + 1;
            u32 word = 0;
            if (cl.flat[d] && ((cl.tmask[d] >> t) & 1u)) {
                const i64 room = dc.cap_eff[t] - ((d == 1 ? mpre : 0) + (d == PP ? mpost : 0) + mxk);
                const int inflight = PP - d + 1, most = cl.wmax[d] < len_cap ? cl.wmax[d] : len_cap;
                const i64 ma = (i64)(pc.M < inflight ? pc.M : inflight) * mak;
                const float room_f = (float)room, mw_f = (float)mwk, ma_f = (float)ma * 9.765625e-4f;
                for (int r = 0; r < R; ++r) {
                    if (!((all_levels >> r) & 1u)) continue;
                    // longest length n with n mwk + floor(xi n ma / 1024) <= room: the quotient, then exact steps from there
                    const i64 xm = (i64)dc.xi_q[r] * ma;
                    auto fits = [&](int n) { return (i64)n * mwk + (((i64)n * xm) >> 10) <= room; };
                    const float guess = room_f / (mw_f + (float)dc.xi_q[r] * ma_f);
                    int lo = guess < 0.0f ? 0 : guess > (float)most ? most : (int)guess;             // (a zero divisor: most, or NaN: 0)
                    while (lo < most && fits(lo + 1)) ++lo;
                    while (lo > 0 && !fits(lo)) --lo;
                    word |= (u32)lo << (8 * r);
                }
            }
            w4[q] = word;
        }
    }
    __syncthreads();
    // ---- policies that cannot be feasible: the longest stages that fit do not add up to N (every warp, for itself) ----
    u32 dead = 0;
    {
        u32 longest = 0;                                                                      // of this lane's depth, a byte per level
        if (lane < PP) {
            const uint4 w = reinterpret_cast<const uint4 *>(w4)[lane];                         // (0 where the depth has no such type)
            longest = cl.flat[lane + 1] ? __vmaxu4(__vmaxu4(w.x, w.y), __vmaxu4(w.z, w.w)) : 0x01010101u * cl.wmax[lane + 1];
        }
        for (int pos = 0; pos < dc.n_rc; ++pos) {
            const u32 levels = dc.rc_masks[dc.rc_order[pos]] * 0x00204081u & 0x01010101u;     // a bit per byte
            u32 v = longest & levels * 255u;
            v = __vmaxu4(v, v >> 16);
            const int most = (int)(max(v & 255u, v >> 8 & 255u));
            const int none = __any_sync(0xffffffffu, lane < PP && most == 0);
            if (none || __reduce_add_sync(0xffffffffu, most) < N) dead |= 1u << pos;
        }
    }
    const bool any = dead != (1u << dc.n_rc) - 1u;                                            // else nothing reads the rows
    // ---- prefix rows of the stage time: per row group the slowest member type of every layer, one warp per group ---
    if (any) {
        double *rows = reinterpret_cast<double *>(rec + cl.o_rows);
        // a lane sums two consecutive layers itself, so that 64 layers take one scan (four spill registers)
        constexpr int kRun = 2;
        const int RW = NL ? 2 : R;
        for (int mr = wib; mr < cl.n_mrows; mr += nwarps) {
            const u32 mk = cl.mask_of_row[mr];
            double *row = rows + (size_t)(mr * RW) * n1;
            double preC = 0.0, preF = 0.0;                                                    // fwd + bwd, fwd of the layers before
            for (int base = 0; base < N; base += 32 * kRun) {
                const int run = N - base < 32 * kRun ? (N - base + 31) / 32 : kRun, l0 = base + lane * run;
                double vC[kRun], vF[kRun], sumC = 0.0, sumF = 0.0;
#pragma unroll
                for (int i = 0; i < kRun; ++i)
                    if (i < run) {
                        double F = 0.0, B = 0.0;
                        if (l0 + i < N) {
                            const double2 *c = sC + l0 + i;
                            for (u32 m = mk; m; m &= m - 1) { const double2 q = c[(__ffs((int)m) - 1) * N]; F = q.x > F ? q.x : F; B = q.y > B ? q.y : B; }
                        }
                        sumC += F + B; sumF += F;
                        vC[i] = sumC; vF[i] = sumF;
                    }
                double upC = sumC, upF = sumF;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const double tC = __shfl_up_sync(0xffffffffu, upC, o), tF = __shfl_up_sync(0xffffffffu, upF, o);
                    if (lane >= o) { upC += tC; upF += tF; }
                }
                const double tC = __shfl_up_sync(0xffffffffu, upC, 1), tF = __shfl_up_sync(0xffffffffu, upF, 1);
                const double befC = lane ? preC + tC : preC, befF = lane ? preF + tF : preF;
                double *dst = row + 1 + l0;
#pragma unroll
                for (int i = 0; i < kRun; ++i)
                    if (i < run && l0 + i < N) {
                        const double c = befC + vC[i], f = befF + vF[i];
                        if (NL) { dst[i] = c; dst[n1 + i] = f; }
                        else {
#pragma unroll
                            for (int r = 0; r < HAP_MAX_RC; ++r) if (r < R) dst[r * n1 + i] = c + in.tau[r] * f;
                        }
                    }
                preC += __shfl_sync(0xffffffffu, upC, 31); preF += __shfl_sync(0xffffffffu, upF, 31);
            }
            if (lane < RW) row[lane * n1] = 0.0;
        }
    }
    // ---- lower bound on the summed stage time: the cheapest type's time of every layer (pruning searches) ----------
    if (lb_sum && !F64) {
        i64 lmin = 0;
        for (int l = tid; l < N; l += nthreads) {
            double m = 0.0;
            for (int h = 0; h < T; ++h) { const double2 q = sC[(size_t)h * N + l]; const double v = q.x + q.y; m = (h == 0 || v < m) ? v : m; }
            lmin += (i64)m;
        }
        lmin = warp_sum_i64(lmin);
        if (lane == 0 && lmin) atomicAdd(reinterpret_cast<unsigned long long *>(lb_sum), (unsigned long long)lmin);
    }
    // ---- the other depths' thresholds: per (type, level, end layer) the longest span ending there that fits; feasibility is
    // monotone in the span, so a thread sweeps a segment of end layers with a split pointer that only moves forward
    if (any && !cl.all_flat) {
        uint8_t *nf = rec + cl.o_thr_nf;
        constexpr int kSeg = 4;
        for (int d = 1; d <= PP; ++d) {
            if (cl.flat[d]) continue;
            const int w = (int)cl.nf_w[d], nseg = (w + kSeg - 1) / kSeg;
            for (int e = tid; e < T * R * nseg; e += nthreads) {
                const int seg = e % nseg, q = e / nseg, r = q % R, t = q / R;
                uint8_t *row = nf + cl.nf_off[d] + (size_t)q * w - cl.jlo[d];
                const int j0 = cl.jlo[d] + seg * kSeg;
                int j1 = j0 + kSeg - 1; if (j1 > cl.jhi[d]) j1 = cl.jhi[d];
                const bool want = ((all_levels >> r) & 1u) && ((cl.tmask[d] >> t) & 1u);
                const i64 extra = (d == 1 ? mpre : 0) + (d == PP ? mpost : 0);
                const int inflight = PP - d + 1;
                const i64 mstore = pc.M < inflight ? pc.M : inflight, cap = dc.cap_eff[t], xi = dc.xi_q[r];
                int k = cl.kmin[d];
                for (int j = j0; j <= j1; ++j) {
                    if (!want) { row[j] = 0; continue; }
                    if (k < j - (int)cl.wmax[d]) k = j - (int)cl.wmax[d];
                    const int kcap = (int)cl.kmax[d] < j - 1 ? (int)cl.kmax[d] : j - 1;      // no cell looks at a split beyond this
                    while (k <= kcap && !span_fits(sW, sA, sK, extra, mx, mstore, cap, xi, k, j)) ++k;
                    row[j] = (uint8_t)(k <= kcap ? j - k : 0);
                }
            }
        }
    }
    if (lb_sum) __syncthreads();
    if (tid == 0) {
        TreeHead h{};
        h.offset = pc.offset; h.m1 = (i64)pc.M - 1; h.p = p; h.dead_policies = dead;
        h.S = lb_sum ? *lb_sum : 0;
        h.lb = h.S + h.m1 * ((h.S + PP - 1) / PP);
        *reinterpret_cast<TreeHead *>(rec) = h;
    }
}

// Persistent blocks over the configurations on the classes' lists: entry i of a class's list becomes its record i.  What
// bounds a configuration is a chain of dependent steps (constants, layer costs, scans), hidden by the resident blocks.
constexpr int kTreePrepBlocksPerSm = 9;
template <bool F64, bool NL>
__global__ void __launch_bounds__(kTreePrepThreads, kTreePrepBlocksPerSm)
tree_prep_kernel(const __grid_constant__ DevConst dc, const __grid_constant__ TreeArgs ta, const __grid_constant__ TreeInput in, DpOut out, int search)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ TreeClass cl;
    __shared__ u32 s_first[HAP_MAX_PP + 3];         // entries of the lists before class c; dead ones behind the last class
    __shared__ i64 s_lb;
    const int tid = threadIdx.x, nthreads = kTreePrepThreads, lane = tid & 31, wib = tid >> 5;
    constexpr int nwarps = kTreePrepThreads / 32;
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < 32) {
        // exclusive sums of the list lengths
        const u32 n = tid <= ta.n_cls ? __ldcg(&ta.state->live[tid]) : 0u;
        u32 v = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u32 t = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += t; }
        if (tid <= ta.n_cls) s_first[tid] = v - n;
    }
    if (tid == 0) s_lb = 0;
    __syncthreads();
    const u32 n_live = s_first[ta.n_cls];
    int loaded = -1;
  for (u32 item = blockIdx.x; item < n_live; item += gridDim.x) {
    int ci = 0;
    while (item >= s_first[ci + 1]) ++ci;
    const u32 s_slot = item - s_first[ci];
    const u32 p = __ldcg(ta.live_list + ta.p_lo[ci] + s_slot);
    if (ci != loaded) {
        static_assert(sizeof(TreeClass) % 4 == 0, "copied in words");
        const u32 *src = reinterpret_cast<const u32 *>(ta.cls + ci);
        u32 *dst = reinterpret_cast<u32 *>(&cl);
        for (int q = tid; q < (int)(sizeof(TreeClass) / 4); q += nthreads) dst[q] = src[q];
        loaded = ci;
        __syncthreads();
    }
    const hap_pconf pc = dc.pconf[p];
    tree_record<F64, NL>(dc, cl, p, pc, in, out.range_flag, smem_raw, smem_raw + cl.rec_bytes, search ? &s_lb : nullptr);
    if (tid == 0) {
        const i64 sum = s_lb;
        if (search && out.prune) {
            // candidates are counted as pruned until a part is evaluated
            const u64 c1 = pc.offset + pc.nmap * (u64)dc.n_rc, a = pc.offset > out.first ? pc.offset : out.first;
            const u64 b = c1 < out.first + out.count ? c1 : out.first + out.count;
            if (a < b) atomicAdd(&ta.state->n_pruned, b - a);
            if (ta.order) {
                const int bk = order_bucket(sum + (i64)(pc.M - 1) * ((sum + pc.PP - 1) / pc.PP));
                const u64 before = atomicAdd(ta.hist + bk, (u64)cl.items_per_conf << 32 | 1ull);
                __stcg(ta.order_key + item, make_uint4((u32)ci | (u32)bk << 8, s_slot, (u32)before, (u32)(before >> 32)));
            }
        }
    }
    __syncthreads();
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(smem_raw);
        uint4 *dst = reinterpret_cast<uint4 *>(ta.rec + cl.rec_off + (u64)s_slot * cl.rec_bytes);
        for (u32 q = (u32)tid; q < cl.rec_bytes / 16; q += nthreads) dst[q] = src[q];
    }
    if (tid == 0) s_lb = 0;                             // (added to behind the next record's first barrier)
    __syncthreads();                                    // the shared arrays are free for the next configuration
  }
    if (search) {
        if (!ta.order) return;
        // the last block turns the buckets into the order
        __shared__ u64 s_sum[nwarps];
        __shared__ int s_last;
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(&ta.state->prep_done, 1u) + 1u == gridDim.x;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        constexpr int kPer = kOrderBuckets / kTreePrepThreads;
        static_assert(kPer * kTreePrepThreads == kOrderBuckets, "a whole number of buckets per thread");
        u64 n[kPer], sum = 0;
#pragma unroll
        for (int q = 0; q < kPer; ++q) { n[q] = __ldcg(ta.hist + tid * kPer + q); sum += n[q]; }
        u64 v = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u64 t = __shfl_up_sync(0xffffffffu, v, o); if (lane >= o) v += t; }
        if (lane == 31) s_sum[wib] = v;
        __syncthreads();
        v -= sum;
        for (int q = 0; q < wib; ++q) v += s_sum[q];
#pragma unroll
        for (int q = 0; q < kPer; ++q) { __stcg(ta.hist + tid * kPer + q, v); v += n[q]; }
        if (tid == kTreePrepThreads - 1) __stcg(ta.order + n_live, make_uint4((u32)(v >> 32), 0, 0, 0));
        __syncthreads();
        for (u32 i = (u32)tid; i < n_live; i += nthreads) {
            const uint4 k = __ldcg(ta.order_key + i);
            const u64 base = __ldcg(ta.hist + (k.x >> 8));
            const u32 at = (u32)base + k.z;
            if (HAP_CHECK_OK(4, at < n_live)) __stcg(ta.order + at, make_uint4((u32)(base >> 32) + k.w, k.x, k.y, 0));
        }
        return;
    }
    const u32 n_dead = __ldcg(&ta.state->live[ta.n_cls]);
    // a warp per configuration; one with many candidates is shared by sixteen
    constexpr u32 kSlices = 16;
    constexpr u64 kMany = 1024;
    for (u32 w = blockIdx.x * nwarps + wib; w < n_dead; w += gridDim.x * nwarps) {
        const hap_pconf *pc = dc.pconf + __ldcg(ta.dead_list + w);
        if (pc->nmap * (u64)dc.n_rc <= kMany) tree_fill_dead<F64>(out, pc->offset, pc->offset + pc->nmap * (u64)dc.n_rc, lane);
    }
    u64 most = 0;
    for (int c = 0; c < ta.n_cls; ++c) { const u64 n = ta.nmap[c] * (u64)dc.n_rc; most = n > most ? n : most; }
    if (most <= kMany) return;
    for (u32 q = blockIdx.x * nwarps + wib; q < n_dead * kSlices; q += gridDim.x * nwarps) {
        const hap_pconf *pc = dc.pconf + __ldcg(ta.dead_list + q / kSlices);
        const u64 c0 = pc->offset, n = pc->nmap * (u64)dc.n_rc;
        if (n > kMany) tree_fill_dead<F64>(out, c0 + n * (q % kSlices) / kSlices, c0 + n * (q % kSlices + 1) / kSlices, lane);
    }
}

// ------------------------------------------------------------------------------------------------------------------
// recurrence
// ------------------------------------------------------------------------------------------------------------------

// Levels of a policy at one (depth, capacity type): level of a stage of n layers = number of the bounds below n, longest
// stage that fits at all = nx.  A level that is not allowed or never the lowest that fits has the bound of the one before it.
struct TreeLevels { int b0, b1, b2, nx; };

template <int RK>
__device__ __forceinline__ TreeLevels tree_levels(int R, unsigned rc_mask, u32 len4)
{
    TreeLevels lv;
    if (RK == 2) {                                  // two levels at most (a level that does not exist has length 0)
        const int l0 = (int)(len4 & 255u), l1 = (int)(len4 >> 8 & 255u);
        lv.b0 = rc_mask & 1u ? l0 : -1;
        lv.b1 = lv.b2 = lv.nx = rc_mask & 2u && l1 > lv.b0 ? l1 : lv.b0;
        return lv;
    }
    int run = -1;                                   // (level 0 not allowed: every length is above it)
    auto step = [&](int r) { if ((rc_mask >> r) & 1u) { const int l = (int)((len4 >> (8 * r)) & 255u); run = l > run ? l : run; } return run; };
    lv.b0 = step(0);
    lv.b1 = R > 1 ? step(1) : run;
    lv.b2 = R > 2 ? step(2) : run;
    lv.nx = R > 3 ? step(3) : run;
    return lv;
}

// Stage cost over layers (k, j] with the stage constant, from the row entries of j and k.
//   combined rows (one per level): row[j] - row[k] + K; integer mode adds K to row[j] first, exact in any order
//   NL: rows C (fwd + bwd) and F (fwd): C[j] - C[k] + floor(tau (F[j] - F[k])) + K; the product of an integer below 2^36 N
//       and tau = tau_q / 1024 is exact in a double (the host checks N tau_q < 2^17), adding 2^52 rounding down floors it
template <bool F64, bool NL>
__device__ __forceinline__ double tree_span(double Cj, double Ck, double Fj, double Fk, double K, double tau)
{
    double c = Cj - Ck;
    if (NL) {
        const double t = (Fj - Fk) * tau;
        if (F64) c = c + t;
        else c = c + (__dadd_rd(t, 4503599627370496.0) - 4503599627370496.0);
    }
    return F64 ? c + K : c;
}

// what tree_dp_kernel leaves: results of every candidate, the best candidate, or the candidates that a refinement may make best
constexpr int kTreePass = 0, kTreeSearch = 1, kTreeList = 2;
constexpr int kNever = 1 << 20;
__device__ __forceinline__ int tree_bound(const TreeLevels &lv, int r) { return r == 0 ? lv.b0 : r == 1 ? lv.b1 : r == 2 ? lv.b2 : lv.nx; }

// J consecutive end layers at once: DP[j] = min over stage lengths n in [a, b] of max(prev[j - n], cost), longest stage
// (smallest split) on ties.  The lane holds a window of J entries of prev and of the row, prev[j0 + i - n], that moves by
// one entry per length: two loads serve J splits, and the J minima are independent chains.  Entries of prev outside the
// parent's row are infinite (padding), so nothing is clipped per split; lengths run level by level, the bounds in lv.
// Lengths are taken in pairs without a branch between them: the second of a pair counts where the level has it, and both
// entries a pair moves on by are asked for before its first split, so that their latency lies behind it.  What bounds it is
// instruction issue: eight instructions a split, half of the arithmetic pipe's time for selects.  Pairs against a test and a branch
// per length: 1,024 devices 378 us a pass (393), 256 devices 439 (452).
//   a_prev: address of prev[j0 - a]; a_row0: address of entry 0 of the row group's first row, `stride` bytes per row
template <int J, int RK, bool F64, bool NL, bool COUNT>
__device__ __forceinline__ void tree_scan(const TreeArgs &ta, u32 a_prev, u32 a_row0, u32 stride, int j0, int cnt, int a, int b, const TreeLevels &lv,
                                          double K, double (&best)[J], int (&arg)[J], u32 &splits)
{
    static_assert(J == 1 || J % 2 == 0, "pairs of lengths");
#pragma unroll
    for (int i = 0; i < J; ++i) { best[i] = kTreeBound; arg[i] = 0; }
    const int end = b < lv.nx ? b : lv.nx;
    if (a > end) return;
    int n = a, r = RK == 2 && !NL ? (int)(a > lv.b0) : (a > lv.b0) + (a > lv.b1) + (a > lv.b2);
    int seg = 0;                                                  // last length of the level at hand
    u32 a_row = 0, pa = a_prev, k0 = 8u * (u32)(j0 - a);          // cell 0's entries: prev, and offset in a row
    double tau = 0.0, C[J], F[J], p[J], q[J], f[J];
    // a level begins at length n: rows of the level, the window of length n; cell i's entries lie in place (i - h) mod J
    auto level = [&](const int h) {
        const int top = tree_bound(lv, r);
        seg = RK == 2 && !NL && r ? end : end < top ? end : top;
        a_row = a_row0 + (NL ? 0u : (u32)r * stride);
        if (NL) tau = ta.tau[r];
        const u32 aj = a_row + 8u * (u32)j0;
#pragma unroll
        for (int i = 0; i < J; ++i) {
            const int w = (i - h) & (J - 1);
            C[i] = lds_f64(aj + 8u * i);                          // (entries past the last layer are other words of the block)
            F[i] = NL ? lds_f64(aj + 8u * i + stride) : 0.0;
            p[w] = lds_f64(pa + 8u * i);
            q[w] = lds_f64(a_row + k0 + 8u * i);
            f[w] = NL ? lds_f64(a_row + k0 + 8u * i + stride) : 0.0;
        }
        if (!F64)
#pragma unroll
            for (int i = 0; i < J; ++i) C[i] += K;
    };
    level(0);
    while (true) {
        double last[J];
#pragma unroll
        for (int h = 0; h < J; h += 2) {
            double tp[2], tq[2], tf[2];                           // the entries below cell 0's
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                tp[s] = lds_f64(pa - 8u * (s + 1));
                tq[s] = lds_f64(a_row + k0 - 8u * (s + 1));
                tf[s] = NL ? lds_f64(a_row + k0 + stride - 8u * (s + 1)) : 0.0;
            }
            const bool both = n < seg;
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int i = 0; i < J; ++i) {
                    const int w = (i - s - h) & (J - 1);
                    const bool below = i < s;
                    const double c = tree_span<F64, NL>(C[i], below ? tq[0] : q[w], F[i], below ? tf[0] : f[w], K, tau);
                    const double x = below ? tp[0] : p[w], v = x > c ? x : c;
                    if (v <= best[i] && (s == 0 || both)) { best[i] = v; arg[i] = n + s; }
                    last[i] = c;
                    if (COUNT) splits += i < cnt && (s == 0 || both) ? 1u : 0u;
                }
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int w = (-1 - s - h) & (J - 1);
                p[w] = tp[s]; q[w] = tq[s];
                if (NL) f[w] = tf[s];
            }
            n += 2; pa -= 16u; k0 -= 16u;
            if (n > seg) {
                if (seg >= end) return;
                const u32 back = 8u * (u32)(n - seg - 1);         // to the first length of the next level
                n = seg + 1; pa += back; k0 += back;
                do ++r; while (RK != 2 && n > tree_bound(lv, r));
                level((h + 2) & (J - 1));
#pragma unroll
                for (int i = 0; i < J; ++i) last[i] = 0.0;
            }
        }
        // costs grow with the length (the host sends policies whose higher levels repeat less forward work to the general
        // kernel): once they exceed all the minima, longer stages cannot win
        bool over = true;
#pragma unroll
        for (int i = 0; i < J; ++i) over = over && last[i] > best[i];
        if (over) return;
    }
}

// The last block of a pass (all of its threads): leaves the report and, for a search, the winner; clears the counters.
template <int THREADS, bool SEARCH, bool F64>
__device__ __forceinline__ void tree_finish(const TreeArgs &ta, const DevConst &dc, u64 n_feasible, u64 n_pruned, u64 again, i64 *s_cost, u64 *s_index, u32 *s_item)
{
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const i64 inf_bits = F64 ? 0x7ff0000000000000ll : kInf;
    const int n_rc = ta.n_rc;
    if (tid == 0) {
        ta.report->n_feasible = n_feasible; ta.report->n_pruned = n_pruned;
        ta.report->splits = __ldcg(&ta.state->splits);
        ta.report->stamp[2] = global_timer();
    }
    __syncthreads();
    static_assert(sizeof(TreeState) % 4 == 0, "cleared in words");
    for (int q = tid; q < (int)(sizeof(TreeState) / 4); q += THREADS) reinterpret_cast<u32 *>(ta.state)[q] = 0;
    if (!SEARCH || !ta.res_dev) return;
    i64 bc = inf_bits; u64 bi = ~0ull; u32 at = 0;
    for (u32 q = (u32)tid; q < ta.blocks_total; q += THREADS) {
        const i64 v = __ldcg(ta.slot_cost + q); const u64 ix = __ldcg(ta.slot_index + q);
        if (v < bc || (v == bc && ix < bi)) { bc = v; bi = ix; at = q; }
    }
    const u64 mine = bi;
    const i64 mine_c = bc;
    warp_argmin(bc, bi);
    if (lane == 0) { s_cost[wib] = bc; s_index[wib] = bi; }
    __syncthreads();
    bc = s_cost[0]; bi = s_index[0];
    for (int q = 1; q < THREADS / 32; ++q) if (s_cost[q] < bc || (s_cost[q] == bc && s_index[q] < bi)) { bc = s_cost[q]; bi = s_index[q]; }
    // the winner's slot: (cost, index) pairs are distinct unless nothing is feasible
    if (bc < inf_bits && mine == bi && mine_c == bc) *s_item = at;
    __syncthreads();
    if (wib != 0) return;
    // (the slot names the winner's configuration: a search for it in the table is a chain of a dozen loads, 6 us)
    TreeResult *w = ta.res_host ? ta.res_host : ta.res_dev;
    if (lane == 0) {
        w->range_flag = __ldcg(ta.range_flag);
        w->n_feasible = n_feasible; w->n_pruned = n_pruned;
        w->cost = bc; w->index = bi; w->again = again;
        for (int q = 0; q < 3; ++q) w->stamp[q] = __ldcg(&ta.report->stamp[q]);
    }
    if (bc < inf_bits) {
        const PlanSlot *ps = ta.slots + *s_item;
        const u64 p = __ldcg(&ps->p);
        const hap_pconf pc = dc.pconf[p];
        const u64 loc = bi - pc.offset, map_idx = loc / (u64)n_rc;
        const StageMap sm = decode_stage(dc, pc, map_idx, lane);
        if (lane == 0) {
            w->pconf = (u32)p; w->rc_mask = ta.rc_masks[loc - map_idx * (u64)n_rc];
            w->bott = __ldcg(&ps->bott); w->T_pipe = __ldcg(&ps->T_pipe); w->T_sync = __ldcg(&ps->T_sync); w->T_opt = __ldcg(&ps->T_opt);
        }
        w->mask[lane] = lane < pc.PP ? (uint8_t)sm.mask : 0;
        w->n[lane] = lane < pc.PP ? __ldcg(ps->n + lane) : 0;
        w->r[lane] = lane < pc.PP ? __ldcg(ps->r + lane) : 0;
    }
    __threadfence_system();
}

// GROUP: items of several configurations (TreeClass::group), in a form of its own because the record's place in shared memory is then
// an address in a register: 2 % of a pass whose classes have no use for it.
template <int MODE, bool F64, int RK, bool NL, bool COUNT, int BLOCKS = kTreeBlocksPerSm, bool GROUP = false>
__global__ void __launch_bounds__(kTreeThreads, BLOCKS)
tree_dp_kernel(const TreeArgs ta, const DevConst dc, DpOut out)
{
    constexpr bool SEARCH = MODE != kTreePass, LIST = MODE == kTreeList;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ u32 s_item, s_unit, s_total[HAP_MAX_PP + 2];
    __shared__ uint4 s_entry;
    __shared__ double s_zero[kTreeAhead + 2 * kTreePad + 1];    // the row before the first stage: 0 at layer 0
    __shared__ i64 s_cost[kTreeWarps];
    __shared__ u64 s_index[kTreeWarps];
    __shared__ int s_last, s_pos[2];
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int N = ta.N, R = ta.R, n1 = N + 1, n_rc = ta.n_rc, RW = NL ? 2 : R;
    const int kind_last = layer_kind(dc, N - 1);
    const i64 inf_bits = F64 ? 0x7ff0000000000000ll : kInf;
    const double dInfOut = F64 ? __longlong_as_double(0x7ff0000000000000ll) : kTreeInf;

    i64 best_cost = inf_bits;               // (non-negative doubles order like their bit patterns)
    u64 best_index = ~0ull;
    u32 n_feas = 0, splits = 0;
    u64 plan_n[2][HAP_MAX_PP / 8], plan_r[2][HAP_MAX_PP / 8];    // the plan at hand and the plan of the thread's best candidate
    i64 plan_val[2][5];
    u32 plan_cur = 0;

    // A second launch of the same pass starts once every block of the first is running, i.e. past the first one's wait for
    // the records; it waits for the first launch itself only at its end.
    if (ta.launch == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const bool ordered = SEARCH && !F64 && ta.order != nullptr;
    if (tid == 0) {
        if (blockIdx.x == 0 && ta.launch == 0) ta.report->stamp[1] = global_timer();
        for (int q = 0; q < kTreeAhead + 2 * kTreePad + 1; ++q) s_zero[q] = q == kTreeAhead + kTreePad ? 0.0 : kTreeInf;
        u32 t = 0;                          // items before class c (in order of the bounds: configurations)
        for (int c = ta.c_lo; c < ta.c_hi; ++c) {
            s_total[c - ta.c_lo] = t;
            const u32 live = __ldcg(&ta.state->live[c]);
            t += ordered ? live : tree_groups(live, GROUP ? ta.cls[c].group : 1) * (u32)(ta.cls[c].items_per_conf * (ta.by_policy ? ta.cls[c].policy_items : 1));
        }
        s_total[ta.c_hi - ta.c_lo] = t;
        s_item = blockIdx.x;
    }
    __syncthreads();
    const u32 a_zero = smem_u32(s_zero), n_total = s_total[ta.c_hi - ta.c_lo];
    // in order of the bounds: the configuration an item belongs to, by one warp; none left where the bucket of the next one
    // lies above the incumbent, like those of all that follow
    auto locate = [&](u32 item) {
        u32 lo = 0, hi = n_total + 1;       // order[lo].x <= item; order[hi].x > item, or hi is past the last one
        while (hi - lo > 1) {
            const u32 step = (hi - lo + 31) / 32, at = lo + (u32)lane * step;
            const u32 n = __popc(__ballot_sync(0xffffffffu, at < hi && __ldcg(&ta.order[at].x) <= item));
            lo += (n - 1) * step;
            hi = lo + step < hi ? lo + step : hi;
        }
        const uint4 en = __ldcg(ta.order + lo);
        if (lane == 0) {
            const bool none = lo >= n_total || (u64)order_edge((int)(en.y >> 8)) > ~*reinterpret_cast<volatile const u64 *>(&ta.state->incumbent);
            s_item = none ? ~0u : item;
            s_entry = en;
        }
    };
    if (ordered) {
        __syncthreads();
        if (wib == 0) locate(blockIdx.x);
        __syncthreads();
    }

    while (true) {
        const u32 item = s_item;
        if (item >= (ordered ? ~0u : n_total)) break;
        u32 next_item = 0;
        if (tid == 0) next_item = atomicAdd(&ta.state->ticket[ta.launch], 1u) + gridDim.x;
        int ci = ta.c_lo;
        if (ordered) ci = (int)(s_entry.y & 255u);
        else while (item >= s_total[ci + 1 - ta.c_lo]) ++ci;
        const TreeClass *cl = ta.cls + ci;
        const u32 ipc = (u32)cl->items_per_conf;
        u32 local = ordered ? item - s_entry.x : item - s_total[ci - ta.c_lo];
        {
            int lo = 0, hi = n_rc;
            if (!ordered && ta.by_policy && cl->policy_items > 1) {
                // items of one policy each: the first policy's come first (they take longest)
                const u32 items = tree_groups(__ldcg(&ta.state->live[ci]), GROUP ? cl->group : 1) * ipc;
                lo = (int)(local / items); hi = lo + 1; local -= (u32)lo * items;
            }
            if (tid == 0) { s_pos[0] = lo; s_pos[1] = hi; }     // (in shared memory: registers are short below)
        }
        // (quotients by the inverse: one too large at most; divisions took a tenth of an item's instructions)
        u32 conf = ipc == 1 ? local : __umulhi(local, cl->ipc_inverse), sub = local - conf * ipc;
        if ((int)sub < 0) { --conf; sub += ipc; }
        u32 n_rec = 1;                                          // configurations of the item: their records follow one another
        if (ordered) conf = s_entry.z;
        else if (GROUP) {
            conf *= (u32)cl->group;
            n_rec = min((u32)cl->group, __ldcg(&ta.state->live[ci]) - conf);
        }
        const u32 n_parts = (u32)cl->n_parts, per = ipc == 1 ? n_parts : __umulhi(n_parts, cl->ipc_inverse), more = n_parts - per * ipc;
        const u32 part0 = sub * per + (sub < more ? sub : more), part1 = part0 + per + (sub < more ? 1u : 0u);
        const u32 rec_bytes = cl->rec_bytes;
        const int PP = cl->PP;
        // the configuration's record into shared memory
        if (tid == 0) s_unit = 0;
        {
            const unsigned char *src = ta.rec + cl->rec_off + (u64)conf * rec_bytes;
            const u32 dst = smem_u32(smem_raw);
            for (u32 q = (u32)tid * 16u; q < n_rec * rec_bytes; q += kTreeThreads * 16u)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst + q), "l"(src + q) : "memory");
            asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const u32 slice_bytes = (cl->buf_cells[0] + cl->buf_cells[1]) * 8u + cl->ch_bytes;
        const u32 a_slice = smem_u32(smem_raw) + (GROUP ? (u32)cl->group : 1u) * rec_bytes + (u32)wib * slice_bytes;
        const u32 a_buf[2] = {a_slice, a_slice + cl->buf_cells[0] * 8u};
        const u32 a_ch = a_buf[1] + cl->buf_cells[1] * 8u;
        const bool all_flat = cl->all_flat != 0;
        // sync and optimizer terms from the longest stage per row group, of the stages behind the last change of kind (256 devices with
        // a dense first layer, partitions: 412 us against 419 with every stage's own terms)
        const bool packed = cl->n_mrows <= 4;
        const u32 row_stride = (u32)n1 * 8u, row_group = (u32)RW * row_stride;

        while (true) {
            u32 u = 0;
            if (lane == 0) u = atomicAdd(&s_unit, 1u);
            u = __shfl_sync(0xffffffffu, u, 0);
            if (u >= n_rec * (part1 - part0)) break;
            const unsigned char *rec = smem_raw;
            if (GROUP)
                for (; u >= part1 - part0; u -= part1 - part0) rec += rec_bytes;
            const TreePart *pt = cl->parts + part0 + u;
            const TreeHead *hd = reinterpret_cast<const TreeHead *>(rec);
            const u32 a_rec = smem_u32(rec), a_rows = a_rec + cl->o_rows;
            const u32 nmap = pt->nmap;
            const u64 c_lo = hd->offset + (u64)pt->m_lo * (u64)n_rc, c_hi = c_lo + (u64)nmap * (u64)n_rc;
            const u64 w_lo = out.first, w_hi = out.first + out.count;
            if (c_hi <= w_lo || c_lo >= w_hi) continue;
            const bool whole = c_lo >= w_lo && c_hi <= w_hi;
            if (SEARCH && out.prune) {
                // a part whose configuration's lower bound exceeds the incumbent cannot hold the minimum (strict); one lane
                // reads the moving incumbent and the warp follows it as a whole
                int skip = 0;
                if (lane == 0) skip = (u64)hd->lb > ~*reinterpret_cast<volatile const u64 *>(&ta.state->incumbent);
                skip = __shfl_sync(0xffffffffu, skip, 0);
                if (skip) continue;
                if (lane == 0) atomicAdd(&ta.state->n_pruned, 0ull - ((c_hi < w_hi ? c_hi : w_hi) - (c_lo > w_lo ? c_lo : w_lo)));
            }
            unsigned without_plan = 0;          // positions in rc_order under which no mapping was feasible
            const TreeTask *tasks = pt->tasks + lane;
            // what the last stages and the way back read first, behind the rows
            if (lane < PP) asm volatile("prefetch.global.L1 [%0];" :: "l"(pt->path + (size_t)lane * nmap));
            if (lane == 0) asm volatile("prefetch.global.L1 [%0];" :: "l"(pt->leaf));

            for (int pos = s_pos[0]; pos < s_pos[1]; ++pos) {
                const int rc_idx = ta.rc_order[pos];
                const unsigned rc_mask = ta.rc_masks[rc_idx];
                bool dead = ((hd->dead_policies >> pos) & 1u) || (ta.rc_sup[pos] & without_plan) != 0;
                // levels at a depth whose spans mix layer kinds: per end layer
                auto nf_levels = [&](int d, int capt, int j) {
                    const u32 w = cl->nf_w[d], a = a_rec + cl->o_thr_nf + cl->nf_off[d] + (u32)(capt * R) * w + (u32)(j - (int)cl->jlo[d]);
                    u32 len4 = 0;
                    for (int r = 0; r < R; ++r) len4 |= (u32)lds_u8(a + (u32)r * w) << (8 * r);
                    return tree_levels<NL ? 4 : RK>(R, rc_mask, len4);
                };

                // ---- rows of the tree, depth by depth ------------------------------------------------------
                if (!dead && PP > 1) {
                    const TreeTask *next = tasks;
                    TreeTask nxt = __ldg(next);
                    u32 a_prv = a_zero, a_cur = a_buf[1];
                    bool alive = false;
                    for (u32 it = pt->n_iter; it > 0; --it) {
                        const TreeTask t = nxt;
                        next += 32;
                        nxt = __ldg(next);                                          // comes in behind this scan
                        const int j0 = (int)(t.y & 255u), a = (int)(t.y >> 8) & 255, b = (int)(t.y >> 16) & 255, cnt = (int)(t.y >> 24) & 7;
                        const u32 kidx = t.z & 255u, mrow = (t.z >> 8) & 255u, thr = t.z >> 16, slot = t.x >> 16, choice = t.w & 0xffffu;
                        const double K = lds_f64(a_rec + kTreeOffKtab + 8u * kidx);
                        const u32 a_row0 = a_rows + mrow * row_group;
                        const u32 a_prev = a_prv + 8u * (t.x & 0xffffu), a_out = a_cur + 8u * slot, a_cho = a_ch + choice;
                        (void)HAP_CHECK_OK(0, a > b || a_prev >= a_prv + 8u * (u32)(b - a + 2));      // the lowest entry a scan reads
                        auto put = [&](int i, double v, int n) {
                            if (HAP_CHECK_OK(1, slot + i < cl->buf_cells[a_cur == a_buf[1]])) sts_f64(a_out + 8u * i, n ? v : kTreeInf);
                            if (HAP_CHECK_OK(2, choice + i < cl->ch_bytes)) sts_u8(a_cho + i, (u32)n);
                            alive |= n != 0;
                        };
                        TreeLevels lv;
                        if (t.w & kTaskByLayer) lv = nf_levels((int)(thr >> 2) + 1, (int)(thr & 3u), j0);      // (one end layer a task)
                        else lv = tree_levels<NL ? 4 : RK>(R, rc_mask, lds_u32(a_rec + kTreeOffThr + 4u * thr));
                        auto scan = [&](auto width, int h) {
                            constexpr int J = decltype(width)::value;
                            double best[J];
                            int arg[J];
                            tree_scan<J, RK, F64, NL, COUNT>(ta, a_prev + 8u * h, a_row0, row_stride, j0 + h, cnt - h, a, b, lv, K, best, arg, splits);
#pragma unroll
                            for (int i = 0; i < J; ++i)
                                if (h + i < cnt) put(h + i, best[i], arg[i]);
                        };
                        if (t.w & (1u << 16)) scan(TreeWidth<1>(), 0);
                        else if (t.w & (2u << 16)) scan(TreeWidth<2>(), 0);
                        else if (!NL) scan(TreeWidth<kTreeJ>(), 0);
                        else {                                                      // (a window of two rows a level: two halves)
                            scan(TreeWidth<kTreeJ / 2>(), 0);
                            if (cnt > kTreeJ / 2) scan(TreeWidth<kTreeJ / 2>(), kTreeJ / 2);
                        }
                        if (t.y & (1u << 27)) {                                     // the row's padding
#pragma unroll
                            for (int i = 1; i <= kTreePad; ++i) sts_f64(a_out - 8u * i, kTreeInf);
                        }
                        if (t.y & (1u << 28)) {
#pragma unroll
                            for (int i = 0; i < kTreePad; ++i) sts_f64(a_out + 8u * (cnt + i), kTreeInf);
                        }
                        if (t.w & kTaskEnds) {
                            __syncwarp();
                            if (!__any_sync(0xffffffffu, alive)) { dead = true; break; }          // no cell of this depth is finite: nothing below is
                            alive = false;
                            a_prv = a_cur; a_cur = a_buf[0] + a_buf[1] - a_cur;
                        }
                    }
                }
                // ---- one lane per mapping: cell (PP, N), walk back, Eq. 4 ----------------------------------------
                bool any_plan = false;
                const u32 a_last = PP == 1 ? a_zero : a_buf[(PP - 1) & 1];
                auto leaf = [&](u32 m, double &bott) {
                    const u64 c = c_lo + (u64)m * (u64)n_rc + (u64)rc_idx;
                    if (c < w_lo || c >= w_hi) return;
                    const u64 o = c - w_lo;
                    if (!HAP_CHECK_OK(3, o < out.count)) return;
                    int n = 0;
                    const u32 *path = pt->path + m;
                    u32 pw = 0;
                    if (!dead) {
                        pw = __ldg(path + (size_t)(PP - 1) * nmap);
                        const u32 lf = __ldg(pt->leaf + m);
                        const int a = (int)(lf & 255u), b = (int)(lf >> 8) & 255;
                        const u32 kidx = (pw >> 20) & 63u, mrow = (pw >> 26) & 15u;
                        const int capt = (int)(pw >> 30);
                        if (a <= b) {
                            const double K = lds_f64(a_rec + kTreeOffKtab + 8u * kidx) + lds_f64(a_rec + kTreeOffMinfo + (mrow * kTreeMinfo + 6) * 8u);
                            const TreeLevels lv = all_flat || cl->flat[PP] ? tree_levels<NL ? 4 : RK>(R, rc_mask, lds_u32(a_rec + kTreeOffThr + 4u * (u32)((PP - 1) * HAP_MAX_TYPES + capt)))
                                                                           : nf_levels(PP, capt, N);
                            (void)HAP_CHECK_OK(0, (pw & 0xfffffu) >= (u32)(b - a + 2));
                            double best[1];
                            int arg[1];
                            tree_scan<1, RK, F64, NL, COUNT>(ta, a_last + 8u * (pw & 0xfffffu), a_rows + mrow * row_group, row_stride, N, 1, a, b, lv, K,
                                                             best, arg, splits);
                            bott = best[0]; n = arg[0];
                        }
                    }
                    if (n == 0) {
                        bott = kTreeInf;
                        if (!SEARCH) {
                            if (out.cost) out.cost[o] = inf_bits;
                            if (out.bottleneck) out.bottleneck[o] = inf_bits;
                            const uint4 z = make_uint4(0, 0, 0, 0);
                            if (out.partition) { uint4 *d = reinterpret_cast<uint4 *>(out.partition + o * HAP_MAX_PP); d[0] = z; d[1] = z; }
                            if (out.recompute) { uint4 *d = reinterpret_cast<uint4 *>(out.recompute + o * HAP_MAX_PP); d[0] = z; d[1] = z; }
                        }
                        return;
                    }
                    double sum = 0.0, t_sync = 0.0, t_opt = 0.0, het = 0.0;
                    u32 most = 0;                                                  // per row group the longest stage, a byte each (packed)
                    u64 acc_n = 0, acc_r = 0;
                    const bool want_plan = LIST ? false : SEARCH ? true : (out.partition != nullptr || out.recompute != nullptr);
                    int b = N;
                    for (int d = PP; d >= 1; --d) {
                        const u32 pn = d > 1 ? __ldg(path + (size_t)(d - 2) * nmap) : 0u;       // the stage before: asked for early
                        const int kidx = (int)(pw >> 20) & 63, capt = (int)(pw >> 30);
                        const u32 mrow = (pw >> 26) & 15u;
                        if (!HAP_CHECK_OK(5, n >= 1 && n <= b && b <= N)) break;
                        double K = lds_f64(a_rec + kTreeOffKtab + 8u * (u32)kidx);
                        const u32 a_mi = a_rec + kTreeOffMinfo + mrow * (kTreeMinfo * 8u);
                        if (d == PP) K += lds_f64(a_mi + 48u);
                        // lowest allowed level whose longest stage holds n layers
                        const TreeLevels lv = all_flat || cl->flat[d] ? tree_levels<NL ? 4 : RK>(R, rc_mask, lds_u32(a_rec + kTreeOffThr + 4u * (u32)((d - 1) * HAP_MAX_TYPES + capt)))
                                                                      : nf_levels(d, capt, b);
                        const int r = RK == 2 && !NL ? (int)(n > lv.b0) : (n > lv.b0) + (n > lv.b1) + (n > lv.b2);
                        const u32 a_row = a_rows + mrow * row_group + (NL ? 0u : (u32)r * row_stride);
                        double cst = lds_f64(a_row + 8u * (u32)b) - lds_f64(a_row + 8u * (u32)(b - n));
                        if (NL) {
                            const double t = (lds_f64(a_row + 8u * (u32)(n1 + b)) - lds_f64(a_row + 8u * (u32)(n1 + b - n))) * ta.tau[r];
                            cst += F64 ? t : __dadd_rd(t, 4503599627370496.0) - 4503599627370496.0;
                        }
                        cst += K;
                        sum += cst;
                        int n_moe = n;
                        if (packed && b - n >= dc.kind_uniform_from) {         // their terms follow below
                            most = __vmaxu4(most, (u32)n << (8u * mrow));
                            n_moe = kind_last == HAP_MOE ? n : 0;
                        } else {
                            // (behind the last change of kind the count needs no look at the layers)
                            n_moe = b - n >= dc.kind_uniform_from ? (kind_last == HAP_MOE ? n : 0) : moe_before(dc, b) - moe_before(dc, b - n);
                            const double dm = (double)n_moe, dd = (double)(n - n_moe);
                            const double sy = lds_f64(a_mi) + dd * lds_f64(a_mi + 8u) + dm * lds_f64(a_mi + 16u);
                            const double op = dd * lds_f64(a_mi + 24u) + dm * lds_f64(a_mi + 32u);
                            t_sync = sy > t_sync ? sy : t_sync; t_opt = op > t_opt ? op : t_opt;
                        }
                        if (ta.eta_q > 0) {                                    // Pruning 3: cross-type transfer into the stage; dispatch of a mixed-type stage
                            if (d > 1 && (kidx - 16) % 6 >= 2) het += lds_f64(a_rec + kTreeOffKtab + 8u * (u32)kidx);
                            het += (double)n_moe * lds_f64(a_mi + 40u);
                        }
                        if (want_plan) {
                            // layers and levels of eight stages in a word, stage d in byte (d - 1) & 7
                            acc_n = (acc_n << 8) | (u64)(u32)n; acc_r = (acc_r << 8) | (u64)(u32)r;
                            if (((d - 1) & 7) == 0) {
                                const int w = (d - 1) >> 3;
                                if (SEARCH) { plan_n[plan_cur][w] = acc_n; plan_r[plan_cur][w] = acc_r; }
                                else {
                                    if (out.partition) reinterpret_cast<u64 *>(out.partition + o * HAP_MAX_PP)[w] = acc_n;
                                    if (out.recompute) reinterpret_cast<u64 *>(out.recompute + o * HAP_MAX_PP)[w] = acc_r;
                                }
                                acc_n = 0; acc_r = 0;
                            }
                        }
                        b -= n;
                        pw = pn;
                        if (d > 1) {
                            const u32 at = (pw & 0xfffffu) + (u32)b - 256u;
                            if (!HAP_CHECK_OK(2, at < cl->ch_bytes)) break;
                            n = lds_u8(a_ch + at);
                        }
                    }
                    if (packed)
                        for (int g = 0; g < cl->n_mrows; ++g) {                // the terms grow with the stage: the longest one of a row group counts
                            const u32 len = (most >> (8 * g)) & 255u;
                            const u32 a_mi = a_rec + kTreeOffMinfo + (u32)(g * kTreeMinfo) * 8u;
                            const double dn = (double)len;
                            const double sy = lds_f64(a_mi) + dn * lds_f64(a_mi + 8u + 8u * (u32)kind_last), op = dn * lds_f64(a_mi + 24u + 8u * (u32)kind_last);
                            if (len) { t_sync = sy > t_sync ? sy : t_sync; t_opt = op > t_opt ? op : t_opt; }
                        }
                    const double mxc = bott;                                   // the largest stage cost is the cell's value
                    i64 T_iter, T_pipe;                                        // (bit patterns in fp64 mode)
                    bool keep = true;
                    if (F64) {
                        const double tp = sum + (double)hd->m1 * mxc;
                        if (ta.eta_q > 0 && het * (double)PP * 1024.0 > (double)ta.eta_q * sum) keep = false;
                        T_pipe = __double_as_longlong(keep ? tp : dInfOut);
                        T_iter = __double_as_longlong(keep ? tp + t_sync + t_opt : dInfOut);
                    } else {
                        const i64 s = (i64)sum;
                        T_pipe = s + hd->m1 * (i64)mxc;
                        T_iter = T_pipe + (i64)t_sync + (i64)t_opt;
                        if (ta.eta_q > 0 && (i64)het * (i64)PP * 1024 > (i64)ta.eta_q * s) { keep = false; T_iter = kInf; T_pipe = kInf; }   // Pruning 3
                    }
                    const i64 bott_bits = F64 ? __double_as_longlong(bott) : (i64)bott;
                    if (SEARCH) {
                        if (LIST) { n_feas++; any_plan = true; }               // (a refined partition may pass Pruning 3 where this one does not)
                        else if (keep) { n_feas++; any_plan = true; }
                        if (T_iter < best_cost || (T_iter == best_cost && c < best_index)) {
                            best_cost = T_iter; best_index = c;
                            plan_val[plan_cur][0] = bott_bits; plan_val[plan_cur][1] = T_pipe;
                            plan_val[plan_cur][2] = F64 ? __double_as_longlong(t_sync) : (i64)t_sync;
                            plan_val[plan_cur][3] = F64 ? __double_as_longlong(t_opt) : (i64)t_opt;
                            plan_val[plan_cur][4] = (i64)hd->p;
                            plan_cur ^= 1u;                                    // the place just filled is kept, the other one is written next
                        }
                    } else {
                        any_plan = true;
                        if (out.cost) out.cost[o] = T_iter;
                        if (out.bottleneck) out.bottleneck[o] = bott_bits;
                        for (int w = keep ? (PP + 7) >> 3 : 0; w < HAP_MAX_PP / 8; ++w) {
                            if (out.partition) reinterpret_cast<u64 *>(out.partition + o * HAP_MAX_PP)[w] = 0;
                            if (out.recompute) reinterpret_cast<u64 *>(out.recompute + o * HAP_MAX_PP)[w] = 0;
                        }
                    }
                };
                if (LIST) {
                    for (u32 m0 = 0; m0 < nmap; m0 += 32u) {
                        const u32 m = m0 + (u32)lane;
                        double bott = kTreeInf;
                        if (m < nmap) leaf(m, bott);
                        __syncwarp();
                        if (!__any_sync(0xffffffffu, bott < kTreeBound)) continue;
                        // the incumbent moves first, then the candidates that it leaves are listed
                        i64 v = best_cost;
#pragma unroll
                        for (int s = 16; s > 0; s >>= 1) { const i64 x = __shfl_xor_sync(0xffffffffu, v, s); v = x < v ? x : v; }
                        if (lane == 0) { const u64 was = ~atomicMax(&ta.state->incumbent, v < inf_bits ? ~(u64)v : 0ull); v = was < (u64)v ? (i64)was : v; }
                        v = shfl_i64(v, 0);
                        const i64 lb = bott < kTreeBound ? hd->S + hd->m1 * (i64)bott : kInf;
                        const bool keep = bott < kTreeBound && lb <= v;
                        const u32 kept = __ballot_sync(0xffffffffu, keep);
                        u64 at = 0;
                        if (lane == 0 && kept) at = atomicAdd(&ta.state->n_surv, (u64)__popc(kept));
                        at = (u64)shfl_i64((i64)at, 0) + (u64)__popc(kept & ((1u << lane) - 1u));
                        if (keep && at < ta.max_surv) {
                            Survivor sv;
                            sv.c = c_lo + (u64)m * (u64)n_rc + (u64)rc_idx; sv.lb = lb; sv.bott = (i64)bott; sv.ci = (u32)ci; sv.slot = conf;
                            ta.surv[at] = sv;
                        }
                    }
                } else
                    for (u32 m = (u32)lane; m < nmap; m += 32u) { double bott = kTreeInf; leaf(m, bott); }
                // (also keeps the next policy from overwriting rows and choices that other lanes still read)
                const int plan = __any_sync(0xffffffffu, any_plan);
                // a policy under which none of the part's mappings has a feasible partition settles its subsets
                if (!plan && whole && ta.eta_q <= 0) without_plan |= 1u << pos;
                __syncwarp();
            }
            if (SEARCH && !LIST && out.prune) {
                // the incumbent moves on after every part
                i64 bc = best_cost;
#pragma unroll
                for (int s = 16; s > 0; s >>= 1) { const i64 v = __shfl_xor_sync(0xffffffffu, bc, s); bc = v < bc ? v : bc; }
                if (lane == 0 && bc < inf_bits) atomicMax(&ta.state->incumbent, ~(u64)bc);
            }
        }
        __syncthreads();                        // every warp is done with the item's records
        if (ordered) { if (wib == 0) locate(__shfl_sync(0xffffffffu, next_item, 0)); }
        else if (tid == 0) s_item = next_item;
        __syncthreads();
    }

    if (COUNT) {
        const u64 s = (u64)warp_sum_i64((i64)splits);
        if (lane == 0 && s) atomicAdd(&ta.state->splits, s);
    }
    if (LIST) {
        const u64 nf = (u64)warp_sum_i64((i64)n_feas);
        if (lane == 0 && nf) atomicAdd(&ta.state->n_finite, nf);
        return;                             // the refinement follows
    }
    if (SEARCH) {
        const u64 nf = (u64)warp_sum_i64((i64)n_feas);
        if (lane == 0 && nf) atomicAdd(&ta.state->n_feasible, nf);
        i64 bc = best_cost; u64 bi = best_index;
        warp_argmin(bc, bi);
        if (lane == 0) { s_cost[wib] = bc; s_index[wib] = bi; }
        __syncthreads();
        bc = s_cost[0]; bi = s_index[0];
        for (int q = 1; q < kTreeWarps; ++q) if (s_cost[q] < bc || (s_cost[q] == bc && s_index[q] < bi)) { bc = s_cost[q]; bi = s_index[q]; }
        const u32 slot = ta.slot_lo + blockIdx.x;
        if (tid == 0) { ta.slot_cost[slot] = bc; ta.slot_index[slot] = bi; }
        if (bc < inf_bits && best_index == bi) {
            // the thread that evaluated the block's best candidate leaves its plan
            PlanSlot *ps = ta.slots + slot;
            const u32 kp = plan_cur ^ 1u;
            ps->bott = plan_val[kp][0]; ps->T_pipe = plan_val[kp][1]; ps->T_sync = plan_val[kp][2]; ps->T_opt = plan_val[kp][3];
            ps->p = (u64)plan_val[kp][4];
            for (int w = 0; w < HAP_MAX_PP / 8; ++w) {                       // (words of later stages are whatever the thread's memory held)
                reinterpret_cast<u64 *>(ps->n)[w] = plan_n[kp][w];
                reinterpret_cast<u64 *>(ps->r)[w] = plan_r[kp][w];
            }
        }
    }
    // ---- the last block of the pass -------------------------------------------------------------------------------------
    if (ta.launch != 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&ta.state->blocks_done, 1u) + 1u == ta.blocks_total;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    tree_finish<kTreeThreads, SEARCH, F64>(ta, dc, __ldcg(&ta.state->n_feasible), __ldcg(&ta.state->n_pruned), 0, s_cost, s_index, &s_item);
}

// ------------------------------------------------------------------------------------------------------------------
// refinement objectives
// ------------------------------------------------------------------------------------------------------------------

// A warp per listed candidate: among its partitions without a stage above the bottleneck the one of the smallest sum, or (exact)
// the one of the smallest sum + (M - 1) max of all, by an additive recurrence over the candidate's bands whose limit on the
// stage cost is swept over the costs that occur.  Lanes run over the end layers.  Few candidates get here -- 169 of 1.35
// million at 256 devices -- so a chain of recurrences bounds it: the unlimited one comes first, because its sum tells
// whether the candidate can still beat the best one so far, and the sweep stops where it cannot any more.  An exact search
// of those 1.35 million: 1,316 us when a plain pass over all of them was followed by a warp per candidate of every block
// that held one left, 305 us in this form.
constexpr int kRefineWarps = 4;
inline size_t refine_smem_bytes(int N, int max_pp) { return (size_t)kRefineWarps * ((size_t)2 * (N + 1) * 8 + ((size_t)max_pp * (N + 1) + 15) / 16 * 16); }

template <bool NL>
__global__ void __launch_bounds__(kRefineWarps * 32)
tree_refine_kernel(const TreeArgs ta, const DevConst dc, int exact, int max_pp)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ i64 s_cost[kRefineWarps];
    __shared__ u64 s_index[kRefineWarps];
    __shared__ u32 s_item;
    __shared__ int s_last;
    const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
    const int N = ta.N, R = ta.R, n1 = N + 1, n_rc = ta.n_rc, RW = NL ? 2 : R;
    double *rows = reinterpret_cast<double *>(smem_raw) + (size_t)wib * 2 * n1;
    uint8_t *ch = smem_raw + (size_t)kRefineWarps * 2 * n1 * 8 + (size_t)wib * (((size_t)max_pp * n1 + 15) / 16 * 16);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const u64 listed = __ldcg(&ta.state->n_surv), n = listed < ta.max_surv ? listed : ta.max_surv;
    const u64 plain = ~__ldcg(&ta.state->incumbent);
    i64 best_cost = kInf, best_bott = 0, best_pipe = 0, best_sync = 0, best_opt = 0;
    u64 best_index = ~0ull, best_p = 0, n_refined = 0, n_ok = 0;
    int best_n = 0, best_r = 0;

    while (true) {
        u32 at = 0;
        if (lane == 0) at = atomicAdd(&ta.state->ticket[1], 1u);
        at = __shfl_sync(0xffffffffu, at, 0);
        if (at >= n) break;
        u64 bar = 0;                                        // nothing above it can win (one lane reads, the warp follows)
        if (lane == 0) { bar = ~*reinterpret_cast<volatile const u64 *>(&ta.state->refined); bar = plain < bar ? plain : bar; }
        bar = (u64)shfl_i64((i64)bar, 0);
        if ((u64)__ldcg(&ta.surv[at].lb) > bar) continue;
        const u64 c = __ldcg(&ta.surv[at].c);
        const double bott = (double)__ldcg(&ta.surv[at].bott);
        const TreeClass *cl = ta.cls + __ldcg(&ta.surv[at].ci);
        const unsigned char *rec = ta.rec + cl->rec_off + (u64)__ldcg(&ta.surv[at].slot) * cl->rec_bytes;
        const TreeHead *hd = reinterpret_cast<const TreeHead *>(rec);
        const hap_pconf pc = dc.pconf[hd->p];
        const int PP = pc.PP;
        const i64 M1 = hd->m1;
        const u64 loc = c - pc.offset, map_idx = loc / (u64)n_rc;
        const unsigned rc_mask = ta.rc_masks[loc - map_idx * (u64)n_rc];
        const double *ktab = reinterpret_cast<const double *>(rec + kTreeOffKtab), *minfo = reinterpret_cast<const double *>(rec + kTreeOffMinfo);
        const double *row0 = reinterpret_cast<const double *>(rec + cl->o_rows);

        // ---- this lane's stage: row group, capacity type, constant, window, band (the formulas of pipeline_dp_kernel) -----
        int mrow = 0, capt = 0, nmin = 0, nmax = 0, bl = 0, bh = 0, kidx = 0;
        double K = 0.0;
        i64 Pmin = 0;
        const StageMap sm = decode_stage(dc, pc, map_idx, lane);
        if (lane < PP) {
            bool seen = false;
            i64 cap = 0;
            for (int h = 0; h < dc.T; ++h)
                if (sm.mask >> h & 1) {
                    if (!seen || dc.P[h] < Pmin) Pmin = dc.P[h];
                    if (!seen || dc.cap_eff[h] < cap) { cap = dc.cap_eff[h]; capt = h; }
                    seen = true;
                }
            mrow = cl->mrow_of[sm.mask];
            kidx = lane == 0 ? mrow : 16 + sm.hb * 6 + (sm.cls == HAP_CROSS ? 2 + sm.ha : sm.cls);
            K = ktab[kidx] + (lane == PP - 1 ? minfo[mrow * kTreeMinfo + 6] : 0.0);
        }
        {
            const i64 Ps = warp_sum_i64(Pmin);
            if (lane < PP) {
                nmin = 1; nmax = N - PP + 1;
                if (dc.uniform) { nmin = N / PP; nmax = (N + PP - 1) / PP; }
                else if (dc.delta_q >= 0) {
                    const i64 den = 1024 * Ps;
                    const i64 lo = ((i64)(1024 - dc.delta_q) * Pmin * N) / den, hi = ((i64)(1024 + dc.delta_q) * Pmin * N + den - 1) / den;
                    nmin = lo < 1 ? 1 : (int)lo; nmax = hi > N - PP + 1 ? N - PP + 1 : (int)hi;
                }
            }
            int smin = nmin, smax = nmax;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, smin, o), b = __shfl_up_sync(0xffffffffu, smax, o);
                if (lane >= o) { smin += a; smax += b; }
            }
            const int tmin = __shfl_sync(0xffffffffu, smin, PP - 1), tmax = __shfl_sync(0xffffffffu, smax, PP - 1), i = lane + 1;
            bl = smin > i ? smin : i; bh = smax < N - PP + i ? smax : N - PP + i;
            const int rl = N - (tmax - smax), rh = N - (tmin - smin);
            bl = bl > rl ? bl : rl; bh = bh < rh ? bh : rh;
        }
        auto levels = [&](int d, int ct, int j) {
            u32 len4 = 0;
            if (cl->flat[d]) len4 = __ldg(reinterpret_cast<const u32 *>(rec + kTreeOffThr) + (d - 1) * HAP_MAX_TYPES + ct);
            else if (HAP_CHECK_OK(6, j >= (int)cl->jlo[d] && j <= (int)cl->jhi[d]))
                for (int r = 0; r < R; ++r) len4 |= (u32)__ldg(rec + cl->o_thr_nf + cl->nf_off[d] + (u32)(ct * R + r) * cl->nf_w[d] + (u32)(j - (int)cl->jlo[d])) << (8 * r);
            return tree_levels<4>(R, rc_mask, len4);
        };
        auto span = [&](int mr, int r, int k, int j, double kk) {
            if (!HAP_CHECK_OK(5, k >= 0 && k <= j && j <= N && r < R)) return kk;
            const double *row = row0 + (size_t)(mr * RW + (NL ? 0 : r)) * n1;
            return tree_span<false, NL>(__ldg(row + j), __ldg(row + k), NL ? __ldg(row + n1 + j) : 0.0, NL ? __ldg(row + n1 + k) : 0.0, 0.0, NL ? ta.tau[r] : 0.0) + kk;
        };
        auto level_of = [&](const TreeLevels &lv, int len) { return (len > lv.b0) + (len > lv.b1) + (len > lv.b2); };
        // cost of this lane's stage over (a, b]
        auto stage_of_lane = [&](int a, int b) -> double {
            if (lane >= PP) return 0.0;
            return span(mrow, level_of(levels(lane + 1, capt, b), b - a), a, b, K);
        };
        // one recurrence under a limit on the stage cost: false if no partition respects it; else the sum, the largest stage
        // cost of the chosen partition, this lane's span, and in nxt the smallest stage cost above the limit
        auto pass = [&](double limit, double &psum, double &pmax, double &nxt, int &pa, int &pb) -> bool {
            int pbl = 0, pbh = 0;
            double skipped = kTreeInf;
            for (int i = 1; i <= PP; ++i) {
                const int mr = __shfl_sync(0xffffffffu, mrow, i - 1), ct = __shfl_sync(0xffffffffu, capt, i - 1);
                const int lo_n = __shfl_sync(0xffffffffu, nmin, i - 1), hi_n = __shfl_sync(0xffffffffu, nmax, i - 1);
                const int lo_j = __shfl_sync(0xffffffffu, bl, i - 1), hi_j = __shfl_sync(0xffffffffu, bh, i - 1);
                const double kk = __shfl_sync(0xffffffffu, K, i - 1);
                const double *prev = rows + (size_t)(i & 1) * n1;
                double *cur = rows + (size_t)((i - 1) & 1) * n1;
                for (int j = lo_j + lane; j <= hi_j; j += 32) {
                    double best = kTreeInf;
                    int arg = 255;
                    const TreeLevels lv = levels(i, ct, j);
                    int a = lo_n > j - pbh ? lo_n : j - pbh, b = hi_n < j - pbl ? hi_n : j - pbl;
                    if (b > lv.nx) b = lv.nx;
                    for (int len = a; len <= b; ++len) {
                        const double cst = span(mr, level_of(lv, len), j - len, j, kk);
                        if (cst > limit) { skipped = cst < skipped ? cst : skipped; continue; }
                        const double v = (i == 1 ? 0.0 : prev[j - len]) + cst;
                        if (v <= best && v < kTreeBound) { best = v; arg = j - len; }
                    }
                    cur[j] = best;
                    if (HAP_CHECK_OK(2, i <= max_pp)) ch[(size_t)(i - 1) * n1 + j] = (uint8_t)arg;
                }
                __syncwarp();
                pbl = lo_j; pbh = hi_j;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) { const double t = __shfl_xor_sync(0xffffffffu, skipped, o); skipped = t < skipped ? t : skipped; }
            nxt = skipped;
            psum = rows[(size_t)((PP - 1) & 1) * n1 + N];
            pa = 0; pb = 0;
            if (!(psum < kTreeBound)) { __syncwarp(); return false; }
            int j = N;
            for (int i = PP; i >= 1; --i) {
                const int k = ch[(size_t)(i - 1) * n1 + j];
                if (lane == i - 1) { pa = k; pb = j; }
                if (!HAP_CHECK_OK(5, k < j)) break;
                j = k;
            }
            double m = stage_of_lane(pa, pb);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) { const double t = __shfl_xor_sync(0xffffffffu, m, o); m = t > m ? t : m; }
            pmax = m;
            __syncwarp();
            return true;
        };
        auto value = [&](double sum, double most) { return (i64)sum + M1 * (i64)most; };
        int a_me = 0, b_me = 0, ua = 0, ub = 0;
        double bs, bm, nx, us = 0.0, um = 0.0, unx;
        if (exact) {
            if (!pass(kTreeBound, us, um, unx, ua, ub)) continue;
            // the sum without a limit and the smallest maximum (whether Pruning 3 drops it, only its partition tells)
            if (ta.eta_q <= 0 && (u64)value(us, bott) > bar) { n_refined++; n_ok++; continue; }
        }
        n_refined++;
        if (!pass(bott, bs, bm, nx, a_me, b_me)) continue;  // (always feasible: the min-max partition respects the limit)
        if (exact) {
            // the first limit that reaches the smallest value wins
            i64 best = value(bs, bm);
            double t = nx;
            while (t < kTreeBound && value(us, t) < best && (ta.eta_q > 0 || (u64)value(us, t) <= bar)) {
                double cs, cm, cn;
                int ca, cb;
                if (pass(t, cs, cm, cn, ca, cb) && value(cs, cm) < best) { best = value(cs, cm); a_me = ca; b_me = cb; }
                t = cn;
            }
            if (value(us, um) < best) { a_me = ua; b_me = ub; }
        }
        // ---- Eq. 4 --------------------------------------------------------------------------------------------------
        const int len = b_me - a_me;
        int my_r = 0;
        double cst = 0.0, sy = 0.0, op = 0.0, het = 0.0;
        if (lane < PP) {
            my_r = level_of(levels(lane + 1, capt, b_me), len);
            cst = span(mrow, my_r, a_me, b_me, K);
            const int n_moe = moe_before(dc, b_me) - moe_before(dc, a_me);
            const double dm = (double)n_moe, dd = (double)(len - n_moe);
            const double *mi = minfo + mrow * kTreeMinfo;
            sy = mi[0] + dd * mi[1] + dm * mi[2];
            op = dd * mi[3] + dm * mi[4];
            if (ta.eta_q > 0) {
                if (lane > 0 && (kidx - 16) % 6 >= 2) het += ktab[kidx];
                het += dm * mi[5];
            }
        }
        double sum = cst, mxc = cst;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double t1 = __shfl_xor_sync(0xffffffffu, mxc, o), t2 = __shfl_xor_sync(0xffffffffu, sy, o), t3 = __shfl_xor_sync(0xffffffffu, op, o);
            sum += __shfl_xor_sync(0xffffffffu, sum, o); het += __shfl_xor_sync(0xffffffffu, het, o);
            mxc = t1 > mxc ? t1 : mxc; sy = t2 > sy ? t2 : sy; op = t3 > op ? t3 : op;
        }
        const i64 T_pipe = value(sum, mxc);
        i64 T_iter = T_pipe + (i64)sy + (i64)op;
        if (ta.eta_q > 0 && (i64)het * (i64)PP * 1024 > (i64)ta.eta_q * (i64)sum) T_iter = kInf;        // Pruning 3
        if (T_iter < kInf) n_ok++;
        if (T_iter < best_cost || (T_iter == best_cost && T_iter < kInf && c < best_index)) {
            best_cost = T_iter; best_index = c; best_bott = (i64)bott; best_pipe = T_pipe; best_sync = (i64)sy; best_opt = (i64)op;
            best_n = len; best_r = my_r; best_p = hd->p;
            if (lane == 0) atomicMax(&ta.state->refined, ~(u64)T_iter);
        }
    }

    if (lane == 0) {
        s_cost[wib] = best_cost; s_index[wib] = best_index;
        if (n_refined) { atomicAdd(&ta.state->n_refined, n_refined); atomicAdd(&ta.state->n_refined_ok, n_ok); }
    }
    __syncthreads();
    int win = 0;
    for (int q = 1; q < kRefineWarps; ++q) if (s_cost[q] < s_cost[win] || (s_cost[q] == s_cost[win] && s_index[q] < s_index[win])) win = q;
    if (wib == win) {
        PlanSlot *ps = ta.slots + blockIdx.x;
        if (lane == 0) {
            ta.slot_cost[blockIdx.x] = best_cost; ta.slot_index[blockIdx.x] = best_index;
            ps->bott = best_bott; ps->T_pipe = best_pipe; ps->T_sync = best_sync; ps->T_opt = best_opt; ps->p = best_p;
        }
        ps->n[lane] = (uint8_t)best_n; ps->r[lane] = (uint8_t)best_r;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&ta.state->blocks_done, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // candidates were dropped against the smallest plain T_iter: that decides the search unless every refined one is above it
    const u64 refined = ~__ldcg(&ta.state->refined), finite = __ldcg(&ta.state->n_finite), done = __ldcg(&ta.state->n_refined);
    const u64 again = listed > ta.max_surv || (finite > 0 && refined > plain) ? 1 : 0;
    tree_finish<kRefineWarps * 32, true, false>(ta, dc, __ldcg(&ta.state->n_refined_ok), __ldcg(&ta.state->n_pruned) + finite - done, again, s_cost, s_index, &s_item);
}

}  // namespace hap
